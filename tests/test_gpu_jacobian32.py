"""The FP32 Jacobian of a mixed-precision context, bit for bit.

get_jacobian and apply_jacobian hand FP32 entries out in FP64, so a caller who repeats a
computation sees any change in the order of the FP32 sums (about 1e-7).  The entries are
held here: tests/golden/jacobian_fp32.json has those of every assembly form (both
quadratures, with and without a transmission field, Newton and Picard, rates of one
context and of an ensemble's table) on a distorted 3x3 mesh whose inputs are dyadic
fractions.  They were recorded on a GB300 (CUDA 13.0) from the form whose FP32 and FP64
kernels summed alike; the tolerance is zero.  On the CPU the recorded entries
are held against the oracle's FP64 matrix: the sums of an entry have at most 60 terms
and factors, each rounded to 2^-24 of the magnitudes summed.
"""
import base64
import json
import os

import numpy as np
import pytest

from oracle import seird_oracle as O
from oracle import seird_variants as V
from paper_2208_01839_gb300 import inputs as I

from paper_2208_01839_gb300 import build as _b

_b.build()
from paper_2208_01839_gb300 import seird as S  # noqa: E402

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "jacobian_fp32.json")
CASES = {  # quadrature, field, Picard, samples
    "deg5": (0, False, 0, 1),
    "deg5_field": (0, True, 0, 1),
    "vertex_field": (1, True, 0, 1),
    "picard_field": (0, True, 1, 1),
    "ensemble": (0, False, 0, 2),
    "ensemble_picard_vertex": (1, True, 1, 2),
}


def _inputs(name):
    rule, field, picard, samples = CASES[name]
    k = np.arange(9)
    xy = np.stack([(k % 3) / 2 + ((3 * k) % 5) / 64, (k // 3) / 2 + ((2 * k) % 7) / 64], axis=1)
    tri = []
    for j in range(2):
        for i in range(2):
            a = 3 * j + i
            tri += [[a, a + 1, a + 4], [a, a + 4, a + 3]]
    tri = np.array(tri, dtype=np.int32)
    i, c = np.meshgrid(np.arange(9 * samples), np.arange(5), indexing="ij")
    U = 1.0 + ((7 * i + 3 * c + i * c) % 23) / 8
    rates = [I.Params(A=1.5 + s / 4, beta_i=0.375 + s / 8, beta_e=0.3125, sigma=0.140625, gamma_e=0.15625 + s / 16,
                      gamma_r=0.046875, gamma_d=0.015625, alpha=0.0078125, mu=0.00390625,
                      nu=(0.03125, 0.0625, 0.001953125, 0.0234375 + s / 64)) for s in range(samples)]
    b = (1.0 + ((5 * k) % 9) / 16) if field else None
    return xy, tri, rates, U, b


def _matrix(name):
    """FP32 entries [nnzb, 5, 5] and the product with a dyadic vector."""
    rule, _, picard, samples = CASES[name]
    xy, tri, rates, U, b = _inputs(name)
    with S.Solver(xy, tri, rates if samples > 1 else rates[0], beta_field=b, n_subdomains=1, dt=0.5, overlap=0,
                  precision=1, quadrature=rule, nonlinear=picard) as sv:
        sv.jacobian(U)
        rp, col, val = sv.get_jacobian()
        x = np.where(np.arange(U.size) % 3 == 0, 1.0, -0.5).reshape(U.shape)
        return rp, col, val, x, sv.apply_jacobian(x)


def _golden(name):
    return np.frombuffer(base64.b64decode(json.load(open(GOLDEN))[name]), dtype="<f4").reshape(-1, 5, 5)


@pytest.mark.parametrize("name", CASES)
def test_recorded_entries_are_the_oracles_in_single_precision(name):
    rule, _, picard, samples = CASES[name]
    xy, tri, rates, U, b = _inputs(name)
    got = _golden(name).reshape(samples, -1, 5, 5)
    for s in range(samples):
        f = V.picard_matrix if picard else O.jacobian
        ref = O.to_bsr(f(xy, tri, rates[s], 0.5, U[9 * s:9 * s + 9], bfield=b, rule="vertex" if rule else "deg5"))[2]
        assert got[s].shape == ref.shape
        assert np.abs(got[s] - ref).max() <= 60 * 2.0 ** -24 * np.abs(ref).max()


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_entries_and_products_repeat_to_the_bit(name):
    rp, col, val, x, y = _matrix(name)
    gold = _golden(name).astype(np.float64)
    assert np.array_equal(val, gold)
    # the product accumulates in FP64, block by block in column order
    prod = np.einsum("bij,bj->bi", gold, x.reshape(-1, 5)[col])
    ref, mag = np.zeros_like(y), np.zeros_like(y)
    row = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    np.add.at(ref, row, prod)
    np.add.at(mag, row, np.einsum("bij,bj->bi", np.abs(gold), np.abs(x.reshape(-1, 5)[col])))
    assert np.all(np.abs(y - ref) <= 45 * 2.0 ** -53 * mag)
