"""The subdomain solve's forms: the factor ring that a context gets by its number of
subdomains (and precision), the split of small stages' rows when there are no more
subdomains than SMs, and both launch shapes of each, on either side of every change,
against the oracle's block ILU(1) sweeps.  The sums of a row are the same for every
launch shape, so those agree bit for bit.  Tolerances as for the preconditioner
elsewhere: 1e-10 in FP64, 1e-4 with FP32 factors."""
import functools

import numpy as np
import pytest

from oracle import seird_oracle as O
from paper_2208_01839_gb300 import inputs as I

from paper_2208_01839_gb300 import build as _b

_b.build()
from paper_2208_01839_gb300 import seird as S  # noqa: E402

COUNTS = [1, 152, 153, 304, 305, 456, 457, 608, 609]


@functools.lru_cache(maxsize=None)
def _problem():
    xy, tri, _ = I.irregular_mesh(3, 2600)
    dens = I.urban_density(3)
    U0 = I.urban_ic(xy, dens, 3)
    p = I.params_ontario(float(U0.sum(axis=1).max()))
    return xy, tri, p, U0, O.to_bsr(O.jacobian(xy, tri, p, 0.5, U0))


def _owner(n, count):
    return (np.arange(n) * count // n).astype(np.int32)


@functools.lru_cache(maxsize=None)
def _reference(count):
    xy, tri, p, U0, (rp, col, val) = _problem()
    r = np.random.default_rng(count).standard_normal(5 * len(xy))
    return r, O.ras_apply(rp, col, val, _owner(len(xy), count), 1, r, coarse=False, ilu_fill=1)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", COUNTS)
def test_stage_placement_holds_for_every_ring(count, precision):
    xy, tri = _problem()[:2]
    st = S.setup_check(xy, tri, owner=_owner(len(xy), count), overlap=1, ilu_fill=1, precision=precision)
    assert st["violations"] == 0 and st["n_subdomains"] == count


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", COUNTS)
def test_every_form_matches_the_oracle(count, precision):
    xy, tri, p, U0, _ = _problem()
    r, ref = _reference(count)
    outs = []
    with S.Solver(xy, tri, p, owner=_owner(len(xy), count), dt=0.5, overlap=1, ilu_fill=1, precision=precision) as sv:
        sv.jacobian(U0)
        sv.precond_setup()
        for ring in (236, 118):
            for warps in (7, 3):
                sv.set_launch_shapes(ilu_warps=warps, ilu_ring=ring)
                outs.append(sv.precond_apply(r.reshape(-1, 5)).ravel())
    for o in outs[1:]:
        assert np.array_equal(outs[0], o)
    assert np.linalg.norm(outs[0] - ref) <= (1e-4 if precision else 1e-10) * np.linalg.norm(ref)


def _wheel_strip(spokes, cells):
    """Triangle fan of `spokes` triangles around one node, on a strip of cells: the hub's row
    of the factors has spokes + 1 blocks."""
    t = np.linspace(0.0, 2.0 * np.pi, spokes, endpoint=False)
    xy = [np.array([[0.0, 0.0]]), np.stack([np.cos(t), np.sin(t)], 1)]
    tri = [[0, 1 + k, 1 + (k + 1) % spokes] for k in range(spokes)]
    sxy, stri = I.structured_mesh(cells, 4, x0=3.0, x1=5.0)
    xy.append(sxy)
    off = 1 + spokes
    return np.concatenate(xy), np.concatenate([np.array(tri), stri + off]).astype(np.int32)


@pytest.mark.parametrize("spokes,hub_last,accepted", [(117, False, True), (118, False, False),
                                                      (118, True, True), (119, True, False)])
def test_longest_row_of_the_one_stage_ring(spokes, hub_last, accepted):
    """118 blocks in a row's sweep: its lower ones, or its pivot and its upper ones."""
    xy, tri = _wheel_strip(spokes, 40)
    if hub_last:
        xy, tri = xy[::-1].copy(), (len(xy) - 1 - tri).astype(np.int32)
    check = functools.partial(S.setup_check, xy, tri, owner=np.zeros(len(xy), dtype=np.int32), overlap=0, ilu_fill=1)
    if accepted:
        assert check()["violations"] == 0
    else:
        with pytest.raises(S.SeirdError, match="stage exceeds the rings"):
            check()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("spokes", [5, 30, 31, 32, 33, 40, 100])
def test_rows_longer_than_a_warp_holds(spokes, precision):
    """A hub node numbered last has a lower row of `spokes` blocks: on either side of the 32
    blocks that a warp keeps in shared memory, and far beyond."""
    xy, tri = _wheel_strip(spokes, 40)
    n = len(xy)
    flip = (n - 1 - tri).astype(np.int32)  # the hub last
    xy, tri = xy[::-1].copy(), flip
    p = I.params_ontario(40.0)
    U0 = np.random.default_rng(spokes).uniform(1.0, 2.0, (n, 5))
    owner = np.zeros(n, dtype=np.int32)
    rp, col, val = O.to_bsr(O.jacobian(xy, tri, p, 0.5, U0))
    r = np.random.default_rng(1).standard_normal(5 * n)
    ref = O.ras_apply(rp, col, val, owner, 0, r, coarse=False, ilu_fill=1)
    with S.Solver(xy, tri, p, owner=owner, dt=0.5, overlap=0, ilu_fill=1, precision=precision) as sv:
        sv.jacobian(U0)
        sv.precond_setup()
        got = sv.precond_apply(r.reshape(-1, 5)).ravel()
    assert np.linalg.norm(got - ref) <= (1e-4 if precision else 1e-10) * np.linalg.norm(ref)
