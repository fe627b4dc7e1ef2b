"""SpMV on a caller's own matrix: rows taken by length within a CTA (51 rows), and FP32
values widened without the conversion instruction.  The sums of a row do not depend on
the order of the rows, and widening is exact, so every result equals that of FP64
values to the bit."""
import numpy as np
import pytest

from paper_2208_01839_gb300 import build as _b

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

_b.build()
from paper_2208_01839_gb300 import seird as S  # noqa: E402


def _spmv(rp, col, val, x):
    t = lambda a: torch.tensor(a, device="cuda")
    y = torch.full((5 * (len(rp) - 1),), np.nan, dtype=torch.float64, device="cuda")
    S.bsr_spmv(t(rp), t(col), t(val), t(x), y)
    torch.cuda.synchronize()
    return y.cpu().numpy()


@pytest.mark.parametrize("n", [1, 51, 52, 62016, 62017, 62067, 62068, 70001])
def test_rows_of_every_length_mix(n):
    """Rows of 0 to 19 blocks: below and above the size from which a CTA sorts its rows
    (62016 rows), with a last CTA of one row, of all but one and of all."""
    rng = np.random.default_rng(n)
    cnt = rng.integers(0, 20, n)
    rp = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int32)
    col = rng.integers(0, 40, rp[-1]).astype(np.int32)
    val = rng.standard_normal((len(col), 5, 5))
    x = rng.standard_normal(200)
    got = _spmv(rp, col, val, x)
    xb = x.reshape(-1, 5)[col]
    ref, mag = np.zeros((n, 5)), np.zeros((n, 5))
    row = np.repeat(np.arange(n), cnt)
    np.add.at(ref, row, np.einsum("bij,bj->bi", val, xb))
    np.add.at(mag, row, np.einsum("bij,bj->bi", np.abs(val), np.abs(xb)))
    assert np.all(np.abs(got.reshape(n, 5) - ref) <= 1e-13 * mag)


def test_float32_values_are_widened_exactly():
    special = np.array([0.0, -0.0, 1e-45, -1e-45, 1.1754942e-38, 1.17549435e-38, -1.17549435e-38, 3.4028235e38,
                        -3.4028235e38, np.inf, -np.inf, np.nan, 1.0, -1.5, 0.1, 2.0 ** -126, 2.0 ** 127],
                       dtype=np.float32)
    rng = np.random.default_rng(3)
    bits = rng.integers(0, 2 ** 32, 25 * 64 - len(special), dtype=np.uint32).view(np.float32)
    val = np.concatenate([special, bits]).reshape(64, 5, 5)
    val = val[~np.isnan(val).any(axis=(1, 2))]  # NaN payloads aside (one block keeps its NaN below)
    val[0, 4, 4] = np.nan
    rp = np.arange(len(val) + 1, dtype=np.int32)
    col = np.zeros(len(val), dtype=np.int32)
    for c in range(5):  # one column at a time: y holds the widened values themselves
        only = np.zeros_like(val)
        only[:, :, c] = val[:, :, c]
        x = np.zeros(5)
        x[c] = 1.0
        a, b = _spmv(rp, col, only, x), _spmv(rp, col, only.astype(np.float64), x)
        assert np.array_equal(a, b, equal_nan=True)
        assert np.array_equal(a, val[:, :, c].astype(np.float64).ravel(), equal_nan=True)


def test_float32_special_values_are_widened_exactly():
    """Zeros, the smallest and largest subnormals, the ends of every power of two (so of each
    exponent), infinities and a NaN, in blocks of five rows of one value each."""
    ends = np.arange(1, 255, dtype=np.uint32) << 23
    bits = np.concatenate([[0, 1, 2, 0x3fffff, 0x400000, 0x7ffffe, 0x7fffff], ends, ends | 0x7fffff, ends | 0x2aaaaa,
                           [0x7f800000, 0x7fc00000]]).astype(np.uint32)
    val = np.concatenate([bits, bits | 0x80000000]).astype(np.uint32).view(np.float32)
    assert len(val) == 1542 and (val == 0).sum() == 2 and np.isinf(val).sum() == 2 and np.isnan(val).sum() == 2
    assert np.isin(np.float32([1e-45, 1.1754942e-38, 1.17549435e-38, 3.4028235e38, 1.0, -1.0, 2.0 ** 127]), val).all()
    val = np.concatenate([val, np.zeros(-len(val) % 25, np.float32)]).reshape(-1, 5, 5)
    rp = np.arange(len(val) + 1, dtype=np.int32)
    col = np.zeros(len(val), dtype=np.int32)
    for c in range(5):  # one column at a time: y holds the widened values themselves
        only = np.zeros_like(val)
        only[:, :, c] = val[:, :, c]
        x = np.zeros(5)
        x[c] = 1.0
        assert np.array_equal(_spmv(rp, col, only, x), val[:, :, c].astype(np.float64).ravel(), equal_nan=True)
