"""The launch-shape autotuner with few Krylov vectors: its Gram-Schmidt candidates run on
at most the gmres_restart + 1 vectors that a context holds.  Every restart length on
either side of the eight vectors it times otherwise: the tuned solve reaches its tolerance
(1e-10 of |b|; 1e-8 asked of the oracle's product, and with an FP32 operator its entries'
rounding, at most 60 terms of 2^-24 each), and the state that the context holds is untouched."""
import numpy as np
import pytest

from oracle import seird_oracle as O
from paper_2208_01839_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2208_01839_gb300 import build as _b  # noqa: E402

_b.build()
from paper_2208_01839_gb300 import seird as S  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("restart", [1, 2, 6, 7, 8, 30])
def test_tuning_stays_within_the_krylov_basis(restart, precision):
    wl = I.square_workload(17)
    J = O.jacobian(wl.xy, wl.tri, wl.params, 0.01, wl.U0)  # near the mass matrix: one vector a cycle converges
    b = np.random.default_rng(restart).standard_normal((wl.n, 5))
    with S.Solver(wl.xy, wl.tri, wl.params, n_subdomains=1, dt=0.01, overlap=0, ilu_fill=3, precision=precision,
                  gmres_restart=restart, gmres_rtol=1e-10, gmres_maxit=2000, autotune=1) as sv:
        sv.set_state(wl.U0)
        sv.jacobian(wl.U0)
        sv.precond_setup()
        x, its = sv.linear_solve(b)
        info = sv.info()
        assert np.array_equal(sv.get_state(), wl.U0)
    assert its > 0 and info["cgs_tile"] in (128, 256) and info["cgs_ctas"] > 0
    rounding = 60 * 2.0 ** -24 * np.linalg.norm(abs(J) @ np.abs(x).ravel()) if precision else 0.0
    assert np.linalg.norm(J @ x.ravel() - b.ravel()) <= 1e-8 * np.linalg.norm(b) + rounding
