"""The subdomain solve and factorisation where the small cases of test_gpu_solve_shapes do
not reach: subdomains of thousands of rows whose dependencies leave the window of 256
results that a CTA keeps in shared memory, in every ring; rows longer than the 32 blocks a
warp holds in the 256-thread factorisation (more than 152 subdomains); and rows of 119 to
236 blocks, which a context takes with the longer ring only.  Against the oracle's block
ILU sweeps, with its tolerances: 1e-10 in FP64, 1e-4 with FP32 factors."""
import functools

import numpy as np
import pytest

from oracle import seird_oracle as O
from paper_2208_01839_gb300 import inputs as I

from paper_2208_01839_gb300 import build as _b

_b.build()
from paper_2208_01839_gb300 import seird as S  # noqa: E402

WINDOW = 256
COUNTS = [2, 152, 153, 305, 457, 609]  # one ring each: one to four CTAs an SM, and more


@functools.lru_cache(maxsize=None)
def _scattered():
    """3,300 nodes in a random numbering: a seventh of a subdomain's rows has no lower
    neighbour, so its first level alone is longer than the window."""
    xy, tri, _ = I.irregular_mesh(3, 3300)
    at = np.random.default_rng(8).permutation(len(xy)).astype(np.int32)  # new number of each node
    new = np.empty_like(xy)
    new[at] = xy
    tri = at[tri]
    U0 = np.random.default_rng(9).uniform(1.0, 2.0, (len(xy), 5))
    p = I.params_ontario(12.0)
    return new, tri, p, U0, O.to_bsr(O.jacobian(new, tri, p, 0.5, U0))


def _uneven(n, count):
    """Two subdomains of more than 1,200 nodes each; the others share the rest."""
    big = (n - 900) // 2
    rest = np.arange(n - 2 * big)
    return np.concatenate([np.arange(2 * big) // big, 2 + rest * (count - 2) // len(rest)] if count > 2 else
                          [np.arange(n) * 2 // n]).astype(np.int32)


def test_the_first_level_of_a_large_subdomain_is_longer_than_the_window():
    xy, tri, _, _, (rp, col, _) = _scattered()
    for count in COUNTS:
        owner = _uneven(len(xy), count)
        assert len(np.unique(owner)) == count
        for q in (0, 1):
            rows = np.flatnonzero(owner == q)  # the nodes of the overlap only add rows after these
            low = [np.any((owner[c] == q) & (c < i)) for i in rows for c in [col[rp[i]:rp[i + 1]]]]
            assert len(rows) > 1200 and len(rows) - sum(low) > WINDOW - 64


@functools.lru_cache(maxsize=None)
def _scattered_reference(count):
    xy, tri, p, U0, (rp, col, val) = _scattered()
    r = np.random.default_rng(count).standard_normal(5 * len(xy))
    return r, O.ras_apply(rp, col, val, _uneven(len(xy), count), 1, r, coarse=False, ilu_fill=1)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", COUNTS)
def test_set_up_of_uneven_subdomains(count, precision):
    xy, tri = _scattered()[:2]
    st = S.setup_check(xy, tri, owner=_uneven(len(xy), count), overlap=1, ilu_fill=1, precision=precision)
    assert st["violations"] == 0 and st["n_subdomains"] == count


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", COUNTS)
def test_results_that_left_the_window(count, precision):
    xy, tri, p, U0, _ = _scattered()
    r, ref = _scattered_reference(count)
    outs = []
    with S.Solver(xy, tri, p, owner=_uneven(len(xy), count), dt=0.5, overlap=1, ilu_fill=1, precision=precision) as sv:
        sv.jacobian(U0)
        sv.precond_setup()
        for ring in (236, 118):
            for warps in (7, 3):
                sv.set_launch_shapes(ilu_warps=warps, ilu_ring=ring)
                outs.append(sv.precond_apply(r.reshape(-1, 5)).ravel())
    for o in outs[1:]:
        assert np.array_equal(outs[0], o)
    assert np.linalg.norm(outs[0] - ref) <= (1e-4 if precision else 1e-10) * np.linalg.norm(ref)


def _wheel(spokes, hub_last, count):
    """Triangle fan of `spokes` triangles around one node (subdomain 0: the hub's row has
    spokes + 1 blocks) and a strip of 880 nodes in count - 1 subdomains."""
    t = np.linspace(0.0, 2.0 * np.pi, spokes, endpoint=False)
    k = np.arange(spokes)
    tri = np.stack([0 * k, 1 + k, 1 + (k + 1) % spokes], axis=1)
    sxy, stri = I.structured_mesh(220, 4, x0=3.0, x1=5.0)
    xy = np.concatenate([[[0.0, 0.0]], np.stack([np.cos(t), np.sin(t)], 1), sxy])
    tri = np.concatenate([tri, stri + 1 + spokes]).astype(np.int32)
    owner = np.concatenate([np.zeros(1 + spokes), 1 + np.arange(880) * (count - 1) // 880]).astype(np.int32)
    if count == 1:
        owner[:] = 0
    if hub_last:
        xy, tri, owner = xy[::-1].copy(), (len(xy) - 1 - tri).astype(np.int32), owner[::-1].copy()
    return xy, tri, owner


def _wheel_apply(spokes, hub_last, count, fill, precision):
    """Relative distance of the preconditioner's application from the oracle's."""
    xy, tri, owner = _wheel(spokes, hub_last, count)
    p = I.params_ontario(40.0)
    U0 = np.random.default_rng(spokes).uniform(1.0, 2.0, (len(xy), 5))
    rp, col, val = O.to_bsr(O.jacobian(xy, tri, p, 0.5, U0))
    r = np.random.default_rng(1).standard_normal(5 * len(xy))
    ref = O.ras_apply(rp, col, val, owner, 0, r, coarse=False, ilu_fill=fill)
    with S.Solver(xy, tri, p, owner=owner, dt=0.5, overlap=0, ilu_fill=fill, precision=precision) as sv:
        sv.jacobian(U0)
        sv.precond_setup()
        if spokes > 118:
            with pytest.raises(S.SeirdError):
                sv.set_launch_shapes(ilu_ring=118)
        got = sv.precond_apply(r.reshape(-1, 5)).ravel()
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [153, 609])
@pytest.mark.parametrize("spokes", [31, 32, 33, 100])
def test_long_rows_in_the_256_thread_factorisation(spokes, count, precision):
    assert _wheel_apply(spokes, True, count, 1, precision) <= (1e-4 if precision else 1e-10)


RING_COUNTS = [1, 153, 305, 457, 609]
LONGEST = [(119, True), (187, True), (188, True), (189, True), (236, True), (119, False), (187, False), (188, False),
           (235, False)]  # lower blocks, or upper ones besides the pivot: 236 blocks at most


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", RING_COUNTS)
@pytest.mark.parametrize("spokes,hub_last", LONGEST)
def test_placement_of_rows_beyond_the_one_stage_ring(spokes, hub_last, count, precision):
    """The check reports such a stage only after it has found its place in the longer ring sound."""
    xy, tri, owner = _wheel(spokes, hub_last, count)
    with pytest.raises(S.SeirdError, match="stage exceeds the rings"):
        S.setup_check(xy, tri, owner=owner, overlap=0, ilu_fill=0, precision=precision)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", RING_COUNTS)
@pytest.mark.parametrize("spokes,hub_last", LONGEST)
def test_rows_beyond_the_one_stage_ring(spokes, hub_last, count, precision):
    assert _wheel_apply(spokes, hub_last, count, 0, precision) <= (1e-4 if precision else 1e-10)


@pytest.mark.gpu
@pytest.mark.parametrize("spokes,hub_last", [(237, True), (236, False)])
def test_rows_beyond_the_longer_ring_are_refused(spokes, hub_last):
    xy, tri, owner = _wheel(spokes, hub_last, 1)
    with pytest.raises(S.SeirdError, match="more blocks than the solve's shared-memory ring"):
        S.Solver(xy, tri, I.params_ontario(40.0), owner=owner, dt=0.5, overlap=0)
