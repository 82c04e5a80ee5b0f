"""Work splits that depend on the GPU's size and on shared memory: the trajectory
recursion's second and later turns of a warp (the batch sizes follow from the number of
SMs), and the reverse pair kernel with its pairs staged and not, by the warp count that
decides it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2406_07048_gb300 import synth
from tests.test_gpu_edges import GRAD_KW, _face_differences, _faces_scene, _mixed
from tests.test_gpu_traj import _bicycles

pytestmark = pytest.mark.gpu

BACK_KW = {k: GRAD_KW[k] for k in ("sigma", "prox", "rho_box", "damp")}


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2406_07048_gb300 import _build, binding
    _build.build()
    return binding


def _batch(per_sm, more):
    """per_sm scenarios per SM and `more`, horizons 1..12 with a few long ones, and
    scenarios from every turn of the deal (longest first, two to a group once there are
    more than four per SM): its first, last and middle places."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n = per_sm * n_sm + more
    horizons = [1 + (5 * s) % 12 for s in range(n)]
    for k, N in enumerate((33, 97, 40, 64)):
        horizons[(k * n) // 4] = N
    order = sorted(range(n), key=lambda s: -horizons[s])
    turn = 8 * n_sm if n > 4 * n_sm else 4 * n_sm
    places = {0, 1, n // 2, n - 2, n - 1}
    for t in range(0, n, turn):
        places |= {t, t + 1, t + turn // 2, t + turn - 2, t + turn - 1}
    return horizons, sorted({order[p] for p in places if 0 <= p < n})


SIZES = [(4, 0), (4, 1), (8, 1), (16, 1), (24, 1)]


@pytest.mark.parametrize("per_sm,more", SIZES)
def test_recursion_turns_match_oracle(B, ora, per_sm, more):
    """Two FP64 iterations against the oracle (1e-9 relative, the fixed-iteration parity
    bound) on scenarios of every turn."""
    horizons, picks = _batch(per_sm, more)
    sc = _bicycles(horizons)
    pb = B.Problem(B.DeviceScene(B.Context(0), sc, torch.float64))
    rep = pb.solve(max_iter=2, eps_pri=0.0, eps_dual=0.0)
    torch.cuda.synchronize()
    assert (rep["iters"].cpu().numpy() == 2).all()
    ref = ora.admm_batch(sc, max_iter=2, eps_pri=0.0, eps_dual=0.0, scenarios=picks)
    s_g, u_g = pb.s.cpu().numpy(), pb.u.cpu().numpy()
    for s in picks:
        a, b = int(sc.state_begin[s]), int(sc.state_begin[s + 1])
        c, d = int(sc.ctrl_begin[s]), int(sc.ctrl_begin[s + 1])
        for got, want in ((s_g[a:b], ref["s"][a:b]), (u_g[c:d], ref["u"][c:d])):
            assert np.abs(got - want).max() <= 1e-9 * (1.0 + np.abs(want).max()), (s, horizons[s])


def _gradients(B, sc, K=2):
    ds = B.DeviceScene(B.Context(0), sc, torch.float64)
    ds.warps = 2
    pb = B.Problem(ds)
    tape = B.new_tape(ds, K)
    rep = B.admm_solve(ds, pb.s_ref, pb.s, pb.u, pb.y, pb.zeta, pb.xi, tape=tape, max_iter=K, **GRAD_KW)
    g = B.admm_backward(ds, pb.s_ref, tape, rep["iters"], torch.ones(sc.n_scen, dtype=torch.float64, device=ds.device),
                        max_iter=K, **BACK_KW)
    return {k: v.cpu().numpy() for k, v in g.items()}


@pytest.mark.parametrize("per_sm,more", [(16, 1), (24, 1)])
def test_later_turns_leave_the_same_bits(B, per_sm, more):
    """Scenarios of every turn against the same scenarios in the first turn of a smaller
    batch that also takes two to a warp: solved and reversed by the same operations, so the
    same bits (the obstacles' gradients are added by atomics in any order: 1e-9)."""
    horizons, picks = _batch(per_sm, more)
    sc = _bicycles(horizons)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    fill = [s for s, N in enumerate(horizons) if N == 1 and s not in picks]
    fill = (fill * (4 * n_sm // len(fill) + 1))[:4 * n_sm + 1]
    full, first = _gradients(B, sc), _gradients(B, synth.subset(sc, picks + fill))
    for k, s in enumerate(picks):
        assert (first["state0"][k] == full["state0"][s]).all(), (s, horizons[s])
        j0, j1 = int(sc.obs_begin[s]), int(sc.obs_begin[s + 1])
        assert np.allclose(first["obs_offset"][3 * k:3 * k + 3], full["obs_offset"][j0:j1], rtol=1e-9, atol=1e-12)


# A staged warp of the reverse pair kernel keeps two pairs: 91 rows of 32 numbers each at 4
# robot and 24 obstacle faces in 2-D, 97 at 6 and 24 in 3-D, so in FP64 four warps (three in
# 3-D) are staged within 200 KB and five are not; the face reduction's third group starts at 17 faces.
@pytest.mark.parametrize("dim,faces,n_obs,N,warps",
                         [(2, 16, 3, 8, 2), (2, 17, 3, 8, 2), (2, 24, 3, 8, 2), (2, 24, 7, 8, 6), (3, 24, 2, 5, 2), (3, 24, 6, 5, 5)])
def test_pair_adjoint_face_groups(B, ora, dim, faces, n_obs, N, warps):
    """Offset gradients against central differences of the oracle (the bounds of the
    adjoint's test of face counts)."""
    sc, K = _faces_scene(dim, faces, n_obs, N), 3
    ds = B.DeviceScene(B.Context(0), sc, torch.float64)
    ds.warps = warps
    pb = B.Problem(ds)
    tape = B.new_tape(ds, K)
    rep = B.admm_solve(ds, pb.s_ref, pb.s, pb.u, pb.y, pb.zeta, pb.xi, tape=tape, max_iter=K, **GRAD_KW)
    g = B.admm_backward(ds, pb.s_ref, tape, rep["iters"], torch.ones(1, dtype=torch.float64, device=ds.device),
                        max_iter=K, **BACK_KW)
    got = g["obs_offset"].cpu().numpy()
    pairs = {(j, m) for j in (0, n_obs - 1) for m in (0, 7, 8, 15, faces - 1)}
    pairs |= {(int(i) // got.shape[1], int(i) % got.shape[1]) for i in np.argsort(-np.abs(got).ravel())[:5]}
    for j, m, fd, cost in _face_differences(ora, sc, K, GRAD_KW, sorted(pairs)):
        assert abs(got[j, m] - fd) <= 1e-4 * abs(fd) + 1e-8 * cost + 1e-8, (j, m, got[j, m], fd)


@pytest.mark.parametrize("scene", [lambda: _mixed(torch.float32), lambda: _faces_scene(3, 24, 17, 5)])
def test_pair_adjoint_staged_and_not_in_fp32(B, scene):
    """One FP32 tape, reversed with two warps a tile (staged) and eight (8 x (25 + 1) KB: not
    staged): the same adjoints with sums over lanes and warps in another order.  Every sum
    has fewer than 256 terms (2^8 roundings of 2^-24, 1.5e-5 of its terms), carried through
    two more reverse steps: 1e-3 of the largest gradient of the scene."""
    sc, K = scene(), 3
    ds = B.DeviceScene(B.Context(0), sc, torch.float32)
    ds.warps = 2
    pb = B.Problem(ds)
    tape = B.new_tape(ds, K)
    rep = B.admm_solve(ds, pb.s_ref, pb.s, pb.u, pb.y, pb.zeta, pb.xi, tape=tape, max_iter=K, **GRAD_KW)
    grads = []
    for w in (2, 8):
        ds.warps = w
        g = B.admm_backward(ds, pb.s_ref, tape, rep["iters"], torch.ones(sc.n_scen, device=ds.device), max_iter=K, **BACK_KW)
        grads.append({k: v.cpu().numpy() for k, v in g.items()})
    for k in ("obs_offset", "state0"):
        a, b = grads[0][k], grads[1][k]
        assert np.isfinite(a).all() and np.abs(b).max() > 0
        assert np.abs(a - b).max() <= 1e-3 * np.abs(b).max()
