"""Kernels on a scene whose tiles mix what the benchmark's scenes keep apart: five
parts of 3 to 8 faces per scenario (so that neighbouring lanes sit on parts with
different face counts), horizons from 1, one to 17 obstacles of 3 to 24 faces."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2406_07048_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2406_07048_gb300 import _build, binding
    _build.build()
    return binding


def _ngon(k, r, off):
    ang = 2.0 * math.pi * np.arange(k) / k + 0.1
    return np.stack([np.cos(ang), np.sin(ang)], 1), np.full(k, r), 0, np.array([off, 0.0])


def _mixed(dtype):
    model = synth.bicycle_model()
    scens = []
    for s, (N, M) in enumerate([(1, 1), (2, 9), (5, 17), (13, 3), (40, 8)]):
        rng = np.random.default_rng([31, s])
        obs = []
        for j in range(M):
            C, off = synth.random_polygon(rng, [3, 24, 7, 12][j % 4], 0.5, 2.0)
            obs.append((C, off, np.array([rng.uniform(5.0, 40.0), rng.uniform(0.0, 10.0)])))
        parts = [_ngon(k, 0.5 + 0.1 * k, 0.3 * k) for k in (3, 8, 4, 5, 6)]
        scens.append(synth._Scen(obs, parts, N, synth._ref_2d(model, N, 0.0, 2.0 * N, 5.0), np.zeros((N, model.nu))))
    sc = synth._assemble(model, scens, "mixed-parts")
    if dtype == torch.float32:  # the geometry as the library stores it
        for f in ("obs_C", "obs_d", "part_A", "part_b", "part_off", "s_ref", "s_init"):
            setattr(sc, f, getattr(sc, f).astype(np.float32).astype(np.float64))
    return sc


def _rounded(a, dtype):
    return a.astype(np.float32).astype(np.float64) if dtype == torch.float32 else a


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("warps", [1, 5])
def test_cert_margin_mixed_parts(B, ora, dtype, warps):
    """Margins of random sparse duals (with a negative, an infinite and a NaN one)
    against the oracle's FP64 bound on the same stored numbers: sums of at most 32
    products in another order (1e-12, floored at 1)."""
    sc = _mixed(dtype)
    rng = np.random.default_rng(5)
    states = _rounded(synth.random_states(sc, rng, 1.0, 0.4), dtype)
    P = sc.n_pairs
    lam = _rounded(rng.exponential(1.0, (P, sc.fr_max)) * (rng.uniform(size=(P, sc.fr_max)) < 0.5), dtype)
    mu = _rounded(rng.exponential(1.0, (P, sc.fo_max)) * (rng.uniform(size=(P, sc.fo_max)) < 0.2), dtype)
    bad = {3: -1.0, 40: np.inf, 77: np.nan}
    for p, v in bad.items():
        mu[p, 0] = v
    ds = B.DeviceScene(B.Context(0), sc, dtype)
    ds.warps = warps
    m_g = B.cert_margin(ds, ds.tensor(states), ds.to_device_pairs(lam), ds.to_device_pairs(mu)).cpu().numpy()
    pb, sb = sc.pair_begin, sc.state_begin
    for p in range(P):
        if p in bad:
            assert m_g[p] < -1e300
            continue
        s = int(np.searchsorted(pb, p, side="right")) - 1
        N, NP, l = int(sc.horizon[s]), sc.n_parts(s), p - int(pb[s])
        gm, gp, t = int(sc.obs_begin[s]) + l // (N * NP), int(sc.part_begin[s]) + l // N % NP, l % N + 1
        nr, nf = int(sc.part_nf[gp]), int(sc.obs_nf[gm])
        rho, R = ora.part_pose(sc.model, 0, sc.part_off[gp], states[int(sb[s]) + t])[:2]
        Cb, db = sc.obs_C[gm, :nf] @ R, sc.obs_d[gm, :nf] - sc.obs_C[gm, :nf] @ rho
        want = ora.cert_margin(sc.part_A[gp, :nr], sc.part_b[gp, :nr], Cb, db, lam[p, :nr], mu[p, :nf])
        if not np.isfinite(want):
            assert m_g[p] < -1e300
        else:
            assert abs(m_g[p] - want) <= 1e-12 * max(1.0, abs(want)), (p, m_g[p], want)


@pytest.mark.parametrize("ns,nu,N,S", [(2, 1, 63, 3), (5, 2, 64, 1), (12, 4, 65, 3), (7, 3, 71, 2), (6, 4, 520, 1), (4, 2, 72, 40)])
@pytest.mark.parametrize("method", [0, 1])
def test_lq_chunked_rollout_edges(B, ora, ns, nu, N, S, method):
    """Horizons around the chunked rollout's start and its remainders, unrolled and
    run-time dimensions, against the oracle's textbook recursion (1e-9 relative)."""
    from tests.test_oracle_riccati import _rand_lq
    rng = np.random.default_rng(100 * ns + N)
    probs = [_rand_lq(rng, N, ns, nu) for _ in range(S)]
    for pr in probs:
        pr[0][:] *= 0.9  # the closed loop stays bounded over the longer horizons
    dev = [torch.as_tensor(np.stack([pr[i] for pr in probs]), dtype=torch.float64, device="cuda") for i in range(8)]
    out = B.lq_solve(B.Context(0), *dev, method=method)
    torch.cuda.synchronize()
    assert (out["status"].cpu().numpy() == 0).all()
    for k in {0, S // 2, S - 1}:
        s_o, u_o, st = ora.riccati(*probs[k])
        assert st == 0
        for got, want in ((out["s"][k], s_o), (out["u"][k], u_o)):
            assert np.abs(got.cpu().numpy() - want).max() <= 1e-9 * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_cold_start_on_the_device(B, dtype):
    """The device's cold start is the scene's, element for element."""
    for sc in (_mixed(dtype), synth.config3(n_scen=5), synth.config4(n_scen=2, n_obs=8, N=5), synth.config_max()):
        ds = B.DeviceScene(B.Context(0), sc, dtype)
        assert torch.equal(ds.cold_y(), ds.to_device_pairs(sc.cold_y()))


def _faces_scene(dim, faces, n_obs, N):
    """One scenario whose obstacles all have `faces` faces."""
    rng = np.random.default_rng([31, dim, faces, n_obs])
    if dim == 2:
        model = synth.trailer_model()
        return synth._assemble(model, [synth._trailer_scen(rng, model, N, n_obs, faces, faces, 2.0 * N, 20.0, 2)], "faces")
    model = synth.quad_model()
    obs = []
    for _ in range(n_obs):
        C, off = synth.random_polyhedron(rng, faces, 0.3, 0.6)
        obs.append((C, off, np.array([rng.uniform(1.0, 3.0), rng.uniform(-1.5, 1.5), rng.uniform(1.5, 3.5)])))
    ref = np.zeros((N + 1, model.ns))
    ref[:, 2] = 2.5
    ref[:, 0] = 4.0 * np.arange(N + 1) / N
    ref[:, 3] = 4.0 / (N * model.dt)
    return synth._assemble(model, [synth._Scen(obs, synth._quad_parts(), N, ref, np.zeros((N, model.nu)))], "faces")


# faces: fewer than the eight summed together, eight, a second group, three; the last
# one is too large to be staged in FP64; obstacles: one warp, fewer and more than warps
FACES = [(2, 3, 1, 5), (2, 8, 5, 20), (2, 9, 9, 17), (2, 24, 20, 8), (3, 7, 3, 7), (3, 24, 9, 5)]


def _face_differences(ora, sc, K, kw, pairs, h=1e-4):
    """Central differences of the oracle's cost by obstacle offsets (step 1e-4: see the
    trajectory split's gradient test)."""
    import dataclasses
    out = []
    for j, m in pairs:
        costs = []
        for e in (h, -h):
            d = sc.obs_d.copy()
            d[j, m] += e
            costs.append(ora.admm_batch(dataclasses.replace(sc, obs_d=d), max_iter=K, **kw)["cost"].sum())
        out.append((j, m, (costs[0] - costs[1]) / (2 * h), abs(costs[0])))
    return out


GRAD_KW = dict(sigma=300.0, eps_pri=0.0, eps_dual=0.0, prox=0.1, rho_box=100.0, damp=100.0)


@pytest.mark.parametrize("dim,faces,n_obs,N", FACES)
def test_pair_adjoint_face_counts(B, ora, dim, faces, n_obs, N):
    """Offset gradients of staged and unstaged pairs against central differences of the
    oracle (FP64; the tolerance of the trajectory split's gradient test)."""
    sc, K = _faces_scene(dim, faces, n_obs, N), 3
    ds = B.DeviceScene(B.Context(0), sc, torch.float64)
    pb = B.Problem(ds)
    tape = B.new_tape(ds, K)
    rep = B.admm_solve(ds, pb.s_ref, pb.s, pb.u, pb.y, pb.zeta, pb.xi, tape=tape, max_iter=K, **GRAD_KW)
    g = B.admm_backward(ds, pb.s_ref, tape, rep["iters"], torch.ones(1, dtype=torch.float64, device=ds.device),
                        max_iter=K, **{k: GRAD_KW[k] for k in ("sigma", "prox", "rho_box", "damp")})
    got = g["obs_offset"].cpu().numpy()
    # the corners of the table and its five largest entries
    pairs = {(j, m) for j in (0, n_obs - 1) for m in (0, faces // 2, faces - 1)}
    pairs |= {(int(i) // got.shape[1], int(i) % got.shape[1]) for i in np.argsort(-np.abs(got).ravel())[:5]}
    for j, m, fd, cost in _face_differences(ora, sc, K, GRAD_KW, sorted(pairs)):
        assert abs(got[j, m] - fd) <= 1e-4 * abs(fd) + 1e-8 * cost + 1e-8, (j, m, got[j, m], fd)
