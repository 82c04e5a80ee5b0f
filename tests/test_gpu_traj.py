"""The 2-D trajectory kernels at the sizes where their work split changes: one
scenario per warp and two, an odd count (a warp with one scenario), a second round
of the longest-first deal, horizons of a lane block and around it.  FP64, against
the oracle's ADMM on sampled scenarios; both run the same iterations in FP64 with
sums in another order (tolerance 1e-9 relative, the fixed-iteration parity bound)."""
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


def _bicycles(horizons):
    """One bicycle scenario of 3 obstacles per horizon."""
    model = synth.bicycle_model()
    scens = []
    for s, N in enumerate(horizons):
        rng = np.random.default_rng([21, s])
        keep = [np.array([0.0, 5.0]), np.array([2.0 * N, 5.0])]
        obs = synth._place_2d(rng, 3, 3, 8, 0.0, 2.0 * N + 30.0, 0.0, 10.0, keep, 5.0)
        scens.append(synth._Scen(obs, [synth._bicycle_body()], N, synth._ref_2d(model, N, 0.0, 2.0 * N, 5.0),
                                 np.zeros((N, model.nu))))
    return synth._assemble(model, scens, "traj-split")


@pytest.mark.parametrize("n_scen", [1, 608, 609, 1217])
def test_trajectory_split_matches_oracle(B, ora, n_scen):
    # 4 schedulers on each of 152 SMs: up to 608 scenarios take a warp each
    edge = [1, 2, 31, 32, 33, 95, 96, 97, 128]
    horizons = [edge[s % len(edge)] if s < 18 or s >= n_scen - 9 else 3 for s in range(n_scen)]
    sc = _bicycles(horizons)
    ds = B.DeviceScene(B.Context(0), sc, torch.float64)
    pb = B.Problem(ds)
    rep = pb.solve(max_iter=3, eps_pri=0.0, eps_dual=0.0)
    torch.cuda.synchronize()
    assert (rep["iters"].cpu().numpy() == 3).all()
    picks = sorted(set(range(min(n_scen, 18))) | set(range(max(0, n_scen - 9), n_scen)) | {n_scen // 2})
    ref = ora.admm_batch(sc, max_iter=3, eps_pri=0.0, eps_dual=0.0, scenarios=picks)
    s_g, u_g = pb.s.cpu().numpy(), pb.u.cpu().numpy()
    for s in picks:
        a, b = int(sc.state_begin[s]), int(sc.state_begin[s + 1])
        c, d = int(sc.ctrl_begin[s]), int(sc.ctrl_begin[s + 1])
        for got, want in ((s_g[a:b], ref["s"][a:b]), (u_g[c:d], ref["u"][c:d])):
            assert np.abs(got - want).max() <= 1e-9 * (1.0 + np.abs(want).max()), (s, horizons[s])


@pytest.mark.parametrize("extra", [0, 600])
def test_adjoint_split_matches_finite_differences(B, ora, extra):
    """Reverse steps over horizons around a block of steps (32 in the chain rule, 96 in
    the assembly) and over counts that take one and two scenarios per warp: gradients
    by the initial state and by the first obstacle's translation, against central
    differences of the oracle's costs per scenario (step 1e-4: the rounding of the
    costs, divided by the step, falls below the bound, which allows for
    two FP64 costs with a hundredfold growth over the steps and a step of 1e-6:
    1e-8 of the cost); 1e-4 relative is the bound of the other gradient tests."""
    import dataclasses

    horizons = [1, 2, 5, 31, 32, 33, 63, 64, 95, 96, 97] + [1] * extra
    sc, K, h = _bicycles(horizons), 3, 1e-4
    kw = dict(sigma=300.0, eps_pri=0.0, eps_dual=0.0, prox=0.1, rho_box=100.0, damp=100.0)
    row0 = np.concatenate([[0], np.cumsum([n + 1 for n in horizons])[:-1]])
    obs0 = np.asarray(sc.obs_begin)[:-1]

    def differences(change):
        costs = [ora.admm_batch(change(e), max_iter=K, **kw)["cost"] for e in (h, -h)]
        return (costs[0] - costs[1]) / (2 * h), np.abs(costs[0])

    def state(i):
        def change(e):
            s = sc.s_init.copy()
            s[row0, i] += e
            return dataclasses.replace(sc, s_init=s)
        return change

    def shift(i):
        def change(e):
            d = sc.obs_d.copy()
            d[obs0] += e * sc.obs_C[obs0][:, :, i]
            return dataclasses.replace(sc, obs_d=d)
        return change

    ctx = B.Context(0)
    ds = B.DeviceScene(ctx, sc, torch.float64)
    pb = B.Problem(ds)
    tape = B.new_tape(ds, K)
    rep = B.admm_solve(ds, pb.s_ref, pb.s, pb.u, pb.y, pb.zeta, pb.xi, tape=tape, max_iter=K, **kw)
    g = B.admm_backward(ds, pb.s_ref, tape, rep["iters"], torch.ones(sc.n_scen, dtype=torch.float64, device=ds.device),
                        max_iter=K, **{k: kw[k] for k in ("sigma", "prox", "rho_box", "damp")})
    g = {k: v.cpu().numpy() for k, v in g.items()}
    for i in range(sc.model.ns):
        fd, cost = differences(state(i))
        assert np.all(np.abs(g["state0"][:, i] - fd) <= 1e-4 * np.abs(fd) + 1e-8 * cost + 1e-8), i
    for i in range(2):
        fd, cost = differences(shift(i))
        assert np.all(np.abs(g["obs_center"][obs0, i] - fd) <= 1e-4 * np.abs(fd) + 1e-8 * cost + 1e-8), i
