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
