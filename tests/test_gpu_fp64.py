"""The FP64 operations that the LQ solves form without a division or a compare
(oca_fp64.cuh), against IEEE arithmetic over the whole range of their operands, and the
entry points at operands near the ends of that range."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests.test_gpu_traj import _bicycles

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2406_07048_gb300 import _build, binding
    _build.build()
    return binding


@pytest.fixture(scope="module")
def ops(B, tmp_path_factory):
    from paper_2406_07048_gb300 import _build
    so = str(tmp_path_factory.mktemp("fp64") / "fp64.so")
    r = subprocess.run([_build.nvcc()] + _build.ARCH + _build.FLAGS + ["-shared", "-o", so,
                       os.path.join(ROOT, "tests", "gpu", "fp64.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return C.CDLL(so)


def _apply(fn, x, out):
    xt = torch.as_tensor(x, device="cuda")
    yt = torch.zeros(len(x), dtype=out, device="cuda")
    assert fn(C.c_void_p(xt.data_ptr()), C.c_void_p(yt.data_ptr()), C.c_int(len(x)),
              C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return yt.cpu().numpy()


def _operands():
    """Every exponent, subnormal ones among them, with random mantissas, the smallest and
    the largest; both signs."""
    rng = np.random.default_rng(11)
    bits = [np.uint64(e) << np.uint64(52) | m for e in range(2047)
            for m in (np.uint64(0), np.uint64(1), np.uint64(2**52 - 1), *rng.integers(0, 2**52, 40, dtype=np.uint64))]
    x = np.array(bits, dtype=np.uint64).view(np.float64)
    return np.concatenate([x, -x])


def test_recip_over_the_range(ops):
    """At most 0.57 units in the last place from 1 / x, whose own rounding moves the
    quotient by half a unit: not more than one number away from the correctly rounded one;
    the same number where 1 / x is formed by division."""
    x = _operands()
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
    got = _apply(ops.run_recip, x, torch.float64)
    sub = (np.abs(x) < 2.0**-1021) | (np.abs(x) >= 2.0**1021)
    assert (got[sub].view(np.int64) == want[sub].view(np.int64)).all()
    away = np.abs(got[~sub].view(np.int64) - want[~sub].view(np.int64))
    print(f"[recip] {np.mean(away != 0):.3g} of the quotients are not the rounded one")
    assert away.max() <= 1
    got = _apply(ops.run_recip, np.array([np.inf, -np.inf, np.nan]), torch.float64)
    assert got[0] == 0.0 and got[1] == 0.0 and np.isnan(got[2])


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_classes_over_the_range(ops, dtype):
    """positive_finite and finite are x > 0 and isfinite, also at both zeros, the smallest
    and largest numbers, the infinities and NaNs of both signs."""
    with np.errstate(over="ignore"):
        x = _operands().astype(dtype)
    ends = np.array([0.0, np.inf, np.nan, np.finfo(dtype).max, np.finfo(dtype).tiny], dtype=dtype)
    x = np.concatenate([x, ends, -ends])
    want = (np.isfinite(x) & (x > 0)) + 2 * np.isfinite(x)
    got = _apply(ops.run_classes if dtype == np.float64 else ops.run_classes_f32, x, torch.int32)
    assert (got == want).all()


@pytest.mark.parametrize("method", [0, 1])
def test_lq_with_a_huge_control_cost(B, method):
    """R = 1.5e308, r = 1e308 and controls that reach no state: u = -r / R (the reciprocal of
    R is a subnormal number of 51 bits: 1e-14)."""
    N, ns, nu = 3, 2, 2
    z = lambda *shape: torch.zeros(1, *shape, dtype=torch.float64, device="cuda")
    eye = lambda n, k: torch.eye(n, dtype=torch.float64, device="cuda").repeat(1, k, 1, 1)
    out = B.lq_solve(B.Context(0), eye(ns, N), z(N, ns, nu), z(N, ns), eye(ns, N + 1), z(N + 1, ns),
                     1.5e308 * eye(nu, N), z(N, nu) + 1e308, z(ns) + 1.0, method=method)
    torch.cuda.synchronize()
    assert int(out["status"][0]) == 0
    assert (out["u"] + 1e308 / 1.5e308).abs().max().item() <= 1e-14


def _one_step(B, ora, damp, speed):
    """One FP64 iteration of three bicycles of horizon 1 at `speed`, and the oracle's."""
    sc = _bicycles([1, 1, 1])
    sc.u_init[:] = 0.25
    sc.s_init[:, 3] = speed
    kw = dict(max_iter=1, eps_pri=0.0, eps_dual=0.0, damp=damp)
    pb = B.Problem(B.DeviceScene(B.Context(0), sc, torch.float64))
    rep = pb.solve(**kw)
    torch.cuda.synchronize()
    return pb, rep, ora.admm_batch(sc, **kw)


def test_trajectory_step_with_a_huge_damping(B, ora):
    """damp = 1e154 at 5 m/s: the 2 x 2 control Hessian is about damp diag(1.01, 1.25), its
    determinant 1.26e308 (above 2^1022), its product with the right-hand sides (up to 0.75
    damp) below the largest number.  Against the oracle (1e-9, the fixed-iteration parity
    bound)."""
    pb, rep, ref = _one_step(B, ora, 1e154, 5.0)
    assert (rep["iters"].cpu().numpy() == ref["iters"]).all() and (rep["status"].cpu().numpy() == ref["status"]).all()
    for got, want in ((pb.s, ref["s"]), (pb.u, ref["u"])):
        assert np.abs(got.cpu().numpy() - want).max() <= 1e-9 * (1.0 + np.abs(want).max())


@pytest.mark.parametrize("damp", [0.5e154, 0.9e154])
def test_an_overflow_in_the_gains_fails_the_scenario(B, ora, damp):
    """At 20 m/s the Hessian is about damp diag(1.01, 5) and the first right-hand side 2.2
    damp: their product, and at 0.9e154 the determinant too, passes the largest number.  The
    scenario is reported as failed, not returned with other gains."""
    _, rep, _ = _one_step(B, ora, damp, 20.0)
    assert rep["status"].cpu().tolist() == [2, 2, 2]


@pytest.mark.parametrize("growth,start,N", [(1e20, 0.0, 1024), (3.0, 1.0, 2176)])
@pytest.mark.parametrize("ns", [2, 12])
def test_lq_rollout_of_a_mode_that_feedback_does_not_reach(B, growth, start, N, ns):
    """A mode that grows per step, which no control reaches and no cost sees, at its
    equilibrium s = growth s + c: step by step it stays there, exactly (small whole numbers).
    Its map over a chunk of the horizon overflows or passes 2^53."""
    nu = 4 if ns == 12 else 1
    f = dict(dtype=torch.float64, device="cuda")
    A = torch.eye(ns, **f) * 0.5
    A[0, 0] = growth
    Bm, c, Q, s0 = torch.zeros(ns, nu, **f), torch.zeros(ns, **f), torch.eye(ns, **f), torch.ones(ns, **f)
    Bm[1:1 + nu, :] = torch.eye(min(nu, ns - 1), **f)
    Q[0, 0] = 0.0
    s0[0], c[0] = start, start * (1.0 - growth)
    rep = lambda x, k: x.repeat(1, k, *([1] * x.dim()))
    out = B.lq_solve(B.Context(0), rep(A, N), rep(Bm, N), rep(c, N), rep(Q, N + 1), torch.zeros(1, N + 1, ns, **f),
                     rep(torch.eye(nu, **f), N), torch.zeros(1, N, nu, **f), s0[None], method=0)
    torch.cuda.synchronize()
    assert int(out["status"][0]) == 0
    assert (out["s"][0, :, 0] == start).all()
    assert torch.isfinite(out["s"]).all() and torch.isfinite(out["u"]).all()
    assert out["s"][0, -1, 1:].abs().max().item() < 1e-100


@pytest.mark.parametrize("nu", [1, 2, 3, 4])
@pytest.mark.parametrize("method", [0, 1])
def test_lq_singular_is_relative_to_the_matrix(B, nu, method):
    """R = 1e-15 I is solved for every number of inputs (u = -r / R; one division and one
    product: 1e-15 and the product's rounding), R with equal rows, or 0, is refused."""
    N, ns = 2, 5
    z = lambda *shape: torch.zeros(2, *shape, dtype=torch.float64, device="cuda")
    eye = lambda n, k: torch.eye(n, dtype=torch.float64, device="cuda").repeat(2, k, 1, 1)
    R = 1e-15 * eye(nu, N)
    R[1, 1] = 1e-15 if nu > 1 else 0.0
    out = B.lq_solve(B.Context(0), eye(ns, N), z(N, ns, nu), z(N, ns), eye(ns, N + 1), z(N + 1, ns), R,
                     z(N, nu) + 3e-15, z(ns) + 1.0, method=method)
    torch.cuda.synchronize()
    assert out["status"].cpu().tolist() == [0, 1]
    assert (out["u"][0] + 3.0).abs().max().item() <= 1e-14
