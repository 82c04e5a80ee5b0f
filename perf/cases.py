"""Performance cases of the library: what a user's program calls, over the sizes it calls it with.

A case is a dict of plain values.  `op` names the public entry point (paper_2406_07048_gb300.binding):

  solve   admm_solve from a cold start: planning one scene, or a batch of scenes
  loop    mpc_run: closed-loop control steps of a batch of quadrotor runs
  grad    admm_solve with a tape, then admm_backward: gradients of the plan's cost
  detect  scale_detect: alpha*, certificates, margins and verdicts of a plan
  margin  cert_margin: FP64 certificate margins of given duals
  qp      pair_qp: one batch of pair QPs (step 1 alone), prox > 0 or the QP as printed (prox = 0)
  lq      lq_solve: batched step-2 LQ problems, parallel in time or sequential

Scenes are shaped like the repository's own configurations (synth.config1 .. config5, closed_loop): ragged horizons, obstacle
counts and face counts between the bounds that a case gives; the geometry is drawn from the seed.  Iteration counts stay below
the counts at which rounding alone moves the nonconvex iteration's result (blocked scenes amplify it with every iteration).
"""
import math

import numpy as np
import torch

from paper_2406_07048_gb300 import binding as B
from paper_2406_07048_gb300 import synth

DTYPES = {"f32": torch.float32, "f64": torch.float64}
NS = {"bicycle": 4, "trailer": 5, "quad": 12}
NU = {"bicycle": 2, "trailer": 2, "quad": 4}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _scene_case(name, op, kind, dtype, S, n, m, f, **more):
    c = {"name": name, "op": op, "kind": kind, "dtype": dtype, "S": S, "n0": n[0], "n1": n[1], "m0": m[0], "m1": m[1],
         "f0": f[0], "f1": f[1]}
    c.update(more)
    return c


def listed():
    return [
        # one vehicle plans once (synth.config1): the smallest whole solve, a chain of small launches
        _scene_case("solve-one-bicycle-f64", "solve", "bicycle", "f64", 1, (20, 20), (4, 4), (4, 8), iters=30, prox=1.0),
        # a fleet or a training set plans at once (synth.config3, the benchmark's step): 5.5 M pairs per iteration
        _scene_case("solve-batch-trailer-f32", "solve", "trailer", "f32", 2048, (20, 80), (8, 64), (3, 16), iters=3, prox=1.0),
        # 3-D: quadrotors among polyhedra (synth.config4), 983,040 pairs per iteration
        _scene_case("solve-batch-quad-f32", "solve", "quad", "f32", 64, (40, 40), (128, 128), (6, 20), iters=4, prox=1.0),
        # the paper's closed loop (synth.closed_loop): short horizons, many control steps, warm starts
        _scene_case("loop-quad-f32", "loop", "quad", "f32", 256, (16, 16), (32, 32), (6, 20), iters=4, prox=1.0, steps=30),
        # gradients of planned costs w.r.t. the obstacles (synth.config5)
        _scene_case("grad-batch-trailer-f32", "grad", "trailer", "f32", 256, (50, 50), (32, 32), (3, 12), iters=2, prox=1.0),
        # one plan checked before it is driven (synth.config2): the smallest call
        _scene_case("detect-one-trailer-f32", "detect", "trailer", "f32", 1, (50, 50), (32, 32), (3, 12)),
        # the plans of a whole batch checked (the benchmark's final check)
        _scene_case("detect-batch-trailer-f32", "detect", "trailer", "f32", 1024, (20, 80), (8, 64), (3, 16)),
        # FP64 margins of an ADMM's own duals, every pair of the batch
        _scene_case("margin-batch-trailer-f32", "margin", "trailer", "f32", 2048, (20, 80), (8, 64), (3, 16)),
        # step 1 alone on the 3-D scenes
        _scene_case("qp-batch-quad-f32", "qp", "quad", "f32", 64, (40, 40), (128, 128), (6, 20), prox=1.0),
        # step 1 as the paper prints it (prox = 0, the entry point's default)
        _scene_case("qp-printed-trailer-f32", "qp", "trailer", "f32", 128, (20, 80), (8, 64), (3, 16), prox=0.0),
        # one long-horizon LQ problem: the parallel-in-time form's use
        {"name": "lq-scan-one", "op": "lq", "method": "scan", "S": 1, "N": 256, "ns": 12, "nu": 4},
        # a batch of LQ problems: the sequential form's use
        {"name": "lq-sequential-batch", "op": "lq", "method": "sequential", "S": 256, "N": 64, "ns": 12, "nu": 4},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "detect", "margin", "qp", "loop", "grad", "lq"])
    if op == "lq":
        scan = rng.random() < 0.5
        ns, nu = rng.choice([(4, 2), (5, 2), (12, 4), (rng.randint(2, 12), rng.randint(1, 4))])
        return {"op": "lq", "method": "scan" if scan else "sequential", "S": _logint(rng, 1, 16 if scan else 256),
                "N": _logint(rng, 16, 256 if scan else 64), "ns": ns, "nu": nu}
    if op == "loop":
        n = rng.randint(10, 16)
        m = _logint(rng, 8, 32)
        return {"op": op, "kind": "quad", "dtype": "f32", "S": _logint(rng, 4, 256), "n0": n, "n1": n, "m0": m, "m1": m,
                "f0": 6, "f1": rng.randint(8, 20), "iters": rng.randint(2, 4), "prox": 1.0, "steps": rng.randint(3, 30)}
    if op == "grad":
        n = rng.randint(20, 50)
        return {"op": op, "kind": rng.choice(["bicycle", "trailer", "trailer"]), "dtype": "f32", "S": _logint(rng, 4, 256),
                "n0": n, "n1": rng.randint(n, 50), "m0": 4, "m1": rng.randint(8, 32), "f0": 3, "f1": rng.randint(5, 12),
                "iters": rng.randint(1, 2), "prox": 1.0}
    kind = rng.choice(["bicycle", "trailer", "trailer", "quad"])
    f64 = rng.random() < 0.25
    if kind == "quad":
        n = rng.randint(10, 40)
        m = _logint(rng, 8, 128)
        c = {"S": _logint(rng, 1, 16 if f64 else 64), "n0": n, "n1": rng.randint(n, 40), "m0": m, "m1": rng.randint(m, 128),
             "f0": 6, "f1": rng.randint(8, 20)}
    else:
        n, m = rng.randint(10, 60), rng.randint(4, 32)
        c = {"S": _logint(rng, 1, 128 if f64 else 1024), "n0": n, "n1": rng.randint(n, 80), "m0": m, "m1": rng.randint(m, 64),
             "f0": 3, "f1": rng.randint(4, 16)}
    c = {"op": op, "kind": kind, "dtype": "f64" if f64 else "f32", **c}
    if op == "solve":
        c["iters"] = rng.randint(3, 8) if f64 else rng.randint(2, 4) if kind == "quad" else rng.randint(2, 3)
        c["prox"] = rng.choice([1.0, 1.0, 0.3, 3.0])
    if op == "qp":
        c["prox"] = rng.choice([1.0, 1.0, 0.3, 0.0])
        if c["prox"] == 0.0:
            c["S"] = max(1, c["S"] // 8)
    return c


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
def _polygons(rng, nf, fmax):
    """Convex polygons: sorted uniform normal angles, every angular gap below pi (as synth.random_polygon), all at once."""
    M = len(nf)
    C, todo = np.zeros((M, fmax, 2)), np.arange(M)
    valid = np.arange(fmax)[None, :] < nf[:, None]
    while len(todo):
        v = valid[todo]
        a = np.sort(np.where(v, rng.uniform(0.0, 2.0 * math.pi, v.shape), np.inf), axis=1)
        last = a[np.arange(len(todo)), nf[todo] - 1]
        a1 = np.where(v, a, last[:, None])
        gap = np.maximum(np.diff(a1, axis=1).max(1), a1[:, 0] + 2.0 * math.pi - last)
        ok = gap < math.pi - 0.05
        C[todo[ok]] = np.where(v[ok][:, :, None], np.stack([np.cos(a1[ok]), np.sin(a1[ok])], 2), 0.0)
        todo = todo[~ok]
    return C, np.where(valid, rng.uniform(0.5, 2.0, (M, fmax)), 1.0)


def _polyhedra(rng, nf, fmax):
    """Bounded polyhedra: four normals of a randomly turned regular tetrahedron, the others uniform on the sphere."""
    M = len(nf)
    valid = np.arange(fmax)[None, :] < nf[:, None]
    C = rng.normal(size=(M, fmax, 3))
    turn, _ = np.linalg.qr(rng.normal(size=(M, 3, 3)))
    C[:, :4] = np.einsum("kj,mij->mki", np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]) / math.sqrt(3.0), turn)
    C /= np.linalg.norm(C, axis=2, keepdims=True)
    return np.where(valid[:, :, None], C, 0.0), np.where(valid, rng.uniform(0.3, 1.5, (M, fmax)), 1.0)


def _rejected(rng, n, draw_points, bad):
    pts, todo = draw_points(np.arange(n)), np.arange(n)
    todo = todo[bad(pts, todo)]
    while len(todo):
        pts[todo] = draw_points(todo)
        todo = todo[bad(pts[todo], todo)]
    return pts


def _scene(case, seed):
    """The scene of a case, and (for the closed loop) the reference of every control step."""
    rng = np.random.default_rng([int(seed), 7])
    S, kind = case["S"], case["kind"]
    # the sizes are the case's own: every seed gives another geometry of the same ragged sizes
    size = np.random.default_rng([S, case["n0"], case["n1"], case["m0"], case["m1"], case["f0"], case["f1"]])
    N = size.integers(case["n0"], case["n1"] + 1, S)
    M = size.integers(case["m0"], case["m1"] + 1, S)
    ob = np.concatenate([[0], np.cumsum(M)])
    scen = np.repeat(np.arange(S), M)
    mt = int(ob[-1])
    nf = size.integers(case["f0"], case["f1"] + 1, mt)
    fo = int(nf.max())
    ref_loop = None
    if kind == "quad":
        model = synth.quad_model()
        halves = [np.array([0.15, 0.15, 0.05]), np.array([0.25, 0.025, 0.025]), np.array([0.025, 0.25, 0.025])]
        links, offs, NP = [0, 0, 0], [np.zeros(3)] * 3, np.full(S, 3)
        C, off = _polyhedra(rng, nf, fo)
        if case["op"] == "loop":
            T = case["steps"]
            start, goal = np.array([0.0, 0.0, 1.0]), np.array([0.0, 70.0, 1.0])
            dense = np.arange(mt) - ob[scen] >= np.maximum(1, M[scen] // 4)

            def pts(i):
                # the first seconds of a run in its dense part: the obstacles stand along the stretch that is flown
                y = np.where(dense[i], rng.uniform(3, 3 + 0.9 * T, len(i)), rng.uniform(3, 68, len(i)))
                return np.stack([rng.uniform(-10, 10, len(i)), y, rng.uniform(0, 6, len(i))], 1)
            ctr = _rejected(rng, mt, pts, lambda p, i: np.minimum(np.linalg.norm(p - start, axis=1),
                                                                  np.linalg.norm(p - goal, axis=1)) < 2.5)
            Nm, duration = int(N.max()), 25.0
            tt = np.arange(T + Nm + 1) * model.dt
            refs = []
            for _ in range(S):
                way = np.stack([rng.uniform(-5, 5, 5), np.sort(rng.uniform(5.0, 65.0, 5)), rng.uniform(1.0, 3.0, 5)], 1)
                p = np.vstack([start, way, goal])
                seg = np.linalg.norm(np.diff(p, axis=0), axis=1)
                tk = np.concatenate([[0.0], np.cumsum(seg)]) / seg.sum() * duration
                ref = np.zeros((len(tt), 12))
                for i in range(3):
                    ref[:, i] = np.interp(tt, tk, p[:, i])
                ref[:-1, 3:6] = np.diff(ref[:, 0:3], axis=0) / model.dt
                refs.append(ref)
            ref_loop = np.stack(refs)
            s_ref = np.concatenate([ref_loop[s, :N[s] + 1] for s in range(S)])
        else:
            start, goal = np.array([0.0, 10.0, 2.5]), np.array([20.0, 10.0, 2.5])
            ctr = _rejected(rng, mt, lambda i: rng.uniform([0, 0, 0], [20, 20, 5], (len(i), 3)),
                            lambda p, i: np.minimum(np.linalg.norm(p - start, axis=1), np.linalg.norm(p - goal, axis=1)) < 2.0)
            # half of the obstacles beside the path, in pairs that leave a gap of 0.6 to 1 m
            k = np.arange(mt) - ob[scen]
            near = k < M[scen] // 2
            pair = np.cumsum(k % 2 == 0) - 1
            npr = int(pair.max()) + 1
            a, gap, up = rng.uniform(0.15, 0.85, npr)[pair], rng.uniform(0.6, 1.0, npr)[pair], (rng.uniform(size=npr) < 0.5)[pair]
            away = (gap / 2 + np.where(np.arange(fo)[None, :] < nf[:, None], off, 0.0).max(1)) * np.where(k % 2 == 0, 1.0, -1.0)
            side = start + a[:, None] * (goal - start) + away[:, None] * np.where(up[:, None], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0])
            ctr = np.where(near[:, None], side, ctr)
            tt = np.concatenate([np.arange(n + 1) / n for n in N])
            s_ref = np.zeros((len(tt), 12))
            s_ref[:, 0:3] = start + tt[:, None] * (goal - start)
            s_ref[:, 3:6] = (goal - start) / (np.repeat(N, N + 1)[:, None] * model.dt)
    else:
        one = kind == "bicycle"
        model = synth.bicycle_model() if one else synth.trailer_model()
        length = (2.0 if one or case["n0"] != case["n1"] else 100.0 / case["n0"]) * N
        width, v = (10.0, 20.0) if one else (20.0, 10.0)
        reach, keep = np.minimum(length, v * N * model.dt), 5.0 if one else 8.0
        halves = [np.array([2.25, 1.0])] if one else [np.array([2.0, 1.0]), np.array([3.0, 1.1])]
        links, offs = ([0], [np.array([1.25, 0.0])]) if one else ([0, 1], [np.array([1.5, 0.0]), np.array([-3.5, 0.0])])
        NP = np.ones(S, int) if one else (size.integers(1, 3, S) if case["n0"] != case["n1"] else np.full(S, 2))
        C, off = _polygons(rng, nf, fo)
        room = np.maximum(length, 2.0 * keep + 8.0)

        def pts2(i):
            return np.stack([rng.uniform(0.0, 1.0, len(i)) * room[scen[i]], rng.uniform(0.0, width, len(i))], 1)

        def bad2(p, i):
            return np.minimum(np.hypot(p[:, 0], p[:, 1] - width / 2),
                              np.hypot(p[:, 0] - reach[scen[i]], p[:, 1] - width / 2)) < keep
        ctr = _rejected(rng, mt, pts2, bad2)
        t = np.concatenate([np.arange(n + 1) for n in N])
        vel = np.repeat(reach / (N * model.dt), N + 1)
        s_ref = np.zeros((len(t), model.ns))
        s_ref[:, 0], s_ref[:, 1], s_ref[:, 3] = vel * model.dt * t, width / 2, vel
    boxes = [synth.box_halfspaces(h) for h in halves]
    which = np.concatenate([np.arange(n) for n in NP])
    off = np.where(np.arange(fo)[None, :] < nf[:, None], off, 0.0)
    d = np.where(np.arange(fo)[None, :] < nf[:, None], off + np.einsum("mfi,mi->mf", C, ctr), 1.0)
    i32 = lambda a: np.asarray(a, np.int32)  # noqa: E731
    sc = synth.Scene(dim=model.dim, model=model, obs_begin=i32(ob), obs_nf=i32(nf), obs_C=C, obs_d=d, obs_center=ctr, obs_off=off,
                     part_begin=i32(np.concatenate([[0], np.cumsum(NP)])), part_nf=i32([len(boxes[w][1]) for w in which]),
                     part_A=np.stack([boxes[w][0] for w in which]), part_b=np.stack([boxes[w][1] for w in which]),
                     part_link=i32([links[w] for w in which]), part_off=np.stack([offs[w] for w in which]), horizon=i32(N),
                     s_ref=s_ref, s_init=s_ref.copy(), u_init=np.zeros((int(N.sum()), model.nu)), name="case")
    return sc, ref_loop


def _pair_index(sc):
    """Obstacle, part and state row of every pair, as int64 arrays on the GPU (obstacle slowest, step fastest)."""
    M, NP, N = np.diff(sc.obs_begin), np.diff(sc.part_begin), sc.horizon
    scen = np.repeat(np.arange(sc.n_scen), M * NP)
    first = np.concatenate([[0], np.cumsum(M * NP)])
    k = np.arange(len(scen)) - first[scen]
    g = lambda a: torch.as_tensor(a.astype(np.int64), device="cuda")  # noqa: E731
    n = g(N[scen])
    rep = lambda a: torch.repeat_interleave(g(a), n)  # noqa: E731
    begin = torch.cumsum(n, 0) - n
    t = torch.arange(sc.n_pairs, device="cuda") - torch.repeat_interleave(begin, n) + 1
    return rep(sc.obs_begin[scen] + k // NP[scen]), rep(sc.part_begin[scen] + k % NP[scen]), rep(sc.state_begin[scen]) + t


def _cold_y(sc, part, dtype):
    """The cold start of synth.Scene.cold_y, component-major on the GPU."""
    y = torch.zeros(sc.ny_max, sc.n_pairs, dtype=dtype, device="cuda")
    e = np.argmax(sc.part_b, axis=1)
    val = torch.as_tensor(1.0 / sc.part_b[np.arange(len(e)), e], dtype=dtype, device="cuda")[part]
    ek = torch.as_tensor(e, device="cuda")[part]
    return y.scatter_(0, ek[None, :], val[None, :])


def _duals(sc, gen, obs, part, row, states, sparse):
    """Feasible duals: lambda on the simplex b.lambda = 1, mu on a share of the obstacle's faces, smaller when it is far."""
    r = lambda n: torch.rand(n, sc.n_pairs, generator=gen, dtype=torch.float64, device="cuda")  # noqa: E731
    g = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    b, FR, FO = g(sc.part_b)[part].T, sc.fr_max, sc.fo_max
    lam = r(FR) * (r(FR) < 0.4)
    lam[0] += (lam.sum(0) == 0).double()
    lam = lam / (b * lam).sum(0)
    far = (g(sc.obs_center)[obs] - g(states)[row][:, :sc.dim]).norm(dim=1)
    nf = torch.as_tensor(sc.obs_nf, device="cuda")[obs]
    mu = r(FO) * (r(FO) < sparse) * (torch.arange(FO, device="cuda")[:, None] < nf) / (1.0 + far)
    return torch.cat([lam, mu, 0.1 * r(1) * (r(1) < 0.3)])


def _lq_data(case, seed):
    rng = np.random.default_rng([int(seed), 8])
    S, N, n, m = case["S"], case["N"], case["ns"], case["nu"]
    spd = lambda L, k: L @ np.swapaxes(L, -1, -2) / k + 0.1 * np.eye(k)  # noqa: E731
    # mildly contracting dynamics: a long horizon stays as bounded as a controlled vehicle's linearisation
    out = [0.98 * (np.eye(n) + 0.05 * rng.normal(size=(S, N, n, n))), 0.2 * rng.normal(size=(S, N, n, m)), 0.1 * rng.normal(size=(S, N, n)),
           spd(rng.normal(size=(S, N + 1, n, n)), n), rng.normal(size=(S, N + 1, n)), spd(rng.normal(size=(S, N, m, m)), m),
           rng.normal(size=(S, N, m)), rng.normal(size=(S, n))]
    return [torch.as_tensor(a, dtype=torch.float64, device="cuda") for a in out]


_CTX = []


def _context():
    if not _CTX:
        _CTX.append(B.Context(0))
    return _CTX[0]


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    op = case["op"]
    st = {"case": dict(case)}
    if op == "lq":
        st["data"] = _lq_data(case, seed)
        n = B.lq_workspace_bytes(case["ns"], case["nu"], case["N"], case["S"])
        st["work"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        return st
    dtype = DTYPES[case["dtype"]]
    sc, ref = _scene(case, seed)
    ds = B.DeviceScene(_context(), sc, dtype)
    st["ds"] = ds
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if op == "loop":
        st["ref"], st["x0"] = ref, ref[:, 0].copy()
        return st
    obs, part, row = _pair_index(sc)
    if op in ("solve", "grad"):
        st["s_ref"] = ds.tensor(sc.s_ref)
        st["start"] = [ds.tensor(sc.s_init), ds.tensor(sc.u_init), _cold_y(sc, part, dtype),
                       torch.zeros(sc.n_pairs, dtype=dtype, device="cuda"), torch.zeros(sc.dim, sc.n_pairs, dtype=dtype, device="cuda")]
        st["live"] = [t.clone() for t in st["start"]]
        if op == "grad":
            st["tape"] = B.new_tape(ds, case["iters"])
            st["seed"] = torch.rand(sc.n_scen, generator=gen, dtype=dtype, device="cuda") + 0.5
        return st
    states = synth.random_states(sc, np.random.default_rng([int(seed), 9]), 1.0, 0.3)
    st["states"] = ds.tensor(states)
    if op == "margin":
        y = _duals(sc, gen, obs, part, row, states, 0.2).to(dtype)
        st["lam"], st["mu"] = y[:sc.fr_max].contiguous(), y[sc.fr_max:sc.fr_max + sc.fo_max].contiguous()
    elif op == "qp":
        st["y"] = _duals(sc, gen, obs, part, row, states, 0.15).to(dtype)
        st["zeta"] = 0.3 * torch.randn(sc.n_pairs, generator=gen, dtype=dtype, device="cuda")
        st["xi"] = 0.3 * torch.randn(sc.dim, sc.n_pairs, generator=gen, dtype=dtype, device="cuda")
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "lq":
        return B.lq_solve(_context(), *st["data"], method=B.OCA_LQ_SCAN if case["method"] == "scan" else B.OCA_LQ_SEQUENTIAL,
                          work=st["work"])
    ds = st["ds"]
    if op == "detect":
        return B.scale_detect(ds, st["states"])
    if op == "margin":
        return B.cert_margin(ds, st["states"], st["lam"], st["mu"])
    if op == "qp":
        return B.pair_qp(ds, st["states"], st["zeta"], st["xi"], st["y"], prox=case["prox"])
    if op == "loop":
        out = B.mpc_run(ds, st["ref"], ds.scene.obs_center, st["x0"], case["steps"], max_iter=case["iters"], prox=case["prox"])
        # the plan, its duals y and the run; the scaled duals of collision-free pairs are sums of rounding errors around zero
        return {k: out[k] for k in ("x", "x_hist", "u_hist", "iters", "collided", "s", "u", "y")}
    for dst, src in zip(st["live"], st["start"]):
        dst.copy_(src)
    s, u, y, zeta, xi = st["live"]
    rep = B.admm_solve(ds, st["s_ref"], s, u, y, zeta, xi, max_iter=case["iters"], prox=case["prox"], tape=st.get("tape"))
    out = {"s": s, "u": u, "y": y, "zeta": zeta, "xi": xi, **rep}
    if op == "grad":
        out.update(B.admm_backward(ds, st["s_ref"], st["tape"], rep["iters"], st["seed"], max_iter=case["iters"],
                                   prox=case["prox"]))
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: each input read once, each output written once.  Flops: expected face counts times what a pair cannot do without
    (per face of one evaluation of its dual 4 V + 4 with V = dim + 1; two evaluations, one Newton system and the sums of y per
    pair QP), and per stage of the trajectory step the products of the recursion over the model's nonzeros."""
    if case["op"] == "lq":
        S, N, n, m = case["S"], case["N"], case["ns"], case["nu"]
        per = n * n + n * m + n + n * n + n + m * m + m + n + m + n * n + n
        return {"bytes": 8.0 * S * N * per, "flops": 2.0 * S * N * (1.5 * n * n * n + 2 * n * n * m + 2 * n * m * m + 4 * n * n)}
    es = 4 if case["dtype"] == "f32" else 8
    kind, S = case["kind"], case["S"]
    D, ns, nu = (3, 12, 4) if kind == "quad" else (2, NS[kind], 2)
    V = D + 1
    N, M, nf = (case["n0"] + case["n1"]) / 2, (case["m0"] + case["m1"]) / 2, (case["f0"] + case["f1"]) / 2
    NP = 3 if kind == "quad" else 1 if kind == "bicycle" else 1.5 if case["n0"] != case["n1"] else 2
    nr = 6 if kind == "quad" else 4
    P = S * N * M * NP
    ny = nr + nf + 1
    face = 4 * V + 4
    if case["op"] == "detect":
        return {"bytes": P * (es * (1 + nr + nf) + 8 + 4 + 4), "flops": P * (nr + nf) * 2 * V * (V + 1)}
    if case["op"] == "margin":
        return {"bytes": P * (es * (nr + nf) + 8), "flops": P * (nr * 2 * (D + 1) + nf * 2 * (D + 1) + 4 * D * D)}
    qp = 2 * (nr + nf) * face + V * V * V + (nr + nf) * 2 * V
    if case["op"] == "qp":
        return {"bytes": P * (es * (2 * ny + 1 + D + V + 1) + 4), "flops": P * qp}
    its = case["iters"] * case.get("steps", 1)
    stage = 1600 if kind == "quad" else 400
    state = S * (N + 1) * ns + S * N * nu
    moved = es * (P * (2 * ny + 2 * (1 + D)) + 3 * state)
    flops = its * (P * qp + S * N * stage)
    if case["op"] == "grad":
        moved += es * S * M * (nf + D)
        flops *= 3
    if case["op"] == "loop":
        moved += es * S * case["steps"] * (2 * ns + nu)
    return {"bytes": float(moved), "flops": float(flops)}


# ---------------------------------------------------------------------------
# exact: the same results in plain FP64 torch
# ---------------------------------------------------------------------------
class _Geo:
    """A scene's geometry as the library holds it (rounded to the case's type), in FP64 on the GPU."""

    def __init__(self, sc, dtype):
        self.sc, self.dtype = sc, dtype
        g = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda").double()  # noqa: E731
        self.g = g
        self.C, self.d, self.A, self.b, self.off = g(sc.obs_C), g(sc.obs_d), g(sc.part_A), g(sc.part_b), g(sc.part_off)
        i = lambda a: torch.as_tensor(a.astype(np.int64), device="cuda")  # noqa: E731
        self.nf, self.nr, self.link = i(sc.obs_nf), i(sc.part_nf), i(sc.part_link)
        self.obs, self.part, self.row = _pair_index(sc)
        m = sc.model
        self.p = [float(v) for v in m.param]
        self.dt = float(m.dt)

    def pose1(self, s, link, off):
        """rho and R of one part at one state (functional torch: differentiable in s)."""
        if self.sc.dim == 2:
            tr = link.double()
            a = s[2] if len(s) == 4 else s[2] * (1 - tr) + s[4] * tr
            c, n = torch.cos(a), torch.sin(a)
            R = torch.stack([torch.stack([c, -n]), torch.stack([n, c])])
            hitch = self.p[1] * tr if len(s) == 5 else 0.0 * tr
            rho = s[:2] + R @ off - hitch * torch.stack([torch.cos(s[2]), torch.sin(s[2])])
            return rho, R
        cf, sf, ct, st, cp, sp = (f(s[6 + i]) for i in range(3) for f in (torch.cos, torch.sin))
        R = torch.stack([torch.stack([cp * ct, cp * st * sf - sp * cf, cp * st * cf + sp * sf]),
                         torch.stack([sp * ct, sp * st * sf + cp * cf, sp * st * cf - cp * sf]),
                         torch.stack([-st, ct * sf, ct * cf])])
        return s[:3] + R @ off, R

    def dyn1(self, s, u):
        if self.sc.dim == 2:
            f = [s[3] * torch.cos(s[2]), s[3] * torch.sin(s[2]), s[3] * u[1], u[0]]
            if len(s) == 5:
                a = s[2] - s[4]
                f.append((s[3] * torch.sin(a) - s[3] * self.p[1] * u[1] * torch.cos(a)) / self.p[2])
            return torch.stack(f)
        mass, grav, Jx, Jy, Jz, arm, km = self.p[:7]
        _, R = self.pose1(s, None, torch.zeros(3, dtype=torch.float64, device=s.device))
        thrust = mass * grav + u.sum()
        p, q, r = s[9], s[10], s[11]
        cf, sf, ct, tt = torch.cos(s[6]), torch.sin(s[6]), torch.cos(s[7]), torch.tan(s[7])
        acc = R[:, 2] * thrust / mass
        return torch.stack([s[3], s[4], s[5], acc[0], acc[1], acc[2] - grav, p + (sf * q + cf * r) * tt, cf * q - sf * r,
                            (sf * q + cf * r) / ct, (arm * (u[1] - u[3]) + q * r * (Jy - Jz)) / Jx,
                            (arm * (u[2] - u[0]) + p * r * (Jz - Jx)) / Jy, (km * (u[0] - u[1] + u[2] - u[3]) + p * q * (Jx - Jy)) / Jz])

    def poses(self, s, row, part):
        return torch.func.vmap(self.pose1)(s[row], self.link[part], self.off[part])

    def faces(self, rho, p):
        """Offsets d' and world normals of the pairs p (padded faces: 0)."""
        o = self.obs[p]
        c = self.C[o]
        own = torch.arange(c.shape[1], device="cuda")[None, :] < self.nf[o][:, None]
        return torch.where(own, self.d[o] - (c * rho[:, None, :]).sum(2), 0.0), c * own[:, :, None], own


def _qp_exact(geo, p, rho, R, zeta, xi, y, prox):
    """argmin 0.5 |K^T y + bq|^2 + 0.5 prox sum |K_g|^2 (y_g - ybar_g)^2, b.lambda = 1, y >= 0, by Newton's method on its dual."""
    D, FR = geo.sc.dim, geo.sc.fr_max
    dp, c, own = geo.faces(rho, p)
    K = torch.cat([dp[:, :, None], c], 2)
    Dm = torch.where(own, (K * K).sum(2), 1.0)
    pt = geo.part[p]
    rob = torch.arange(FR, device="cuda")[None, :] < geo.nr[pt][:, None]
    A = geo.A[pt] * rob[:, :, None]
    Kr = torch.einsum("pij,pkj->pki", R, A)
    n2 = torch.where(rob, (A * A).sum(2), 1.0)
    b = torch.where(rob, geo.b[pt], 1.0)
    yl, ym, yg = y[:, :FR], y[:, FR:-1] * own, y[:, -1]
    bq = torch.cat([(1.0 + zeta)[:, None], torch.einsum("pij,pj->pi", R, xi)], 1)
    wt = torch.where(rob, b * b / n2, 0.0)

    def at(w):
        mu = (ym - (K * w[:, None, :]).sum(2) / (prox * Dm)).clamp_min(0) * own
        gam = (yg - w[:, 0] / prox).clamp_min(0)
        t = torch.where(rob, (yl - (Kr * w[:, None, 1:]).sum(2) / (prox * n2)) * n2 / b, -1e30)
        ts, order = t.sort(1, descending=True)
        ws = wt.gather(1, order)
        s1, s2 = (ws * ts).cumsum(1), ws.cumsum(1)
        tk = (s1 - 1) / s2
        k = ((ts > tk) & (ws > 0)).sum(1, keepdim=True) - 1
        tau = tk.gather(1, k.clamp_min(0))[:, 0]
        x = (t - tau[:, None]).clamp_min(0) * rob
        lam = b / n2 * x
        Kty = torch.cat([((mu * dp).sum(1) + gam)[:, None], (lam[:, :, None] * Kr).sum(1) + (mu[:, :, None] * c).sum(1)], 1)
        psi = 0.5 * (w * w).sum(1) - (bq * w).sum(1) + 0.5 * prox * ((mu * mu * Dm).sum(1) + gam * gam + (n2 * lam * lam).sum(1)) + prox * tau
        return lam, mu, gam, Kty, psi

    w = bq.clone()
    w[:, 0] += (ym * dp).sum(1) + yg
    w[:, 1:] += (yl[:, :, None] * Kr).sum(1) + (ym[:, :, None] * c).sum(1)
    cur = at(w)
    eye = torch.eye(D + 1, dtype=torch.float64, device="cuda")
    for _ in range(80):
        lam, mu, gam, Kty, psi = cur
        F = w - bq - Kty
        scale = 1.0 + w.abs().amax(1) + bq.abs().amax(1)
        if bool((F.abs().amax(1) <= 1e-13 * scale).all()):
            break
        on = ((mu > 0) & own).double()
        H = eye + torch.einsum("pf,pfi,pfj->pij", on / (prox * Dm), K, K)
        H[:, 0, 0] += (gam > 0) / prox
        act = ((lam > 0) & rob).double()
        ba = torch.einsum("pk,pki->pi", act * b / n2, Kr)
        bb = (act * wt).sum(1).clamp_min(1e-300)
        H[:, 1:, 1:] += (torch.einsum("pk,pki,pkj->pij", act / n2, Kr, Kr) - ba[:, :, None] * ba[:, None, :] / bb[:, None, None]) / prox
        step = -torch.linalg.solve(H, F)
        gd = (F * step).sum(1)
        tl = torch.ones_like(psi)
        for _ in range(40):
            new = at(w + tl[:, None] * step)
            bad = new[4] > psi + 1e-4 * tl * gd + 1e-13 * (1 + psi.abs())
            if not bool(bad.any()):
                break
            tl = torch.where(bad, 0.5 * tl, tl)
        w = w + tl[:, None] * step
        cur = at(w)
    return cur[0], cur[1], cur[2], cur[3] + bq


def _chunks(n, k):
    return [torch.arange(i, min(n, i + k), device="cuda") for i in range(0, n, k)]


def _alpha_exact(geo, states):
    """alpha* of every pair: the scale LP's dual by a batched simplex."""
    D, out = geo.sc.dim, []
    V, FR = D + 1, geo.sc.fr_max
    for p in _chunks(geo.sc.n_pairs, 400_000):
        pt = geo.part[p]
        rho, R = geo.poses(states, geo.row[p], pt)
        dp, c, own = geo.faces(rho, p)
        rob = torch.arange(FR, device="cuda")[None, :] < geo.nr[pt][:, None]
        n = len(p)
        cols = torch.cat([torch.cat([geo.b[pt][:, :, None], torch.einsum("pij,pkj->pki", R, geo.A[pt])], 2),
                          torch.cat([torch.zeros_like(c[:, :, :1]), c], 2),
                          torch.eye(V, dtype=torch.float64, device="cuda").expand(n, V, V)], 1)
        nc = cols.shape[1] - V
        dead = torch.cat([~rob, ~own, torch.ones(n, V, dtype=torch.bool, device="cuda")], 1)
        cost2 = torch.cat([torch.zeros_like(geo.b[pt]), dp, torch.zeros(n, V, dtype=torch.float64, device="cuda")], 1)
        cost1 = torch.zeros_like(cost2)
        cost1[:, nc:] = 1.0
        Bi = torch.eye(V, dtype=torch.float64, device="cuda").repeat(n, 1, 1)
        x = torch.zeros(n, V, dtype=torch.float64, device="cuda")
        x[:, 0] = 1.0
        bas = torch.arange(nc, nc + V, device="cuda").repeat(n, 1)
        for phase, cost in ((1, cost1), (2, cost2)):
            for it in range(200):
                pi = torch.einsum("pi,pij->pj", cost.gather(1, bas), Bi)
                rc = cost - (cols * pi[:, None, :]).sum(2)
                rc = torch.where(dead, math.inf, rc.scatter(1, bas, 0.0))
                # steepest cost first, the lowest index after many pivots (no cycling)
                neg = rc < -1e-11 * (1 + cost.abs() + (cols * pi[:, None, :]).abs().sum(2))
                ent = torch.where(neg, rc, 0.0).argmin(1) if it < 60 else neg.double().argmax(1)
                go = neg.any(1)
                if not bool(go.any()):
                    break
                dc = torch.einsum("pij,pj->pi", Bi, cols.gather(1, ent[:, None, None].expand(n, 1, V))[:, 0])
                ratio = torch.where(dc > 1e-11, x / dc.clamp_min(1e-300), math.inf)
                # a zero-level artificial leaves first
                art = (bas >= nc) & (dc.abs() > 1e-9) & (x <= 1e-14) if phase == 2 else torch.zeros_like(dc, dtype=torch.bool)
                ratio = torch.where(art, -1.0, ratio)
                r = ratio.argmin(1, keepdim=True)
                pr = dc.gather(1, r)
                brow = Bi.gather(1, r[:, :, None].expand(n, 1, V)) / pr[:, :, None]
                xr = x.gather(1, r) / pr
                Bn = (Bi - dc[:, :, None] * brow).scatter(1, r[:, :, None].expand(n, 1, V), brow)
                xn = (x - dc * xr).clamp_min(0).scatter(1, r, xr.clamp_min(0))
                Bi = torch.where(go[:, None, None], Bn, Bi)
                x = torch.where(go[:, None], xn, x)
                bas = torch.where(go[:, None], bas.scatter(1, r, ent[:, None]), bas)
        Bm = cols.gather(1, bas[:, :, None].expand(n, V, V)).transpose(1, 2)
        e1 = torch.zeros(n, V, dtype=torch.float64, device="cuda")
        e1[:, 0] = 1.0
        out.append(-(cost2.gather(1, bas) * torch.linalg.solve(Bm, e1)).sum(1))
    return torch.cat(out)


def _lq_exact(case, seed):
    A, Bm, c, Q, q, R, r, s0 = _lq_data(case, seed)
    N = case["N"]
    P, p = [Q[:, N]], [q[:, N]]
    K, k = [], []
    for t in range(N - 1, -1, -1):
        PA, PB, w = P[-1] @ A[:, t], P[-1] @ Bm[:, t], (P[-1] @ c[:, t, :, None])[..., 0] + p[-1]
        Bt, At = Bm[:, t].transpose(1, 2), A[:, t].transpose(1, 2)
        G = -torch.linalg.solve(R[:, t] + Bt @ PB, torch.cat([Bt @ PA, (r[:, t] + (Bt @ w[..., None])[..., 0])[..., None]], 2))
        K.append(G[:, :, :-1])
        k.append(G[:, :, -1])
        H = Bt @ PA
        Pt = Q[:, t] + At @ PA + H.transpose(1, 2) @ K[-1]
        P.append(0.5 * (Pt + Pt.transpose(1, 2)))  # rounding would grow in the antisymmetric part
        p.append(q[:, t] + (At @ w[..., None])[..., 0] + (H.transpose(1, 2) @ k[-1][..., None])[..., 0])
    s, u = [s0], []
    for t in range(N):
        u.append((K[N - 1 - t] @ s[-1][..., None])[..., 0] + k[N - 1 - t])
        s.append((A[:, t] @ s[-1][..., None])[..., 0] + (Bm[:, t] @ u[-1][..., None])[..., 0] + c[:, t])
    return {"s": torch.stack(s, 1), "u": torch.stack(u, 1), "P": torch.stack(P[::-1], 1), "p": torch.stack(p[::-1], 1), "status": None}


def _solve_exact(case, seed):
    """The ADMM of Sec. IV-B in FP64: pair QPs, one LQ step per iteration, box block, dual updates, stopping rule."""
    sc, _ = _scene(case, seed)
    geo = _Geo(sc, DTYPES[case["dtype"]])
    m, D, S = sc.model, sc.dim, sc.n_scen
    ns, nu, FR = m.ns, m.nu, sc.fr_max
    sigma, rho_b, damp, eps, prox, its = 300.0, 100.0, 100.0, 1e-4, case["prox"], case["iters"]
    t64 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    idx = lambda a: torch.as_tensor(np.asarray(a, np.int64), device="cuda")  # noqa: E731
    N, sb, cb = idx(sc.horizon), idx(sc.state_begin[:-1]), idx(sc.ctrl_begin[:-1])
    Nm = int(N.max())
    s_ref, s, u = geo.g(sc.s_ref), geo.g(sc.s_init), geo.g(sc.u_init)
    y = _cold_y(sc, geo.part, geo.dtype).double().T.contiguous()
    P = sc.n_pairs
    zeta, xi = torch.zeros(P, dtype=torch.float64, device="cuda"), torch.zeros(P, D, dtype=torch.float64, device="cuda")
    Qs, Qu = t64(m.Qs), t64(m.Qu)
    bound = [t64(np.clip(v, -1e30, 1e30)) for v in (m.s_lo, m.s_hi, m.u_lo, m.u_hi)]
    sbox, ubox = (bound[0] > -1e29) | (bound[1] < 1e29), (bound[2] > -1e29) | (bound[3] < 1e29)
    # lanes: (part, step) of every scenario; pair -> lane, lane -> state row, part
    NP, Nh = np.diff(sc.part_begin), sc.horizon
    lane_part = idx(np.repeat(np.arange(len(sc.part_nf)), np.repeat(Nh, NP)))
    pscen = np.repeat(np.arange(S), NP)
    lane_row = idx(np.concatenate([sc.state_begin[a] + 1 + np.arange(Nh[a]) for a in pscen]))
    qb = np.concatenate([[0], np.cumsum(NP * Nh)])
    scen_of = lambda b, n: torch.repeat_interleave(torch.arange(S, device="cuda"), idx(n))  # noqa: E731
    pair_scen, row_scen, ctrl_scen = scen_of(None, sc.pair_counts), scen_of(None, Nh + 1), scen_of(None, Nh)
    lane = idx(qb[:-1])[pair_scen] + (torch.arange(P, device="cuda") - idx(sc.pair_begin[:-1])[pair_scen]) % idx(NP * Nh)[pair_scen]
    row_t = torch.arange(len(s), device="cuda") - sb[row_scen]
    zs, zu = s.clamp(bound[0], bound[1]), u.clamp(bound[2], bound[3])
    ws, wu = torch.zeros_like(zs), torch.zeros_like(zu)
    box_p = torch.zeros(S, dtype=torch.float64, device="cuda")
    box_d, rdual = box_p.clone(), box_p.clone()
    live = torch.ones(S, dtype=torch.bool, device="cuda")
    rep = {k: torch.zeros(S, dtype=torch.float64, device="cuda") for k in ("r_pri", "r_dual", "cost")}
    ssum = lambda v, who: torch.zeros(S, dtype=torch.float64, device="cuda").index_add_(0, who, v)  # noqa: E731
    jp = torch.func.vmap(torch.func.jacfwd(geo.pose1))
    jd = torch.func.vmap(torch.func.jacfwd(geo.dyn1, argnums=(0, 1)))
    for j in range(its + 1):
        if j:
            rpri = torch.zeros(S, dtype=torch.float64, device="cuda")
            for p in _chunks(P, 1_000_000):
                rho, R = geo.poses(s, geo.row[p], geo.part[p])
                dp, c, _ = geo.faces(rho, p)
                yp = y[p]
                Tr = 1.0 + (yp[:, FR:-1] * dp).sum(1) + yp[:, -1]
                Rr = (yp[:, :FR, None] * geo.A[geo.part[p]]).sum(1) + torch.einsum("pij,pi->pj", R, (yp[:, FR:-1, None] * c).sum(1))
                on = live[pair_scen[p]].double()
                zeta[p] += on * Tr
                xi[p] += on[:, None] * Rr
                rpri.index_add_(0, pair_scen[p], Tr * Tr + (Rr * Rr).sum(1))
            rp, rd = rpri + box_p, rdual + box_d
            stop = live & (((rp <= eps) & (rd <= eps)) | (j >= its))
            e = s - s_ref
            F = ssum((Qs * e * e).sum(1), row_scen) + ssum((Qu * u * u).sum(1), ctrl_scen)
            for k, v in (("r_pri", rp), ("r_dual", rd), ("cost", F)):
                rep[k] = torch.where(stop, v, rep[k])
            live = live & ~stop
            if not bool(live.any()):
                break
        nl = len(lane_row)
        W, Wc, E = (torch.zeros(nl, *sh, dtype=torch.float64, device="cuda") for sh in ((D, D), (D,), (D, D)))
        rdual = torch.zeros(S, dtype=torch.float64, device="cuda")
        for p in _chunks(P, 500_000):
            rho, R = geo.poses(s, geo.row[p], geo.part[p])
            lam, mu, gam, _ = _qp_exact(geo, p, rho, R, zeta[p], xi[p], y[p], prox)
            o, pt = geo.obs[p], geo.part[p]
            new = torch.cat([lam, mu, gam[:, None]], 1)
            rdual.index_add_(0, pair_scen[p], ((new - y[p])[:, :-1] ** 2).sum(1))
            w = (mu[:, :, None] * geo.C[o]).sum(1)
            cc = 1.0 + (mu * geo.d[o]).sum(1) + gam + zeta[p]
            ee = (lam[:, :, None] * geo.A[pt]).sum(1) + xi[p]
            W.index_add_(0, lane[p], w[:, :, None] * w[:, None, :])
            Wc.index_add_(0, lane[p], cc[:, None] * w)
            E.index_add_(0, lane[p], w[:, :, None] * ee[:, None, :])
            y[p] = torch.where(live[pair_scen[p]][:, None], new, y[p])
        # Gauss-Newton terms of every lane, summed over the parts of a step
        sl = s[lane_row]
        rho, R = geo.poses(s, lane_row, lane_part)
        dr, dR = jp(sl, geo.link[lane_part], geo.off[lane_part])
        Hs = torch.einsum("lia,lij,ljb->lab", dr, W, dr) + torch.einsum("lika,ljkb,lij->lab", dR, dR, W)
        gg = (-torch.einsum("lia,li->la", dr, Wc - torch.einsum("lij,lj->li", W, rho)) + torch.einsum("lija,lij->la", dR, E)
              + torch.einsum("lika,ljk,lij->la", dR, R, W))
        later = (row_t > 0).double()[:, None]
        Q = torch.diag_embed(2 * Qs + later * (damp + rho_b * sbox.double()))
        q = -2 * Qs * s_ref - later * (damp * s + torch.where(sbox, rho_b * (zs - ws), 0.0))
        Q.index_add_(0, lane_row, sigma * Hs)
        q.index_add_(0, lane_row, sigma * (gg - torch.einsum("lab,lb->la", Hs, sl)))
        srow = torch.arange(len(u), device="cuda") + ctrl_scen
        sc0 = s[srow]
        fs, fu = jd(sc0, u)
        A = torch.eye(ns, dtype=torch.float64, device="cuda") + geo.dt * fs
        Bm = geo.dt * fu
        cv = sc0 + geo.dt * torch.func.vmap(geo.dyn1)(sc0, u) - torch.einsum("tij,tj->ti", A, sc0) - torch.einsum("tij,tj->ti", Bm, u)
        Ru = torch.diag(2 * Qu + damp + rho_b * ubox.double())
        r = -damp * u - torch.where(ubox, rho_b * (zu - wu), 0.0)
        Pv, pv = Q[sb + N].clone(), q[sb + N].clone()
        Ks = torch.zeros(Nm, S, nu, ns + 1, dtype=torch.float64, device="cuda")
        for t in range(Nm - 1, -1, -1):
            on = t < N
            tc, tr = cb + torch.minimum(torch.full_like(N, t), N - 1), sb + torch.minimum(torch.full_like(N, t), N)
            PA, PB, w = Pv @ A[tc], Pv @ Bm[tc], (Pv @ cv[tc][..., None])[..., 0] + pv
            Bt, At = Bm[tc].transpose(1, 2), A[tc].transpose(1, 2)
            Hm = torch.cat([Bt @ PA, (r[tc] + (Bt @ w[..., None])[..., 0])[..., None]], 2)
            G = -torch.linalg.solve(Ru + Bt @ PB, Hm)
            Ks[t] = G
            Pn = Q[tr] + At @ PA + Hm[:, :, :-1].transpose(1, 2) @ G[:, :, :-1]
            pn = q[tr] + (At @ w[..., None])[..., 0] + (Hm[:, :, :-1].transpose(1, 2) @ G[:, :, -1:])[..., 0]
            Pn = 0.5 * (Pn + Pn.transpose(1, 2))  # rounding would grow in the antisymmetric part
            Pv, pv = torch.where(on[:, None, None], Pn, Pv), torch.where(on[:, None], pn, pv)
        x = s[sb]
        sn, un = s.clone(), u.clone()
        for t in range(Nm):
            on = (t < N) & live
            tc = cb + torch.minimum(torch.full_like(N, t), N - 1)
            ut = (Ks[t][:, :, :-1] @ x[..., None])[..., 0] + Ks[t][:, :, -1]
            x = (A[tc] @ x[..., None])[..., 0] + (Bm[tc] @ ut[..., None])[..., 0] + cv[tc]
            un[tc[on]] = ut[on]
            sn[(sb + t + 1)[on]] = x[on]
        s, u = sn, un
        box_p, box_d = torch.zeros_like(box_p), torch.zeros_like(box_d)
        for v, z, w, k, who, use in ((s, zs, ws, 0, row_scen, sbox[None] & (row_t > 0)[:, None]), (u, zu, wu, 2, ctrl_scen, ubox[None].expand_as(u))):
            zn = (v + w).clamp(bound[k], bound[k + 1])
            on = (use & live[who][:, None]).double()
            box_d += ssum((on * (zn - z) ** 2).sum(1), who)
            box_p += ssum((on * (v - zn) ** 2).sum(1), who)
            w += on * (v - zn)
            z += on * (zn - z)
    return {"s": s, "u": u, "y": y.T.contiguous(), "zeta": zeta, "xi": xi.T.contiguous(), "iters": None, "status": None, **rep}


def exact(case, seed):
    op = case["op"]
    if op == "lq":
        return _lq_exact(case, seed)
    if op == "loop":
        return None  # control steps of whole solves, each from the last one's plan: over 20 seconds in this form
    if op == "solve":
        return _solve_exact(case, seed)
    if op == "grad":
        out = _solve_exact(case, seed)
        out.update(obs_offset=None, obs_center=None, state0=None)  # the reverse sweep of all iterations: over 20 seconds
        return out
    dtype = DTYPES[case["dtype"]]
    st = prepare(case, seed)
    sc = st["ds"].scene
    geo = _Geo(sc, dtype)
    states = st["states"].double()
    if op == "detect":
        # the certificates belong to whichever optimal basis is found, and the margin to them
        return {"alpha": _alpha_exact(geo, states), "lam": None, "mu": None, "margin": None, "verdict": None, "status": None}
    if op == "margin":
        out = []
        radius = _part_radius(geo)
        for p in _chunks(sc.n_pairs, 500_000):
            pt = geo.part[p]
            rho, R = geo.poses(states, geo.row[p], pt)
            dp, c, own = geo.faces(rho, p)
            lam, mu = st["lam"][:, p].double().T, st["mu"][:, p].double().T * own
            r = (lam[:, :, None] * geo.A[pt]).sum(1) + torch.einsum("pij,pi->pj", R, (mu[:, :, None] * c).sum(1))
            out.append(-(dp * mu).sum(1) / ((geo.b[pt] * lam).sum(1) + r.norm(dim=1) * radius[pt]))
        return torch.cat(out)
    if case["prox"] == 0.0:
        return None  # y is not unique; v is, but as the limit of hundreds of proximal steps in this form: over 20 seconds
    ys, vs = [], []
    for p in _chunks(sc.n_pairs, 300_000):
        rho, R = geo.poses(states, geo.row[p], geo.part[p])
        lam, mu, gam, v = _qp_exact(geo, p, rho, R, st["zeta"][p].double(), st["xi"][:, p].double().T, st["y"][:, p].double().T, case["prox"])
        ys.append(torch.cat([lam, mu, gam[:, None]], 1))
        vs.append(torch.cat([v[:, :1], torch.einsum("pij,pi->pj", R, v[:, 1:])], 1))
    v = torch.cat(vs)
    return {"y": torch.cat(ys).T.contiguous(), "v": v.T.contiguous(), "obj": 0.5 * (v * v).sum(1), "status": None}


def _part_radius(geo):
    """Largest vertex norm of every part (the parts are boxes about their centres)."""
    return torch.stack([b[geo.A[i].abs().sum(1) > 0][::2].norm() for i, b in enumerate(geo.b)])
