"""Launch configuration of the tile kernels, read from captured launches (a stream capture
records the kernel nodes; nothing of it is run)."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

from paper_2406_07048_gb300 import synth
from tests.test_gpu_edges import _faces_scene, _mixed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2406_07048_gb300 import _build, binding
    _build.build()
    return binding


class _KernelNode(C.Structure):
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("shared", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _launches(call):
    """The kernel launches of call(stream=...): (block, dynamic shared bytes, a function that
    reads the kernel's limit of dynamic shared memory)."""
    cu = C.CDLL("libcuda.so.1")
    ok = lambda r: r == 0 or pytest.fail(f"driver call: {r}")
    call(stream=None)  # allocations, and what is looked up once
    torch.cuda.synchronize()
    st, graph, n = torch.cuda.Stream(), C.c_void_p(), C.c_size_t(0)
    ok(cu.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2))
    try:
        out = call(stream=st)
    finally:
        r = cu.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph))
    ok(r)
    ok(cu.cuGraphGetNodes(graph, None, C.byref(n)))
    nodes = (C.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, C.byref(n)))
    found = []
    for node in nodes:
        kind = C.c_int()
        ok(cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
        if kind.value != 0:
            continue
        p = _KernelNode()
        ok(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)))
        func = C.c_void_p(p.func)
        if not func:
            ok(cu.cuKernelGetFunction(C.byref(func), C.c_void_p(p.kern)))

        def limit(func=func):
            v = C.c_int()
            ok(cu.cuFuncGetAttribute(C.byref(v), 8, func))
            return v.value

        found.append((tuple(p.block), p.shared, limit))
    ok(cu.cuGraphDestroy(graph))
    del out
    return found


def _states(ds):
    return ds.tensor(ds.scene.s_init)


@pytest.mark.parametrize("entry", ["scale", "noalloc", "pair"])
def test_a_smaller_call_leaves_the_shared_memory_limit(B, entry):
    """The limit of dynamic shared memory belongs to the kernel, not to the call: a call with
    less of it must not lower the limit below that of a call that another thread is about to
    launch (both calls need more than the 48 KB that need no limit)."""
    ctx = B.Context(0)
    scene = lambda sc, dtype: B.DeviceScene(ctx, sc, dtype)
    if entry == "scale":
        big, small = scene(_mixed(torch.float32), torch.float32), scene(_faces_scene(2, 8, 16, 5), torch.float32)
        run = lambda ds: lambda stream: B.scale_detect(ds, _states(ds), stream=stream)
    elif entry == "noalloc":
        big, small = (scene(_faces_scene(2, f, 33, 5), torch.float64) for f in (24, 12))
        run = lambda ds: lambda stream: B.scale_detect_noalloc(ds, _states(ds), stream=stream)
    else:
        big, small = (scene(_faces_scene(2, f, 16, 5), torch.float32) for f in (24, 9))
        big.warps = small.warps = 8

        def run(ds):
            pb = B.Problem(ds)
            return lambda stream: B.pair_qp(ds, pb.s, pb.zeta, pb.xi, pb.y, prox=1.0, stream=stream)
    _, need, limit = max(_launches(run(big)), key=lambda f: f[1])
    after = max(shared for _, shared, _ in _launches(run(small)))
    assert 48 * 1024 < after < need
    assert limit() >= need


def test_warps_of_the_pair_and_of_the_lp_kernels(B):
    """The pair kernels' count of warps, set or tuned, leaves the LP and margin kernels'
    count, also on a scene derived with other offsets; theirs changes no result."""
    ds = B.DeviceScene(B.Context(0), synth.config3(n_scen=64), torch.float32)
    pb = B.Problem(ds)

    def lp_warps(ds):
        out = B.scale_detect(ds, pb.s)
        shapes = _launches(lambda stream: B.scale_detect(ds, pb.s, stream=stream))
        shapes += _launches(lambda stream: B.cert_margin(ds, pb.s, out["lam"], out["mu"], stream=stream))
        return sorted(block[1] for block, _, _ in shapes if block[0] == 32)

    own = lp_warps(ds)
    assert len(own) == 2 and own[0] == own[1] > 2
    ds.warps = 2
    assert lp_warps(ds) == own
    assert lp_warps(ds.with_offsets(ds.obs_d)) == own
    ds.autotune_warps(pb, candidates=(1, 3), iters=1)
    assert lp_warps(ds) == own
    ref = B.scale_detect(ds, pb.s)
    for w in (1, 5):
        ds.lp_warps = w
        assert lp_warps(ds) == [w, w] == lp_warps(ds.with_offsets(ds.obs_d))
        got = B.scale_detect(ds, pb.s)
        assert all(torch.equal(got[k], ref[k]) for k in ref)
        assert torch.equal(B.cert_margin(ds, pb.s, got["lam"], got["mu"]), B.cert_margin(ds, pb.s, ref["lam"], ref["mu"]))
    with pytest.raises(B.OcaError) as e:
        ds.lp_warps = 17
    assert e.value.code == 1


def test_cold_start_is_there_when_the_call_returns(B):
    """The solve that takes the cold start may run on another stream than the one that
    forms it: nothing of it is pending when cold_y returns."""
    ds = B.DeviceScene(B.Context(0), synth.config3(n_scen=2048), torch.float32)
    torch.cuda.synchronize()
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(stream):
            ds.cold_y()
            assert stream.query()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_lp_warps_follow_what_an_sm_holds(B, dtype):
    """More than four warps a tile only while the launch stays within two and a half times
    the warps whose staged columns (32 lanes x 4 numbers a face) an SM's 227 KB hold."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    counts = []
    for n in (1, 64, 256, 512, 1024):
        ds = B.DeviceScene(B.Context(0), synth.config3(n_scen=n), dtype)
        held = 227 * 1024 // (32 * 4 * (ds.scene.fr_max + ds.scene.fo_max) * ds.dtype.itemsize)
        counts.append(ds.lp_warps)
        assert ds.lp_warps <= 4 or ds.n_tiles * ds.lp_warps <= 2.5 * n_sm * held
    # one scene of 12 obstacles, 181 tiles, ..., 2,892 tiles
    assert counts[:2] == [12, 16] and counts[-1] == 4
