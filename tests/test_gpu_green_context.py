"""Calls on a stream of a green context (a part of the SMs): the cooperative
launches have to be sized for it, plain and while a graph is captured."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


class DevResource(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sm_count", ctypes.c_uint),
                ("rest", ctypes.c_ubyte * 44)]


@pytest.fixture(scope="module")
def m():
    import paper_2409_03771_gb300 as msc
    from paper_2409_03771_gb300 import _build

    _build.build()
    msc.load()
    return msc


@pytest.fixture(scope="module")
def green():
    """(torch stream, SMs) of a green context of a few SMs."""
    torch.zeros(1, device="cuda")  # the primary context
    cu = ctypes.CDLL("libcuda.so.1")
    P = ctypes.c_void_p
    if not hasattr(cu, "cuGreenCtxCreate"):
        pytest.skip("the driver has no green contexts")

    def ok(code):
        assert code == 0, code

    whole, part, rest = DevResource(), DevResource(), DevResource()
    ok(cu.cuDeviceGetDevResource(0, ctypes.byref(whole), 1))
    groups = ctypes.c_uint(1)
    ok(cu.cuDevSmResourceSplitByCount(ctypes.byref(part), ctypes.byref(groups), ctypes.byref(whole), ctypes.byref(rest), 0, 16))
    assert 0 < part.sm_count < whole.sm_count
    desc, ctx, st = P(), P(), P()
    ok(cu.cuDevResourceGenerateDesc(ctypes.byref(desc), ctypes.byref(part), 1))
    ok(cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, 0, 1))  # CU_GREEN_CTX_DEFAULT_STREAM
    ok(cu.cuGreenCtxStreamCreate(ctypes.byref(st), ctx, 1, 0))  # CU_STREAM_NON_BLOCKING
    yield torch.cuda.ExternalStream(st.value), int(part.sm_count)
    torch.cuda.synchronize()
    ok(cu.cuStreamDestroy_v2(st))
    ok(cu.cuGreenCtxDestroy(ctx))


@pytest.mark.parametrize("dims", [(9, 7, 5), (64, 64, 64), (100, 110, 120), (150, 140, 130)])
def test_segment_on_a_part_of_the_sms(m, green, dims):
    f = torch.rand(dims[0] * dims[1] * dims[2], device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    want = m.segment(f, dims)
    torch.cuda.synchronize()
    with torch.cuda.stream(green[0]):
        got = m.segment(f, dims)
    assert got[4] == want[4]
    for g, w in zip(got[:4], want[:4]):
        assert torch.equal(g, w)


def test_captured_compress_on_a_part_of_the_sms(m, green):
    n = 3000000
    p = (torch.arange(n, dtype=torch.int32, device="cuda") - 1).clamp_(min=0)
    ws = torch.empty(m.msc_workspace_bytes(m.OP_COMPRESS, n), dtype=torch.uint8, device="cuda")
    st = torch.full((1,), 9, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=green[0], capture_error_mode="thread_local"):
        assert m.msc_compress(p, n, ws, ws.numel(), st) == m.OK
    graph.replay()
    torch.cuda.synchronize()
    assert int(st) == m.OK and int(p.max()) == 0


def test_batch_plan_launched_on_a_part_of_the_sms(m, green):
    b = m.Batch([(40, 41, 42), (64, 64, 64)])
    b.f.copy_(torch.rand(b.total, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2)))
    b.run()
    want = [t.clone() for t in (b.order, b.asc, b.desc, b.ms, b.num_cells)]
    b.plan()
    for t in (b.order, b.asc, b.desc, b.ms, b.num_cells):
        t.fill_(-1)
    torch.cuda.synchronize()
    with torch.cuda.stream(green[0]):
        b.launch()
    for t, w in zip((b.order, b.asc, b.desc, b.ms, b.num_cells), want):
        assert torch.equal(t, w)
