"""A bounded wait inside the library that runs out leaves its stage's outputs
unfinished, while the call's later stages are already enqueued: those that
would follow indices from those outputs without a test must not start.

The stages are called one by one (tests/native/stages.cu, linked with the
library's objects) on inputs that are valid all the same: with the status word
of a wait that ran out nothing may be written, with a clean one, or one that
holds another error, the results are the usual ones."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import paper_2409_03771_gb300 as msc
    from paper_2409_03771_gb300 import _build

    _build.build(force=not glob.glob(os.path.join(_build.BUILD, "*.o")))
    msc.load()
    out = str(tmp_path_factory.mktemp("native") / "libstages.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.INCLUDE, "-I", _build.CSRC, "-shared",
                    "-o", out, os.path.join(HERE, "native", "stages.cu"),
                    *(os.path.join(_build.BUILD, os.path.splitext(s)[0] + ".o") for s in _build.SOURCES)], check=True)
    so = ctypes.CDLL(out)
    for name in ("order", "compress", "ms_id"):
        getattr(so, f"stage_{name}_bytes").restype = ctypes.c_size_t
        getattr(so, f"stage_{name}_bytes").argtypes = [ctypes.c_int64]
    P, I, Z = ctypes.c_void_p, ctypes.c_int32, ctypes.c_size_t
    so.stage_order.argtypes = [P, ctypes.c_int64, P, P, Z, P, P]
    so.stage_compress.argtypes = [P, I, P, Z, P, P]
    so.stage_ms_id.argtypes = [P, P, I, P, P, P, Z, P, P]
    so.stage_lonely_barrier.argtypes = [P, P, P, P]
    return so


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def word(v):
    return torch.full((1,), v, dtype=torch.int32, device="cuda")


def ws_for(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")


def stream():
    return torch.cuda.current_stream().cuda_stream


def call(fn, *args):
    assert fn(*(a.data_ptr() if isinstance(a, torch.Tensor) else a for a in args), stream()) == 0
    torch.cuda.synchronize()


@pytest.mark.parametrize("n", [5000, 70001, (1 << 20) + 3, (1 << 24) + 5])  # the tail alone, four and eight sweeps before it
@pytest.mark.parametrize("code", [0, -4, -7])
def test_trusted_jumping(lib, n, code):
    ptr = np.maximum(np.arange(n, dtype=np.int32) - 1, 0)
    p, st = cuda(ptr), word(code)
    ws = ws_for(lib.stage_compress_bytes(n))
    call(lib.stage_compress, p, n, ws, ws.numel(), st)
    assert int(st) == code
    if code == -7:
        np.testing.assert_array_equal(p.cpu().numpy(), ptr)
    else:
        assert int(p.max()) == 0


@pytest.mark.parametrize("n", [3000000, (1 << 24) + 5])  # a direct last pass, an inverse permutation
@pytest.mark.parametrize("code", [0, -7])
def test_order_passes(lib, n, code):
    f = torch.rand(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(n))
    order, st = torch.full((n,), -5, dtype=torch.int32, device="cuda"), word(code)
    ws = ws_for(lib.stage_order_bytes(n))
    call(lib.stage_order, f, n, order, ws, ws.numel(), st)
    assert int(st) == code
    if code:
        assert bool((order == -5).all())
    else:
        assert bool((torch.empty_like(order).scatter_(0, torch.argsort(f, stable=True),
                                                      torch.arange(n, dtype=torch.int32, device="cuda")) == order).all())


@pytest.mark.parametrize("n", [4000, 3 << 20])
@pytest.mark.parametrize("code", [0, -7])
def test_cell_ids(lib, n, code):
    lab = (torch.arange(n, device="cuda") // 5 * 5).int()
    ms, cells, st = torch.full((n,), -5, dtype=torch.int32, device="cuda"), word(0), word(code)
    ws = ws_for(lib.stage_ms_id_bytes(n))
    call(lib.stage_ms_id, lab, lab, n, ms, cells, ws, ws.numel(), st)
    assert int(st) == code
    if code:
        assert bool((ms == -5).all())
    else:
        assert bool((ms == lab // 5).all()) and int(cells) == (n + 4) // 5


@pytest.mark.parametrize("code", [0, -4, -1])
def test_barrier_that_runs_out_is_reported_over_other_errors(lib, code):
    count, passed, st = torch.zeros(1, dtype=torch.int32, device="cuda"), word(9), word(code)
    call(lib.stage_lonely_barrier, count, passed, st)
    assert int(passed) == 0 and int(st) == -7
