"""A run of norms whose blocks stop waiting for one another's sums: the library is rebuilt with waits that end before
the first poll.  The normalised rows are then NaN throughout and the residual is that of the calls in order; nothing
hangs, and the device goes on working."""
import ctypes

import pytest
import torch

import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import binding, build as astra_build

pytestmark = pytest.mark.gpu
CODE = {torch.bfloat16: 0, torch.float16: 1, torch.float32: 2}


@pytest.fixture(scope="module")
def hasty_lib(tmp_path_factory):
    path = str(tmp_path_factory.mktemp("waits") / "libastra_hasty.so")
    astra_build.build_variant(path, {"ASTRA_RUN_WAIT_POLLS": 0})
    lib = ctypes.CDLL(path)
    vp, i64, i32, f32 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_float
    lib.astra_issue_run.argtypes = [i32, ctypes.c_int32, vp, ctypes.POINTER(i64), f32, i32, vp]
    return lib


@pytest.mark.parametrize("dtype", list(CODE))
@pytest.mark.parametrize("T,H,n", [(1, 8, 2), (16, 2048, 8), (16, 2048, 20), (37, 4096, 33), (74, 1032, 64)])
def test_a_wait_that_runs_out_gives_nan_rows(hasty_lib, dtype, T, H, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(T + n)
    mk = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(dtype)  # noqa: E731
    xs, r, ws = mk(n, T, H), mk(T, H), mk(n, H)
    want = r.clone()
    for x in xs.clone():
        astra.astra_fused_add_rmsnorm(x, want, ws[0], 1e-5)
    calls = (ctypes.c_void_p * (6 * n))(*(p for x, w in zip(xs, ws) for p in (x.data_ptr(), r.data_ptr(), w.data_ptr(), 0, 0, 0)))
    ext = (ctypes.c_int64 * 4)(T, H, 0, 0)
    torch.cuda.synchronize()
    assert hasty_lib.astra_issue_run(binding._fast.KIND_RMSNORM, n, calls, ext, 1e-5, CODE[dtype], None) == 0
    torch.cuda.synchronize()
    assert xs.isnan().all()
    assert torch.equal(r.view(torch.uint8), want.view(torch.uint8))
