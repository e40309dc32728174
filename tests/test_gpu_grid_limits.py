"""Both sides of the grid sizes at which silu_and_mul changes between 16- and 32-byte vectors and merge_attn_states_lse between
blocks of 128 and 256 threads, with whole and partial last blocks and at offsets that forbid the wider access."""
import pytest

from paper_2509_07506_b200 import workloads as wl
from test_gpu_parity import run_merge, run_silu

pytestmark = pytest.mark.gpu
BF16, FP16, FP32 = wl.BF16, wl.FP16, wl.FP32


def blocks(T, D, dtype):
    """256-thread blocks of one 32-byte vector per thread"""
    return -(-T * (D * (2 if dtype == FP32 else 1) // 16) // 256)


@pytest.mark.parametrize("dtype", [BF16, FP16, FP32])
@pytest.mark.parametrize("T,D,want", [(959, 4096, 959), (960, 4096, 960), (961, 4096, 961), (956, 4112, 960), (957, 4112, 961),
                                      (800, 5120, 1000), (300, 14336, 1050)])
@pytest.mark.parametrize("offset", [0, 16, 8])
def test_silu_from_960_blocks(T, D, want, dtype, offset):
    if dtype == FP32:
        D, offset = D // 2, offset // 2
    assert blocks(T, D, dtype) == want
    run_silu(wl.silu_inputs(T, D, dtype, std=2.0, seed=T + D), offset=offset)


@pytest.mark.parametrize("T,want", [(8192, 8192), (8193, 8193)])
def test_silu_to_8192_blocks(T, want):
    assert blocks(T, 4096, BF16) == want
    run_silu(wl.silu_inputs(T, 4096, BF16, std=2.0, seed=T))


@pytest.mark.parametrize("dtype", [BF16, FP16, FP32])
@pytest.mark.parametrize("T,Hh,D", [(1024, 32, 128), (32767, 1, 128), (32769, 1, 128), (52428, 1, 80), (52429, 1, 80)])
@pytest.mark.parametrize("offset", [0, 8])
def test_merge_to_262144_vectors(T, Hh, D, dtype, offset):
    if dtype == FP32:
        D //= 2
    run_merge(wl.merge_inputs(T, Hh, D, dtype, seed=T + D, neg_inf_frac=0.05), offset=offset)
