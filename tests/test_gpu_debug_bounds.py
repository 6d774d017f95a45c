"""The bounds-checking build (-DLT_DEBUG_BOUNDS) stands in for a memory checker: every global store / gather
with a known bound is checked, a failing access is skipped and LT_STATUS_BOUNDS is recorded.  Ordinary cases
must leave the bit clear and return the release build's bits; a page table that points outside the pool must be
caught before the access happens."""
import numpy as np
import pytest
import torch

from paper_2607_11976_b200 import binding as lt
from paper_2607_11976_b200 import build as lt_build
from workloads import make_config, make_knn

from gpu_util import run_topk
from test_gpu_paged import make_pool, run_paged

pytestmark = pytest.mark.gpu


@pytest.fixture()
def debug_library():
    path = lt_build.build(debug_bounds=True)
    lt.use_library(path)
    yield path
    lt.use_library(None)


CASES = [("fp8_ar1", 72, 30000, 512), ("dsa_bf16", 40, 12000, 256), ("tiny_f32", 16, 1500, 64), ("adv_ties_exact", 24, 6000, 300)]


@pytest.mark.parametrize("name,T,N,topk", CASES)
def test_ordinary_cases_leave_the_bounds_bit_clear(name, T, N, topk, debug_library):
    inp = make_config(name, T=T, N=N, topk=topk)
    lt.use_library(None)
    want = run_topk(inp)
    lt.use_library(debug_library)
    fused = [] if inp.dtype == "f32" else [lt.Tunables(path=lt.LT_PATH_FUSED)]  # the sampled form, which small problems leave out
    for tun in [None, lt.Tunables(cap_mult=1, sample_rank=1)] + fused:  # the second one forces rows through the exact fallback
        got = run_topk(inp, tun)
        if tun in fused:
            assert got[2][3] > 0
        assert got[2][0] & lt.LT_STATUS_BOUNDS == 0, "a bounds check failed on a valid problem"
        assert got[2][0] & lt.LT_STATUS_TIMEOUT == 0
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1].view(np.uint32), want[1].view(np.uint32))


def test_paged_cache_is_clean_and_a_bad_page_table_is_caught(debug_library):
    inp = make_config("fp8_ar1", T=40, N=9000, topk=256)
    pool, scale, table = make_pool(inp, seed=5)
    lt.use_library(None)
    want = run_paged(inp, pool, scale, table)
    lt.use_library(debug_library)
    got = run_paged(inp, pool, scale, table)
    assert got[2][0] & lt.LT_STATUS_BOUNDS == 0
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1].view(np.uint32), want[1].view(np.uint32))
    # host-made fault: one visible logical page points far outside the pool.  The checks replace the page by
    # page 0 before any address is formed from it, flag the call, and the call completes.
    bad = table.copy()
    bad[3] = pool.shape[0] // 64 + 1000
    got = run_paged(inp, pool, scale, bad)
    assert got[2][0] & lt.LT_STATUS_BOUNDS, "the page-table entry outside the pool was not caught"
    assert got[2][0] & lt.LT_STATUS_TIMEOUT == 0


@pytest.mark.parametrize("tun", [None, lt.Tunables(path=lt.LT_PATH_FUSED)], ids=["dense", "sampled"])
def test_knn_is_clean(tun, debug_library):
    from test_gpu_knn import gpu_topk  # the driver of the k-NN parity tests
    inp = make_knn(T=64, N=20000, D=256, topk=128)
    lt.use_library(None)
    want = gpu_topk(inp)
    lt.use_library(debug_library)
    got = gpu_topk(inp, tun)
    assert got[2][0] & lt.LT_STATUS_BOUNDS == 0 and (got[2][3] > 0) == (tun is not None)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1].view(np.uint32), want[1].view(np.uint32))


@pytest.mark.parametrize("T,N,tun", [(3, 5000, {}), (2, 40000, {}), (70, 9000, dict(path=lt.LT_PATH_FUSED)), (40, 9000, dict(path=lt.LT_PATH_FUSED, grid=296)),
                                     (40, 9000, dict(path=lt.LT_PATH_FUSED, cap_mult=1, sample_rank=1))])
def test_status_block_opens_as_in_the_release_build(T, N, tun, debug_library):
    """A workspace full of ones: the status bytes and counters are cleared by the call's own kernels in this build too, and checked."""
    inp = make_config("fp8_ar1", T=T, N=N, topk=64)
    lt.use_library(None)
    want = run_topk(inp)
    lt.use_library(debug_library)
    tun = lt.Tunables(**tun)
    q, w, k, ks = lt.to_device(inp)
    ws = lt.alloc_workspace(inp.dtype, T, N, inp.H, inp.D, 64, tun).fill_(0xff)
    idx, score = torch.empty((T, 64), dtype=torch.int32, device="cuda"), torch.empty((T, 64), device="cuda")
    lt.lt_indexer_topk_ex(inp.dtype, q, w, k, ks, 64, inp.causal_offset, idx, score, ws, tun)
    status = lt.lt_read_status(ws)
    assert status[0] & ~lt.LT_STATUS_FALLBACK == 0 and 0 <= status[4] <= T and status[6] == 0 and status[7] == 0, status
    assert np.array_equal(idx.cpu().numpy(), want[0]) and np.array_equal(score.cpu().numpy().view(np.uint32), want[1].view(np.uint32))


def test_status_block_opens_as_in_the_release_build_knn(debug_library):
    inp = make_knn(T=70, N=30000, D=64, topk=10)
    q, x = (torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda() for a in (inp.q, inp.x))
    ws = torch.full((lt.lt_knn_topk_workspace_bytes(70, 30000, 64, 10),), 0xff, dtype=torch.uint8, device="cuda")
    idx = torch.empty((70, 10), dtype=torch.int32, device="cuda")
    lt.lt_knn_topk(q, x, 10, idx, None, ws)
    status = lt.lt_read_status(ws)
    assert status[0] & ~lt.LT_STATUS_FALLBACK == 0 and status[6] == 0 and status[7] == 0, status
