"""Edges of the forms that sizes, alignments and counts choose: whole masks of the union, digits of the position ranking, sample
statistics beyond what a CTA holds and beyond the bins it looks at first, the status block that a call's own kernels open, work items of
a triangular mask.  Integer results and bits only: nothing here has a tolerance."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import frequent_positions, pack_mask_words, union_and_masks
from paper_2607_11976_b200 import binding as lt
from workloads import make_config, make_knn

from gpu_util import run_topk, run_unfused

pytestmark = pytest.mark.gpu


# rows whose masks come one at a time and whole (4 positions to a thread, 16-byte pieces), and those that just miss it
@pytest.mark.parametrize("T,topk,N,group,shift", [(64, 2048, 131072, 64, 0), (63, 2048, 131072, 63, 0), (70, 2048, 65536, 64, 0), (64, 2048, 131072, 64, 1),
                                                  (64, 1030, 90000, 64, 0), (128, 1024, 600000, 128, 0), (9, 12, 70, 2, 0), (6, 16, 100, 3, 0),
                                                  (64, 2052, 131072, 32, 0)])
def test_union_masks_by_whole_rows(T, topk, N, group, shift):
    rng = np.random.default_rng(T * 31 + topk)
    shared = rng.integers(0, N, size=topk)
    idx = np.where(rng.random((T, topk)) < 0.5, shared[None, :], rng.integers(0, N, size=(T, topk))).astype(np.int32)
    idx[rng.random(idx.shape) < 0.02] = -1
    flat = torch.empty(T * topk + shift, dtype=torch.int32, device="cuda")
    dev = flat[shift:].view(T, topk)  # shift: rows that do not start on 16-byte boundaries
    dev.copy_(torch.from_numpy(idx))
    n_groups, cap = -(-T // group), group * topk
    words = (cap + 31) // 32
    pos = torch.full((n_groups, cap), 12345, dtype=torch.int32, device="cuda")
    length = torch.full((n_groups,), -3, dtype=torch.int32, device="cuda")
    mask = torch.full((T, words), -1, dtype=torch.int32, device="cuda")
    lt.lt_dsa_union_mask(dev, N, group, pos, length, mask)
    unions, masks = union_and_masks(idx.astype(np.int64), N, group)
    pos, length, mask = pos.cpu().numpy(), length.cpu().numpy(), mask.cpu().numpy().view(np.uint32)
    for g, u in enumerate(unions):
        assert length[g] == u.size and np.array_equal(pos[g, :u.size].astype(np.int64), u) and np.all(pos[g, u.size:] == -1)
    for t in range(T):
        assert np.array_equal(mask[t], pack_mask_words(masks[t], words)), t


# whole rows beside every size of bitmap, by CTAs of both sizes, around the longest single window, and one position to a row
@pytest.mark.parametrize("T,topk,N,group", [(32, 2048, 1200000, 32), (32, 2048, 1572864, 32), (32, 2048, 1572865, 32), (8, 2048, 200000, 8), (8, 2048, 400000, 8),
                                            (130, 1024, 262145, 128), (33, 2044, 90000, 32), (5, 4, 40, 5), (1, 4096, 131072, 1)])
def test_union_masks_by_whole_rows_everywhere(T, topk, N, group):
    test_union_masks_by_whole_rows(T, topk, N, group, 0)


# around a digit of 2048 positions, a CTA's 4096, one block of 256 keys more or less, and as many keys as a workspace holds
@pytest.mark.parametrize("N,n_out", [(2047, 256), (2048, 257), (2049, 255), (4096, 4096), (4097, 1), (8193, 8192), (1 << 18, 6144)])
def test_frequent_positions_around_digits(N, n_out):
    rng = np.random.default_rng(N + n_out)
    idx = np.where(rng.random((40, 300)) < 0.5, rng.integers(0, max(1, N // 50), size=(40, 300)), rng.integers(-2, N + 2, size=(40, 300)))
    dev = torch.from_numpy(idx.astype(np.int32)).cuda()
    out = torch.full((2, n_out), -5, dtype=torch.int32, device="cuda")
    ws = torch.full((lt.lt_topk_frequent_workspace_bytes(N),), 0xff, dtype=torch.uint8, device="cuda")
    lt.lt_topk_frequent(dev, N, out[0], out[1], ws)
    clean = np.where((idx >= 0) & (idx < N), idx, -1)
    want_pos, want_count = frequent_positions(clean, N, n_out)
    assert np.array_equal(out[0].cpu().numpy().astype(np.int64), want_pos)
    assert np.array_equal(out[1].cpu().numpy().astype(np.int64), want_count)


# samples that a CTA holds in registers or reads again, for its three sizes; the paper's rank lies below the bins looked at first
@pytest.mark.parametrize("T", [5, 300])
@pytest.mark.parametrize("tun", [dict(sample_mult=1), dict(sample_mult=15), dict(sample_mult=17), dict(sample_mult=36), dict(sample_mult=33, sample_rank=-1),
                                 dict(sample_rank=-1), dict(sample_rank=10 ** 6)])
def test_any_sample_gives_the_same_bits(T, tun):
    inp = make_config("fp8_ar1", T=T, N=20000, topk=256)
    want = run_unfused(inp, rows_per_pass=304)
    idx, score, status = run_topk(inp, lt.Tunables(path=lt.LT_PATH_FUSED, **tun))
    assert status[0] & lt.LT_STATUS_TIMEOUT == 0
    assert np.array_equal(idx, want[0]) and np.array_equal(score.view(np.uint32), want[1].view(np.uint32))


# either side of the rank and the size from which a sample is cut before it is counted (an eighth, 2048 scores), in one batch of loads and
# in several, in a sample smaller than its rank, and with keys that stretch every row's range
@pytest.mark.parametrize("T", [5, 300])
@pytest.mark.parametrize("outliers", [False, True])
@pytest.mark.parametrize("topk,offset,tun", [(256, 19000, dict(sample_mult=8, sample_rank=-1)), (256, 19000, dict(sample_mult=8, sample_rank=255)),
                                             (255, 19000, dict(sample_mult=8, sample_rank=200)), (256, 19000, dict(sample_mult=70, sample_rank=-1)),
                                             (2048, 19000, dict(sample_mult=8, sample_rank=-1)),
                                             (256, 100, dict(sample_rank=-1)), (1, 19000, dict(sample_mult=1, sample_rank=-1))])
def test_sample_ranks_around_the_cut(T, outliers, topk, offset, tun):
    inp = make_config("fp8_ar1", T=T, N=20000, topk=topk)
    inp = dataclasses.replace(inp, causal_offset=offset)
    if outliers:
        scale = inp.k_scale.copy()
        scale[::911] *= np.float32(50.0)
        inp = dataclasses.replace(inp, k_scale=scale)
    want = run_unfused(inp, rows_per_pass=304)
    idx, score, status = run_topk(inp, lt.Tunables(path=lt.LT_PATH_FUSED, **tun))
    assert status[0] & lt.LT_STATUS_TIMEOUT == 0
    assert np.array_equal(idx, want[0]) and np.array_equal(score.view(np.uint32), want[1].view(np.uint32))


# dense form (one CTA per row, clusters), sampled form, no common prefix to sample, more CTAs than status bytes
@pytest.mark.parametrize("T,N,offset,tun", [(3, 5000, 4997, None), (2, 40000, 39998, None), (40, 9000, 8960, dict(path=lt.LT_PATH_FUSED)),
                                            (40, 9000, -5, dict(path=lt.LT_PATH_FUSED)), (6, 3000, -4, None),
                                            (40, 9000, 8960, dict(path=lt.LT_PATH_FUSED, grid=296, segment_tiles=2))])
def test_status_block_of_a_workspace_full_of_ones(T, N, offset, tun):
    inp = dataclasses.replace(make_config("fp8_ar1", T=T, N=N, topk=64), causal_offset=offset)
    tun = lt.Tunables(**tun) if tun else None
    q, w, k, ks = lt.to_device(inp)
    ws = lt.alloc_workspace(inp.dtype, T, N, inp.H, inp.D, 64, tun)
    idx = torch.empty((T, 64), dtype=torch.int32, device="cuda")
    score = torch.empty((T, 64), device="cuda")
    want = run_unfused(inp)
    for _ in range(2):
        ws.fill_(0xff)
        lt.lt_indexer_topk_ex(inp.dtype, q, w, k, ks, 64, offset, idx, score, ws, tun)
        status = lt.lt_read_status(ws)
        assert status[0] & ~lt.LT_STATUS_FALLBACK == 0 and status[4] == 0 and status[6] == 0 and status[7] == 0, status
        assert 0 <= status[2] <= N and 0 <= status[3] <= T * N, status
        assert np.array_equal(idx.cpu().numpy(), want[0]) and np.array_equal(score.cpu().numpy().view(np.uint32), want[1].view(np.uint32))


@pytest.mark.parametrize("T,N", [(4, 3000), (70, 30000)])
def test_status_block_of_the_knn_variant(T, N):
    inp = make_knn(T=T, N=N, D=64, topk=10)
    q, x = (torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda() for a in (inp.q, inp.x))
    ws = torch.full((lt.lt_knn_topk_workspace_bytes(T, N, 64, 10),), 0xff, dtype=torch.uint8, device="cuda")
    idx = torch.empty((T, 10), dtype=torch.int32, device="cuda")
    lt.lt_knn_topk(q, x, 10, idx, None, ws)
    status = lt.lt_read_status(ws)
    assert status[0] & ~lt.LT_STATUS_FALLBACK == 0 and status[6] == 0 and status[7] == 0, status


# row blocks of very different length, enough of them for whole rows to be one item each; a ragged last block and last tile
@pytest.mark.parametrize("name", ["dsa_bf16", "fp8_ar1"])
@pytest.mark.parametrize("offset,path", [(0, lt.LT_PATH_AUTO), (0, lt.LT_PATH_FUSED), (-700, lt.LT_PATH_AUTO), (900, lt.LT_PATH_FUSED)])
def test_triangular_mask(name, offset, path):
    inp = dataclasses.replace(make_config(name, T=2405, N=2405, topk=64), causal_offset=offset)
    want = run_unfused(inp, rows_per_pass=1208)
    idx, score, status = run_topk(inp, lt.Tunables(path=path))
    assert status[0] & lt.LT_STATUS_TIMEOUT == 0
    assert np.array_equal(idx, want[0]) and np.array_equal(score.view(np.uint32), want[1].view(np.uint32))


# "do not split": a segment longer than any row, in the forms that scan with one unit, two units, a sample, vectors, and through the fallback
@pytest.mark.parametrize("segment_tiles", [1 << 24, 1 << 30, 2 ** 31 - 1])
@pytest.mark.parametrize("T,N,tun", [(1, 40000, {}), (64, 9000, {}), (70, 9000, dict(path=lt.LT_PATH_FUSED)), (9, 40000, dict(path=lt.LT_PATH_FUSED, grid=296)),
                                     (40, 9000, dict(path=lt.LT_PATH_FUSED, cap_mult=1, sample_rank=1)), (20, 9000, dict(path=lt.LT_PATH_FUSED_ABS))])
def test_segments_longer_than_the_context(segment_tiles, T, N, tun):
    inp = make_config("fp8_ar1", T=T, N=N, topk=128)
    want = run_topk(inp, lt.Tunables(**tun))
    idx, score, status = run_topk(inp, lt.Tunables(segment_tiles=segment_tiles, **tun))
    assert status[0] & lt.LT_STATUS_TIMEOUT == 0 and (status[1] > 0) == (want[2][1] > 0)
    assert np.array_equal(idx, want[0]) and np.array_equal(score.view(np.uint32), want[1].view(np.uint32))


@pytest.mark.parametrize("segment_tiles", [1 << 24, 2 ** 31 - 1])
@pytest.mark.parametrize("path", [lt.LT_PATH_AUTO, lt.LT_PATH_FUSED])
def test_segments_longer_than_the_corpus(segment_tiles, path):
    inp = make_knn(T=70, N=9000, D=64, topk=100)
    q, x = (torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda() for a in (inp.q, inp.x))
    bits = []
    for tun in (lt.Tunables(path=path), lt.Tunables(path=path, segment_tiles=segment_tiles)):
        ws = torch.empty(lt.lt_knn_topk_workspace_bytes(70, 9000, 64, 100, tun), dtype=torch.uint8, device="cuda")
        idx, score = torch.empty((70, 100), dtype=torch.int32, device="cuda"), torch.empty((70, 100), device="cuda")
        lt.lt_knn_topk(q, x, 100, idx, score, ws, tun)
        assert lt.lt_read_status(ws)[0] & lt.LT_STATUS_TIMEOUT == 0
        bits.append((idx.cpu().numpy(), score.cpu().numpy().view(np.uint32)))
    assert np.array_equal(bits[0][0], bits[1][0]) and np.array_equal(bits[0][1], bits[1][1])
