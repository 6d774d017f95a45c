"""The dense form of small problems (scores of whole rows, then a full-row select): the sizes at which the select changes
hands (one CTA per row, clusters of 2 to 16 CTAs) and at which the sampled form takes over, rows that see few or no keys, score
distributions that overfill a bin (heavy tails, mass ties).  Arbiter: the library's own dense dump, bit for bit; the sampled
form, asked for by path, must give the same bits."""
import numpy as np
import pytest
import torch

from paper_2607_11976_b200 import binding as lt
from workloads import make_inputs

from gpu_util import assert_matches_oracle, assert_own_scores_rule, dump_scores, run_topk

pytestmark = pytest.mark.gpu


def _check(inp, oracle_rows=()):
    idx, score, status = run_topk(inp)
    assert status[0] == 0 and status[3] == 0  # no candidates were filtered: the dense form ran
    dumped = dump_scores(inp, 0, inp.T)
    assert_own_scores_rule(inp, idx, score, dumped, range(inp.T))
    if oracle_rows:
        assert_matches_oracle(inp, idx, score, list(oracle_rows), dumped)
    f_idx, f_score, _ = run_topk(inp, lt.Tunables(path=lt.LT_PATH_FUSED))
    assert np.array_equal(idx, f_idx) and np.array_equal(score.view(np.uint32), f_score.view(np.uint32))


@pytest.mark.parametrize("recipe,dtype", [("iid", "bf16"), ("ar1", "e4m3")])
@pytest.mark.parametrize("T,N,topk", [(1, 16384, 2048), (1, 16385, 2047), (3, 16389, 1), (2, 32769, 500), (4, 65537, 8191),
                                      (1, 131073, 2048), (5, 131077, 3000), (10, 200001, 64), (31, 131071, 64),
                                      (300, 4097, 2048), (9, 127, 127)])
def test_sizes(recipe, dtype, T, N, topk):
    inp = make_inputs(recipe, dtype, T=T, N=N, H=64, D=128, topk=topk, seed=N)
    _check(inp, oracle_rows=(0, T - 1))


@pytest.mark.parametrize("recipe", ["ties", "ties_exact", "planted", "cluster"])
@pytest.mark.parametrize("N,topk", [(5000, 700), (20011, 64), (40000, 5001), (140000, 2048)])
def test_crowded_scores(recipe, N, topk):
    _check(make_inputs(recipe, "bf16", T=3, N=N, H=64, D=128, topk=topk, seed=N))


@pytest.mark.parametrize("N", [3000, 50000])
@pytest.mark.parametrize("offset", [-5, 0, 100, 2040])
def test_rows_with_few_keys(N, offset):
    _check(make_inputs("iid", "bf16", T=20, N=N, H=64, D=128, topk=2048, seed=N, causal_offset=offset))


def test_one_score_everywhere():
    inp = make_inputs("iid", "bf16", T=2, N=70001, H=64, D=128, topk=2000, seed=4)
    inp.k[:] = inp.k[0]
    _check(inp)
    inp.w[:] = 0.0  # all scores are +0
    _check(inp)


@pytest.mark.parametrize("N,topk", [(16388, 64), (20011, 2048), (131072, 8192), (300001, 64), (500000, 2048)])
@pytest.mark.parametrize("values", [2, 50])
def test_few_different_scores(values, N, topk):
    """A threshold bin of one value: its keys are told apart by their indices, in the clusters' slices and at their borders."""
    inp = make_inputs("iid", "bf16", T=3, N=N, H=64, D=128, topk=topk, seed=N)
    inp.k[:] = inp.k[np.random.default_rng(values).integers(0, values, size=N)]
    _check(inp)
    inp.k[N // 3:] = inp.k[0]  # two thirds of the row are one run of ties
    _check(inp)


def test_paged_keys_take_the_dense_form_too():
    N, T = 30011, 3
    inp = make_inputs("ar1", "e4m3", T=T, N=N, H=64, D=128, topk=600, seed=8)
    want_idx, want_score, _ = run_topk(inp)
    q, w, k, ks = lt.to_device(inp)
    n_pages = (N + 63) // 64
    table = torch.randperm(n_pages + 7, device="cuda")[:n_pages]
    pool = torch.zeros(((n_pages + 7), 64, 128), dtype=torch.uint8, device="cuda")
    pool_scale = torch.zeros((n_pages + 7, 64), device="cuda")
    pool[table] = torch.nn.functional.pad(k, (0, 0, 0, n_pages * 64 - N)).reshape(n_pages, 64, 128)
    pool_scale[table] = torch.nn.functional.pad(ks, (0, n_pages * 64 - N)).reshape(n_pages, 64)
    idx = torch.empty((T, 600), dtype=torch.int32, device="cuda")
    score = torch.empty((T, 600), device="cuda")
    ws = torch.empty(lt.lt_indexer_topk_paged_workspace_bytes("e4m3", T, N, 64, 128, 600), dtype=torch.uint8, device="cuda")
    lt.lt_indexer_topk_paged("e4m3", q, w, pool.reshape(-1, 128), pool_scale.reshape(-1), table.to(torch.int32), N, 600,
                             inp.causal_offset, idx, score, ws)
    assert lt.lt_read_status(ws)[0] == 0
    assert np.array_equal(idx.cpu().numpy(), want_idx) and np.array_equal(score.cpu().numpy().view(np.uint32), want_score.view(np.uint32))


def test_a_workspace_of_the_default_size_serves_every_path():
    inp = make_inputs("ar1", "e4m3", T=64, N=16384, H=64, D=128, topk=256, seed=3)
    want_idx, want_score, _ = run_topk(inp)
    q, w, k, ks = lt.to_device(inp)
    ws = lt.alloc_workspace("e4m3", 64, 16384, 64, 128, 256)
    for topk, path in ((256, lt.LT_PATH_FUSED), (256, lt.LT_PATH_AUTO), (100, lt.LT_PATH_FUSED)):
        idx = torch.empty((64, topk), dtype=torch.int32, device="cuda")
        score = torch.empty((64, topk), device="cuda")
        lt.lt_indexer_topk_ex("e4m3", q, w, k, ks, topk, inp.causal_offset, idx, score, ws, lt.Tunables(path=path))
        assert lt.lt_read_status(ws)[0] == 0
        assert np.array_equal(idx.cpu().numpy(), want_idx[:, :topk])
        assert np.array_equal(score.cpu().numpy().view(np.uint32), want_score[:, :topk].view(np.uint32))
