"""The distribution sort behind the final select and the full-row select, at the sizes where it changes course: one batch of
registers (4096 candidates, 8192 visible keys) more or less, rows with fewer keys than topk, scores that crowd into few bins
(heavy tails, mass ties).  Arbiter: the library's own dense dump, ranked on the host, bit for bit."""
import pytest
import torch

from paper_2607_11976_b200 import binding as lt
from workloads import make_inputs

from gpu_util import assert_own_scores_rule, dump_scores, run_topk, run_unfused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recipe", ["iid", "ties_exact", "planted", "cluster"])
@pytest.mark.parametrize("n", [1, 2, 33, 4095, 4097, 8191, 8193, 8200])
def test_full_row_select(recipe, n):
    for topk in sorted({1, min(n, 2), min(n, 700), min(n, 2049), min(n, 8192)}):
        inp = make_inputs(recipe, "bf16", T=3, N=n + 1, H=64, D=128, topk=topk, seed=n, causal_offset=n - 2)
        idx, score, _ = run_unfused(inp, rows_per_pass=2)
        assert_own_scores_rule(inp, idx, score, dump_scores(inp, 0, 3), range(3))


@pytest.mark.parametrize("recipe", ["iid", "ties_exact", "planted", "cluster"])
@pytest.mark.parametrize("n,topk", [(4095, 4000), (4096, 17), (4097, 4097), (12289, 3000), (20000, 6000)])
def test_final_select(recipe, n, topk):
    # accept everything (rank rule with a sample smaller than topk): every visible key is a candidate
    tun = lt.Tunables(path=lt.LT_PATH_FUSED, sample_rank=-1, sample_mult=1)
    inp = make_inputs(recipe, "bf16", T=5, N=n, H=64, D=128, topk=topk, seed=n + topk, causal_offset=n - 3)
    idx, score, status = run_topk(inp, tun)
    assert status[0] & lt.LT_STATUS_TIMEOUT == 0
    assert_own_scores_rule(inp, idx, score, dump_scores(inp, 0, 5), range(5))


def test_no_visible_key():
    inp = make_inputs("iid", "bf16", T=4, N=500, H=64, D=128, topk=100, seed=1, causal_offset=-3)
    for idx, score, _ in (run_topk(inp, lt.Tunables(path=lt.LT_PATH_FUSED)), run_unfused(inp, rows_per_pass=4)):
        assert (idx[:2] == -1).all() and torch.isneginf(torch.from_numpy(score[:2])).all()
        assert_own_scores_rule(inp, idx, score, dump_scores(inp, 0, 4), range(4))
