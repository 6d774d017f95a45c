"""The generic scoring kernel at the edges of its tiles (8 query rows, 128 keys, 8 heads, 16 coordinates): dense scores within
the tolerance of the oracle (fp32 sums of at most 33 x 17 terms: far inside 1e-3 of the row's RMS), masked keys -inf, top-k exact
on the library's own scores."""
import numpy as np
import pytest

from oracle import indexer_scores
from oracle.acceptance import REL_TOL
from paper_2607_11976_b200 import binding as lt
from workloads import make_inputs

from gpu_util import assert_own_scores_rule, dump_scores, run_topk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "e4m3"])
@pytest.mark.parametrize("T,N,H,D", [(1, 127, 1, 1), (1, 128, 8, 16), (4, 129, 9, 17), (5, 513, 7, 15), (8, 300, 16, 32), (9, 1025, 17, 33),
                                     (3, 40001, 3, 5), (17, 640, 8, 48)])
def test_tile_edges(dtype, T, N, H, D):
    inp = make_inputs("iid", dtype, T=T, N=N, H=H, D=D, topk=min(N, 50), seed=N + H)
    want = indexer_scores(inp.q, inp.w, inp.k, inp.k_scale, inp.dtype, inp.causal_offset, rows=list(range(T)))
    got = dump_scores(inp, 0, T, lt.LT_PATH_GENERIC)
    for r in range(T):
        vis = np.isfinite(want[r])
        assert np.all(np.isneginf(got[r][~vis]))
        assert np.abs(got[r][vis] - want[r][vis]).max() <= REL_TOL * np.sqrt(np.mean(want[r][vis] ** 2))
    part = dump_scores(inp, T // 2, T, lt.LT_PATH_GENERIC)  # another launch shape, the same bits
    assert np.array_equal(part.view(np.uint32), got[T // 2:].view(np.uint32))
    idx, score, _ = run_topk(inp, lt.Tunables(path=lt.LT_PATH_GENERIC))
    assert_own_scores_rule(inp, idx, score, got, range(T))
