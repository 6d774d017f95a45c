"""What the size functions promise (host arithmetic, no GPU): a workspace sized once with default tunables serves the same problem by
every path, and a problem whose topk, rows or keys are fewer.  Around the lines where LT_PATH_AUTO changes its form."""
import pytest

from paper_2607_11976_b200 import binding as lt
from paper_2607_11976_b200 import build


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def sizes(T, N, topk, tun=None):
    return {"dense keys": lt.lt_indexer_topk_workspace_bytes("e4m3", T, N, 64, 128, topk, tun),
            "paged keys": lt.lt_indexer_topk_paged_workspace_bytes("e4m3", T, N, 64, 128, topk, tun),
            "k-NN": lt.lt_knn_topk_workspace_bytes(T, N, 128, topk, tun)}


SHAPES = [(64, 16384, 256), (1, 131072, 2048), (4, 524288, 2048), (4096, 4096, 2048), (4096, 16384, 2048), (4096, 16384, 512), (8, 300000, 64),
          (300, 16384, 64), (1025, 16384, 511), (64, 65536, 2048), (65, 65536, 512), (1, 8192, 8192), (9, 100, 1)]


@pytest.mark.parametrize("T,N,topk", SHAPES)
def test_the_default_size_serves_every_path(T, N, topk):
    auto = sizes(T, N, topk)
    for path in (lt.LT_PATH_FUSED, lt.LT_PATH_GENERIC):
        need = lt.lt_indexer_topk_workspace_bytes("e4m3", T, N, 64, 128, topk, lt.Tunables(path=path))
        assert 0 < need <= auto["dense keys"]
    # the sampled form asked for by path or by a tunable that does not enlarge it
    for tun in (lt.Tunables(path=lt.LT_PATH_FUSED), lt.Tunables(cap_mult=1), lt.Tunables(segment_tiles=3, grid=7)):
        for what, need in sizes(T, N, topk, tun).items():
            assert 0 < need <= auto[what], (what, need, auto[what])


@pytest.mark.parametrize("T,N,topk", SHAPES)
def test_a_smaller_problem_never_needs_more(T, N, topk):
    auto = sizes(T, N, topk)
    # (a topk that is a large part of the keys draws a smaller sample than one of half its size, and the sample is kept in the workspace)
    sample = lambda k: lt.lt_indexer_sample_plan(N, k, N - 1)[0]
    smaller = [(T, N, k) for k in (topk // 2, topk // 5, 511, 1) if 0 < k < topk and sample(k) <= sample(topk)]
    smaller += [(t, N, topk) for t in (T // 2, T - 1, 8, 1) if 0 < t < T]
    smaller += [(T, n, topk) for n in (N // 2, N - 1, 16384, 8192) if topk <= n < N]
    for t, n, k in smaller:
        for what, need in sizes(t, n, k).items():
            assert need <= auto[what], (what, (t, n, k), need, auto[what])
