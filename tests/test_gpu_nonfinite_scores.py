"""Finite inputs whose scores overflow fp32: rows with infinite and NaN scores, and rows whose range is wider than a float, at the sizes
where the full-row select changes hands (one CTA per row, clusters).  Arbiter: the library's own dense dump, ranked on the host
by the order of the bit patterns, in which every score has a place."""
import numpy as np
import pytest

from paper_2607_11976_b200 import binding as lt
from workloads import make_inputs

from gpu_util import assert_own_scores_rule, dump_scores, run_topk, run_unfused

pytestmark = pytest.mark.gpu


def rank_bits(row, topk):
    """(indices, score bits) of the topk largest scores of a row in the order of their bit patterns, ties to the lower index."""
    bits = np.ascontiguousarray(row, dtype=np.float32).view(np.uint32)
    key = np.where(bits >> 31, ~bits, bits | np.uint32(0x80000000)).astype(np.int64)
    order = np.argsort(-key, kind="stable")[:topk]
    return order, bits[order]


def overflowing(kind, dtype, T, N, H, D, topk):
    inp = make_inputs("iid", dtype, T=T, N=N, H=H, D=D, topk=topk, seed=N + topk)

    def put(a, v):  # a value into (part of) an array of fp32 values or of bf16 bit patterns
        a[...] = v if dtype == "f32" else np.float32(v).view(np.uint32) >> 16

    # the even heads look at the first half of the coordinates, the odd ones at the second; the latter count negative
    put(inp.q, 0.0)
    half = D // 2
    inp.w[:, ::2], inp.w[:, 1::2] = 1.0, -1.0
    big = 3e38 / (H // 2 * half) if kind == "wide" else 1e20
    put(inp.q[:, ::2, :half], 1.0 if kind == "wide" else big)
    put(inp.q[:, 1::2, half:], 1.0 if kind == "wide" else big)
    if kind == "one_inf":
        put(inp.k[777:778, :half], big)
    elif kind == "all_minus_inf":
        put(inp.k, 0.0)
        put(inp.k[:, half:], big)
    elif kind == "some_minus_inf":
        put(inp.k[N // 2:, :half], 0.0)
        put(inp.k[N // 2:, half:], big)
    elif kind == "some_nan":
        put(inp.k[2::4], big)
    else:  # mixed: infinities of both signs, NaN, finite ones; wide: finite scores of both signs, more than a float apart
        put(inp.k[::4], 0.0)
        put(inp.k[::4, :half], big)
        put(inp.k[1::4], 0.0)
        put(inp.k[1::4, half:], big)
        if kind == "mixed":
            put(inp.k[2::4], big)
    return inp


@pytest.mark.parametrize("kind", ["one_inf", "all_minus_inf", "some_minus_inf", "some_nan", "wide", "mixed"])
@pytest.mark.parametrize("N,topk", [(9000, 500), (20000, 500), (20001, 500), (140000, 64), (20000, 8192)])
def test_generic_path(kind, N, topk):
    inp = overflowing(kind, "f32", T=3, N=N, H=2, D=8, topk=topk)
    idx, score, _ = run_topk(inp)
    u_idx, u_score, _ = run_unfused(inp, rows_per_pass=2)
    dumped = dump_scores(inp, 0, inp.T, lt.LT_PATH_GENERIC)
    for t in range(inp.T):
        vis = inp.visible(t)
        if kind in ("mixed", "some_nan"):
            assert np.isnan(dumped[t][:vis]).any()
        want_idx, want_bits = rank_bits(dumped[t][:vis], topk)
        for i, s in ((idx, score), (u_idx, u_score)):
            assert np.array_equal(i[t], want_idx) and np.array_equal(s[t].view(np.uint32), want_bits)


@pytest.mark.parametrize("kind", ["one_inf", "all_minus_inf", "some_minus_inf", "wide"])
@pytest.mark.parametrize("N,topk", [(9000, 500), (20011, 2000), (65540, 64), (140000, 2048)])
def test_dense_form(kind, N, topk):
    inp = overflowing(kind, "bf16", T=3, N=N, H=64, D=128, topk=topk)
    idx, score, status = run_topk(inp)
    assert status[0] == 0 and status[3] == 0  # the dense form ran
    dumped = dump_scores(inp, 0, inp.T)
    assert not np.isnan(dumped).any()
    assert_own_scores_rule(inp, idx, score, dumped, range(inp.T))


@pytest.mark.parametrize("dtype,N", [("bf16", 70000), ("bf16", 30000)])
def test_nan_in_the_sample_costs_the_row_nothing(dtype, N):
    """Key 0 is in every sample.  Its score is NaN, which the gate never passes: the row is selected from the other keys, by the
    sampled form's own means and not by its fallback."""
    inp = make_inputs("iid", dtype, T=20, N=N, H=64, D=128, topk=100, seed=5)
    inp.w[:, ::2], inp.w[:, 1::2] = np.abs(inp.w[:, ::2]), -np.abs(inp.w[:, 1::2])
    inp.q[:, 0], inp.q[:, 1] = inp.q[:, 0] & 0x7FFF, inp.q[:, 0] & 0x7FFF  # a head of each sign that sees key 0 overflow
    inp.k[0] = np.float32(3e38).view(np.uint32) >> 16
    idx, score, status = run_topk(inp, lt.Tunables(path=lt.LT_PATH_FUSED))
    assert status[0] == 0 and status[1] == 0  # no row took the fallback
    dumped = dump_scores(inp, 0, inp.T)
    assert np.isnan(dumped[:, 0]).all() and not np.isnan(dumped[:, 1:]).any()
    assert_own_scores_rule(inp, idx, score, dumped, range(inp.T))  # (the host's ranking puts NaN last)


@pytest.mark.parametrize("N,topk", [(9000, 500), (20011, 2000), (65540, 64), (140000, 2048), (5000, 5000), (30000, 8192)])
@pytest.mark.parametrize("nan", ["some", "most"])
def test_nan_scores_rank_alike_in_both_forms(nan, N, topk):
    """The gate of the sampled form lets no NaN pass, and a row that is then short of keys is redone by the order of the bit patterns:
    the dense form of the same problem has to put NaN scores last where there are enough others, first where there are not."""
    inp = make_inputs("iid", "bf16", T=3, N=N, H=64, D=128, topk=topk, seed=5)
    inp.w[:, ::2], inp.w[:, 1::2] = np.abs(inp.w[:, ::2]), -np.abs(inp.w[:, 1::2])
    inp.q[:, 0], inp.q[:, 1] = inp.q[:, 0] & 0x7FFF, inp.q[:, 0] & 0x7FFF  # a head of each sign that sees the large keys overflow
    large = np.random.default_rng(N).permutation(N)[:20 if nan == "some" else N - topk // 2]
    inp.k[large] = np.float32(3e38).view(np.uint32) >> 16
    dumped = dump_scores(inp, 0, inp.T)
    idx, score, status = run_topk(inp)
    assert status[3] == 0  # the dense form ran
    f_idx, f_score, _ = run_topk(inp, lt.Tunables(path=lt.LT_PATH_FUSED))
    assert np.array_equal(idx, f_idx) and np.array_equal(score.view(np.uint32), f_score.view(np.uint32))
    for t in range(inp.T):
        row = dumped[t][:inp.visible(t)]
        enough = np.count_nonzero(~np.isnan(row)) >= min(topk, row.size)
        if nan == "some" and topk < N - 100:
            assert enough and np.isnan(row).any()
        want_idx, want_bits = rank_bits(np.where(np.isnan(row), -np.inf, row) if enough else row, topk)
        n = want_idx.size
        assert np.array_equal(idx[t][:n], want_idx) and np.array_equal(score[t][:n].view(np.uint32), want_bits)
