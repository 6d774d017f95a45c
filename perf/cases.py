"""The workloads by which the library's speed is judged, each through the public entry points of the binding.

A case is a plain dict: an operation ("op") with its sizes and options.  The sizes are those of the repository's own
configurations (`workloads/gen.py`), its benchmark and its tests, or generic ones between them:

  chunk     lt_indexer_topk_ex over a dense key cache: prefill chunks of every length, decode steps, verification of a
            few drafted tokens; e4m3 and bf16 keys with the indexer's 64 heads of 128, other shapes and fp32 on the
            generic path
  paged     lt_indexer_topk_paged: the same over a paged key cache, pages in random order
  next      one chunk of a long prompt served with the previous chunk's result: lt_topk_frequent over the previous
            chunk's indices, then lt_indexer_topk_sampled with the positions it returned
  knn       lt_knn_topk: exact inner-product search over a corpus of embeddings
  union     lt_dsa_union_mask: union list and membership masks of groups of adjacent rows
"""
import math

import torch

from paper_2607_11976_b200 import binding as lt


def listed():
    return [
        # the generic path: fp32 and a head shape the tensor-core kernels do not take (the repository's smallest
        # configuration; a debugging or research model)
        dict(name="generic_f32", op="chunk", dtype="f32", T=64, N=4096, H=8, D=64, topk=256, offset=4032, recipe="iid", scores=True),
        # one token of one sequence, serving cache: the smallest call there is, latency counts
        dict(name="decode_paged_fp8_128k", op="paged", dtype="e4m3", T=1, N=131072, H=64, D=128, topk=2048, offset=131071, recipe="ar1", scores=False),
        # four drafted tokens verified at once at the longest context
        dict(name="verify_fp8_1m", op="chunk", dtype="e4m3", T=4, N=1048576, H=64, D=128, topk=2048, offset=1048572, recipe="ar1", scores=True),
        # the short last chunk of a prompt, odd sizes
        dict(name="tail_chunk_fp8_300k", op="chunk", dtype="e4m3", T=77, N=300017, H=64, D=128, topk=2048, offset=299940, recipe="ar1", scores=True),
        # the first chunk of a prompt: triangular mask, the first half of the rows sees fewer keys than topk
        dict(name="first_chunk_bf16_4k", op="chunk", dtype="bf16", T=4096, N=4096, H=64, D=128, topk=2048, offset=0, recipe="drift", scores=True),
        # an ordinary prefill chunk in bf16
        dict(name="chunk_bf16_64k", op="chunk", dtype="bf16", T=4096, N=65536, H=64, D=128, topk=2048, offset=61440, recipe="drift", scores=True),
        # a large prefill chunk over fp8 keys
        dict(name="chunk_fp8_128k", op="chunk", dtype="e4m3", T=8192, N=131072, H=64, D=128, topk=2048, offset=122880, recipe="ar1", scores=True),
        # the headline configuration and the largest case
        dict(name="chunk_fp8_1m", op="chunk", dtype="e4m3", T=4096, N=1048576, H=64, D=128, topk=2048, offset=1044480, recipe="ar1", scores=True),
        # a ragged prefill chunk over the serving cache
        dict(name="chunk_paged_fp8_200k", op="paged", dtype="e4m3", T=1000, N=200003, H=64, D=128, topk=2048, offset=199003, recipe="ar1", scores=True),
        # a chunk whose sample is taken from the previous chunk's result
        dict(name="next_chunk_fp8_256k", op="next", dtype="e4m3", T=1024, N=262144, H=64, D=128, topk=2048, offset=261120, recipe="hot", scores=True),
        # retrieval: a batch of 64 queries over a million 768-d embeddings
        dict(name="knn_bf16_1m", op="knn", dtype="bf16", T=64, N=1048576, D=768, topk=1024),
        # the union lists and masks of a chunk whose rows share part of their keys
        dict(name="union_128k", op="union", T=4096, N=131072, topk=2048, group=64),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["chunk", "chunk", "chunk", "decode", "decode", "paged", "next", "knn", "union", "generic"])
    if op == "generic":
        T, N, H, D = _log_int(rng, 1, 128), _log_int(rng, 512, 16384), rng.choice([4, 8, 16, 32]), rng.choice([32, 64, 96, 128])
        return dict(op="chunk", dtype=rng.choice(["f32", "f32", "bf16"]), T=T, N=N, H=H, D=D, topk=min(N, rng.choice([64, 256, 512])),
                    offset=max(0, N - T), recipe="iid", scores=True)
    if op == "knn":
        N, D = _log_int(rng, 20000, 1 << 20), 64 * rng.randint(2, 12)
        return dict(op="knn", dtype="bf16", T=_log_int(rng, 1, 256), N=N, D=D, topk=rng.choice([10, 100, 128, 1024, 4096]))
    if op == "union":
        return dict(op="union", T=_log_int(rng, 256, 4096), N=_log_int(rng, 16384, 1 << 20), topk=rng.choice([512, 1024, 2048]),
                    group=rng.choice([16, 32, 64, 128]))
    dtype = rng.choice(["e4m3", "e4m3", "bf16"])
    N = _log_int(rng, 4096, 1 << 20)
    if op == "decode":
        op, T = rng.choice(["chunk", "paged"]), rng.choice([1, 1, 2, 4, 7, 8])
    else:
        # no more (row, key) pairs than the largest listed case; bf16 pairs cost twice as much
        most = (1 << 31 if dtype == "bf16" else 1 << 32) // N
        T = _log_int(rng, 16, min(8192, N, most))
    topk = 2048 if rng.random() < 0.6 else rng.choice([64, 512, 1024, 4096])
    recipe = "hot" if op == "next" else ("ar1" if dtype == "e4m3" else "drift")
    return dict(op=op, dtype=dtype, T=T, N=N, H=64, D=128, topk=min(N, topk), offset=N - T, recipe=recipe, scores=rng.random() < 0.7)


# ---------------------------------------------------------------------------------------------
# inputs (device-side counterparts of the recipes in workloads/gen.py)
# ---------------------------------------------------------------------------------------------
def _quantize(x):
    """Per-token absmax e4m3 codes and scales."""
    flat = x.reshape(x.shape[0], -1)
    absmax = flat.abs().amax(dim=1)
    scale = torch.where(absmax > 0, absmax / 448.0, torch.ones_like(absmax))
    codes = (flat / scale[:, None]).clamp_(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8)
    return codes.reshape(x.shape), scale


def _indexer_inputs(case, g, dev):
    T, N, H, D = case["T"], case["N"], case["H"], case["D"]
    sd = D ** -0.5
    q = torch.randn((T, H * D), generator=g, device=dev).mul_(sd)
    w = torch.randn((T, H), generator=g, device=dev).mul_(H ** -0.5)
    k = torch.randn((N, D), generator=g, device=dev).mul_(sd)
    hot = None
    if case["recipe"] == "ar1":  # neighbouring tokens have similar queries
        c = (1.0 - 0.81) ** 0.5
        for t in range(1, T):
            q[t].mul_(c).add_(q[t - 1], alpha=0.9)
    elif case["recipe"] == "drift":  # keys carry a slow drift along one direction
        u = torch.nn.functional.normalize(torch.randn(D, generator=g, device=dev), dim=0)
        k += (0.2 * torch.sin(torch.arange(N, device=dev, dtype=torch.float64) / 4096.0)).float()[:, None] * u
    elif case["recipe"] == "hot":  # positions of the first half of the context that every chunk selects
        u = torch.nn.functional.normalize(torch.randn(D, generator=g, device=dev), dim=0)
        hot = torch.randperm(N // 2, generator=g, device=dev)[:min(N // 8, 3 * case["topk"] // 2)]
        k[hot] += u
        q += (0.5 * u).repeat(H)
        w = w.abs()
    q = q.reshape(T, H, D)
    if case["dtype"] == "e4m3":
        q, q_scale = _quantize(q)
        k, k_scale = _quantize(k)
        return q, w * q_scale[:, None], k, k_scale, hot
    if case["dtype"] == "bf16":
        q, k = q.to(torch.bfloat16), k.to(torch.bfloat16)
    return q, w, k, None, hot


def _embeddings(rows, D, centres, g, dev):
    """Unit vectors drawn around a few dozen centres."""
    out = torch.empty((rows, D), dtype=torch.bfloat16, device=dev)
    for r in range(0, rows, 1 << 18):
        n = min(1 << 18, rows - r)
        which = torch.randint(0, centres.shape[0], (n,), generator=g, device=dev)
        v = torch.randn((n, D), generator=g, device=dev).mul_(D ** -0.5).add_(centres[which], alpha=0.7)
        out[r:r + n] = torch.nn.functional.normalize(v, dim=1).to(torch.bfloat16)
    return out


def prepare(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    op = case["op"]
    s = dict(case=case)
    i32 = dict(dtype=torch.int32, device=dev)
    if op == "union":
        # rows of a group share about half of their keys, the others are scattered over what they can see
        T, N, topk, group = case["T"], case["N"], case["topk"], case["group"]
        shared = torch.randint(0, N, ((T + group - 1) // group, topk), generator=g, device=dev)
        idx = torch.randint(0, N, (T, topk), generator=g, device=dev)
        pick = torch.rand((T, topk), generator=g, device=dev) < 0.5
        idx = torch.where(pick, shared.repeat_interleave(group, dim=0)[:T], idx).to(torch.int32).contiguous()
        words = (group * topk + 31) // 32
        n_groups = (T + group - 1) // group
        s.update(idx=idx, pos=torch.empty((n_groups, group * topk), **i32), length=torch.empty(n_groups, **i32), mask=torch.empty((T, words), **i32))
        return s
    T, topk = case["T"], case["topk"]
    s.update(out_idx=torch.empty((T, topk), **i32), out_score=torch.empty((T, topk), device=dev) if case.get("scores", True) else None)
    if op == "knn":
        centres = torch.nn.functional.normalize(torch.randn((64, case["D"]), generator=g, device=dev), dim=1)
        s["x"] = _embeddings(case["N"], case["D"], centres, g, dev)
        s["q"] = _embeddings(T, case["D"], centres, g, dev)
        nbytes = lt.lt_knn_topk_workspace_bytes(T, case["N"], case["D"], topk)
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device=dev)
        return s
    q, w, k, ks, hot = _indexer_inputs(case, g, dev)
    args = (case["dtype"], T, case["N"], case["H"], case["D"], topk)
    if op == "paged":
        # the context's pages, scattered over a pool that other sequences use as well
        n_pages = (case["N"] + 63) // 64
        pool_pages = n_pages + n_pages // 4 + 1
        table = torch.randperm(pool_pages, generator=g, device=dev)[:n_pages]
        pool = torch.zeros((pool_pages, 64, case["D"]), dtype=k.dtype, device=dev)
        pad = torch.zeros((n_pages * 64, case["D"]), dtype=k.dtype, device=dev)
        pad[:case["N"]] = k
        pool[table] = pad.reshape(n_pages, 64, -1)
        pool_scale = None
        if ks is not None:
            pool_scale = torch.ones((pool_pages, 64), device=dev)
            pad_scale = torch.ones(n_pages * 64, device=dev)
            pad_scale[:case["N"]] = ks
            pool_scale[table] = pad_scale.reshape(n_pages, 64)
            pool_scale = pool_scale.reshape(-1)
        s.update(q=q, w=w, k=pool.reshape(pool_pages * 64, -1), ks=pool_scale, table=table.to(torch.int32))
        s["ws"] = torch.empty(lt.lt_indexer_topk_paged_workspace_bytes(*args), dtype=torch.uint8, device=dev)
        return s
    s.update(q=q, w=w, k=k, ks=ks)
    if op == "next":
        # the previous chunk's result: most of its rows' keys are the ones every chunk selects
        n_sample = min(3 * topk, case["N"])
        prev = torch.randint(0, case["offset"] + 1, (T, topk), generator=g, device=dev)
        pick = torch.rand((T, topk), generator=g, device=dev) < 0.8
        among = hot[torch.randint(0, hot.numel(), (T, topk), generator=g, device=dev)]
        s["prev"] = torch.where(pick, among, prev).to(torch.int32).contiguous()
        s["sample"] = torch.empty(n_sample, **i32)
        s["freq_ws"] = torch.empty(lt.lt_topk_frequent_workspace_bytes(case["N"]), dtype=torch.uint8, device=dev)
        nbytes = lt.lt_indexer_topk_sampled_workspace_bytes(*args, n_sample)
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device=dev)
        return s
    s["ws"] = lt.alloc_workspace(*args)
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "union":
        lt.lt_dsa_union_mask(s["idx"], case["N"], case["group"], s["pos"], s["length"], s["mask"])
        return s["pos"], s["length"], s["mask"]
    if op == "knn":
        lt.lt_knn_topk(s["q"], s["x"], case["topk"], s["out_idx"], s["out_score"], s["ws"])
        return s["out_idx"], s["out_score"]
    if op == "paged":
        lt.lt_indexer_topk_paged(case["dtype"], s["q"], s["w"], s["k"], s["ks"], s["table"], case["N"], case["topk"], case["offset"],
                                 s["out_idx"], s["out_score"], s["ws"])
    elif op == "next":
        lt.lt_topk_frequent(s["prev"], case["N"], s["sample"], None, s["freq_ws"])
        lt.lt_indexer_topk_sampled(case["dtype"], s["q"], s["w"], s["k"], s["ks"], case["topk"], case["offset"], s["sample"],
                                   s["out_idx"], s["out_score"], s["ws"])
        return s["sample"], s["out_idx"], s["out_score"]
    else:
        lt.lt_indexer_topk_ex(case["dtype"], s["q"], s["w"], s["k"], s["ks"], case["topk"], case["offset"], s["out_idx"], s["out_score"], s["ws"])
    return s["out_idx"], s["out_score"]


def _pairs(case):
    """Visible (row, key) pairs: row t sees keys 0 .. offset + t."""
    T, N, off = case["T"], case["N"], case["offset"]
    full = min(T, max(0, T - (N - 1 - off)))  # rows that see all N keys
    part = T - full
    return full * N + part * (off + 1) + part * (part - 1) // 2


def work(case):
    op = case["op"]
    if op == "union":
        T, topk, group = case["T"], case["topk"], case["group"]
        n_groups, words = (T + group - 1) // group, (group * topk + 31) // 32
        return dict(bytes=4 * (T * topk + n_groups * (group * topk + 1) + T * words), flops=0)
    T, N, D, topk = case["T"], case["N"], case["D"], case["topk"]
    out = T * topk * (8 if case.get("scores", True) else 4)
    if op == "knn":
        return dict(bytes=2 * D * (N + T) + out, flops=2 * T * N * D)
    H = case["H"]
    elem = {"f32": 4, "bf16": 2, "e4m3": 1}[case["dtype"]]
    nbytes = elem * D * (T * H + N) + 4 * T * H + (4 * N if case["dtype"] == "e4m3" else 0) + out
    if op == "next":
        nbytes += 4 * (T * topk + min(3 * topk, N))
    return dict(bytes=nbytes, flops=2 * H * D * _pairs(case))


def tolerance(case):
    """Scores are exact products summed in fp32 (64 heads or up to 768 coordinates): another order of the sums moves
    them by about 1e-6 of their size.  Indices are exact up to scores that close, which then change places."""
    if case["op"] == "union":
        return "exact"
    return {"rel": 5e-6, "max": 5e-5, "differ": 0.01}
