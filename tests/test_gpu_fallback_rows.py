"""The exact fallback with more flagged rows than it launches CTAs: every CTA then selects several rows one after the other, of different
kinds, over the same shared memory.  Bits only."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2607_11976_b200 import binding as lt
from workloads import make_config, make_knn

from gpu_util import run_topk, run_unfused

pytestmark = pytest.mark.gpu

ALL_ROWS = dict(path=lt.LT_PATH_FUSED, cap_mult=1, sample_rank=1)  # a gate so tight that every row is short of keys


# rows of one, two and more batches of registers, rows that see fewer keys than topk, and rows that one CTA cannot hold
@pytest.mark.parametrize("name,T,N,topk,offset", [("fp8_ar1", 700, 3000, 300, 2300), ("dsa_bf16", 1300, 9000, 600, 7700), ("fp8_ar1", 905, 2000, 500, 100),
                                                  ("fp8_ar1", 640, 17000, 2048, 16360)])
def test_several_rows_per_cta(name, T, N, topk, offset):
    inp = make_config(name, T=T, N=N, topk=topk)
    w = inp.w.copy()
    w[5::7] = 0.0           # mass ties: the radix select, between rows that the distribution sort takes
    w[3::11] *= np.float32(1e-30)
    inp = dataclasses.replace(inp, w=w, causal_offset=offset)
    want = run_unfused(inp, rows_per_pass=656)
    idx, score, status = run_topk(inp, lt.Tunables(**ALL_ROWS))
    assert status[0] & lt.LT_STATUS_TIMEOUT == 0 and status[1] > 2 * 296
    assert np.array_equal(idx, want[0]) and np.array_equal(score.view(np.uint32), want[1].view(np.uint32))


@pytest.mark.parametrize("T,N,topk", [(700, 5000, 100), (605, 20000, 1024)])
def test_several_rows_per_cta_knn(T, N, topk):
    inp = make_knn(T=T, N=N, D=64, topk=topk)
    q, x = (torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda() for a in (inp.q, inp.x))
    q[4::9] = 0  # every score of these is zero
    bits = []
    for tun in (lt.Tunables(path=lt.LT_PATH_FUSED), lt.Tunables(**ALL_ROWS)):
        ws = torch.empty(lt.lt_knn_topk_workspace_bytes(T, N, 64, topk, tun), dtype=torch.uint8, device="cuda")
        idx, score = torch.empty((T, topk), dtype=torch.int32, device="cuda"), torch.empty((T, topk), device="cuda")
        lt.lt_knn_topk(q, x, topk, idx, score, ws, tun)
        status = lt.lt_read_status(ws)
        assert status[0] & lt.LT_STATUS_TIMEOUT == 0
        bits.append((idx.cpu().numpy(), score.cpu().numpy().view(np.uint32), status[1]))
    assert bits[1][2] > 2 * 296 - T // 9 and np.array_equal(bits[0][0], bits[1][0]) and np.array_equal(bits[0][1], bits[1][1])
