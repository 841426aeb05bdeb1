"""The sparse attention's split of the selected rows over warps and CTAs and the merges that follow, against float64:
pairs (sequence, KV head) held by one warp, by several warps of a CTA and by many CTAs, groups served in passes of 16
heads, empty sequences, and a workspace that holds arbitrary data before the call.
"""
import math

import numpy as np
import pytest
import torch

from parity_util import check_attn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill
    build.build()
    hill.load()
    return hill


# (B, H, Hkv, tokens, kept per sequence)
CASES = [
    (1, 1, 1, 4096, [1]),                    # one batch: one warp
    (1, 2, 2, 4096, [33]),                   # two batches per pair
    (1, 1, 1, 40000, [40000]),               # one pair over all CTAs (1250 batches, two per warp)
    (1, 32, 1, 20000, [19999]),              # two passes of 16 heads, each over half of the CTAs
    (2, 20, 1, 4096, [4000, 0]),             # passes of 16 and 4 heads, an empty sequence
    (3, 40, 1, 2048, [2048, 31, 32]),        # passes of 16, 16 and 8
    (2, 24, 8, 4096, [3000, 257]),           # groups of 3
    (4, 32, 32, 4096, [819, 0, 1, 300]),     # many short pairs
    (8, 32, 32, 2048, [1999, 7, 0, 1024, 33, 64, 65, 2048]),
    (5, 14, 2, 5000, [5000, 4999, 1, 0, 2500]),   # groups of 7
]


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"B{c[0]}H{c[1]}kv{c[2]}n{max(c[4])}")
def test_attention_over_every_split(H, case, dtype):
    B, Hq, Hkv, n, kept = case
    g = torch.Generator(device="cuda").manual_seed(n + Hq)
    K, V = (torch.randn(B, Hkv, n, 128, generator=g, device="cuda").to(dtype) for _ in range(2))
    q = torch.randn(B, Hq, 128, generator=g, device="cuda").to(dtype)
    desc = H.make_desc(q, K, V)
    max_k = max(kept)
    idx = torch.full((B, max_k), -1, dtype=torch.int32, device="cuda")
    sets = []
    for b, m in enumerate(kept):
        t = torch.randperm(n, generator=g, device="cuda")[:m].sort().values
        idx[b, :m] = t.int()
        sets.append(t)
    count = torch.tensor(kept, dtype=torch.int32, device="cuda")
    out = torch.full((B, Hq, 128), float("nan"), device="cuda")
    ws = H.alloc_workspace(desc, 0, max_k)
    ws.fill_(0xFF)
    ref = np.zeros((B, Hq, 128))
    G = Hq // Hkv
    for b, t in enumerate(sets):
        for h in range(Hq if len(t) else 0):
            z = K[b, h // G, t].double() @ q[b, h].double() / math.sqrt(128)
            ref[b, h] = (torch.softmax(z, 0) @ V[b, h // G, t].double()).cpu().numpy()
    first = None
    for _ in range(2):   # (the second call finds what the first one left in the workspace)
        H.hill_gather_sparse_attn(desc, q, K, V, idx, count, max_k, out, ws)
        H.hill_sync_status()
        check_attn(out.cpu().numpy(), ref)
        if first is not None:
            assert torch.equal(out, first), "the order of the merge is fixed"
        first = out.clone()
        out.fill_(float("nan"))


@pytest.mark.parametrize("B,Hq,Hkv,n,kept,max_k,launches", [
    (8, 32, 32, 4096, [819] * 8, 819, 1), (8, 32, 32, 4096, [819] + [0] * 7, 819, 1),
    (8, 32, 32, 4096, [947, 0, 1, 31, 600, 0, 0, 33], 947, 1),
    (8, 32, 8, 5000, [4600, 0, 1, 31, 600, 4000, 0, 33], 4600, 1),   # groups: one round more
    (8, 32, 8, 6000, [5600, 0, 1, 31, 600, 4000, 0, 33], 5600, 2),
    (4, 32, 32, 4096, [3277, 200, 0, 200], 3277, 2),    # one long sequence: its batches over all warps
    (6, 40, 40, 2048, [1500, 50, 50, 0, 50, 1], 1500, 2),
    (1, 32, 32, 4096, [3277], 3277, 1), (2, 32, 32, 4096, [3277, 1], 3277, 1),
    (16, 32, 1, 7000, [6400] + [50] * 15, 6400, 1),     # two passes over the heads
    (4, 32, 8, 4096, [100] * 4, 4000, 1),               # an index width far above the counts
])
def test_form_by_index_width(H, B, Hq, Hkv, n, kept, max_k, launches):
    """Which widths take clusters per (sequence, KV head) (one launch) and which the even split and its merge (152 SMs):
    where the counts may differ, a single long sequence must not be left to a few CTAs."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes of 152 SMs")
    g = torch.Generator(device="cuda").manual_seed(max_k + B)
    K, V = (torch.randn(B, Hkv, n, 128, generator=g, device="cuda").half() for _ in range(2))
    q = torch.randn(B, Hq, 128, generator=g, device="cuda").half()
    desc = H.make_desc(q, K, V)
    idx = torch.full((B, max_k), -1, dtype=torch.int32, device="cuda")
    for b, m in enumerate(kept):
        idx[b, :m] = torch.randperm(n, generator=g, device="cuda")[:m].sort().values.int()
    count = torch.tensor(kept, dtype=torch.int32, device="cuda")
    out = torch.full((B, Hq, 128), float("nan"), device="cuda")
    ws = H.alloc_workspace(desc, 0, max_k)
    ws.fill_(0xFF)
    before = H.hill_kernel_launches()
    H.hill_gather_sparse_attn(desc, q, K, V, idx, count, max_k, out, ws)
    assert H.hill_kernel_launches() - before == launches
    H.hill_sync_status()
    ref = torch.zeros(B, Hq, 128, dtype=torch.float64, device="cuda")
    for b, m in enumerate(kept):
        t = idx[b, :m].long()
        for h in range(Hq if m else 0):
            g_ = h * Hkv // Hq
            p = torch.softmax(K[b, g_, t].double() @ q[b, h].double() / math.sqrt(128), 0)
            ref[b, h] = p @ V[b, g_, t].double()
    check_attn(out.cpu().numpy(), ref.cpu().numpy())
