"""The normalisation of the ATTN importance against float64: head counts that are not a multiple of the 8 taken at a
time or exceed the 32 held at a time, many partials per head (several warps per KV head), one and two kernels, ragged
and empty sequences; with the running importance and the selection that is fed by its digit counts.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# (B, H, Hkv, tokens of each sequence)
CASES = [
    (1, 1, 1, [1]),
    (2, 9, 3, [257, 0]),
    (1, 32, 1, [6000]),              # 1216 partials per head, combined in the one kernel
    (3, 8, 1, [30000, 16000, 1]),    # the same in two kernels
    (1, 71, 1, [8000]),              # and over three passes of heads
    (2, 20, 2, [5000, 40]),
    (2, 28, 4, [3001, 2999]),
    (2, 64, 8, [9000, 4097]),        # two rounds of 32 heads
    (1, 72, 8, [70001]),             # three, in two kernels
    (5, 40, 40, [700, 31, 32, 33, 640]),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"B{c[0]}H{c[1]}kv{c[2]}n{max(c[3])}")
def test_scores_and_selection(case):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    B, Hq, Hkv, lens = case
    n, G = max(lens), Hq // Hkv
    g = torch.Generator(device="cuda").manual_seed(n + Hq)
    K = torch.randn(B, Hkv, n, 128, generator=g, device="cuda").half()
    q = (3 * torch.randn(B, Hq, 128, generator=g, device="cuda")).half()
    accum = torch.rand(B, n, generator=g, device="cuda") * Hq / n
    before = accum.double()
    desc = H.make_desc(q, K)
    kept = [max(1, m // 5) if m else 0 for m in lens]
    dev = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")  # noqa: E731
    scores = torch.zeros(B, n, device="cuda")
    idx = torch.zeros(B, max(kept), dtype=torch.int32, device="cuda")
    count = torch.zeros(B, dtype=torch.int32, device="cuda")
    ws = H.alloc_workspace(desc, 0, max(kept))
    H.hill_evict_step(desc, q, K, None, dev(lens), dev(kept), max(kept), 0, accum, scores, idx, count, None, ws)
    H.hill_sync_status()
    assert count.tolist() == kept
    for b, m in enumerate(lens):
        z = torch.stack([K[b, h // G, :m].double() @ q[b, h].double() for h in range(Hq)]) / np.sqrt(128)
        ref = torch.softmax(z, -1).sum(0)
        # 32-bit logits of magnitude up to ~15: a few 2^-24 of them in the exponent, and as much in the sums
        assert torch.all((scores[b, :m].double() - ref).abs() <= 2e-5 * ref.clamp_min(1e-30)) or m == 0
        assert torch.all((accum[b, :m].double() - before[b, :m] - scores[b, :m].double()).abs() <= 1e-6)
        # the selection is exact on the kernel's own sums
        order = torch.sort(accum[b, :m], descending=True, stable=True).indices[:kept[b]]
        assert torch.equal(idx[b, :kept[b]].long(), order.sort().values)


@pytest.mark.parametrize("H_,Hkv", [(6, 3), (12, 3), (20, 20), (9, 3), (72, 9), (48, 2), (40, 8)])
def test_group_sums(H_, Hkv):
    """Per-KV-head importance for groups of 1, 2, 4, 8, 24 and odd sizes, head counts that are no multiple of 8."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    B, n, G, lens = 2, 700, H_ // Hkv, [700, 333]
    g = torch.Generator(device="cuda").manual_seed(H_)
    K = torch.randn(B, Hkv, n, 128, generator=g, device="cuda").half()
    q = (2 * torch.randn(B, H_, 128, generator=g, device="cuda")).half()
    desc = H.make_desc(q, K)
    dev = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")  # noqa: E731
    scores = torch.zeros(B, Hkv, n, device="cuda")
    idx = torch.zeros(B, Hkv, 70, dtype=torch.int32, device="cuda")
    count = torch.zeros(B, Hkv, dtype=torch.int32, device="cuda")
    H.hill_evict_step_kvh(desc, q, K, None, dev(lens), dev([70, 33]), 70, 0, None, scores, idx, count, None,
                          H.alloc_workspace(desc, 0, 70))
    H.hill_sync_status()
    for b, m in enumerate(lens):
        z = torch.stack([K[b, h // G, :m].double() @ q[b, h].double() for h in range(H_)]) / np.sqrt(128)
        ref = torch.softmax(z, -1).reshape(Hkv, G, m).sum(1)
        assert torch.all((scores[b, :, :m].double() - ref).abs() <= 2e-5 * ref)
        assert not scores[b, :, m:].any()


def _claims(ws, desc):
    """The counts of the eight claim counters (tag 0 once closed, count, a pad word) in a workspace that held 0x5A bytes
    before a hill_score call; None where nothing was claimed. The logits, which come first, are skipped: their lines are
    discarded from L2 and may read as anything."""
    start = -ws.data_ptr() % 256 + (4 * desc.batch * desc.num_q_heads * (-(-desc.capacity // 32) * 32) + 255) // 256 * 256
    rows = ws[start:start + (ws.numel() - start) // 256 * 256].view(torch.int32).view(-1, 64)
    filler = 0x5A5A5A5A
    head = rows[:, :32].view(-1, 8, 4)
    hit = (head[..., :2] == 0).all(-1).all(-1) & (head[..., 3] == filler).all(-1) & (rows[:, 32:] == filler).all(-1)
    assert int(hit.sum()) <= 1
    counts = head[hit][..., 2].flatten().tolist()
    return counts if counts and filler not in counts else None


@pytest.mark.parametrize("B,Hq,Hkv,n,launches", [
    (4, 32, 8, 10000, 2), (1, 32, 8, 65536, 2), (16, 32, 1, 4096, 2), (8, 32, 32, 8192, 2),   # up to two blocks per SM
    (1, 32, 1, 4096, 2), (2, 32, 1, 16000, 2),   # several rounds of partials per head
    (4, 32, 1, 16384, 3), (1, 32, 1, 65536, 3),  # the same on more than one block per SM
    (1, 32, 8, 80000, 3), (1, 32, 32, 80000, 3),
])
def test_launches_of_the_normalisation(B, Hq, Hkv, n, launches):
    """Which sizes combine the partials in a kernel of their own (152 SMs), and the scores of both forms at the sizes
    where they meet, in a cache that is filled and in one that is nearly empty."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes of 152 SMs")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    g = torch.Generator(device="cuda").manual_seed(n + Hkv)
    K = torch.randn(B, Hkv, n, 128, generator=g, device="cuda").half()
    q = (2 * torch.randn(B, Hq, 128, generator=g, device="cuda")).half()
    desc = H.make_desc(q, K)
    ws = H.alloc_workspace(desc, 0, 0)
    ws.fill_(0xFF)
    for m in (n, n // 10):
        scores = torch.zeros(B, n, device="cuda")
        before = H.hill_kernel_launches()
        H.hill_score(desc, q, K, torch.full((B,), m, dtype=torch.int32, device="cuda"), 0, scores, None, ws)
        assert H.hill_kernel_launches() - before == launches
        H.hill_sync_status()
        for b in (0, B - 1):
            z = torch.stack([K[b, h * Hkv // Hq, :m].double() @ q[b, h].double() for h in range(Hq)]) / np.sqrt(128)
            ref = torch.softmax(z, -1).sum(0)
            assert torch.all((scores[b, :m].double() - ref).abs() <= 2e-5 * ref)


@pytest.mark.parametrize("lens,claimed", [([8192] * 8, True), ([8192] * 7 + [8160], False), ([1000] * 8, False),
                                          ([65536] + [0] * 7, True), ([65504] + [0] * 7, False)])
def test_claims_by_the_tokens_present(lens, claimed):
    """A cache that could hold more than 512 MB of keys: the tail is claimed where the sequences in it do (65536 tokens
    of 32 heads), and not where they are short."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    cap = max(10000, max(lens) + 64)   # (more than two blocks of tokens per SM)
    K = torch.randn(len(lens), 32, cap, 128, dtype=torch.float16, device="cuda")
    q = torch.randn(len(lens), 32, 128, dtype=torch.float16, device="cuda")
    desc = H.make_desc(q, K)
    assert K.numel() * 2 >= 512 << 20
    ws = H.alloc_workspace(desc, 0, 0)
    ws.fill_(0x5A)
    scores = torch.zeros(len(lens), cap, device="cuda")
    H.hill_score(desc, q, K, torch.tensor(lens, dtype=torch.int32, device="cuda"), 0, scores, None, ws)
    H.hill_sync_status()
    counts = _claims(ws, desc)
    assert (counts is not None) == claimed
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = sum((m + 31) // 32 for m in lens)
    # every warp index claims each tile past the shares once, and then once more per CTA
    assert not claimed or counts == [tiles - sms * (tiles // 16 * 13 // sms) + sms] * 8


@pytest.mark.parametrize("B,Hq,Hkv,cap,claims", [(1, 32, 8, 131072, False), (4, 32, 16, 32768, False), (4, 40, 40, 32768, False),
                                                 (4, 32, 32, 12000, False), (4, 32, 1, 16384, False), (4, 32, 32, 32768, True)])
def test_workspace_without_claims(B, Hq, Hkv, cap, claims):
    """A layout that never claims holds one partial slot per scoring CTA (and warp share), as hill_score_noalloc
    documents it; one that may claim holds more."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    K = torch.zeros(1, 1, 1, 128, dtype=torch.float16, device="cuda").expand(B, Hkv, cap, 128)
    desc = H.make_desc(torch.zeros(B, Hq, 128, dtype=torch.float16, device="cuda"), K)
    attn = H.hill_workspace_bytes(desc, 0, 0) - H.hill_workspace_bytes(desc, 1, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = 8 // Hkv if Hkv <= 4 and Hq // Hkv >= 5 else 1
    up = lambda n: (n + 255) // 256 * 256  # noqa: E731
    tiles = (cap + 31) // 32
    bound = up(4 * B * Hq * tiles * 32) + up(8 * B * Hq * min(sms, B * tiles) * warps) + up(8 * B * Hq)
    assert (attn > bound) == claims


@pytest.mark.parametrize("lens,claimed", [
    ([8200] * 8, True), ([30000, 0, 1, 20000, 641, 16000, 33, 100], True), ([65537] + [0] * 7, True),
    ([0] * 7 + [66000], True), ([0, 31, 32, 33, 66000, 0, 7, 1], True), ([640, 641, 639, 7, 0, 0, 1500, 3], False),
])
@pytest.mark.parametrize("Hq,Hkv,dtype", [(32, 32, torch.float16), (64, 32, torch.bfloat16), (96, 32, torch.bfloat16),
                                          (24, 24, torch.bfloat16), (40, 20, torch.float16), (136, 17, torch.bfloat16)])
def test_claimed_tail_of_a_large_cache(Hq, Hkv, dtype, lens, claimed):
    """A cache large enough for the scoring kernel's tail to be claimed, full, ragged, with empty sequences anywhere and
    nearly empty; groups of 1 to 8, uneven heads per warp: right against float64, the same bits every time and in the
    fused step, and the workspace's counters say that tiles were claimed (from 512 MB of keys on: lengths are given for
    32 KV heads)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    lens = [-(-m * 32 // Hkv) for m in lens]
    B, G, cap = 8, Hq // Hkv, max(max(lens), 10000 * 32 // Hkv)
    g = torch.Generator(device="cuda").manual_seed(sum(lens) + Hq)
    K = torch.empty(B, Hkv, cap, 128, dtype=dtype, device="cuda")
    for b, m in enumerate(lens):
        K[b, :, :m] = torch.randn(Hkv, m, 128, generator=g, device="cuda").to(dtype)
        K[b, :, m:] = float("nan")
    q = (2 * torch.randn(B, Hq, 128, generator=g, device="cuda")).to(dtype)
    desc = H.make_desc(q, K)
    lens_t = torch.tensor(lens, dtype=torch.int32, device="cuda")
    kept = torch.tensor([min(m, 50) for m in lens], dtype=torch.int32, device="cuda")
    ws = H.alloc_workspace(desc, 0, 50)
    first = None
    for fill in (0, 0xFF, 0x5A):
        ws.fill_(fill)
        scores = torch.zeros(B, cap, device="cuda")
        H.hill_score(desc, q, K, lens_t, 0, scores, None, ws)
        H.hill_sync_status()
        assert first is None or torch.equal(scores, first)
        first = scores
    assert (_claims(ws, desc) is not None) == claimed
    accum, scores = torch.zeros(B, cap, device="cuda"), torch.zeros(B, cap, device="cuda")
    idx = torch.zeros(B, 50, dtype=torch.int32, device="cuda")
    H.hill_evict_step(desc, q, K, None, lens_t, kept, 50, 0, accum, scores, idx, torch.empty_like(kept), None, ws)
    H.hill_sync_status()
    assert torch.equal(scores, first) and torch.equal(accum, first)
    # and with sets of their own for the KV heads, whose importance adds up to the sequence's
    group = torch.zeros(B, Hkv, cap, device="cuda")
    H.hill_evict_step_kvh(desc, q, K, None, lens_t, kept, 50, 0, None, group,
                          torch.zeros(B, Hkv, 50, dtype=torch.int32, device="cuda"),
                          torch.zeros(B, Hkv, dtype=torch.int32, device="cuda"), None, ws)
    H.hill_sync_status()
    assert torch.all((group.double().sum(1) - first.double()).abs() <= 1e-5 * first.double())
    for b, m in enumerate(lens):
        assert not scores[b, m:].any()
        if m == 0:
            continue
        ref = torch.zeros(m, dtype=torch.float64, device="cuda")
        for h in range(Hq):
            ref += torch.softmax(K[b, h // G, :m].double() @ q[b, h].double() / np.sqrt(128), -1)
        assert torch.all((scores[b, :m].double() - ref).abs() <= 2e-5 * ref)
        order = torch.sort(scores[b, :m], descending=True, stable=True).indices[:min(m, 50)]
        assert torch.equal(idx[b, :min(m, 50)].long(), order.sort().values)


@pytest.mark.parametrize("Hq,Hkv,cap", [(32, 32, 24000), (48, 24, 32000)])
@pytest.mark.parametrize("fused", [False, True])
def test_claims_in_a_replayed_graph(fused, Hq, Hkv, cap):
    """A call whose tail is claimed, captured once and replayed over lengths and queries that change between the
    replays, the first sequence, all of them or none empty: every replay gives the bits of an eager call on a workspace
    of its own."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill as H
    build.build()
    B, max_k = 4, 64
    g = torch.Generator(device="cuda").manual_seed(cap)
    K = torch.randn(B, Hkv, cap, 128, generator=g, device="cuda").bfloat16()
    q = torch.empty(B, Hq, 128, dtype=torch.bfloat16, device="cuda")
    desc = H.make_desc(q, K)
    lens = torch.full((B,), cap, dtype=torch.int32, device="cuda")
    k = torch.full((B,), max_k, dtype=torch.int32, device="cuda")

    def buffers():
        ws = H.alloc_workspace(desc, 0, max_k)
        ws.fill_(0x5A)
        return {"ws": ws, "scores": torch.zeros(B, cap, device="cuda"), "accum": torch.zeros(B, cap, device="cuda"),
                "idx": torch.zeros(B, max_k, dtype=torch.int32, device="cuda"),
                "count": torch.zeros(B, dtype=torch.int32, device="cuda")}

    def call(y):
        if fused:
            H.hill_evict_step(desc, q, K, None, lens, k, max_k, 0, y["accum"], y["scores"], y["idx"], y["count"], None,
                              y["ws"])
        else:
            H.hill_score(desc, q, K, lens, 0, y["scores"], y["accum"], y["ws"])

    call(buffers())   # (kernels loaded)
    H.hill_sync_status()
    y = buffers()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(y)
    empty, full = [0] * B, [cap] * B
    first = [0] + [cap] * (B - 1)
    for step, n in enumerate([full, first, full, first, first, empty, full, [cap, 0, cap - 33, cap], [0, 0, 0, cap], full]):
        q.copy_(2 * torch.randn(q.shape, generator=g, device="cuda"))
        lens.copy_(torch.tensor(n, dtype=torch.int32))
        want = buffers()
        for o in ("scores", "accum"):
            want[o].copy_(y[o])
        call(want)
        graph.replay()
        H.hill_sync_status()
        for o in ("scores", "accum", "idx", "count"):
            assert torch.equal(y[o], want[o]), f"{o} of replay {step}, lengths {n}"
