"""The selection kernel alone against the oracle's sort, bit for bit: row lengths at the edges of a CTA's and a
cluster's chunks, keys whose crossing bin fits the exchanged list and keys whose crossing bin does not (shared leading
digits, heavy ties), every budget edge, with and without a pinned window and hit counts.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_18750_gb300 import build, hill
    build.build()
    hill.load()
    return hill


def _keys(kind, rows, cap, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(rows, cap, generator=g)
    if kind == "narrow":     # one leading digit for every key: the crossing bin is the whole row
        x = 1.0 + 0.249 * torch.rand(rows, cap, generator=g)
    elif kind == "ties":     # few values, both signs, both zeros
        x = torch.randint(-3, 4, (rows, cap), generator=g).float() * 0.5 * torch.sign(x)
    elif kind == "flat":
        x = torch.full((rows, cap), -0.0)
    elif kind == "bins":     # 512 tokens in [1, 1.25), spread over the row, the rest far below
        x = -x.abs()
        at = torch.linspace(0, cap - 1, min(cap, 512)).long()
        x[:, at] = 1.0 + 0.2 * torch.rand(rows, len(at), generator=g)
    return x


@pytest.mark.parametrize("kind", ["random", "narrow", "ties", "flat", "bins"])
@pytest.mark.parametrize("cap", [1, 33, 1024, 1025, 4159, 8193, 16384, 16385, 32831, 65537, 131135])
def test_select_matches_sort(H, oracle_mod, cap, kind):
    rows = 5
    x = _keys(kind, rows, cap, cap)
    lens = [cap, cap, max(cap - 1, 0), cap // 2, cap]
    budgets = [max(1, cap // 5), cap - 1, 1, cap // 4, min(cap, 256)]
    K = torch.zeros(rows, 1, 1, 128, dtype=torch.float16, device="cuda").expand(rows, 1, cap, 128)
    desc = H.make_desc(torch.zeros(rows, 1, 128, dtype=torch.float16, device="cuda"), K)
    dev = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")  # noqa: E731
    for recent, hits in ((0, None), (70, torch.randint(0, 65536, (rows, cap), generator=torch.Generator().manual_seed(3)))):
        max_k = max(budgets) + recent
        idx = torch.full((rows, max_k), -9, dtype=torch.int32, device="cuda")
        count = torch.full((rows,), -9, dtype=torch.int32, device="cuda")
        h0 = None if hits is None else hits.numpy().astype(np.uint16)
        hd = None if h0 is None else torch.from_numpy(h0.view(np.int16).copy()).cuda()
        H.hill_topk_select_bkp(desc, x.cuda(), dev(lens), dev(budgets), recent, max_k, idx, count, hd)
        H.hill_sync_status()
        want_i, want_c, rc, want_h = oracle_mod.bkp_select(x.numpy(), lens, budgets, recent, max_k, h0)
        assert np.array_equal(count.cpu().numpy(), want_c) and np.array_equal(idx.cpu().numpy(), want_i)
        if h0 is not None:
            assert np.array_equal(hd.cpu().numpy().view(np.uint16), want_h)


def test_select_longest_row(H, oracle_mod):
    """The longest row the selection takes (48128 keys in each of 8 CTAs); one more is refused."""
    cap = 8 * 48128
    q = torch.zeros(1, 1, 128, dtype=torch.float16, device="cuda")
    K = torch.zeros(1, 1, 1, 128, dtype=torch.float16, device="cuda")
    desc = H.make_desc(q, K.expand(1, 1, cap, 128))
    one = lambda v: torch.tensor([v], dtype=torch.int32, device="cuda")  # noqa: E731
    idx, count = torch.zeros(1, 40000, dtype=torch.int32, device="cuda"), one(0)
    for kind in ("random", "narrow"):
        x = _keys(kind, 1, cap, 1)
        H.hill_topk_select(desc, x.cuda(), one(cap), one(40000), 40000, idx, count)
        H.hill_sync_status()
        want_i, want_c, _ = oracle_mod.topk(x.numpy(), [cap], [40000], 40000)
        assert np.array_equal(idx.cpu().numpy(), want_i) and int(count) == want_c[0]
    desc = H.make_desc(q, K.expand(1, 1, cap + 1, 128))
    with pytest.raises(H.HillError):
        H.hill_topk_select(desc, torch.zeros(1, cap + 1, device="cuda"), one(cap), one(1), 1, idx, count)


@pytest.mark.parametrize("kind", ["random", "narrow", "ties", "flat", "bins"])
@pytest.mark.parametrize("cap", [8193, 16385, 40002, 131135])
def test_short_rows_of_a_large_cache(H, oracle_mod, cap, kind):
    """Rows at and around the 8192 ranked tokens up to which a cluster's first CTA works alone, for every place of a
    row's first key in its 16 bytes (odd capacities), beside rows that all CTAs search; budgets at both ends."""
    lens = [1, 2, 33, 4096, 8188, 8189, 8190, 8191, 8192, 8193, 8000, cap]
    budgets = [1, 1, 32, 64, 8187, 1, 819, 65, 4096, 700, 8000, 1000]
    rows = len(lens)
    x = _keys(kind, rows, cap, cap)
    K = torch.zeros(rows, 1, 1, 128, dtype=torch.float16, device="cuda").expand(rows, 1, cap, 128)
    desc = H.make_desc(torch.zeros(rows, 1, 128, dtype=torch.float16, device="cuda"), K)
    dev = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")  # noqa: E731
    for recent, hits in ((0, None), (3, torch.randint(0, 65536, (rows, cap), generator=torch.Generator().manual_seed(5)))):
        max_k = max(budgets) + recent
        idx = torch.full((rows, max_k), -9, dtype=torch.int32, device="cuda")
        count = torch.full((rows,), -9, dtype=torch.int32, device="cuda")
        h0 = None if hits is None else hits.numpy().astype(np.uint16)
        hd = None if h0 is None else torch.from_numpy(h0.view(np.int16).copy()).cuda()
        H.hill_topk_select_bkp(desc, x.cuda(), dev(lens), dev(budgets), recent, max_k, idx, count, hd)
        H.hill_sync_status()
        want_i, want_c, rc, want_h = oracle_mod.bkp_select(x.numpy(), lens, budgets, recent, max_k, h0)
        assert np.array_equal(count.cpu().numpy(), want_c) and np.array_equal(idx.cpu().numpy(), want_i)
        if h0 is not None:
            assert np.array_equal(hd.cpu().numpy().view(np.uint16), want_h)


@pytest.mark.parametrize("cap", [16385, 70001])
def test_short_rows_counted_by_the_normalisation(H, cap):
    """The same with the leading digits counted by the ATTN normalisation."""
    lens, g = [1000, 8191, 8192, 8193, 1, cap], torch.Generator(device="cuda").manual_seed(cap)
    K = torch.randn(len(lens), 2, cap, 128, generator=g, device="cuda").half()
    q = torch.randn(len(lens), 4, 128, generator=g, device="cuda").half()
    kept = [max(1, m // 7) for m in lens]
    dev = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")  # noqa: E731
    scores = torch.zeros(len(lens), cap, device="cuda")
    idx = torch.zeros(len(lens), max(kept), dtype=torch.int32, device="cuda")
    count = torch.zeros(len(lens), dtype=torch.int32, device="cuda")
    desc = H.make_desc(q, K)
    H.hill_evict_step(desc, q, K, None, dev(lens), dev(kept), max(kept), 0, None, scores, idx, count, None,
                      H.alloc_workspace(desc, 0, max(kept)))
    H.hill_sync_status()
    assert count.tolist() == kept
    for b, m in enumerate(lens):
        order = torch.sort(scores[b, :m], descending=True, stable=True).indices[:kept[b]]
        assert torch.equal(idx[b, :kept[b]].long(), order.sort().values)
        assert torch.all(idx[b, kept[b]:] == -1)
