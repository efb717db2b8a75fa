"""The ordered compactions past the tiles whose counts are added up one by one:
4.3 million chunks with 17.2 million edges.  The hub plan and the kept lists against
a store that has neither, the deletion's lists against the same deletion in torch,
the compaction's directory against its definition."""
import pytest

from test_gpu_out_of_memory import _store

pytestmark = pytest.mark.gpu


def test_lists_of_many_tiles(monkeypatch):
    import torch
    n, links = 4_300_000, 4                      # 4200 tiles of rows, 4200 of edges
    st, emb = _store(n, 0, links=links)
    monkeypatch.setenv("AKASHIC_SPLIT_T", str(1 << 40))
    monkeypatch.setenv("AKASHIC_HOP_PRUNE", "0")
    plain, _ = _store(n, 0, links=links)
    q = emb[::100_000][:20].contiguous()

    def same(hops):
        a, b = st.retrieve(q, 10, 0.5, hops), plain.retrieve(q, 10, 0.5, hops)
        st.sync()
        plain.sync()
        hit = a[0] == b[0]
        assert hit.float().mean() > 0.98
        # fp32 sums of up to 10^6 in-edges in another order
        assert ((a[1] - b[1]).abs() <= 2e-4 * b[1])[hit].all()

    same(1)
    rp, col, aff, _ = st.export_csr()
    # three quarters of every 1000th page and some chunks elsewhere
    page = torch.arange(0, n // 64, 1000, device="cuda")
    gone = (page[:, None] * 64 + torch.arange(48, device="cuda")).flatten()
    gone = torch.cat([gone, torch.arange(7, n, 99_991, device="cuda")]).unique()
    for s in (st, plain):
        s.delete(gone)
    dead = torch.zeros(n, dtype=torch.bool, device="cuda")
    dead[gone] = True
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    keep = ~dead[rows] & ~dead[col.long()]
    g_rp, g_col, g_aff, _ = st.export_csr()
    want = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    want[1:] = torch.bincount(rows[keep], minlength=n).cumsum(0)
    assert torch.equal(g_rp, want)
    assert torch.equal(g_col, col[keep]) and torch.equal(g_aff, aff[keep])
    same(1)
    # the pages three quarters gone are packed anew, in the order of their chunks
    before = st.export_pages()
    bad = torch.bincount(before[gone].long(), minlength=n // 64 + 1) >= 48
    assert st.compact_pages(0.75, 0.7) == int(bad.sum())
    moved = torch.nonzero(bad[before.long()] & ~dead).flatten()
    after = before.clone()
    after[moved] = int(before.max()) + 1 + (torch.arange(moved.numel(), device="cuda") // 64).int()
    got = st.export_pages()
    assert torch.equal(got[~dead], after[~dead])
