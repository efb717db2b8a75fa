"""The relation update's graph insert where its pieces can go wrong: the sorts
around the size that one launch takes, edges moved across tiles with and without
cuts in them, targets chosen by every new chunk, new chunks in page order, with
and without reciprocal edges; the whole CSR against the oracle's neighbours, then
two hops over it (the in-edges)."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from _parity import assert_retrieval_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,new,M,recip,paged", [
    (70, 1, 1, True, False),
    (300, 64, 32, True, True),        # 2048 pairs: the last that one launch sorts
    (300, 65, 32, True, True),        # 2080
    (2050, 7, 64, True, False),
    (2050, 200, 3, False, True),
    (16384, 33, 16, True, True),      # 2^19 old edges: many tiles without a cut
    (5000, 700, 8, True, True),
])
def test_insert(n, new, M, recip, paged):
    import torch
    from paper_2607_05708_gb300 import MemStore
    base = synth.workload(2, scale=1 / 64)
    rng = np.random.default_rng(n + new)
    emb = base.emb[:n]
    if n <= 300:       # one component: all new chunks choose among the same targets
        emb = np.ascontiguousarray(base.emb[np.argsort(base.component, kind="stable")][:n])
    rp, col, aff = base.row_ptr[:n + 1], base.col, base.aff
    e = int(rp[-1])
    keep = col[:e] < n
    deg = np.add.reduceat(keep, rp[:-1].astype(np.int64))
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    col, aff = col[:e][keep], aff[:e][keep]
    store = MemStore.from_arrays(emb, base.page_of["clustered"][:n], rp, col, aff,
                                 capacity=n + new, temperature=base.tau)
    more = synth.bf16_to_f32(emb[rng.integers(0, n, new)])
    more = synth.to_bf16(more + rng.normal(0, 0.004, more.shape).astype(np.float32))
    pages = (rng.permutation(new) // 4 + 10 ** 4).astype(np.int32)
    first = store.append_chunks(torch.from_numpy(more.view(np.int16)).cuda(),
                                torch.from_numpy(pages).cuda() if paged else None)
    store.update_relations(first, new, M, recip)
    g_rp, g_col, g_aff, g_w = (t.cpu().numpy() for t in store.export_csr())
    # the new rows: the M prior chunks of largest fp64 cosine (near-ties may swap)
    cos = synth.bf16_to_f32(more).astype(np.float64) @ synth.bf16_to_f32(emb).astype(np.float64).T
    nbr = np.empty((new, M), np.int64)
    for a in range(new):
        nbr[a] = g_col[g_rp[n + a]:g_rp[n + a + 1]]
        kth = np.sort(cos[a])[-M]
        assert len(set(nbr[a])) == M and (cos[a][nbr[a]] >= kth - 1e-4).all()
        # 10 times an fp32 sum of products whose parts reach 1, one truncation a
        # 16-wide MMA step: 10 * (dim / 16) * 2^-23 (dim 768: 5.7e-5)
        np.testing.assert_allclose(g_aff[g_rp[n + a]:g_rp[n + a + 1]], 10 * cos[a][nbr[a]],
                                   atol=10 * emb.shape[1] / 16 * 2.0 ** -23, rtol=0)
    # the whole CSR from those choices
    rows = [(col[rp[j]:rp[j + 1]].tolist(), aff[rp[j]:rp[j + 1]].tolist()) for j in range(n)]
    logit = {(a, j): g_aff[g_rp[n + a] + t] for a in range(new) for t, j in enumerate(nbr[a])}
    if recip:
        for a in range(new):
            for j in nbr[a]:
                rows[j][0].append(n + a)
                rows[j][1].append(logit[a, j])
    for a in range(new):
        rows.append((nbr[a].tolist(), [logit[a, j] for j in nbr[a]]))
    want = np.concatenate([[0], np.cumsum([len(r[0]) for r in rows])])
    assert (g_rp == want).all()
    assert (g_col == np.concatenate([r[0] for r in rows])).all()
    assert (g_aff == np.concatenate([np.asarray(r[1], np.float32) for r in rows])).all()
    np.testing.assert_allclose(g_w, oracle.row_softmax(g_rp, g_aff), rtol=2e-5, atol=0)
    # the transpose: two hops over it
    both = np.concatenate([emb, more])
    page = store.export_pages().cpu().numpy()
    wl = dataclasses.replace(base, emb=both, row_ptr=g_rp, col=g_col, aff=g_aff, hops=2, k=10,
                             page_of={"p": page})
    q = base.queries[:20]
    out = store.retrieve(torch.from_numpy(np.ascontiguousarray(q).view(np.int16)).cuda(), 10,
                         wl.alpha, 2)
    store.sync()
    got = dict(zip(("ids", "scores", "page_ids", "n_pages"), (t.cpu().numpy() for t in out)))
    ref = oracle.retrieve(both, q, g_rp, g_col, oracle.row_softmax(g_rp, g_aff), tau=base.tau,
                          alpha=wl.alpha, hops=2, k=10, page_of=page, want_final=True)
    assert_retrieval_parity(wl, "p", got, ref)


@pytest.mark.parametrize("n,new,M,recip", [
    (2000, 140_000, 2, True),     # pairs in the large sort, new rows in the small, one scratch
    (64, 100_000, 64, True),      # every new chunk chooses every old one
    (3, 5001, 3, False),
])
def test_many_new_chunks_of_few_targets(n, new, M, recip):
    import torch
    from paper_2607_05708_gb300 import MemStore
    dim = 64
    rng = np.random.default_rng(7)
    emb = rng.normal(0, 1, (n + new, dim)).astype(np.float32)
    emb = synth.to_bf16(emb / np.linalg.norm(emb, axis=1, keepdims=True))
    dev = torch.from_numpy(emb.view(np.int16)).cuda()
    store = MemStore(dim, n + new, chunks_per_page=32, relation_scale=10.0)
    store.append_chunks(dev[:n])
    store.update_relations(1, n - 1, 1, True)           # some old edges to move
    old_rp, old_col, old_aff, _ = (t.cpu().numpy() for t in store.export_csr())
    pages = torch.from_numpy((rng.permutation(new) // 8 + 1000).astype(np.int32)).cuda()
    first = store.append_chunks(dev[n:], pages)         # (rows in another order than IDs)
    assert first == n
    store.set_profiling(True)
    store.update_relations(n, new, M, recip)
    # 12.8 million edges placed, sorted and moved: a few ms, seconds where a place
    # costs a scan of all the new chunks that chose its target
    assert store.phase_times()["transpose"][0] < 50
    store.set_profiling(False)
    rp, col, aff, w = (t.cpu().numpy() for t in store.export_csr())
    nbr, logit = col[rp[n]:].reshape(new, M), aff[rp[n]:].reshape(new, M)
    assert (nbr < n).all() and (np.diff(nbr, axis=1) > 0).all()
    # the old rows: their old edges, then the new chunks that chose them, ascending
    tgt, src = nbr.ravel(), np.repeat(np.arange(n, n + new), M)
    order = np.argsort(tgt, kind="stable") if recip else np.empty(0, np.int64)
    rows = np.concatenate([np.repeat(np.arange(n), np.diff(old_rp[:n + 1])), tgt[order]])
    at = np.argsort(rows, kind="stable")
    assert (rp[:n + 1] == np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))])).all()
    assert (col[:rp[n]] == np.concatenate([old_col, src[order]])[at]).all()
    assert (aff[:rp[n]] == np.concatenate([old_aff, logit.ravel()[order]])[at]).all()
    np.testing.assert_allclose(w, oracle.row_softmax(rp, aff), rtol=2e-5, atol=0)
    # the transpose: one hop over it
    k, q, page = 10, emb[:9], store.export_pages().cpu().numpy()
    out = store.retrieve(dev[:9], k, 0.5, 1)
    store.sync()
    got = dict(zip(("ids", "scores", "page_ids", "n_pages"), (t.cpu().numpy() for t in out)))
    ref = oracle.retrieve(emb, q, rp, col, oracle.row_softmax(rp, aff), tau=dim ** -0.5, alpha=0.5,
                          hops=1, k=k, page_of=page, want_final=True)
    wl = dataclasses.replace(synth.workload(2, scale=1 / 64), emb=emb, hops=1, k=k,
                             row_ptr=rp, col=col, aff=aff, page_of={"p": page})
    assert_retrieval_parity(wl, "p", got, ref)


def test_refused_updates_say_why_and_change_nothing():
    """Rows that have out-edges, and a chunk that an edge points at already."""
    import torch
    from paper_2607_05708_gb300 import AkashicError, MemStore
    rng = np.random.default_rng(2)
    emb = torch.from_numpy(synth.to_bf16(rng.normal(0, 0.1, (300, 64)).astype(np.float32))
                           .view(np.int16)).cuda()
    st = MemStore(64, 300, chunks_per_page=16)
    st.append_chunks(emb[:200])
    st.update_relations(100, 100, 4, True)
    rp = torch.zeros(51, dtype=torch.int64, device="cuda")
    rp[10:] = 1                                          # chunk 209 links to 220
    st.append_chunks(emb[200:250], None, rp, torch.tensor([220], dtype=torch.int32, device="cuda"),
                     torch.ones(1, device="cuda"))
    before = [t.cpu().numpy() for t in st.export_csr()]
    for first, n, code, why in ((150, 20, "EINVAL", "already have out-edges"),
                                (200, 50, "EINVAL", "already have out-edges"),
                                (210, 40, "EDEVICE", "update")):
        with pytest.raises(AkashicError, match=why) as e:
            st.update_relations(first, n, 4, True)
        assert e.value.code == code
        for a, b in zip(st.export_csr(), before):
            assert (a.cpu().numpy() == b).all()
    st.sync()                                            # nothing is left in the status word
    st.update_relations(221, 29, 4, True)
