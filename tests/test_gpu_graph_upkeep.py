"""Deletion's two-pass compaction at the edges of its words and tiles, and the
hub plan with more source windows than a warp has lanes.  Against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from _parity import assert_retrieval_parity, gpu_retrieve, gpu_store, oracle_retrieve

pytestmark = pytest.mark.gpu


def _check_graph(store, rp, col, aff):
    g_rp, g_col, g_aff, g_w = (t.cpu().numpy() for t in store.export_csr())
    assert (g_rp == rp).all() and (g_col == col).all() and (g_aff == aff).all()
    np.testing.assert_allclose(g_w, oracle.row_softmax(rp, aff), rtol=2e-5, atol=0)


@pytest.mark.parametrize("n,deg,gone", [
    (64, 2, 1),             # 128 edges: a few words of one tile
    (67, 31, 5),            # rows that cross words
    (517, 8, 33),           # 4136 edges: one tile and a bit
    (4096, 33, 700),        # many tiles, rows of an odd length
    (512, 8, 511),          # all but one: nothing left but empty rows
])
def test_deletions_in_turn(n, deg, gone):
    """Three deletions in a row (the second repeats part of the first), then a
    retrieval over the graph that is left."""
    import torch
    base = synth.workload(2, scale=1 / 64)
    rng = np.random.default_rng(n + deg)
    col = np.stack([np.sort(rng.choice(n - 1, deg, replace=False)) for _ in range(n)])
    col += col >= np.arange(n)[:, None]
    # chunk 3 is a hub: every other row that lacks it links to it
    for i in range(n):
        if i != 3 and 3 not in col[i]:
            col[i, 0] = 3
            col[i].sort()
    aff = rng.normal(0, 1, (n, deg)).astype(np.float32)
    wl = dataclasses.replace(base, emb=base.emb[:n], hops=2, k=1, queries=base.queries[:8],
                             row_ptr=np.arange(0, n * deg + 1, deg, dtype=np.int64),
                             col=col.astype(np.int32).ravel(), aff=aff.ravel(),
                             page_of={"clustered": base.page_of["clustered"][:n]},
                             component=base.component[:n])
    store = gpu_store(wl, "clustered")
    rp, c, a = wl.row_ptr, wl.col, wl.aff
    dead = np.zeros(n, bool)
    victims = rng.permutation(n)[:gone]
    for part in (victims[:gone // 2 + 1], victims[gone // 3:], np.array([3])):
        dead[part] = True
        if dead.all():
            break
        store.delete(torch.from_numpy(part.astype(np.int64)).cuda())
        rp, c, a = oracle.drop_dead(rp, c, a, dead)
        _check_graph(store, rp, c, a)
    if dead.sum() <= n - 2:
        q = torch.from_numpy(np.ascontiguousarray(wl.queries).view(np.int16)).cuda()
        ids, sc, pg, npg = store.retrieve(q, 1, wl.alpha, 2)
        store.sync()
        ref = oracle.retrieve(wl.emb, wl.queries, rp, c, oracle.row_softmax(rp, a), tau=wl.tau,
                              alpha=wl.alpha, hops=2, k=1, page_of=wl.page_of["clustered"],
                              want_final=True, dead=dead)
        assert_retrieval_parity(wl, "clustered", dict(ids=ids.cpu().numpy(), scores=sc.cpu().numpy(),
                                                      page_ids=pg.cpu().numpy(),
                                                      n_pages=npg.cpu().numpy()), ref)


@pytest.mark.parametrize("win,seg,split", [(97, 64, 100), (500, 512, 256), (16384, 1, 300)])
def test_hub_plan_shapes(win, seg, split, monkeypatch):
    """169 windows (several rounds of a warp's lanes), one-edge segments, and
    the ordinary ones: two hops through the plan."""
    monkeypatch.setenv("AKASHIC_REACH", "0")
    monkeypatch.setenv("AKASHIC_WIN_ROWS", str(win))
    monkeypatch.setenv("AKASHIC_SEG_LEN", str(seg))
    monkeypatch.setenv("AKASHIC_SPLIT_T", str(split))
    wl = synth.workload(2, scale=1 / 64)
    q = wl.queries[:40]
    _, got = gpu_retrieve(wl, "random", queries=q)
    assert_retrieval_parity(wl, "random", got, oracle_retrieve(wl, "random", queries=q))
