"""The selection of small stores straight from the slab: sizes around its keys a
thread, every list length, ties across the k-th score, scopes that leave too
few candidates, deleted chunks; against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from _parity import assert_retrieval_parity, assert_scoped_parity, gpu_retrieve, oracle_retrieve

pytestmark = pytest.mark.gpu


def _cut(n, **kw):
    base = synth.workload(2, scale=1 / 64)
    e = int(base.row_ptr[n])
    keep = base.col[:e] < n
    deg = np.add.reduceat(keep, base.row_ptr[:n].astype(np.int64))
    return dataclasses.replace(base, emb=base.emb[:n], component=base.component[:n],
                               page_of={"clustered": base.page_of["clustered"][:n]},
                               row_ptr=np.concatenate([[0], np.cumsum(deg)]).astype(np.int64),
                               col=base.col[:e][keep], aff=base.aff[:e][keep], **kw)


@pytest.mark.parametrize("n,B,hops,k", [(64, 3, 1, 64), (1023, 1, 0, 1), (1024, 33, 2, 64),
                                        (1025, 5, 1, 7), (2049, 256, 1, 32), (4096, 300, 3, 16),
                                        (4097, 17, 0, 64), (8192, 129, 2, 33), (8193, 20, 1, 8)])
def test_sizes(n, B, hops, k):
    wl = _cut(n, hops=hops, k=k)
    q = np.concatenate([wl.queries, wl.queries])[:B]
    _, got = gpu_retrieve(wl, "clustered", queries=q)
    assert_retrieval_parity(wl, "clustered", got, oracle_retrieve(wl, "clustered", queries=q))


@pytest.mark.parametrize("hops", [0, 1])
def test_ties_take_the_lowest_ids(hops):
    """3000 equal embeddings on a ring: all scores equal."""
    n = 3000
    wl = _cut(n, hops=hops, k=50)
    wl = dataclasses.replace(wl, emb=np.repeat(wl.emb[:1], n, axis=0),
                             row_ptr=np.arange(n + 1, dtype=np.int64),
                             col=((np.arange(n) + 1) % n).astype(np.int32),
                             aff=np.zeros(n, np.float32))
    _, got = gpu_retrieve(wl, "clustered", queries=wl.queries[:5])
    assert (np.sort(got["ids"], axis=1) == np.arange(50)).all()


@pytest.mark.parametrize("hops,by_time", [(0, False), (2, True)])
def test_scope_and_deletions(hops, by_time):
    import torch
    from _parity import gpu_store
    wl = _cut(3001, hops=hops, k=20)
    rng = np.random.default_rng(5)
    ns_of = rng.integers(0, 4, wl.n).astype(np.int32)
    ns_of[rng.choice(wl.n, 7, replace=False)] = 9          # fewer than k
    q_ns = rng.choice([0, 1, 2, 9, 77], 40).astype(np.int32)
    dead = np.zeros(wl.n, bool)
    dead[rng.choice(wl.n, 300, replace=False)] = True
    store = gpu_store(wl, "clustered")
    store.set_namespace(0, torch.from_numpy(ns_of).cuda())
    store.delete(torch.from_numpy(np.nonzero(dead)[0]).cuda())
    rp, col, aff = oracle.drop_dead(wl.row_ptr, wl.col, wl.aff, dead)
    q = wl.queries[:40]
    out = store.retrieve(torch.from_numpy(np.ascontiguousarray(q).view(np.int16)).cuda(), wl.k,
                         wl.alpha, hops, q_ns=torch.from_numpy(q_ns).cuda(), sort_by_time=by_time)
    store.sync()
    got = dict(zip(("ids", "scores", "page_ids", "n_pages"), (t.cpu().numpy() for t in out)))
    ref = oracle.retrieve(wl.emb, q, rp, col, oracle.row_softmax(rp, aff), tau=wl.tau,
                          alpha=wl.alpha, hops=hops, k=wl.k, page_of=wl.page_of["clustered"],
                          want_final=True, ns_of=ns_of, q_ns=q_ns, sort_by_time=by_time, dead=dead)
    assert_scoped_parity(wl, "clustered", got, ref, ns_of, q_ns, by_time)
    assert (got["ids"][q_ns == 77] == -1).all()
