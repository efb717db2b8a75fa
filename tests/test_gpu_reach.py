"""Two to four hops from reach coefficients, in fp32 (batches of at most 32
queries) or on the tensor cores (33 to 64 queries, or three hops and more): the
path is taken once the hops have run often enough on one graph, selects what
the hops select, and its scores agree with theirs within the bound below; a
graph whose candidates do not suffice goes through the hops."""
import dataclasses

import numpy as np
import pytest

import synth
from _parity import assert_retrieval_parity, gpu_retrieve, gpu_store, oracle_retrieve

pytestmark = pytest.mark.gpu

# fp32: sums of non-negative terms in two orders, at most a few hundred
# roundings on any path (a warp's rows, the warps, the CTAs; a hop's segments),
# 2^-24 each.  Tensor cores: split-bf16 products of u - u_min, each within
# 3 * 2^-16 = 4.6e-5, and u - u_min is at most 1 - exp(-2 tau |q| |e|) = 6% of u
# here (dim 1024): 2.9e-6 of the sum.
REL = 1e-5


def _launches(store, wl, q):
    store.set_profiling(True)
    store.phase_times()
    _, out = gpu_retrieve(wl, "clustered", store=store, queries=q)
    ph = store.phase_times()
    store.set_profiling(False)
    return out, ph["last_hop"][1]


@pytest.mark.parametrize("B,hops,spread,same", [
    (48, 2, 1.0, True), (100, 3, 2.0, True), (48, 4, 1.0, True),   # too sharp for 16-bit pairs
    (48, 2, 0.375, False), (100, 3, 0.25, False),
])
def test_sharp_temperatures_keep_the_hops_precision(B, hops, spread, same, monkeypatch):
    """Scores between exp(-spread) and 1: with a wide spread the tensor-core pass
    would be less exact than the hops, so they run and give their own bits; below
    the limit (0.375) the candidates are used."""
    import torch
    from paper_2607_05708_gb300 import MemStore
    wl = synth.workload(2, scale=1 / 64)
    norm = lambda x: np.linalg.norm(synth.bf16_to_f32(x), axis=1).max()
    tau = 0.999 * spread / (2 * norm(wl.queries[:B]) * norm(wl.emb))
    q = torch.from_numpy(np.ascontiguousarray(wl.queries[:B]).view(np.int16)).cuda()
    out = []
    for reach in ("0", "1"):
        monkeypatch.setenv("AKASHIC_REACH", reach)
        store = MemStore.from_arrays(wl.emb, wl.page_of["clustered"], wl.row_ptr, wl.col, wl.aff,
                                     temperature=tau)
        for _ in range(12):
            got = store.retrieve(q, 4, 0.5, hops)
        store.sync()
        out.append([t.cpu().numpy() for t in got])
    (ids, scores, _, _), (ids0, scores0, _, _) = out[1], out[0]
    assert ((ids == ids0).all() and (scores == scores0).all()) == same
    hit = ids == ids0
    # the products' 4.6e-5 of the part above the smallest score (see REL), and the
    # hops' and the candidates' sums
    np.testing.assert_allclose(scores[hit], scores0[hit], atol=0,
                               rtol=REL + 4.6e-5 * (1 - np.exp(-spread)) * (not same))


@pytest.mark.parametrize("n,B,hops,k", [
    (16384, 1, 2, 32),          # one column tile of 8
    (16383, 9, 2, 8),           # 16 columns, ragged rows
    (16384, 33, 2, 32),         # two tiles of 32
    (9001, 64, 3, 16),
    (16384, 200, 3, 64),        # both halves of the candidates
    (16001, 256, 4, 5),
])
def test_equals_the_hops(n, B, hops, k, monkeypatch):
    base = synth.workload(2, scale=1 / 64)
    rp = base.row_ptr[:n + 1]
    keep = base.col[:rp[-1]] < n
    new_rp = np.concatenate([[0], np.cumsum(np.add.reduceat(keep, rp[:-1].astype(np.int64)))])
    wl = dataclasses.replace(base, emb=base.emb[:n], row_ptr=new_rp.astype(np.int64),
                             col=base.col[:rp[-1]][keep], aff=base.aff[:rp[-1]][keep],
                             page_of={"clustered": base.page_of["clustered"][:n]},
                             component=base.component[:n], hops=hops, k=k)
    q = wl.queries[:B]
    monkeypatch.setenv("AKASHIC_REACH", "0")
    _, ref = gpu_retrieve(wl, "clustered", queries=q)
    monkeypatch.setenv("AKASHIC_REACH", "1")
    store = gpu_store(wl, "clustered")
    for _ in range(12):                      # the hops, until the coefficients pay
        got, launches = _launches(store, wl, q)
    assert launches == (5 if B <= 32 else 4), launches   # the candidates' and the last hop's
    hit = got["ids"] == ref["ids"]
    assert hit.mean() > 0.99
    np.testing.assert_allclose(got["scores"][hit], ref["scores"][hit], rtol=REL, atol=0)
    assert_retrieval_parity(wl, "clustered", got, oracle_retrieve(wl, "clustered", queries=q))
    # a change of the graph starts over with the hops
    import torch
    victims = got["ids"][0][:1].astype(np.int64)
    store.delete(torch.from_numpy(victims).cuda())
    got, launches = _launches(store, wl, q)
    assert launches == 2 and victims[0] not in got["ids"]


def test_candidates_that_do_not_suffice():
    """304 rows of the same in-weight above the split limit, and no links among them:
    more rows reach the floor than there are candidates, so every call goes through
    the hops."""
    base = synth.workload(2, scale=1 / 64)
    n = base.n
    rng = np.random.default_rng(3)
    hubs = rng.choice(n, 304, replace=False)
    col = np.sort(hubs[(np.arange(8 * n) % 304).reshape(n, 8)], axis=1)   # 431 each, +-1
    ok = ~np.isin(np.arange(n), hubs)
    rp = np.concatenate([[0], np.cumsum(8 * ok)]).astype(np.int64)
    wl = dataclasses.replace(base, row_ptr=rp, col=col[ok].astype(np.int32).ravel(),
                             aff=np.zeros(8 * int(ok.sum()), np.float32), k=16, hops=2)
    q = wl.queries[:20]
    store = gpu_store(wl, "clustered")
    ref = oracle_retrieve(wl, "clustered", queries=q)
    seen = []
    for _ in range(40):
        got, launches = _launches(store, wl, q)
        assert_retrieval_parity(wl, "clustered", got, ref)
        seen.append(launches)
    # the hops until they have cost as much as the tables (192 columns x hops, 64 a
    # call); the candidates tried (first combined, two launches more), the hops run
    # behind them; 15 calls of hops alone
    assert seen == ([2] * 3 + [7] + [2] * 15 + ([5] + [2] * 15) * 2)[:40], seen


def test_tables_wait_where_they_did_not_pay():
    """A store that is written every few reads builds tables once, then does without;
    once it is read long enough again, they come after the least work again."""
    import torch
    wl = synth.workload(2, scale=1 / 64)
    q = wl.queries[:20]
    store = gpu_store(wl, "clustered")
    victims = iter(range(100, 200))

    def reads(n):
        seen = [_launches(store, wl, q)[1] for _ in range(n)]
        store.delete(torch.tensor([next(victims)], device="cuda"))
        return [x > 2 for x in seen]

    hops, cand = [False], [True]
    assert reads(4) == hops * 3 + cand          # built, used once
    assert reads(4) == hops * 4                 # twice the work now
    assert reads(8) == hops * 6 + cand * 2      # again dropped too early
    assert reads(12) == hops * 12               # four times
    assert reads(16) == hops * 12 + cand * 4    # they pay (3 calls' work saved)
    assert reads(4) == hops * 3 + cand


def test_the_path_does_not_depend_on_timing():
    """Batches whose candidates suffice and batches (too sharp) whose do not, under
    one key: enqueued at once they take the paths that they take one by one."""
    import torch
    from paper_2607_05708_gb300 import MemStore
    wl = synth.workload(2, scale=1 / 64)
    norm = lambda x: np.linalg.norm(synth.bf16_to_f32(x), axis=1).max()
    soft = wl.queries[:48]
    sharp = synth.to_bf16(2 * synth.bf16_to_f32(soft))
    tau = 0.25 / (2 * norm(soft) * norm(wl.emb))             # 0.25 and 0.5 about 0.375
    qs = [torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).cuda() for x in (soft, sharp)]
    turns = np.random.default_rng(5).random(60) < 0.15       # True: the sharp one
    out = []
    for wait in (True, False):
        store = MemStore.from_arrays(wl.emb, wl.page_of["clustered"], wl.row_ptr, wl.col, wl.aff,
                                     temperature=tau)
        bufs = [(torch.empty((48, 4), dtype=torch.int64, device="cuda"),
                 torch.empty((48, 4), device="cuda")) for _ in turns]
        torch.cuda.synchronize()
        for t, (ids, scores) in zip(turns, bufs):
            store.retrieve(qs[int(t)], 4, 0.5, 2, ids=ids, scores=scores)
            if wait:
                store.sync()
        store.sync()
        out.append([(i.cpu().numpy(), s.cpu().numpy()) for i, s in bufs])
    for (i0, s0), (i1, s1) in zip(*out):
        assert (i0 == i1).all() and (s0 == s1).all()
    # both paths were taken by the soft batch
    bits = {s.tobytes() for (_, s), t in zip(out[0], turns) if not t}
    assert len(bits) == 2
