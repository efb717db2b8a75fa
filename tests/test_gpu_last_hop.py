"""The last hop's filter bound (the hop's own values on a row sample) and what
the hop leaves out, on graphs where they can go wrong: no hubs at all, rows
around the sample's edge limit and the split limit, fewer hubs than k, ties
everywhere.  Against the oracle, with the tolerances of `_parity`."""
import dataclasses

import numpy as np
import pytest

import synth
from _parity import assert_retrieval_parity, gpu_retrieve, oracle_retrieve

pytestmark = pytest.mark.gpu


def _graph(base, degrees, seed):
    """Row j gets degrees[j] in-edges from distinct other rows, random logits."""
    rng = np.random.default_rng(seed)
    n = base.n
    tgt = np.repeat(np.arange(n), degrees)
    src = np.concatenate([(j + 1 + rng.choice(n - 1, d, replace=False)) % n
                          for j, d in enumerate(degrees) if d])
    order = np.lexsort((tgt, src))
    row_ptr = np.zeros(n + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(src, minlength=n))
    return dataclasses.replace(base, row_ptr=row_ptr, col=tgt[order].astype(np.int32),
                               aff=rng.normal(0, 1, tgt.size).astype(np.float32))


def _store(n):
    base = synth.workload(2, scale=1 / 64)
    return dataclasses.replace(base, emb=base.emb[:n],
                               page_of={"clustered": base.page_of["clustered"][:n]},
                               component=base.component[:n])


@pytest.mark.parametrize("n,B,hops,k,heavy", [
    (2048, 1, 1, 1, 0),         # the sample holds every row
    (5003, 33, 1, 64, 0),       # ragged, two lane groups a row
    (16384, 8, 2, 16, 0),       # whole tiles of 1024 rows
    (16383, 100, 3, 5, 3),      # fewer split rows than k
    (9001, 256, 1, 8, 40),      # more split rows than k: the sample's edge limit
    (9001, 129, 2, 64, 64),
])
def test_graphs_with_few_hubs(n, B, hops, k, heavy):
    base = _store(n)
    rng = np.random.default_rng(n + B)
    deg = rng.choice([0, 1, 7, 31, 32, 33, 40], n)
    deg[rng.choice(n, heavy, replace=False)] = rng.integers(257, 900, heavy)
    deg[rng.choice(n, 4, replace=False)] = [255, 256, 64, 65]
    wl = dataclasses.replace(_graph(base, deg, n), hops=hops, k=k, queries=base.queries[:B])
    _, got = gpu_retrieve(wl, "clustered")
    assert_retrieval_parity(wl, "clustered", got, oracle_retrieve(wl, "clustered"))


@pytest.mark.parametrize("hops", [1, 2])
def test_equal_scores_overflow_the_buffers(hops):
    """16384 equal embeddings on a ring of 4 successors with equal logits:
    every score is the same after every hop, so all rows reach the bound, the
    8192-key buffers overflow and the merge recomputes the columns; the k
    lowest IDs win."""
    base = synth.workload(2, scale=1 / 64)
    n = base.n
    col = np.sort((np.arange(n)[:, None] + np.arange(1, 5)[None, :]) % n, axis=1)
    wl = dataclasses.replace(base, emb=np.repeat(base.emb[:1], n, axis=0), hops=hops, k=8,
                             row_ptr=np.arange(0, 4 * n + 1, 4, dtype=np.int64),
                             col=col.astype(np.int32).ravel(), aff=np.zeros(4 * n, np.float32),
                             queries=base.queries[:4])
    _, got = gpu_retrieve(wl, "clustered")
    assert (np.sort(got["ids"], axis=1) == np.arange(8)).all()
