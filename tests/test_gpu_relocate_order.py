"""Relocation's 32 requests at a time: batches around that number, requests that
move each other's chunks, sets of one chunk and of 64, exact against the
oracle.  Then the pair table's growth by the pairs that it holds."""
import numpy as np
import pytest

from oracle.memory_manager import MemoryManager
from test_gpu_memory_manager import _built, _check, _store  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_req,s_len,pool,P", [
    (1, 2, 40, 4), (31, 3, 12, 1), (32, 5, 30, 16), (33, 64, 90, 16), (100, 8, 9, 64), (64, 1, 50, 4),
])
def test_conflicting_requests_in_order(n_req, s_len, pool, P):
    import torch
    n = 256
    page_of = np.random.default_rng(1).permutation(n) // P
    st, mm = _store(n, 64, page_of, P), MemoryManager(page_of, P)
    rng = np.random.default_rng(n_req + s_len)
    for tau in (0.0, 0.4, 0.7):
        S = rng.integers(-1, pool, (n_req, s_len))
        st.relocate(torch.from_numpy(S).cuda(), tau)
        mm.relocate(S, tau)
        _check(st, mm)
        assert st.compact_pages(0.75, tau) == len(mm.compact(0.75, tau))
        _check(st, mm)


def test_repeated_requests_and_new_pairs():
    """The same pairs again and again, then 600 requests of 64 new chunks each:
    1.2 million pairs, past half of the first table."""
    import torch
    n, P = 40_000, 64
    page_of = np.arange(n) // P
    st, mm = _store(n, 64, page_of, P), MemoryManager(page_of, P)
    rng = np.random.default_rng(9)
    same = rng.integers(0, 200, (50, 5))
    for _ in range(4):
        st.relocate(torch.from_numpy(same).cuda(), 0.7)
        mm.relocate(same, 0.7)
    _check(st, mm)
    S = np.arange(600 * 64).reshape(600, 64)
    st.relocate(torch.from_numpy(S).cuda(), 0.99)
    mm.relocate(S, 0.99)
    _check(st, mm)
    st.relocate(torch.from_numpy(S[:, ::-1].copy()).cuda(), 0.99)
    mm.relocate(S[:, ::-1], 0.99)
    _check(st, mm)


@pytest.mark.parametrize("pages,keep,namespaces", [(1, 1, 1), (40, 4, 3), (512, 4, 2), (513, 4, 5),
                                                   (1000, 4, 64)])
def test_compaction_sizes(pages, keep, namespaces):
    """Compactions of 1 to 4000 chunks, around the 2048 that one CTA repacks,
    grouped by pairs that a relocation left in place."""
    import torch
    n, P = 16384, 16
    page_of = np.arange(n) // P
    ns = np.random.default_rng(2).integers(-2, namespaces - 2, n)
    st, mm = _store(n, 64, page_of, P, ns), MemoryManager(page_of, P, ns_of=ns)
    rng = np.random.default_rng(pages)
    left = []
    gone = []
    for p in rng.choice(n // P, pages, replace=False):
        c = rng.permutation(np.arange(p * P, (p + 1) * P))
        left += c[:keep].tolist()
        gone += c[keep:].tolist()
    S = rng.choice(left, (200, 6))
    st.relocate(torch.from_numpy(S).cuda(), 1.0)
    mm.relocate(S, 1.0)
    st.delete(torch.from_numpy(np.array(gone, np.int64)).cuda())
    mm.delete(np.array(gone, np.int64))
    for tau in (0.3, 0.0):
        assert st.compact_pages(0.75, tau) == len(mm.compact(0.75, tau))
        _check(st, mm)


@pytest.mark.parametrize("P", [2 ** 31 - 1, 2 ** 31 - 3, 2 ** 30])
def test_pages_of_any_size(P):
    """Relocation and compaction with the largest chunks_per_page: a group is one
    page, a namespace's share of a compaction one."""
    import torch
    n = 400
    page_of = np.arange(n) // 40
    ns = np.arange(n) % 4 - 2
    st, mm = _store(n, 64, page_of, P, ns), MemoryManager(page_of, P, ns_of=ns)
    S = np.arange(96).reshape(12, 8) * 4
    st.relocate(torch.from_numpy(S).cuda(), 0.5)
    mm.relocate(S, 0.5)
    _check(st, mm)
    gone = np.array([i for i in range(n) if i % 40 > 9], np.int64)
    st.delete(torch.from_numpy(gone).cuda())
    mm.delete(gone)
    for _ in range(2):
        assert st.compact_pages(0.75, 0.5) == len(mm.compact(0.75, 0.5))
        _check(st, mm)
