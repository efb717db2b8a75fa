"""Calls that do not get the device memory they ask for: they fail, or go on
another way, and leave the store as it was.  The memory is taken by ordinary
allocations beside the store, in blocks that are given back one by one, so that
every allocation of a call gets to fail."""
import contextlib
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


class _Held:
    """All free device memory but `left` bytes, and blocks to give back; from the
    driver, so that a block given back is free at once."""

    def __init__(self, left, blocks, size):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.cuda = ctypes.CDLL("libcuda.so.1")
        self.blocks, self.rest, part = [], [], 1 << 38
        while len(self.blocks) < blocks:
            self.blocks.append(self._new(size))
            assert self.blocks[-1], "no room to begin with"
        while part >= 8 * MB:                 # the rest in pieces of a power of two
            fits = torch.cuda.mem_get_info()[0] - left >= part
            p = self._new(part) if fits else None
            if p:
                self.rest.append(p)
            else:                             # (or no piece of that size in one)
                part >>= 1

    def _new(self, size):
        p = ctypes.c_uint64()
        rc = self.cuda.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(size))
        assert rc in (0, 2), rc               # CUDA_SUCCESS, CUDA_ERROR_OUT_OF_MEMORY
        return p if rc == 0 else None

    def give_back(self):
        assert self.cuda.cuMemFree_v2(self.blocks.pop()) == 0

    def give_all(self):
        self.blocks, rest = [], self.blocks + self.rest
        self.rest = []
        for p in rest:
            assert self.cuda.cuMemFree_v2(p) == 0


@contextlib.contextmanager
def _memory(left, blocks=0, size=16 * MB):
    held = _Held(left, blocks, size)
    try:
        yield held
    finally:
        held.give_all()


def _store(n, room, dim=64, links=32, seed=3, **kw):
    """n unit chunks, `links` targets each, three quarters of them few popular ones."""
    import torch
    from paper_2607_05708_gb300 import MemStore
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n + room, dim), generator=gen, device="cuda")
    emb = (x / x.norm(dim=1, keepdim=True)).to(torch.bfloat16).view(torch.int16)
    u = torch.rand((n, links), generator=gen, device="cuda")
    t = (u.pow(6) * (n - 2 * links)).long()
    t = t.sort(dim=1).values + torch.arange(links, device="cuda")   # distinct, ascending
    t += (t >= torch.arange(n, device="cuda")[:, None]).long()      # not the chunk itself
    aff = torch.rand((n, links), generator=gen, device="cuda")
    st = MemStore(dim, n + room, chunks_per_page=64, relation_scale=10.0, **kw)
    st.append_chunks(emb[:n], None, torch.arange(n + 1, device="cuda") * links,
                     t.int().view(-1), aff.view(-1))
    return st, emb


def _csr(st):
    return [t.cpu().numpy() for t in st.export_csr()]


def test_an_update_that_does_not_fit_changes_nothing():
    from paper_2607_05708_gb300 import AkashicError
    n, new, M = 262_144, 256, 32
    want, emb = _store(n, new)                # (its kernels are loaded by now)
    before = _csr(want)
    want.append_chunks(emb[n:])
    want.update_relations(n, new, M, True)
    want = _csr(want)
    st, emb = _store(n, new)
    st.append_chunks(emb[n:])
    failed = 0
    with _memory(24 * MB, blocks=40) as held:
        while True:
            try:
                st.update_relations(n, new, M, True)
                break
            except AkashicError as e:
                assert e.code == "ENOMEM", e
                failed += 1
                assert st.size()[1] == n * 32
                held.give_back()
    got = _csr(st)
    assert failed >= 3
    for a, b in zip(got, want):
        assert (a == b).all()
    assert len(before[1]) == n * 32


def _two(st, q, stream, hops, k=8):
    import torch
    with torch.cuda.stream(stream):
        out = st.retrieve(q, k, 0.5, hops, stream=stream)
    return out


def test_tables_that_do_not_fit_are_not_seen_half_built(monkeypatch):
    """Two streams with different hop counts after a deletion: the one with three
    hops does not get its third table.  The other's answers come from tables that
    are finished, at once and later."""
    import torch
    n = 262_144
    monkeypatch.setenv("AKASHIC_REACH", "0")
    plain, emb = _store(n, 0)
    monkeypatch.setenv("AKASHIC_REACH", "1")
    st, _ = _store(n, 0)
    q = emb[5:6].contiguous()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(6):                        # two hops: the tables are built
        _two(st, q, b, 2)
    _two(st, q, a, 3)                         # a's own slabs
    torch.cuda.synchronize()
    gone = torch.tensor([int(_two(st, q, b, 2)[0][0, 0])], device="cuda")
    torch.cuda.synchronize()
    plain.delete(gone)
    st.delete(gone)
    want = [t.cpu().numpy() for t in plain.retrieve(q, 8, 0.5, 2)]
    out = []
    with _memory(16 * MB):
        for _ in range(8):                    # (the hops, until the tables pay)
            _two(st, q, a, 3)
        for _ in range(4):
            out.append(_two(st, q, b, 2))
        st.sync(a)
        st.sync(b)
    out.append(_two(st, q, b, 2))
    st.sync(b)
    for ids, scores, _, _ in out:
        hit = ids.cpu().numpy() == want[0]
        assert hit.mean() >= 0.75
        np.testing.assert_allclose(scores.cpu().numpy(), want[1], rtol=1e-5, atol=0)


def _candidates(st, q, stream=None):
    """Whether a call of two hops queues the candidates' pass."""
    st.set_profiling(True)
    st.phase_times()
    st.retrieve(q, 8, 0.5, 2, stream=stream)
    st.sync(stream)
    ph = st.phase_times()
    st.set_profiling(False)
    return ph["last_hop"][1] > 2


def test_tables_give_way(monkeypatch):
    """An update and a wide retrieval that fit only in the place of the tables."""
    import torch
    n, new = 262_144, 256
    monkeypatch.setenv("AKASHIC_REACH", "0")
    plain, emb = _store(n, new)
    monkeypatch.setenv("AKASHIC_REACH", "1")
    st, _ = _store(n, new)
    few, many = emb[5:6].contiguous(), emb[:256].contiguous()
    wide = [t.cpu().numpy() for t in plain.retrieve(many, 5, 0.5, 0)]
    first = [t.cpu().numpy() for t in plain.retrieve(few, 8, 0.5, 2)]
    assert [_candidates(st, few) for _ in range(5)][-1]
    with _memory(16 * MB):                       # the tables are 0.4 GB, the slab 0.27
        got = [t.cpu().numpy() for t in st.retrieve(many, 5, 0.5, 0)]
        st.sync()
        assert not any(_candidates(st, few) for _ in range(8))
        out = [t.cpu().numpy() for t in st.retrieve(few, 8, 0.5, 2)]
    for a, b in zip(got, wide):
        assert (a == b).all()
    for a, b in zip(out, first):
        assert (a == b).all()                    # the hops: the same bits
    st, _ = _store(n, new)
    assert [_candidates(st, few) for _ in range(5)][-1]
    plain.append_chunks(emb[n:])
    plain.update_relations(n, new, 32, True)
    want = _csr(plain)
    with _memory(48 * MB):                       # (an update takes 0.35 GB)
        st.append_chunks(emb[n:])
        st.update_relations(n, new, 32, True)
    for a, b in zip(_csr(st), want):
        assert (a == b).all()


def test_tables_leave_as_much_free():
    """The tables of one query and two hops (three tables of 512 bytes a chunk) are
    not taken where less than twice that is free."""
    import torch
    n = 262_144
    st, emb = _store(n, 0)
    q = emb[5:6].contiguous()
    st.retrieve(q, 8, 0.5, 2)                    # the slabs
    st.sync()
    with _memory(3 * 512 * n * 3 // 2):
        free = torch.cuda.mem_get_info()[0]
        assert not any(_candidates(st, q) for _ in range(8))
        assert torch.cuda.mem_get_info()[0] > free - 8 * MB      # (the outputs)
    st, _ = _store(n, 0)
    assert [_candidates(st, q) for _ in range(8)][-1]
