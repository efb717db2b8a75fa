"""Calls that do not get the device memory they ask for: they fail, or go on
another way, and leave the store as it was.  The memory is taken by ordinary
allocations beside the store, in blocks that are given back one by one, so that
every allocation of a call gets to fail."""
import contextlib

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MB = 1 << 20


class _Held:
    """All free device memory but `left` bytes, and blocks to give back."""

    def __init__(self, left, blocks, size):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        new = lambda b: torch.empty(b, dtype=torch.uint8, device="cuda")
        self.blocks = [new(size) for _ in range(blocks)]
        self.rest, part = [], 1 << 38
        while part >= 8 * MB:                 # the rest in pieces of a power of two
            free = torch.cuda.mem_get_info()[0]
            if free - left < part:
                part >>= 1
                continue
            try:
                self.rest.append(new(part))
            except torch.OutOfMemoryError:    # no piece of that size in one
                part >>= 1

    def give_back(self):
        import torch
        self.blocks.pop()
        torch.cuda.empty_cache()


@contextlib.contextmanager
def _memory(left, blocks=0, size=16 * MB):
    import torch
    held = _Held(left, blocks, size)
    try:
        yield held
    finally:
        held.blocks.clear()
        held.rest.clear()
        torch.cuda.empty_cache()


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
