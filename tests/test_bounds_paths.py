"""The row bounds' widening for split rows: the roundings on a term's path are
those of a segment (at most seg_len terms in sequence) and of the sum over the
row's segments, not the in-degree.  The hop's and the bound's own sums emulated
in numpy fp32, with every product rounded and one chain per segment (worse than
the device's fused, many-lane sums), against the widened bounds."""
import numpy as np
import pytest

EPS = np.float32(5.9604645e-8)
F = np.float32


def _chain(v):
    return np.cumsum(v.astype(F), dtype=F)[-1] if v.size else F(0)


def _segmented(w, x, cuts):
    """fp32: a chain per segment, then a chain over the segments."""
    p = (w * x).astype(F)
    return _chain(np.array([_chain(p[a:b]) for a, b in zip(cuts[:-1], cuts[1:])], F))


@pytest.mark.parametrize("edges,seg_len,windows", [(257, 512, 1), (5000, 512, 3), (60_000, 512, 32),
                                                   (300_000, 512, 128), (20_000, 64, 7)])
@pytest.mark.parametrize("spread", [0.0, 1.0])
def test_split_row_widening_covers_the_sums(edges, seg_len, windows, spread):
    rng = np.random.default_rng(edges + windows)
    w = rng.uniform(0.01, 1.0, edges).astype(F) if spread else np.full(edges, 0.031, F)
    s = (1.0 + spread * rng.uniform(0, 0.04, edges)).astype(F)     # the sources' values
    U, L = F(s.max()), F(s.min())
    edge_of_window = np.sort(rng.choice(np.arange(1, edges), windows - 1, replace=False))
    cuts = [0]
    for b in list(edge_of_window) + [edges]:
        while b - cuts[-1] > seg_len:
            cuts.append(cuts[-1] + seg_len)
        cuts.append(b)
    n = min(edges, seg_len + len(cuts) - 1)                        # as k_split_bound takes it
    x = F(3.25) * F(n + 8) * EPS
    alpha, u = F(0.5), s[0]
    hop = F(alpha * _segmented(w, s, cuts) + u)
    up = F(F(F(alpha * _segmented(w, np.full(edges, U), cuts)) * F(F(1) + x + x * x) + U) * F(1 + 4e-6))
    dn = F(F(F(alpha * _segmented(w, np.full(edges, L), cuts)) * F(F(1) - x) + L) * F(1 - 4e-6))
    exact = float(alpha) * float(np.dot(w.astype(np.float64), s.astype(np.float64))) + float(u)
    assert dn <= hop <= up and dn <= exact <= up
    # and it stays tight: far below the in-degree's own widening for a hub
    if edges >= 60_000:
        assert float(x) < 0.05 * 3.25 * (edges + 8) * float(EPS)
