"""The scratch sizes of the radix sort and the prefix sum never fall as the count
grows: one scratch, sized by the largest count, serves shorter sorts too.
Compiles csrc/ak_sizes.h (plain C++) and reads the sizes it gives."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_05708_gb300", "csrc")


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("sizes")
    src = d / "sizes.cpp"
    src.write_text('#include "ak_sizes.h"\n#include <stdio.h>\n'
                   'int main() { long long n;\n'
                   '  while (scanf("%lld", &n) == 1)\n'
                   '    printf("%zu %zu\\n", ak::radix_tmp_bytes(n), ak::scan_tmp_bytes(n)); }\n')
    exe = str(d / "sizes")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)

    def get(ns):
        out = subprocess.run([exe], input="\n".join(map(str, ns)), capture_output=True, text=True,
                             check=True).stdout.split()
        return [int(x) for x in out[::2]], [int(x) for x in out[1::2]]
    return get


def test_sizes_never_fall(sizes):
    ns = list(range(1, 10_000)) + list(range(10_000, 2_000_000, 997))
    for t in (2048, 262_144, 1 << 20, 1 << 24, 2 ** 31 - 1):     # a small sort's limits, large ones
        ns += [t - 1, t, t + 1]
    for got in sizes(sorted(set(ns))):
        assert all(a <= b for a, b in zip(got, got[1:]))


@pytest.mark.parametrize("new,m", [(140_000, 2), (200_000, 2), (262_144, 2), (262_144, 64)])
def test_the_new_rows_sort_in_the_pairs_scratch(sizes, new, m):
    """A reciprocal update sorts its new * m pairs, then its new rows."""
    (rows, pairs), _ = sizes([new, new * m])
    assert rows <= pairs
