"""The arithmetic by which the line kernels find a line's cells and its class, on the
host: below and beyond 2^32 lines, against integers of any size."""
import random
import subprocess

import pytest

from paper_1702_08521_gb300 import _build

PROBE = r"""
#include <cstdio>
#include "vp_internal.cuh"
int main() {
    LineShape s{};
    long long outer, n;
    while (scanf("%lld %lld %lld %u %d %d %lld", &outer, &s.inner, &s.cdiv, &s.cmod, &s.from_inner, &s.L, &n) == 7) {
        s.lines = outer * s.inner;
        s.prepare();
        for (; n > 0; --n) {
            long long line, base;
            if (scanf("%lld", &line) != 1) return 1;
            const unsigned cls = s.place(line, base);
            printf("%lld %u\n", base, cls);
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def place(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(PROBE)
    exe = str(d / "probe")
    subprocess.run([_build._nvcc(), "-std=c++17", "-I", _build.INCLUDE, "-I", _build.CSRC, str(d / "probe.cu"), "-o", exe],
                   check=True, capture_output=True)

    def run(outer, inner, cdiv, cmod, from_inner, L, lines):
        text = "%d %d %d %d %d %d %d\n%s\n" % (outer, inner, cdiv, cmod, from_inner, L, len(lines), "\n".join(map(str, lines)))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in row.split()) for row in out.splitlines()]
    return run


@pytest.mark.parametrize("outer,inner,cdiv,cmod,from_inner", [
    # drifts: classes of the inner index; fewer lines than 2^32, and just as many
    (1, 12, 1, 12, 1), (6, 7 * 33 * 30, 30, 33, 1), (3, 1000003, 7, 1001, 1), (1, 2 ** 32 - 1, 65537, 65537, 1),
    (1, 2 ** 32, 65536, 65536, 1), (2, 2 ** 31, 2 ** 15, 2 ** 16, 1),
    # inner indices beyond 2^32, also a multiple of it
    (1, 65538 * 65537, 65537, 65538, 1), (5, 3 * 2 ** 32, 2 ** 20, 3 * 2 ** 12, 1), (2, 2 ** 33 + 6, 3, 2 ** 20 + 1, 1),
    # kicks: classes of the outer index, up to cdiv beyond 2^32
    (9, 1, 1, 1, 0), (40 * 31, 30, 31, 1, 0), (2 ** 32 - 1, 1, 77, 1, 0), (2 ** 32 + 12345, 1, 1001, 1, 0),
    (2 ** 20, 2 ** 13, 2 ** 5, 1, 0), (3 * 2 ** 32, 2, 2 ** 32, 1, 0)])
def test_lines_and_classes_of_grids_of_any_size(place, outer, inner, cdiv, cmod, from_inner):
    L, n = 3, outer * inner
    rng = random.Random(outer + inner)
    edges = [0, 1, inner - 1, inner, n - inner, n - 1, cdiv - 1, cdiv, 2 ** 32 - 1, 2 ** 32, 2 ** 32 + 1, 2 ** 32 + cdiv]
    lines = sorted({v for v in edges if 0 <= v < n} | {rng.randrange(n) for _ in range(200)})
    got = place(outer, inner, cdiv, cmod, from_inner, L, lines)
    for line, (base, cls) in zip(lines, got):
        o, c = divmod(line, inner)
        assert base == o * L * inner + c, line
        assert cls == (c // cdiv % cmod if from_inner else o // cdiv), line
    assert len(got) == len(lines)
