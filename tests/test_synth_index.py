"""Index arithmetic of the synthesis at the largest arrays its arguments can name (2^31 - 1
elements), compiled for the host with checks for signed overflow, against integers of
any size. Kernels of that size take most of a GPU's memory and are not run."""
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_10006_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "synth_index.cuh"
int main() {
    long long a, b, c;
    while (scanf("%lld %lld %lld", &a, &b, &c) == 3)
        printf("%lld %lld %lld %lld\n", (long long)sbr::xyz_at(b), (long long)sbr::tiles_of((int32_t)c, 256),
               (long long)sbr::dl_size(a + 1, c), (long long)sbr::dl_index((int32_t)a, (int32_t)b, (int32_t)c));
}
"""


def dl_index(q, p, Nt):
    block = (q // 8) * -(-Nt // 16) + p // 16
    return block * 128 + ((q % 8) * 4 + (p % 8) // 2) * 4 + (p // 8 % 2) * 2 + p % 2


@pytest.mark.parametrize("top", [300, 1 << 20, 2 ** 31 - 1])
def test_indexes(tmp_path, top):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", CSRC,
                    str(tmp_path / "t.cpp"), "-o", exe], check=True)
    rng = random.Random(top)
    cases = [(0, top - 1, top), (7, 0, top), (top - 1, 0, 1), (9, top - 1, top)]
    cases += [(rng.randrange(100), rng.randrange(n), n) for n in (rng.randint(1, top) for _ in range(200))]
    out = subprocess.run([exe], input="".join("%d %d %d\n" % c for c in cases), capture_output=True, text=True, check=True).stdout
    want = [(3 * p, -(-n // 256), -(-(q + 1) // 8) * -(-n // 16) * 128, dl_index(q, p, n)) for q, p, n in cases]
    assert [tuple(map(int, l.split())) for l in out.splitlines()] == want
    # distinct places within the table of one array
    if top == 300:
        for Nr, Nt in ((1, 1), (9, 33), (16, 64)):
            at = {dl_index(q, p, Nt) for q in range(Nr) for p in range(Nt)}
            assert len(at) == Nr * Nt and max(at) < -(-Nr // 8) * -(-Nt // 16) * 128
