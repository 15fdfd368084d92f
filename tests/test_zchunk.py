"""The z-chunk rules of the persistent launches (csrc/mhd_zmarch.cuh) on the
CPU: the chunk lengths they choose, and that a launch of a tall box does not walk
every number of chunks to find one."""
import importlib
import os
import subprocess

import pytest

build = importlib.import_module("paper_1908_08557_gb300.build")

PROBE = r"""
#include <cstdio>
#include "mhd_zmarch.cuh"
int main() {
  int nz, tiles, ctas;
  while (std::scanf("%d %d %d", &nz, &tiles, &ctas) == 3) {
    int n = 1;
    for (int kc = nz; (kc = mhd::zm::shorter_chunk(nz, kc)) > 0;) ++n;
    std::printf("%d %d %d\n", mhd::zm::zchunk(nz, tiles, ctas), mhd::zm::zchunk_claimed(nz, tiles, ctas, 1.35), n);
  }
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("zchunk")
    (d / "p.cu").write_text(PROBE)
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O2", "-I", build.CSRC, "-I",
                        os.path.join(build.ROOT, "include"), str(d / "p.cu"), "-o", str(d / "p")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "p")


def _lengths(nz):
    """Every chunk length ceil(nz / n), by the number of chunks n, first n of each."""
    out = {}
    for n in range(1, nz + 1):
        out.setdefault(-(-nz // n), n)
    return list(out)


def _zchunk(nz, tiles, ctas):
    best, eff_best = nz, 0.0
    for kc in _lengths(nz):
        items = tiles * -(-nz // kc)
        waves = -(-items // ctas)
        eff = items / (waves * ctas) * kc / (kc + 6)
        if eff > eff_best + 1e-9:
            best, eff_best = kc, eff
    return best


def _claimed(nz, tiles, ctas, lead):
    cost = lambda kc: tiles * nz / ctas * (1.0 + lead / kc) + 0.5 * (kc + lead)  # noqa: E731
    return min(_lengths(nz), key=cost)


def test_chunks_are_the_best_of_all_numbers_of_chunks(probe):
    cases = [(nz, t, c) for nz in (7, 13, 16, 31, 64, 97, 256, 997, 4000) for t in (1, 3, 8, 64, 256, 4096)
             for c in (152, 304)]
    r = subprocess.run([probe], input="".join(f"{a} {b} {c}\n" for a, b, c in cases), capture_output=True, text=True,
                       check=True)
    for case, line in zip(cases, r.stdout.splitlines(), strict=True):
        z, zc, n = map(int, line.split())
        assert z == _zchunk(*case) and zc == _claimed(*case, 1.35), case
        assert n == len(_lengths(case[0])) <= 2 * case[0] ** 0.5 + 1
