"""Launch shapes of the NTT's phases (csrc/phase_shape.h, compiled here as plain
C++): for every ring degree and every accepted tile size a phase covers its limb
exactly within the kernels' threads and an SM's shared memory, and the values
the autotuner searches are the different launches, each once."""
import os
import shutil
import subprocess

import pytest

from paper_2601_15401_gb300 import executor as E

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "paper_2601_15401_gb300/csrc/phase_shape.h"
#include <cstdio>
using namespace ckks;
int main() {
    for (int log_n = 4; log_n <= 16; ++log_n)
        for (int cols = 0; cols < 2; ++cols)
            for (int tile = 512; tile <= 8192; tile *= 2) {
                int a, b;
                ntt_geometry(log_n, a, b);
                if (cols && a == 0) continue;
                const PhaseShape s = cols ? phase_shape(log_n, true, tile, 1024) : phase_shape(log_n, false, 4096, tile);
                printf("%d %d %d %d %d %d %d %d %zu %d\n", log_n, cols, tile, s.shape, s.logn, s.tiles, s.threads,
                       s.limbs, s.smem, a);
            }
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("shapes")
    (d / "s.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", ROOT, "-o", str(d / "s"), str(d / "s.cpp")], check=True)
    out = subprocess.run([str(d / "s")], capture_output=True, text=True, check=True).stdout
    return {r[:3]: r[3:] for r in (tuple(map(int, x.split())) for x in out.splitlines())}


def test_every_tile_covers_the_limb(shapes):
    for (log_n, cols, tile), (shape, logn, tiles, threads, limbs, smem, log_n1) in shapes.items():
        n, n1, n2 = 1 << logn, 1 << log_n1, 1 << (log_n - log_n1)
        assert smem <= 227 * 1024 and 1 <= threads <= 256
        if shape == 0:
            groups = threads // n           # n threads take 16 columns
            assert threads == groups * n and tiles * groups * 16 == n2
            assert smem == groups * 16 * n * 8 + n * 16
        elif shape == 2:
            assert (tiles, threads, limbs) == (1, n // 16, 1)
        elif log_n1 == 0:
            assert (tiles, threads) == (1, 32 * limbs) and smem % (16 * limbs) == 0
        else:
            blocks = threads // (n // 16)   # n / 16 threads take a block
            assert threads % 32 == 0 and tiles * blocks == n1 and limbs == 1
            assert smem == blocks * ((n + n // 16) * 8 + (n - 1) * 16)


def test_the_search_times_each_launch_once(shapes):
    for log_n in range(9, 17):
        for name, cols in (("ntt_tile_cols", 1), ("ntt_tile_blocks", 0)):
            values = E.tune_values(name, log_n)
            accepted = {tile: s for (l, c, tile), s in shapes.items() if (l, c) == (log_n, cols)}
            if not accepted:                # no column phase
                assert values == [E.TUNE_DEFAULTS[name]]
                continue
            launches = [accepted[v] for v in values]
            assert len(set(launches)) == len(launches)
            assert set(launches) == set(accepted.values())
            assert E.TUNE_DEFAULTS[name] in values
    # a difference within two timings of one launch does not move a tunable
    assert E.pick({128: 1.0, 256: 1.009}, 256) == 256 and E.pick({128: 1.0, 256: 1.02}, 256) == 128
    assert E.pick({}, 256) == 256 and E.pick({128: 2.0, 64: 1.0}, 256) == 64
    # the other tunables: every value within what the kernels run
    for name in ("bconv_threads", "mac_threads"):
        assert E.tune_values(name, 16) == E.TUNE_SPACE[name] and max(E.TUNE_SPACE[name]) <= 256
