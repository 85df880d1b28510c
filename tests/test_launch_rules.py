"""The rules that choose launch shapes, compiled from the engine's header: what
they pick on both sides of their lines, and that the scratch they imply exists."""
import os
import subprocess

import pytest

from paper_2207_05535_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """Evaluate an expression of pa_internal.cuh for each tuple of arguments."""
    tmp = tmp_path_factory.mktemp("rules")

    def run(expr, names, rows):
        src, exe = tmp / "r.cpp", tmp / "r"
        args = ", ".join(f"unsigned {n}" for n in names)
        calls = "".join(f"  f({', '.join(str(v) + 'u' for v in r)});\n" for r in rows)
        src.write_text(f"""#include <cstdio>
#include <cuda_runtime.h>
#include "pa_internal.cuh"
static void f({args}) {{ std::printf("%llu\\n", (unsigned long long)({expr})); }}
int main() {{
{calls}  return 0;
}}
""")
        subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                        os.path.join(ROOT, "paper_2207_05535_gb300", "csrc"), "-I", CUDA_INCLUDE, str(src), "-o",
                        str(exe)], check=True)
        out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
        return [int(v) for v in out]

    return run


def test_few_threads_only_where_the_levels_allow(rule):
    """128 threads per run scan a large lattice's levels slower than 512, while those fit the GPU at once."""
    rows = {(1, 100, 64): 128, (1, 1024, 256): 128, (1, 1025, 256): 512, (100, 300, 1024): 512, (153, 300, 1024): 128,
            (1, 300, 4096): 512, (304, 300, 4096): 512, (305, 300, 4096): 128, (304, 300, 16384): 512,
            (609, 300, 16384): 128, (100000, 300, 65536): 512}
    got = rule("pa::measure_threads(n, cap, N)", ("n", "cap", "N"), list(rows))
    assert got == list(rows.values())
    rows = {(1, 244): 128, (1, 512): 128, (1, 972): 512, (152, 972): 512, (153, 972): 128, (2048, 1025): 512}
    got = rule("pa::resample_threads(n, cap)", ("n", "cap"), list(rows))
    assert got == list(rows.values())


def test_clusters_grow_only_with_the_sweeps_work(rule):
    """16 CTAs lengthen a temperature's chain: few sweeps stay on 8 (theta = 2, R = 700 12.3 us against 13.2)."""
    names = ("L", "n", "t", "th")
    # threads that 8 CTAs take for R = 300, 500, 700, 1000 at L = 16 and 8: 4 lanes per replica
    rows = {(16, 1, 448, 2): 8, (16, 5, 448, 1): 8, (16, 1, 448, 3): 16, (16, 1, 352, 3): 8, (16, 1, 352, 4): 16,
            (16, 8, 328, 10): 8, (16, 1, 204, 5): 8, (16, 1, 204, 10): 16, (16, 9, 388, 4): 16, (16, 1, 628, 1): 16, (8, 1, 328, 10): 8, (8, 1, 328, 20): 16,
            (8, 1, 447, 8): 8, (8, 1, 447, 10): 16, (8, 20, 328, 10): 8, (16, 1, 0, 1 << 22): 8}
    assert rule("pa::small_largest_cluster_ahead(L, n, t, th)", names, list(rows)) == list(rows.values())
    rows = {(16, 1, 384): 8, (16, 1, 385): 16, (16, 9, 461): 8, (16, 9, 568): 16, (32, 1, 9999): 8}
    assert rule("pa::small_largest_cluster(L, n, t)", names[:3], list(rows)) == list(rows.values())
    rows = {(16, 1500, 2): 0, (16, 1500, 10): 1, (8, 1500, 2): 0, (8, 1500, 10): 1, (8, 2000, 10): 1, (8, 2000, 1 << 22): 1}
    assert rule("pa::small_steps_per_stage(L, R, th)", ("L", "R", "th"), list(rows)) == list(rows.values())


def test_scratch_holds_every_split(tmp_path):
    """The CTAs that a run gets in a launch of any others: its scratch tail holds their totals and family statistics."""
    prog, exe = tmp_path / "s.cpp", tmp_path / "s"
    prog.write_text(r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "pa_internal.cuh"
int main()
{
    const unsigned caps[] = {1, 64, 500, 1024, 1365, 1366, 1367, 2048, 2731, 4096, 4097, 5632, 8192, 9824, 16384, 16385,
                             24576, 40000, 65536, 100000, 311296, 1000000, 5000000, 4200000000u};
    const unsigned runs[] = {1, 2, 3, 5, 9, 10, 16, 19, 38, 76, 77, 101, 152, 153, 304, 305, 4096};
    unsigned widest = 0;
    for (unsigned n : runs)
        for (unsigned most : caps) {
            const unsigned grid = pa::split_ctas(n, most), per_cta = (most + grid - 1) / grid;
            if (grid < 1 || grid > pa::MAX_RUN_CTAS) return 1;
            if (pa::resample_nearest_launches(n, most) != (grid == 1 ? 1u : 2u)) return 2;
            for (unsigned cap : caps) {
                if (cap > most) continue;
                const unsigned need = (unsigned)(((unsigned long long)cap + per_cta - 1) / per_cta);  // as the kernels
                const unsigned nc = need < grid ? need : grid;
                if (nc > widest) widest = nc;
                if (nc > 1 && cap <= 1365ull * (nc - 1)) return 3;
                for (unsigned N : {16u, 256u, 65536u}) {
                    const unsigned long long tail = pa::scratch_words(N, cap) - pa::scr_tail_off(N);
                    if (tail < pa::MEASURE_PART_WORDS * nc || 2 * tail < nc) return 4;
                }
            }
        }
    std::printf("%u\n", widest);
    return 0;
}
""")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2207_05535_gb300", "csrc"), "-I", CUDA_INCLUDE, str(prog), "-o", str(exe)],
                   check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0 and int(res.stdout) > 32
