"""Shared memory of a launch of teams (team_smem_bytes in csrc/gfmc_internal.h,
compiled for the host): the launch never asks for more than the room when every work
area fits it alone, holds what each of its chains uses, and a chain's vectors stand there
by its own sizes and the room, whatever other chains the launch has.  Chains are
those of gfmc_run_batch: packed ones of one CTA or a tile, others, K from 16 to 8192."""
import shutil
import subprocess

import pytest

from test_tile_plan import INTERNAL

DRIVER = r"""
int main()
{
    const size_t room = 232448 - 2208, dev = 232448;
    unsigned long long rng = 1;
    auto next = [&](unsigned n) { rng = rng * 6364136223846793005ull + 1442695040888963407ull; return (unsigned)(rng >> 33) % n; };
    auto chain = [&]() {
        TeamChainSmem q{};
        const size_t K = (size_t)16 << next(10);
        q.packed = next(2);
        q.work = 16 * K;
        if (!q.packed && q.work < 57568) q.work = 57568;
        q.vec = next(4) == 0 ? SIZE_MAX : 1000 + next(300000);
        q.want = q.vec == SIZE_MAX ? 0 : q.vec + next(200000);
        return q;
    };
    int bad = 0, resident = 0, global = 0;
    for (int t = 0; t < 20000; ++t) {
        TeamChainSmem c[6], alone;
        const int n = 1 + next(6);
        for (int k = 0; k < n; ++k) c[k] = chain();
        const int total = team_smem_bytes(c, n, room);
        if ((size_t)total > room) ++bad;
        for (int k = 0; k < n; ++k) {
            const size_t need = c[k].packed ? ((size_t)c[k].at > c[k].work ? (size_t)c[k].at : c[k].work) : c[k].at + c[k].work;
            if (need > (size_t)total || c[k].at % 16) ++bad;
            if (c[k].at && (size_t)c[k].at < c[k].vec) ++bad;
            alone = c[k];
            team_smem_bytes(&alone, 1, room);
            if (alone.at != c[k].at) ++bad;
            ++(c[k].at ? resident : global);
        }
    }
    // FP32 on K = 8192 nodes: L = 8 on one CTA beside L = 24 on one CTA, whose vectors stay in global memory
    TeamChainSmem two[2] = {{73728, 131072, 0, true, 0}, {2 * 13824 * 8, 131072, 0, true, 0}};
    if (team_smem_bytes(two, 2, room) > (int)room || two[0].at == 0) ++bad;
    (void)dev;
    std::printf("resident %d, global %d, bad %d\n", resident, global, bad);
    return bad || !resident || !global;
}
"""


def test_team_shared_memory_fits_and_is_each_chains_own(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = open(INTERNAL).read()
    a = src.index("struct TeamChainSmem")
    fn = src[a:src.index("\n}\n", src.index("inline int team_smem_bytes")) + 3]
    f = tmp_path / "smem.cpp"
    f.write_text("#include <cstdint>\n#include <cstdio>\n#include <cstddef>\n" + fn + DRIVER)
    exe = tmp_path / "smem"
    subprocess.run([cxx, "-O1", "-std=c++17", "-o", str(exe), str(f)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
