"""The per-CTA buffers of a chain (phase sums, magnetisation partials, flags) hold
every launch of the chain, whatever teams it has run on in between: a single
chain's own launches take as many CTAs as its packed engine (pk_ctas), which may
be more than its tiles (ncta), and a team of a size between the two replaces
buffers that are too small for the team, and only those.  The sizes, the
capacity and ensure_team_capacity are taken from csrc/gfmc_api.cu and compiled for
the host, with an allocator that records sizes, over every even L and team size."""
import re
import shutil
import subprocess

import pytest

from test_fixed_point import ROOT
from test_tile_plan import API, INTERNAL, extract

PRELUDE = r"""
#include <algorithm>
#include <cstdio>
#include <map>
#include <vector>
#include <cstddef>
#define __host__
#define __device__
enum gfmc_status { GFMC_OK = 0 };
typedef int cudaError_t;
constexpr int cudaSuccess = 0;
struct Params { double *qpart = nullptr, *magpart = nullptr; unsigned* flags = nullptr; };
struct gfmc_ctx { int cap_ncta = 0, pk_ctas = 0; Params P; };
static std::map<void*, size_t> made;
template <class T> cudaError_t dalloc(gfmc_ctx*, T** p, size_t n)
{
    *p = (T*)(new char);
    made[*p] = n;
    return cudaSuccess;
}
static void release(gfmc_ctx*, void*) {}
static gfmc_status cuda_fail(gfmc_ctx*, cudaError_t, const char*) { return GFMC_OK; }
namespace gfmc {
"""

DRIVER = r"""
static void create(gfmc_ctx* h, int ncta)
{
    Params& P = h->P;
    cudaError_t e;
    (void)e;
    CREATE
}

int main()
{
    int bad = 0, replaced = 0;
    for (int L = 4; L <= 64; L += 2)
        for (int K : {16, 1024, 8192})
            for (int sms : {148, 152}) {
                const int N = L * L * L, ncta = std::max(1, std::min(N / 64, sms));
                // every engine a chain may run alone: a cluster of up to 16 CTAs, or the grid
                std::vector<int> own = {1, 16};
                int cy, cz, bytes;
                if (gfmc::pk_grid_split(L, K, sms, 225 * 1024, &cy, &cz, &bytes)) own.push_back(cy * cz);
                for (int pk : own)
                    for (int tc = 1; tc <= std::min(N, 200); ++tc) {
                        gfmc_ctx h;
                        h.pk_ctas = pk;
                        create(&h, ncta);
                        const int before = h.cap_ncta;
                        ensure_team_capacity(&h, tc);
                        replaced += h.cap_ncta != before;
                        const size_t need = std::max({ncta, pk, tc});
                        if (made[h.P.qpart] < 2 * need || made[h.P.magpart] < 3 * need || made[h.P.flags] < (size_t)std::max(ncta, tc))
                            ++bad;
                        if ((size_t)h.cap_ncta < need) ++bad;
                    }
            }
    std::printf("replaced %d, bad %d\n", replaced, bad);
    return bad != 0 || replaced == 0;
}
"""


def test_buffers_hold_every_launch_of_the_chain(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = open(API).read()
    internal = open(INTERNAL).read()
    split = internal[internal.index("// Shared memory of a CTA of the packed cluster engine"):
                     internal.index("// One-CTA chains of a few sites per thread")]
    # the allocations and the capacity as gfmc_create states them
    create = "".join(re.findall(r"    const int cap = .*?;\n", src))
    for name in ("qpart", "magpart", "flags"):
        call = re.search(r"\(e = (dalloc\(h, &P\." + name + r",.*?)\) != cudaSuccess", src).group(1)
        create += f"    e = {call};\n"
    create += re.findall(r"    h->cap_ncta = \w+;\n", src)[-1]
    fn = extract(API, r"gfmc_status ensure_team_capacity\(gfmc_ctx\* h, int tc\).*?\n\}\n")
    f = tmp_path / "cap.cpp"
    f.write_text(PRELUDE + split + "}\n" + fn + DRIVER.replace("CREATE", create))
    exe = tmp_path / "cap"
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-o", str(exe), str(f)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
