"""How the descriptor kernel's calls are spread over it (desc_plan) and its shared memory, over all bases the library takes; and
which of its paths the parametrised GPU tests reach.  Host arithmetic, compiled from the library's own headers."""
import os
import subprocess

import pytest

from paper_2609_05709_b200 import build
from test_gpu_descriptor_quads import BASES, MOLECULES, R_CUT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "basis_host.h"
#include "desc_layout.h"
using namespace soap;
const size_t max_smem = 227 * 1024;                                // what a CTA of this architecture may have
const int64_t sms = 148;
int layouts() {
    for (int S = 1; S <= kMaxSpecies; ++S)
        for (int n = 1; n <= 16; ++n)
            for (int l = 0; l <= 12; ++l) {
                const int np = desc_np(n), L1 = l + 1;
                if (n * L1 * L1 > kMaxElements) continue;
                for (const int plain : {0, 1})
                    for (const int64_t work : {1, 27, 592, 593, 740, 741, 900, 3000, 100000})
                        for (const int intervals : {0, 40, 90}) {
                            const size_t words = (size_t)intervals * L1 * np * 6;
                            for (const int64_t atoms : {(int64_t)0, work}) {
                                const DescPlan p = desc_plan(S, np, l, plain, false, words, work, atoms, sms, max_smem);
                                const DescLayout o = make_desc_layout(S, np, l, p.warps, p.table ? (int)words : 0, p.team != 0, plain);
                                bool ok = p.bytes <= max_smem && p.warps >= 1 && (int64_t)p.grid * p.warps >= (p.team ? work * p.warps : 1);
                                ok = ok && p.bytes == (size_t)o.total * 4 + (p.team ? desc_search_bytes(atoms, p.warps) : 0);
                                ok = ok && (p.team ? work <= 740 && p.warps == p.team : p.warps <= kDescMaxWarps);
                                // a team's slots for what it finds, 8 bytes each, lie behind everything else; a slot per atom
                                ok = ok && o.total % 2 == 0 && (!p.team || (int64_t)desc_search_share(atoms, p.warps) * p.warps >= atoms);
                                const int starts[] = {o.blocks, o.warp0, o.per_warp, o.c, o.sS, o.sG, o.ring};
                                for (const int at : starts) ok = ok && at % 4 == 0;
                                ok = ok && o.blocks >= (p.table ? (int)words : 0) && o.sS >= o.c + S * np * L1 * L1 && o.total == o.warp0 + p.warps * o.per_warp;
                                if (!ok) printf("species %d n_max %d l_max %d plain %d centres %lld\n", S, n, l, plain, (long long)work);
                            }
                        }
            }
    return 0;
}
int main(int argc, char** argv) {
    if (argc == 1) return layouts();
    // n_max, l_max, r_cut, centres, weighted -> quads of a lane that keeps its quad, of a list, or pairs; and where the table is
    const int n = atoi(argv[1]), l = atoi(argv[2]);
    const bool weighted = atoi(argv[5]);
    HostBasis b;
    std::string err;
    if (build_basis(0, atof(argv[3]), n, l, 0.5, b, err)) return 1;
    const int np = desc_np(n);
    const DescPlan p = desc_plan(2, np, l, !weighted, weighted, (size_t)b.n_intervals_values * (l + 1) * np * 6, atoi(argv[4]), 0, sms, max_smem);
    printf("%s %s\n", desc_quad_span(np, l) ? "kept" : desc_quads(np, l) ? "list" : "pairs", p.team ? "team" : p.table ? "shared" : "global");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    (d / "layout.cpp").write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-I", build.CSRC, "-I", build.INCLUDE, "-I", cuda, str(d / "layout.cpp"),
                    os.path.join(build.CSRC, "basis_host.cpp"), "-o", str(d / "layout"), "-lquadmath"], check=True)
    return lambda *a: subprocess.run([str(d / "layout"), *map(str, a)], check=True, capture_output=True, text=True).stdout.strip()


def test_regions_and_plans(program):
    assert program() == ""


def test_the_radial_factors_are_tested_on_every_path(program):
    """The bases of test_gpu_descriptor_quads.py: each way of taking radial factors, by teams and with the table in shared and in
    global memory."""
    reached = {name: {tuple(program(n, l, R_CUT, 3 * molecules, int(weighted)).split()) for n, l in BASES}
               for name, (molecules, weighted) in MOLECULES.items()}
    for way in ("pairs", "kept", "list"):
        assert (way, "team") in reached["team"] and (way, "shared") in reached["shared"] and (way, "global") in reached["global"]
    assert {place for _, place in reached["team"]} == {"team"} and {place for _, place in reached["global"]} == {"global"}
