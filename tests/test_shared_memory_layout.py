"""The shared-memory layout of the per-centre derivative kernels over all bases the library takes: host arithmetic,
compiled from the library's own headers."""
import os
import subprocess

from paper_2609_05709_b200 import build

PROGRAM = r"""
#include <cstdio>
#include "smem_plan.h"
using namespace soap;
int main() {
    const size_t max_smem = 227 * 1024;                        // what a CTA of this architecture may have
    int bases = 0, planned = 0;
    for (int S = 1; S <= kMaxSpecies; ++S)
        for (int n = 1; n <= 16; ++n)
            for (int l = 0; l <= 12; ++l) {
                const int L1 = l + 1, LM = L1 * L1, LMP = LM | 1, NCH = n * L1, CT = S * n * LMP;
                if (n * LM > kMaxElements) continue;
                ++bases;
                for (int weighted = 0; weighted < 2; ++weighted)
                    for (const int warps : {8, 4}) {
                        int P = 0;
                        size_t bytes = 0;
                        if (!plan_chunk(S, n, l, weighted, warps, 0, max_smem, P, bytes)) continue;
                        ++planned;
                        const SmemLayout o = make_layout(S, n, l, P, warps, weighted);
                        bool ok = P >= 4 && (size_t)o.total * 4 == bytes;
                        // the regions one after the other, on 16-byte boundaries, with room for what the kernel puts there
                        const int starts[] = {o.c, o.geo, o.tri, o.xdec, o.zero, o.D, o.sSD, o.sG};
                        for (const int at : starts) ok = ok && at % 4 == 0;
                        const int uv = warps * S * NCH * 4;
                        ok = ok && o.c == 0 && o.geo >= CT && o.tri >= o.geo + kGeoWords + (weighted ? 2 * kGeoPairs : 0);
                        ok = ok && 2 * (o.xdec - o.tri) >= n * (n + 1) / 2 * L1 && 2 * (o.zero - o.xdec) >= (cross_table_wanted(S, n, l) ? n * NCH : 0);
                        ok = ok && o.D >= o.zero + zero_words(S, n, l) && o.wUV == o.D;
                        ok = ok && o.sG >= o.sSD + 4 * P * LMP && o.total >= o.sG + 2 * P * (NCH + (row_table_wanted(n, l) ? 1 : 0));
                        // the slab lies behind everything that is still needed when it is written (coefficients, geometry,
                        // decode tables, zeros, D), and apart from what stays staged where pass 2 relies on that
                        ok = ok && o.slab % 4 == 0 && o.slab >= o.D + 3 * CT && o.slab >= o.wUV + uv && o.slab + o.slab_words <= o.total;
                        if (o.keep) ok = ok && o.slab + o.slab_words <= o.sSD;
                        // rows by the table of operands: the zero behind a pair's channels, in sG, is never written again
                        // (with crossover off: `t`; with crossover the layout does not ask, and the features must fit before it)
                        const int F = S * n * (S * n + 1) / 2 * L1;
                        if (row_table_wanted(n, l) && F <= kKeepFeatures) ok = ok && o.slab + (4 * F < o.slab_words ? 4 * F : o.slab_words) <= o.sG;
                        const SmemLayout t = make_layout(S, n, l, P, warps, weighted, true);
                        ok = ok && t.slab_words > 0 && t.slab + t.slab_words <= t.sG && t.slab == o.slab && t.sG == o.sG && t.total == o.total;
                        if (!ok) printf("species %d n_max %d l_max %d weighted %d warps %d\n", S, n, l, weighted, warps);
                    }
            }
    fprintf(stderr, "%d %d\n", bases, planned);
}
"""


def test_regions_of_the_layout(tmp_path):
    (tmp_path / "layout.cpp").write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", cuda, str(tmp_path / "layout.cpp"), "-o", str(tmp_path / "layout")], check=True)
    out = subprocess.run([str(tmp_path / "layout")], check=True, capture_output=True, text=True)
    assert out.stdout == ""
    bases, planned = map(int, out.stderr.split())
    assert bases > 1000 and planned > 2 * bases
