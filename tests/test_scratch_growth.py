"""Scratch that cannot grow: the bookkeeping with an allocator that fails (host), and a handle on a full device (GPU)."""
import subprocess

import pytest

from paper_2609_05709_b200 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "scratch.h"
using namespace soap;
static int live = 0;
#define CHECK(x) do { if (!(x)) { printf("after %d allocations: %s\n", good, #x); } } while (0)
int main() {
    for (int good = 0; good <= 3; ++good) {                   // allocations that succeed when the group grows
        void *a = nullptr, *b = nullptr, *c = nullptr;
        int64_t cap = 0;
        int left = 3;
        auto get = [&](void** p, size_t n) { if (left-- <= 0) return false; *p = malloc(n); ++live; return true; };
        auto put = [&](void* p) { free(p); --live; };
        CHECK(regrow_group(cap, 10, {{&a, 40}, {&b, 80}, {&c, 10}}, get, put) && cap == 10 && live == 3);
        left = good;
        const bool grown = regrow_group(cap, 20, {{&a, 80}, {&b, 160}, {&c, 20}}, get, put);
        CHECK(grown == (good == 3));
        if (grown) CHECK(cap == 20 && a && b && c && live == 3);
        else CHECK(cap == 0 && !a && !b && !c && live == 0);
        left = 3;                                             // memory is back
        CHECK(regrow_group(cap, 5, {{&a, 20}, {&b, 40}, {&c, 5}}, get, put) && cap == 5 && a && b && c && live == 3);
        put(a); put(b); put(c);
    }
}
"""


def test_a_group_is_whole_or_gone(tmp_path):
    (tmp_path / "scratch.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, str(tmp_path / "scratch.cpp"), "-o", str(tmp_path / "scratch")], check=True)
    assert subprocess.run([str(tmp_path / "scratch")], check=True, capture_output=True, text=True).stdout == ""


@pytest.mark.gpu
@pytest.mark.parametrize("weighting", [None, {"function": "poly", "r0": 5.0, "c": 1.0, "m": 2.0, "w0": 1.0}], ids=["plain", "weighted"])
@pytest.mark.parametrize("n_atoms,spacing,left", [(12_000_000, 4.0, 1000 << 20), (40_000, 0.7, 300 << 20)], ids=["atoms", "pairs"])
def test_a_handle_on_a_full_device(n_atoms, spacing, left, weighting):
    """The search of a structure whose scratch does not fit reports that, and the handle goes on with others."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    from soap_inputs import water_cluster
    s = water_cluster(8, 0)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    side = round(n_atoms ** (1 / 3)) + 1
    at = torch.arange(n_atoms, device="cuda")
    big_pos = spacing * torch.stack([at // (side * side), at // side % side, at % side], 1).float()
    big_num = torch.full((n_atoms,), 8, dtype=torch.int32, device="cuda")
    soap, other = (pkg.Soap([1, 8], 5.0, 4, 3, 0.5, weighting=weighting) for _ in range(2))
    want = soap.derivatives(pos, num)
    totals = other.neighbors(big_pos, big_num)                               # (and the kernels are loaded)
    del other
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        for _ in range(2):
            with pytest.raises(pkg.SoapError):
                soap.neighbors(big_pos, big_num)
            again = soap.derivatives(pos, num)
            for name in ("descriptor", "jacobian", "row_ptr", "row_atom"):
                assert torch.equal(getattr(again, name), getattr(want, name))
    finally:
        del filler
        torch.cuda.empty_cache()
    assert soap.neighbors(big_pos, big_num) == totals
