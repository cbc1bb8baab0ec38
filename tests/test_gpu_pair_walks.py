"""The two walks of the pair kernels, over runs of the sorted atoms and over images, at the edges of what takes which kernel: the pairs
against the exact fp64 test over all atoms and images, bit for bit."""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R_CUT = 3.0


def exact_pairs(pos, cell, pbc, centers):
    """(pair_ptr, atom, shift) by the definition, every operation in fp64 on the fp32 inputs, sorted by (atom, shift)."""
    p = pos.astype(np.float64)
    ptr, found = [0], []
    shifts = list(itertools.product(*[(-2, -1, 0, 1, 2) if f else (0,) for f in pbc]))
    for c in centers:
        d = p - p[c]
        n = []
        for a, b, e in shifts:
            x = d + ((a * cell[0] + b * cell[1]) + e * cell[2])
            d2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
            n += [(int(j), a, b, e) for j in np.nonzero((d2 < R_CUT * R_CUT) & (d2 > 0.0))[0]]
        found += sorted(n)
        ptr.append(len(found))
    found = np.array(found, dtype=np.int64).reshape(-1, 4)
    return np.array(ptr), found[:, 0], found[:, 1:]


# 700 and 3000 atoms lie on both sides of the line between four candidates in flight and one; neighbours: some ten (small key
# buffers), some 110 (large ones) and some 700 (more than either holds, found by a second walk)
@pytest.mark.parametrize("density", [0.1, 1.0, 6.0])
@pytest.mark.parametrize("n", [700, 3000])
@pytest.mark.parametrize("pbc", [(False, False, False), (True, True, True), (False, True, False)], ids=["free", "periodic", "mixed"])
def test_pairs_are_exact(pbc, n, density):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    rng = np.random.default_rng(n)
    edge = (n / density) ** (1 / 3)
    cell = np.diag([edge, 1.1 * edge, 0.9 * edge])
    cell[1, 0] = 0.2 * edge
    pos = (rng.random((n, 3)) @ cell).astype(np.float32)
    at, num = torch.from_numpy(pos).cuda(), torch.ones(n, dtype=torch.int32, device="cuda")
    soap = pkg.Soap([1], R_CUT, 2, 2, 0.5, pkg.GTO, pbc)
    soap.neighbors(at, num, cell)                                 # (the key buffers follow the pairs of the last plan)
    ptr, atom, shift = (x.cpu().numpy() for x in soap.neighbor_list(at, num, cell))
    some = rng.permutation(n)[:40]
    want_ptr, want_atom, want_shift = exact_pairs(pos, cell, pbc, some)
    for i, c in enumerate(some):
        mine, theirs = slice(ptr[c], ptr[c + 1]), slice(want_ptr[i], want_ptr[i + 1])
        assert np.array_equal(atom[mine], want_atom[theirs]) and np.array_equal(shift[mine], want_shift[theirs])
    # the kernels that leave their pairs unsorted: descriptors within the parity tolerance of the sorted ones, column by column, a
    # column's scale floored at 1e-3 of the largest entry (two orders of summation)
    got, want = soap.descriptor(at, num, cell).double(), soap.derivatives(at, num, cell, torch.from_numpy(some.astype(np.int32)).cuda()).descriptor.double()
    scale = torch.maximum(want.abs().amax(0), 1e-3 * want.abs().max())
    assert float(((got[torch.from_numpy(some).cuda()] - want).abs().amax(0) / scale).max()) < 1e-5
    soap.status()
