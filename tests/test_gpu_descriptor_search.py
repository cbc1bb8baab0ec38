"""Descriptors of small structures, whose kernel searches for itself: against the search of the derivative calls, at the edges of
what takes that route."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as p
    return p


def close(a, b):
    """Column by column against the parity tolerance, a column's scale floored at 1e-3 of the largest entry: two orders of summation."""
    a, b = a.double(), b.double()
    scale = torch.maximum(b.abs().amax(0), 1e-3 * b.abs().max())
    return float(((a - b).abs().amax(0) / scale).max()) < TOL


def box(n, edge, seed=0, tilt=0.0):
    rng = np.random.default_rng(seed)
    cell = np.diag([edge] * 3).astype(float)
    cell[1, 0] = cell[2, 1] = tilt
    m = int(np.ceil(n ** (1 / 3)))
    grid = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    frac = (grid[rng.permutation(len(grid))[:n]] + 0.5 + 0.2 * (rng.random((n, 3)) - 0.5)) / m
    frac += rng.integers(-3, 4, (n, 3))                            # atoms outside the cell
    pos = torch.from_numpy((frac @ cell).astype(np.float32)).cuda()
    return pos, torch.from_numpy(rng.choice([1, 6, 8], n).astype(np.int32)).cuda(), cell


# shares of 32 atoms per warp and their remainders, four warps per team, two, and beyond (740 on 148 SMs)
@pytest.mark.parametrize("n", [1, 2, 31, 33, 128, 129, 592, 593, 740, 741, 1030])
@pytest.mark.parametrize("pbc", [(False, False, False), (True, True, True), (True, False, True)], ids=["free", "periodic", "mixed"])
def test_equals_the_search_of_the_derivatives(pkg, n, pbc):
    edge = max(8.2, (n / 0.06) ** (1 / 3))
    pos, num, cell = box(n, edge, n, tilt=0.3)
    soap = pkg.Soap([1, 6, 8], 3.9, 4, 3, 0.5, pkg.GTO, pbc)
    d = soap.derivatives(pos, num, cell)
    pairs, _ = soap.neighbors(pos, num, cell)
    got = soap.descriptor(pos, num, cell)
    assert soap.status() == (pairs, 0)
    assert close(got, d.descriptor)
    assert n > 740 or torch.equal(got, soap.descriptor(pos, num, cell))       # (bit for bit: found in a fixed order)


# heights of two cutoffs, and a little below and above: the nearest image is the only one from there on
@pytest.mark.parametrize("edge", [7.99, 8.0, 8.0001, 8.2])
def test_heights_of_two_cutoffs(pkg, edge):
    pos, num, cell = box(60, edge)
    soap = pkg.Soap([1, 6, 8], 4.0, 3, 2, 0.4, pkg.GTO, (True, True, True))
    d = soap.derivatives(pos, num, cell)
    assert close(soap.descriptor(pos, num, cell), d.descriptor)
    assert soap.status()[0] == soap.neighbors(pos, num, cell)[0]


def test_many_neighbours_and_options(pkg):
    """More neighbours than are held in registers at once, all of them in one warp's share; no crossover."""
    rng = np.random.default_rng(3)
    pos = torch.from_numpy((2.2 * rng.random((300, 3))).astype(np.float32)).cuda()
    num = torch.from_numpy(rng.choice([1, 6], 300).astype(np.int32)).cuda()
    for crossover in (True, False):
        soap = pkg.Soap([1, 6], 5.0, 5, 4, 0.5, crossover=crossover)
        assert close(soap.descriptor(pos, num), soap.derivatives(pos, num).descriptor)


def test_errors_are_reported_and_cleared(pkg):
    pos, num, cell = box(40, 9.0)
    soap = pkg.Soap([1, 6, 8], 4.0, 2, 2, 0.5, pkg.GTO, (True, True, True))
    good = soap.descriptor(pos, num, cell)
    bad = num.clone()
    bad[17] = 7
    soap.descriptor(pos, bad, cell)
    with pytest.raises(pkg.SoapError) as e:
        soap.status()
    assert e.value.code == -2
    away = pos.clone()
    away[5] += 9.0 * 150
    soap.descriptor(away, num, cell)
    with pytest.raises(pkg.SoapError) as e:
        soap.status()
    assert e.value.code == -1
    with pytest.raises(pkg.SoapError):                             # no list to export
        ptr = torch.empty(41, dtype=torch.int64, device="cuda")
        soap._check(soap._lib.soap_neighbor_list(soap._h, ptr.data_ptr(), ptr.data_ptr(), None, 41, soap._stream()))
    assert torch.equal(soap.descriptor(pos, num, cell), good)
    soap.status()


def test_a_denser_structure_than_planned_is_refused(pkg):
    """As where the pairs are kept: planned sizes hold the pairs of the structures seen (and half as many again)."""
    pos, num, _ = box(200, 40.0)
    soap = pkg.Soap([1, 6, 8], 4.0, 2, 2, 0.5)
    soap.neighbors(pos, num)
    soap.descriptor(0.01 * pos, num)
    with pytest.raises(pkg.SoapError) as e:
        soap.status()
    assert e.value.code == -3
    soap.neighbors(0.01 * pos, num)
    soap.descriptor(0.01 * pos, num)
    soap.status()
