"""The descriptor kernel where its dispatch changes: teams of four and of two warps per centre, a warp per centre, the
table in shared memory; chunks of 16 and of 32 pairs; feature rows that the copy engine takes and rows that it cannot."""
import numpy as np
import pytest

from oracle.soap import GTO, SoapOracle
from soap_inputs import multispecies_box, water_cluster
from test_gpu_parity import DESC_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as p
    return p


def col_err(a, ref):
    """Largest error over the column's largest magnitude, which counts as 1e-3 of the output's largest entry at least: the
    bound include/soap.h states for few centres, whose columns can all be small at once."""
    a = np.asarray(a, np.float64)
    return float((np.abs(a - ref).max(axis=0) / np.maximum(np.abs(ref).max(axis=0), 1e-3 * np.abs(ref).max())).max())


def check(pkg, s, args, sample, centers=None):
    soap, oracle = pkg.Soap(*args), SoapOracle(*args)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    cen = None if centers is None else torch.tensor(centers, dtype=torch.int32, device="cuda")
    got = soap.descriptor(pos, num, s.cell, cen)
    soap.status()
    of = [k if centers is None else centers[k] for k in sample]
    ref = oracle.descriptor(s.positions, s.numbers, s.cell, of)
    assert bool(torch.isfinite(got).all())
    assert col_err(got[list(sample)].cpu().numpy(), ref) < DESC_TOL
    return got


# with 148 SMs: up to 592 centres a team of four, up to 740 a team of two, then a warp per centre
@pytest.mark.parametrize("n_centers", [1, 147, 592, 593, 740, 741, 1200])
@pytest.mark.parametrize("n_max,l_max", [(8, 6), (3, 2), (5, 4), (12, 7)])
def test_centre_counts(pkg, n_centers, n_max, l_max):
    s = water_cluster(400, 1)
    args = ([1, 8], 5.0, n_max, l_max, 0.5, GTO)
    rng = np.random.default_rng(n_centers)
    centers = rng.permutation(s.n_atoms)[:n_centers].tolist()
    sample = sorted({0, n_centers // 3, n_centers // 2, n_centers - 1})
    a = check(pkg, s, args, sample, centers)
    full = check(pkg, s, args, [0, 600, 1199])
    # one row by different kernels: sums in another order
    scale = full.abs().max(dim=0).values.clamp_min(1e-3 * float(full.abs().max()))
    assert float(((a - full[centers]).abs() / scale).max()) < DESC_TOL


@pytest.mark.parametrize("n_species", [1, 3, 8])
@pytest.mark.parametrize("n_max,l_max", [(1, 0), (4, 1), (7, 3), (8, 4), (4, 8), (13, 2), (2, 12)])
def test_bases_and_species_counts(pkg, n_species, n_max, l_max):
    """Tiles of one to eight species (three: a tile whose rows are no power of two), more blocks than the table of blocks holds."""
    s = multispecies_box(60, 2)
    species = [1, 6, 7, 8, 9, 14, 16, 17][:n_species]
    s.numbers = np.random.default_rng(1).choice(species, size=s.n_atoms).astype(np.int32)
    args = (species, 4.0, n_max, l_max, 0.5, GTO, (True, True, True))
    check(pkg, s, args, [0, 17, 59])


def test_centres_with_no_one_few_and_very_many_neighbours(pkg):
    """A lone atom, a pair, and several groups of 64 pairs in one call, on many and on few centres."""
    rng = np.random.default_rng(0)
    for n_ball in (150, 800):
        s = water_cluster(1, 0)
        ball = rng.random((n_ball, 3)) * 2.2
        s.positions = np.concatenate([ball, [[50, 0, 0], [80, 0, 0], [81, 0, 0]]]).astype(np.float32)
        s.numbers = rng.choice([1, 8], size=n_ball + 3).astype(np.int32)
        check(pkg, s, ([1, 8], 4.0, 6, 5, 0.5, GTO), [0, n_ball - 1, n_ball, n_ball + 1, n_ball + 2])


@pytest.mark.parametrize("n_centers", [600, 745])
def test_options_on_many_centres(pkg, n_centers):
    """The kernel that honours the options, with the table in shared memory (from 592 centres on, no weighting) and not."""
    from oracle import modes
    s = water_cluster(250, 4)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    centers = np.random.default_rng(3).permutation(s.n_atoms)[:n_centers].tolist()
    cen = torch.tensor(centers, dtype=torch.int32, device="cuda")
    sample = [0, 11, n_centers - 1]
    of = [centers[k] for k in sample]
    args = ([1, 8], 4.5, 6, 5, 0.5, GTO)
    soap, oracle = pkg.Soap(*args), SoapOracle(*args)
    got = soap.coefficients(pos, num, None, cen)
    ref = modes.coefficient_derivatives(oracle, s.positions, s.numbers, None, of).descriptor
    assert col_err(got[sample].cpu().numpy(), ref) < DESC_TOL
    weighting = {"function": "pow", "r0": 3.0, "c": 1.5, "d": 1.0, "m": 2.0, "w0": 0.7}
    for kw in ({"crossover": False}, {"weighting": weighting}):
        soap, oracle = pkg.Soap(*args, **kw), SoapOracle(*args, **kw)
        got = soap.descriptor(pos, num, None, cen)
        assert col_err(got[sample].cpu().numpy(), oracle.descriptor(s.positions, s.numbers, None, of)) < DESC_TOL


# sixteen warps without the radial table in shared memory, ten or thirteen with it: which of the two runs depends on the
# warps that a second round of centres would keep busy
@pytest.mark.parametrize("crossover", [True, False])
@pytest.mark.parametrize("n_centers", [1480, 1481, 1850, 1851, 2368, 2369])
@pytest.mark.parametrize("n_max,l_max,sigma", [(8, 8, 0.4), (4, 9, 0.5)])
def test_rounds_of_centres(pkg, n_max, l_max, sigma, n_centers, crossover):
    s = water_cluster(100, 1)
    args = ([1, 8], 4.8, n_max, l_max, sigma, GTO)
    soap, oracle = pkg.Soap(*args, crossover=crossover), SoapOracle(*args, crossover=crossover)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    centers = np.random.default_rng(n_centers).integers(0, s.n_atoms, n_centers)
    got = soap.descriptor(pos, num, None, torch.from_numpy(centers.astype(np.int32)).cuda())
    few = soap.descriptor(pos, num)
    scale = few.abs().max(dim=0).values.clamp_min(1e-3 * float(few.abs().max()))
    assert float(((got - few[torch.from_numpy(centers).cuda()]).abs() / scale).max()) < DESC_TOL
    sample = [0, 1479, n_centers - 1]
    ref = oracle.descriptor(s.positions, s.numbers, None, centers[sample].tolist())
    assert col_err(got[sample].cpu().numpy(), ref) < DESC_TOL


# a centre's tile without its padding, at l_max 8 with n_max 13 to 16, and beside it
@pytest.mark.parametrize("n_species,n_max,l_max", [(1, 13, 8), (2, 14, 8), (6, 16, 8), (2, 12, 8), (2, 14, 7)])
@pytest.mark.parametrize("n_centers", [90, 1036, 1037, 3000])
def test_padded_and_plain_tiles(pkg, n_species, n_max, l_max, n_centers):
    s = multispecies_box(90, 2)
    species = [1, 6, 7, 8, 9, 14][:n_species]
    s.numbers = np.random.default_rng(2).choice(species, size=s.n_atoms).astype(np.int32)
    args = (species, 4.0, n_max, l_max, 0.5, GTO, (True, True, True))
    centers = np.random.default_rng(n_centers).integers(0, s.n_atoms, n_centers).tolist()
    got = check(pkg, s, args, [0, n_centers // 2, n_centers - 1], centers)
    few = check(pkg, s, args, [0, 50, 89])
    scale = few.abs().max(dim=0).values.clamp_min(1e-3 * float(few.abs().max()))
    assert float(((got - few[centers]).abs() / scale).max()) < DESC_TOL
