"""The derivative kernel where its dispatch changes for small bases: CTAs of 128 and 256 threads (740 centres on 148 SMs),
rows by the table of operands and by sweeps (20 channels, 512 features), centres that fit the staging area, do not fit
it, and have more pairs than one batch of geometry; images that share a row."""
import numpy as np
import pytest

from oracle.soap import GTO, POLYNOMIAL, SoapOracle
from soap_inputs import multispecies_box, small_periodic_cell, water_cluster
from test_gpu_parity import DESC_TOL, JAC_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as p
    return p


def col_err(a, ref, axes):
    """Column error with the scale floored at 1e-3 of the output's largest entry (include/soap.h: few centres)."""
    a = np.asarray(a, np.float64)
    return float((np.abs(a - ref).max(axis=axes) / np.maximum(np.abs(ref).max(axis=axes), 1e-3 * np.abs(ref).max())).max())


def check(pkg, s, args, centers, sample, **kw):
    soap, oracle = pkg.Soap(*args, **kw), SoapOracle(*args, **kw)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    out = soap.derivatives(pos, num, s.cell, torch.tensor(centers, dtype=torch.int32, device="cuda"))
    ref = oracle.derivatives(s.positions, s.numbers, s.cell, [centers[k] for k in sample])
    ptr = out.row_ptr.cpu().numpy()
    rows = np.concatenate([np.arange(ptr[k], ptr[k + 1]) for k in sample])
    assert np.array_equal(out.row_atom.cpu().numpy()[rows], ref.row_atom)
    assert col_err(out.descriptor.cpu().numpy()[sample], ref.descriptor, 0) < DESC_TOL
    assert col_err(out.jacobian.cpu().numpy()[rows], ref.jacobian, (0, 1)) < JAC_TOL


@pytest.mark.parametrize("n_centers", [739, 740])
@pytest.mark.parametrize("n_max,l_max", [(1, 0), (2, 2), (2, 9), (4, 3), (4, 4), (3, 5), (4, 5), (5, 3), (6, 4), (8, 3), (5, 5), (8, 2), (2, 10)])
def test_thread_counts_and_rows(pkg, n_centers, n_max, l_max):
    s = water_cluster(250, 2)
    centers = np.random.default_rng(l_max).permutation(s.n_atoms)[:n_centers].tolist()
    check(pkg, s, ([1, 8], 4.5, n_max, l_max, 0.5, GTO), centers, [0, 400, n_centers - 1])


@pytest.mark.parametrize("n_max,l_max", [(2, 2), (3, 3), (4, 3), (4, 2), (2, 9)])
@pytest.mark.parametrize("n_species", [1, 3, 4, 8])
def test_species_counts(pkg, n_max, l_max, n_species):
    """Rows on both sides of the table's 512 features; one species has no cross-species block."""
    s = multispecies_box(80, 1)
    species = [1, 6, 7, 8, 9, 14, 16, 17][:n_species]
    s.numbers = np.random.default_rng(1).choice(species, size=s.n_atoms).astype(np.int32)
    args = (species, 4.0, n_max, l_max, 0.4, POLYNOMIAL, (True, True, True))
    check(pkg, s, args, list(range(80)), [0, 33, 79])
    check(pkg, s, args, list(range(80)) * 10, [0, 333, 799])
    check(pkg, s, args, list(range(80)) * 10, [1, 200], crossover=False)


@pytest.mark.parametrize("repeats", [1, 100])
@pytest.mark.parametrize("n_max,l_max", [(3, 3), (4, 3), (6, 3)])
def test_images_that_share_a_row(pkg, repeats, n_max, l_max):
    """Several images of one atom add up in its row, images of the centre contribute to none."""
    s = small_periodic_cell(0)
    weighting = {"function": "poly", "r0": 4.5, "c": 1.0, "m": 2.0, "w0": 1.0}
    for kw in ({}, {"weighting": weighting}):
        check(pkg, s, ([1, 6, 7, 8], 4.5, n_max, l_max, 0.5, GTO, (True, True, True)), list(range(8)) * repeats, [0, 3, 8 * repeats - 1], **kw)


@pytest.mark.parametrize("n_ball", [8, 31, 48, 97, 129, 300])
@pytest.mark.parametrize("n_max,l_max", [(4, 3), (2, 6), (6, 4)])
def test_neighbour_counts(pkg, n_ball, n_max, l_max):
    """From less than a warp of pairs to more than two batches of geometry per centre, beside lone atoms."""
    rng = np.random.default_rng(n_ball)
    s = water_cluster(1, 0)
    s.positions = np.concatenate([rng.random((n_ball, 3)) * 2.0, rng.random((800, 3)) * 0.5 + 50.0 + 10.0 * np.arange(800)[:, None]]).astype(np.float32)
    s.numbers = rng.choice([1, 8], size=n_ball + 800).astype(np.int32)
    args = ([1, 8], 4.0, n_max, l_max, 0.5, GTO)
    check(pkg, s, args, list(range(n_ball)), [0, n_ball - 1])
    check(pkg, s, args, list(range(n_ball + 800)), [0, n_ball - 1, n_ball, n_ball + 799])


@pytest.mark.parametrize("n_ball", [9, 32, 33, 34, 65])
@pytest.mark.parametrize("n_max,l_max", [(2, 2), (4, 4), (2, 8), (3, 9), (4, 12)])
def test_staging_limits(pkg, n_ball, n_max, l_max):
    """Chunks of up to 32 and of more pairs; with and without a slab of its own (l_max 8 and 9)."""
    test_neighbour_counts(pkg, n_ball, n_max, l_max)


@pytest.mark.parametrize("repeats", [1, 10])
@pytest.mark.parametrize("kw", [{}, {"weighting": {"function": "poly", "r0": 4.0, "c": 1.0, "m": 2.0, "w0": 1.0}}], ids=["plain", "weighted"])
@pytest.mark.parametrize("n_max,l_max", [(4, 0), (4, 1), (3, 0), (2, 2)])
def test_absent_operands_are_zero(pkg, n_max, l_max, kw, repeats):
    """Eight species without crossover: rows by the table of operands though the slab shares the staging area ((4, 0) is
    where the two meet).  Only the block of the neighbour's species may differ from zero in its row."""
    s = multispecies_box(80, 1)
    species = [1, 6, 7, 8, 9, 14, 16, 17]
    s.numbers = np.random.default_rng(1).choice(species, size=s.n_atoms).astype(np.int32)
    args = (species, 4.0, n_max, l_max, 0.4, POLYNOMIAL, (True, True, True))
    centers = list(range(80)) * repeats
    check(pkg, s, args, centers, [0, 33, 79], crossover=False, **kw)
    soap = pkg.Soap(*args, crossover=False, **kw)
    out = soap.derivatives(torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda(), s.cell, torch.tensor(centers, dtype=torch.int32, device="cuda"))
    width = soap.n_features // 8
    atom = out.row_atom.cpu().numpy()
    center = np.repeat(centers, np.diff(out.row_ptr.cpu().numpy()))
    block = np.searchsorted(species, s.numbers[atom])
    jac = out.jacobian.cpu().numpy().reshape(-1, 3, 8, width)
    jac[np.arange(atom.size), :, block] = 0.0
    assert not jac[atom != center].any()
