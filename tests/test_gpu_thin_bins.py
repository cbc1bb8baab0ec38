"""The search without periodic axes, whose bins are thin along x and whose runs are cut to the sphere: the pairs against the
exact fp64 test over all atoms, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def pairs_of(pos, centers, r_cut):
    """(pair_ptr, pair_atom) by the definition: every operation in fp64 on the fp32 inputs."""
    p = pos.astype(np.float64)
    ptr, atoms = [0], []
    for c in centers:
        d = p - c.astype(np.float64)
        d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        atoms.append(np.nonzero((d2 < r_cut * r_cut) & (d2 > 0.0))[0])
        ptr.append(ptr[-1] + len(atoms[-1]))
    return np.array(ptr), np.concatenate(atoms)


def spread(kind, n, rng):
    """Extents of 0 to some tens of r_cut = 3 per axis: one bin, a few, many; a lattice puts pairs right at the cutoff and atoms
    right on the edges of bins."""
    if kind == "lattice":
        m = int(np.ceil(n ** (1 / 3)))
        return 0.75 * np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    if kind == "clumps":
        return rng.random((n, 3)) * 18 + 1700.0 * (np.arange(n) % 2)[:, None]
    extent = {"cube": (18, 18, 18), "line x": (300, 1, 1), "line y": (1, 300, 1), "line z": (0, 0, 300), "plane": (40, 40, 0),
              "point": (1.4, 1.4, 1.4), "far": (30, 9, 9), "sparse": (150, 150, 150), "long line": (1200, 1, 1)}[kind]
    return rng.random((n, 3)) * extent + (1.0e5 if kind == "far" else -7.0)


@pytest.mark.parametrize("n", [600, 5000, 70000])                # cell list of one CTA, of a cluster, of many launches
@pytest.mark.parametrize("kind", ["cube", "line x", "line y", "line z", "plane", "point", "far", "lattice"])
def test_pairs_are_exact(kind, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if kind == "point" and n > 600:
        n = 700                                                    # (every atom sees every other: beyond the keys kept on chip)
    import paper_2609_05709_b200 as pkg
    rng = np.random.default_rng(n)
    pos = spread(kind, n, rng).astype(np.float32)
    soap = pkg.Soap([1], 3.0, 1, 0, 0.5)
    at = torch.from_numpy(pos).cuda()
    centers = rng.permutation(n)[:300].astype(np.int32)
    ptr, atom, _ = soap.neighbor_list(at, torch.ones(n, dtype=torch.int32, device="cuda"), None, torch.from_numpy(centers).cuda())
    want_ptr, want = pairs_of(pos, pos[centers], 3.0)
    assert np.array_equal(ptr.cpu().numpy(), want_ptr) and np.array_equal(atom.cpu().numpy(), want)


# where the grid is not the one that r_cut asks for: more bins than the scratch holds (158,012 for 70,000 atoms: 500,000 are wanted,
# and 3e8), more than 1024 along an axis (1600), both
@pytest.mark.parametrize("kind,n", [("sparse", 70000), ("long line", 5000), ("long line", 70000), ("clumps", 70000)])
def test_pairs_are_exact_on_cut_grids(kind, n):
    test_pairs_are_exact(kind, n)


@pytest.mark.parametrize("cell", [np.diag([2.0, 0.5, 7.0]), np.array([[9.0, 1.0, 0.0], [0.0, 8.0, 2.0], [1.0, 0.0, 7.0]])], ids=["square", "skew"])
def test_a_cell_without_periodic_axes(cell):
    """The bins follow the cell's axes then: thin ones only where those are at right angles."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    pos = (np.random.default_rng(1).random((3000, 3)) * 25).astype(np.float32)
    soap = pkg.Soap([1], 3.0, 1, 0, 0.5)
    ptr, atom, _ = soap.neighbor_list(torch.from_numpy(pos).cuda(), torch.ones(3000, dtype=torch.int32, device="cuda"), cell)
    want_ptr, want = pairs_of(pos, pos, 3.0)
    assert np.array_equal(ptr.cpu().numpy(), want_ptr) and np.array_equal(atom.cpu().numpy(), want)


def test_sites_outside_the_atoms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    rng = np.random.default_rng(2)
    pos = (rng.random((4000, 3)) * 15).astype(np.float32)
    sites = (rng.random((500, 3)) * 25 - 5).astype(np.float32)
    soap = pkg.Soap([1], 3.0, 1, 0, 0.5)
    d = soap.derivatives_at(torch.from_numpy(pos).cuda(), torch.ones(4000, dtype=torch.int32, device="cuda"), torch.from_numpy(sites).cuda())
    want_ptr, want = pairs_of(pos, sites, 3.0)
    assert np.array_equal(d.row_ptr.cpu().numpy(), want_ptr) and np.array_equal(d.row_atom.cpu().numpy(), want)
