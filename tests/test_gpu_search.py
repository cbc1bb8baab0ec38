"""The search whose totals come back to the host, and the derivatives of what it found (soap_search_start,
soap_search_finish, soap_derivatives_found), through the calls of the binding that size their own outputs."""
import numpy as np
import pytest

from soap_inputs import multispecies_box, water_cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as p
    return p


def dev(s):
    return torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()


def into(soap, pos, num, cell, c, rows):
    out = (torch.empty((c, soap.n_features), device="cuda"), torch.empty((rows, 3, soap.n_features), device="cuda"),
           torch.empty(c + 1, dtype=torch.int64, device="cuda"), torch.empty(rows, dtype=torch.int32, device="cuda"))
    soap.derivatives_into(pos, num, cell, None, *out)
    soap.status()
    return out


# the brute-force search (up to 512 atoms) and the cell lists of one CTA (up to 4096), of a cluster and of many launches
@pytest.mark.parametrize("molecules", [1, 8, 171, 400, 5600])
def test_sized_call_equals_the_call_into_buffers(pkg, molecules):
    s = water_cluster(molecules, 1)
    soap = pkg.Soap([1, 8], 4.0, 3, 2, 0.5)
    pos, num = dev(s)
    a = soap.derivatives(pos, num)
    b = into(soap, pos, num, None, s.n_atoms, a.jacobian.shape[0])
    for x, y in zip((a.descriptor, a.jacobian, a.row_ptr, a.row_atom), b):
        assert torch.equal(x, y)
    assert int(a.row_ptr[-1]) == a.jacobian.shape[0]


def test_more_pairs_than_the_scratch_holds(pkg):
    """A denser structure of a size that was planned: the search grows the scratch and runs again."""
    loose, dense = water_cluster(60, 0), water_cluster(60, 0)
    dense.positions = (dense.positions * 0.6).astype(np.float32)
    args = ([1, 8], 5.0, 3, 2, 0.5)
    soap, fresh = pkg.Soap(*args), pkg.Soap(*args)
    soap.derivatives(*dev(loose))
    a, b = soap.derivatives(*dev(dense)), fresh.derivatives(*dev(dense))
    assert torch.equal(a.jacobian, b.jacobian) and torch.equal(a.row_ptr, b.row_ptr)
    soap.status()


def test_device_side_error_is_raised_and_cleared(pkg):
    s = water_cluster(8, 0)
    soap = pkg.Soap([1, 8], 5.0, 2, 2, 0.5)
    pos, num = dev(s)
    bad = num.clone()
    bad[3] = 7
    with pytest.raises(pkg.SoapError) as e:
        soap.derivatives(pos, bad)
    assert e.value.code == -2
    soap.status()
    assert soap.derivatives(pos, num).jacobian.shape[0] > 0


def test_derivatives_of_a_search_need_that_search(pkg):
    s = multispecies_box(60, 0)
    soap = pkg.Soap([1, 6, 7, 8], 4.0, 2, 2, 0.5, pkg.GTO, (True, True, True))
    pos, num = dev(s)
    cell, cellp = soap._cell(s.cell)
    out = torch.empty(1, device="cuda")

    def found(n):
        soap._check(soap._lib.soap_derivatives_found(soap._h, 0, pos.data_ptr(), n, cellp, None, None, n, out.data_ptr(), None,
                                                     out.data_ptr(), 1, out.data_ptr(), out.data_ptr(), soap._stream()))

    def finish(n):
        out64 = torch.empty(n + 1, dtype=torch.int64, device="cuda")
        soap._check(soap._lib.soap_search_finish(soap._h, pos.data_ptr(), num.data_ptr(), n, cellp, None, None, n, None, 0,
                                                 out64.data_ptr(), None, None, soap._stream()))

    for call in (found, finish):
        with pytest.raises(pkg.SoapError) as e:           # no search yet
            call(60)
        assert e.value.code == -1
    soap.derivatives(pos, num, s.cell)
    with pytest.raises(pkg.SoapError):                     # a search of another size
        found(59)
    soap.derivatives(pos, num, s.cell)
    soap.descriptor(pos, num, s.cell)                      # a call in between
    for call in (found, finish):
        with pytest.raises(pkg.SoapError):
            call(60)


def all_pairs(pos, r_cut):
    """(pair_ptr, pair_atom) of a non-periodic structure: a k-d tree in fp64, neighbours in atom order."""
    from scipy.spatial import cKDTree
    x = pos.astype(np.float64)
    lists = cKDTree(x).query_ball_point(x, r_cut, return_sorted=True)
    lists = [[j for j in l if j != i] for i, l in enumerate(lists)]
    return np.concatenate([[0], np.cumsum([len(l) for l in lists])]), np.array([j for l in lists for j in l], np.int64)


def check_search(pkg, pos, r_cut):
    ptr, atom = all_pairs(pos, r_cut)
    soap = pkg.Soap([1], r_cut, 1, 0, 0.5)
    p, num = torch.from_numpy(pos).cuda(), torch.ones(len(pos), dtype=torch.int32, device="cuda")
    for _ in range(2):                                       # the second call knows how many pairs a centre has
        got_ptr, got_atom, _ = soap.neighbor_list(p, num)
        assert np.array_equal(got_ptr.cpu().numpy(), ptr) and np.array_equal(got_atom.cpu().numpy(), atom)
        d = soap.derivatives(p, num)
        assert np.array_equal(d.row_ptr.cpu().numpy(), ptr + np.arange(len(pos) + 1))
        row_atom = d.row_atom.cpu().numpy()
        for i in (0, len(pos) // 2, len(pos) - 1):
            a, b = ptr[i] + i, ptr[i + 1] + i + 1
            assert np.array_equal(row_atom[a:b], np.sort(np.append(atom[ptr[i]:ptr[i + 1]], i)))


# one, two, four and eight CTAs of the brute-force search; one CTA, a cluster and many launches for the cell list;
# one CTA and a cluster for the row pointers, and the tiled scan
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 127, 129, 255, 257, 511, 512, 513, 2369, 4095, 4096, 4097, 8193, 32768, 32769, 65536, 65537])
def test_sizes_at_which_the_search_changes(pkg, n):
    rng = np.random.default_rng(n)
    edge = (n / 0.6) ** (1 / 3)
    check_search(pkg, (rng.random((n, 3)) * edge).astype(np.float32), 1.7)


@pytest.mark.parametrize("n_ball,spread", [(100, 1), (128, 1), (129, 40), (300, 150), (512, 1), (513, 90), (300, 100000)])
def test_sort_of_a_centre_s_pairs(pkg, n_ball, spread):
    """Neighbours whose indices are consecutive, evenly spread, or crowded at one end of a long range."""
    rng = np.random.default_rng(spread)
    n = max(20000, n_ball * min(spread, 150) + 1)
    pos = (rng.random((n, 3)) * 1000.0 + 50.0).astype(np.float32)
    ids = np.arange(n_ball) * (spread if spread <= 150 else 1)
    if spread > 150:
        ids[-1] = n - 1
    pos[ids] = (rng.random((n_ball, 3)) * 1.0).astype(np.float32)
    check_search(pkg, pos, 2.5)


@pytest.mark.parametrize("n", [7, 60, 431, 2368, 2369, 4097])
@pytest.mark.parametrize("pbc", [(True, True, True), (True, False, True)])
def test_periodic_search_of_few_and_many_atoms(pkg, n, pbc):
    """With and without a free axis, one and several candidates per lane in flight, against a k-d tree over replicas."""
    from scipy.spatial import cKDTree
    rng = np.random.default_rng(n)
    edge, r_cut = (n / 0.3) ** (1 / 3), 2.2
    cell = np.eye(3) * edge
    pos = (rng.random((n, 3)) * edge).astype(np.float32)
    soap = pkg.Soap([1], r_cut, 1, 0, 0.5, pkg.GTO, pbc)
    p, num = torch.from_numpy(pos).cuda(), torch.ones(n, dtype=torch.int32, device="cuda")
    images = [(a, b, c) for a in (-1, 0, 1) for b in ((-1, 0, 1) if pbc[1] else (0,)) for c in (-1, 0, 1)]
    x = pos.astype(np.float64)
    tree = cKDTree(np.concatenate([x + np.array(t) @ cell for t in images]))
    want = [sorted((j % n, *images[j // n]) for j in near if j != i + n * images.index((0, 0, 0)))
            for i, near in enumerate(tree.query_ball_point(x, r_cut))]
    for _ in range(2):
        ptr, atom, shift = (t.cpu().numpy() for t in soap.neighbor_list(p, num, cell))
        got = np.concatenate([atom[:, None], shift], axis=1)
        assert ptr[-1] == sum(len(w) for w in want)
        for i in range(n):
            assert got[ptr[i]:ptr[i + 1]].tolist() == [list(w) for w in want[i]]
