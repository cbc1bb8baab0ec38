"""The search whose totals come back to the host, and the derivatives of what it found (soap_search,
soap_derivatives_found), through the calls of the binding that size their own outputs."""
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


# the brute-force search (up to 512 atoms), the single-CTA cell list (up to 16384) and the tiled one
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

    with pytest.raises(pkg.SoapError) as e:               # no search yet
        found(60)
    assert e.value.code == -1
    soap.derivatives(pos, num, s.cell)
    with pytest.raises(pkg.SoapError):                     # a search of another size
        found(59)
    soap.derivatives(pos, num, s.cell)
    soap.descriptor(pos, num, s.cell)                      # a call in between
    with pytest.raises(pkg.SoapError):
        found(60)
