"""The calls that compute from a search made before: what they refuse, and that a refusal leaves nothing behind."""
import ctypes as C

import pytest

from soap_inputs import water_cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ERR_INVALID_ARG, ERR_CAPACITY = -1, -3


class Calls:
    """The three calls on one structure, return codes as they are."""

    def __init__(self, pkg, n_molecules):
        s = water_cluster(n_molecules, 0)
        self.soap = pkg.Soap([1, 8], 4.0, 4, 3, 0.5)
        self.pos, self.num, self.n = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda(), s.n_atoms
        self.ptr = torch.empty(self.n + 1, dtype=torch.int64, device="cuda")
        self.search = (self.soap._h, self.pos.data_ptr(), self.num.data_ptr(), self.n, None, None, None, self.n, None, 0, self.ptr.data_ptr())

    def find(self):
        pairs, rows = C.c_int64(), C.c_int64()
        assert self.soap._lib.soap_search_start(*self.search, None) == 0
        assert self.soap._lib.soap_search_finish(*self.search, C.byref(pairs), C.byref(rows), None) == 0
        return rows.value

    def compute(self, kind, rows, capacity):
        width = self.soap.n_coefficients if kind == 2 else self.soap.n_features
        out = [torch.full((self.n, width), 7.0, device="cuda"), torch.full((rows, 3, width), 7.0, device="cuda"), torch.full((rows,), 7, dtype=torch.int32, device="cuda")]
        torch.cuda.synchronize()
        rc = self.soap._lib.soap_derivatives_found(self.soap._h, kind, self.pos.data_ptr(), self.n, None, None, None, self.n, out[0].data_ptr(), None,
                                                   out[1].data_ptr(), capacity, self.ptr.data_ptr(), out[2].data_ptr(), None)
        torch.cuda.synchronize()
        return rc, out


@pytest.fixture(params=[8, 200])
def calls(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    return Calls(pkg, request.param)


def test_too_little_room_is_reported_at_once(calls):
    rows = calls.find()
    rc, out = calls.compute(0, rows, rows - 1)
    assert rc == ERR_CAPACITY and all(bool((o == 7).all()) for o in out)
    calls.soap.status()                                                     # raises if anything were left
    assert calls.compute(0, rows, rows)[0] == 0                             # the search is still at hand
    assert calls.soap.derivatives(calls.pos, calls.num).jacobian.shape[0] == rows


def test_one_search_serves_several_kinds(calls):
    rows = calls.find()
    for kind, want in ((0, calls.soap.derivatives), (2, calls.soap.coefficient_derivatives)):
        calls.find()
        first, second = calls.compute(kind, rows, rows), calls.compute(kind, rows, rows)
        assert first[0] == second[0] == 0
        ref = want(calls.pos, calls.num)
        for got in (first[1], second[1]):
            assert torch.equal(got[0], ref.descriptor) and torch.equal(got[1], ref.jacobian) and torch.equal(got[2], ref.row_atom)


@pytest.mark.parametrize("change", ["crossover", "weighting", "search"])
def test_a_change_takes_the_search_away(calls, change):
    rows = calls.find()
    lib, h = calls.soap._lib, calls.soap._h
    if change == "crossover":
        assert lib.soap_set_crossover(h, 0) == 0
    elif change == "weighting":
        assert lib.soap_set_weighting(h, 1, 4.0, 1.0, 1.0, 2.0, 1.0) == 0
    else:
        calls.soap.descriptor(calls.pos, calls.num)
    assert calls.compute(0, rows, rows)[0] == ERR_INVALID_ARG
    assert calls.compute(0, calls.find(), rows)[0] == 0
