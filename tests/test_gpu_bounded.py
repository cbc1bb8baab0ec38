"""Small calls that size their own outputs, which wait once (soap_derivatives_bounded): against the calls into buffers."""
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


def both(pkg, monkeypatch, soap, other, call, *args):
    """The call as it is, and with the bound at nothing (a search that is waited for); the first must take the short way."""
    seen = []
    whole = soap._lib.soap_derivatives_bounded
    monkeypatch.setattr(soap._lib, "soap_derivatives_bounded", lambda *a: (seen.append(1), whole(*a))[1])
    a = getattr(soap, call)(*args)
    assert seen
    monkeypatch.setattr(pkg.binding, "BOUNDED_BYTES", 0)
    b = getattr(other, call)(*args)
    assert len(seen) == 1
    return a, b


def fields(d):
    return vars(d).values() if hasattr(d, "__dataclass_fields__") else d


@pytest.mark.parametrize("call", ["derivatives", "derivatives_compact", "coefficient_derivatives"])
@pytest.mark.parametrize("n,scale", [(1, 1.0), (2, 1.0), (24, 1.0), (42, 1.0), (42, 0.3)])      # the last: more pairs than a new handle's scratch holds
def test_equals_the_call_that_waits_for_its_rows(pkg, monkeypatch, call, n, scale):
    s = water_cluster(14, 1)
    pos, num = torch.from_numpy((scale * s.positions[:n]).astype(np.float32)).cuda(), torch.from_numpy(s.numbers[:n]).cuda()
    soap, other = (pkg.Soap([1, 8], 5.0, 2, 2, 0.5) for _ in range(2))
    a, b = both(pkg, monkeypatch, soap, other, call, pos, num)
    for x, y in zip(fields(a), fields(b)):
        assert torch.equal(x, y) and x.is_contiguous()
    soap.status()


@pytest.mark.parametrize("weighted", [False, True])
def test_periodic_with_centres(pkg, monkeypatch, weighted):
    s = multispecies_box(60, 0)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    centers = torch.tensor([3, 59, 17], dtype=torch.int32, device="cuda")
    w = {"function": "poly", "r0": 4.0, "c": 1.0, "m": 2.0, "w0": 1.0} if weighted else None
    soap, other = (pkg.Soap([1, 6, 7, 8], 4.0, 2, 2, 0.5, pkg.GTO, (True, True, True), weighting=w) for _ in range(2))
    a, b = both(pkg, monkeypatch, soap, other, "derivatives", pos, num, s.cell, centers)
    for x, y in zip(fields(a), fields(b)):
        assert torch.equal(x, y)


@pytest.mark.parametrize("call", ["derivatives", "derivatives_compact", "coefficient_derivatives"])
@pytest.mark.parametrize("n,centers,scale", [(24, 24, 1.0), (24, 24, 4.0), (120, 8, 1.0), (3000, 1, 1.0)])
def test_results_do_not_keep_the_room(pkg, call, n, centers, scale):
    """Whatever share of its room a call fills, its result holds at most twice the bytes of its rows."""
    s = water_cluster((n + 2) // 3, 1)
    pos, num = torch.from_numpy((scale * s.positions[:n]).astype(np.float32)).cuda(), torch.from_numpy(s.numbers[:n]).cuda()
    soap = pkg.Soap([1, 8], 4.0, 2, 2, 0.5)
    d = getattr(soap, call)(pos, num, None, torch.arange(centers, dtype=torch.int32, device="cuda"))
    rows = int(d.row_ptr[-1])
    assert d.jacobian.shape[0] == d.row_atom.shape[0] == rows > 0
    again = getattr(soap, call)(pos, num, None, torch.arange(centers, dtype=torch.int32, device="cuda"))     # (the other way, after an empty room)
    for x, y in ((d.jacobian, again.jacobian), (d.row_atom, again.row_atom)):
        assert x.is_contiguous() and x.untyped_storage().nbytes() <= 2 * x.nbytes and torch.equal(x, y)


def test_errors(pkg):
    s = water_cluster(4, 0)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    soap = pkg.Soap([1, 8], 5.0, 2, 2, 0.5)
    bad = num.clone()
    bad[3] = 7
    with pytest.raises(pkg.SoapError) as e:
        soap.derivatives(pos, bad)
    assert e.value.code == -2
    assert soap.status()[1] >= 12 and soap.derivatives(pos, num).jacobian.shape[0] > 0
    out = torch.empty(100, device="cuda")
    with pytest.raises(pkg.SoapError) as e:                        # room for fewer rows than there could be
        soap._check(soap._lib.soap_derivatives_bounded(soap._h, 0, pos.data_ptr(), num.data_ptr(), 12, None, None, 12, out.data_ptr(), None,
                                                       out.data_ptr(), 143, out.data_ptr(), out.data_ptr(), None, soap._stream()))
    assert e.value.code == -3
