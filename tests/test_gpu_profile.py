"""The library's own timing of a call's two parts."""
import pytest

from soap_inputs import water_cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WEIGHTING = {"function": "poly", "r0": 6.0, "c": 1.0, "m": 2.0, "w0": 1.0}


@pytest.mark.parametrize("weighting", [None, WEIGHTING], ids=["plain", "weighted"])
@pytest.mark.parametrize("call", ["derivatives", "derivatives_compact", "coefficient_derivatives", "derivatives_at", "derivatives_batch"])
def test_a_call_that_sizes_its_outputs_reports_its_search(call, weighting):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    s = water_cluster(500, 0)
    soap = pkg.Soap([1, 8], 6.0, 4, 3, 0.5, weighting=weighting)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    ptr = torch.tensor([0, 600, s.n_atoms], dtype=torch.int64, device="cuda")
    run = {"derivatives_at": lambda: soap.derivatives_at(pos, num, pos + 0.1), "derivatives_batch": lambda: soap.derivatives_batch(pos, num, ptr)}
    run = run.get(call, lambda: getattr(soap, call)(pos, num))
    # a descriptor of the same structure runs the same kind of search in one call
    alone = {"derivatives_at": lambda: soap.derivatives_at(pos, num, pos + 0.1, jacobian=False),
             "derivatives_batch": lambda: soap.derivatives_batch(pos, num, ptr, jacobian=False)}.get(call, lambda: soap.descriptor(pos, num))
    soap.profile(True)
    times = {}
    for name, f in (("sized", run), ("alone", alone), ("again", run)):
        read = []
        for _ in range(5):
            whole = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            whole[0].record()
            f()
            whole[1].record()
            search, center = soap.profile_read()
            whole[1].synchronize()
            assert search > 0 and center > 0 and search + center <= whole[0].elapsed_time(whole[1]) + 1e-3
            read.append(search)
        times[name] = min(read[1:])
    # sorting and row pointers are extra; the search of the whole structure is in both
    assert times["sized"] > 0.5 * times["alone"] and times["again"] > 0.5 * times["alone"]
