"""Several handles in one process."""
import pytest

from soap_inputs import multispecies_box, water_cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["derivatives", "coefficient_derivatives"])
def test_a_handle_of_fewer_species_takes_nothing_from_another(call):
    """Two handles of one (n_max, l_max) share their kernels; the one with fewer species needs less shared memory, and
    setting it up must not lower the limit that the other one launches with."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    box, water = multispecies_box(100, 0), water_cluster(20, 0)
    big = pkg.Soap([1, 6, 7, 8], 4.0, 8, 6, 0.5, pkg.GTO, (True, True, True))
    pos, num = torch.from_numpy(box.positions).cuda(), torch.from_numpy(box.numbers).cuda()
    first = getattr(big, call)(pos, num, box.cell)
    small = pkg.Soap([8], 4.0, 8, 6, 0.5)
    oxygen = torch.from_numpy(water.positions[::3].copy()).cuda()
    getattr(small, call)(oxygen, torch.full((20,), 8, dtype=torch.int32, device="cuda"))
    again = getattr(big, call)(pos, num, box.cell)
    assert torch.equal(first.jacobian, again.jacobian)


def test_a_kernel_may_be_launched_first_inside_a_capture():
    """A handle loads and prepares a kernel when it first launches it; after soap_neighbors has planned, that may be while a
    graph is recorded."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    water = water_cluster(60, 0)
    pos, num = torch.from_numpy(water.positions).cuda(), torch.from_numpy(water.numbers).cuda()
    args = ([1, 8], 4.0, 11, 5, 0.5)                                          # a basis that no other test uses
    soap = pkg.Soap(*args)
    _, rows = soap.neighbors(pos, num)
    n, f = water.n_atoms, soap.n_features
    out = (torch.zeros((n, f), device="cuda"), torch.zeros((rows, 3, f), device="cuda"), torch.zeros(n + 1, dtype=torch.int64, device="cuda"),
           torch.zeros(rows, dtype=torch.int32, device="cuda"))
    desc = torch.zeros((n, f), device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        soap.derivatives_into(pos, num, None, None, *out)
        soap.descriptor(pos, num, out=desc)
    graph.replay()
    torch.cuda.synchronize()
    direct = pkg.Soap(*args)
    want = direct.derivatives(pos, num)
    assert torch.equal(out[1], want.jacobian) and torch.equal(out[3], want.row_atom) and torch.equal(desc, direct.descriptor(pos, num))
