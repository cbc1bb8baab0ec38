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
