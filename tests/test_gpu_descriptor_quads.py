"""The two ways in which the descriptor kernel takes its radial factors from the table (desc_quads), each on both sides of the rule
between them, with the table in shared and in global memory, one warp per centre and several: against the derivative kernel."""
import pytest

from soap_inputs import water_cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


# quads of a pair: 1, 7, 8 (a lane keeps its quad); 9, 6, 10, 12 (pairs); 14, 15, 16, 18 and 20 (a list of quads), 26, 28 and 32 of 32
@pytest.mark.parametrize("n_max,l_max", [(3, 0), (4, 6), (2, 7), (4, 8), (5, 2), (8, 4), (9, 3), (7, 6), (10, 4), (13, 3), (8, 8), (16, 4), (7, 12), (13, 6), (15, 7)])
@pytest.mark.parametrize("molecules,weighting", [(9, None), (300, None), (300, {"function": "poly", "r0": 4.0, "c": 1.0, "m": 2.0, "w0": 1.0})],
                         ids=["team", "shared", "global"])
def test_radial_factors(n_max, l_max, molecules, weighting):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    s = water_cluster(molecules, 2)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    soap = pkg.Soap([1, 8], 4.0, n_max, l_max, 0.5, weighting=weighting)
    got, want = soap.descriptor(pos, num).double(), soap.derivatives(pos, num).descriptor.double()
    # column by column within the parity tolerance, a column's scale floored at 1e-3 of the largest entry (two fp32 builds)
    scale = torch.maximum(want.abs().amax(0), 1e-3 * want.abs().max())
    assert float(((got - want).abs().amax(0) / scale).max()) < TOL
