"""The two ways in which the descriptor kernel takes its radial factors from the table (desc_quads), each on both sides of the rule
between them, with the table in shared and in global memory, one warp per centre and several: against the derivative kernel.
(test_descriptor_layout.py checks that the bases reach every path; large ones leave the table in global memory in any case.)"""
import pytest

from soap_inputs import water_cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5
R_CUT = 4.0
# quads of a pair: 1 (pairs), 7 and 8 (a lane keeps its quad); 9, 6, 10, 12 (pairs); 14, 15, 16 (kept), 18 and 20 (a list of quads), 26 (a
# list), 28 and 32 (kept)
BASES = [(3, 0), (4, 6), (2, 7), (4, 8), (5, 2), (8, 4), (9, 3), (7, 6), (10, 4), (13, 3), (8, 8), (16, 4), (7, 12), (13, 6), (15, 7)]
MOLECULES = {"team": (9, False), "shared": (300, False), "global": (300, True)}


@pytest.mark.parametrize("n_max,l_max", BASES)
@pytest.mark.parametrize("molecules,weighting", [(m, {"function": "poly", "r0": 4.0, "c": 1.0, "m": 2.0, "w0": 1.0} if w else None) for m, w in MOLECULES.values()],
                         ids=list(MOLECULES))
def test_radial_factors(n_max, l_max, molecules, weighting):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    s = water_cluster(molecules, 2)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    soap = pkg.Soap([1, 8], R_CUT, n_max, l_max, 0.5, weighting=weighting)
    got, want = soap.descriptor(pos, num).double(), soap.derivatives(pos, num).descriptor.double()
    # column by column within the parity tolerance, a column's scale floored at 1e-3 of the largest entry (two fp32 builds)
    scale = torch.maximum(want.abs().amax(0), 1e-3 * want.abs().max())
    assert float(((got - want).abs().amax(0) / scale).max()) < TOL


# teams that search for themselves, of four warps and of two, with one step of the search and several, and more pairs than one group
@pytest.mark.parametrize("n_max,l_max", [(8, 6), (8, 8), (9, 3), (13, 3)])
@pytest.mark.parametrize("molecules", [50, 190, 240])
def test_radial_factors_of_teams(n_max, l_max, molecules):
    test_radial_factors(n_max, l_max, molecules, None)
