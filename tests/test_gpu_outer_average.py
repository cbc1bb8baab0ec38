"""The Jacobian of the outer average on both sides of its dispatch: sums in register tiles (as many tiles as threads at
most, one to eight groups of threads) and a thread per feature; coefficient rows with and without padding."""
import numpy as np
import pytest

from oracle import modes
from oracle.soap import GTO, SoapOracle
from soap_inputs import multispecies_box
from test_gpu_parity import JAC_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# tiles ceil(n/4) ceil(S n/2) (l+1): 1 (eight groups), 12, 126, 216, 256, 260, 288, 396 and more
@pytest.mark.parametrize("n_species,n_max,l_max", [(1, 1, 0), (2, 3, 3), (3, 7, 5), (2, 9, 7), (4, 8, 7), (1, 13, 8), (4, 8, 8), (2, 12, 10), (8, 4, 3), (2, 16, 0)])
def test_tiles_and_features(n_species, n_max, l_max):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05709_b200 as pkg
    s = multispecies_box(30, 3)
    species = [1, 6, 7, 8, 9, 14, 16, 17][:n_species]
    s.numbers = np.random.default_rng(2).choice(species, size=s.n_atoms).astype(np.int32)
    args = (species, 4.0, n_max, l_max, 0.5, GTO, (True, True, True))
    soap, oracle = pkg.Soap(*args), SoapOracle(*args)
    pos, num = torch.from_numpy(s.positions).cuda(), torch.from_numpy(s.numbers).cuda()
    for cross in (True, False):
        if not cross:
            soap, oracle = pkg.Soap(*args, crossover=False), SoapOracle(*args, crossover=False)
        _, ref = modes.average_derivatives(oracle, "outer", s.positions, s.numbers, s.cell)
        _, jac = soap.derivatives_average("outer", pos, num, s.cell)
        soap.status()
        err = np.abs(jac.cpu().numpy().astype(np.float64) - ref).max(axis=(0, 1))
        # single columns cancel for all thirty atoms at once: the scale is at least 1e-3 of the output's largest entry
        scale = np.maximum(np.abs(ref).max(axis=(0, 1)), 1e-3 * np.abs(ref).max())
        assert float((err / scale).max()) < JAC_TOL
        again = soap.derivatives_average("outer", pos, num, s.cell)[1]
        assert torch.equal(again, jac)
