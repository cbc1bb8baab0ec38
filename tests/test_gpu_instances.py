"""Every n_max the derivative kernels are compiled for, and its neighbours that are read at run time, against the
oracle: the plain kernels, the ones that honour the options, the ones of the averages."""
import numpy as np
import pytest

from oracle import modes
from oracle.soap import GTO, SoapOracle
from soap_inputs import water_cluster
from test_gpu_parity import DESC_TOL, JAC_TOL, col_err

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


@pytest.mark.parametrize("n_max", range(1, 14))
def test_plain_and_optioned_kernels(pkg, n_max):
    s = water_cluster(9, 3)
    pos, num = dev(s)
    for l_max in (1, 3, 5 + n_max % 6):
        args = ([1, 8], 4.5, n_max, l_max, 0.5, GTO)
        options = {"crossover": n_max % 2 == 0, "weighting": {"function": "poly", "r0": 4.5, "c": 1.0, "m": 2.0, "w0": 1.0}}
        for kw in ({}, options):
            soap, oracle = pkg.Soap(*args, **kw), SoapOracle(*args, **kw)
            ref = oracle.derivatives(s.positions, s.numbers, None)
            out = soap.derivatives(pos, num)
            assert np.array_equal(out.row_atom.cpu().numpy(), ref.row_atom)
            assert col_err(out.descriptor.cpu().numpy(), ref.descriptor, 0) < DESC_TOL, (l_max, kw)
            assert col_err(out.jacobian.cpu().numpy(), ref.jacobian, (0, 1)) < JAC_TOL, (l_max, kw)


@pytest.mark.parametrize("mode", ["inner", "outer"])
@pytest.mark.parametrize("n_max", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10])
def test_average_kernels(pkg, mode, n_max):
    s = water_cluster(7, 3)
    pos, num = dev(s)
    for l_max in (2, 3 + n_max % 5):
        args = ([1, 8], 4.5, n_max, l_max, 0.5, GTO)
        soap, oracle = pkg.Soap(*args), SoapOracle(*args)
        _, rj = modes.average_derivatives(oracle, mode, s.positions, s.numbers, None)
        _, gj = soap.derivatives_average(mode, pos, num)
        soap.status()
        assert col_err(gj.cpu().numpy(), rj, (0, 1)) < JAC_TOL, l_max
