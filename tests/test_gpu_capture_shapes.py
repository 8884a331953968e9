"""A matvec recorded into a CUDA graph for a state count that has never run before, on a term set that
another state count has used (which uploaded it): the recording builds the layout that this count
needs, and the replay equals the oracle."""
import numpy as np
import pytest

from helpers import TOL, rel, to_dev, torch_or_skip
from oracle import hamiltonian as hm
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B", [("c64", 1), ("c64", 2), ("c64", 4), ("c64", 7), ("c64", 8), ("c64", 16),
                                     ("c128", 1), ("c128", 2)])
@pytest.mark.parametrize("N", [20, 26])
def test_capture_of_a_new_state_count(N, dtype, B):
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    syk.syk_autotune_reset()
    J = inputs.couplings(N, 8)
    terms = syk.syk_build_terms(N, J)
    syk.syk_apply_H(terms, 0, to_dev(torch, inputs.random_states(N, 12, 3), "c64"))  # uploads the term set
    psi = inputs.random_states(N, B, 9)
    x = to_dev(torch, psi, dtype)
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        syk.syk_apply_H(terms, 0, x, out=y)
    H = hm.H_sector_sparse(N, J, 0)
    for _ in range(2):
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert rel(y.cpu().numpy().reshape(-1, B), H @ psi.T) < TOL[dtype]
    # the same count outside a graph, on what the recording built
    z = syk.syk_apply_H(terms, 0, x).cpu().numpy()
    assert np.array_equal(z, y.cpu().numpy())
