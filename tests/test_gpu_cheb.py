"""The Chebyshev evaluation of the Krylov projection's exponential (convergence checks, step
selection and combination coefficients) against the oracle's exact evolution: steps from 1e-9 to
beyond the expansion's range (|z| r > 90, where the eigendecomposition takes over), real and
imaginary time and both, bases that cover the step at once, bases that have to be restarted (the
step search) and bases that reach an invariant subspace.

Bound: the suite's complex128 tolerance 1e-10 of the largest amplitude; the Krylov tolerance is
1e-12 a basis and the expansion's own error about 1e-14 (its sums in FP64 against an
eigendecomposition)."""
import numpy as np
import pytest

from helpers import TOL, rel, to_dev, torch_or_skip
from oracle import evolve
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu

STEPS = [1e-9j, 1e-4, -0.1j, 0.7j, -2.5, 3.0, -4 - 9j, -40j, 150j, -30.0]


@pytest.mark.parametrize("N", [8, 14])
@pytest.mark.parametrize("m", [4, 17, 40, 64])
def test_expmv_steps_vs_exact(N, m):
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    J = inputs.couplings(N, 21)
    terms = syk.syk_build_terms(N, J)
    psi = inputs.random_states(N, 3, 22)
    ref = evolve.SectorSystem(N, J)
    for z in STEPS:
        if m == 4 and abs(z) > 10:
            continue  # thousands of bases
        y, _ = syk.syk_expmv(terms, 1, complex(z), to_dev(torch, psi, "c128"), krylov_dim=m, tol=1e-12)
        assert rel(y.cpu().numpy(), ref.expmv(complex(z), psi.T, 1)) < TOL["c128"], z
        y, _ = syk.syk_expmv(terms, 1, complex(z), to_dev(torch, psi, "c64"), krylov_dim=m, tol=1e-7)
        assert np.isfinite(y.cpu().numpy()).all(), z


def test_zero_columns_and_zero_hamiltonian():
    """A zero state and H = 0 (r = 0: nothing to expand) stay what they are."""
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    N = 10
    psi = inputs.random_states(N, 2, 5)
    psi[1] = 0.0
    x = to_dev(torch, psi, "c128")
    terms = syk.syk_build_terms(N, inputs.couplings(N, 4))
    y, _ = syk.syk_expmv(terms, 0, -1.5j, x, krylov_dim=20, tol=1e-12)
    assert np.all(y.cpu().numpy()[:, 1] == 0.0)
    zero = syk.syk_build_terms(N, np.zeros(inputs.n_terms(N)))
    y, _ = syk.syk_expmv(zero, 0, -1.5j, x, krylov_dim=20, tol=1e-12)
    assert rel(y.cpu().numpy(), psi.T) < 1e-14
