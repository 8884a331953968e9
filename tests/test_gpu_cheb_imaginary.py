"""The Krylov exponential's expansion in imaginary time, where |Re z| r is large (r: half the width of
the projection's spectrum, about 0.74 at N = 14 and 0.8 at N = 16), against the oracle's exact
evolution.  N = 14 with 3 states runs on the one-launch basis of small sectors, N = 16 on the general
path.

Bounds.  A basis leaves an error of at most tol of its result's norm (Saad's estimate), and complex64
about m roundings of 2^-24; rounded couplings and matvecs move the levels by 2^-24 of them.  Later
bases can raise an error against the state by at most 1/|<e|psi>|, e the extreme level that the
evolution projects on.  So the relative error (2-norm) is below
(bases (tol + m 2^-24) + |z| (Emax - Emin) 2^-24) / |<e|psi>|, without the roundings but plus 1e-11 in
complex128."""
import numpy as np
import pytest

from helpers import to_dev, torch_or_skip
from oracle import evolve
from oracle import hamiltonian as hm
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu


def _check(N, z, m, dtype, sector=1, B=3, seed=21):
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    J = inputs.couplings(N, seed)
    terms = syk.syk_build_terms(N, J)
    psi = inputs.random_states(N, B, seed + 1)
    # complex64 squares amplitudes in single precision: keep them in range while they grow
    scale = 1e-17 if dtype == "c64" else 1.0
    tol = 1e-7 if dtype == "c64" else 1e-12
    y, bases = syk.syk_expmv(terms, sector, complex(z), to_dev(torch, psi * scale, dtype), krylov_dim=m, tol=tol)
    y = y.cpu().numpy().astype(np.complex128) / scale
    ref = evolve.SectorSystem(N, J).expmv(complex(z), psi.T, sector)
    E, Q = np.linalg.eigh(hm.H_sector_sparse(N, J, sector).toarray())
    e = Q[:, -1] if z.real > 0 else Q[:, 0]
    over = np.abs(e.conj() @ psi.T) / np.linalg.norm(psi, axis=1)
    rounding = (bases * m + abs(z) * (E[-1] - E[0])) * 2.0 ** -24 if dtype == "c64" else 0.0
    bound = (bases * tol + rounding) / over + (0.0 if dtype == "c64" else 1e-11)
    err = np.linalg.norm(y - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert (err <= bound).all(), (N, z, m, dtype, bases, err, bound)


@pytest.mark.parametrize("N", [14, 16])
@pytest.mark.parametrize("m", [8, 12, 16, 20])
@pytest.mark.parametrize("z", [-60.0, 60.0, -90.0, 90.0, -110.0, 110.0, -75.0 + 30.0j, 70.0 - 40.0j])
def test_step_search_c128(N, m, z):
    """|Re z| r of 45 to 90: the step search starts far above the step that a basis covers."""
    _check(N, complex(z), m, "c128")


@pytest.mark.parametrize("N", [14, 16])
@pytest.mark.parametrize("m,z", [(6, -110.0), (6, 110.0), (8, -105.0), (8, 105.0), (12, -110.0)])
def test_step_search_c64(N, m, z):
    _check(N, complex(z), m, "c64")


@pytest.mark.parametrize("N", [6, 8, 10, 12])
@pytest.mark.parametrize("reach", [-60.0, -40.0, -20.0, 20.0, 40.0, 60.0, -30.0 + 20.0j, 45.0 + 10.0j])
def test_invariant_basis(N, reach):
    """Bases that span the sector (estimate 0: whatever the expansion gives is accepted), with
    |Re z| (half the spectrum's width) of `reach`: the result is far below the scale of the sums."""
    J = inputs.couplings(N, 21)
    for sector in (0, 1):
        E = np.linalg.eigvalsh(hm.H_sector_sparse(N, J, sector).toarray())
        z = reach / (0.5 * (E[-1] - E[0]))
        _check(N, complex(z), 40, "c128", sector=sector)
        _check(N, complex(z), 40, "c64", sector=sector)
