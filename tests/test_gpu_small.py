"""Small sectors run a Krylov basis as one launch (k_small_basis): evolutions, correlators and their
counters against the oracle at the sizes its rule takes and just beyond, both vector types, both
orthogonalisations, and against the general path (profiling switches to it)."""
import numpy as np
import pytest

from helpers import TOL, rel, to_dev, torch_or_skip
from oracle import correlators as co, evolve
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = torch_or_skip()
    syk.load(build_if_missing=True)
    return t


@pytest.mark.parametrize("N,B", [(4, 1), (4, 16), (6, 3), (8, 5), (10, 16), (12, 1), (12, 13), (12, 16), (12, 17), (14, 4),
                                 (14, 5), (16, 1), (16, 2), (18, 1)])
@pytest.mark.parametrize("dt", ["c128", "c64"])
def test_expmv_vs_exact_and_general_path(torch, N, B, dt):
    J = inputs.couplings(N, 31)
    terms = syk.syk_build_terms(N, J)
    psi = inputs.random_states(N, B, 32)
    ref = evolve.SectorSystem(N, J)
    code = syk.SYK_C128 if dt == "c128" else syk.SYK_C64
    tol = 1e-12 if dt == "c128" else 1e-7
    try:
        for orth in (syk.ORTH_FULL, syk.ORTH_LOCAL):
            prev = syk.syk_lanczos_orth(code, orth)
            for z, m in ((-0.1j, 30), (-1.5 - 2j, 40), (-8j, 12)):
                for sector in (0, 1):
                    x = to_dev(torch, psi, dt)
                    y, n1 = syk.syk_expmv(terms, sector, z, x, krylov_dim=m, tol=tol)
                    assert rel(y.cpu().numpy(), ref.expmv(z, psi.T, sector)) < TOL[dt], (z, m, sector, orth)
                    syk.syk_profile_enable(True)
                    g, n2 = syk.syk_expmv(terms, sector, z, x, krylov_dim=m, tol=tol)
                    syk.syk_profile_enable(False)
                    assert n1 == n2 and rel(y.cpu().numpy(), g.cpu().numpy()) < TOL[dt]
            syk.syk_lanczos_orth(code, prev)
    finally:
        syk.syk_profile_enable(False)
        syk.syk_lanczos_orth(syk.SYK_C128, syk.ORTH_FULL)
        syk.syk_lanczos_orth(syk.SYK_C64, syk.ORTH_LOCAL)


def test_G_grid_and_launch_modes(torch):
    N = 12
    J = inputs.couplings(N, 33)
    psi = inputs.random_states(N, 2, 34)
    terms = syk.syk_build_terms(N, J)
    ts = np.linspace(0.0, 3.0, 7)
    ref, Z = co.G_state(evolve.SectorSystem(N, J), 5.0, 3, ts, psi.T)
    x = to_dev(torch, psi, "c128")
    out = []
    for mode in (syk.GRAPHS_OFF, syk.GRAPHS_SEGMENTS, syk.GRAPHS_DEVICE):
        syk.syk_use_graphs(mode)
        syk.syk_counters(reset=True)
        out.append(syk.syk_correlator_G(terms, 5.0, 3, ts, x, krylov_dim=30, tol=1e-12))
        out[-1] += (syk.syk_counters(reset=True)["h_applies"],)
    syk.syk_use_graphs(syk.GRAPHS_SEGMENTS)
    for G, Zg, n in out:
        assert np.array_equal(G, out[0][0]) and n == out[0][2] > 0
        assert rel(G, ref) < TOL["c128"] and rel(Zg, Z) < TOL["c128"]


def test_non_finite_state_is_reported(torch):
    N = 12
    terms = syk.syk_build_terms(N, inputs.couplings(N, 35))
    x = to_dev(torch, inputs.random_states(N, 2, 36), "c128")
    x[3, 1] = complex(float("nan"), 0.0)
    with pytest.raises(syk.SykError, match="code -4"):
        syk.syk_expmv(terms, 0, -1j, x, krylov_dim=20, tol=1e-12)
