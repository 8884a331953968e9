"""The row-block complex64 matvec (k_apply_block) against the oracle, at the edges of its rule:
the smallest sectors and one tile, state counts in and out of powers of two up to 32, every
thread count and cluster size, and the sectors between its 8-row and 32-row kernels.

Bound: a row is a sum of M masks, each product and sum rounded to FP32 (unit 2^-24), so with
random signs its error is about sqrt(M) 2^-24 of |row| (M = 256 at N = 20, 1093 at N = 28:
2e-6); the bound is the suite's complex64 tolerance 1e-5."""
import json

import numpy as np
import pytest

from helpers import TOL, rel, to_dev, torch_or_skip
from oracle import hamiltonian as hm
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = torch_or_skip()
    syk.load(build_if_missing=True)
    yield t
    syk.syk_autotune_reset()


def _check(torch, N, B, H, terms, sector):
    psi = inputs.random_states(N, B, 11 + B)
    syk.syk_matvec_launches(reset=True)
    y = syk.syk_apply_H(terms, sector, to_dev(torch, psi, "c64")).cpu().numpy().reshape(-1, B)
    mv = syk.syk_matvec_launches(reset=True)
    assert syk.syk_status(terms) == syk.SYK_OK
    assert rel(y, H @ psi.T) < TOL["c64"], (N, B, sector)
    return mv


@pytest.mark.parametrize("N", [10, 12, 14, 16, 18, 20, 22, 24])
def test_default_rule_vs_oracle(torch, N):
    syk.syk_autotune_reset()
    J = inputs.couplings(N, 5)
    terms = syk.syk_build_terms(N, J)
    for sector in (0, 1):
        H = hm.H_sector_sparse(N, J, sector)
        for B in (1, 2, 3, 4, 5, 6, 7, 8, 12, 13, 16, 17, 24, 31, 32, 33):
            mv = _check(torch, N, B, H, terms, sector)
            if N >= 22 and B <= 32:
                assert mv["coset"] == 1 and mv["rows"] == 0, (B, mv)


@pytest.mark.parametrize("N,B", [(20, 16), (24, 8), (24, 16), (26, 4), (26, 1)])
def test_every_shape_vs_oracle(torch, N, B):
    J = inputs.couplings(N, 6)
    terms = syk.syk_build_terms(N, J)
    H = hm.H_sector_sparse(N, J, 1)
    for var in (4, 5):
        for ntb in (6, 7, 8):
            for cs in (1, 2, 4, 8):
                syk.syk_autotune_reset()
                syk.syk_autotune_import(json.dumps({"apply_tiles": [
                    {"N": N, "dtype": 1, "batch": B, "ntb": ntb, "cluster": cs, "variant": var}]}))
                _check(torch, N, B, H, terms, 1)
    syk.syk_autotune_reset()


@pytest.mark.parametrize("B", [1, 6, 8, 16])
def test_larger_sector_rows_and_epilogue(torch, B):
    """N = 30 (32 rows per thread from 8 states on): the matvec on sampled rows, and e^{zH}, whose
    Lanczos steps take the scaled output and the dot products of the kernel's output stage,
    against the complex128 result."""
    N = 30
    syk.syk_autotune_reset()
    J = inputs.couplings(N, 7)
    terms = syk.syk_build_terms(N, J)
    psi = inputs.random_states(N, B, 3)
    x = to_dev(torch, psi, "c64")
    rows = np.unique(np.concatenate([[0, (1 << 14) - 1], np.random.default_rng(3).integers(0, 1 << 14, 40)]))
    y = syk.syk_apply_H(terms, 0, x).cpu().numpy().reshape(-1, B)
    assert rel(y[rows], hm.apply_rows(N, J, 0, psi.T, rows).reshape(len(rows), B)) < TOL["c64"]
    z = complex(-0.4, -1.5)
    a = syk.syk_expmv(terms, 0, z, x, krylov_dim=40, tol=1e-7)[0].cpu().numpy()
    b = syk.syk_expmv(terms, 0, z, to_dev(torch, psi, "c128"), krylov_dim=40, tol=1e-12)[0].cpu().numpy()
    assert rel(a, b) < TOL["c64"]


def test_first_launch_under_stream_capture(torch):
    """A state count whose layout is not built yet, first used under stream capture: the row kernel
    is recorded instead (building a layout allocates), and the replayed graph is correct."""
    N = 22
    syk.syk_autotune_reset()
    J = inputs.couplings(N, 8)
    terms = syk.syk_build_terms(N, J)
    H = hm.H_sector_sparse(N, J, 0)
    _check(torch, N, 4, H, terms, 0)  # uploads the term set
    psi = inputs.random_states(N, 5, 9)
    x = to_dev(torch, psi, "c64")
    y = torch.zeros_like(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        syk.syk_apply_H(terms, 0, x, out=y)
    g.replay()
    torch.cuda.synchronize()
    assert rel(y.cpu().numpy(), H @ psi.T) < TOL["c64"]
    _check(torch, N, 5, H, terms, 0)
