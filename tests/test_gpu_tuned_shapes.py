"""Tuned row-block shapes in Krylov calls, whose matvecs write the partial sums of their output stage
into the workspace: every shape that can be imported has to serve e^{zH} too (one with more CTAs
than the workspace has room for gives way to the default rule).  Reference: the same evolution in
complex128; bound: the suite's complex64 tolerance."""
import json

import pytest

from helpers import TOL, rel, to_dev, torch_or_skip
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,B", [(26, 16), (28, 16), (26, 1), (26, 4)])
def test_expmv_with_every_shape(N, B):
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    terms = syk.syk_build_terms(N, inputs.couplings(N, 6))
    psi = inputs.random_states(N, B, 4)
    z = complex(-0.2, -0.9)
    syk.syk_autotune_reset()
    ref = syk.syk_expmv(terms, 1, z, to_dev(torch, psi, "c128"), krylov_dim=30, tol=1e-12)[0].cpu().numpy()
    x = to_dev(torch, psi, "c64")
    try:
        for var in (4, 5):
            for ntb in (6, 7, 8):
                for cs in (1, 2, 4, 8):
                    syk.syk_autotune_reset()
                    syk.syk_autotune_import(json.dumps({"apply_tiles": [
                        {"N": N, "dtype": 1, "batch": B, "ntb": ntb, "cluster": cs, "variant": var}]}))
                    y = syk.syk_expmv(terms, 1, z, x, krylov_dim=30, tol=1e-7)[0].cpu().numpy()
                    assert rel(y, ref) < TOL["c64"], (var, ntb, cs)
    finally:
        syk.syk_autotune_reset()


@pytest.mark.parametrize("B", [1, 2, 4, 8, 16])
def test_complex128_shapes_vs_oracle(B):
    """Every complex128 row-block shape that the table takes, against the FP64 oracle."""
    from oracle import hamiltonian as hm
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    N = 24
    J = inputs.couplings(N, 6)
    terms = syk.syk_build_terms(N, J)
    H = hm.H_sector_sparse(N, J, 1)
    psi = inputs.random_states(N, B, 4)
    x = to_dev(torch, psi, "c128")
    try:
        for ntb in (6, 7, 8):
            for cs in (1, 2, 4, 8):
                syk.syk_autotune_reset()
                syk.syk_autotune_import(json.dumps({"apply_tiles": [
                    {"N": N, "dtype": 2, "batch": B, "ntb": ntb, "cluster": cs, "variant": 5}]}))
                y = syk.syk_apply_H(terms, 1, x).cpu().numpy().reshape(-1, B)
                assert rel(y, H @ psi.T) < TOL["c128"], (ntb, cs)
    finally:
        syk.syk_autotune_reset()
