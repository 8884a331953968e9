"""Rounding of the complex64 matvec: the default kernel's error is no larger than that of the kernel it
took over from, with the launch shape that one had by default (a row's masks split over a cluster of
CTAs, so its FP32 sums were short).  Errors are 2-norms over a whole vector against the complex128
matvec (error below 1e-13), so they repeat to a fraction of a percent."""
import json

import pytest

from helpers import torch_or_skip
from paper_2002_05725_gb300 import inputs, syk

pytestmark = pytest.mark.gpu

# N, states, and the former default: variant, CTA width, cluster
FORMER = [(24, 16, 1, 6, 8), (28, 8, 2, 6, 8), (30, 16, 1, 6, 8), (32, 4, 2, 6, 8), (32, 16, 1, 6, 8),
          (34, 8, 2, 6, 8), (34, 16, 1, 6, 8), (36, 1, 0, 8, 8), (36, 4, 2, 6, 8), (36, 8, 2, 6, 8), (36, 16, 1, 6, 4),
          (38, 8, 2, 7, 4), (38, 16, 1, 7, 2), (40, 1, 0, 8, 4)]


@pytest.mark.parametrize("N,B,variant,ntb,cluster", FORMER)
def test_no_larger_than_the_former_kernel(N, B, variant, ntb, cluster):
    torch = torch_or_skip()
    syk.load(build_if_missing=True)
    terms = syk.syk_build_terms(N, inputs.couplings(N, 3))
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.view_as_complex(torch.randn((1 << (N // 2 - 1), B, 2), generator=g, device="cuda"))
    syk.syk_autotune_reset()
    new = syk.syk_apply_H(terms, 0, x)
    try:
        syk.syk_autotune_import(json.dumps({"apply_tiles": [
            {"N": N, "dtype": 1, "batch": B, "ntb": ntb, "cluster": cluster, "variant": variant}]}))
        old = syk.syk_apply_H(terms, 0, x)
    finally:
        syk.syk_autotune_reset()
    ref = syk.syk_apply_H(terms, 0, x.to(torch.complex128))
    err = [float((y.to(torch.complex128) - ref).norm() / ref.norm()) for y in (new, old)]
    assert err[0] <= err[1], err
