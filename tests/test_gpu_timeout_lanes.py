"""A bounded wait of the row-block matvec that runs out in some lanes of a warp and not in others.

The lanes of a warp poll one after another, so at the end of the budget they may disagree.  The
warp has to give up as one: its other barriers take all 32 lanes.  A variant build gives lane 0
of every warp no polls and the others enough; every launch must then end, with the timeout in the
term set's status word and the context usable, for each form of the kernel (8 and 32 rows per
thread, shared two-spin coefficients, state counts with idle lanes, double-float)."""
import os
import subprocess
import sys
import textwrap

import pytest

from helpers import torch_or_skip

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = textwrap.dedent("""
    import sys
    sys.path.insert(0, {root!r})
    import numpy as np
    import torch
    from oracle import hamiltonian as hm
    from paper_2002_05725_gb300 import inputs, syk
    syk.load()
    for N, B, dt in [(20, 8, torch.complex64), (22, 5, torch.complex64), (24, 1, torch.complex64),
                     (28, 16, torch.complex64), (28, 12, torch.complex64), (24, 1, torch.complex128)]:
        terms = syk.syk_build_terms(N, inputs.couplings(N, 3))
        x = torch.from_numpy(np.ascontiguousarray(inputs.random_states(N, B, 1).T)).to(dt).cuda()
        syk.syk_apply_H(terms, 0, x)
        assert syk.syk_status(terms, reset=True) == syk.SYK_ETIMEOUT, (N, B, dt)
        assert syk.syk_status(terms) == syk.SYK_OK
    # the row kernel (3 states of a small sector) has no waits: the context is usable
    N = 16
    J = inputs.couplings(N, 3)
    terms = syk.syk_build_terms(N, J)
    psi = inputs.random_states(N, 3, 2)
    y = syk.syk_apply_H(terms, 0, torch.from_numpy(np.ascontiguousarray(psi.T)).to(torch.complex64).cuda())
    ref = hm.H_sector_sparse(N, J, 0) @ psi.T
    assert np.abs(y.cpu().numpy() - ref).max() / np.abs(ref).max() < 1e-5
    assert syk.syk_status(terms) == syk.SYK_OK
    print("child ok")
""")


def test_lanes_give_up_together(tmp_path):
    torch_or_skip()
    out = tmp_path / "lanes"
    b = subprocess.run([sys.executable, "-m", "paper_2002_05725_gb300.build", "--out-dir", str(out),
                        "-D", "SYK_WAIT_POLLS=threadIdx.x%32*65536"], cwd=ROOT, capture_output=True, text=True,
                       timeout=1200)
    assert b.returncode == 0, b.stdout[-2000:] + b.stderr[-2000:]
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, SYK_LIBRARY=str(out / "libsyk_gb300.so")))
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
