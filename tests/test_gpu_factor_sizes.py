"""Truncated amplitudes at the edges of the factorisations' size classes.

The compression keeps the columns of its QR and Jacobi steps in registers, in
forms chosen by the column length (a left site has D_k^2 chi rows, a truncated
bond D_k chi).  Each case sits on the last size of a form, on the first of the
next one, or beyond the longest (the general forms), or has bonds with fewer
rows than one register pass has columns; the lattice is just large enough for
the bonds to reach chi.  Against the FP64 oracle; FP32 by the rule
of the full-size tests: 1e-4 where the oracle's own single-precision run
is within 1e-5, else 10 times its distance.
"""

import numpy as np
import pytest

from oracle import vmc

from gpu_helpers import amp_err, configs_for, setup

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [("fp32", False, dk, chi) for dk, chi in
         [(2, 5), (2, 8), (2, 9), (2, 16), (2, 17), (2, 25), (2, 33), (2, 41), (3, 22), (3, 38), (3, 40), (3, 43)]]
CASES += [("fp32", True, dk, chi) for dk, chi in [(2, 8), (2, 9), (2, 17), (2, 32), (2, 33), (3, 22), (3, 37), (3, 38),
                                                  (3, 43)]]
CASES += [("fp64", False, dk, chi) for dk, chi in [(2, 9), (2, 33), (3, 38), (3, 43)]]
CASES += [("fp64", True, dk, chi) for dk, chi in [(2, 8), (2, 9), (2, 17), (2, 33), (3, 15), (3, 22), (3, 36)]]


def _levels(base, n):
    k = 0
    while base ** k < n:
        k += 1
    return k


@pytest.mark.parametrize("prec,cplx,dk,chi", CASES)
def test_truncated_amplitude_at_size_edges(prec, cplx, dk, chi):
    Lx, Ly = 2 * _levels(dk, dk * chi), _levels(dk, chi) + 3
    lat, pe, ctx = setup(Lx, Ly, 2, 2 * dk, chi, seed=31, complex_=cplx, precision=prec)
    cfgs, _, _ = configs_for(lat, 2, seed=32)
    la, ph = (t.cpu().numpy() for t in ctx.amplitude(torch.from_numpy(cfgs)))
    for i, c in enumerate(cfgs):
        ref = vmc.amplitude(pe, c, chi)
        bound = 1e-9
        if prec == "fp32":
            d32 = amp_err(*vmc.amplitude(pe, c, chi, dtype=np.complex64 if cplx else np.float32), *ref)
            bound = 1e-4 if d32 <= 1e-5 else 10 * d32
        assert amp_err(la[i], ph[i], *ref) <= bound, (i, la[i], ph[i], ref)
