"""Truncated bonds beyond the number range.

A bond matrix whose squared norms overflow FP32 has no order of columns; every
rank must still name one column, or the compression reads through an index that
was never written.  The amplitude is then not finite, and the context stays
usable.
"""

import numpy as np
import pytest

import synth
from gpu_helpers import oracle_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cplx", [False, True])
def test_overflowing_bonds_stay_in_bounds(cplx):
    import paper_2503_20566_gb300 as G

    scale = 1e24
    lat, _, vals = oracle_net(7, 6, 2, 4, seed=61, complex_=cplx)
    got = {}
    for prec in ("fp32", "fp64"):
        ctx = G.Context(2, 7, 6, 4, 5, complex_=cplx, precision=prec, seed=1)
        cfg = ctx.init_configs(20, None, synth.plaquette_powers(62, 20, lat.n_plaquettes, 2))
        for name, v in (("before", vals), ("big", vals * scale), ("after", vals)):
            ctx.set_tensors(v)
            got[prec, name] = ctx.amplitude(cfg)[0].cpu().numpy()
    assert not np.isfinite(got["fp32", "big"]).any()
    for prec in ("fp32", "fp64"):
        assert np.isfinite(got[prec, "before"]).all() and np.array_equal(got[prec, "before"], got[prec, "after"])
