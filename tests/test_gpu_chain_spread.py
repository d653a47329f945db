"""Chains do not depend on how many run beside them.

A grouped launch seats one, two or four chains per CTA by the number of chains
and of SMs, and a truncating one-chain launch takes 512 or 256 threads: chain
c of every batch size must equal, bit for bit, chain c of the largest.
"""

import numpy as np
import pytest

import synth
from gpu_helpers import oracle_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Lx,Ly,chi,form", [(4, 4, 4, "group4"), (13, 7, 24, "cta")])
def test_batch_size_leaves_chains_unchanged(Lx, Ly, chi, form, monkeypatch):
    import paper_2503_20566_gb300 as G

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lat, _, vals = oracle_net(Lx, Ly, 2, 4, seed=41)
    n = 2 * sms + 1 if form == "cta" else 4 * sms + 1
    monkeypatch.setenv("GCFVMC_EXEC", form)
    powers = synth.plaquette_powers(42, n, lat.n_plaquettes, 2)
    ctx = G.Context(2, Lx, Ly, 4, chi, g=0.4, seed=1)
    ctx.set_tensors(vals)
    start = ctx.init_configs(n, None, powers)
    ref = None
    for m in (n, 2 * sms, 2 * sms - 1, sms + 1, sms, 5, 1):
        cfg = start[:m].clone()
        out = ctx.sample_batch(cfg, 1, 7)
        got = [cfg] + [out[k].reshape(m, -1) for k in ("log_abs", "e_loc", "O", "accepted")]
        ref = ref or got
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy(), b[:m].cpu().numpy()), m
