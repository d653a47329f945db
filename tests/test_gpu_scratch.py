"""Scratch of later asynchronous launches.

gcf_sample_batch_async takes any number of chains up to that of an earlier
gcf_sample_batch, whatever launch either takes.
"""

import pytest

import synth
from gpu_helpers import oracle_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Lx,Ly,chi,form", [(4, 4, 4, None), (4, 4, 4, "group"), (7, 6, 5, "cta"), (10, 6, 20, "cta")])
def test_async_covers_every_smaller_batch(Lx, Ly, chi, form, monkeypatch):
    import paper_2503_20566_gb300 as G

    if form:
        monkeypatch.setenv("GCFVMC_EXEC", form)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lat, _, vals = oracle_net(Lx, Ly, 2, 4, seed=71)
    for n in (5, sms + 1, 2 * sms + 96, 4 * sms + 1):
        ctx = G.Context(2, Lx, Ly, 4, chi, g=0.4, seed=1)
        ctx.set_tensors(vals)
        start = ctx.init_configs(n, None, synth.plaquette_powers(72, n, lat.n_plaquettes, 2))
        big = start.clone()
        ref = ctx.sample_batch(big, 1, 7)
        for m in {n, n - 1, min(n, 250), min(n, sms), min(n, 2 * sms), n // 2 + 1, 1}:
            cfg = start[:m].clone()
            out = ctx.sample_batch_async(cfg, 1, 7, ctx.alloc_samples(m, 1))
            torch.cuda.synchronize()
            assert torch.equal(cfg, big[:m]), (n, m)
            assert torch.equal(out["log_abs"], ref["log_abs"][:m]), (n, m)
        with pytest.raises(G.GcfError, match="scratch"):
            G.Context(2, Lx, Ly, 4, chi, g=0.4, seed=1).sample_batch_async(start.clone(), 1, 7, ctx.alloc_samples(n, 1))
