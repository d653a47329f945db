"""Short memory: a call that fits with one CTA per SM runs where there is no room
for the scratch of the second."""

import pytest

import synth
from gpu_helpers import oracle_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_short_memory_takes_fewer_ctas_per_sm(monkeypatch):
    import paper_2503_20566_gb300 as G

    monkeypatch.setenv("GCFVMC_EXEC", "cta")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * sms
    lat, _, vals = oracle_net(16, 16, 2, 4, seed=73)
    powers = synth.plaquette_powers(74, n, lat.n_plaquettes, 2)

    def context():
        c = G.Context(2, 16, 16, 4, 16, g=0.4, seed=1)
        c.set_tensors(vals)
        return c

    a, b = context(), context()
    cfg = a.init_configs(n, None, powers)
    ref = a.amplitude(cfg)  # loads the kernel and its stack beside two CTAs per SM
    x0, x1 = cfg[:n].clone(), cfg[:n].clone()
    G.sample_multi([a], [x0], 1, [7])
    slots = sms * a.scratch_bytes_per_chain
    m = context()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(free - 3 * slots // 2 - (64 << 20), dtype=torch.uint8, device="cuda")
    got = b.amplitude(cfg)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    b.close()
    G.sample_multi([m], [x1], 1, [7])
    assert torch.equal(x0, x1)
    del fill
