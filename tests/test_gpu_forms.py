"""The kernel form that runs is the one asked for, and the one reported.

A grouped form seats the chains of a call on as few chains per CTA as the SMs
allow; a form forced by GCFVMC_EXEC keeps its own number, so that the tests
which force one run it.  chains_per_cta and kernel_name report the launch, and the
autotuner times no launch under two names.
"""

import numpy as np
import pytest

import synth
from gpu_helpers import oracle_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("form,per_cta,name", [("cta", 1, "gcf::vmc_kernel"), ("group", 2, "gcf::vmc_kernel_grouped"),
                                               ("group4", 4, "gcf::vmc_kernel_grouped4")])
def test_forced_form_keeps_its_chains_per_cta(form, per_cta, name, monkeypatch):
    import paper_2503_20566_gb300 as G

    monkeypatch.setenv("GCFVMC_EXEC", form)
    ctx = G.Context(2, 4, 4, 4, 4, g=0.4, seed=1)
    for n in (1, 3, 5):
        ctx.amplitude(ctx.init_configs(n))
        assert (ctx.chains_per_cta, ctx.kernel_name) == (per_cta, name), n


def test_default_form_spreads_few_chains_and_leaves_them_unchanged():
    import paper_2503_20566_gb300 as G

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lat, _, vals = oracle_net(4, 4, 2, 4, seed=41)
    n = 4 * sms + 1
    ctx = G.Context(2, 4, 4, 4, 4, g=0.4, seed=1)
    ctx.set_tensors(vals)
    start = ctx.init_configs(n, None, synth.plaquette_powers(42, n, lat.n_plaquettes, 2))
    ref = None
    for m, per_cta in ((n, 4), (2 * sms + 1, 4), (2 * sms, 2), (sms + 1, 2), (sms, 1), (5, 1), (1, 1)):
        cfg = start[:m].clone()
        out = ctx.sample_batch(cfg, 1, 7)
        assert ctx.chains_per_cta == per_cta, m
        assert ctx.kernel_name == "gcf::vmc_kernel_grouped" + ("4" if per_cta == 4 else ""), m
        got = [cfg] + [out[k].reshape(m, -1) for k in ("log_abs", "e_loc", "O", "accepted")]
        ref = ref or got
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy(), b[:m].cpu().numpy()), m


@pytest.mark.parametrize("per_sm,forms", [(1, 4 + 3), (2, 4 + 3), (3, 4 + 3 + 3)])
def test_autotune_times_each_launch_once(per_sm, forms):
    """One-chain-per-CTA at four levels, two groups at three; four groups only
    where the chains outnumber two per SM (below, the launches would be the
    same and noise would choose the name)."""
    import paper_2503_20566_gb300 as G

    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    ctx = G.Context(2, 3, 3, 4, 4, g=0.4, seed=1)
    assert len(ctx.autotune(ctx.init_configs(n))) == forms
    assert per_sm > 2 or ctx.kernel_name != "gcf::vmc_kernel_grouped4"


@pytest.mark.parametrize("prec,cplx,chi", [("fp64", True, 22), ("fp64", False, 43), ("fp32", False, 24), ("fp32", True, 10),
                                           ("fp32", True, 30), ("fp64", True, 10)])
def test_amplitudes_do_not_depend_on_the_batch(prec, cplx, chi):
    """D_k = 3, bonds beyond the register factorisations in the first two (QR
    columns of 9 chi rows, Jacobi columns of 3 chi): the same bits alone, among
    as many chains as there are SMs, among more, and without allocation."""
    import paper_2503_20566_gb300 as G
    from paper_2503_20566_gb300.binding import _ptr

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lat, _, vals = oracle_net(10, 7, 2, 6, seed=51, complex_=cplx, precision=prec)
    ctx = G.Context(2, 10, 7, 6, chi, complex_=cplx, precision=prec, seed=1)
    ctx.set_tensors(vals)
    n = sms + 1
    cfg = ctx.init_configs(n, None, synth.plaquette_powers(52, n, lat.n_plaquettes, 2))
    ref = ctx.amplitude(cfg)
    for m in (sms, 3):
        for a, b in zip(ctx.amplitude(cfg[:m].clone()), ref):
            assert torch.equal(a, b[:m]), m
    la, ph = torch.zeros(3, dtype=torch.float64, device="cuda"), torch.zeros(3, dtype=torch.float64, device="cuda")
    ctx._check(ctx.lib.gcf_amplitude_noalloc(ctx.ctx, 3, _ptr(cfg), _ptr(la), _ptr(ph)), "noalloc")
    torch.cuda.synchronize()
    assert torch.equal(la, ref[0][:3]) and torch.equal(ph, ref[1][:3])


def _two_lattices(prec, cplx, Dk, chi, sizes, n):
    import paper_2503_20566_gb300 as G

    ctxs, cfgs = [], []
    for Lx, Ly in sizes:
        lat, _, vals = oracle_net(Lx, Ly, 2, 2 * Dk, seed=81, complex_=cplx, precision=prec)
        ctxs.append(G.Context(2, Lx, Ly, 2 * Dk, chi, g=0.4, complex_=cplx, precision=prec, seed=1))
        ctxs[-1].set_tensors(vals)
        cfgs.append(ctxs[-1].init_configs(n, None, synth.plaquette_powers(82, n, lat.n_plaquettes, 2)))
    return ctxs, cfgs


def _sampled(ctxs, cfgs, n):
    import paper_2503_20566_gb300 as G

    x = [c[:n].clone() for c in cfgs]
    out = G.sample_multi(ctxs, x, 1, [7, 8])
    return [t for a, o in zip(x, out) for t in (a, o["log_abs"], o["e_loc"].view(n, 2), o["O"].view(n, -1), o["accepted"])]


def test_many_chains_of_several_lattices_share_ctas_and_keep_their_bits():
    """Four chains per CTA from three rounds of one per CTA on (two CTAs fit an SM here)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctxs, cfgs = _two_lattices("fp32", False, 2, 3, ((6, 5), (5, 6)), 3 * sms)
    ref = None
    for n, per_cta in ((3 * sms, 4), (3 * sms - 1, 1), (5, 1)):
        got = _sampled(ctxs, cfgs, n)
        assert ctxs[0].multi_chains_per_cta == per_cta, n
        ref = ref or got
        for a, b in zip(got, ref):
            assert torch.equal(a, b[:n]), n


@pytest.mark.parametrize("prec,cplx,Dk,chi", [("fp32", False, 2, 24), ("tf32", False, 2, 24), ("bf16", False, 2, 16), ("fp32", True, 3, 10),
                                              ("fp64", False, 2, 10), ("fp64", True, 2, 8)])
def test_chains_are_the_same_one_or_four_per_cta(prec, cplx, Dk, chi, monkeypatch):
    """Sums are dealt to 128 threads and products add in one order in every form."""
    got = {}
    for form, per_cta in (("cta", 1), ("group4", 4)):
        monkeypatch.setenv("GCFVMC_MULTI", form)
        ctxs, cfgs = _two_lattices(prec, cplx, Dk, chi, ((11, 6), (9, 7)) if chi > 12 else ((7, 6), (6, 5)), 9)
        got[form] = _sampled(ctxs, cfgs, 9)
        assert ctxs[0].multi_chains_per_cta == per_cta
    for a, b in zip(got["cta"], got["group4"]):
        assert torch.equal(a, b)
