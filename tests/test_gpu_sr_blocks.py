"""SR step over many blocks, odd block sizes, and block ids that name no block.

A vertex of more than 128 blocks (Z5 with matter: 250 at the centre) takes the
sort of one CTA per vertex; D_k = 3 has blocks of 81, 27 and 9 entries, whose
rows are not whole 16-byte vectors.  The update must equal that of
(S + shift) x = F solved in FP64 in the space of the samples or parameters,
whichever is smaller.  Tolerance on x as for the other sizes: 1e-4 in FP32
storage (2^-24 per product and partial sum, times the condition of S + shift,
below 1e3), 1e-9 in FP64.  Ids out of range are refused before anything is read
through them, and the tensors stay as they are.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _problem(N, L, D, n, prec, cplx, matter):
    import paper_2503_20566_gb300 as G

    ctx = G.Context(N, L, L, D, 4, matter=matter, complex_=cplx, precision=prec, seed=1)
    Dk = D // N
    ks = [(x > 0) + (x < L - 1) + (y > 0) + (y < L - 1) for y in range(L) for x in range(L)]
    nb, bs = [(1 + matter) * N ** (k - 1) for k in ks], [Dk ** k for k in ks]
    r = np.random.default_rng(n)
    bid = np.stack([r.integers(0, b, n) for b in nb], 1).astype(np.int32)
    real = lambda: r.standard_normal((n, L * L, Dk ** 4)) * 0.3 + 0.1  # noqa: E731
    O = (real() + 1j * real() if cplx else real()).astype({("fp32", False): np.float32, ("fp32", True): np.complex64,
                                                          ("fp64", False): np.float64, ("fp64", True): np.complex128}[prec, cplx])
    E = r.standard_normal(n) + O[:, 0, 0].real.astype(np.float64)
    return ctx, nb, bs, bid, O, E


def _samples(bid, O, E):
    return dict(e_loc=torch.from_numpy(np.stack([E, 0 * E], 1).reshape(-1)).cuda(),
                block_ids=torch.from_numpy(bid).cuda(), O=torch.from_numpy(O).cuda())


@pytest.mark.parametrize("N,L,D,n,prec,cplx,matter", [
    (5, 3, 10, 600, "fp32", False, True), (5, 3, 10, 1300, "fp64", True, True), (2, 3, 6, 1500, "fp32", False, False),
    (2, 3, 6, 1025, "fp32", True, False), (2, 3, 6, 1500, "fp64", False, False), (3, 2, 3, 2100, "fp32", False, False),
    # a block gathers a sample up to twice as many samples as a row has vectors (36 and 72 here), a warp beyond
    (2, 3, 4, 72, "fp32", False, False), (2, 3, 4, 73, "fp32", False, False), (2, 3, 4, 144, "fp32", True, False),
    (2, 3, 4, 145, "fp32", True, False)])
def test_sr_update_many_blocks_and_odd_sizes(N, L, D, n, prec, cplx, matter):
    _check(*_problem(N, L, D, n, prec, cplx, matter), prec)


def _check(ctx, nb, bs, bid, O, E, prec):
    shift, lr, n, cplx = 0.1, 0.5, len(E), np.iscomplexobj(O)
    off = np.concatenate([[0], np.cumsum([a * b for a, b in zip(nb, bs)])])
    c = np.zeros((n, off[-1]), np.complex128 if cplx else np.float64)
    for v in range(len(nb)):
        np.put_along_axis(c, off[v] + bid[:, v, None] * bs[v] + np.arange(bs[v]), O[:, v, :bs[v]].astype(c.dtype), 1)
    F = c.conj().T @ (E - E.mean()) / n
    c -= c.mean(0)
    if n < off[-1]:  # Woodbury
        x = (F - c.conj().T @ np.linalg.solve(c @ c.conj().T + n * shift * np.eye(n), c @ F)) / shift
    else:
        x = np.linalg.solve(c.conj().T @ c / n + shift * np.eye(off[-1]), F)
    before = ctx.get_tensors()
    ctx.sr_step(_samples(bid, O, E), 1, diag_shift=shift, lr=lr, max_iter=800, tol=1e-8 if prec == "fp32" else 1e-12)
    got = (before - ctx.get_tensors()) / lr
    eps = 2.0 ** -23 if prec == "fp32" else 1e-15
    tol = (1e-4 if prec == "fp32" else 1e-9) * np.abs(x).max() + eps * np.abs(before).max() / lr
    assert np.abs(got - x).max() <= tol, (np.abs(got - x).max(), tol)


@pytest.mark.parametrize("N,D,prec,cplx", [(3, 6, "fp32", True), (3, 6, "fp64", False), (3, 3, "fp32", False)])
def test_sr_update_with_most_samples_on_one_block(N, D, prec, cplx):
    """Short segments on average, long ones among them: warps take 64 rows each,
    so segments of 0, 1, 63, 64, 65, 128 and about a thousand rows meet."""
    ctx, nb, bs, bid, O, E = _problem(N, 3, D, 1400, prec, cplx, False)
    for v in range(9):
        lens = [0, 1, 63, 64, 65, 128][: min(6, nb[v] - 1)]
        bid[:, v] = np.random.default_rng(v).permutation(np.concatenate([np.repeat(np.arange(len(lens)), lens),
                                                                         np.full(1400 - sum(lens), nb[v] - 1)]))
    _check(ctx, nb, bs, bid, O, E, prec)


@pytest.mark.parametrize("N,D,matter,prec,cplx", [(2, 4, False, "fp32", False), (5, 10, True, "fp32", False), (3, 9, False, "fp64", True)])
@pytest.mark.parametrize("bad", [-1, "nb", 2 ** 30, -2 ** 31])
def test_block_ids_out_of_range_are_refused(N, D, matter, prec, cplx, bad):
    import paper_2503_20566_gb300 as G

    ctx, nb, _, bid, O, E = _problem(N, 3, D, 1500, prec, cplx, matter)
    good = bid.copy()
    for s, v in ((0, 0), (700, 4), (1499, 8)):
        bid[s, v] = nb[v] if bad == "nb" else bad
    before = ctx.get_tensors()
    with pytest.raises(G.GcfError, match="block_ids"):
        ctx.sr_step(_samples(bid, O, E), 1, max_iter=5)
    assert np.array_equal(before, ctx.get_tensors())
    st = ctx.sr_step(_samples(good, O, E), 1, diag_shift=0.1, max_iter=400, tol=1e-6)
    assert st[6] == 1.0 and not np.array_equal(before, ctx.get_tensors())
