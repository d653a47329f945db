"""SR step at the edges of its sample-count classes, against a dense solve.

The sort by block works in chunks of 1024 samples, few samples are gathered by
a block each, short segments are scattered by a warp each, and chains of few
samples are averaged by a thread each; the cases sit on both sides of every
line.  Seeded samples (block ids uniform, O normal with an offset, E_loc
correlated with O); the update must equal that of (S + shift) x = F formed and
solved in FP64.  Tolerance on x: 1e-9 in FP64; in FP32 storage products and
partial sums carry 2^-24 relative, amplified by at most the condition of
S + shift, below 1e3 here (shift 1e-1, O of order 1, 100 parameters): 1e-4.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(2, 3, "fp32", False, n, nc) for n, nc in [(1, 1), (1023, 1023), (1025, 5), (16383, 1), (16400, 25), (40000, 40000)]]
CASES += [(3, 3, "fp32", True, 1024, 16), (3, 3, "fp64", True, 2049, 3), (2, 2, "fp64", False, 16385, 5),
          (4, 2, "fp32", True, 20000, 100)]


@pytest.mark.parametrize("N,L,prec,cplx,n,n_chains", CASES)
def test_sr_update_at_size_edges(N, L, prec, cplx, n, n_chains):
    import paper_2503_20566_gb300 as G

    Dk, shift, lr = 2, 0.1, 0.5
    ctx = G.Context(N, L, L, Dk * N, 4, complex_=cplx, precision=prec, seed=1)
    legs = [[(x > 0) + (x < L - 1) + (y > 0) + (y < L - 1) for x in range(L)] for y in range(L)]
    ks = [k for row in legs for k in row]
    nb, bs = [N ** (k - 1) for k in ks], [Dk ** k for k in ks]
    off = np.concatenate([[0], np.cumsum([a * b for a, b in zip(nb, bs)])])
    r = np.random.default_rng(n)
    bid = np.stack([r.integers(0, b, n) for b in nb], 1).astype(np.int32)
    real = lambda: r.standard_normal((n, L * L, Dk ** 4)) * 0.3 + 0.1  # noqa: E731
    O = (real() + 1j * real() if cplx else real()).astype({("fp32", False): np.float32, ("fp32", True): np.complex64,
                                                          ("fp64", False): np.float64, ("fp64", True): np.complex128}[prec, cplx])
    E = r.standard_normal(n) + O[:, 0, 0].real.astype(np.float64)
    dense = np.zeros((n, off[-1]), np.complex128 if cplx else np.float64)
    for v in range(L * L):
        at = off[v] + bid[:, v, None] * bs[v] + np.arange(bs[v])
        np.put_along_axis(dense, at, O[:, v, :bs[v]].astype(dense.dtype), 1)
    F = dense.conj().T @ (E - E.mean()) / n
    c = dense - dense.mean(0)
    x = np.linalg.solve(c.conj().T @ c / n + shift * np.eye(off[-1]), F)
    before = ctx.get_tensors()
    s = dict(e_loc=torch.from_numpy(np.stack([E, 0 * E], 1).reshape(-1)).cuda(), block_ids=torch.from_numpy(bid).cuda(),
             O=torch.from_numpy(O).cuda())
    st = ctx.sr_step(s, n_chains, diag_shift=shift, lr=lr, max_iter=400, tol=1e-8 if prec == "fp32" else 1e-12)
    means = E.reshape(n_chains, -1).mean(1) if n_chains > 1 else E
    assert abs(st[0] - E.mean()) < 1e-12 * n
    assert abs(st[2] - (means.std(ddof=1) / np.sqrt(means.size) if means.size > 1 else 0.0)) < 1e-9
    got = (before - ctx.get_tensors()) / lr
    tol = (1e-4 if prec == "fp32" else 1e-9) * max(np.abs(x).max(), 1e-12) + (2.0 ** -23 * np.abs(before).max() / lr if prec == "fp32" else 1e-15 * np.abs(before).max() / lr)
    assert np.abs(got - x).max() <= tol, (np.abs(got - x).max(), tol)
