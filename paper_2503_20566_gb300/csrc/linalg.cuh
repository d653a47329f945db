// CTA-cooperative dense linear algebra on small matrices: strided GEMM,
// Householder QR and one-sided Jacobi of any size.
//
// Every routine is called by all threads of the executor with identical
// arguments and ends with ex.sync(), so its results are visible on return.
// The QR and Jacobi here serve any size; factor.cuh holds the forms that keep
// the columns in registers and falls back to these.
//
// The algorithms are the textbook ones: Householder QR (Golub & Van Loan,
// "Matrix Computations", Alg. 5.1.1 / 5.2.1, with the complex reflector that
// maps x to -sign(Re x_1) |x| e_1) and the one-sided (Hestenes) Jacobi SVD
// with the round-robin pair schedule.
#pragma once

#include "common.cuh"
#include "mma.cuh"

namespace gcf {

// Rows of a column-major matrix padded to whole 16-byte chunks of any type.
__host__ __device__ inline int pad4(int n) { return (n + 3) & ~3; }

// Row offsets of a matrix whose row index may be a pair i = (i / mr, i % mr).
struct RowMap {
  int mr, s0, s1;  // row i at (i / mr) s0 + (i % mr) s1
  __device__ __forceinline__ int operator()(int i) const {
    const int h = mr == 1 ? i : i / mr;
    return h * s0 + (i - h * mr) * s1;
  }
};

// Address of C(i, j): rows and columns may each be a pair of indices,
// i = (i / mr, i % mr) and j = (j / nc, j % nc).
template <class T>
struct OutMap {
  T* C;
  RowMap row;
  int nc, s2, s3;  // column j at (j / nc) s2 + (j % nc) s3
  __device__ __forceinline__ int col(int j) const {
    const int h = j < nc ? 0 : j / nc;
    return h * s2 + (j - h * nc) * s3;
  }
};

// C (M x N) = A (M x K) B (K x N), strided operands in shared or global
// memory: each thread accumulates TM x TN tiles of C in registers, summing
// over k in order.  C must not overlap A or B.
template <class T, int TM, int TN, class X>
__device__ __noinline__ void gemm_tiled(const X ex, int M, int N, int K, const T* A, const RowMap ra, int sAk,
                                        const T* B, int sBk, int sBn, const OutMap<T> out) {
  const int tm = (M + TM - 1) / TM, tn = (N + TN - 1) / TN;
#pragma unroll 1
  for (int t = ex.tid(); t < tm * tn; t += ex.size()) {
    const int i0 = (t / tn) * TM, j0 = (t - (t / tn) * tn) * TN;
    const T* ap[TM];
    const T* bp[TN];
#pragma unroll
    for (int q = 0; q < TM; ++q) ap[q] = A + ra(min(i0 + q, M - 1));  // rows / columns past the edge repeat the last one
#pragma unroll
    for (int r = 0; r < TN; ++r) bp[r] = B + min(j0 + r, N - 1) * sBn;
    T acc[TM][TN];
#pragma unroll
    for (int q = 0; q < TM; ++q)
#pragma unroll
      for (int r = 0; r < TN; ++r) acc[q][r] = zero<T>();
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      T a[TM], b[TN];
#pragma unroll
      for (int q = 0; q < TM; ++q) a[q] = ap[q][k * sAk];
#pragma unroll
      for (int r = 0; r < TN; ++r) b[r] = bp[r][k * sBk];
#pragma unroll
      for (int q = 0; q < TM; ++q)
#pragma unroll
        for (int r = 0; r < TN; ++r) acc[q][r] = fmac(acc[q][r], a[q], b[r]);
    }
#pragma unroll
    for (int q = 0; q < TM; ++q) {
      if (i0 + q >= M) continue;
      const int ro = out.row(i0 + q);
#pragma unroll
      for (int r = 0; r < TN; ++r)
        if (j0 + r < N) out.C[ro + out.col(j0 + r)] = acc[q][r];
    }
  }
  ex.sync();
}

// gemm_tiled with the tile that needs the fewest cycles over the executor's
// threads (per step of k a tile costs its multiply-adds and its loads).
template <class T, class X>
__device__ __noinline__ void cta_gemm_out(const X ex, int M, int N, int K, const T* A, const RowMap ra, int sAk,
                                          const T* B, int sBk, int sBn, const OutMap<T> out) {
  constexpr int F = Traits<T>::cplx ? 4 : 1;
  const int nt = ex.size();
  auto cost = [&](int tm, int tn) {
    const int tiles = ((M + tm - 1) / tm) * ((N + tn - 1) / tn);
    return ((tiles + nt - 1) / nt) * (F * tm * tn + 2 * (tm + tn));
  };
  const int c44 = cost(4, 4), c42 = cost(4, 2), c22 = cost(2, 2);
  if (c44 <= c42 && c44 <= c22) gemm_tiled<T, 4, 4>(ex, M, N, K, A, ra, sAk, B, sBk, sBn, out);
  else if (c42 <= c22) gemm_tiled<T, 4, 2>(ex, M, N, K, A, ra, sAk, B, sBk, sBn, out);
  else gemm_tiled<T, 2, 2>(ex, M, N, K, A, ra, sAk, B, sBk, sBn, out);
}

// C (M x N) = A B in the scalar's own precision (dense absorption).
template <class T, class X>
__device__ __noinline__ void cta_gemm(const X ex, int M, int N, int K, const T* A, int sAm, int sAk, const T* B,
                                      int sBk, int sBn, T* C, int sCm, int sCn) {
  const int MN = M * N;
#pragma unroll 1
  for (int idx = ex.tid(); idx < MN; idx += ex.size()) {
    const int i = idx / N, j = idx - (idx / N) * N;
    T s = zero<T>();
    const T* a = A + i * sAm;
    const T* b = B + j * sBn;
    for (int k = 0; k < K; ++k) s = fmac(s, a[k * sAk], b[k * sBk]);
    C[i * sCm + j * sCn] = s;
  }
  ex.sync();
}

// Householder reflector for column (alpha; x) with |x|^2 = xn2, in the
// scalar's own precision: H = I - tau v v^H, v = (1; x * scal),
// H^H (alpha; x) = (beta; 0), beta real.
template <class T>
__device__ inline void householder(T alpha, typename Traits<T>::R xn2, T& tau, T& scal, T& beta) {
  using R = typename Traits<T>::R;
  const R ar = re(alpha), ai = im(alpha);
  if (xn2 == R(0) && (ai == R(0) || ar * ar + ai * ai == R(0))) {  // (the second: squares that underflow)
    tau = zero<T>(); scal = zero<T>(); beta = alpha;
    return;
  }
  R b = sqrt(fmac(fmac(xn2, ai, ai), ar, ar));
  if (ar >= R(0)) b = -b;
  tau = make_scalar<T>((b - ar) / b, -ai / b);
  const R dr = ar - b, di = ai;
  const R d2 = fmac(dr * dr, di, di);
  scal = make_scalar<T>(dr / d2, -di / d2);
  beta = make_scalar<T>(b, R(0));
}

// Reciprocal, square root and reciprocal square root of the rotation angles, in
// which a few units in the last place do not matter (FP32: the hardware's; FP64: exact).
__device__ __forceinline__ float jrcpa(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float jsqrta(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// 1 / sqrt(x) to rounding: one Newton step on the hardware's value
__device__ __forceinline__ float jrsqrt1(float x) {
  const float r = rsqrtf(x);
  return fmaf(r, fmaf(-0.5f * x * r, r, 0.5f), r);
}
__device__ __forceinline__ double jrcpa(double x) { return 1.0 / x; }
__device__ __forceinline__ double jsqrta(double x) { return sqrt(x); }
__device__ __forceinline__ double jrsqrt1(double x) { return 1.0 / sqrt(x); }

// Sum of v over the L consecutive lanes (L a power of two <= 32, aligned)
// that share a column pair; every lane of the warp must call it.
template <class R>
__device__ __forceinline__ R lanes_sum(R v, int L) {
#pragma unroll 1
  for (int o = L >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Reciprocal and reciprocal square root of the Jacobi rotation parameters: in
// FP32 the fast forms (a rotation need only be orthogonal to rounding, and the
// kept singular vectors are re-orthogonalised after the sweeps), exact in FP64.
__device__ __forceinline__ float jrcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double jrcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float jrsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double jrsqrt(double x) { return 1.0 / sqrt(x); }

// Lanes per column for `cols` independent column operations on the
// executor: the largest power of two <= 32 whose groups of lanes cover every
// column at once (1 if the columns outnumber the threads).
template <class X>
__device__ __forceinline__ int lanes_per_column(const X ex, int cols) {
  int L = 32;
  while (L > 1 && L * cols > ex.size()) L >>= 1;
  return L;
}

template <class T>
__device__ __forceinline__ T lanes_sum_scalar(T v, int L);
template <>
__device__ __forceinline__ float lanes_sum_scalar<float>(float v, int L) { return lanes_sum(v, L); }
template <>
__device__ __forceinline__ double lanes_sum_scalar<double>(double v, int L) { return lanes_sum(v, L); }
template <>
__device__ __forceinline__ cfloat lanes_sum_scalar<cfloat>(cfloat v, int L) {
  return {lanes_sum(v.x, L), lanes_sum(v.y, L)};
}
template <>
__device__ __forceinline__ cdouble lanes_sum_scalar<cdouble>(cdouble v, int L) {
  return {lanes_sum(v.x, L), lanes_sum(v.y, L)};
}

// Apply the reflector H = I - f v v^H (v = (1; A[j+1.., j])) from the left
// to columns c0 .. c1-1 of M (rows j..m-1): w_c = v^H M_c, M_c -= v (f w_c).
// Each column is served by a group of L lanes that split its rows and sum
// their parts by shuffles, so that all columns proceed at once.
template <class T, class X>
__device__ __forceinline__ void apply_reflector(const X ex, int m, int j, const T* A, int sm, int sn, T f,
                                                T* Mt, int sMm, int sMn, int c0, int c1) {
  const int nc = c1 - c0;
  if (nc <= 0) return;
  const int L = lanes_per_column(ex, nc);
  const int slots = ex.size() / L;
  const int sub = ex.tid() / L, li = ex.tid() - (ex.tid() / L) * L;
  const T* vcol = A + j * sn;  // v_i = A[i][j] below the diagonal, v_j = 1
#pragma unroll 1
  for (int base = 0; base < nc; base += slots) {
    const int c = c0 + base + sub;
    const bool act = c < c1;
    T* mc = Mt + c * sMn;
    T w = zero<T>();
    if (act) {
#pragma unroll 2
      for (int i = j + li; i < m; i += L) {
        const T v = (i == j) ? one<T>() : vcol[i * sm];
        w = fmac(w, conjg(v), mc[i * sMm]);
      }
    }
    w = lanes_sum_scalar(w, L);
    if (act) {
      const T g = f * w;
#pragma unroll 2
      for (int i = j + li; i < m; i += L) {
        const T v = (i == j) ? one<T>() : vcol[i * sm];
        mc[i * sMm] -= v * g;
      }
    }
  }
}

// In-place Householder QR of A (m x n): on return the upper triangle of the
// leading k = min(m,n) rows holds R, the part below the diagonal holds the
// reflector vectors, tau[0..k) their factors.
template <class T, class X>
__device__ __noinline__ void cta_qr(const X ex, int m, int n, T* A, int sm, int sn, T* tau) {
  using R = typename Traits<T>::R;
  const int k = min(m, n);
  for (int j = 0; j < k; ++j) {
    R part = R(0);
#pragma unroll 1
    for (int i = j + 1 + ex.tid(); i < m; i += ex.size()) part += abs2(A[i * sm + j * sn]);
    const R xn2 = ex.template sum<R>(part);
    const T alpha = A[j * sm + j * sn];
    T t, sc, beta;
    householder(alpha, xn2, t, sc, beta);
    ex.sync();
#pragma unroll 1
    for (int i = j + 1 + ex.tid(); i < m; i += ex.size()) A[i * sm + j * sn] = A[i * sm + j * sn] * sc;
    if (ex.tid() == 0) { A[j * sm + j * sn] = beta; tau[j] = t; }
    ex.sync();
    apply_reflector(ex, m, j, A, sm, sn, conjg(t), A, sm, sn, j + 1, n);
    ex.sync();
  }
}

// Shared-memory factorisation workspace of each chain group: the reflectors
// of a QR step and the columns of the Jacobi sweeps (every step of these
// factorisations depends on the previous one, so each access would otherwise
// wait on L2).  Set at kernel entry; null when the launch has none.
__shared__ void* g_fz[4];
__shared__ long long g_fz_elems;  // scalars of each workspace

// One-sided Jacobi on the columns of W (p x q, column-major), any size: on
// return the columns are mutually orthogonal.  Returns the number of sweeps
// used (max_sweeps: not converged).
// Each sweep visits every column pair once in the round-robin order (n - 1
// rounds of n/2 disjoint pairs, n = q rounded up to even).  A pair is served
// by L consecutive lanes (the largest power of two <= 32 with L x n/2 within
// the executor), which split its rows and combine their partial sums by
// shuffles, so that all pairs of a round proceed at once.
template <class T, class X>
__device__ __noinline__ int cta_jacobi(const X ex, int p, int q, T* W, int ldw, int* sflag, int max_sweeps) {
  using R = typename Traits<T>::R;
  const int n = q + (q & 1);
  const int npair = n / 2;
  int L = 32;
  while (L > 1 && L * npair > ex.size()) L >>= 1;
  const int slots = ex.size() / L;
  const int sub = ex.tid() / L, li = ex.tid() - (ex.tid() / L) * L;
  // convergence threshold on |w_a^H w_b| / (|w_a| |w_b|): the rounding of a
  // length-p dot product is about sqrt(p) eps, below which rotations only
  // stir noise (the threshold of LAPACK's one-sided Jacobi, xGESVJ, scaled
  // by 4)
  const R tol = R(4) * sqrt(R(p > 4 ? p : 4)) * Traits<T>::eps();
  // a column whose norm is below eps ||W||_F (rotations keep ||W||_F) is
  // rounding noise of the matrix: pairs with one are left as they are
  R f2 = R(0);
#pragma unroll 1
  for (int idx = sum_first(ex, p * q); idx < p * q; idx += ex.sum_size()) {
    const int c = idx / p, i = idx - (idx / p) * p;
    f2 += abs2(W[i + (long long)c * ldw]);
  }
  f2 = ex.template sum<R>(f2);
  const R negl = Traits<T>::eps() * Traits<T>::eps() * f2;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (ex.tid() == 0) *sflag = 0;
    ex.sync();
#pragma unroll 1
    for (int r = 0; r < n - 1; ++r) {
#pragma unroll 1
      for (int base = 0; base < npair; base += slots) {
        const int kp = base + sub;
        // round-robin pair kp of round r: (r + kp, r - kp) mod (n - 1), and
        // (r, n - 1) for kp = 0; kp < n/2 keeps each sum within one period
        int a = r, b = n - 1;
        if (kp > 0) {
          a = r + kp;
          if (a >= n - 1) a -= n - 1;
          b = r - kp;
          if (b < 0) b += n - 1;
        }
        if (a > b) { const int t = a; a = b; b = t; }
        const bool act = kp < npair && b < q;
        T* pa = W + (long long)a * ldw;
        T* pb = W + (long long)b * ldw;
        R al = R(0), be = R(0), gr = R(0), gi = R(0);
        if (act) {
          T g = zero<T>();
#pragma unroll 2
          for (int i = li; i < p; i += L) {
            const T wa = pa[i], wb = pb[i];
            al += abs2(wa);
            be += abs2(wb);
            g = fmac(g, conjg(wa), wb);
          }
          gr = re(g);
          gi = im(g);
        }
        al = lanes_sum(al, L);
        be = lanes_sum(be, L);
        gr = lanes_sum(gr, L);
        gi = lanes_sum(gi, L);
        const R ga = sqrt(gr * gr + gi * gi);
        // sqrt(al) sqrt(be), not sqrt(al be): the product of two small squared
        // norms can underflow, and a zero threshold would rotate rounding
        // noise forever
        if (!act || ga == R(0) || !(al > negl) || !(be > negl) || !(ga > tol * (sqrt(al) * sqrt(be)))) continue;
        const R iga = jrcp(ga);
        const R zeta = (be - al) * (R(0.5) * iga);
        // tan of the rotation angle; for |zeta| beyond 1e15, zeta^2 would
        // overflow in FP32, and t = 1 / (2 zeta) to rounding
        const R az = fabs(zeta);
        const R t = (zeta >= R(0) ? R(1) : R(-1)) * jrcp(az > R(1e15) ? R(2) * az : az + sqrt(R(1) + zeta * zeta));
        if (t == R(0)) continue;  // a rotation below rounding leaves the pair as it is
        const R c = jrsqrt(R(1) + t * t), s = c * t;
        // G = [[c, s e^{i phi}], [-s e^{-i phi}, c]], e^{i phi} = g / |g|
        const T eph = make_scalar<T>(gr * iga, gi * iga);
        const T s_e = scale(eph, (R)s);                 // s e^{i phi}
        const T s_ec = scale(conjg(eph), (R)s);         // s e^{-i phi}
#pragma unroll 2
        for (int i = li; i < p; i += L) {
          const T wa = pa[i], wb = pb[i];
          pa[i] = scale(wa, (R)c) - wb * s_ec;
          pb[i] = wa * s_e + scale(wb, (R)c);
        }
        if (li == 0) *sflag = 1;
      }
      ex.sync();
    }
    const int any = *sflag;
    ex.sync();
    if (!any) break;
  }
  ex.sync();
  return sweep;
}

}  // namespace gcf
