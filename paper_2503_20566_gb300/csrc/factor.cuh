// Factorisations of the boundary-MPS compression, held in registers.
//
// A truncating absorption spends its time in chains of dependent small
// steps: one Householder reflector or one set of Jacobi rotations after the
// other on matrices of 16 to 324 rows.  Bandwidth and flops are far from
// their limits there; what counts is the length of a step and the number of
// barriers.  So the columns live in registers for a whole factorisation and
// shared memory carries only what the lanes of other columns need: one
// reflector per QR step (one barrier), the column blocks of a Jacobi round
// (one barrier per 4 x 4 column pairs).
//
// Measured against the same steps with every column in shared memory or L2 (a
// barrier and a pass over the matrix per column or column pair) and Q and J
// formed: log-derivatives at 16x16, chi = 24, 304 configurations 117.7 -> 63.8
// ms (43 with two blocks per SM, 40 with IEEE divisions in the reflectors and
// nothing held across a factorisation); 10x10, D_k = 3, chi = 36, complex, 152
// configurations 403 -> 159 ms (94 with 512 threads a chain, 84 with those two).
//
// All matrices are column-major with leading dimensions padded to 4 rows
// (pad4), so a lane moves 16 bytes of a column at a time.
//
// Algorithms: Householder QR (Golub & Van Loan, "Matrix Computations",
// Alg. 5.2.1; the complex reflector maps x to -sign(Re x_1) |x| e_1), panels
// factored left-looking when the columns exceed one register pass; one-sided
// (Hestenes) Jacobi with the round-robin schedule over blocks of four columns.
#pragma once

#include "common.cuh"
#include "linalg.cuh"

namespace gcf {

// Rows of a 16-byte chunk, and the rows that a chunk per lane of 8 covers.
template <class T> struct Chunk {
  static constexpr int E = 16 / (int)sizeof(T);
  static constexpr int ROWS = 8 * E;
};

template <class T>
__device__ __forceinline__ void load_chunk(T* x, const T* p) {
  constexpr int E = Chunk<T>::E;
  union { float4 v; T t[E]; } u;
  u.v = *reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int e = 0; e < E; ++e) x[e] = u.t[e];
}
template <class T>
__device__ __forceinline__ void store_chunk(T* p, const T* x) {
  constexpr int E = Chunk<T>::E;
  union { float4 v; T t[E]; } u;
#pragma unroll
  for (int e = 0; e < E; ++e) u.t[e] = x[e];
  *reinterpret_cast<float4*>(p) = u.v;
}

// Sum over the 8 lanes of a column.  Every lane of the warp calls it: a warp's
// four columns take all branches together (a shuffle under a mask of 8 lanes
// would run the four one after the other).
template <class R>
__device__ __forceinline__ R sum8(R v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}
__device__ __forceinline__ float sum8s(float v) { return sum8(v); }
__device__ __forceinline__ double sum8s(double v) { return sum8(v); }
__device__ __forceinline__ cfloat sum8s(cfloat v) { return {sum8(v.x), sum8(v.y)}; }
__device__ __forceinline__ cdouble sum8s(cdouble v) { return {sum8(v.x), sum8(v.y)}; }

// x <- x - f v (v^H x) on the 8 lanes of a column, v in registers; the chunks
// q < q0 of v are zero.
template <class T, int Q>
__device__ __forceinline__ void reflect_col(T* x, const T* vr, T f, int q0) {
  constexpr int E = Chunk<T>::E;
  T w0 = zero<T>(), w1 = zero<T>();
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (Q < 3 || q >= q0) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if ((q * E + e) & 1) w1 = fmac(w1, conjg(vr[q * E + e]), x[q * E + e]);
        else w0 = fmac(w0, conjg(vr[q * E + e]), x[q * E + e]);
      }
    }
  const T g = -(f * sum8s(w0 + w1));
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (Q < 3 || q >= q0) {
#pragma unroll
      for (int e = 0; e < E; ++e) x[q * E + e] = fmac(x[q * E + e], vr[q * E + e], g);
    }
}
// The same with v read from memory (its first `lim` rows, whole chunks) twice,
// for columns too long to hold v beside x.
template <class T, int Q>
__device__ __forceinline__ void reflect_col_mem(T* x, const T* v, int li, T f, int q0, int lim) {
  constexpr int E = Chunk<T>::E;
  T w0 = zero<T>(), w1 = zero<T>();
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (q >= q0 && E * (li + 8 * q) < lim) {
      T c[E];
      load_chunk(c, v + E * (li + 8 * q));
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if ((q * E + e) & 1) w1 = fmac(w1, conjg(c[e]), x[q * E + e]);
        else w0 = fmac(w0, conjg(c[e]), x[q * E + e]);
      }
    }
  const T g = -(f * sum8s(w0 + w1));
  asm volatile("" ::: "memory");  // read v again rather than hold it
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (q >= q0 && E * (li + 8 * q) < lim) {
      T c[E];
      load_chunk(c, v + E * (li + 8 * q));
#pragma unroll
      for (int e = 0; e < E; ++e) x[q * E + e] = fmac(x[q * E + e], c[e], g);
    }
}

// Reflector of column j held in x (rows E (li + 8 q) + e of the lane):
// publishes v (1 at row j, zero above) to vb and tau to *tb, and leaves
// beta and v below it in x.  All lanes of the column's warp call it; only
// the column's own (`own`) publish and change x.
template <class T, int Q>
__device__ __forceinline__ void make_reflector(T* x, int j, int nq, int li, bool own, T* vb, T* tb) {
  using R = typename Traits<T>::R;
  constexpr int E = Chunk<T>::E;
  R p0 = R(0), p1 = R(0);
  T al = zero<T>();
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int row = E * (li + 8 * q) + e;
      const R a = row > j ? abs2(x[q * E + e]) : R(0);
      if ((q * E + e) & 1) p1 += a;
      else p0 += a;
      if (row == j) al = x[q * E + e];
    }
  const R xn2 = sum8(p0 + p1);
  al = sum8s(al);
  T t, sc, beta;
  householder(al, xn2, t, sc, beta);
  if (own) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      if (q >= nq) continue;
      T c[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int row = E * (li + 8 * q) + e;
        const T s = x[q * E + e] * sc;
        c[e] = row < j ? zero<T>() : row == j ? one<T>() : s;
        x[q * E + e] = row < j ? x[q * E + e] : row == j ? beta : s;
      }
      store_chunk(vb + E * (li + 8 * q), c);
    }
    if (li == 0) *tb = t;
  }
  __syncwarp();
}

// Householder QR of A (m x n, column-major) in register passes: columns c0 ..
// c0 + groups C - 1, a column per group of 8 lanes and slot, its rows
// in chunks of 16 bytes over the lanes (at most Q chunks a lane).  Reflectors
// of earlier passes come from V.  Per step one barrier: the group that
// holds column j + 1 updates it first and publishes its reflector (two
// buffers in vb) while the others are still updating.  Except in real FP32 a warp
// skips a slot whose four columns are finished or beyond the matrix (SKIP): FP64
// and complex multiply-adds are what a step waits for (amplitudes 8x4, D_k = 3,
// chi = 22, FP64, 16 chains 6.50 -> 5.86 ms; sampling 10x10 chi = 16 FP64 69.7 ->
// 64.6 ms), in real FP32 the branches cost more (three boson lattices, 5472
// chains: 15.06 s without, 15.19 s with).
// Outputs: V (explicit reflector columns: zero above, 1 on the diagonal) and
// tau when V is set; the rows 0 .. k - 1 (k = min(m, n)) of R either as
// column-major Rt (leading dimension ldr) or, TRANS, as the columns of
// W = R^H: W[c + i ldr] = conj(R[i][c]).
template <class T, int Q, int C, bool TRANS, class X>
__device__ __noinline__ void qr_pass(const X ex, int m, int n, const T* A, int lda, T* V, T* Vwork, int ldv, T* tau,
                                     T* Rt, int ldr, T* vb) {
  constexpr int E = Chunk<T>::E;
  const int li = ex.tid() & 7, grp = ex.tid() >> 3, ngrp = ex.size() >> 3;
  const int k = min(m, n), mp = (m + E - 1) / E * E, ldb = (m + 8 * E - 1) / (8 * E) * (8 * E), nq = ldb / (8 * E);
  constexpr bool SKIP = sizeof(T) > 4;
  const int w4 = ex.warp() << 2;  // the warp's first group
  T* tb = vb + 2 * ldb;
  if (!V && n > C * ngrp) V = Vwork;
#pragma unroll 1
  for (int c0 = 0; c0 < n; c0 += C * ngrp) {
    T x[C][Q * E];
#pragma unroll
    for (int s = 0; s < C; ++s) {
      const int c = c0 + s * ngrp + grp;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int row = E * (li + 8 * q);
        if (c < n && row < mp) {
          load_chunk(x[s] + q * E, A + (long long)c * lda + row);
#pragma unroll
          for (int e = 0; e < E; ++e)
            if (row + e >= m) x[s][q * E + e] = zero<T>();
        } else {
#pragma unroll
          for (int e = 0; e < E; ++e) x[s][q * E + e] = zero<T>();
        }
      }
    }
    for (int j = 0; j < min(c0, k); ++j) {
      const T f = conjg(tau[j]);
#pragma unroll
      for (int s = 0; s < C; ++s)
        if (c0 + s * ngrp + w4 < n) reflect_col_mem<T, Q>(x[s], V + (long long)j * ldv, li, f, j / (8 * E), mp);
    }
    if (c0 < k && ex.warp() == 0)
      make_reflector<T, Q>(x[0], c0, nq, li, grp == 0, vb + (c0 & 1) * ldb, tb + (c0 & 1));
#pragma unroll
    for (int s = 0; s < C; ++s) {
#pragma unroll 1
      for (int jj = 0; jj < ngrp; ++jj) {
        const int j = c0 + s * ngrp + jj;
        if (j >= k) break;
        ex.sync();
        const T* v = vb + (j & 1) * ldb;
        const T f = conjg(tb[j & 1]);
        const int q0 = j / (8 * E);
        if (ex.tid() == 0 && V) tau[j] = tb[j & 1];
        const bool cur = !SKIP || (w4 + 3 > jj && c0 + s * ngrp + w4 < n);  // columns of slot s left to this warp
        if constexpr (C > 1) {
          if (SKIP && !cur && !(s + 1 < C && c0 + (s + 1) * ngrp + w4 < n)) continue;
          T vr[Q * E];
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            if (q < nq) load_chunk(vr + q * E, v + E * (li + 8 * q));
            else {
#pragma unroll
              for (int e = 0; e < E; ++e) vr[q * E + e] = zero<T>();
            }
          }
          if (cur) reflect_col<T, Q>(x[s], vr, grp > jj ? f : zero<T>(), q0);
          if ((jj + 1) >> 2 == ex.warp() && jj + 1 < ngrp && j + 1 < k)
            make_reflector<T, Q>(x[s], j + 1, nq, li, grp == jj + 1, vb + ((j + 1) & 1) * ldb, tb + ((j + 1) & 1));
#pragma unroll
          for (int s2 = s + 1; s2 < C; ++s2)
            if (c0 + s2 * ngrp + (SKIP ? w4 : 0) < n) reflect_col<T, Q>(x[s2], vr, f, q0);
        } else {
          if (!cur) continue;
          reflect_col_mem<T, Q>(x[s], v, li, grp > jj ? f : zero<T>(), q0, ldb);
          if ((jj + 1) >> 2 == ex.warp() && jj + 1 < ngrp && j + 1 < k)
            make_reflector<T, Q>(x[s], j + 1, nq, li, grp == jj + 1, vb + ((j + 1) & 1) * ldb, tb + ((j + 1) & 1));
        }
        if (s + 1 < C && jj == ngrp - 1 && ex.warp() == 0 && j + 1 < k)
          make_reflector<T, Q>(x[s + 1 < C ? s + 1 : s], j + 1, nq, li, grp == 0, vb + ((j + 1) & 1) * ldb,
                               tb + ((j + 1) & 1));
      }
    }
#pragma unroll
    for (int s = 0; s < C; ++s) {
      const int c = c0 + s * ngrp + grp;
      if (c >= n) continue;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int row = E * (li + 8 * q);
        if (TRANS) {
#pragma unroll
          for (int e = 0; e < E; ++e)
            if (row + e < k) Rt[c + (long long)(row + e) * ldr] = row + e <= c ? conjg(x[s][q * E + e]) : zero<T>();
        } else if (row < ldr) {
          T o[E];
#pragma unroll
          for (int e = 0; e < E; ++e) o[e] = row + e <= c && row + e < k ? x[s][q * E + e] : zero<T>();
          store_chunk(Rt + (long long)c * ldr + row, o);
        }
        if (V && c < k && row < mp) {
          T o[E];
#pragma unroll
          for (int e = 0; e < E; ++e)
            o[e] = row + e < c ? zero<T>() : row + e == c ? one<T>() : x[s][q * E + e];
          store_chunk(V + (long long)c * ldv + row, o);
        }
      }
    }
    ex.sync();
  }
}

// Y = H_0 H_1 .. H_{k-1} [L; 0] in register passes over the columns of L (k x
// nc, column-major; the identity when L is null).  Columns are independent,
// so there is no barrier; v comes straight from V (cached).  Row i p + u of
// column c goes to Y[(u nc + c) ldy + i] (p = pout): the columns of Y viewed
// as cur x (pout nc).
template <class T, int Q, int C, class X>
__device__ __noinline__ void apply_q_pass(const X ex, int m, int k, const T* V, int ldv, const T* tau, const T* L,
                                          int ldl, int nc, int pout, T* Y, int ldy) {
  constexpr int E = Chunk<T>::E;
  const int li = ex.tid() & 7, grp = ex.tid() >> 3, ngrp = ex.size() >> 3;
  const int mp = (m + E - 1) / E * E, w4 = ex.warp() << 2;
#pragma unroll 1
  for (int c0 = 0; c0 + w4 < nc; c0 += C * ngrp) {  // while there is a column for this warp
    T x[C][Q * E];
#pragma unroll
    for (int s = 0; s < C; ++s) {
      const int c = c0 + s * ngrp + grp;
#pragma unroll
      for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int row = E * (li + 8 * q) + e;
          x[s][q * E + e] = (c < nc && row < k) ? (L ? L[(long long)c * ldl + row] : (row == c ? one<T>() : zero<T>()))
                                                : zero<T>();
        }
    }
    // v of the next AHEAD steps are under way while one is applied (the reads
    // come from L2), as far as registers allow; else v is read twice in place
    constexpr int W = Q * E * (int)sizeof(T) / 4;  // registers of a column
    constexpr int AHEAD = C * W >= 80 ? 0 : (80 - C * W) / W < 3 ? (80 - C * W) / W : 3;
    auto fetch = [&](T* r, int j) {
      const T* v = V + (long long)max(j, 0) * ldv;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int row = E * (li + 8 * q);
        if (row < mp) load_chunk(r + q * E, v + row);
        else {
#pragma unroll
          for (int e = 0; e < E; ++e) r[q * E + e] = zero<T>();
        }
      }
    };
    if constexpr (AHEAD > 0) {
      T vr[AHEAD][Q * E];
      T fr[AHEAD];
#pragma unroll
      for (int a = 0; a < AHEAD; ++a) {
        fetch(vr[a], k - 1 - a);
        fr[a] = tau[max(k - 1 - a, 0)];
      }
#pragma unroll 1
      for (int j0 = k - 1; j0 >= 0; j0 -= AHEAD) {
#pragma unroll
        for (int a = 0; a < AHEAD; ++a) {
          const int j = j0 - a;
          if (j < 0) break;
          const int q0 = j / (8 * E);
#pragma unroll
          for (int s = 0; s < C; ++s)
            if (s == 0 || c0 + s * ngrp + w4 < nc) reflect_col<T, Q>(x[s], vr[a], fr[a], q0);
          fetch(vr[a], j - AHEAD);
          fr[a] = tau[max(j - AHEAD, 0)];
        }
      }
    } else {
#pragma unroll 1
      for (int j = k - 1; j >= 0; --j) {
        const T f = tau[j];
#pragma unroll
        for (int s = 0; s < C; ++s)
          if (s == 0 || c0 + s * ngrp + w4 < nc) reflect_col_mem<T, Q>(x[s], V + (long long)j * ldv, li, f, j / (8 * E), mp);
      }
    }
#pragma unroll
    for (int s = 0; s < C; ++s) {
      const int c = c0 + s * ngrp + grp;
      if (c >= nc) continue;
#pragma unroll
      for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int row = E * (li + 8 * q) + e;
          if (row < m) {
            const int i = row / pout, u = row - i * pout;
            Y[(long long)(u * nc + c) * ldy + i] = x[s][q * E + e];
          }
        }
    }
  }
  ex.sync();
}

// qr_factor for columns longer than the register variants take: the same
// outputs from an in-place QR in `work` (m x n, leading dimension ldv; V
// itself when V is wanted).
template <class T, bool TRANS, class X>
__device__ __noinline__ void qr_general(const X ex, int m, int n, const T* A, int lda, bool want_v, T* work, int ldv,
                                        T* tau, T* Rt, int ldr) {
  const int k = min(m, n);
#pragma unroll 1
  for (int idx = ex.tid(); idx < n * m; idx += ex.size()) {
    const int c = idx / m, i = idx - (idx / m) * m;
    work[i + (long long)c * ldv] = A[i + (long long)c * lda];
  }
  ex.sync();
  cta_qr<T>(ex, m, n, work, 1, ldv, tau);
#pragma unroll 1
  for (int idx = ex.tid(); idx < n * k; idx += ex.size()) {
    const int c = idx / k, i = idx - (idx / k) * k;
    const T r = i <= c ? work[i + (long long)c * ldv] : zero<T>();
    if (TRANS) Rt[c + (long long)i * ldr] = conjg(r);
    else Rt[i + (long long)c * ldr] = r;
  }
  ex.sync();
  if (want_v) {
#pragma unroll 1
    for (int idx = ex.tid(); idx < k * m; idx += ex.size()) {
      const int c = idx / m, i = idx - (idx / m) * m;
      if (i <= c) work[i + (long long)c * ldv] = i < c ? zero<T>() : one<T>();
    }
    ex.sync();
  }
}

template <class T, class X>
__device__ __noinline__ void apply_q_general(const X ex, int m, int k, const T* V, int ldv, const T* tau, const T* L,
                                             int ldl, int nc, int pout, T* Y, int ldy, T* work, int ldk) {
#pragma unroll 1
  for (int idx = ex.tid(); idx < nc * m; idx += ex.size()) {
    const int c = idx / m, i = idx - (idx / m) * m;
    work[i + (long long)c * ldk] = i < k ? (L ? L[(long long)c * ldl + i] : (i == c ? one<T>() : zero<T>()))
                                         : zero<T>();
  }
  ex.sync();
  for (int j = k - 1; j >= 0; --j) {
    apply_reflector(ex, m, j, V, 1, ldv, tau[j], work, 1, ldk, 0, nc);
    ex.sync();
  }
#pragma unroll 1
  for (int idx = ex.tid(); idx < nc * m; idx += ex.size()) {
    const int c = idx / m, row = idx - (idx / m) * m;
    const int i = row / pout, u = row - i * pout;
    Y[(long long)(u * nc + c) * ldy + i] = work[row + (long long)c * ldk];
  }
  ex.sync();
}

// Workspace scalars of qr_factor for columns of m rows.
template <class T>
__host__ __device__ inline int qr_vb_elems(int m) {
  constexpr int RC = Chunk<T>::ROWS;
  return 2 * ((m + RC - 1) / RC * RC) + 4;
}

// Longest columns that the register forms of the QR and of the Jacobi take.  The
// general forms behind them deal their sums to all threads of the executor, so
// their last bits depend on its size: a plan that reaches one keeps one block
// size (see cta_block).
template <class T>
constexpr int qr_max_rows() { return Chunk<T>::ROWS * (sizeof(T) == 4 ? 11 : sizeof(T) == 8 ? 21 : 16); }
template <class T>
constexpr int jacobi_max_rows() { return sizeof(T) == 4 ? 256 : sizeof(T) == 8 ? 128 : 64; }

// Register variants: chunks per lane Q (rows up to Q ROWS) and columns per
// group C.  C is what keeps x within about 64 registers a thread (128 are
// available).  The dispatchers hold nothing after the call: a variant takes
// nearly all registers, so whatever a caller keeps across it goes to local
// memory and, with shared memory taking most of L1, on to L2 (this and AbsorbArgs:
// 1824 chains of three boson lattices, four per CTA 4.79 -> 4.44 s; log-derivatives
// 10x10, D_k = 3, chi = 36 91.2 -> 84.4 ms).
#define GCF_QC_CASES(T, CALL)                                                        \
  if constexpr (sizeof(T) == 4) {                                                    \
    if (nq <= 1) { CALL(1, 3) } else if (nq <= 2) { CALL(2, 3) }                     \
    else if (nq <= 3) { CALL(3, 3) } else if (nq <= 4) { CALL(4, 4) }                \
    else if (nq <= 6) { CALL(6, 2) } else if (nq <= 11) { CALL(11, 1) }              \
  } else if constexpr (sizeof(T) == 8) {                                             \
    if (nq <= 2) { CALL(2, 3) } else if (nq <= 4) { CALL(4, 2) }                     \
    else if (nq <= 8) { CALL(8, 2) } else if (nq <= 12) { CALL(12, 1) }              \
    else if (nq <= 21) { CALL(21, 1) }                                               \
  } else {                                                                           \
    if (nq <= 4) { CALL(4, 2) } else if (nq <= 8) { CALL(8, 1) }                     \
    else if (nq <= 16) { CALL(16, 1) }                                               \
  }

// Householder QR of A (m x n, column-major, leading dimension a multiple of
// 4; m >= n when V is set): R or W = R^H to Rt (see qr_pass), the reflectors
// to V and tau; with V null they are dropped, and Vwork (m x n, leading
// dimension ldv) serves columns of several passes.  A is left as it is (V
// must not be A).  vb: qr_vb_elems(m) scalars, 16-byte aligned.
template <class T, bool TRANS, class X>
__device__ __noinline__ void qr_factor(const X ex, int m, int n, const T* A, int lda, T* V, T* Vwork, int ldv, T* tau, T* Rt,
                                       int ldr, T* vb) {
  const int nq = (m + Chunk<T>::ROWS - 1) / Chunk<T>::ROWS;
#define GCF_QR_CALL(Qv, Cv) return qr_pass<T, Qv, Cv, TRANS>(ex, m, n, A, lda, V, Vwork, ldv, tau, Rt, ldr, vb);
  GCF_QC_CASES(T, GCF_QR_CALL)
#undef GCF_QR_CALL
  qr_general<T, TRANS>(ex, m, n, A, lda, V != nullptr, V ? V : Vwork, ldv, tau, Rt, ldr);
}

// Y = Q [L; 0] with Q from qr_factor's V, tau (see apply_q_pass); `work` (m
// rows x nc, leading dimension ldv) serves the general form.
template <class T, class X>
__device__ __noinline__ void apply_q(const X ex, int m, int k, const T* V, int ldv, const T* tau, const T* L, int ldl,
                                     int nc, int pout, T* Y, int ldy, T* work) {
  const int nq = (m + Chunk<T>::ROWS - 1) / Chunk<T>::ROWS;
  const int ngrp = ex.size() >> 3;
#define GCF_AQ_CALL(Qv, Cv)                                                                              \
  if (nc <= ngrp) return apply_q_pass<T, Qv, 1>(ex, m, k, V, ldv, tau, L, ldl, nc, pout, Y, ldy);        \
  return apply_q_pass<T, Qv, Cv>(ex, m, k, V, ldv, tau, L, ldl, nc, pout, Y, ldy);
  GCF_QC_CASES(T, GCF_AQ_CALL)
#undef GCF_AQ_CALL
  apply_q_general(ex, m, k, V, ldv, tau, L, ldl, nc, pout, Y, ldy, work, ldv);
}

// ---------------------------------------------------------------------------
// One-sided Jacobi on blocks of four columns
// ---------------------------------------------------------------------------

// The sums over LG lanes of four values, value q on the lanes of quarter q
// (lanes q LG/4 ..): 2 + 1 + log2(LG/4) shuffles instead of 4 log2(LG).
template <int LG, class R>
__device__ __forceinline__ R quarter_sum(R v0, R v1, R v2, R v3, int li) {
  const bool h = li & (LG / 2), h2 = li & (LG / 4);
  R a = h ? v2 : v0, b = h ? v3 : v1;
  a += __shfl_xor_sync(0xffffffffu, h ? v0 : v2, LG / 2);
  b += __shfl_xor_sync(0xffffffffu, h ? v1 : v3, LG / 2);
  R s = h2 ? b : a;
  s += __shfl_xor_sync(0xffffffffu, h2 ? a : b, LG / 4);
#pragma unroll
  for (int o = LG / 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <class T, int R>
__device__ __forceinline__ T dot_cols(const T* a, const T* b) {
  T s = zero<T>();
#pragma unroll
  for (int q = 0; q < R; ++q) s = fmac(s, conjg(a[q]), b[q]);
  return s;
}
template <class T, int R>
__device__ __forceinline__ typename Traits<T>::R norm_col(const T* a) {
  typename Traits<T>::R s = 0;
#pragma unroll
  for (int q = 0; q < R; ++q) s += abs2(a[q]);
  return s;
}

// Rotation that makes a pair with squared norms al, be and inner product g
// orthogonal: w_a <- c w_a - conj(se) w_b, w_b <- se w_a + c w_b with
// se = s g / |g|.  Leaves c = 1, se = 0 (rot = false) when the pair is
// orthogonal to rounding or a column is noise; moves the norms along.
// In FP32 the angle comes from the hardware's reciprocal and square root: it
// decides how fast the sweeps converge, not how orthogonal they leave the
// columns (c^2 + s^2 = 1 to rounding for any angle, and the last sweep, which
// rotates nothing, tests norms summed afresh).  With IEEE operations in their
// place the errors against FP64 restatements are the same within their scatter
// (two sets of inputs each, IEEE / hardware: amplitudes 32x32 3.0e-8 / 3.0e-8 and
// 3.3e-8 / 3.4e-8; log-derivatives 16x16 1.6e-7 in all four, 10x10 complex 2.6e-7 /
// 2.5e-7 and 2.3e-7 / 2.3e-7; E_loc 12x9 5.2e-7 / 5.1e-7 and 5.2e-7 / 5.2e-7, 16x16 Z3
// 4.1e-7 / 5.9e-7 and 4.1e-6 / 2.0e-6), complex cases take 2 to 3 % longer and real
// ones 1 % less.
template <class T>
__device__ __forceinline__ bool pair_rotation(typename Traits<T>::R& al, typename Traits<T>::R& be, T g,
                                              typename Traits<T>::R negl, typename Traits<T>::R tol,
                                              typename Traits<T>::R& c, T& se) {
  using R = typename Traits<T>::R;
  c = R(1);
  se = zero<T>();
  const R gr = re(g), gi = im(g);
  R ga, iga;
  if constexpr (Traits<T>::cplx) {
    const R g2 = fmac(gr * gr, gi, gi);
    iga = jrsqrt1(g2);
    ga = g2 * iga;
    if (!(g2 > R(0))) return false;
  } else {
    ga = fabs(gr);
    iga = jrcpa(ga);
    if (ga == R(0)) return false;
  }
  // sqrt(al) sqrt(be), not sqrt(al be): the product of two small squared norms can underflow
  if (!(al > negl) || !(be > negl) || !(ga > tol * (jsqrta(al) * jsqrta(be)))) return false;
  const R zeta = (be - al) * (R(0.5) * iga);
  const R az = fabs(zeta);
  // for |zeta| beyond 1e15, zeta^2 would overflow in FP32, and t = 1 / (2 zeta) to rounding
  const R t = (zeta >= R(0) ? R(1) : R(-1)) * jrcpa(az > R(1e15) ? R(2) * az : az + jsqrta(R(1) + zeta * zeta));
  if (t == R(0)) return false;
  c = jrsqrt1(R(1) + t * t);  // c^2 + s^2 = 1 to rounding whatever the error of t
  const R s = c * t;
  if constexpr (Traits<T>::cplx) se = make_scalar<T>(s * (gr * iga), s * (gi * iga));
  else se = gr >= R(0) ? s : -s;
  al -= t * ga;
  be += t * ga;
  return true;
}

__device__ __forceinline__ float lane_of(float v, int src, int w) { return __shfl_sync(0xffffffffu, v, src, w); }
__device__ __forceinline__ double lane_of(double v, int src, int w) { return __shfl_sync(0xffffffffu, v, src, w); }
__device__ __forceinline__ cfloat lane_of(cfloat v, int src, int w) { return {lane_of(v.x, src, w), lane_of(v.y, src, w)}; }
__device__ __forceinline__ cdouble lane_of(cdouble v, int src, int w) { return {lane_of(v.x, src, w), lane_of(v.y, src, w)}; }

template <int LG, class T>
__device__ __forceinline__ T quarter_sum_s(T v0, T v1, T v2, T v3, int li) {
  if constexpr (Traits<T>::cplx)
    return {quarter_sum<LG>(v0.x, v1.x, v2.x, v3.x, li), quarter_sum<LG>(v0.y, v1.y, v2.y, v3.y, li)};
  else
    return quarter_sum<LG>(v0, v1, v2, v3, li);
}

// Rotations of quarters 0..3 applied to the four column pairs.
template <class T, int LG, int R>
__device__ __forceinline__ void apply_rot(T* a, T* b, typename Traits<T>::R c, T se, int quarter) {
  const typename Traits<T>::R cc = lane_of(c, quarter * (LG / 4), LG);
  const T s = lane_of(se, quarter * (LG / 4), LG);
  const T ns = -conjg(s);
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const T x = a[q], y = b[q];
    a[q] = fmac(scale(x, cc), y, ns);
    b[q] = fmac(scale(y, cc), x, s);
  }
}

// One-sided Jacobi on the columns of W (p x kp, column-major, kp a multiple of
// 8 with zero columns beyond the matrix): on return the columns are mutually
// orthogonal.  Blocks of four columns meet in round-robin order; a pair of
// blocks is held in the registers of LG lanes (R rows of each of the 8
// columns a lane) while all 16 cross pairs (in the first round of a sweep also
// the 12 pairs inside the blocks) are rotated, four disjoint pairs at a time.
// Each quarter of the lanes forms the rotation of one pair (quarter i that of a_i); the squared norms
// are summed once per meeting and moved along by the rotations, so a step
// reduces only the four inner products.  Returns the sweeps used (max_sweeps: not
// converged).
template <class T, int LG, int R, class X>
__device__ __noinline__ int jacobi_blocks(const X ex, int p, int kp, T* W, int ldw, int* sflag, int max_sweeps) {
  using S = typename Traits<T>::R;
  const int nb = kp >> 2, npair = nb >> 1;
  const int slots = ex.size() / LG, sub = ex.tid() / LG, li = ex.tid() & (LG - 1);
  const S tol = S(4) * sqrt(S(p > 4 ? p : 4)) * Traits<T>::eps();
  // a column whose norm is below eps ||W||_F is rounding noise of the matrix:
  // pairs with one are left as they are
  S f2 = S(0);
#pragma unroll 1
  for (int idx = sum_first(ex, p * kp); idx < p * kp; idx += ex.sum_size()) {
    const int c = idx / p, i = idx - (idx / p) * p;
    f2 += abs2(W[i + (long long)c * ldw]);
  }
  f2 = ex.template sum<S>(f2);
  const S negl = Traits<T>::eps() * Traits<T>::eps() * f2;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (ex.tid() == 0) *sflag = 0;
    ex.sync();
    bool rotated = false;
#pragma unroll 1
    for (int r = 0; r < nb - 1; ++r) {
#pragma unroll 1
      for (int base = 0; base < npair; base += slots) {
        const int kq = base + sub;
        // whole warps past the last pair have nothing to do
        if (base + (ex.warp() * 32) / LG >= npair) continue;
        const bool act = kq < npair;
        // round-robin pair kq of round r: blocks (r + kq, r - kq) mod (nb - 1), and (r, nb - 1) for kq = 0
        int a = r, b = nb - 1;
        if (kq > 0) {
          a = r + kq;
          if (a >= nb - 1) a -= nb - 1;
          b = r - kq;
          if (b < 0) b += nb - 1;
        }
        T* wa = W + (long long)(4 * a) * ldw;
        T* wb = W + (long long)(4 * b) * ldw;
        T x[8][R];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < R; ++q) {
            const int row = li + LG * q;
            const bool in = act && row < p;
            x[i][q] = in ? wa[row + (long long)i * ldw] : zero<T>();
            x[4 + i][q] = in ? wb[row + (long long)i * ldw] : zero<T>();
          }
        bool any = false;
        if (r == 0) {
          // pairs inside the two blocks
#pragma unroll
          for (int st = 1; st < 4; ++st) {
            // partner of i is i ^ st; the pairs with i < i ^ st
            constexpr int lo[4][2] = {{0, 0}, {0, 2}, {0, 1}, {0, 1}};
            const int i0 = lo[st][0], i1 = lo[st][1];
            S al = quarter_sum<LG>(norm_col<T, R>(x[i0]), norm_col<T, R>(x[i1]), norm_col<T, R>(x[4 + i0]),
                                   norm_col<T, R>(x[4 + i1]), li);
            S be = quarter_sum<LG>(norm_col<T, R>(x[i0 ^ st]), norm_col<T, R>(x[i1 ^ st]),
                                   norm_col<T, R>(x[4 + (i0 ^ st)]), norm_col<T, R>(x[4 + (i1 ^ st)]), li);
            const T g = quarter_sum_s<LG, T>(dot_cols<T, R>(x[i0], x[i0 ^ st]), dot_cols<T, R>(x[i1], x[i1 ^ st]),
                                             dot_cols<T, R>(x[4 + i0], x[4 + (i0 ^ st)]),
                                             dot_cols<T, R>(x[4 + i1], x[4 + (i1 ^ st)]), li);
            S c;
            T se;
            const bool rot = pair_rotation<T>(al, be, g, negl, tol, c, se);
            if (__any_sync(0xffffffffu, rot)) {
              any = true;
              apply_rot<T, LG, R>(x[i0], x[i0 ^ st], c, se, 0);
              apply_rot<T, LG, R>(x[i1], x[i1 ^ st], c, se, 1);
              apply_rot<T, LG, R>(x[4 + i0], x[4 + (i0 ^ st)], c, se, 2);
              apply_rot<T, LG, R>(x[4 + i1], x[4 + (i1 ^ st)], c, se, 3);
            }
          }
        }
        // cross pairs: quarter i holds the norm of a_i and, in step st, of b_(i + st)
        S al = quarter_sum<LG>(norm_col<T, R>(x[0]), norm_col<T, R>(x[1]), norm_col<T, R>(x[2]), norm_col<T, R>(x[3]), li);
        S be = quarter_sum<LG>(norm_col<T, R>(x[4]), norm_col<T, R>(x[5]), norm_col<T, R>(x[6]), norm_col<T, R>(x[7]), li);
#pragma unroll
        for (int st = 0; st < 4; ++st) {
          const T g = quarter_sum_s<LG, T>(dot_cols<T, R>(x[0], x[4 + (st & 3)]), dot_cols<T, R>(x[1], x[4 + ((1 + st) & 3)]),
                                           dot_cols<T, R>(x[2], x[4 + ((2 + st) & 3)]),
                                           dot_cols<T, R>(x[3], x[4 + ((3 + st) & 3)]), li);
          S c;
          T se;
          const bool rot = pair_rotation<T>(al, be, g, negl, tol, c, se);
          if (__any_sync(0xffffffffu, rot)) {
            any = true;
            apply_rot<T, LG, R>(x[0], x[4 + (st & 3)], c, se, 0);
            apply_rot<T, LG, R>(x[1], x[4 + ((1 + st) & 3)], c, se, 1);
            apply_rot<T, LG, R>(x[2], x[4 + ((2 + st) & 3)], c, se, 2);
            apply_rot<T, LG, R>(x[3], x[4 + ((3 + st) & 3)], c, se, 3);
          }
          be = lane_of(be, (li + LG / 4) & (LG - 1), LG);
        }
        if (any) {
          rotated = true;
          if (act) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int q = 0; q < R; ++q) {
                const int row = li + LG * q;
                if (row < p) {
                  wa[row + (long long)i * ldw] = x[i][q];
                  wb[row + (long long)i * ldw] = x[4 + i][q];
                }
              }
          }
        }
      }
      ex.sync();
    }
    if (rotated && ex.lane() == 0) *sflag = 1;
    ex.sync();
    const int any = *sflag;
    ex.sync();
    if (!any) break;
  }
  return sweep;
}

// Lanes per block pair and rows a lane by the column length p: 16 lanes while
// 8 columns fit about 64 registers, else a warp.
template <class T, class X>
__device__ __noinline__ int jacobi_columns(const X ex, int p, int kp, T* W, int ldw, int* sflag, int max_sweeps) {
  if constexpr (sizeof(T) == 4) {
    if (p <= 16) return jacobi_blocks<T, 16, 1>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 32) return jacobi_blocks<T, 16, 2>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 48) return jacobi_blocks<T, 16, 3>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 80) return jacobi_blocks<T, 16, 5>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 128) return jacobi_blocks<T, 32, 4>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 256) return jacobi_blocks<T, 32, 8>(ex, p, kp, W, ldw, sflag, max_sweeps);
  } else if constexpr (sizeof(T) == 8) {
    if (p <= 16) return jacobi_blocks<T, 16, 1>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 32) return jacobi_blocks<T, 16, 2>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 64) return jacobi_blocks<T, 32, 2>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 128) return jacobi_blocks<T, 32, 4>(ex, p, kp, W, ldw, sflag, max_sweeps);
  } else {
    if (p <= 16) return jacobi_blocks<T, 16, 1>(ex, p, kp, W, ldw, sflag, max_sweeps);
    if (p <= 64) return jacobi_blocks<T, 32, 2>(ex, p, kp, W, ldw, sflag, max_sweeps);
  }
  return cta_jacobi<T>(ex, p, kp, W, ldw, sflag, max_sweeps);
}

// G (kk x kk, column-major) <- (3 I - V^H V) / 2 for V (p x kk, column-major).
template <class T, class X>
__device__ __noinline__ void gram_3i(const X ex, int p, int kk, const T* V, int ldv, T* G) {
  using R = typename Traits<T>::R;
  // 2 x 2 tiles: the four products of a tile share its four columns
  const int t2 = (kk + 1) >> 1;
#pragma unroll 1
  for (int t = ex.tid(); t < t2 * t2; t += ex.size()) {
    const int i0 = 2 * (t / t2), j0 = 2 * (t - (t / t2) * t2);
    const int i1 = min(i0 + 1, kk - 1), j1 = min(j0 + 1, kk - 1);
    const T *a0 = V + i0 * ldv, *a1 = V + i1 * ldv, *b0 = V + j0 * ldv, *b1 = V + j1 * ldv;
    T s00 = zero<T>(), s01 = zero<T>(), s10 = zero<T>(), s11 = zero<T>();
#pragma unroll 4
    for (int q = 0; q < p; ++q) {
      const T x0 = conjg(a0[q]), x1 = conjg(a1[q]), y0 = b0[q], y1 = b1[q];
      s00 = fmac(s00, x0, y0);
      s01 = fmac(s01, x0, y1);
      s10 = fmac(s10, x1, y0);
      s11 = fmac(s11, x1, y1);
    }
    auto put = [&](int i, int j, T s) {
      s = scale(s, R(-0.5));
      if (i == j) s += make_scalar<T>(R(1.5), R(0));
      G[i + j * kk] = s;
    };
    put(i0, j0, s00);
    if (j1 > j0) put(i0, j1, s01);
    if (i1 > i0) put(i1, j0, s10);
    if (i1 > i0 && j1 > j0) put(i1, j1, s11);
  }
  ex.sync();
}

}  // namespace gcf
