// Device layer of the GCF-PEPS contraction: sector gather (Sec. S-2, Eq. S5),
// boundary-MPS row absorption with QR / truncated-SVD compression, and
// the environment steps of the 4-layer strip (plaquette and vertical-hop
// ratios) and of the 3-layer row (gradient and horizontal-hop ratios).
//
// One CTA owns one Markov chain at a time; all tensors of that chain live in
// the CTA's slice of a global scratch arena (L2-resident for the active CTAs).
//
// Tensor layouts (row-major):
//   PEPS tensor at a vertex, "box" of D_k^4: W[l][r][d][u]; missing legs of
//     the open boundary use index 0 only (dimension 1).
//   boundary-MPS site: M[a][i][b] (left bond, physical, right bond); the
//     bond dimensions of every MPS come from host-computed tables bd[0..Lx]
//     with bd[0] = bd[Lx] = 1 and bd[c] = left bond of site c.
//   strip environment: E[a][i][j][b] (B bond, row-r bond, row-(r+1) bond,
//     T bond); row environment: E[a][l][b].
#pragma once

#include "common.cuh"
#include "factor.cuh"
#include "linalg.cuh"
#include "envsteps.cuh"

namespace gcf {

enum { MAX_L = 64 };

// Everything a VMC kernel needs; plain pointers into device memory.
template <class T>
struct KParams {
  // model
  int N, Lx, Ly, Dk, chi, matter, P;
  int n_h, n_v, n_s, cfg_len, n_plaq, n_slots;
  double h, g, J, m;
  double elink[8];         // g (2 - 2 cos(2 pi n / N)) for n = 0..N-1
  const int* Q;            // [Ly*Lx]
  const long long* voff;   // [Lx*Ly] parameter offset of each vertex
  const int* vbs;          // [Lx*Ly] block size of each vertex
  const T* params;
  // MPS tables (see host planner): bond dims of stored MPS and per-step
  // QR dims / SVD flags, each row of Lx+1 ints.
  const int* bondB;  // slot j = B[j-1], j = 0..Ly-1
  const int* bondT;  // slot r = T[r], r = 1..Ly (index 0 unused)
  const int* qrB;    // B-step r (absorbing row r), r = 0..Ly-2
  const int* svdB;
  const int* qrT;    // T-step r, r = 1..Ly-1
  const int* svdT;
  // all tables in one block: the six above, then the derived offB, offT
  // (site offsets per B / T slot, rows of Lx+1) and denseB, denseT (Ly+1
  // flags each: the step takes the identity + core form)
  const int* tab;
  int tab_ints;
  // scratch
  T* scratch;
  long long ws_stride;     // elements per CTA
  long long o_net, o_prop, o_B, o_T, o_Q, o_M1, o_M2, o_M3, o_tau, o_envR, o_envL,
      o_envX, o_envY, o_t1, o_t2, o_t3, o_env3R, o_env3L, o_env3X, o_env3Y, o_G;
  long long mps_stride;
  // Boundary-MPS store.  ck_every = 0: every B[r] / T[r] of the chain is kept
  // (B slot j at o_B + j mps_stride, T slot r at o_T + r mps_stride).
  // ck_every = K >= 2: only every K-th is kept (B slot j with j % K == 0 at
  // o_B + (j / K) mps_stride; T slot r with (Ly - r) % K == 0 at
  // o_T + ((Ly - r) / K) mps_stride) and the slots of one segment between
  // two kept ones live in a segment buffer (o_Bseg / o_Tseg + position
  // mps_stride), recomputed from the segment's kept slot when a pass needs
  // them.
  int ck_every;
  long long o_Bseg, o_Tseg;
  int env_stride, env3_stride;
  int max_sweeps_svd;
  // hot buffers: in dynamic shared memory when hot_in_smem, else in scratch
  int hot_in_smem;
  long long o_sigma, o_sel, o_Z, o_X, o_W1, o_W2, o_W4;
  long long so_net, so_prop, so_cop, so_envL, so_envX, so_envY, so_env3L, so_env3X, so_env3Y,
      so_t1, so_t2, smem_cfg_bytes;
  long long group_smem_bytes;  // grouped kernel: shared bytes per chain group
  int group_threads;          // grouped kernel: threads per chain (128)
  int lockstep;               // grouped kernels: keep a CTA's chains at the same row
  int lock_fault;             // test hook: group 0 never counts in, so the others' waits run out
  int gemm_mode;              // GemmMode of the environment GEMMs (the absorption keeps the scalar's own precision)
  int row_gemm_mode;          // GemmMode of the row environments (O, amplitude, hops)
  // BF16 GEMMs of real chains on the fifth-generation tensor cores
  // (tcgen05.cuh): 1 if used, the bytes of a chain's operand staging area and
  // its byte offset from the start of the chain's dynamic shared memory
  int tc_bf16;
  long long tc_bytes, tc_off;
  // shared-memory factorisation workspace of a chain (linalg.cuh): scalars
  // (0: none) and byte offset from the start of the chain's dynamic shared
  // memory
  long long fz_elems, fz_off;
  // right environments and the staged B / T rows of the current pass
  int mps_in_smem, renv_in_smem;
  long long so_envR, so_env3R, so_sB, so_sT;
  // per-run
  int n_chains, n_sweeps, mode, want;  // mode 0: measure given configs, 1: sample
  unsigned long long seed;
  int8_t* configs;
  double* log_abs;
  double* phase;
  double* e_loc;
  int* block_ids;
  T* O;
  int* accepted;
  int* proposed;
  int* status;       // [4] counters: Gauss violations, tensor-core waits run out, SVDs not converged, lockstep waits run out
};

enum { WANT_AMP = 1, WANT_ELOC = 2, WANT_GRAD = 4 };
enum { ST_GAUSS = 0, ST_TC_TIMEOUT = 1, ST_SVD = 2, ST_PHASE_TIMEOUT = 3 };

// What an absorption keeps across its factorisations, in shared memory: the
// same for every thread of the chain, and those routines leave no registers for
// it (one copy here instead of one per thread in local memory, i.e. L2).
struct AbsorbArgs {
  void *M1, *M2, *M3, *tau, *Qs, *Z, *Xb, *W1, *Vw, *W4, *sigma, *sel, *mout;
  const void *net, *mps_in;
  const int *bdi, *bdo, *qr, *svd;
  int Lx, Dk, pin, pout, row, sd, su, max_sweeps;
  int* status;  // KParams::status
  void *w, *vs, *gg;  // truncate_bond
};

struct Shared {
  AbsorbArgs ab_args;
  double red[64];
  double bcast;
  int iflag[4];
  int ab[MAX_L + 1];
  int zoff[MAX_L + 1];
  int qoff[MAX_L + 1];
  int bd_off[MAX_L + 1];
  int bd_off2[MAX_L + 1];
};

__device__ inline int hl_dim(int c, int Dk) { return c == 0 ? 1 : Dk; }
__device__ inline int hr_dim(int c, int Lx, int Dk) { return c == Lx - 1 ? 1 : Dk; }
__device__ inline int dn_dim(int r, int Dk) { return r == 0 ? 1 : Dk; }
__device__ inline int up_dim(int r, int Ly, int Dk) { return r == Ly - 1 ? 1 : Dk; }

// ---------------------------------------------------------------------------
// Configuration helpers (int8 layout documented in the public header)
// ---------------------------------------------------------------------------
template <class T>
__device__ inline void leg_values(const KParams<T>& k, const int8_t* cfg, int x, int y, int& nl,
                                  int& nr, int& nd, int& nu, int& p) {
  nl = x > 0 ? cfg[y * (k.Lx - 1) + x - 1] : 0;
  nr = x < k.Lx - 1 ? cfg[y * (k.Lx - 1) + x] : 0;
  nd = y > 0 ? cfg[k.n_h + (y - 1) * k.Lx + x] : 0;
  nu = y < k.Ly - 1 ? cfg[k.n_h + y * k.Lx + x] : 0;
  p = cfg[k.n_h + k.n_v + y * k.Lx + x];
}

// Block id selected at (x, y) by cfg, or -1 if the Gauss law (Eq. 1) fails.
template <class T>
__device__ inline int block_of(const KParams<T>& k, const int8_t* cfg, int x, int y) {
  int nl, nr, nd, nu, p;
  leg_values(k, cfg, x, y, nl, nr, nd, nu, p);
  if (p < 0 || p >= k.P) return -1;
  int tot = p + nl + nd - nr - nu - k.Q[y * k.Lx + x];
  tot %= k.N;
  if (tot != 0) return -1;
  const int n[4] = {nl, nr, nd, nu};
  const bool has[4] = {x > 0, x < k.Lx - 1, y > 0, y < k.Ly - 1};
  int last = 3;
  while (!has[last]) --last;
  int bid = p;
  for (int i = 0; i < last; ++i)
    if (has[i]) bid = bid * k.N + n[i];
  return bid;
}

// Copy the selected block of (x, y) into a D_k^4 box (thread-parallel).
template <class T, class X>
__device__ inline void gather_box(const X ex, const KParams<T>& k, int x, int y, int bid, T* box) {
  const int Dk = k.Dk;
  const int dl = hl_dim(x, Dk), dr = hr_dim(x, k.Lx, Dk), dd = dn_dim(y, Dk),
            du = up_dim(y, k.Ly, Dk);
  const int v = y * k.Lx + x;
  const T* src = k.params + k.voff[v] + (long long)bid * k.vbs[v];
  const int bs = dl * dr * dd * du;
#pragma unroll 1
  for (int e = ex.tid(); e < bs; e += ex.size()) {
    int t = e;
    const int iu = t % du; t /= du;
    const int id = t % dd; t /= dd;
    const int ir = t % dr; t /= dr;
    const int il = t;
    box[((il * Dk + ir) * Dk + id) * Dk + iu] = src[e];
  }
}

// Address of B slot j (B[j-1]) and of T slot r (T[r]) in a chain's scratch.
template <class T>
__device__ inline T* bslot_ptr(const KParams<T>& k, T* ws, int j) {
  const int K = k.ck_every;
  if (!K) return ws + k.o_B + (long long)j * k.mps_stride;
  if (j % K == 0) return ws + k.o_B + (long long)(j / K) * k.mps_stride;
  return ws + k.o_Bseg + (long long)(j % K) * k.mps_stride;
}
template <class T>
__device__ inline T* tslot_ptr(const KParams<T>& k, T* ws, int r) {
  const int K = k.ck_every;
  if (!K) return ws + k.o_T + (long long)r * k.mps_stride;
  const int d = k.Ly - r;
  if (d % K == 0) return ws + k.o_T + (long long)(d / K) * k.mps_stride;
  return ws + k.o_Tseg + (long long)(d % K) * k.mps_stride;
}

template <class T>
__device__ inline T* net_box(const KParams<T>& k, T* ws, int x, int y) {
  return ws + k.o_net + (long long)(y * k.Lx + x) * (k.Dk * k.Dk * k.Dk * k.Dk);
}

// ---------------------------------------------------------------------------
// Rescaling by exact powers of two; the returned integer e means
// "tensor_in = 2^e * tensor_out".
// ---------------------------------------------------------------------------
template <class T, class X>
__device__ __noinline__ int rescale(const X ex, T* a, int n) {
  using R = typename Traits<T>::R;
  float mx = 0.f;
#pragma unroll 1
  for (int i = ex.tid(); i < n; i += ex.size()) mx = fmaxf(mx, (float)absmax1(a[i]));
  mx = ex.maxf(mx);
  if (!(mx > 0.f) || !isfinite(mx)) return 0;
  const int e = exp2_of(mx);
  const R s = pow2r<R>(-e);
#pragma unroll 1
  for (int i = ex.tid(); i < n; i += ex.size()) a[i] = scale(a[i], s);
  ex.sync();
  return e;
}

// sum_k A[k] B[k] (no conjugation), broadcast to all threads as (re, im)
template <class T, class X>
__device__ __noinline__ void cta_dot(const X ex, const T* A, const T* B, int n, typename Traits<T>::R& r,
                               typename Traits<T>::R& i) {
  using R = typename Traits<T>::R;
  T s = zero<T>();
#pragma unroll 1
  for (int k = sum_first(ex, n); k < n; k += ex.sum_size()) s = fmac(s, A[k], B[k]);
  r = re(s);
  i = im(s);
  ex.template sum2<R>(r, i);
}

// ---------------------------------------------------------------------------
// Exact compression in identity + core form.
// When every output bond of a step is at full rank, bd[c] = min(p^c, p^(L-c))
// (p = D_k, L = Lx; no truncation), the compressed boundary state is an
// exact MPS whose sites left of m = floor(L/2) are identity isometries
// M[a][i][a*p + i], whose sites right of m are identity isometries
// M[i*p^(L-1-c) + b][i][b], and whose site m holds the normalised dense state
// v[(u_0..u_{m-1})][u_m][(u_{m+1}..u_{L-1})].  It is the same state the sweeps
// of the general path produce, in a different gauge.  The dense state is obtained by
// contracting the input MPS to a vector and applying the row MPO site by site.
// Returns the binary exponent e of the scale (state = 2^e * output).
// ---------------------------------------------------------------------------
template <class T, class X>
__device__ __noinline__ int dense_absorb(const X ex, const KParams<T>& k, Shared& sh, const T* net, const T* mps_in,
                                            const int* bdi, int pin, int row, int flip, T* mout,
                                            const int* bdo, int pout, T* bufA, T* bufB) {
  const int Lx = k.Lx, Dk = k.Dk;
  const int D3 = Dk * Dk * Dk, D2 = Dk * Dk;
  const int sd = flip ? 1 : Dk, su = flip ? Dk : 1;
  // 1. input vector v[(i_0..i_{L-1})], i_0 most significant
  if (ex.tid() == 0) bufA[0] = one<T>();
  ex.sync();
  int rows = 1;
  for (int c = 0; c < Lx; ++c) {
    const T* M = mps_in + sh.bd_off[c];
    // bufB[(p, i)][b] = sum_a bufA[p][a] M[a][(i b)]
    cta_gemm<T>(ex, rows, pin * bdi[c + 1], bdi[c], bufA, bdi[c], 1, M, pin * bdi[c + 1], 1, bufB,
                pin * bdi[c + 1], 1);
    rows *= pin;
    T* t = bufA; bufA = bufB; bufB = t;
  }
  // 2. MPO sweep: t_c[h][U][u][Dr] = sum_{h', d} W_c[h'][h][d][u] t_{c-1}[h'][U][d][Dr]
  int NU = 1, ND = rows / pin;  // ND = pin^(L-1) before position 0
  for (int c = 0; c < Lx; ++c) {
    const int hl = hl_dim(c, Dk), hr = hr_dim(c, Lx, Dk);
    const T* W = net + (long long)(row * Lx + c) * (Dk * Dk * Dk * Dk);
    const int nout = hr * NU * pout * ND;
#pragma unroll 1
    for (int idx = ex.tid(); idx < nout; idx += ex.size()) {
      int t = idx;
      const int Dr = t % ND; t /= ND;
      const int u = t % pout; t /= pout;
      const int U = t % NU; t /= NU;
      const int h = t;
      T s = zero<T>();
      for (int hp = 0; hp < hl; ++hp)
        for (int d = 0; d < pin; ++d)
          s = fmac(s, W[hp * D3 + h * D2 + d * sd + u * su], bufA[((hp * NU + U) * pin + d) * ND + Dr]);
      bufB[idx] = s;
    }
    ex.sync();
    T* tt = bufA; bufA = bufB; bufB = tt;
    NU *= pout;
    if (c < Lx - 1) ND /= pin;
  }
  // 3. scale v' (length pout^L, bufA) by a power of two near its norm
  using R = typename Traits<T>::R;
  const int nv = NU;
  R s2 = R(0);
#pragma unroll 1
  for (int i = sum_first(ex, nv); i < nv; i += ex.sum_size()) s2 += abs2(bufA[i]);
  s2 = ex.template sum<R>(s2);
  const int e = (s2 > R(0) && isfinite((float)s2)) ? exp2_of((float)sqrt(s2)) : 0;
  const R inv = pow2r<R>(-e);
  // 4. identity sites and the core
  const int m = Lx / 2;
  for (int c = 0; c < Lx; ++c) {
    const int a = bdo[c], b = bdo[c + 1];
    T* site = mout + sh.bd_off2[c];
    const int n = a * pout * b;
    if (c == m) {
#pragma unroll 1
      for (int i = ex.tid(); i < n; i += ex.size()) site[i] = scale(bufA[i], inv);
    } else {
#pragma unroll 1
      for (int i = ex.tid(); i < n; i += ex.size()) {
        const int ib = i % b, ii = (i / b) % pout, ia = i / (b * pout);
        const bool on = (c < m) ? (ib == ia * pout + ii) : (ia == ii * b + ib);
        site[i] = on ? one<T>() : zero<T>();
      }
    }
  }
  ex.sync();
  return e;
}

// sel[0..kk) <- the indices of the kk largest of sigma[0..k0), largest first
// (ties: lower index first; NaN above all, so that every rank is taken once).
template <class R, class X>
__device__ inline void select_largest(const X ex, int k0, int kk, const R* sigma, int* sel) {
#pragma unroll 1
  for (int j = ex.tid(); j < k0; j += ex.size()) {
    int rank = 0;
    const R sj = sigma[j];
    for (int i = 0; i < k0; ++i) {
      const R si = sigma[i];
      const bool above = si > sj || (si != si && sj == sj);
      const bool below = sj > si || (sj != sj && si == si);
      rank += above || (!below && i < j);
    }
    if (rank < kk) sel[rank] = j;
  }
  ex.sync();
}

// The Frobenius norm of a column-major matrix scaled to [0.5, 1) by an exact
// power of two; the returned integer e means "matrix in = 2^e * matrix out".
template <class T, class X>
__device__ __noinline__ int frob_rescale_cm(const X ex, int rows, int cols, T* a, int ld) {
  using R = typename Traits<T>::R;
  R s2 = R(0);
#pragma unroll 1
  for (int idx = sum_first(ex, cols * rows); idx < cols * rows; idx += ex.sum_size()) {
    const int c = idx / rows, i = idx - (idx / rows) * rows;
    s2 += abs2(a[c * ld + i]);
  }
  s2 = ex.template sum<R>(s2);
  if (!(s2 > R(0)) || !isfinite((float)s2)) return 0;
  const int e = exp2_of((float)sqrt(s2));
  const R s = pow2r<R>(-e);
#pragma unroll 1
  for (int idx = ex.tid(); idx < cols * rows; idx += ex.size()) {
    const int c = idx / rows, i = idx - (idx / rows) * rows;
    a[c * ld + i] = scale(a[c * ld + i], s);
  }
  ex.sync();
  return e;
}

// X[(i u)][(b r)] = sum_{l,d} T1[(l d b)][i] W[l][r][d][u] (column-major X, T1
// with i contiguous): a thread holds the l, d values of one (i, b).
struct SiteDims {
  int l, r, pin, pout, sd, su, rows, nb, ldt, ldx;
};
template <class T, int DK, class X>
__device__ __noinline__ void site_product(const X ex, const SiteDims d, const T* W, const T* T1, T* Xc) {
#pragma unroll 1
  for (int idx = ex.tid(); idx < d.rows * d.nb; idx += ex.size()) {
    const int ib = idx / d.rows, i = idx - (idx / d.rows) * d.rows;
    T t[DK][DK];
#pragma unroll
    for (int il = 0; il < DK; ++il)
#pragma unroll
      for (int dd = 0; dd < DK; ++dd)
        t[il][dd] = (il < d.l && dd < d.pin) ? T1[((il * d.pin + dd) * d.nb + ib) * d.ldt + i] : zero<T>();
#pragma unroll
    for (int ir = 0; ir < DK; ++ir)
#pragma unroll
      for (int iu = 0; iu < DK; ++iu) {
        if (ir >= d.r || iu >= d.pout) continue;
        T s = zero<T>();
#pragma unroll
        for (int il = 0; il < DK; ++il)
#pragma unroll
          for (int dd = 0; dd < DK; ++dd)
            if (il < d.l && dd < d.pin)
              s = fmac(s, t[il][dd], W[il * (DK * DK * DK) + ir * (DK * DK) + dd * d.sd + iu * d.su]);
        Xc[(ib * d.r + ir) * d.ldx + i * d.pout + iu] = s;
      }
  }
  ex.sync();
}

// Truncated step of a bond: Y (yr x yc, column-major) ~ carry site, with site
// the kk x yc (row-major) isometry of Y's kk leading right singular vectors
// and carry = Y site^H (yr x kk, column-major).  Y = Q R by Householder QR; of
// it only R is formed, as the columns of W = R^H, whose one-sided Jacobi gives
// W J = V Sigma: the rotated columns themselves are the right singular vectors
// of Y, so neither Q nor J is ever needed (R^H, not Y^H, because its columns
// are closer to orthogonal and converge in fewer sweeps).  The kk columns of
// largest norm are normalised, and one Newton-Schulz step V (3 I - V^H V) / 2
// brings them from the sweeps' threshold to orthogonal at rounding.  Columns
// of norm below eps |Y| are rounding noise, which the sweeps leave alone: their
// directions are dropped (zero rows of site), with the rounding of the sums of
// squares (below 2^-10 for a thousand terms in any order) on top: the sweeps
// add the same squares in another order, and a column that they left alone may
// lie along a leading one, so none of those may be kept.
// Work: W, V and the Gram matrix in the chain's shared-memory workspace as
// far as they fit it, else in M1, M2, M3 (mat_max each); Vw, tau for the QR.
// Returns whether the sweeps converged.
template <class T, class X>
__device__ __noinline__ bool truncate_bond(const X ex, Shared& sh, int yr, int yc, int kk, const T* Y, int ldy, T* carry,
                                           int ldl, T* site) {
  using R = typename Traits<T>::R;
  AbsorbArgs& g = sh.ab_args;
  const int k0 = min(yr, yc), kp = (k0 + 7) & ~7, ldw = pad4(yc);
  {
    const int nvb = qr_vb_elems<T>(yr), nw = ldw * kp, nv = ldw * kk, ng = pad4(kk * kk);
    T* fz = (T*)g_fz[ex.slot()];
    long long room = fz ? g_fz_elems : 0;
    auto place = [&](long long n, void* other) {
      if (n > room) return (T*)other;
      T* q = fz;
      fz += n;
      room -= n;
      return q;
    };
    T* vb = place(nvb, carry);  // the carry is written last
    T* w = place(nw, g.M1);
    T* vs = place(nv, g.M2);
    T* gg = place(ng, g.M3);
    if (ex.tid() == 0) { g.w = w; g.vs = vs; g.gg = gg; }
#pragma unroll 1
    for (int idx = ex.tid(); idx < (kp - k0) * ldw; idx += ex.size()) w[k0 * ldw + idx] = zero<T>();
    qr_factor<T, true>(ex, yr, yc, Y, ldy, (T*)nullptr, (T*)g.Vw, ldy, (T*)g.tau, w, ldw, vb);
  }
  const bool conv = jacobi_columns<T>(ex, yc, kp, (T*)g.w, ldw, &sh.iflag[0], g.max_sweeps) < g.max_sweeps;
  {
    const T* w = (const T*)g.w;
    T* vs = (T*)g.vs;
    R* sigma = (R*)g.sigma;
    int* sel = (int*)g.sel;
#pragma unroll 1
    for (int j = ex.warp(); j < k0; j += ex.nwarps()) {
      R s2 = R(0);
      for (int i = ex.lane(); i < yc; i += 32) s2 += abs2(w[j * ldw + i]);
      s2 = warp_sum(s2);
      if (ex.lane() == 0) sigma[j] = s2;
    }
    ex.sync();
    R f2 = R(0);
    for (int j = ex.lane(); j < k0; j += 32) f2 += sigma[j];
    f2 = warp_sum(f2);
    const R negl = Traits<T>::eps() * Traits<T>::eps() * f2 * R(1 + 1.0 / 1024);
    select_largest(ex, k0, kk, sigma, sel);
#pragma unroll 1
    for (int idx = ex.tid(); idx < kk * yc; idx += ex.size()) {
      const int n = idx / yc, i = idx - (idx / yc) * yc;
      const R s2 = sigma[sel[n]];
      vs[n * ldw + i] = s2 > negl ? scale(w[sel[n] * ldw + i], R(1) / sqrt(s2)) : zero<T>();
    }
    ex.sync();
  }
  gram_3i<T>(ex, yc, kk, (const T*)g.vs, ldw, (T*)g.gg);
  // V' over W, which is not needed any more
  cta_gemm_out<T>(ex, yc, kk, kk, (const T*)g.vs, {1, 1, 0}, ldw, (const T*)g.gg, 1, kk,
                  OutMap<T>{(T*)g.w, {1, 1, 0}, kk, 0, ldw});
  cta_gemm_out<T>(ex, yr, kk, yc, Y, {1, 1, 0}, ldy, (const T*)g.w, 1, ldw, OutMap<T>{carry, {1, 1, 0}, kk, 0, ldl});
  const T* w = (const T*)g.w;
#pragma unroll 1
  for (int idx = ex.tid(); idx < kk * yc; idx += ex.size()) {
    const int n = idx / yc, i = idx - (idx / yc) * yc;
    site[idx] = conjg(w[n * ldw + i]);
  }
  ex.sync();
  return conv;
}

// ---------------------------------------------------------------------------
// Row absorption + compression.
//   in : MPS `mps_in` (bond table bdi, physical dim pin) and row `row` whose
//        tensors are boxes net_box(x=c, y=row); flip=1 swaps the d and u legs
//        (absorption from above).
//   out: MPS `mout` with bond table bdo, physical dim pout; qr/svd: the
//        step's QR left dims and SVD flags.  Returns the binary exponent e of
//        the scale (output state = 2^e * mout, up to the discarded weight).
// Algorithm: QR left to right on the absorbed MPS (left-canonical form),
// then right to left the truncated SVD of every bond above chi.  Where a
// bond needs no factorisation none is made: a left site with no more rows
// than columns has the identity as its isometry (its matrix is the carry),
// and so has a right site whose outer dimensions already fit the bond.  The
// isometries of the left sweep stay products of reflectors, applied to the
// carry of the right sweep (kc columns) instead of being formed.
// ---------------------------------------------------------------------------
template <class T, class X>
__device__ __noinline__ int absorb_general(const X ex, Shared& sh) {
  const AbsorbArgs& g = sh.ab_args;
  const int Lx = g.Lx;
  int logs = 0;
  // General path.  Z_c (absorbed sites) right of cL; then a QR sweep from the
  // left over the bonds that must shrink (all bonds if the step truncates),
  // then a sweep from the right over the bonds that must shrink (truncated SVD,
  // or the identity where the outer dimensions fit); sites in between are the
  // absorbed tensors with the carries multiplied in.  Without truncation this
  // reaches the exact state with the step's bond dimensions; with truncation it
  // is the full canonical sweep.  Where no bond shrinks from the left (cL = 0:
  // the first rows of a lattice) every site is a Z_c, and one that needs no
  // carry either goes to the output as it is: those steps are short, and the
  // code of a longer way through them costs more than their work (16 amplitudes on
  // 4x4, D_k = 3, chi = 9, complex FP32: 166 -> 156 us; 608 FP32 chains of 4x4
  // with bosons, four sweeps: 6.13 -> 5.80 ms).
  if (ex.tid() == 0) {
    const int *bdi = g.bdi, *qr = g.qr, *svd = g.svd;
    const int Dk = g.Dk, pout = g.pout;
    int any_svd = 0;
    for (int c = 1; c < Lx; ++c) any_svd |= svd[c];
    int zo = 0, qo = 0;
    for (int c = 0; c <= Lx; ++c) sh.ab[c] = (c == 0 || c == Lx) ? 1 : bdi[c] * Dk;
    for (int c = 0; c < Lx; ++c) {
      sh.zoff[c] = zo;
      zo += sh.ab[c] * pout * sh.ab[c + 1];
      // reflectors and their factors (the isometry of a QR site)
      sh.qoff[c] = qo;
      if (qr[c] * pout > qr[c + 1]) qo += (pad4(qr[c] * pout) + 1) * qr[c + 1] + 32;
      qo = (qo + 31) & ~31;
    }
    int cl = 0;
    while (cl < Lx - 1 && (any_svd || qr[cl] * pout < sh.ab[cl + 1])) ++cl;
    sh.iflag[1] = cl;
  }
  ex.sync();
  const int cL = sh.iflag[1];
  for (int c = cL ? cL + 1 : 0; c < Lx; ++c) {
    const int Dk = g.Dk, pin = g.pin, pout = g.pout, sd = g.sd, su = g.su;
    const int a = g.bdi[c], b = g.bdi[c + 1];
    const int l = hl_dim(c, Dk), r = hr_dim(c, Lx, Dk);
    const T* M = (const T*)g.mps_in + sh.bd_off[c];
    const T* W = (const T*)g.net + (long long)(g.row * Lx + c) * (Dk * Dk * Dk * Dk);
    const int nZ = a * l * pout * b * r;
    T* Zc = (T*)g.Z + sh.zoff[c];
#pragma unroll 1
    for (int idx = ex.tid(); idx < nZ; idx += ex.size()) {
      int t = idx;
      const int ir = t % r; t /= r;
      const int ib = t % b; t /= b;
      const int iu = t % pout; t /= pout;
      const int il = t % l; t /= l;
      const int ia = t;
      T s = zero<T>();
      for (int d = 0; d < pin; ++d)
        s = fmac(s, M[(ia * pin + d) * b + ib], W[il * Dk * Dk * Dk + ir * Dk * Dk + d * sd + iu * su]);
      Zc[idx] = s;
    }
  }
  // ---- left QR sweep over sites 0..cL-1 (site cL: X only); carry Rc (Rrows x ab[c], column-major)
  T* Rc = (T*)g.M3;
  if (ex.tid() == 0) Rc[0] = one<T>();
  ex.sync();
  int Rrows = 1, ldr = 4, ldxb = 4;
  for (int c = 0; c <= cL && cL; ++c) {
    const int rows = Rrows * g.pout, ldx = pad4(rows);
    // X ((Rrows pout) x (b, r)) = sum R[.][(a l)] M[a][d][b] W[l][r][d][u], the
    // MPS site first: its a bond is the large one
    T* Xc = (T*)(c == cL ? g.Xb : Rc == g.M3 ? g.M1 : g.M3);
    {
      const int nb = g.bdi[c + 1], pin = g.pin, Dk = g.Dk, l = hl_dim(c, Dk), ldt = pad4(Rrows);
      T* T1 = (T*)g.M2;  // [(l d b)][Rrows]
      cta_gemm_out<T>(ex, l * Rrows, pin * nb, g.bdi[c], Rc, {Rrows, ldr, 1}, l * ldr, (const T*)g.mps_in + sh.bd_off[c],
                      pin * nb, 1, OutMap<T>{T1, {Rrows, pin * nb * ldt, 1}, pin * nb, 0, ldt});
    }
    {
      const int Dk = g.Dk;
      const T* W = (const T*)g.net + (long long)(g.row * Lx + c) * (Dk * Dk * Dk * Dk);
      const SiteDims d{hl_dim(c, Dk), hr_dim(c, Lx, Dk), g.pin, g.pout, g.sd, g.su, Rrows, g.bdi[c + 1], pad4(Rrows), ldx};
      switch (Dk) {
        case 1: site_product<T, 1>(ex, d, W, (const T*)g.M2, Xc); break;
        case 2: site_product<T, 2>(ex, d, W, (const T*)g.M2, Xc); break;
        default: site_product<T, 3>(ex, d, W, (const T*)g.M2, Xc); break;
      }
    }
    ldxb = ldx;
    if (c == cL) break;
    const int cols = sh.ab[c + 1];
    if (rows <= cols) {
      Rc = Xc;
      ldr = ldx;
      Rrows = rows;
    } else {
      T* V = (T*)g.Qs + sh.qoff[c];
      T* fz = (T*)g_fz[ex.slot()];
      ldr = pad4(cols);
      qr_factor<T, false>(ex, rows, cols, Xc, ldx, V, (T*)nullptr, ldx, V + ldx * cols, Rc, ldr,
                          (fz && qr_vb_elems<T>(rows) <= g_fz_elems) ? fz : (T*)g.M2);
      Rrows = cols;
    }
    logs += frob_rescale_cm(ex, Rrows, sh.ab[c + 1], Rc, ldr);
  }
  // ---- right sweep over every site.  The carry Lc (rd x kc, column-major) is
  // the identity while no bond to the right has been reduced.
  // Y (cur x (pout, kc), column-major): site c times the carry.
  bool ident = true;
  int kc = 1, ldl = 4;
  T* Y = (T*)g.W1;
  T* Lc = (T*)g.W4;
  for (int c = Lx - 1; c >= 0; --c) {
    const int cur = (c < cL) ? g.qr[c] : (c == cL ? Rrows : sh.ab[c]);
    const int rd = (c < cL) ? g.qr[c + 1] : sh.ab[c + 1];
    const int pout = g.pout, n = ident ? rd : kc, yc = pout * n, ldy = pad4(cur), rows = cur * pout;
    const bool from_x = c == cL && cL, shrinks = c >= 1 && (g.svd[c] || g.bdo[c] < cur);
    T* site = (T*)g.mout + sh.bd_off2[c];
    if (ident && c >= cL && !shrinks) {
      // the absorbed site as it is
      const T* S = from_x ? (const T*)g.Xb : (const T*)g.Z + sh.zoff[c];
#pragma unroll 1
      for (int idx = ex.tid(); idx < rows * n; idx += ex.size())
        site[idx] = from_x ? S[(idx % n) * ldxb + idx / n] : S[idx];
      ex.sync();
      logs += rescale(ex, site, rows * n);
      continue;
    }
    if (c < cL && rows > rd) {
      const T* V = (const T*)g.Qs + sh.qoff[c];
      const int ldv = pad4(rows);
      apply_q<T>(ex, rows, rd, V, ldv, V + ldv * rd, ident ? (const T*)nullptr : Lc, ldl, n, pout, Y, ldy, (T*)g.M1);
    } else if (c < cL || ident) {
      // identity isometry (Y = the carry) or identity carry (Y = the site)
      const T* S = from_x ? (const T*)g.Xb : (const T*)g.Z + sh.zoff[c];
#pragma unroll 1
      for (int idx = ex.tid(); idx < rows * n; idx += ex.size()) {
        const int m = idx / rows, q = idx - (idx / rows) * rows;
        const int i = q / pout, u = q - (q / pout) * pout;
        T v;
        if (c < cL) v = ident ? (q == m ? one<T>() : zero<T>()) : Lc[m * ldl + q];
        else v = from_x ? S[m * ldxb + q] : S[q * rd + m];
        Y[(u * n + m) * ldy + i] = v;
      }
      ex.sync();
    } else {
      const T* S = from_x ? (const T*)g.Xb : (const T*)g.Z + sh.zoff[c];
      cta_gemm_out<T>(ex, rows, n, rd, S, {1, from_x ? 1 : rd, 0}, from_x ? ldxb : 1, Lc, 1, ldl,
                      OutMap<T>{Y, {pout, 1, n * ldy}, n, 0, ldy});
    }
    if (shrinks) {
      const int kk = g.bdo[c];
      if (!g.svd[c]) {
        // yc = kk columns already fit the bond: the identity is the isometry
#pragma unroll 1
        for (int idx = ex.tid(); idx < kk * yc; idx += ex.size())
          site[idx] = idx / yc == idx % yc ? one<T>() : zero<T>();
        T* t = Lc; Lc = Y; Y = t;
        ldl = ldy;
      } else {
        ldl = pad4(cur);
        if (!truncate_bond<T>(ex, sh, cur, yc, kk, Y, ldy, Lc, ldl, site) && ex.tid() == 0)
          atomicAdd(&g.status[ST_SVD], 1);
      }
      logs += frob_rescale_cm(ex, cur, g.bdo[c], Lc, ldl);
      kc = g.bdo[c];
      ident = false;
    } else {
      // no reduction at this site's left bond (cur == bdo[c]): keep Y
#pragma unroll 1
      for (int idx = ex.tid(); idx < cur * yc; idx += ex.size()) {
        const int i = idx / yc, j = idx - (idx / yc) * yc;
        site[idx] = Y[j * ldy + i];
      }
      ex.sync();
      logs += rescale(ex, site, cur * yc);
      ident = true;
    }
  }
  return logs;
}

template <class T, class X>
__device__ __noinline__ int absorb_compress(const X ex, const KParams<T>& k, T* ws, T* hot_base, Shared& sh, const T* net,
                                  const T* mps_in, const int* bdi, int pin, int row, int flip, T* mout,
                                  const int* bdo, int pout, const int* qr, const int* svd, const int* offi,
                                  const int* offo, int dense) {
#pragma unroll 1
  for (int c = ex.tid(); c <= k.Lx; c += ex.size()) {
    sh.bd_off[c] = offi[c];
    sh.bd_off2[c] = offo[c];
  }
  ex.sync();
  // Dense (identity + core) path: every output bond at full rank and the
  // dense state small enough (flag planned on the host).
  if (dense) {
    T* bufA = k.hot_in_smem ? hot_base + k.so_t1 : ws + k.o_t1;
    T* bufB = k.hot_in_smem ? hot_base + k.so_t2 : ws + k.o_t2;
    return dense_absorb<T>(ex, k, sh, net, mps_in, bdi, pin, row, flip, mout, bdo, pout, bufA, bufB);
  }
  if (ex.tid() == 0) {
    AbsorbArgs& a = sh.ab_args;
    a.M1 = ws + k.o_M1; a.M2 = ws + k.o_M2; a.M3 = ws + k.o_M3; a.tau = ws + k.o_tau; a.Qs = ws + k.o_Q;
    a.Z = ws + k.o_Z; a.Xb = ws + k.o_X; a.W1 = ws + k.o_W1; a.Vw = ws + k.o_W2; a.W4 = ws + k.o_W4; a.sigma = ws + k.o_sigma; a.sel = ws + k.o_sel;
    a.mout = mout; a.net = net; a.mps_in = mps_in; a.bdi = bdi; a.bdo = bdo; a.qr = qr; a.svd = svd;
    a.Lx = k.Lx; a.Dk = k.Dk; a.pin = pin; a.pout = pout; a.row = row;
    a.sd = flip ? 1 : k.Dk; a.su = flip ? k.Dk : 1; a.max_sweeps = k.max_sweeps_svd; a.status = k.status;
  }
  ex.sync();
  return absorb_general<T>(ex, sh);
}
}  // namespace gcf
