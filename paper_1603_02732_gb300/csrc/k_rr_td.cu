// FP64 Rayleigh-Ritz, one CTA or one cluster of CTAs per problem (orthonormalisation + subspace
// diagonalisation of Algorithm 1): S = L L^T, C = L^-1 Hs L^-T, C = V diag(eps) V^T, Tm = L^-T V, so
// that X Tm is orthonormal and diagonalises H in the subspace.
//
//  1. Cholesky of S.
//  2. W = L^-1 Hs and C = W L^-T by forward substitution down columns.
//  3. Householder tridiagonalisation of C (Golub & Van Loan, section 8.3.1).
//  4. Divide and conquer on the tridiagonal matrix (Cuppen, Numer. Math. 36, 177 (1981)): leaves of
//     two rows, merged pairwise, a merge being the rank-one problem diag(delta) + rho z z^T.  Roots of
//     its secular equation by the two-pole rational interpolation of Bunch, Nielsen & Sorensen (Numer.
//     Math. 31, 31 (1978)), each as an offset from its nearest pole; z is then recomputed from the
//     roots (Gu & Eisenstat, SIAM J. Matrix Anal. 15, 1266 (1994)), which makes the vectors orthogonal
//     to rounding however close the roots lie.  Nothing is deflated: poles closer than one unit of
//     rounding of the matrix are moved that far apart and weights below rounding are raised to it,
//     both of the size of the rounding errors already there; a negligible rho leaves the two halves as
//     they are.
//  5. V = Householder reflectors applied to the eigenvectors; Tm = L^-T V by back substitution.
//
// What bounds it, and why this form: one CTA (one SM) works on a chain of dependent steps, so the
// time is barriers, latencies and the two FP64 lanes of the SM (a warp's DFMA holds them 16 cycles).
// A cyclic Jacobi eigensolve (k_rr) takes about 200 rounds of two block barriers and 6 n^2 operations
// each.  Here the matrices stay in the registers of MW matrix warps, row i in warp i / RPW, column j in
// lane j mod 32 (few warps with 8 to 16 rows each: the overhead of a step is paid per warp); the
// Cholesky needs one barrier per RPW columns, the tridiagonalisation two per column, the
// substitutions and the back transformation none (a warp owns whole columns).
// In a cluster the rows are dealt to the CTAs' warps in order; a CTA has its own copy of L, the
// reflectors and the vectors, into which their owner writes (Team::put), and takes the roots, merge
// columns and vectors of its own rows.  The leaves and the sorting are done by every CTA alike.
// Results do not depend on the number of CTAs or warps (the sums over lanes have one shape, fused
// multiply-adds are written out).
// Measured, mean per launch over an evaluation, Jacobi kernel -> here: 24 bands 317 -> 207 us, 70 bands
// 2500 -> 772 us, up to 80 bands in six members 3550 -> 829 us.
#include "kernels.h"

namespace sgo {

namespace {

// Near-dependent directions of the block [X, W] (blk = 2): a W vector whose component orthogonal
// to the basis vectors before it has squared norm at most TD_DROP (its own norm is 1) is left out
// of the subspace instead of failing the Cholesky (the preconditioned residuals of a random start
// are nearly collinear): its column of L and its row of L^-1 are zero, and its diagonal entry of
// C is set above the spectrum, so that it ranks after every kept Ritz value.
constexpr double TD_DROP = 1e-3;
// Lanes per root of a merge of m poles out of n.  A root's own arithmetic is done by all its lanes,
// so more lanes only pay while they shorten a chain of terms that is long against it, and only until
// about four warps keep the FP64 lanes busy.  (Not a function of the block
// size: the sums must not depend on the batch a member is in.)
__device__ __forceinline__ int td_lanes(int m, int n) {
  if (n > 32) return m > 32 ? 4 : m > 8 ? 2 : 1;
  return m > 8 ? 4 : m > 4 ? 2 : 1;
}

using T = double;
template <typename F>
struct TdNum;  // (float: the starting phase of the roots)
template <>
struct TdNum<float> {
  static constexpr float eps = 1.1920929e-7f, ztiny = 1e-7f, floor = 1e-30f, step = 3e-5f;
};
template <>
struct TdNum<double> {
  static constexpr double eps = 2.220446049250313e-16, ztiny = 1e-16, floor = 1e-280, step = 1e-9;
};
// (step: a relative step below which the quadratically convergent root iteration is done, its
// square being below rounding)
constexpr int TD_ITERS = 60;  // cap of the root iteration (typically 4)

// (correctly rounded over the whole range, subnormal numbers among it)
__device__ __forceinline__ float td_rcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double td_rcp(double x) { return __drcp_rn(x); }

__device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// sum over the g lanes of a root
template <typename F>
__device__ __forceinline__ F gsum(F v, int g) {
  for (int o = g >> 1; o > 0; o >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Root in the pole interval of the two-pole model c + s / (p - mu) + S / (q - mu) = 0; right:
// offsets from the right pole (p = -w, q = 0), else from the left one (p = 0, q = w).  S = 0: no
// right pole (the last root; the quadratic would lose the root to its other one at w).
template <typename F>
__device__ __forceinline__ F two_pole_root(F c, F s, F S, F w, bool right) {
  if (S == F(0)) return s * td_rcp(c);
  const F b = right ? fma(-c, w, s + S) : fma(c, w, s) + S;
  const F d = right ? -S * w : s * w;
  const F disc = fma(b, b, -(F(4) * c * d));
  const F r = sqrt(disc > F(0) ? disc : F(0));
  const F num = b >= F(0) ? F(2) * d : b - r, den = b >= F(0) ? b + r : F(2) * c;
  return num * td_rcp(den);
}

// poles relative to the nearest one, in F
template <typename F>
struct Poles {
  const T* d;
  T b;
  __device__ __forceinline__ F operator()(int j) const { return (F)(d[j] - b); }
};

// Iteration for root ii of poles lo .. hi - 1 (weights zw), starting at x in the bracket (a, b)
// of offsets from the nearest pole; lane sub of the root's g lanes takes every g-th term.  Returns
// whether it converged; all lanes of the warp take part until the last root is done.
template <typename F, typename PO>
__device__ __forceinline__ bool secular(const PO& pole, const F* zw, int lo, int hi, int ii, int sub, int g, F w,
                                        bool right, bool last, F a, F b, bool done, int iters, F* xio) {
  const F pl = right ? -w : F(0), ql = right ? F(0) : w;  // the two poles of the interval
  F x = *xio;
  for (int it = 0; it < iters; ++it) {
    if (!__any_sync(0xffffffffu, !done)) break;
    F ps = F(0), dp = F(0), ph = F(0), dq = F(0);  // the sums left and right of the root, their slopes
    if (!done)
      for (int j = lo + sub; j < hi; j += g) {
        const F r = td_rcp(pole(j) - x);
        const F t = zw[j] * r, u = t * r;
        if (j <= ii) {
          ps += t;
          dp += u;
        } else {
          ph += t;
          dq += u;
        }
      }
    for (int o = g >> 1; o > 0; o >>= 1) {
      ps += __shfl_xor_sync(0xffffffffu, ps, o);
      dp += __shfl_xor_sync(0xffffffffu, dp, o);
      ph += __shfl_xor_sync(0xffffffffu, ph, o);
      dq += __shfl_xor_sync(0xffffffffu, dq, o);
    }
    if (!done) {
      const F f = F(1) + ps + ph;
      if (f < F(0)) a = x;
      else b = x;
      if (fabs(f) <= F(2) * TdNum<F>::eps * (F(1) + fabs(ps) + fabs(ph))) {
        done = true;
      } else {
        const F dl = pl - x, dr = ql - x;
        F c = fma(-dl, dp, f);
        if (!last) c = fma(-dr, dq, c);
        F y = two_pole_root(c, dl * dl * dp, last ? F(0) : dr * dr * dq, w, right);
        const bool in = y > a && y < b;
        if (!in) y = a == F(0) ? b * F(0.01) : b == F(0) ? a * F(0.01) : F(0.5) * (a + b);
        if ((in && fabs(y - x) <= TdNum<F>::step * fabs(x)) || !(b - a > TdNum<F>::eps * fmax(fabs(a), fabs(b)))) done = true;
        x = y;
      }
    }
  }
  *xio = x;
  return done;
}

// Largest block the divide and conquer starts from: 2 rows (one rotation), since longer QL iterations
// are chains of FP64 operations (8 rows 100 us, three merge levels instead 40).
constexpr int TD_LEAF = 2;

// Eigenvectors of a symmetric tridiagonal leaf of m0 <= M rows by implicit QL steps with
// Wilkinson's shift (EISPACK's tql2: Bowdler, Martin, Reinsch & Wilkinson, Numer. Math. 11, 293
// (1968)): every lane carries the whole of d and e and one row z of the vectors.
template <int M>
__device__ __forceinline__ void td_leaf(T (&d)[M], T (&e)[M], T (&z)[M], int m0, T norm) {
  const T tiny = T(1e-3) * TdNum<T>::eps * norm;
  for (int l = 0; l + 1 < m0; ++l) {
    for (int it = 0; it < 30; ++it) {
      int m = m0 - 1;  // the first negligible e at or after l ends the active block
      T dl = T(0), dl1 = T(0), el = T(0), dm = T(0);
#pragma unroll
      for (int i = M - 2; i >= 0; --i) {
        const T x = fabs(e[i]);
        if (i >= l && i < m0 - 1 && !(x > TdNum<T>::eps * (fabs(d[i]) + fabs(d[i + 1])) && x > tiny)) m = i;
        if (i == l) {
          dl = d[i];
          dl1 = d[i + 1];
          el = e[i];
        }
      }
      if (m == l) break;
#pragma unroll
      for (int i = 0; i < M; ++i)
        if (i == m) dm = d[i];
      T g = (dl1 - dl) * td_rcp(T(2) * el);
      g = fma(el, td_rcp(g + copysign(sqrt(fma(g, g, T(1))), g)), dm - dl);
      T s = T(1), c = T(1), q = T(0);
      bool cut = false;  // an exact zero ended the sweep early
#pragma unroll
      for (int i = M - 2; i >= 0; --i)
        if (i < m && i >= l && !cut) {
          const T f = s * e[i], b = c * e[i], h = fma(f, f, g * g);
          const T ir = rsqrt(h);
          if (h > TdNum<T>::floor) {
            e[i + 1] = h * ir;
            s = f * ir;
            c = g * ir;
            g = d[i + 1] - q;
            const T r = fma(d[i] - g, s, T(2) * c * b);
            q = s * r;
            d[i + 1] = g + q;
            g = fma(c, r, -b);
            const T zi = z[i + 1];
            z[i + 1] = fma(s, z[i], c * zi);
            z[i] = fma(c, z[i], -(s * zi));
          } else {
            e[i + 1] = T(0);
            d[i + 1] = d[i + 1] - q;
            cut = true;
          }
        }
#pragma unroll
      for (int i = 0; i < M; ++i) {
        if (i == l && !cut) {
          d[i] = d[i] - q;
          e[i] = g;
        }
        if (i == m) e[i] = T(0);
      }
    }
  }
}

// The CTAs of a problem: writes to every CTA's copy of a shared variable, barriers over all of them
// (CL = 1: the CTA's own copy, the matrix warps).
template <int CL>
struct Team {
  unsigned off[CL];  // from a shared address to CTA r's copy of it
  int rank;
  __device__ __forceinline__ void init(void* smem) {
    rank = 0;
    off[0] = 0;
    if constexpr (CL > 1) {
      asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
      const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        unsigned b;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(r));
        off[r] = b - a;
      }
    }
  }
  static __device__ __forceinline__ void st(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
  }
  static __device__ __forceinline__ void st(unsigned a, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
  }
  template <typename X>
  __device__ __forceinline__ void put(X* p, X v) const {  // *p = v in every CTA
    if constexpr (CL == 1) {
      *p = v;
    } else {
      const unsigned a = (unsigned)__cvta_generic_to_shared(p);
#pragma unroll
      for (int r = 0; r < CL; ++r) st(a + off[r], v);
    }
  }
  __device__ __forceinline__ void barrier() const {  // all threads of all CTAs
    if constexpr (CL == 1) {
      __syncthreads();
    } else {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }
  __device__ __forceinline__ void matrix_barrier(int threads) const {  // the matrix warps of all CTAs
    if constexpr (CL == 1) asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
    else barrier();
  }
};

// R consecutive shared values (aligned to 16 bytes) as vector loads
template <int R>
__device__ __forceinline__ void ldv(const T* p, T (&o)[R]) {
  static_assert(R % 2 == 0, "whole vectors");
#pragma unroll
  for (int i = 0; i < R / 2; ++i) {
    const double2 v = reinterpret_cast<const double2*>(p)[i];
    o[2 * i] = v.x; o[2 * i + 1] = v.y;
  }
}

__host__ __device__ inline int td_zs(int n) { return n > 16 ? ((n + 1) / 2) | 1 : 9; }  // row stride of the vectors
__host__ __device__ inline int td_us(int n) { return (n + 3) & ~3; }        // row stride of the merge matrix
constexpr int TD_RED = 64;  // one value for each matrix warp of a cluster
constexpr int TD_PAD = 32;  // vectors are read in whole groups of rows past n
__host__ __device__ inline int td_vn(int n) { return ((n + 3) & ~3) + TD_PAD; }
__host__ __device__ inline size_t td_vec_bytes(int n) {
  return ((size_t)(13 * td_vn(n) + TD_RED) * sizeof(T) + (size_t)(3 * td_vn(n) + 16) * 4 + 15) / 16 * 16;
}

}  // namespace

// all: L, the reflectors, U and Z in shared memory; else L, the reflectors and the transposes go
// through the member's global scratch (3 n^2 elements) and share U's place in turn.
template <int NR, int MW, int NW, int CL>
__global__ void __launch_bounds__(32 * NW, 1)
    k_rr_td(KArgs ka, T* gscratch, size_t gstride, int all, int blk) {
  static_assert(CL == 1 || MW == NW, "in a cluster every warp is a matrix warp");
  constexpr int RPW = 32 * NR / (MW * CL), NT = 32 * NW, MT = 32 * MW;
  static_assert(RPW * MW * CL == 32 * NR && RPW % 2 == 0, "whole vectors of rows");
  static_assert(MW * CL <= TD_RED && NW <= TD_RED, "a value of red for every warp");
  using N = TdNum<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = blockIdx.x / CL;
  if (!ka.active[p]) return;
  const Prob& P = ka.probs[p];
  Team<CL> team;
  team.init(smem_raw);
  const int n = blk * P.nb, ns = n | 1, zs = td_zs(n), us = td_us(n), vn = td_vn(n);
  const double* Sin = blk == 2 ? P.S2 : P.S;
  const double* Hin = blk == 2 ? P.H2 : P.Hs;
  const int tid = threadIdx.x, lane = tid & 31, lwarp = tid >> 5;
  const int warp = team.rank * MW + lwarp;  // (a matrix warp's number)
  // vectors
  T* dk = reinterpret_cast<T*>(smem_raw);  // 1 / L_kk; 0 marks a left-out direction
  T* vbuf = dk + vn;                       // [2][vn] Householder vectors in turn
  T* pv = vbuf + 2 * vn;                   // C v
  T* wv = pv + vn;                         // the rank-two update's w
  T* tau = wv + vn;
  T* dg = tau + vn;                        // diagonal, then the blocks' eigenvalues
  T* eo = dg + vn;                         // off-diagonal
  T* zv = eo + vn;                         // z recomputed from the roots
  T* ds = zv + vn;                         // sorted poles
  T* zw = ds + vn;                         // rho z^2, sorted
  T* zh = zw + vn;                         // z, sorted
  T* mu = zh + vn;                         // root i = ds[kx[i]] + mu[i]
  T* red = mu + vn;                        // [TD_RED]
  T* nd = vbuf;                            // new eigenvalues (the reflectors are done with by then)
  int* perm = reinterpret_cast<int*>(red + TD_RED);
  int* kx = perm + vn;
  int* bk = kx + vn;                       // block of each index: lo | mid << 10 | hi << 20
  float* fz = reinterpret_cast<float*>(wv);  // the weights as floats
  int* flags = bk + vn;                      // [0] Cholesky failed, [1] left-out directions, [2] close poles, [3] capped
  T* Ub = reinterpret_cast<T*>(smem_raw + td_vec_bytes(n));  // [n][us]; L or the reflectors [n][ns]
  T* Zb = Ub + (size_t)n * (ns > us ? ns : us);                        // [n][zs]
  T* Lb = all ? Zb + ((size_t)n * zs + 3) / 4 * 4 : Ub;                // L: row k holds column k
  T* Vb = all ? Lb + (size_t)n * ns : Ub;                              // reflectors, row k
  T* gW = gscratch ? gscratch + (size_t)p * gstride : nullptr;         // transposes
  T* gL = gW + (size_t)n * n;
  T* gV = gL + (size_t)n * n;
  if (tid < 16) flags[tid] = 0;
  team.barrier();

  // row i = i0 + a, column (or, for column-owning steps, row) j = lane + 32 c
  const int i0 = warp * RPW;
  const int c0 = team.rank * MW * RPW, c1 = CL == 1 ? n : min(n, c0 + MW * RPW);  // the CTA's rows
  T A[RPW][NR];
  if (CL > 1 || lwarp < MW) {
    // ---- 1. Cholesky: a warp factors its RPW columns, one barrier, the others update ----
#pragma unroll
    for (int a = 0; a < RPW; ++a)
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        const int i = i0 + a, j = lane + 32 * c;
        A[a][c] = T(0);
        if (i < n && j < n) {
          A[a][c] = Sin[(size_t)i * n + j];
        }
      }
    // (only entries j >= i of the trailing rows are kept up to date)
    for (int pw = 0; pw * RPW < n; ++pw) {
      if (pw == warp) {
#pragma unroll 1
        for (int a = 0; a < RPW && i0 + a < n; ++a) {
          const int k = i0 + a;
          T row[NR], x = T(0);
#pragma unroll
          for (int c = 0; c < NR; ++c) row[c] = A[0][c];
#pragma unroll
          for (int b = 1; b < RPW; ++b)
#pragma unroll
            for (int c = 0; c < NR; ++c)
              if (b == a) row[c] = A[b][c];
#pragma unroll
          for (int c = 0; c < NR; ++c)
            if (c == (k >> 5)) x = row[c];
          x = __shfl_sync(0xffffffffu, x, k & 31);
          const bool drop = blk == 2 && k >= P.nb && x <= TD_DROP;
          const bool bad = !drop && !(x > T(0));  // (S not positive definite; the bands need no norm of 1)
          const T inv = drop ? T(0) : rsqrt(bad ? T(1) : x);
          if (lane == 0) {
            team.put(&dk[k], inv);
            if (bad) team.put(&flags[0], 1);
            if (drop) team.put(&flags[1], 1);
          }
#pragma unroll
          for (int c = 0; c < NR; ++c) {
            const int j = lane + 32 * c;
            row[c] = j > k && j < n ? row[c] * inv : T(0);
            if (j < n) team.put(&Lb[(size_t)k * ns + j], row[c]);
          }
          __syncwarp();
#pragma unroll
          for (int b = 1; b < RPW; ++b)
            if (b > a) {
              const T li = i0 + b < n ? Lb[(size_t)k * ns + i0 + b] : T(0);
#pragma unroll
              for (int c = 0; c < NR; ++c) A[b][c] = fma(-li, row[c], A[b][c]);
            }
        }
      }
      team.matrix_barrier(MT);
      if (warp > pw && i0 < n) {
        for (int k = pw * RPW; k < (pw + 1) * RPW; ++k) {
          T lj[NR];
#pragma unroll
          for (int c = 0; c < NR; ++c) lj[c] = lane + 32 * c < n ? Lb[(size_t)k * ns + lane + 32 * c] : T(0);
#pragma unroll
          for (int a = 0; a < RPW; ++a) {
            const T li = i0 + a < n ? Lb[(size_t)k * ns + i0 + a] : T(0);
#pragma unroll
            for (int c = 0; c < NR; ++c)
              if (32 * c + 31 >= i0) A[a][c] = fma(-li, lj[c], A[a][c]);
          }
        }
      }
    }
    // ---- 2. W = L^-1 Hs, C = W L^-T (a warp owns columns i0 .. i0 + RPW - 1; no barriers) ----
    // forward substitution: x_k = h_k / L_kk, h_r -= L_rk x_k for r > k
    auto forward = [&](T(&X)[RPW][NR]) {
#pragma unroll
      for (int ck = 0; ck < NR; ++ck) {
        const int kn = min(32, n - 32 * ck);
        for (int t = 0; t < kn; ++t) {
          const int k = 32 * ck + t;
          const T inv = dk[k];
          T x[RPW], l[NR];
#pragma unroll
          for (int c = ck; c < NR; ++c) l[c] = lane + 32 * c < n ? Lb[(size_t)k * ns + lane + 32 * c] : T(0);  // zero for r <= k
#pragma unroll
          for (int a = 0; a < RPW; ++a) {
            x[a] = __shfl_sync(0xffffffffu, X[a][ck], t) * inv;
            if (lane == t) X[a][ck] = x[a];
          }
#pragma unroll
          for (int c = ck; c < NR; ++c)
#pragma unroll
            for (int a = 0; a < RPW; ++a) X[a][c] = fma(-l[c], x[a], X[a][c]);
        }
      }
    };
    // (Hs is symmetric to rounding; its rows are taken as columns, and C is symmetrised below)
    if (i0 < n) {
#pragma unroll
      for (int a = 0; a < RPW; ++a)
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          const int i = i0 + a, j = lane + 32 * c;
          A[a][c] = i < n && j < n ? (T)Hin[(size_t)i * n + j] : T(0);
        }
      forward(A);
    }
    // transpose through U's place (or the global scratch, where L occupies it)
    T* const Tb = all ? Ub : gW;
    const int ts = all ? ns : n;
    auto put = [&]() {  // Tb[i][j] = A (in a cluster, for the CTA of row j)
#pragma unroll
      for (int a = 0; a < RPW; ++a)
#pragma unroll
        for (int c = 0; c < NR; ++c)
          if (i0 + a < n && lane + 32 * c < n) {
            T* const q = &Tb[(size_t)(i0 + a) * ts + lane + 32 * c];
            if (CL == 1 || !all) {
              *q = A[a][c];
            } else {
              const int to = (lane + 32 * c) / (MW * RPW);
              unsigned o = 0;
#pragma unroll
              for (int r = 0; r < CL; ++r)
                if (r == to) o = team.off[r];
              Team<CL>::st((unsigned)__cvta_generic_to_shared(q) + o, A[a][c]);
            }
          }
    };
    put();
    team.matrix_barrier(MT);
#pragma unroll
    for (int a = 0; a < RPW; ++a)
#pragma unroll
      for (int c = 0; c < NR; ++c)
        A[a][c] = i0 + a < n && lane + 32 * c < n ? Tb[(size_t)(lane + 32 * c) * ts + i0 + a] : T(0);
    if (i0 < n) forward(A);
    team.matrix_barrier(MT);
    put();
    if (!all)  // L is needed again at the end; its place is U's
      for (int e = team.rank * MT + tid; e < n * n; e += CL * MT) gL[e] = Lb[(size_t)(e / n) * ns + e % n];
    team.matrix_barrier(MT);
    T rs = T(0);  // largest row sum of |C|
#pragma unroll
    for (int a = 0; a < RPW; ++a) {
      T s = T(0);
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        if (i0 + a < n && lane + 32 * c < n) A[a][c] = T(0.5) * (A[a][c] + Tb[(size_t)(lane + 32 * c) * ts + i0 + a]);
        s += fabs(A[a][c]);
      }
      if (flags[1]) rs = fmax(rs, wsum(s));
    }
    if (flags[1]) {  // (blk = 2) left-out directions above the spectrum
      if (lane == 0) team.put(&red[warp], rs);
      team.matrix_barrier(MT);
      for (int w = 0; w < MW * CL; ++w) rs = fmax(rs, red[w]);
#pragma unroll
      for (int a = 0; a < RPW; ++a)
#pragma unroll
        for (int c = 0; c < NR; ++c)
          if (i0 + a < n && i0 + a == lane + 32 * c && dk[i0 + a] == T(0)) A[a][c] = T(2) * rs + T(1);
    }
    // ---- 3. tridiagonalisation: reflector k from row k (warp k / RPW), v_{k+1} = 1 ----
    for (int k = 0; k + 2 < n; ++k) {
      T* v = vbuf + (k & 1) * vn;
      if (k / RPW == warp) {
        T x[NR], x1 = T(0), dd = T(0);
#pragma unroll
        for (int c = 0; c < NR; ++c) x[c] = T(0);
#pragma unroll
        for (int a = 0; a < RPW; ++a)
          if (i0 + a == k)
#pragma unroll
            for (int c = 0; c < NR; ++c) x[c] = A[a][c];
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          if (c == (k >> 5)) dd = x[c];
          if (c == ((k + 1) >> 5)) x1 = x[c];
        }
        x1 = __shfl_sync(0xffffffffu, x1, (k + 1) & 31);
        T sg = T(0);
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          if (lane + 32 * c <= k + 1) x[c] = T(0);
          sg = fma(x[c], x[c], sg);
        }
        sg = wsum(sg);
        T beta = x1, f = T(0), tk = T(0);
        if (sg > T(0)) {
          const T s2 = fma(x1, x1, sg), r = rsqrt(s2), m = s2 * r;  // |x| = m
          beta = x1 > T(0) ? -m : m;
          f = td_rcp(x1 - beta);
          tk = fma(fabs(x1), r, T(1));
        }
        if (lane == (k & 31)) team.put(&dg[k], dd);
        if (lane == 0) {
          team.put(&eo[k], beta);
          team.put(&tau[k], tk);
        }
        T* vd = all ? Vb + (size_t)k * ns : gV + (size_t)k * n;
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          const int j = lane + 32 * c;
          const T vj = j == k + 1 ? T(1) : x[c] * f;
          if (j < n) {
            team.put(&v[j], vj);
            if (all) team.put(&vd[j], vj);
            else vd[j] = vj;
          }
        }
      }
      team.matrix_barrier(MT);
      const T tk = tau[k];
      if (tk == T(0)) continue;  // (uniform) nothing to eliminate
      const bool busy = i0 + RPW - 1 > k && i0 < n;
      T vj[NR];
#pragma unroll
      for (int c = 0; c < NR; ++c) vj[c] = lane + 32 * c < n ? v[lane + 32 * c] : T(0);
      if (busy) {
        T q[RPW];
#pragma unroll
        for (int a = 0; a < RPW; ++a) q[a] = T(0);
#pragma unroll
        for (int c = 0; c < NR; ++c)
          if (32 * c + 31 > k)
#pragma unroll
            for (int a = 0; a < RPW; ++a) q[a] = fma(A[a][c], vj[c], q[a]);
        const T s = fold_sums<T, RPW, 32>(q, lane);
        constexpr int S = fold_shift<RPW, 32>();
        const int a = lane >> S;
        if ((lane & ((1 << S) - 1)) == 0 && a < RPW && i0 + a < n) team.put(&pv[i0 + a], s);
      }
      team.matrix_barrier(MT);
      if (busy) {
        T pj[NR], kk = T(0);
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          const int j = lane + 32 * c;
          pj[c] = j > k && j < n ? pv[j] : T(0);
          kk = fma(pj[c], vj[c], kk);
        }
        kk = T(0.5) * tk * wsum(kk);
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          pj[c] = tk * fma(-kk, vj[c], pj[c]);  // w_j
          const int j = lane + 32 * c;
          if (j >= i0 && j < i0 + RPW && j < n) wv[j] = pj[c];
        }
        __syncwarp();
        T vi[RPW], wi[RPW];
        ldv(v + i0, vi);
        ldv(wv + i0, wi);
#pragma unroll
        for (int c = 0; c < NR; ++c)
          if (32 * c + 31 > k)
#pragma unroll
            for (int a = 0; a < RPW; ++a)
              if (i0 + a < n) A[a][c] = fma(-vi[a], pj[c], fma(-wi[a], vj[c], A[a][c]));
      }
    }
#pragma unroll
    for (int a = 0; a < RPW; ++a)
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        const int i = i0 + a, j = lane + 32 * c;
        if (i < n && i + 2 >= n && j < n) {
          if (i == j) team.put(&dg[i], A[a][c]);
          if (i == n - 2 && j == n - 1) team.put(&eo[i], A[a][c]);
        }
      }
  }
  team.barrier();
  // ---- 4. divide and conquer (in a cluster, the leaves, sorting and poles in every CTA alike; a CTA
  // takes the roots, weights and vectors of its own rows) ----
  // blocks: at shift sh, block q holds the indices (q n) >> sh .. ((q + 1) n) >> sh.  The leaves are
  // the blocks of at most TD_LEAF rows, torn apart at their ends (d -= |e| on either side of a
  // tear).
  {
    T nm = T(0);
    for (int i = tid; i < n; i += NT) {
      nm = fmax(nm, fabs(dg[i]) + (i > 0 ? fabs(eo[i - 1]) : T(0)) + (i + 1 < n ? fabs(eo[i]) : T(0)));
      perm[i] = i;  // (stays a valid index where the input is not finite)
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nm = fmax(nm, __shfl_xor_sync(0xffffffffu, nm, o));
    if (lane == 0) red[lwarp] = nm;
  }
  __syncthreads();
  T norm = T(0);
  for (int w = 0; w < NW; ++w) norm = fmax(norm, red[w]);
  int lev = 0;  // merge levels
  while (((n + (1 << lev) - 1) >> lev) > TD_LEAF) ++lev;
  const T gap = N::eps * norm;
  for (int t = tid; t < (TD_LEAF << lev); t += NT) {  // TD_LEAF lanes per leaf
    const int q = t / TD_LEAF, r = t % TD_LEAF;
    const int lo = (q * n) >> lev, hi = ((q + 1) * n) >> lev, m0 = hi - lo;
    T d[TD_LEAF], e[TD_LEAF], z[TD_LEAF];
#pragma unroll
    for (int i = 0; i < TD_LEAF; ++i) {
      d[i] = i < m0 ? dg[lo + i] : T(0);
      e[i] = i + 1 < m0 ? eo[lo + i] : T(0);
      if (i == 0 && lo > 0) d[i] -= fabs(eo[lo - 1]);
      if (i == m0 - 1 && hi < n) d[i] -= fabs(eo[hi - 1]);
      z[i] = i == r ? T(1) : T(0);
    }
    td_leaf(d, e, z, m0, norm);
    // ascending: vector i goes to row lo + rank of the leaf's part of Z
#pragma unroll
    for (int i = 0; i < TD_LEAF; ++i) {
      int rk = 0;
#pragma unroll
      for (int k = 0; k < TD_LEAF; ++k) rk += k < m0 && (d[k] < d[i] || (d[k] == d[i] && k < i));
      if (i < m0) {
        if (r < m0) Zb[(size_t)(lo + rk) * zs + r] = z[i];
        if (r == 0) nd[lo + rk] = d[i];
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < n; i += NT) dg[i] = nd[i];
  // the merged vectors: A[a][c] = component lane + 32 c of vector i0 + a
  if (CL > 1 || lwarp < MW)
#pragma unroll
    for (int a = 0; a < RPW; ++a)
#pragma unroll
      for (int c = 0; c < NR; ++c)  // (kept where one leaf is the whole matrix)
        A[a][c] = lev == 0 && i0 + a < n && lane + 32 * c < n ? Zb[(size_t)(i0 + a) * zs + lane + 32 * c] : T(0);
  for (int l = 0; l < lev; ++l) {
    const int sh = lev - l - 1;
    const int g = td_lanes((n + (1 << sh) - 1) >> sh, n);  // lanes per root
    const int sub = tid & (g - 1), GR = NT / g, root0 = tid / g;
    const int slots = (c1 - c0 + GR - 1) / GR;
    team.barrier();
    // sort the poles of the two halves together
    for (int i = tid; i < n; i += NT) {
      const int q = (((i + 1) << sh) - 1) / n;  // the block of index i at this level
      const int lo = (q * n) >> sh, hi = ((q + 1) * n) >> sh, mid = ((2 * q + 1) * n) >> (sh + 1);
      bk[i] = lo | mid << 10 | hi << 20;
      const T d = dg[i];
      int b0 = i < mid ? mid : lo, b1 = i < mid ? hi : mid;
      const int s0 = b0;
      while (b0 < b1) {
        const int h = (b0 + b1) >> 1;
        if (i < mid ? dg[h] < d : dg[h] <= d) b0 = h + 1;
        else b1 = h;
      }
      const int pos = (i < mid ? i : lo + i - mid) + (b0 - s0);
      T z = T(1), rho = T(0);
      if (mid > lo && mid < hi) {
        z = i < mid ? Zb[(size_t)i * zs + mid - 1 - lo] : Zb[(size_t)i * zs];
        const T e = eo[mid - 1];
        if (i >= mid && e < T(0)) z = -z;
        rho = fabs(e);
      }
      if (fabs(z) < N::ztiny) z = z < T(0) ? -N::ztiny : N::ztiny;
      ds[pos] = d;
      zh[pos] = z;
      zw[pos] = z * z * rho;
      perm[pos] = i;
    }
    if (tid == 0) flags[2] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += NT)
      if (i > (bk[i] & 1023) && !(ds[i] - ds[i - 1] >= gap)) flags[2] = 1;
    if constexpr (CL == 1) {
      for (int e = tid; e < n * us / 2; e += NT) reinterpret_cast<double2*>(Ub)[e] = make_double2(0.0, 0.0);
    } else {  // the CTA's own columns
      constexpr int CW = MW * RPW / 2;
      for (int e = tid; e < n * CW; e += NT) {
        const int j = c0 + e % CW * 2;
        if (j < us) *reinterpret_cast<double2*>(&Ub[(size_t)(e / CW) * us + j]) = make_double2(0.0, 0.0);
      }
    }
    __syncthreads();
    if (flags[2]) {  // (few or none) poles closer than rounding: one thread per block moves them apart
      for (int i = tid; i < n; i += NT) {
        const int lo = bk[i] & 1023, hi = bk[i] >> 20;
        if (i == lo)
          for (int j = lo + 1; j < hi; ++j)
            if (!(ds[j] - ds[j - 1] >= gap)) {
              // (the step may round to less than gap where |ds| is large: take the next step up)
              const T up = ds[j - 1] + gap;
              ds[j] = up > ds[j - 1] ? up : ds[j - 1] + T(2) * gap;
            }
      }
      __syncthreads();
    }
    for (int i = tid; i < n; i += NT) fz[i] = (float)zw[i];
    __syncthreads();
    // roots
    for (int sl = 0; sl < slots; ++sl) {
      const int i = c0 + sl * GR + root0;
      const bool live = i < c1;
      const int b3 = bk[live ? i : n - 1], lo = b3 & 1023, mid = (b3 >> 10) & 1023, hi = b3 >> 20;
      const T rho = mid > lo && mid < hi ? fabs(eo[mid - 1]) : T(0);
      const bool solve = live && rho > T(0.01) * gap;
      const int ii = live ? i : lo;
      const bool last = ii == hi - 1;
      const int nx = last ? ii : ii + 1;
      using F = float;
      T tot = T(0);
      for (int j = lo + sub; j < hi; j += g) tot += zw[j];
      tot = gsum(tot, g);
      const T w = last ? tot : ds[nx] - ds[ii];
      // the sign at the middle tells the nearer pole; the root of the two-pole model there starts
      // the iteration.  Both in floats, then two or three FP64 steps.
      const F wf = (F)w, hf = 0.5f * wf;
      const F* zf = fz;
      auto fpole = [&](int K) { return Poles<F>{ds, ds[K]}; };
      F fm = 0.f;
      if (solve) {
        const auto po = fpole(ii);
        for (int j = lo + sub; j < hi; j += g) fm = fma(zf[j], td_rcp(po(j) - hf), fm);
      }
      fm = gsum(fm, g) + 1.f;
      const bool right = !last && fm < 0.f;
      const int K = right ? ii + 1 : ii;
      F xf = two_pole_root(fma(2.f * (zf[ii] - (last ? 0.f : zf[nx])), td_rcp(wf), fm), zf[ii], last ? 0.f : zf[nx], wf, right);
      const F af = right ? -wf : 0.f, bf = right ? 0.f : wf;
      if (!(xf > af && xf < bf)) xf = right ? -0.5f * hf : 0.5f * hf;
      secular(fpole(K), zf, lo, hi, ii, sub, g, wf, right, last, af, bf, !solve, 12, &xf);
      T x = (T)xf;
      const T a = right ? -w : T(0), b = right ? T(0) : w;
      if (!(x > a && x < b)) x = right ? -0.25 * w : 0.25 * w;
      const bool done = secular(Poles<T>{ds, ds[K]}, zw, lo, hi, ii, sub, g, w, right, last, a, b, !solve, TD_ITERS, &x);
      if (live && sub == 0) {
        team.put(&kx[i], solve ? K : -1);  // -1: the halves stay as they are
        team.put(&mu[i], solve ? x : T(0));
        team.put(&nd[i], solve ? ds[K] + x : ds[i]);
        if (solve && !done) team.put(&flags[3], 1);
      }
    }
    team.barrier();
    // z from the roots: z_j^2 ~ (lam_last - ds_j) prod_{i<j} (lam_i - ds_j) / (ds_i - ds_j)
    //                          prod_{j<=i<last} (lam_i - ds_j) / (ds_{i+1} - ds_j), every factor positive
    for (int sl = 0; sl < slots; ++sl) {
      const int j = c0 + sl * GR + root0;
      const bool live = j < c1 && kx[j < c1 ? j : 0] >= 0;
      T pr = T(1);
      if (live) {
        const int lo = bk[j] & 1023, hi = bk[j] >> 20;
        const T dj = ds[j];
        for (int i = lo + sub; i < hi; i += g) {
          const T num = (ds[kx[i]] - dj) + mu[i];
          pr *= i == hi - 1 ? num : num * td_rcp(ds[i < j ? i : i + 1] - dj);
        }
      }
      for (int o = g >> 1; o > 0; o >>= 1) pr *= __shfl_xor_sync(0xffffffffu, pr, o);
      if (live && sub == 0) {
        const T q = sqrt(fmax(fabs(pr), N::floor));
        team.put(&zv[j], zh[j] < T(0) ? -q : q);
      }
    }
    team.barrier();
    // U[original index of pole j - lo][i] = z_j / (ds_j - lam_i), normalised
    for (int sl = 0; sl < slots; ++sl) {
      const int i = c0 + sl * GR + root0;
      const bool live = i < c1;
      const int b3 = bk[live ? i : n - 1], lo = b3 & 1023, hi = b3 >> 20;
      const int K = live ? kx[i] : -1;
      T s = T(0);
      if (K >= 0) {
        const T base = ds[K], m = mu[i];
        for (int j = lo + sub; j < hi; j += g) {
          const T v = zv[j] * td_rcp((ds[j] - base) - m);
          Ub[(size_t)perm[j] * us + i] = v;
          s = fma(v, v, s);
        }
      }
      s = gsum(s, g);
      if (K >= 0) {
        const T f = rsqrt(s);
        for (int j = lo + sub; j < hi; j += g) Ub[(size_t)perm[j] * us + i] *= f;
      } else if (live && sub == 0) {
        Ub[(size_t)perm[i] * us + i] = T(1);
      }
    }
    __syncthreads();
    // vectors: component r of vector i = sum over the poles j of r's half, U[j][i] Z[j][r]
    if ((CL > 1 || lwarp < MW) && i0 < n) {
#pragma unroll
      for (int a = 0; a < RPW; ++a)
#pragma unroll
        for (int c = 0; c < NR; ++c) A[a][c] = T(0);
      const int jlo = bk[i0] & 1023, jhi = bk[min(i0 + RPW, n) - 1] >> 20;
      for (int jh = jlo; jh < jhi;) {  // half blocks: poles j0 .. j1 - 1, whose vectors span rows j0 .. j1 - 1
        const int b3 = bk[jh], mid = (b3 >> 10) & 1023;
        const int j0 = jh, j1 = jh < mid ? mid : b3 >> 20;
        const T* z[NR];
        bool on[NR];
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          const int r = lane + 32 * c;
          on[c] = r >= j0 && r < j1;
          z[c] = Zb + (size_t)j0 * zs + (on[c] ? r - j0 : 0);
        }
#pragma unroll 4
        for (int j = j0; j < j1; ++j) {
          T u[RPW];
          ldv(Ub + (size_t)j * us + i0, u);
#pragma unroll
          for (int c = 0; c < NR; ++c)
            if (32 * c < j1 && 32 * c + 31 >= j0) {
              const T zr = on[c] ? z[c][(j - j0) * zs] : T(0);
#pragma unroll
              for (int a = 0; a < RPW; ++a) A[a][c] = fma(u[a], zr, A[a][c]);
            }
        }
        jh = j1;
      }
    }
    team.barrier();
    for (int i = tid; i < n; i += NT) dg[i] = nd[i];
    if (sh > 0 && (CL > 1 || lwarp < MW)) {
#pragma unroll
      for (int a = 0; a < RPW; ++a) {
        const int b3 = bk[min(i0 + a, n - 1)], lo = b3 & 1023, hi = b3 >> 20;
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          const int r = lane + 32 * c;
          if (i0 + a < n && r >= lo && r < hi) team.put(&Zb[(size_t)(i0 + a) * zs + r - lo], A[a][c]);
        }
      }
    }
  }
  team.barrier();
  // ---- 5. reflectors from the last to the first, then back substitution with L^T ----
  if (CL == 1 && lwarp >= MW) return;  // (the matrix warps go on alone)
  if (!all) {
    for (int e = tid; e < (n - 2) * n; e += MT) Ub[(size_t)(e / n) * ns + e % n] = gV[e];
    team.matrix_barrier(MT);
  }
  if (i0 < n)
    for (int k = n - 3; k >= 0; --k) {
      const T tk = tau[k];
      if (tk == T(0)) continue;
      T v[NR], q[RPW];
#pragma unroll
      for (int a = 0; a < RPW; ++a) q[a] = T(0);
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        v[c] = T(0);
        if (32 * c + 31 > k) {
          if (lane + 32 * c < n) v[c] = Vb[(size_t)k * ns + lane + 32 * c];
#pragma unroll
          for (int a = 0; a < RPW; ++a) q[a] = fma(v[c], A[a][c], q[a]);
        }
      }
      const T s = fold_sums<T, RPW, 32>(q, lane) * tk;
#pragma unroll
      for (int a = 0; a < RPW; ++a) q[a] = __shfl_sync(0xffffffffu, s, a << fold_shift<RPW, 32>());
#pragma unroll
      for (int c = 0; c < NR; ++c)
        if (32 * c + 31 > k)
#pragma unroll
          for (int a = 0; a < RPW; ++a) A[a][c] = fma(-q[a], v[c], A[a][c]);
    }
  if (!all) {
    team.matrix_barrier(MT);
    for (int e = tid; e < n * n; e += MT) Ub[(size_t)(e / n) * ns + e % n] = gL[e];
    team.matrix_barrier(MT);
  }
  if (i0 < n) {
#pragma unroll
    for (int ci = 0; ci < NR; ++ci) {
      constexpr int top = NR - 1;
      const int ck = top - ci;
      const int kn = min(32, n - 32 * ck);
      for (int t = kn - 1; t >= 0; --t) {
        const int k = 32 * ck + t;
        const T inv = dk[k];
        T x[RPW], lr[NR];
#pragma unroll
        for (int c = 0; c < NR; ++c)
          if (c <= ck) lr[c] = lane + 32 * c < k ? Lb[(size_t)(lane + 32 * c) * ns + k] : T(0);  // L_kr
#pragma unroll
        for (int a = 0; a < RPW; ++a) {
          x[a] = __shfl_sync(0xffffffffu, A[a][ck], t) * inv;
          if (lane == t) A[a][ck] = x[a];
        }
#pragma unroll
        for (int c = 0; c < NR; ++c)
          if (c <= ck)
#pragma unroll
            for (int a = 0; a < RPW; ++a) A[a][c] = fma(-lr[c], x[a], A[a][c]);
      }
    }
    // the lowest n_b Ritz pairs: rows r < n_b are the coefficients on X, the others those on W
#pragma unroll
    for (int a = 0; a < RPW; ++a) {
      const int i = i0 + a;
      if (i >= n || i >= P.nb) continue;
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        const int r = lane + 32 * c;
        if (r >= n) continue;
        if (r < P.nb) P.Tm[(size_t)r * P.nb + i] = A[a][c];
        else P.Cm[(size_t)(r - P.nb) * P.nb + i] = A[a][c];
      }
      if (lane == 0) P.eps[i] = dg[i];
    }
  }
  if (warp == 0 && lane == 0) {
    if (flags[3]) P.scal[SC_RRCAP] += 1.0;
    if (flags[0]) P.status[0] = 1;
  }
}

namespace {
size_t td_smem(int n, bool all) {
  const size_t ns = n | 1, us = td_us(n), u = (size_t)n * (ns > us ? ns : us), z = ((size_t)n * td_zs(n) + 3) / 4 * 4;
  return td_vec_bytes(n) + (u + z + (all ? 2 * (size_t)n * ns + 32 : 0)) * sizeof(T);  // (32: rows are read on past n)
}
constexpr size_t TD_SMEM_MAX = 227 * 1024;
}  // namespace

// Subspaces the kernel takes: an 8 x 4 tile of the matrix per thread.
int rr_td_max() { return 128; }

// bytes of global scratch per problem (0: everything fits in shared memory)
size_t rr_td_scratch_bytes(int n) { return td_smem(n, true) <= TD_SMEM_MAX ? 0 : 3 * (size_t)n * n * sizeof(T); }

template <int NR, int MW, int NW, int CL>
static void td_launch(const Launch& L, int n, unsigned char* scratch, size_t stride, int blk) {
  const bool all = td_smem(n, true) <= TD_SMEM_MAX;
  const size_t smem = td_smem(n, all);
  auto* fn = k_rr_td<NR, MW, NW, CL>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = L.ka.nprob * CL;
  cfg.blockDim = 32 * NW;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = L.stream;
  cudaLaunchAttribute at[1] = {};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CL > 1 ? 1 : 0;
  cuda_ok(cudaLaunchKernelEx(&cfg, fn, L.ka, reinterpret_cast<T*>(scratch), stride / sizeof(T), all ? 1 : 0, blk),
          "subspace eigensolve launch");
}

// n: the largest subspace of the launch (n_b, or 2 n_b for blk = 2).  CTAs per problem: more of them
// shorten the column-owning steps and share the FP64 lanes' work; each barrier costs 0.4 us more.  So
// a cluster wherever the launch leaves half the SMs to the sub-batches that run beside it.  Measured,
// one problem, 1 / 4 / 8 CTAs: 24 bands 269 / 219 / 191 us, 52 bands 851 / 550 / 472, 70 bands 1825 /
// 925 / 724, 119 bands 5074 / 1953 / 1438.  (In one CTA: 8 to 16 rows in as few warps as the registers
// allow, since every warp's own sums use the FP64 lanes too.)
void launch_rr_td(const Launch& L, int n, unsigned char* scratch, size_t stride, int blk) {
  constexpr int SMS = 152 / 2;
  const int np = L.ka.nprob;
  if (np * 8 <= SMS) {
    if (n <= 32) td_launch<1, 2, 2, 8>(L, n, scratch, stride, blk);
    else if (n <= 64) td_launch<2, 4, 4, 8>(L, n, scratch, stride, blk);
    else if (n <= 96) td_launch<3, 6, 6, 8>(L, n, scratch, stride, blk);
    else td_launch<4, 8, 8, 8>(L, n, scratch, stride, blk);
  } else if (np * 4 <= SMS) {
    if (n <= 32) td_launch<1, 2, 2, 4>(L, n, scratch, stride, blk);
    else if (n <= 64) td_launch<2, 4, 4, 4>(L, n, scratch, stride, blk);
    else if (n <= 96) td_launch<3, 6, 6, 4>(L, n, scratch, stride, blk);
    else td_launch<4, 8, 8, 4>(L, n, scratch, stride, blk);
  } else {
    if (n <= 32) td_launch<1, 4, 8, 1>(L, n, scratch, stride, blk);
    else if (n <= 64) td_launch<2, 8, 8, 1>(L, n, scratch, stride, blk);
    else if (n <= 96) td_launch<3, 8, 8, 1>(L, n, scratch, stride, blk);
    else td_launch<4, 8, 8, 1>(L, n, scratch, stride, blk);
  }
}

// (Every size's limit, once per engine: the limit belongs to the process, so that one set before each
// launch could be lowered by another thread's smaller structure in between.)
template <int NR, int MW, int NW, int CL>
static void td_limit() {
  cudaFuncSetAttribute(k_rr_td<NR, MW, NW, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TD_SMEM_MAX);
}
void rr_td_set_smem_limits() {
  td_limit<1, 2, 2, 8>(), td_limit<2, 4, 4, 8>(), td_limit<3, 6, 6, 8>(), td_limit<4, 8, 8, 8>();
  td_limit<1, 2, 2, 4>(), td_limit<2, 4, 4, 4>(), td_limit<3, 6, 6, 4>(), td_limit<4, 8, 8, 4>();
  td_limit<1, 4, 8, 1>(), td_limit<2, 8, 8, 1>(), td_limit<3, 8, 8, 1>(), td_limit<4, 8, 8, 1>();
}

}  // namespace sgo
