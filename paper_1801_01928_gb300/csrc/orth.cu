// FP64 Householder orthogonalisation of TT-cores (the left- and right-orthogonal forms that
// the tangent-space operations of the paper's Section 3.2 are built on).
//
// Three sweeps over an FP64 working copy of the cores: right-to-left on X (LQ steps: QR of
// the transposed r_{k-1} x (n_k r_k) unfolding, R^T pushed into core k-1), left-to-right on
// the result (QR of the (r_{k-1} n_k) x r_k unfolding, R pushed into core k+1) giving U, and
// right-to-left on U giving V. Every QR normalises diag(R) >= 0, which makes the factors of a
// full-rank unfolding unique.
//
// GB300 runs FP64 at a small fraction of its FP32 rate, so one QR is spread over a cluster
// of P CTAs (P = 16 when the device allows it, else 8): the m rows of the unfolding W are
// split into P contiguous blocks held in shared memory. Column j's Householder reflector
// (LAPACK dlarfg convention, Golub & Van Loan Algorithm 5.1.1) needs the norm of x = W[j:, j]
// and the products v . W[:, l] with the trailing columns; both follow from one set of
// partial sums per CTA (x.x and x.W[:, l] below the diagonal, plus row j), exchanged through
// distributed shared memory behind a single cluster barrier per column (the publish slots
// alternate between two buffers). R is then broadcast to every CTA and Q = W R^{-1} is
// recovered row by row by a triangular solve that needs no further communication.
//
// Tall unfoldings of 4 to 32 columns first try a factorisation with two exchanges instead of
// one per column (cqr_step): a Cholesky factor R1 of the Gram matrix taken in FP32 preconditions
// W, Q1 = W R1^{-1} in FP64 is orthonormal to some 1e-6, and one FP64 Gram matrix of Q1 corrects
// both factors to FP64 accuracy. The departure of Q1 from orthonormality is measured; where it
// is not small (ill-conditioned or nearly square unfoldings) the Householder columns run. X of
// config 5 (d = 20, n = 16, r = 32, 57 factorisations): 6.80 ms with Householder columns alone (3.3
// us each: one cluster barrier, four block barriers and the FP64 chain of the reflector), 2.53 ms
// now, 40 us a factorisation, of which the 2.3 thousand FP64 warp instructions of a CTA's 32 rows
// at some 16 clocks each are 18 us. The left-to-right and the last sweep factor unfoldings that carry the
// singular values of X; with sigma_1 / sigma_r = 100, 300 and 1000 or more at every interface the same size
// takes 3.07, 3.37 and 4.45 ms (the refused steps pay for both ways), with Householder columns alone 6.90.
//
// The working cores keep their original row strides so every in-place update touches only the
// rows or columns its CTA owns.
#include <cooperative_groups.h>
#include <math.h>

#include "t3f_internal.cuh"

namespace cg = cooperative_groups;

namespace t3f {

constexpr int kOrthThreads = 256;
constexpr int kOrthMaxRows = 4096;

struct OrthArgs {
  TTV X, U, V;
  int P;                      // CTAs per cluster
  int rows_per;               // max rows of W per CTA (ceil(kOrthMaxRows / P) bound)
  double* work;               // per object: padded working cores
  long long obj_stride;       // doubles per object
  long long coff[T3F_MAX_D];  // offset of working core k
  int R1[T3F_MAX_D];          // padded row stride of core k (= original r_{k+1})
};

struct Dims {
  int r0, n, r1;
};

struct OrthSmem {
  double* W;      // rows_per x c working block (row-major, ld = c)
  double* Rs;     // T3F_MAX_RANK x T3F_MAX_RANK
  double* pub;    // [2][T3F_MAX_RANK] published partial dots (index j holds the squared norm)
  double* rowj;   // [2][T3F_MAX_RANK] published row j (owner only)
  double* gsum;   // T3F_MAX_RANK gathered dots
  double* wj;     // T3F_MAX_RANK row j of W
  double* rinv;   // T3F_MAX_RANK reciprocals of diag(R)
  double* tv;     // rows_per: tau * v_r of the owned rows
  double* refl;   // 4: beta, tau, scale of the current reflector
};

// Address of element (row q, col l) of W inside the padded working core.
//   lr = 1: W = left unfolding, row q = a * n + i, col l = b   -> (a n + i) R1 + l
//   lr = 0: W = transposed right unfolding, row q = i * r1 + b, col l = a
__device__ __forceinline__ long long w_addr(int lr, int q, int l, const Dims& dm, int R1) {
  if (lr) return (long long)q * R1 + l;
  const int i = q / dm.r1, b = q % dm.r1;
  return ((long long)l * dm.n + i) * R1 + b;
}

// Entry e of a packed upper triangle, column by column: row p <= column q.
__device__ __forceinline__ void tri_pq(int e, int* p, int* q) {
  int c = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while (c * (c + 1) / 2 > e) --c;
  while ((c + 1) * (c + 2) / 2 <= e) ++c;
  *q = c;
  *p = e - c * (c + 1) / 2;
}

// The same triangle of order c row by row (p = c - 1 first), and by diagonals q - p (longest first):
// the lanes of a warp then run sums of nearly equal length.
__device__ __forceinline__ void tri_row(int e, int c, int* p, int* q) {
  int a, b;
  tri_pq(e, &a, &b);
  *p = c - 1 - b;
  *q = *p + a;
}
__device__ __forceinline__ void tri_diag(int e, int c, int* p, int* q) {
  int a, b;
  tri_pq(e, &a, &b);
  *p = a;
  *q = a + c - 1 - b;
}

constexpr int kCqrMax = 32;            // columns
constexpr int kCqrLd = kCqrMax + 1;
constexpr int kCqrTri = kCqrMax * (kCqrMax + 1) / 2;
constexpr int kCqrPer = (kCqrTri + kOrthThreads - 1) / kOrthThreads;  // triangle entries per thread

// U <- phi(E - U^T U), `its` times from U = phi(E) (phi: strict upper part plus half the
// diagonal), so that (I + U)^T (I + U) = I + E up to |E|^(its + 2); then C <- U - U C from C = U,
// so that (I + U)(I - C) = I to the same order. The second-order products run in T on Ub / Cb, the
// leading terms in FP64 (e: this thread's entries of E, by rows; results in Um and Cm).
template <typename T>
__device__ void cqr_series(const double* e, int c, int its, T* Ub, T* Cb, double* Um, double* Cm) {
  const int tid = threadIdx.x, nt = c * (c + 1) / 2;
  int p[kCqrPer], q[kCqrPer];
#pragma unroll
  for (int x = 0; x < kCqrPer; ++x) {
    const int en = tid + x * kOrthThreads;
    p[x] = 0;
    q[x] = -1;
    if (en < nt) {
      tri_row(en, c, &p[x], &q[x]);
      Ub[p[x] * kCqrLd + q[x]] = (T)(p[x] == q[x] ? 0.5 * e[x] : e[x]);
    }
  }
  __syncthreads();
  for (int it = 0; it < its; ++it) {
    T t[kCqrPer];
#pragma unroll
    for (int x = 0; x < kCqrPer; ++x) {
      t[x] = (T)0;
      if (q[x] >= 0)
#pragma unroll 8
        for (int r = 0; r <= p[x]; ++r) t[x] += Ub[r * kCqrLd + p[x]] * Ub[r * kCqrLd + q[x]];
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < kCqrPer; ++x)
      if (q[x] >= 0) {
        const double v = e[x] - (double)t[x], u = p[x] == q[x] ? 0.5 * v : v;
        Ub[p[x] * kCqrLd + q[x]] = (T)u;
        if (it == its - 1) {
          Um[p[x] * kCqrLd + q[x]] = u;
          Cb[p[x] * kCqrLd + q[x]] = (T)u;
        }
      }
    __syncthreads();
  }
#pragma unroll
  for (int x = 0; x < kCqrPer; ++x)
    if (q[x] >= 0) tri_diag(tid + x * kOrthThreads, c, &p[x], &q[x]);
  for (int it = 0; it < its; ++it) {
    T t[kCqrPer];
#pragma unroll
    for (int x = 0; x < kCqrPer; ++x) {
      t[x] = (T)0;
      if (q[x] >= 0)
#pragma unroll 8
        for (int r = p[x]; r <= q[x]; ++r) t[x] += Ub[p[x] * kCqrLd + r] * Cb[r * kCqrLd + q[x]];
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < kCqrPer; ++x)
      if (q[x] >= 0) {
        const double u = Um[p[x] * kCqrLd + q[x]] - (double)t[x];
        Cb[p[x] * kCqrLd + q[x]] = (T)u;
        if (it == its - 1) Cm[p[x] * kCqrLd + q[x]] = u;
      }
    __syncthreads();
  }
}

// Rows x (8 lanes a row, lane g keeps the columns l = g mod 8 in registers) <- x U^{-1}, U unit upper
// triangular with row stride T3F_MAX_RANK, then column l times scale[l].
__device__ __forceinline__ void unit_solve_rows(double* W, int nrow, int c, const double* U, const double* scale) {
  const int tid = threadIdx.x, g = tid % 8, uend = (c + 7) / 8;
  for (int q0 = 0; q0 < nrow; q0 += kOrthThreads / 8) {
    const int q = q0 + tid / 8;
    const bool qv = q < nrow;
    double* qr = W + (qv ? q : 0) * c;
    double x[kCqrMax / 8];
#pragma unroll
    for (int u = 0; u < kCqrMax / 8; ++u) {
      const int l = g + 8 * u;
      x[u] = (qv && l < c) ? qr[l] : 0.0;
    }
#pragma unroll
    for (int UB = 0; UB < kCqrMax / 8; ++UB) {
      if (UB >= uend) break;
      for (int ob = 0; ob < 8; ++ob) {
        const int b = 8 * UB + ob;
        if (b >= c) break;
        const double xb = __shfl_sync(0xffffffffu, x[UB], ob, 8);
        const double* rb = U + b * T3F_MAX_RANK;
#pragma unroll
        for (int u = UB; u < kCqrMax / 8; ++u) {
          const int l = g + 8 * u;
          if (u < uend && l > b && l < c) x[u] = fma(-xb, rb[l], x[u]);
        }
      }
    }
    if (qv)
#pragma unroll
      for (int u = 0; u < kCqrMax / 8; ++u) {
        const int l = g + 8 * u;
        if (l < c) qr[l] = x[u] * scale[l];
      }
  }
}

// QR of the cluster's m x c unfolding (c <= 32, m >= c), this CTA's rows in s.W (row-major, ld c):
// on success s.W holds the rows of Q, s.Rs the factor R (diag(R) > 0), and true is returned in every
// CTA; false (in every CTA: they decide on the same sums) where W is too ill-conditioned for it,
// with s.W overwritten.
//   G = W^T W and G = U1^T D^2 U1 in FP32, R1 = D U1 (exact in FP64);  Q1 = W R1^{-1} in FP64;
//   E = Q1^T Q1 - I in FP64;  (I + U)^T (I + U) = I + E;  Q = Q1 (I + U)^{-1}, R = (I + U) R1.
// With |E| <= 3e-5 the terms of second order and up are below 1e-9 and FP32 holds them to 1e-16;
// up to 1e-2 they run in FP64; the series is cut where |E|^(its + 2) < 1e-17.
__device__ bool cqr_step(const OrthArgs& a, const OrthSmem& s, int nrow, int c, cg::cluster_group& cluster) {
  const int P = a.P, tid = threadIdx.x, lane = tid & 31, nt = c * (c + 1) / 2;
  // the second half of the W region is free (c <= 32 of T3F_MAX_RANK = 64 columns)
  float* Wf = reinterpret_cast<float*>(s.W + (size_t)a.rows_per * kCqrMax);  // rows x c
  float* pubf = Wf + (size_t)a.rows_per * kCqrMax;                           // triangle
  double* pubd = reinterpret_cast<double*>(pubf + kCqrTri + (kCqrTri & 1));  // triangle
  double* sumd = pubd + kCqrTri;                                             // a P-th of it, summed
  double* Um = sumd + (kCqrTri + 7) / 8;
  double* Cm = Um + kCqrMax * kCqrLd;
  float* Uf = reinterpret_cast<float*>(Cm + kCqrMax * kCqrLd);
  float* Cf = Uf + kCqrMax * kCqrLd;
  __shared__ float red[kOrthThreads / 32];
  __shared__ int bad;
  for (int e = tid; e < nrow * c; e += kOrthThreads) Wf[e] = (float)s.W[e];
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int e = tid; e < nt; e += kOrthThreads) {
    int p, q;
    tri_pq(e, &p, &q);
    float v = 0.0f, w = 0.0f;  // two chains: half the accumulated rounding and latency
    int r = 0;
    for (; r + 1 < nrow; r += 2) {
      v = fmaf(Wf[r * c + p], Wf[r * c + q], v);
      w = fmaf(Wf[(r + 1) * c + p], Wf[(r + 1) * c + q], w);
    }
    if (r < nrow) v = fmaf(Wf[r * c + p], Wf[r * c + q], v);
    pubf[e] = v + w;
  }
  cluster.sync();
  for (int e = tid; e < nt; e += kOrthThreads) {
    int p, q;
    tri_pq(e, &p, &q);
    float v[16], t = 0.0f;
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = r < P ? cluster.map_shared_rank(pubf, r)[e] : 0.0f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)  // pairwise: the least rounding
#pragma unroll
      for (int r = 0; r < o; ++r) v[r] += v[r + o];
    t = v[0];
    Uf[p * kCqrLd + q] = t;
    Uf[q * kCqrLd + p] = t;
  }
  __syncthreads();
  // G = U1^T D^2 U1: warp 0, lane = column
  if (tid < 32) {
    float g[kCqrMax];
#pragma unroll
    for (int p = 0; p < kCqrMax; ++p) g[p] = p < c && lane < c ? Uf[p * kCqrLd + lane] : 0.0f;
    bool ok = true;
    float dj = 1.0f;  // this lane's pivot
#pragma unroll
    for (int j = 0; j < kCqrMax; ++j)
      if (j < c) {
        const float piv = __shfl_sync(0xffffffffu, g[j], j);
        ok = ok && piv > 0.0f && piv < 3.0e38f;
        const float gj = g[j], u = lane == j ? 1.0f : gj * __fdividef(1.0f, piv);
        if (lane >= j) Uf[j * kCqrLd + lane] = u;
        dj = lane == j ? piv : dj;
#pragma unroll
        for (int p = j + 1; p < kCqrMax; ++p) g[p] = fmaf(-__shfl_sync(0xffffffffu, u, p), gj, g[p]);
      }
    if (lane < c) {
      s.wj[lane] = (double)sqrtf(dj);
      s.rinv[lane] = 1.0 / s.wj[lane];
    }
    if (!ok && lane == 0) bad = 1;
  }
  __syncthreads();
  if (bad) return false;
  for (int e = tid; e < c * c; e += kOrthThreads) {
    const int p = e / c, q = e % c;
    if (q >= p) s.Rs[p * T3F_MAX_RANK + q] = (double)Uf[p * kCqrLd + q];
  }
  __syncthreads();
  unit_solve_rows(s.W, nrow, c, s.Rs, s.rinv);  // Q1 = W U1^{-1} D^{-1}
  __syncthreads();
  for (int e = tid; e < nt; e += kOrthThreads) {  // R1 = D U1 (exact: a product of two FP32 values)
    int p, q;
    tri_pq(e, &p, &q);
    s.Rs[p * T3F_MAX_RANK + q] *= s.wj[p];
  }
  for (int e = tid; e < nt; e += kOrthThreads) {
    int p, q;
    tri_pq(e, &p, &q);
    double v = 0.0;
    for (int r = 0; r < nrow; ++r) v = fma(s.W[r * c + p], s.W[r * c + q], v);
    pubd[e] = v;
  }
  cluster.sync();
  // E: CTA r sums the cluster's entries r npc .. (r + 1) npc - 1, sixteen lanes an entry, and every
  // CTA then gathers the sums (sixteen remote reads and FP64 additions per entry and CTA otherwise)
  const int npc = (nt + P - 1) / P, e0 = (int)cluster.block_rank() * npc, e1 = min(nt, e0 + npc);
  for (int w0 = 0; w0 < 16 * npc; w0 += kOrthThreads) {
    const int e = e0 + (w0 + tid) / 16, r = tid % 16;
    double v = e < e1 && r < P ? cluster.map_shared_rank(pubd, r)[e] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (r == 0 && e < e1) sumd[e - e0] = v;
  }
  cluster.sync();
  double ev[kCqrPer];
  float nrm = 0.0f;
#pragma unroll
  for (int x = 0; x < kCqrPer; ++x) {
    const int en = tid + x * kOrthThreads;
    ev[x] = 0.0;
    if (en >= nt) continue;
    int p, q;
    tri_row(en, c, &p, &q);
    const int e = q * (q + 1) / 2 + p;
    const double v = cluster.map_shared_rank(sumd, e / npc)[e % npc];
    ev[x] = p == q ? v - 1.0 : v;
    const float f = (float)ev[x];
    nrm += (p == q ? 1.0f : 2.0f) * f * f;
  }
  for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
  if (lane == 0) red[tid >> 5] = nrm;
  __syncthreads();
  nrm = 0.0f;
  for (int w = 0; w < kOrthThreads / 32; ++w) nrm += red[w];
  nrm = sqrtf(nrm);  // |E| in the Frobenius norm, the same bits in every CTA
  if (!(nrm < 1e-2f)) return false;
  if (nrm < 3e-5f) cqr_series<float>(ev, c, nrm < 2e-6f ? 1 : 2, Uf, Cf, Um, Cm);
  else cqr_series<double>(ev, c, nrm < 1e-4f ? 3 : (nrm < 1e-3f ? 4 : 7), Um, Cm, Um, Cm);
  // R = (I + U) R1
  double rv[kCqrPer];
#pragma unroll
  for (int x = 0; x < kCqrPer; ++x) {
    const int e = tid + x * kOrthThreads;
    if (e >= nt) continue;
    int p, q;
    tri_diag(e, c, &p, &q);
    double v = s.Rs[p * T3F_MAX_RANK + q];
#pragma unroll 4
    for (int r = p; r <= q; ++r) v = fma(Um[p * kCqrLd + r], s.Rs[r * T3F_MAX_RANK + q], v);
    rv[x] = v;
  }
  // Q = Q1 - Q1 C: sixteen lanes a row, lane l takes the columns l and c2 - 1 - l (c2 = c rounded up
  // to even), c2 + 1 steps for every lane
  const int half = (c + 1) / 2, c2 = 2 * half;
  for (int r0 = 0; r0 < nrow; r0 += kOrthThreads / 16) {
    const int r = r0 + tid / 16, l = tid % 16;
    const bool on = r < nrow && l < half;
    double lo = 0.0, hi = 0.0;
    const int ch = c2 - 1 - l;
    const double* w = s.W + (size_t)(on ? r : 0) * c;
    if (on) {
      const int cs = min(ch, c - 1);  // (c odd: lane 0 has no second column)
      double acc = w[l];
      hi = w[cs];
      for (int t = 0; t <= c2; ++t) {  // one fused multiply-add per step for every lane
        const bool sec = t > l;
        if (t == l + 1) {
          lo = acc;
          acc = hi;
        }
        const int r = min(sec ? t - l - 1 : t, cs);
        acc = fma(-w[r], Cm[r * kCqrLd + (sec ? cs : l)], acc);
      }
      hi = acc;
    }
    __syncwarp();
    if (on) {
      s.W[(size_t)r * c + l] = lo;
      if (ch < c) s.W[(size_t)r * c + ch] = hi;
    }
    __syncwarp();
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < kCqrPer; ++x) {
    const int e = tid + x * kOrthThreads;
    if (e >= nt) continue;
    int p, q;
    tri_diag(e, c, &p, &q);
    s.Rs[p * T3F_MAX_RANK + q] = rv[x];
  }
  __syncthreads();
  return true;
}

// Householder QR of the cluster's m x c unfolding W (this CTA's nrow rows from row0 in s.W): R (kk x c,
// diag(R) >= 0) in every CTA's s.Rs, the rows of Q in s.W (ld c).
__device__ void householder_step(const OrthArgs& a, const double* core, const Dims& dm, int R1, int lr, int m, int c,
                                 int rp, int row0, int nrow, const OrthSmem& s, cg::cluster_group& cluster) {
  const int P = a.P, tid = threadIdx.x, nth = blockDim.x;
  const int kk = m < c ? m : c;
  for (int j = 0; j < kk; ++j) {
    const int par = j & 1;
    double* pub = s.pub + par * T3F_MAX_RANK;
    double* rowj = s.rowj + par * T3F_MAX_RANK;
    const bool own_j = j >= row0 && j < row0 + nrow;
    // (1) partials over the owned rows strictly below the diagonal:
    //     pub[j] = sum x_r^2, pub[l] = sum x_r W[r][l] (l > j); the owner publishes row j.
    //     Eight lanes per column split the rows and combine with three shuffles.
    const int q_lo = max(0, j + 1 - row0);
    for (int cb = j; cb < c; cb += nth / 8) {
      const int l = cb + tid / 8, g = tid % 8;
      double acc = 0.0;
      if (l < c)
        for (int q = q_lo + g; q < nrow; q += 8) acc = fma(s.W[q * c + j], s.W[q * c + l], acc);
      acc += __shfl_xor_sync(0xffffffffu, acc, 4, 8);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2, 8);
      acc += __shfl_xor_sync(0xffffffffu, acc, 1, 8);
      if (g == 0 && l < c) pub[l] = acc;
    }
    if (own_j)
      for (int l = j + tid; l < c; l += nth) rowj[l] = s.W[(j - row0) * c + l];
    __syncthreads();
    cluster.sync();
    // (2) gather the cluster sums (8 lanes per column, each reading the partials of ranks g
    //     and g + 8 in one round trip); the lane that owns column j also forms the reflector
    //     (LAPACK dlarfg convention: beta = -sign(w) |x|, tau = (beta - w) / beta,
    //     scale = 1 / (w - beta), with 1 / |x| from one reciprocal square root)
    const int jown = j / rp;
    const int ng = ((c - j) * 8 + 31) & ~31;  // whole warps take part in the shuffles
    for (int e = tid; e < ng; e += nth) {
      const int l = j + e / 8, p = e % 8;
      double v = 0.0, v2 = 0.0, wl = 0.0;
      if (l < c) {
        if (p < P) v = cluster.map_shared_rank(pub, p)[l];
        if (p + 8 < P) v2 = cluster.map_shared_rank(pub, p + 8)[l];
        if (p == 0) wl = cluster.map_shared_rank(rowj, jown)[l];  // issued with v
      }
      v += v2;
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, 8);
      if (p == 0 && l < c) {
        s.gsum[l] = v;
        s.wj[l] = wl;
        if (l == j) {
          double beta = wl, tau = 0.0, scale = 0.0;
          if (v != 0.0) {
            const double x2 = wl * wl + v, rn = rsqrt(x2), nrm = x2 * rn;
            const bool pos = wl >= 0.0;
            beta = pos ? -nrm : nrm;
            tau = pos ? 1.0 + wl * rn : 1.0 - wl * rn;  // 1 - wl / beta
            scale = 1.0 / (wl - beta);
          }
          s.refl[0] = beta;
          s.refl[1] = tau;
          s.refl[2] = scale;
        }
      }
    }
    __syncthreads();
    const double beta = s.refl[0], tau = s.refl[1], scale = s.refl[2];
    // (3) w_l = v . W[:, l] for the trailing columns and tau v_r for the owned rows, then the
    //     rank-one update of the owned rows
    for (int l = j + 1 + tid; l < c; l += nth) s.gsum[l] = s.wj[l] + scale * s.gsum[l];
    const int q_j = max(0, j - row0);
    for (int q = q_j + tid; q < nrow; q += nth) s.tv[q] = row0 + q == j ? tau : tau * scale * s.W[q * c + j];
    __syncthreads();
    const int wc = c - j - 1, wr = nrow - q_j;
    for (int e = tid; e < wr * wc; e += nth) {
      const int q = q_j + e / wc, l = j + 1 + e % wc;
      s.W[q * c + l] -= s.tv[q] * s.gsum[l];
    }
    if (own_j && tid == 0) s.W[(j - row0) * c + j] = beta;
    __syncthreads();
  }
  cluster.sync();  // every row of R is final in its owner's shared memory
  // (C) R (kk x c) from the owners of rows 0..kk-1, normalised to diag(R) >= 0
  for (int e = tid; e < kk * c; e += nth) {
    const int j = e / c, l = e % c;
    double v = 0.0;
    if (l >= j) {
      const int own = j / rp;
      v = cluster.map_shared_rank(s.W, own)[(j - own * rp) * c + l];
    }
    s.Rs[j * T3F_MAX_RANK + l] = v;
  }
  __syncthreads();
  for (int e = tid; e < kk * c; e += nth) {
    const int j = e / c, l = e % c;
    if (s.Rs[j * T3F_MAX_RANK + j] < 0.0 && l != j) s.Rs[j * T3F_MAX_RANK + l] = -s.Rs[j * T3F_MAX_RANK + l];
  }
  __syncthreads();
  for (int j = tid; j < kk; j += nth) {
    const double dg = fabs(s.Rs[j * T3F_MAX_RANK + j]);
    s.Rs[j * T3F_MAX_RANK + j] = dg;
    s.rinv[j] = 1.0 / dg;
  }
  cluster.sync();  // all CTAs are done reading remote W before it is reused below
  // (D) Q rows = W rows R[:kk,:kk]^{-1}: reload the original rows, forward substitution
  for (int e = tid; e < nrow * kk; e += nth) {
    const int q = e / kk, l = e % kk;
    s.W[q * c + l] = core[w_addr(lr, row0 + q, l, dm, R1)];
  }
  __syncthreads();
  // right-looking substitution: once q_b is known it is removed from every later column.
  // Eight lanes share a row: lane g keeps the columns l = g (mod 8) of the row in registers
  // and the owner of column b broadcasts q_b with a shuffle.
  if (kk <= 64) {
    const int g = tid % 8;
    const int nq = (nrow + (nth / 8) - 1) / (nth / 8);
    for (int it = 0; it < nq; ++it) {
      const int q = it * (nth / 8) + tid / 8;
      const bool qv = q < nrow;
      double* qr = s.W + (qv ? q : 0) * c;
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int l = g + 8 * u;
        x[u] = (qv && l < kk) ? qr[l] : 0.0;
      }
      const int uend = (kk + 7) / 8;  // register slots holding columns < kk
      // column b = 8 UB + ob lives in slot UB of lane ob; only the slots UB .. uend-1 hold
      // columns l > b, so the loops start at UB at compile time and no update is issued
      // for the slots below it (the FP64 pipe is the scarce one)
#pragma unroll
      for (int UB = 0; UB < 8; ++UB) {
        if (UB >= uend) break;
        for (int ob = 0; ob < 8; ++ob) {
          const int b = 8 * UB + ob;
          if (b >= kk) break;
          double xb = __shfl_sync(0xffffffffu, x[UB] * s.rinv[b], ob, 8);
          if (g == ob) x[UB] = xb;
          const double* rb = s.Rs + b * T3F_MAX_RANK;
#pragma unroll
          for (int u = UB; u < 8; ++u) {
            const int l = g + 8 * u;
            if (u < uend && l > b && l < kk) x[u] = fma(-xb, rb[l], x[u]);
          }
        }
      }
      if (qv) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int l = g + 8 * u;
          if (l < kk) qr[l] = x[u];
        }
      }
    }
  }
  __syncthreads();
}

// out(a, x) = sum_{al >= a} R(a, al) in(al, x) for a < kk, x < nx: the lanes of a warp run over x with
// one row a (sums of equal length), and a thread takes the rows a and kk - 1 - a together, so every
// thread does the same work on two independent chains (up to three rows: one element a thread).
template <class FR, class FI, class FO>
__device__ __forceinline__ void push_rows(int kk, int c, int nx, FR R, FI in, FO out) {
  if (kk < 4) {
    for (int e = threadIdx.x; e < kk * nx; e += blockDim.x) {
      const int a = e / nx, x = e % nx;
      double u = 0.0;
      for (int al = a; al < c; ++al) u = fma(R(a, al), in(al, x), u);
      out(a, x, u);
    }
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int na = (kk + 1) / 2, ng = (nx + 31) / 32;
  for (int w = warp; w < na * ng; w += nw) {
    const int a = w % na, b = kk - 1 - a, x = (w / na) * 32 + lane;  // a <= b
    if (x >= nx) continue;
    double u = 0.0, v = 0.0;
    int al = a;
    for (; al < b; ++al) u = fma(R(a, al), in(al, x), u);
    for (; al < c; ++al) {
      const double t = in(al, x);
      u = fma(R(a, al), t, u);
      v = fma(R(b, al), t, v);
    }
    out(a, x, u);
    if (b != a) out(b, x, v);
  }
}

// One QR step of a sweep on core k (updates dims for core k and its neighbour).
__device__ void qr_step(const OrthArgs& a, double* base, Dims* dims, int k, int lr,
                        const OrthSmem& s, cg::cluster_group& cluster) {
  const int P = a.P;
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, nth = blockDim.x;
  const Dims dm = dims[k];
  const int m = lr ? dm.r0 * dm.n : dm.n * dm.r1;
  const int c = lr ? dm.r1 : dm.r0;
  const int kk = m < c ? m : c;
  const int rp = (m + P - 1) / P;
  const int row0 = rank * rp;
  const int nrow = max(0, min(m, row0 + rp) - row0);
  double* core = base + a.coff[k];
  const int R1 = a.R1[k];

  cluster.sync();  // previous step's global writes are visible; remote smem reads are done
  for (int e = tid; e < nrow * c; e += nth) {
    const int q = e / c, l = e % c;
    s.W[e] = core[w_addr(lr, row0 + q, l, dm, R1)];
  }
  __syncthreads();

  // A Householder column is 2.5 to 3.5 us, cqr_step some 12 to 15 us up to eight columns, and a square
  // unfolding is often refused. d = 8, n = 8, Householder against cqr_step, us: r = 1 148, 229; r = 2 222, 261;
  // r = 3 283, 269; r = 4 338, 280; r = 5 394, 286; d = 10, n = 4: r = 3 361, 342; 4 x 4 and 4 x 5 unfoldings
  // (d = 2, n = 4) 52, 58.
  bool done = false;
  if (c >= 4 && c <= kCqrMax && m >= (c < 6 ? c + 1 : c)) {
    done = cqr_step(a, s, nrow, c, cluster);
    if (!done) {  // the rows again, for the Householder columns
      __syncthreads();
      for (int e = tid; e < nrow * c; e += nth) {
        const int q = e / c, l = e % c;
        s.W[e] = core[w_addr(lr, row0 + q, l, dm, R1)];
      }
      __syncthreads();
    }
  }
  if (!done) householder_step(a, core, dm, R1, lr, m, c, rp, row0, nrow, s, cluster);
  Dims nd = dm;
  if (lr) nd.r1 = kk; else nd.r0 = kk;
  for (int e = tid; e < nrow * kk; e += nth) {
    const int q = e / kk, l = e % kk;
    // L->R: new core (r0, n, kk) row q col l; R->L: new core (kk, n, r1) = Q^T
    core[w_addr(lr, row0 + q, l, nd, R1)] = s.W[q * c + l];
  }
  __syncthreads();
  // (E) push R into the neighbour core, split across the cluster; operands staged in smem
  if (lr) {
    const Dims nx = dims[k + 1];  // (c, n', r2)
    double* nb = base + a.coff[k + 1];
    const int R1n = a.R1[k + 1];
    const int cols = nx.n * nx.r1;
    const int cp = (cols + P - 1) / P, c0 = rank * cp, nc = max(0, min(cols, c0 + cp) - c0);
    for (int e = tid; e < c * nc; e += nth) {
      const int al = e / nc, q = c0 + e % nc;
      const int i = q / nx.r1, b = q % nx.r1;
      s.W[e] = nb[((long long)al * nx.n + i) * R1n + b];
    }
    __syncthreads();
    push_rows(kk, c, nc, [&](int a2, int al) { return s.Rs[a2 * T3F_MAX_RANK + al]; },
              [&](int al, int qq) { return s.W[al * nc + qq]; },
              [&](int a2, int qq, double v) {
                const int q = c0 + qq, i = q / nx.r1, b = q % nx.r1;
                nb[((long long)a2 * nx.n + i) * R1n + b] = v;
              });
  } else {
    const Dims pv = dims[k - 1];  // (r0', n', c)
    double* pb = base + a.coff[k - 1];
    const int R1p = a.R1[k - 1];
    const int rows = pv.r0 * pv.n;
    const int rq = (rows + P - 1) / P, q0 = rank * rq, nq = max(0, min(rows, q0 + rq) - q0);
    // rows are read across the lanes: an odd stride where it fits the W region (sized for stride
    // T3F_MAX_RANK; c = 64 with 253 rows or more does not fit and keeps the even one)
    const int ldw = nq * (c | 1) <= a.rows_per * T3F_MAX_RANK ? c | 1 : c;
    for (int e = tid; e < nq * c; e += nth) {
      const int q = e / c, b = e % c;
      s.W[q * ldw + b] = pb[(long long)(q0 + q) * R1p + b];
    }
    __syncthreads();
    push_rows(kk, c, nq, [&](int a2, int b) { return s.Rs[a2 * T3F_MAX_RANK + b]; },
              [&](int b, int q) { return s.W[q * ldw + b]; },
              [&](int a2, int q, double v) { pb[(long long)(q0 + q) * R1p + a2] = v; });
  }
  __syncthreads();  // (the cluster barrier that opens the next step publishes the global writes)
  if (tid == 0) {
    if (lr) {
      dims[k].r1 = kk;
      dims[k + 1].r0 = kk;
    } else {
      dims[k].r0 = kk;
      dims[k - 1].r1 = kk;
    }
  }
  __syncthreads();
}

__device__ void write_out(const OrthArgs& a, const TTV& O, int obj, const double* base,
                          const Dims* dims, cg::cluster_group& cluster) {
  cluster.sync();
  const int P = a.P, rank = (int)cluster.block_rank();
  for (int k = 0; k < O.d; ++k) {
    const Dims dm = dims[k];
    const long long sz = (long long)dm.r0 * dm.n * dm.r1;
    const long long ob = core_base(O, k, obj);
    for (long long e = (long long)rank * blockDim.x + threadIdx.x; e < sz; e += (long long)P * blockDim.x) {
      const int b = (int)(e % dm.r1);
      const long long ai = e / dm.r1;
      const double v = base[a.coff[k] + ai * a.R1[k] + b];
      if (O.dtype == T3F_F64) static_cast<double*>(O.p)[ob + e] = v;
      else static_cast<float*>(O.p)[ob + e] = (float)v;
    }
  }
}

__global__ void __launch_bounds__(kOrthThreads) k_orth(const __grid_constant__ OrthArgs a) {
  extern __shared__ double smd[];
  __shared__ Dims dims[T3F_MAX_D];
  cg::cluster_group cluster = cg::this_cluster();
  const int obj = blockIdx.x / a.P;
  const int rank = (int)cluster.block_rank();
  const TTV& X = a.X;
  const int d = X.d;
  OrthSmem s;
  s.W = smd;
  s.Rs = s.W + (size_t)a.rows_per * T3F_MAX_RANK;
  s.pub = s.Rs + T3F_MAX_RANK * T3F_MAX_RANK;
  s.rowj = s.pub + 2 * T3F_MAX_RANK;
  s.gsum = s.rowj + 2 * T3F_MAX_RANK;
  s.wj = s.gsum + T3F_MAX_RANK;
  s.rinv = s.wj + T3F_MAX_RANK;
  s.tv = s.rinv + T3F_MAX_RANK;
  s.refl = s.tv + a.rows_per;
  double* base = a.work + (long long)obj * a.obj_stride;
  for (int k = threadIdx.x; k < d; k += blockDim.x) dims[k] = Dims{X.r[k], X.n[k], X.r[k + 1]};
  // load X (split across the cluster) into the padded FP64 working cores
  for (int k = 0; k < d; ++k) {
    const long long sz = X.osz[k];
    const long long ob = core_base(X, k, obj);
    for (long long e = (long long)rank * blockDim.x + threadIdx.x; e < sz; e += (long long)a.P * blockDim.x) {
      const double v = X.dtype == T3F_F64 ? static_cast<const double*>(X.p)[ob + e]
                                          : (double)static_cast<const float*>(X.p)[ob + e];
      base[a.coff[k] + e] = v;  // the padded stride equals the original one for X
    }
  }
  __threadfence();
  __syncthreads();
  for (int k = d - 1; k >= 1; --k) qr_step(a, base, dims, k, 0, s, cluster);
  for (int k = 0; k < d - 1; ++k) qr_step(a, base, dims, k, 1, s, cluster);
  __threadfence();
  write_out(a, a.U, obj, base, dims, cluster);
  for (int k = d - 1; k >= 1; --k) qr_step(a, base, dims, k, 0, s, cluster);
  __threadfence();
  write_out(a, a.V, obj, base, dims, cluster);
}

static long long orth_obj_stride(const TTV& X, long long* coff, int* R1) {
  long long o = 0;
  for (int k = 0; k < X.d; ++k) {
    if (coff) coff[k] = o;
    if (R1) R1[k] = X.r[k + 1];
    o += X.osz[k];
  }
  return (o + 31) & ~31LL;
}

static size_t orth_smem(int rows_per) {
  return sizeof(double) * ((size_t)rows_per * T3F_MAX_RANK + T3F_MAX_RANK * T3F_MAX_RANK + 7 * T3F_MAX_RANK + rows_per + 4);
}

// Largest supported cluster size (16 if allowed, else 8), cached per process.
static int orth_cluster_size(size_t* smem_out) {
  static int P = -1;
  static size_t smem = 0;
  if (P >= 0) {
    *smem_out = smem;
    return P;
  }
  P = 0;
  for (int cand : {16, 8}) {
    const int rows_per = (kOrthMaxRows + cand - 1) / cand;
    const size_t sm = orth_smem(rows_per);
    if (cudaFuncSetAttribute(k_orth, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (cand > 8 && cudaFuncSetAttribute(k_orth, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cand;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(cand);
    cfg.blockDim = dim3(kOrthThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, k_orth, &cfg) == cudaSuccess && nclusters > 0) {
      P = cand;
      smem = sm;
      break;
    }
    cudaGetLastError();
  }
  *smem_out = smem;
  return P;
}

size_t ws_orth(const TTV& X) {
  return kWsHeader + align256(sizeof(double) * orth_obj_stride(X, nullptr, nullptr) * X.batch);
}

}  // namespace t3f

using namespace t3f;

extern "C" t3f_status t3f_orthogonalize(const t3f_tt* X, t3f_tt* U, t3f_tt* V, void* ws,
                                        size_t ws_bytes, t3f_stream_t stream) {
  TTV vx, vu, vv;
  T3F_CHECK(make_view(X, &vx, -1, false));
  if (vx.dtype == T3F_BF16) return T3F_ERR_DTYPE;
  T3F_CHECK(make_view(U, &vu, -1, false));
  T3F_CHECK(make_view(V, &vv, -1, false));
  if (vu.dtype == T3F_BF16 || vv.dtype == T3F_BF16) return T3F_ERR_DTYPE;
  if (vx.rmax > T3F_MAX_RANK) return T3F_ERR_UNSUPPORTED;
  for (int k = 0; k < vx.d; ++k) {
    if ((long long)vx.r[k] * vx.n[k] > kOrthMaxRows) return T3F_ERR_UNSUPPORTED;
    if ((long long)vx.n[k] * vx.r[k + 1] > kOrthMaxRows) return T3F_ERR_UNSUPPORTED;
  }
  int ru[T3F_MAX_D + 1];
  int xn[T3F_MAX_D], xr[T3F_MAX_D + 1];
  for (int k = 0; k < vx.d; ++k) xn[k] = vx.n[k];
  for (int k = 0; k <= vx.d; ++k) xr[k] = vx.r[k];
  T3F_CHECK(t3f_orth_ranks(vx.d, xn, xr, ru));
  for (const TTV* o : {&vu, &vv}) {
    if (o->batch != vx.batch || o->d != vx.d) return T3F_ERR_SHAPE;
    for (int k = 0; k <= vx.d; ++k)
      if (o->r[k] != ru[k] || (k < vx.d && o->n[k] != vx.n[k])) return T3F_ERR_SHAPE;
  }
  T3F_CHECK(check_ws(ws, ws_bytes, ws_orth(vx)));
  size_t smem = 0;
  const int P = orth_cluster_size(&smem);
  if (P == 0) return T3F_ERR_UNSUPPORTED;
  OrthArgs args;
  memset(&args, 0, sizeof(args));
  args.X = vx;
  args.U = vu;
  args.V = vv;
  args.P = P;
  args.rows_per = (kOrthMaxRows + P - 1) / P;
  args.work = reinterpret_cast<double*>(static_cast<char*>(ws) + kWsHeader);
  args.obj_stride = orth_obj_stride(vx, args.coff, args.R1);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = P;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(P * vx.batch));
  cfg.blockDim = dim3(kOrthThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k_orth, args) != cudaSuccess) {
    cudaGetLastError();
    return T3F_ERR_CUDA;
  }
  return launch_status();
}
