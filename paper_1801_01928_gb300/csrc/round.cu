// TT rounding (paper Section 3, t3f.round: the best approximation of lower TT-rank), the
// TT-SVD recompression of Oseledets (2011) in FP64, one CTA per object:
//   1. right to left, k = d-1..1: Householder QR of the transposed unfolding
//      W_k^T = ((n_k r_k) x r_{k-1}) = Q R with diag(R) >= 0, in place (the reflectors stay in
//      W_k below the diagonal of R, Q is never formed), W_{k-1} <- W_{k-1} R^T;
//   2. left to right, k = 0..d-2: SVD of the (r_{k-1} n_k) x r_k unfolding M = U S V^T through
//      the eigen-decomposition (cyclic Jacobi, FP64, shared memory) of the smaller of M M^T and
//      M^T M, truncated to the leading p = min(max_rank, rows, cols) triplets; every kept left
//      singular vector has its entry of largest magnitude positive; W_k <- U,
//      W_{k+1} <- (S V^T) Q_{k+1}^T, the reflectors applied to the p rows.
// The working cores live in the workspace in FP64 (each core keeps its input capacity; ranks
// only shrink); the output is written in FP32. The eigen-decompositions are limited to
// T3F_ROUND_MAX_SIDE rows (160 KB of shared memory for the matrix and its eigenvectors).
//
// What bounds it: an SM runs about two FP64 multiply-adds per clock, so the work is counted in
// those. The reflectors are applied to p rows instead of forming Q (p / r of its cost); the QR
// takes panels of eight columns, one column per warp in registers while the panel is factored,
// and then passes the panel's eight reflectors over two trailing columns at a time held in
// registers (one read and one write of a column per panel instead of per reflector; two
// columns share their lane reductions); W R^T runs the triangle only. 100 objects of rank 100
// (d = 10, n = 4) to rank 10: 57.0 ms with Q formed column by column through L2, 27.4 ms this
// way, the FP64 pipe of the 100 busy SMs 62 % active (28.1 ms and 70 % with one register count for all
// column heights, of which the QR took 43 %, W R^T 17 %, Jacobi 27 %, reflectors on the kept rows 10 %).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "t3f_internal.cuh"

namespace t3f {

namespace {

constexpr int kRoundThreads = 256;
constexpr int kMaxSide = 100;  // largest eigenproblem (rows of the Gram matrix)
constexpr int kPanel = kRoundThreads / 32;  // columns of a QR panel: one per warp
constexpr int kRegRows = 16;                // register slots of a column (32 rows each)
constexpr int kDynDoubles = 2 * kMaxSide * (kMaxSide + 1);  // dynamic shared memory
constexpr int kRtRows = 7;   // W R^T: 32-row groups of a tile
constexpr int kRtK = 64;     // W R^T: steps staged at a time
constexpr int kRtLd = 32 * kRtRows + 1;
static_assert(kRtK * (kRtLd + 17) <= kDynDoubles, "W R^T staging");
static_assert(kPanel * 32 * kRegRows <= kDynDoubles, "QR panel");

struct RoundArgs {
  TTV X, Y;
  int maxr;
  long long coff[T3F_MAX_D];  // FP64 offset of core k inside an object's working set
  long long maxcore;          // largest core (elements)
  long long per_obj;          // doubles per object: cores + 2 scratch buffers
  double* ws;
  int* err;
};

__device__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;
}

// Lane sums of two values at once: lanes 0-15 end with the sum of a, lanes 16-31 with that of
// b (five additions for both instead of ten); every lane receives both.
__device__ __forceinline__ void warp_sum2(double& a, double& b) {
  const bool hi = (threadIdx.x & 16) != 0;
  double mine = hi ? b : a;
  mine += __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  a = __shfl_sync(0xffffffffu, mine, 0);
  b = __shfl_sync(0xffffffffu, mine, 16);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// y0, y1 <- (I - tau v v^T) y0, y1 with the vectors spread over the lanes (element 32 c + lane
// in slot c); the slots below c0 hold zeros of v. NC: the slots a column of this height can use, at
// compile time, since an FP64 instruction that is predicated off takes its turn on the pipe all the same
// (16 slots for every height: 21 objects of rank 46, d = 8, n = 2, to rank 12 2970 us, now 1390).
template <int NC>
__device__ __forceinline__ void reflect2(const double (&v)[NC], double tau, int c0, int nch, double (&y0)[NC],
                                         double (&y1)[NC]) {
  double s0 = 0.0, s1 = 0.0;
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (c >= c0 && c < nch) {
      s0 = fma(v[c], y0[c], s0);
      s1 = fma(v[c], y1[c], s1);
    }
  warp_sum2(s0, s1);
  s0 *= -tau;
  s1 *= -tau;
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (c >= c0 && c < nch) {
      y0[c] = fma(s0, v[c], y0[c]);
      y1[c] = fma(s1, v[c], y1[c]);
    }
}

template <int NC>
__device__ __forceinline__ void reflect1(const double (&v)[NC], double tau, int c0, int nch, double (&y)[NC]) {
  double s0 = 0.0, s1 = 0.0;  // two chains: one column alone is latency-bound
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (c >= c0 && c < nch) {
      if (c & 1) s1 = fma(v[c], y[c], s1);
      else s0 = fma(v[c], y[c], s0);
    }
  const double s = -tau * warp_sum(s0 + s1);
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (c >= c0 && c < nch) y[c] = fma(s, v[c], y[c]);
}

template <int NC>
__device__ __forceinline__ void load_col(const double* p, int m, int nch, double (&y)[NC]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    y[c] = 0.0;
    if (c < nch && 32 * c + lane < m) y[c] = p[32 * c + lane];
  }
}

template <int NC>
__device__ __forceinline__ void store_col(double* p, int m, int nch, const double (&y)[NC]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (c < nch && 32 * c + lane < m) p[32 * c + lane] = y[c];
}

// f with the register slots of a column of m <= 32 kRegRows rows.
template <class F>
__device__ __forceinline__ void by_slots(int m, F f) {
  if (m <= 32) f(std::integral_constant<int, 1>());
  else if (m <= 64) f(std::integral_constant<int, 2>());
  else if (m <= 128) f(std::integral_constant<int, 4>());
  else if (m <= 256) f(std::integral_constant<int, 8>());
  else f(std::integral_constant<int, kRegRows>());
}

// The QR below for columns of at most 32 NC rows, panel by panel.
template <int NC>
__device__ void qr_panels(double* A, int m, int c, double* vp, double* tp) {
  const int q = min(m, c);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kRoundThreads / 32;
  const int nch = (m + 31) / 32;
  for (int j0 = 0; j0 < q; j0 += kPanel) {
    const int nb = min(kPanel, q - j0), cb = j0 / 32;
    {  // factor the panel: warp w holds column j0 + w
      double y[NC];
      const bool mine = warp < nb;
      if (mine) load_col(A + (long long)(j0 + warp) * m, m, nch, y);
      for (int jj = 0; jj < nb; ++jj) {
        const int j = j0 + jj;
        double* vj = vp + jj * (32 * NC);
        if (warp == jj) {
          double part = 0.0, x0 = 0.0;
#pragma unroll
          for (int c2 = 0; c2 < NC; ++c2)
            if (c2 >= cb && c2 < nch) {
              const int i = 32 * c2 + lane;
              if (i >= j) part = fma(y[c2], y[c2], part);
              if (i == j) x0 = y[c2];
            }
          part = warp_sum(part);
          x0 = __shfl_sync(0xffffffffu, x0, j & 31);
          double alpha = 0.0, tau = 0.0, inv = 0.0;
          if (part > 0.0) {
            const double rn = rsqrt(part);
            alpha = x0 >= 0.0 ? -(part * rn) : part * rn;
            tau = fma(fabs(x0), rn, 1.0);  // -v0 / alpha
            inv = 1.0 / (x0 - alpha);
          }
#pragma unroll
          for (int c2 = 0; c2 < NC; ++c2)
            if (c2 < nch) {
              const int i = 32 * c2 + lane;
              if (i >= j) y[c2] = i == j ? alpha : y[c2] * inv;
              vj[i] = i > j ? y[c2] : (i == j ? 1.0 : 0.0);
            }
          if (lane == 0) tp[jj] = tau;
        }
        __syncthreads();
        if (mine && warp > jj) {
          double s = 0.0;
#pragma unroll
          for (int c2 = 0; c2 < NC; ++c2)
            if (c2 >= cb && c2 < nch) s = fma(vj[32 * c2 + lane], y[c2], s);
          s = -tp[jj] * warp_sum(s);
#pragma unroll
          for (int c2 = 0; c2 < NC; ++c2)
            if (c2 >= cb && c2 < nch) y[c2] = fma(s, vj[32 * c2 + lane], y[c2]);
        }
      }
      if (mine) store_col(A + (long long)(j0 + warp) * m, m, nch, y);
    }
    // the panel's reflectors over the trailing columns, two per warp at a time (one per warp when
    // at most eight are left, so that the last round spreads over all warps)
    for (int l0 = j0 + nb; l0 < c; l0 += 2 * nw) {
      const bool pairs = c - l0 > nw;
      const int l = l0 + (pairs ? 2 * warp : warp);
      if (l >= c) break;
      double y0[NC], y1[NC], v[NC];
      const bool two = pairs && l + 1 < c;
      if (!two) {
        load_col(A + (long long)l * m, m, nch, y0);
        for (int jj = 0; jj < nb; ++jj) {
          const double* vj = vp + jj * (32 * NC);
#pragma unroll
          for (int c2 = 0; c2 < NC; ++c2) v[c2] = c2 >= cb && c2 < nch ? vj[32 * c2 + lane] : 0.0;
          reflect1(v, tp[jj], cb, nch, y0);
        }
        store_col(A + (long long)l * m, m, nch, y0);
        continue;
      }
      load_col(A + (long long)l * m, m, nch, y0);
      load_col(A + (long long)(l + 1) * m, m, nch, y1);
      for (int jj = 0; jj < nb; ++jj) {
        const double* vj = vp + jj * (32 * NC);
#pragma unroll
        for (int c2 = 0; c2 < NC; ++c2) v[c2] = c2 >= cb && c2 < nch ? vj[32 * c2 + lane] : 0.0;
        reflect2(v, tp[jj], cb, nch, y0, y1);
      }
      store_col(A + (long long)l * m, m, nch, y0);
      store_col(A + (long long)(l + 1) * m, m, nch, y1);
    }
    __syncthreads();
  }
}

// Householder QR in place of the column-major m x c matrix A (column a at A + a*m), q =
// min(m, c) reflectors: on return column j holds R[0..j][j] on and above the diagonal (signs as
// they come) and below it the reflector v_j (v_j[j] = 1 not stored; H_j = I - tau_j v_j v_j^T,
// tau_j = 2 / |v_j|^2, or 0 where R[j][j] = 0). vp: kPanel x 32 kRegRows doubles of shared
// memory, tp: kPanel. Columns longer than 32 kRegRows go through memory one reflector at a time.
__device__ void householder_qr(double* A, int m, int c, double* vp, double* tp, double* red) {
  const int q = min(m, c);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kRoundThreads / 32;
  if (m > 32 * kRegRows) {
    for (int j = 0; j < q; ++j) {
      double* x = A + (long long)j * m;
      double part = 0.0;
      for (int i = j + tid; i < m; i += kRoundThreads) part += x[i] * x[i];
      const double nrm2 = block_sum(part, red);
      const double x0 = x[j];
      const double alpha = x0 >= 0.0 ? -sqrt(nrm2) : sqrt(nrm2);
      const double v0 = x0 - alpha, tau = nrm2 > 0.0 ? -v0 / alpha : 0.0, inv = nrm2 > 0.0 ? 1.0 / v0 : 0.0;
      __syncthreads();
      for (int i = j + tid; i < m; i += kRoundThreads) x[i] = i == j ? alpha : x[i] * inv;
      __syncthreads();
      for (int l = j + 1 + warp; l < c; l += nw) {
        double* y = A + (long long)l * m;
        double s = 0.0;
        for (int i = j + 1 + lane; i < m; i += 32) s += x[i] * y[i];
        s = tau * (warp_sum(s) + y[j]);
        __syncwarp();
        if (lane == 0) y[j] -= s;
        for (int i = j + 1 + lane; i < m; i += 32) y[i] -= s * x[i];
      }
      __syncthreads();
    }
    return;
  }
  by_slots(m, [&](auto nc) { qr_panels<decltype(nc)::value>(A, m, c, vp, tp); });
}

// The kept rows below for at most 32 NC columns, in registers.
template <int NC>
__device__ void apply_rows(const double* A, int m, int q, const double* B, int p, double* out, const double* tau) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kRoundThreads / 32;
  const int nch = (m + 31) / 32;
  for (int b0 = 0; b0 < p; b0 += 2 * nw) {
    // up to 16 rows a round: the first `dbl` warps take two, so that no scheduler holds more
    // than one above its share
    const int rem = min(p - b0, 2 * nw), dbl = max(0, rem - nw);
    const bool two = warp < dbl;
    const int b = b0 + (two ? 2 * warp : warp + dbl);
    if (b >= b0 + rem) continue;
    double y0[NC], y1[NC], v[NC], vn[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int i = 32 * c + lane;
      y0[c] = y1[c] = 0.0;
      if (c < nch && i < q) {
        const double sg = A[(long long)i * m + i] < 0.0 ? -1.0 : 1.0;
        y0[c] = sg * B[(long long)b * q + i];
        if (two) y1[c] = sg * B[(long long)(b + 1) * q + i];
      }
    }
    load_col(A + (long long)(q - 1) * m, m, nch, vn);
    for (int j = q - 1; j >= 0; --j) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int i = 32 * c + lane;
        v[c] = i > j ? vn[c] : (i == j ? 1.0 : 0.0);
      }
      if (j > 0) load_col(A + (long long)(j - 1) * m, m, nch, vn);  // in flight during this reflector
      if (two) reflect2(v, tau[j], j / 32, nch, y0, y1);
      else reflect1(v, tau[j], j / 32, nch, y0);
    }
    store_col(out + (long long)b * m, m, nch, y0);
    if (two) store_col(out + (long long)(b + 1) * m, m, nch, y1);
  }
}

// rows b < p of out (p x m, row-major) <- (b-th row of B (p x q) diag(sgn)) Q^T with Q from the
// reflectors left in A by householder_qr; sgn_j = sign of R[j][j] (the diag(R) >= 0 convention).
// tau: q doubles of shared memory.
__device__ void apply_q(const double* A, int m, int q, const double* B, int p, double* out, double* tau) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kRoundThreads / 32;
  for (int j = warp; j < q; j += nw) {
    const double* v = A + (long long)j * m;
    double s = 0.0;
    for (int i = j + 1 + lane; i < m; i += 32) s = fma(v[i], v[i], s);
    s = warp_sum(s);
    if (lane == 0) tau[j] = v[j] == 0.0 ? 0.0 : 2.0 / (1.0 + s);
  }
  __syncthreads();
  if (m > 32 * kRegRows) {
    for (int b = warp; b < p; b += nw) {
      double* y = out + (long long)b * m;
      for (int i = lane; i < m; i += 32)
        y[i] = i < q ? (A[(long long)i * m + i] < 0.0 ? -B[(long long)b * q + i] : B[(long long)b * q + i]) : 0.0;
      __syncwarp();
      for (int j = q - 1; j >= 0; --j) {
        const double* v = A + (long long)j * m;
        double s = 0.0;
        for (int i = j + 1 + lane; i < m; i += 32) s = fma(v[i], y[i], s);
        s = tau[j] * (warp_sum(s) + y[j]);
        __syncwarp();
        if (lane == 0) y[j] -= s;
        for (int i = j + 1 + lane; i < m; i += 32) y[i] = fma(-s, v[i], y[i]);
        __syncwarp();
      }
    }
    return;
  }
  by_slots(m, [&](auto nc) { apply_rows<decltype(nc)::value>(A, m, q, B, p, out, tau); });
}

// out (rows x q, row-major) = Wp (rows x c) R^T with R (q x c, upper trapezoid, rows normalised
// to diag(R) >= 0) in the column-major A (ld m). Tiles of up to 224 rows x 16 columns: a warp
// owns two columns j and starts its sum at the first a >= j (the zero triangle is skipped); a
// lane owns one row of each of the tile's 32-row groups, which are shared out evenly over the
// tiles. 64 steps are staged at a time. wt: kRtK x kRtLd, rt: kRtK x 17 doubles of shared memory.
// NX: the most 32-row groups of a tile here.
template <int NX>
__device__ void mul_rt_tiles(const double* Wp, int rows, int c, const double* A, int m, int q, double* out, double* wt,
                             double* rt) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ng = (rows + 31) / 32, nt = (ng + kRtRows - 1) / kRtRows;
  for (int t = 0; t < nt; ++t) {
    const int g0 = (int)((long long)t * ng / nt), nx = (int)((long long)(t + 1) * ng / nt) - g0;
    const int i0 = 32 * g0, nr = min(32 * nx, rows - i0);
    for (int j0 = 0; j0 < q; j0 += 16) {
      double acc[NX][2];
#pragma unroll
      for (int x = 0; x < NX; ++x) acc[x][0] = acc[x][1] = 0.0;
      const int ja = j0 + 2 * warp;
      for (int a0 = j0; a0 < c; a0 += kRtK) {
        const int na = min(kRtK, c - a0);
        __syncthreads();
        for (int e = tid; e < kRtK * nr; e += kRoundThreads) {
          const int r = e / kRtK, aa = e % kRtK;
          if (aa < na) wt[aa * kRtLd + r] = Wp[(long long)(i0 + r) * c + a0 + aa];
        }
        for (int e = tid; e < na * 16; e += kRoundThreads) {
          const int aa = e >> 4, j = j0 + (e & 15), col = a0 + aa;
          double v = 0.0;
          if (j < q && j <= col) {
            v = A[(long long)col * m + j];
            if (A[(long long)j * m + j] < 0.0) v = -v;
          }
          rt[aa * 17 + (e & 15)] = v;
        }
        __syncthreads();
        if (ja < q)
          for (int aa = max(0, ja - a0); aa < na; ++aa) {
            const double r0 = rt[aa * 17 + 2 * warp], r1 = rt[aa * 17 + 2 * warp + 1];
#pragma unroll
            for (int x = 0; x < NX; ++x)
              if (x < nx) {
                const double w = wt[aa * kRtLd + 32 * x + lane];
                acc[x][0] = fma(w, r0, acc[x][0]);
                acc[x][1] = fma(w, r1, acc[x][1]);
              }
          }
      }
#pragma unroll
      for (int x = 0; x < NX; ++x) {
        const int r = 32 * x + lane;
        if (r < nr) {
          if (ja < q) out[(long long)(i0 + r) * q + ja] = acc[x][0];
          if (ja + 1 < q) out[(long long)(i0 + r) * q + ja + 1] = acc[x][1];
        }
      }
    }
  }
  __syncthreads();
}

__device__ void mul_rt(const double* Wp, int rows, int c, const double* A, int m, int q, double* out, double* wt,
                       double* rt) {
  if (rows <= 32) mul_rt_tiles<1>(Wp, rows, c, A, m, q, out, wt, rt);
  else if (rows <= 96) mul_rt_tiles<3>(Wp, rows, c, A, m, q, out, wt, rt);
  else mul_rt_tiles<kRtRows>(Wp, rows, c, A, m, q, out, wt, rt);
}

// Cyclic Jacobi eigen-decomposition of the symmetric positive semidefinite s x s matrix S
// (row-major with leading dimension ld, odd: its columns spread over the banks; shared memory)
// with rotations of s/2 disjoint pairs at a time (round-robin
// ordering); V receives the eigenvectors (columns), diag(S) the eigenvalues. The matrix is
// scaled by a power of two to a largest diagonal entry in [1, 2) meanwhile, so that the
// tangent of a rotation can be taken in FP32 and corrected by one FP64 Newton step (relative
// error ~1e-13, against an FP64 divide / root / divide chain of some 2000 clocks per round); c and
// s are FP64 with c^2 + s^2 = 1 to rounding, so the similarity is exact to FP64 for any tangent.
// A round updates S in 2 x 2 blocks (pair t1 x pair t2, t1 <= t2, both mirror images written)
// and V in the same barrier interval.
__device__ void jacobi_eig(double* S, double* V, int s, int ld, int* pp, int* pq, double* pc, double* ps, double* red,
                           unsigned short* tri) {
  const int tid = threadIdx.x;
  if (s == 1) {
    if (tid == 0) V[0] = 1.0;
    __syncthreads();
    return;
  }
  const int se = s + (s & 1);  // even count; index s is a dummy
  const int np = se / 2, ns = np * (np + 1) / 2;
  double dmax = 0.0;
  for (int i = 0; i < s; ++i) dmax = fmax(dmax, S[i * ld + i]);
  int ex = 0;
  frexp(dmax, &ex);
  const bool scale = dmax > 0.0 && isfinite(dmax);
  for (int t1 = tid; t1 < np; t1 += kRoundThreads)
    for (int t2 = t1; t2 < np; ++t2) tri[t1 * np - t1 * (t1 - 1) / 2 + t2 - t1] = (unsigned short)(t1 << 8 | t2);
  __syncthreads();
  for (int e = tid; e < s * s; e += kRoundThreads) {
    const int o = (e / s) * ld + e % s;
    V[o] = (e / s) == (e % s) ? 1.0 : 0.0;
    if (scale) S[o] = ldexp(S[o], 1 - ex);
  }
  __syncthreads();
  for (int sweep = 0; sweep < 40; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int e = tid; e < s * s; e += kRoundThreads) {
      const double v = S[(e / s) * ld + e % s];
      if ((e / s) == (e % s)) dia += v * v; else off += v * v;
    }
    off = block_sum(off, red);
    dia = block_sum(dia, red);
    if (off <= 1e-30 * dia || off == 0.0) break;
    for (int rnd = 0; rnd < se - 1; ++rnd) {
      // round-robin pairs: position 0 fixed, positions 1..se-1 rotate
      for (int t = tid; t < np; t += kRoundThreads) {
        auto at = [&](int pos) { return pos == 0 ? 0 : 1 + (pos - 1 + rnd) % (se - 1); };
        int p = at(t), q = at(se - 1 - t);
        if (p > q) { const int tmp = p; p = q; q = tmp; }
        double c = 1.0, sn = 0.0;
        if (q < s) {
          const double apq = S[p * ld + q], dd = S[q * ld + q] - S[p * ld + p];
          const float af = (float)apq, df = (float)dd;
          if (af != 0.0f) {
            // t^2 apq + t dd - apq = 0, the root of smaller magnitude
            const float z = df / (2.0f * af), az = fabsf(z);
            float tf = az > 1e9f ? 0.5f / az : 1.0f / (az + sqrtf(fmaf(z, z, 1.0f)));
            tf = z >= 0.0f ? tf : -tf;
            double t2 = (double)tf;
            const double f = fma(t2, fma(t2, apq, dd), -apq);
            const float fp = fmaf(2.0f * tf, af, df);
            if (fp != 0.0f) {
              const float corr = (float)f / fp;
              if (fabsf(corr) < 0.01f) t2 -= (double)corr;
            }
            c = rsqrt(fma(t2, t2, 1.0));
            sn = t2 * c;
          }
        }
        pp[t] = p;
        pq[t] = q;
        pc[t] = c;
        ps[t] = sn;
      }
      __syncthreads();
      for (int e = tid; e < ns + s * np; e += kRoundThreads) {
        if (e < ns) {
          const int t1 = tri[e] >> 8, t2 = tri[e] & 255;  // block (t1, t2), t1 <= t2
          const int p1 = pp[t1], q1 = pq[t1], p2 = pp[t2], q2 = pq[t2];
          const bool v1 = q1 < s, v2 = q2 < s;  // the dummy index has no row or column
          const double c1 = pc[t1], s1 = ps[t1], c2 = pc[t2], s2 = ps[t2];
          const double a = S[p1 * ld + p2], b = v2 ? S[p1 * ld + q2] : 0.0;
          const double cc = v1 ? S[q1 * ld + p2] : 0.0, dv = v1 && v2 ? S[q1 * ld + q2] : 0.0;
          // B <- J1^T B J2 with J = [[c, s], [-s, c]]
          const double a1 = c2 * a - s2 * b, b1 = s2 * a + c2 * b;
          const double g1 = c2 * cc - s2 * dv, d1 = s2 * cc + c2 * dv;
          const double a2 = c1 * a1 - s1 * g1, g2 = s1 * a1 + c1 * g1;
          const double b2 = c1 * b1 - s1 * d1, d2 = s1 * b1 + c1 * d1;
          S[p1 * ld + p2] = a2;
          S[p2 * ld + p1] = a2;
          if (v2) {
            S[p1 * ld + q2] = b2;
            S[q2 * ld + p1] = b2;
          }
          if (v1 && t1 != t2) {
            S[q1 * ld + p2] = g2;
            S[p2 * ld + q1] = g2;
          }
          if (v1 && v2) {
            S[q1 * ld + q2] = d2;
            S[q2 * ld + q1] = d2;
          }
        } else {
          const int ev = e - ns, i = ev / np, t = ev % np, p = pp[t], q = pq[t];
          if (q >= s) continue;
          const double c = pc[t], sn = ps[t];
          const double va = V[i * ld + p], vb = V[i * ld + q];
          V[i * ld + p] = c * va - sn * vb;
          V[i * ld + q] = sn * va + c * vb;
        }
      }
      __syncthreads();
    }
  }
  if (scale) {
    for (int i = tid; i < s; i += kRoundThreads) S[i * ld + i] = ldexp(S[i * ld + i], ex - 1);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kRoundThreads) k_round(const __grid_constant__ RoundArgs a) {
  extern __shared__ double dsm[];
  __shared__ double red[kRoundThreads / 32];
  __shared__ double sh_tau[kMaxSide + T3F_MAX_RANK];
  __shared__ double pc[kMaxSide / 2 + 1], ps[kMaxSide / 2 + 1], sig[kMaxSide];
  __shared__ unsigned short tri[(kMaxSide / 2) * (kMaxSide / 2 + 1) / 2];
  __shared__ int pp[kMaxSide / 2 + 1], pq[kMaxSide / 2 + 1], perm[kMaxSide];
  __shared__ int rk[T3F_MAX_D + 1];
  const int obj = blockIdx.x, tid = threadIdx.x, d = a.X.d;
  double* W = a.ws + (long long)obj * a.per_obj;
  double* S1 = W + a.coff[d - 1] + a.X.osz[d - 1];
  double* S2 = S1 + a.maxcore;
  // FP64 working copy of the object
  const float* Xp = static_cast<const float*>(a.X.p);
  for (int k = 0; k < d; ++k) {
    const float* src = Xp + core_base(a.X, k, obj);
    for (long long e = tid; e < a.X.osz[k]; e += blockDim.x) W[a.coff[k] + e] = (double)src[e];
  }
  if (tid <= d) rk[tid] = a.X.r[tid];
  __syncthreads();
  // 1. right-to-left orthogonalisation; W_k row-major r0 x (n r1) is W_k^T column-major
  for (int k = d - 1; k >= 1; --k) {
    const int r0 = rk[k], n = a.X.n[k], r1 = rk[k + 1];
    const int m = n * r1, c = r0, q = min(m, c);
    double* Wk = W + a.coff[k];
    householder_qr(Wk, m, c, dsm, sh_tau, red);
    // W_{k-1} <- W_{k-1} R^T: rows (r_{k-2} n_{k-1}), c -> q columns
    double* Wp = W + a.coff[k - 1];
    const int rows = rk[k - 1] * a.X.n[k - 1];
    mul_rt(Wp, rows, c, Wk, m, q, S2, dsm, dsm + kRtK * kRtLd);
    for (long long e = tid; e < (long long)rows * q; e += kRoundThreads) Wp[e] = S2[e];
    __syncthreads();  // every thread has read rk[k]
    if (tid == 0) rk[k] = q;
    __syncthreads();
  }
  // 2. left-to-right truncated SVDs
  for (int k = 0; k + 1 < d; ++k) {
    const int r0 = rk[k], n = a.X.n[k], c = rk[k + 1];
    const int m = r0 * n;
    const bool rows_side = m <= c;  // eigen-decompose M M^T (else M^T M)
    const int s = rows_side ? m : c;
    const int p = min(a.maxr, s);
    double* Sg = dsm;
    const int lds = s | 1;
    double* Vg = Sg + s * lds;
    // M staged in shared memory (odd row stride) where it fits beside the eigenproblem
    const int ldm = c | 1;
    const bool staged = 2LL * s * lds + (long long)m * ldm <= kDynDoubles;
    double* Ms = Vg + s * lds;
    double* M = W + a.coff[k];
    if (staged) {
      for (int e = tid; e < m * c; e += kRoundThreads) Ms[(e / c) * ldm + e % c] = M[e];
      __syncthreads();
    }
    const double* Mr = staged ? Ms : M;
    const long long ld = staged ? ldm : c;
    for (int e = tid; e < s * s; e += kRoundThreads) {
      const int x = e / s, y = e % s;
      if (x > y) continue;
      double v = 0.0;
      if (rows_side)
        for (int b = 0; b < c; ++b) v = fma(Mr[x * ld + b], Mr[y * ld + b], v);
      else
        for (int row = 0; row < m; ++row) v = fma(Mr[row * ld + x], Mr[row * ld + y], v);
      Sg[x * lds + y] = v;
      Sg[y * lds + x] = v;
    }
    __syncthreads();
    jacobi_eig(Sg, Vg, s, lds, pp, pq, pc, ps, red, tri);
    // order by eigenvalue, largest first (ties by index)
    for (int j = tid; j < s; j += kRoundThreads) {
      const double lj = Sg[j * lds + j];
      int pos = 0;
      for (int l = 0; l < s; ++l) {
        const double ll = Sg[l * lds + l];
        pos += (ll > lj || (ll == lj && l < j)) ? 1 : 0;
      }
      perm[pos] = j;
    }
    __syncthreads();
    for (int j = tid; j < p; j += kRoundThreads) sig[j] = sqrt(fmax(Sg[perm[j] * lds + perm[j]], 0.0));
    __syncthreads();
    // U (m x p, row-major) in S1, S V^T (p x c, row-major) in S2
    for (long long e = tid; e < (long long)m * p; e += kRoundThreads) {
      const int x = (int)(e / p), j = (int)(e % p), col = perm[j];
      double u;
      if (rows_side) {
        u = Vg[x * lds + col];
      } else {
        double t = 0.0;
        for (int b = 0; b < c; ++b) t = fma(Mr[x * ld + b], Vg[b * lds + col], t);
        u = sig[j] > 0.0 ? t / sig[j] : 0.0;
      }
      S1[e] = u;
    }
    __syncthreads();
    for (long long e = tid; e < (long long)p * c; e += kRoundThreads) {
      const int j = (int)(e / c), b = (int)(e % c);
      double v;
      if (rows_side) {
        v = 0.0;
        for (int x = 0; x < m; ++x) v = fma(Vg[x * lds + perm[j]], Mr[x * ld + b], v);
      } else {
        v = sig[j] * Vg[b * lds + perm[j]];
      }
      S2[e] = v;
    }
    __syncthreads();
    // sign convention: the entry of largest magnitude of every kept column of U is positive
    for (int j = tid; j < p; j += kRoundThreads) {
      int best = 0;
      double bv = -1.0;
      for (int x = 0; x < m; ++x) {
        const double v = fabs(S1[(long long)x * p + j]);
        if (v > bv) {
          bv = v;
          best = x;
        }
      }
      sig[j] = S1[(long long)best * p + j] < 0.0 ? -1.0 : 1.0;
    }
    __syncthreads();
    for (long long e = tid; e < (long long)m * p; e += kRoundThreads) M[e] = S1[e] * sig[e % p];
    for (long long e = tid; e < (long long)p * c; e += kRoundThreads) S2[e] *= sig[e / c];
    __syncthreads();
    // W_{k+1} <- (S V^T) Q_{k+1}^T: p x (n_{k+1} r_{k+2})
    double* Wn = W + a.coff[k + 1];
    const int cols = a.X.n[k + 1] * rk[k + 2];
    apply_q(Wn, cols, c, S2, p, S1, sh_tau);
    __syncthreads();
    for (long long e = tid; e < (long long)p * cols; e += kRoundThreads) Wn[e] = S1[e];
    if (tid == 0) rk[k + 1] = p;
    __syncthreads();
  }
  // FP32 output with the final ranks
  float* Yp = static_cast<float*>(a.Y.p);
  for (int k = 0; k < d; ++k) {
    float* dst = Yp + core_base(a.Y, k, obj);
    for (long long e = tid; e < a.Y.osz[k]; e += blockDim.x) dst[e] = (float)W[a.coff[k] + e];
  }
}

struct RoundPlan {
  long long coff[T3F_MAX_D];
  long long maxcore, per_obj;
  size_t total;
};

RoundPlan round_plan(const TTV& X) {
  RoundPlan p;
  long long o = 0, mx = 1;
  for (int k = 0; k < X.d; ++k) {
    p.coff[k] = o;
    o += X.osz[k];
    mx = std::max(mx, X.osz[k]);
  }
  p.maxcore = mx;
  p.per_obj = o + 2 * mx;
  p.total = kWsHeader + align256(sizeof(double) * (size_t)p.per_obj * X.batch);
  return p;
}

void round_ranks_host(int d, const int* n, const int* ranks, int maxr, int* out, int* rr) {
  for (int k = 0; k <= d; ++k) rr[k] = ranks[k];
  for (int k = d - 1; k >= 1; --k) rr[k] = (int)std::min<long long>(rr[k], (long long)n[k] * rr[k + 1]);
  out[0] = 1;
  for (int k = 1; k < d; ++k)
    out[k] = (int)std::min<long long>(std::min<long long>((long long)out[k - 1] * n[k - 1], rr[k]), maxr);
  out[d] = 1;
}

}  // namespace

size_t ws_round(const TTV& X) { return round_plan(X).total; }

}  // namespace t3f

using namespace t3f;

extern "C" t3f_status t3f_round_ranks(int32_t d, const int32_t* n, const int32_t* ranks, int32_t max_rank,
                                      int32_t* out_ranks) {
  if (d < 1 || d > T3F_MAX_D || !n || !ranks || !out_ranks || max_rank < 1) return T3F_ERR_ARG;
  if (ranks[0] != 1 || ranks[d] != 1) return T3F_ERR_SHAPE;
  for (int k = 0; k <= d; ++k)
    if (ranks[k] < 1) return T3F_ERR_SHAPE;
  for (int k = 0; k < d; ++k)
    if (n[k] < 1) return T3F_ERR_SHAPE;
  int rr[T3F_MAX_D + 1];
  round_ranks_host(d, n, ranks, max_rank, out_ranks, rr);
  return T3F_OK;
}

extern "C" t3f_status t3f_round(const t3f_tt* X, int32_t max_rank, t3f_tt* Y, void* ws, size_t ws_bytes,
                                t3f_stream_t stream) {
  TTV vx, vy;
  T3F_CHECK(make_view(X, &vx, T3F_F32, false));
  T3F_CHECK(make_view(Y, &vy, T3F_F32, false));
  if (max_rank < 1) return T3F_ERR_ARG;
  if (vy.batch != vx.batch || vy.d != vx.d) return T3F_ERR_SHAPE;
  int want[T3F_MAX_D + 1], rr[T3F_MAX_D + 1];
  round_ranks_host(vx.d, vx.n, vx.r, max_rank, want, rr);
  for (int k = 0; k <= vx.d; ++k)
    if (vy.r[k] != want[k] || (k < vx.d && vy.n[k] != vx.n[k])) return T3F_ERR_SHAPE;
  // limits: the QR reflector count and every eigenproblem side
  for (int k = 1; k < vx.d; ++k)
    if (std::min<long long>((long long)vx.n[k] * rr[k + 1], vx.r[k]) > kMaxSide + T3F_MAX_RANK) return T3F_ERR_UNSUPPORTED;
  for (int k = 0; k + 1 < vx.d; ++k)
    if (std::min<long long>((long long)want[k] * vx.n[k], rr[k + 1]) > kMaxSide) return T3F_ERR_UNSUPPORTED;
  const RoundPlan p = round_plan(vx);
  T3F_CHECK(check_ws(ws, ws_bytes, p.total));
  cudaStream_t s = (cudaStream_t)stream;
  RoundArgs a;
  memset(&a, 0, sizeof(a));
  a.X = vx;
  a.Y = vy;
  a.maxr = max_rank;
  for (int k = 0; k < vx.d; ++k) a.coff[k] = p.coff[k];
  a.maxcore = p.maxcore;
  a.per_obj = p.per_obj;
  a.ws = reinterpret_cast<double*>(static_cast<char*>(ws) + kWsHeader);
  a.err = static_cast<int*>(ws);
  const size_t smem = sizeof(double) * kDynDoubles;
  if (cudaFuncSetAttribute(k_round, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  k_round<<<(unsigned)vx.batch, kRoundThreads, smem, s>>>(a);
  return launch_status();
}
