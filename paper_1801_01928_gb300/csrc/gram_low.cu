// Gram sweep and its adjoint for uniform batches of low rank (both ranks <= 16), FP32.
//
// A tile of na x nb pairs (a, b) keeps its r x r partials as the rows and columns of one matrix
// [(a, alpha)][(b, beta)], and every product of a sweep step is a row or a column of it times a
// core slice:
//   rows     T[(a, alpha)][(b, .)]  = M[(a, alpha)][(b, .)] B_b,i      Y, R' likewise with B_b,i^T
//   columns  M'[(a, .)][(b, beta')] += A_a,i^T T[(a, .)][(b, beta')]    X likewise with A_a,i
// so a lane owns rows (a, alpha) or columns (b, beta') in registers, R = the rank rounded up to
// even, compile time, and only the slice is read from shared memory, the same addresses for the
// R lanes of an object: no padding of 10 to 12 or 16, R multiply-adds per 16-byte read of
// four slice values, and one block barrier per slice, between the row and the column role (the
// matrix passes through shared memory there). Row role: warp a, lanes (b_sub, alpha); column
// role: warp b, lanes (a_sub, beta'); S = 32 / R sub-objects, two objects per lane. In the adjoint
//   column role  X = A_i R (kept for the row role),  dB_b,i = sum_a (g M)^T X
//   row role     R' += X B_i^T,  Y = R B_i^T,  dA_a,i = sum_b (g M) Y^T
// a lane sums dB (dA) over its objects, the S sub-objects meet by shuffles and one atomic per
// element and tile goes to the gradient. The left partials of every interface go through a scratch
// area per tile (t R x t RP floats each, R of the larger rank on both sides: as much as the 4 x 4 block
// kernels' on equal sides, ranks 6 and 4 48 floats a pair and interface instead of 32).
//
// 100 x 100 pairs, d = 10, n = 10, r = 10: forward 388 us with 4 x 4 blocks on padded ranks (three
// barriers per slice) -> 203 us, adjoint 1826 -> 783 us. Bound by the issue of the two or three warps a
// scheduler holds (48 % of slots, FMA pipe 28 %): 17 x 17 tiles of 6 warps are 1.9 blocks per SM.
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "t3f_internal.cuh"

namespace t3f {

namespace {

template <int R>
struct Low {
  static constexpr int RP = (R + 3) & ~3;          // stored columns of a row
  static constexpr int S = 32 / R;                 // sub-objects of a warp
  static constexpr int O = 2;                      // objects of a lane
  static constexpr int W = O * S;                  // most objects a side, and warps
  static constexpr int P = ((W * RP) & 7) == 4 ? W * RP : W * RP + 4;  // row stride (odd multiple of 4)
  static constexpr int MAT = W * R * P;            // floats of a pair matrix
  static constexpr int OS = R * RP + 4;            // floats of a staged slice
  static constexpr int RING = 3;
  static constexpr size_t smem = sizeof(float) * (3 * (size_t)MAT + RING * 2 * W * OS + W * W);
  static_assert(smem <= 227 * 1024 && 32 * W <= 1024, "one block must fit");
};

struct GramLowArgs {
  TTV A, B;
  int t;                 // objects a side of a tile
  int cut;               // forward: padded ranks run with the row test
  float* out;            // forward
  const float* dG;       // adjoint
  float* dA;
  float* dB;
  float* scratch;        // adjoint: [CTA][interface 0 .. d - 1][t R rows][t RP]
};

template <int R>
__device__ __forceinline__ void ld_row(float (&v)[R], const float* p) {
#pragma unroll
  for (int q = 0; q + 4 <= R; q += 4) {
    const float4 f = *reinterpret_cast<const float4*>(p + q);
    v[q] = f.x;
    v[q + 1] = f.y;
    v[q + 2] = f.z;
    v[q + 3] = f.w;
  }
  if (R & 2) {
    const float2 f = *reinterpret_cast<const float2*>(p + (R & ~3));
    v[R - 2] = f.x;
    v[R - 1] = f.y;
  }
}

template <int R>
__device__ __forceinline__ void st_row(float* p, const float (&v)[R]) {
#pragma unroll
  for (int q = 0; q + 4 <= R; q += 4) *reinterpret_cast<float4*>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  if (R & 2) *reinterpret_cast<float2*>(p + (R & ~3)) = make_float2(v[R - 2], v[R - 1]);
}

template <int R>
__device__ __forceinline__ float dot_row(const float (&a)[R], const float (&b)[R]) {
  float s = a[0] * b[0], t = a[1] * b[1];  // two chains
#pragma unroll
  for (int q = 2; q < R; q += 2) {
    s = fmaf(a[q], b[q], s);
    t = fmaf(a[q + 1], b[q + 1], t);
  }
  return s + t;
}

// The slices of one tile: a ring of three, filled by 4-byte asynchronous copies, zero outside the
// ranks. Slices are counted along the sweep (dir = 0: cores ascending, 1: descending). Warp w copies
// its A and its B object; a lane's element offsets within a slice change with the core only.
template <int R>
struct LowSlices {
  static constexpr int NJ = (R * Low<R>::RP + 31) / 32;
  float* ring;
  int a0, b0, na, nb;
  int k, i, cnt;  // next slice to issue, its running number
  int n;          // modes of core k
  const float *pa, *pb;    // this warp's objects, core k, the next slice
  int oa[NJ], ob[NJ];      // element offsets, -1 outside the ranks
  __device__ void core(const GramLowArgs& g) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    n = g.A.n[k];
    pa = static_cast<const float*>(g.A.p) + core_base(g.A, k, a0 + min(w, na - 1));
    pb = static_cast<const float*>(g.B.p) + core_base(g.B, k, b0 + min(w, nb - 1));
    const int ra0 = g.A.r[k], ra1 = g.A.r[k + 1], rb0 = g.B.r[k], rb1 = g.B.r[k + 1];
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int e = lane + 32 * j, row = e / Low<R>::RP, col = e % Low<R>::RP;
      oa[j] = row < ra0 && col < ra1 ? row * n * ra1 + col : -1;
      ob[j] = row < rb0 && col < rb1 ? row * n * rb1 + col : -1;
    }
  }
  __device__ void start(const GramLowArgs& g, int kfirst, int kend) {
    k = kfirst;
    i = cnt = 0;
    if (k != kend) core(g);
  }
  __device__ __forceinline__ void issue(const GramLowArgs& g, int dir, int kend) {
    using L = Low<R>;
    if (k != kend) {
      const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
      float* bufa = ring + (cnt % L::RING) * 2 * L::W * L::OS + w * L::OS;
      const unsigned sa = (unsigned)__cvta_generic_to_shared(bufa) + 4 * lane, sb = sa + 4 * L::W * L::OS;
      if (w < na)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          if (lane + 32 * j < R * L::RP)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa + 128 * j), "l"(pa + max(oa[j], 0)),
                         "r"(oa[j] >= 0 ? 4 : 0));
      if (w < nb)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          if (lane + 32 * j < R * L::RP)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sb + 128 * j), "l"(pb + max(ob[j], 0)),
                         "r"(ob[j] >= 0 ? 4 : 0));
      pa += g.A.r[k + 1];
      pb += g.B.r[k + 1];
      if (++i >= n) {
        i = 0;
        k += dir ? -1 : 1;
        if (k != kend) core(g);
      }
    }
    ++cnt;
    asm volatile("cp.async.commit_group;\n" ::);
  }
};

// How a core's ranks lie to R. kExact: all R (those that a product sums over). kPadded: they come up to R
// when padded to four, and its rows are run without a test (the operands are zero there), which lets
// their loads run ahead. kCut: row al runs where the core has it. Zero on both sides: a partial is cut
// to its core's ranks (keep) wherever it passes on to the next role or core, since an infinity in a
// padded row or column meets a zero of the slice there and would reach the real ones as NaN (a pair
// that overflows FP32 before its last core is +-inf). Bits are masked instead of selected: the products
// were branched around behind a select (adjoint of 100 x 100 pairs of rank 9 1201 us, with masks 797,
// without either 784; forward 201 against 199, rank 7 95 against 82).
enum { kCut, kPadded, kExact };

template <int R, class F>
__device__ __forceinline__ void by_ranks(int lo, bool cut, F f) {
  if (lo == R) f(std::integral_constant<int, kExact>());
  else if (((lo + 3) & ~3) >= R && !cut) f(std::integral_constant<int, kPadded>());
  else f(std::integral_constant<int, kCut>());
}
template <int MODE>
__device__ __forceinline__ bool row_on(int al, int e) {
  return MODE != kCut || al < e;
}
template <int MODE = kPadded>
__device__ __forceinline__ float keep(float v, bool real) {
  return MODE == kPadded ? __uint_as_float(__float_as_uint(v) & (real ? 0xffffffffu : 0u)) : v;
}

// Left sweep over cores 0 .. kend - 1. On return acc holds the column role's last partial (of interface
// kend). With `scr`, the partials of interfaces 1 .. kend go there (interface 0 is the caller's).
template <int R, bool SAVE>
__device__ void low_left(const GramLowArgs& g, float* sm, int a0, int na, int b0, int nb, int kend, float* scr,
                         float (&acc)[Low<R>::O][R]) {
  using L = Low<R>;
  constexpr int P = L::P, RP = L::RP, S = L::S;
  float* Ms = sm;
  float* Ts = Ms + L::MAT;  // two buffers
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane / R, x = lane % R;
  const bool on = sub < S;
  LowSlices<R> sl;
  sl.ring = Ts + 2 * L::MAT;
  sl.a0 = a0;
  sl.b0 = b0;
  sl.na = na;
  sl.nb = nb;
  sl.start(g, 0, kend);
  sl.issue(g, 0, kend);
  sl.issue(g, 0, kend);
  float m[Low<R>::O][R];
#pragma unroll
  for (int o = 0; o < Low<R>::O; ++o)
#pragma unroll
    for (int q = 0; q < R; ++q) m[o][q] = x == 0 && q == 0 ? 1.0f : 0.0f;
  asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  __syncthreads();
  int c = 0;  // running slice
  for (int k = 0; k < kend; ++k) {
    const int n = g.A.n[k], eA0 = g.A.r[k], eA1 = g.A.r[k + 1], eB0 = g.B.r[k], eB1 = g.B.r[k + 1];
#pragma unroll
    for (int o = 0; o < Low<R>::O; ++o)
#pragma unroll
      for (int q = 0; q < R; ++q) acc[o][q] = 0.0f;
    auto slices = [&](auto mode) {
      constexpr int MODE = decltype(mode)::value;
      for (int i = 0; i < n; ++i, ++c) {
        const float* As = sl.ring + (c % L::RING) * 2 * L::W * L::OS;
        const float* Bs = As + L::W * L::OS;
        float* T = Ts + (c & 1) * L::MAT;
        // row role: a = w, alpha = x
        if (on && w < na && row_on<MODE>(x, eA0))
#pragma unroll
          for (int o = 0; o < Low<R>::O; ++o) {
            const int b = sub + o * S;
            if (b >= nb) continue;
            float t[R], br[R];
            const float* Bb = Bs + b * L::OS;
#pragma unroll
            for (int q = 0; q < R; ++q) t[q] = 0.0f;
#pragma unroll
            for (int be = 0; be < R; ++be)
              if (row_on<MODE>(be, eB0)) {
                ld_row<R>(br, Bb + be * RP);
#pragma unroll
                for (int q = 0; q < R; ++q) t[q] = fmaf(m[o][be], br[q], t[q]);
              }
#pragma unroll
            for (int q = 0; q < R; ++q) t[q] = keep<MODE>(t[q], x < eA0);
            st_row<R>(T + (w * R + x) * P + b * RP, t);
          }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();  // T complete; slice c + 1 has landed; the column role of slice c - 1 is done
        sl.issue(g, 0, kend);
        // column role: b = w, beta' = x
        if (on && w < nb)
#pragma unroll
          for (int o = 0; o < Low<R>::O; ++o) {
            const int a = sub + o * S;
            if (a >= na) continue;
            const float* Aa = As + a * L::OS;
            const float* tc = T + a * R * P + w * RP + x;
#pragma unroll
            for (int al = 0; al < R; ++al)
              if (row_on<MODE>(al, eA0)) {
                float ar[R];
                const float tv = tc[al * P];
                ld_row<R>(ar, Aa + al * RP);
#pragma unroll
                for (int q = 0; q < R; ++q) acc[o][q] = fmaf(ar[q], tv, acc[o][q]);
              }
          }
      }
    };
    by_ranks<R>(min(eA0, eB0), g.cut, slices);
    if (k + 1 == kend && !SAVE) break;
    // the columns of M' become the rows of the next core's M
    if (on && w < nb)
#pragma unroll
      for (int o = 0; o < Low<R>::O; ++o) {
        const int a = sub + o * S;
        if (a >= na) continue;
#pragma unroll
        for (int q = 0; q < R; ++q) Ms[(a * R + q) * P + w * RP + x] = acc[o][q];
      }
    __syncthreads();
    if (on && w < na)
#pragma unroll
      for (int o = 0; o < Low<R>::O; ++o) {
        const int b = sub + o * S;
        if (b >= nb) continue;
        ld_row<R>(m[o], Ms + (w * R + x) * P + b * RP);
#pragma unroll
        for (int q = 0; q < R; ++q) m[o][q] = keep(m[o][q], x < eA1 && q < eB1);
        if (SAVE) st_row<R>(scr + ((size_t)(k + 1) * g.t * R + w * R + x) * (g.t * RP) + b * RP, m[o]);
      }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Blocks an SM to leave registers for. Forward us with 1, 2, 3: R = 6, 40 x 40 pairs (d = 6, n = 10) 33, 35, 44
// and 350 x 350 (d = 5, n = 8) 338, 266, 282; R = 14, 40 x 40 86, -, 90 and 350 x 350 2143, -, 1920 (2112 with 4).
// Left to the compiler R = 8 had 80 registers for three blocks (100 x 100 of rank 7, d = 6, n = 10: 95, now 80) and
// R = 16 168 (471, now 408).
template <int R>
__global__ void __launch_bounds__(32 * Low<R>::W, R <= 8 ? 2 : R == 14 ? 3 : 1) k_gram_low(const __grid_constant__ GramLowArgs g) {
  extern __shared__ __align__(16) float sm[];
  const int ntb = (g.B.batch + g.t - 1) / g.t;
  const int a0 = (blockIdx.x / ntb) * g.t, b0 = (blockIdx.x % ntb) * g.t;
  const int na = min(g.t, g.A.batch - a0), nb = min(g.t, g.B.batch - b0);
  float acc[Low<R>::O][R];
  low_left<R, false>(g, sm, a0, na, b0, nb, g.A.d, nullptr, acc);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane / R, x = lane % R;
  if (sub < Low<R>::S && x == 0 && w < nb)
#pragma unroll
    for (int o = 0; o < Low<R>::O; ++o) {
      const int a = sub + o * Low<R>::S;
      if (a < na) g.out[(long long)(a0 + a) * g.B.batch + b0 + w] = acc[o][0];
    }
}

// Sum of the lanes of equal index within their object (lanes s R + x), complete in the lanes < R.
template <int R>
__device__ __forceinline__ float sum_subs(float v) {
  float s = v;
#pragma unroll
  for (int q = 1; q < Low<R>::S; ++q) s += __shfl_down_sync(0xffffffffu, v, q * R);
  return s;
}

template <int R>
__global__ void __launch_bounds__(32 * Low<R>::W, Low<R>::W <= 8 ? 2 : 1) k_gram_low_bwd(const __grid_constant__ GramLowArgs g) {
  extern __shared__ __align__(16) float sm[];
  using L = Low<R>;
  constexpr int P = L::P, RP = L::RP, S = L::S;
  float* Ms = sm;                 // g M of the current core
  float* Xs = Ms + L::MAT;        // two buffers (T of the left sweep)
  float* gs = Xs + 2 * L::MAT + L::RING * 2 * L::W * L::OS;  // cotangents [a][b]
  float* scr = g.scratch + (size_t)blockIdx.x * g.A.d * (g.t * R) * (g.t * RP);
  const int ntb = (g.B.batch + g.t - 1) / g.t;
  const int a0 = (blockIdx.x / ntb) * g.t, b0 = (blockIdx.x % ntb) * g.t;
  const int na = min(g.t, g.A.batch - a0), nb = min(g.t, g.B.batch - b0);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, sub = lane / R, x = lane % R, d = g.A.d;
  const bool on = sub < S;
  for (int p = tid; p < na * nb; p += blockDim.x)
    gs[p] = g.dG[(long long)(a0 + p / nb) * g.B.batch + b0 + p % nb];
  {
    float acc[Low<R>::O][R];
    low_left<R, true>(g, sm, a0, na, b0, nb, d - 1, scr, acc);
  }
  // R of interface d: rows (a = w, x; b) and columns (b = w, x; a)
  float rrow[Low<R>::O][R], rcol[Low<R>::O][R], racc[Low<R>::O][R];
#pragma unroll
  for (int o = 0; o < Low<R>::O; ++o)
#pragma unroll
    for (int q = 0; q < R; ++q) {
      rrow[o][q] = x == 0 && q == 0 ? 1.0f : 0.0f;
      rcol[o][q] = rrow[o][q];
    }
  LowSlices<R> sl;
  sl.ring = Xs + 2 * L::MAT;
  sl.a0 = a0;
  sl.b0 = b0;
  sl.na = na;
  sl.nb = nb;
  sl.start(g, d - 1, -1);
  __syncthreads();  // the left sweep is done with the ring
  sl.issue(g, 1, -1);
  sl.issue(g, 1, -1);
  int c = 0;
  for (int k = d - 1; k >= 0; --k) {
    const int n = g.A.n[k];
    const int eA0 = g.A.r[k], eA1 = g.A.r[k + 1], eB0 = g.B.r[k], eB1 = g.B.r[k + 1];
    // g M at interface k
    for (int e = tid; e < na * R * nb * RP; e += blockDim.x) {
      const int col = e % (nb * RP), row = e / (nb * RP), q = col % RP;
      float v = 0.0f;
      if (q < R) v = k == 0 ? 1.0f : scr[((size_t)k * g.t * R + row) * (g.t * RP) + col];
      Ms[row * P + col] = keep(gs[(row / R) * nb + col / RP] * v, q < eB0 && row % R < eA0);
    }
#pragma unroll
    for (int o = 0; o < Low<R>::O; ++o)
#pragma unroll
      for (int q = 0; q < R; ++q) racc[o][q] = 0.0f;
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();  // M complete, slice c has landed
    auto slices = [&](auto mode) {
      constexpr int MODE = decltype(mode)::value;
      for (int i = 0; i < n; ++i, ++c) {
        const float* As = sl.ring + (c % L::RING) * 2 * L::W * L::OS;
        const float* Bs = As + L::W * L::OS;
        float* X = Xs + (c & 1) * L::MAT;
        // column role: b = w, beta' = x
        float grad[R];
#pragma unroll
        for (int q = 0; q < R; ++q) grad[q] = 0.0f;
        if (on && w < nb && row_on<MODE>(x, eB1))
#pragma unroll
          for (int o = 0; o < Low<R>::O; ++o) {
            const int a = sub + o * S;
            if (a >= na) continue;
            const float* Aa = As + a * L::OS;
            float* xc = X + a * R * P + w * RP + x;
            const float* mr = Ms + a * R * P + w * RP;
#pragma unroll
            for (int al = 0; al < R; ++al)
              if (row_on<MODE>(al, eA0)) {
                float ar[R], mv[R];
                ld_row<R>(ar, Aa + al * RP);
                ld_row<R>(mv, mr + al * P);
                const float xv = keep<MODE>(dot_row<R>(ar, rcol[o]), al < eA0 && x < eB1);
                xc[al * P] = xv;
#pragma unroll
                for (int q = 0; q < R; ++q) grad[q] = fmaf(mv[q], xv, grad[q]);
              }
          }
        if (g.dB && w < nb) {
          float* dst = g.dB + core_base(g.B, k, b0 + w) + (long long)i * eB1 + x;
          const int step = n * eB1;
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (q < eB0) {
              const float v = sum_subs<R>(on ? grad[q] : 0.0f);
              if (lane < R && x < eB1) atomicAdd(dst + q * step, v);
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();  // X complete; slice c + 1 has landed; the row role of slice c - 1 is done
        sl.issue(g, 1, -1);
        // row role: a = w, alpha (alpha') = x
#pragma unroll
        for (int q = 0; q < R; ++q) grad[q] = 0.0f;
        if (on && w < na)
#pragma unroll
          for (int o = 0; o < Low<R>::O; ++o) {
            const int b = sub + o * S;
            if (b >= nb) continue;
            const float* Bb = Bs + b * L::OS;
            float xr[R], y[R];
            ld_row<R>(xr, X + (w * R + x) * P + b * RP);
            if (MODE == kCut) {  // rows and columns past the ranks were not written
#pragma unroll
              for (int q = 0; q < R; ++q) xr[q] = x < eA0 && q < eB1 ? xr[q] : 0.0f;
            }
#pragma unroll
            for (int be = 0; be < R; ++be) {
              y[be] = 0.0f;
              if (row_on<MODE>(be, eB0)) {
                float br[R];
                ld_row<R>(br, Bb + be * RP);
                racc[o][be] += dot_row<R>(br, xr);
                y[be] = keep<MODE>(dot_row<R>(br, rrow[o]), be < eB0);
              }
            }
            const float* mr = Ms + w * R * P + b * RP;
#pragma unroll
            for (int al = 0; al < R; ++al)
              if (row_on<MODE>(al, eA0)) {
                float mv[R];
                ld_row<R>(mv, mr + al * P);
                grad[al] += dot_row<R>(mv, y);
              }
          }
        if (g.dA && w < na) {
          float* dst = g.dA + core_base(g.A, k, a0 + w) + (long long)i * eA1 + x;
          const int step = n * eA1;
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (q < eA0) {
              const float v = sum_subs<R>(on ? grad[q] : 0.0f);
              if (lane < R && x < eA1) atomicAdd(dst + q * step, v);
            }
        }
      }
    };
    by_ranks<R>(min(min(eA0, eA1), min(eB0, eB1)), false, slices);
    if (k == 0) break;
    // R' : rows to columns through the X buffer that the last slice did not use
    float* Rs = Xs + (c & 1) * L::MAT;
    if (on && w < na)
#pragma unroll
      for (int o = 0; o < Low<R>::O; ++o) {
        const int b = sub + o * S;
#pragma unroll
        for (int q = 0; q < R; ++q) rrow[o][q] = keep(racc[o][q], x < eA0 && q < eB0);
        if (b < nb) st_row<R>(Rs + (w * R + x) * P + b * RP, rrow[o]);
      }
    __syncthreads();  // (also: every read of M is done)
    if (on && w < nb)
#pragma unroll
      for (int o = 0; o < Low<R>::O; ++o) {
        const int a = sub + o * S;
        if (a >= na) continue;
#pragma unroll
        for (int q = 0; q < R; ++q) rcol[o][q] = Rs[(a * R + q) * P + w * RP + x];
      }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Objects a side of a tile, t: the t warps of a tile run o = ceil(t / S) objects a lane, and the
// busiest SM has c of the tiles. c (t o + 3) + 2 o follows the measured times of both kernels to a
// fifth over t = 1 .. W, ranks 4 .. 16 and batches of 8 x 9 .. 128 x 128 (3: a tile's staging and
// barriers in units of a warp's object, 2: latency of a lane's chain).
template <int R>
int low_tile(const TTV& A, const TTV& B) {
  const int sms = device_sm_count();
  int best = 1;
  long long cost = -1;
  for (int t = 1; t <= Low<R>::W; ++t) {
    const long long tiles = (long long)((A.batch + t - 1) / t) * ((B.batch + t - 1) / t), o = (t + Low<R>::S - 1) / Low<R>::S;
    const long long v = (tiles + sms - 1) / sms * (t * o + 3) + 2 * o;
    if (cost < 0 || v <= cost) {
      cost = v;
      best = t;
    }
  }
  return best;
}

template <class F>
auto low_dispatch(const TTV& A, const TTV& B, F f) {
  const int r = std::max(A.rmax, B.rmax);
  if (r <= 4) return f(std::integral_constant<int, 4>());
  if (r <= 6) return f(std::integral_constant<int, 6>());
  if (r <= 8) return f(std::integral_constant<int, 8>());
  if (r <= 10) return f(std::integral_constant<int, 10>());
  if (r <= 12) return f(std::integral_constant<int, 12>());
  if (r <= 14) return f(std::integral_constant<int, 14>());
  return f(std::integral_constant<int, 16>());
}

}  // namespace

// FP32 storage and ranks that fill most of R, where these kernels were the faster ones (us, this
// file against the 4 x 4 block kernels; n modes a core, d cores):
//   largest rank 1 .. 10, the sides within a half of one another (a side of 6 against 10 gains
//   nothing at all; up to rank 4 every pair of ranks): forward 34 .. 208 against 90 .. 401 and adjoint
//   92 .. 821 against 250 .. 1856 over batches of 8 x 9 .. 128 x 128, 1.1 to 4.2 times as fast. Forward of
//   many pairs of ranks 1 and 2 (d = 10, n = 10): 200 x 200 115 against 148, 350 x 350 247 against 225, 500 x
//   500 445 against 421, 800 x 800 1062 against 1198, so not from 500 to 3000 pairs an SM; ranks 5 and 4 (d = 5, n = 8): 150 x
//   150 60 against 82, 250 x 250 156 against 123, 350 x 350 265 against 238, 500 x 500 488 against 545, so not
//   from 200 to 1500;
//   11 and 12, forward only and up to 46 pairs an SM: 80 x 80 138 against 172, but 90 x 90 of ranks 12 and 9 177
//   against 168, 128 x 128 with n = 16, d = 4 311 against 290 (two objects of 12 rows a warp); the adjoint 966
//   against 927 at 96 x 104;
//   13 .. 16, both sides: forward 92 .. 802 against 283 .. 1068, except many pairs whose inner cores are of
//   lower rank (61 x 304 of ranks 1 to 15 727 against 619; 24 x 5 of ranks 3 to 16 148 against 294). The
//   adjoint's three sets of rows take all registers, 551 against 424 on 8 x 9 pairs and 952 against 789 on
//   25 x 56, but 552 against 919 on 64 x 64 and 2487 against 3304 on 128 x 128, so from 4096 pairs on, and
//   only where no inner core is of much lower rank (1-4-16-16-16-4-1, 100 x 100: 790 against 727).
static bool low_ranks(const TTV& A, const TTV& B) {
  const int hi = std::max(A.rmax, B.rmax), lo = std::min(A.rmax, B.rmax);
  if (A.dtype != T3F_F32 || B.dtype != T3F_F32 || hi > 16) return false;
  for (int k = 0; k < A.d; ++k)  // offsets within a core are 32-bit here
    if ((long long)hi * hi * A.n[k] > 0x7fffffffLL) return false;
  if (hi <= 4) return true;
  return hi <= 10 ? 3 * lo >= 2 * hi : ((lo + 3) & ~3) >= hi;
}

// Every inner core of the ranks that only R = 14 and 16 hold.
static bool inner_full(const TTV& A, const TTV& B) {
  for (int k = 1; k < A.d; ++k)
    if (std::min(A.r[k], B.r[k]) <= 12) return false;
  return true;
}

bool gram_low_supported(const TTV& A, const TTV& B) {
  if (!low_ranks(A, B)) return false;
  const int hi = std::max(A.rmax, B.rmax), lo = std::min(A.rmax, B.rmax);
  const long long pairs = (long long)A.batch * B.batch, sms = device_sm_count();
  if (hi <= 2) return pairs <= 500 * sms || pairs >= 3000 * sms;
  if (hi <= 6 && hi > 4 && lo <= 4) return pairs <= 200 * sms || pairs >= 1500 * sms;
  if (hi <= 10) return true;
  if (hi <= 12) return pairs <= 46 * sms;
  return pairs <= 64 * sms || inner_full(A, B);
}

bool gram_low_bwd_supported(const TTV& A, const TTV& B) {
  if (!low_ranks(A, B)) return false;
  const int hi = std::max(A.rmax, B.rmax);
  if (hi <= 10) return true;
  return hi > 12 && (long long)A.batch * B.batch >= 4096 && inner_full(A, B);
}

size_t ws_gram_low_bwd(const TTV& A, const TTV& B) {
  return low_dispatch(A, B, [&](auto rc) -> size_t {
    constexpr int R = decltype(rc)::value;
    const int t = low_tile<R>(A, B);
    const long long tiles = (long long)((A.batch + t - 1) / t) * ((B.batch + t - 1) / t);
    return kWsHeader + align256(sizeof(float) * (size_t)tiles * A.d * (t * R) * (t * Low<R>::RP));
  });
}

template <int R, class K>
static t3f_status launch_low(K kern, GramLowArgs& g, cudaStream_t s) {
  g.t = low_tile<R>(g.A, g.B);
  // Many pairs of ranks 1 to 3 (R = 4): the additions for padding count, not the loads' latency (padded
  // against cut, ranks 2, d = 10, n = 10, us: 100 x 100 47.6, 49.7; 200 x 200 123, 115; 500 x 500 538, 445).
  g.cut = R == 4 && (long long)g.A.batch * g.B.batch > 150LL * device_sm_count();
  const long long tiles = (long long)((g.A.batch + g.t - 1) / g.t) * ((g.B.batch + g.t - 1) / g.t);
  if (tiles > 0x7fffffff) return T3F_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Low<R>::smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<(unsigned)tiles, 32 * g.t, Low<R>::smem, s>>>(g);
  return launch_status();
}

t3f_status run_gram_low(const TTV& A, const TTV& B, float* out, cudaStream_t s) {
  GramLowArgs g;
  memset(&g, 0, sizeof(g));
  g.A = A;
  g.B = B;
  g.out = out;
  return low_dispatch(A, B, [&](auto rc) -> t3f_status {
    constexpr int R = decltype(rc)::value;
    return launch_low<R>(k_gram_low<R>, g, s);
  });
}

t3f_status run_gram_low_bwd(const TTV& A, const TTV& B, const float* dG, float* dA, float* dB, void* ws, size_t ws_bytes,
                            cudaStream_t s) {
  T3F_CHECK(check_ws(ws, ws_bytes, ws_gram_low_bwd(A, B)));
  GramLowArgs g;
  memset(&g, 0, sizeof(g));
  g.A = A;
  g.B = B;
  g.dG = dG;
  g.dA = dA;
  g.dB = dB;
  g.scratch = reinterpret_cast<float*>(static_cast<char*>(ws) + kWsHeader);
  return low_dispatch(A, B, [&](auto rc) -> t3f_status {
    constexpr int R = decltype(rc)::value;
    if constexpr (R == 12) return T3F_ERR_UNSUPPORTED;  // (gram_low_bwd_supported takes no rank of 11 or 12)
    else return launch_low<R>(k_gram_low_bwd<R>, g, s);
  });
}

}  // namespace t3f
