// Element gather, completion loss and its adjoint (paper Section 1's completion example;
// Section 3.2's Riemannian gradient of that loss).
//
// For a tuple t with indices i_{t,1..d}:
//   prefix  l_{t,0} = 1,          l_{t,k} = l_{t,k-1} G^k[:, i_{t,k}, :]
//   suffix  rho_{t,d+1} = 1,      rho_{t,k} = G^k[:, i_{t,k}, :] rho_{t,k+1}
//   X(i_t) = l_{t,d} = rho_{t,1}
//   cotangent of sum_t w_t X(i_t):  dG^k[:, i, :] = sum_{t: i_{t,k} = i} w_t l_{t,k-1} rho_{t,k+1}^T
// One thread owns one tuple. The cores are staged in shared memory as zero-padded R x R
// mode slices, so the chains run fully unrolled in registers. The adjoint stores the
// suffix vectors of its tuple in shared memory, evaluates the residual, then walks the
// prefix and scatters the outer products into a per-CTA shared accumulator; a second
// kernel reduces the per-CTA partials in a fixed order.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "t3f_internal.cuh"

namespace t3f {

constexpr int kGatherThreads = 128;

struct GatherArgs {
  int d;
  long long N;
  int nmax;
  int rl[T3F_MAX_D + 1];     // ranks of the prefix cores (X or U)
  int rr[T3F_MAX_D + 1];     // ranks of the suffix cores (X or V)
  int n[T3F_MAX_D];
  const float* L;            // prefix cores, packed, batch 1
  long long Loff[T3F_MAX_D];
  const float* Rg;           // suffix cores, packed, batch 1
  long long Roff[T3F_MAX_D];
  long long Lnfl, Rnfl;      // floats of the packed prefix / suffix object
  int same;                  // L and R are the same cores
  const int* idx;            // [d][N]
  const float* y;            // nullable
  const float* w;            // nullable
  float* vals;               // nullable
  double* loss_part;         // [gridDim.x] nullable
  float* grad_part;          // [gridDim.x][gsize] nullable
  long long goff[T3F_MAX_D]; // compact per-core offsets of the gradient (r^L_k x n_k x r^R_{k+1})
  long long gsize;
  int* err;                  // device error word
};

// ---- whole-object staging through the TMA unit -------------------------------------------
// One cp.async.bulk copies the packed cores of a batch-1 TT (rounded out to 16-byte
// boundaries: the copy may start up to 12 bytes before the object and end up to 15 bytes
// after it, always inside the same 16-byte block, hence the same page) into a landing zone
// of shared memory; stage_from_raw then lays the slices out on chip. The landing zone is
// the first core rounded down by delta floats: raw[delta + element offset].

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > (1ll << 31)) return false;  // about one second
  }
}

__device__ __forceinline__ void bar_init(uint64_t* bar) {
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

__host__ __device__ __forceinline__ uint32_t raw_bytes(const float* src, long long nfl) {
  const uintptr_t s = reinterpret_cast<uintptr_t>(src);
  return (uint32_t)(((s & 15) + (uintptr_t)nfl * 4 + 15) & ~uintptr_t(15));
}

__device__ __forceinline__ int raw_delta(const float* src) { return (int)((reinterpret_cast<uintptr_t>(src) & 15) >> 2); }

// thread 0: one bulk copy of [src, src + nfl) (rounded out) into raw, completing on bar
__device__ __forceinline__ void tma_copy(float* raw, const float* src, long long nfl, uint64_t* bar) {
  const uintptr_t s0 = reinterpret_cast<uintptr_t>(src) & ~uintptr_t(15);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(raw)),
               "l"(s0), "r"(raw_bytes(src, nfl)), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tma_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// zero-padded R x R slices with slice stride SS from the landed object
template <int R>
__device__ __forceinline__ void stage_from_raw(float* dst, int SS, const float* raw, const long long* off,
                                               const int* r, const int* n, int d, int nmax) {
  const int total = d * nmax * SS;
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int q = e % SS, i = (e / SS) % nmax, k = e / (SS * nmax);
    const int a = q / R, b = q % R;
    float v = 0.0f;
    if (q < R * R && i < n[k] && a < r[k] && b < r[k + 1]) v = raw[off[k] + ((long long)a * n[k] + i) * r[k + 1] + b];
    dst[e] = v;
  }
}

// land one object and stage it (every thread; bar used at `parity`); false on a timeout
template <int R>
__device__ bool stage_object_tma(float* dst, int SS, float* landing, const float* src, long long nfl,
                                 const long long* off, const int* r, const int* n, int d, int nmax, uint64_t* bar,
                                 uint32_t parity) {
  if (threadIdx.x == 0) {
    tma_expect(bar, raw_bytes(src, nfl));
    tma_copy(landing, src, nfl, bar);
  }
  const bool ok = bar_wait(smem_u32(bar), parity);
  stage_from_raw<R>(dst, SS, landing + raw_delta(src), off, r, n, d, nmax);
  return ok;
}

__device__ __forceinline__ int load_index(const GatherArgs& g, int k, long long t) {
  int i = __ldg(g.idx + (long long)k * g.N + t);
  if (i < 0 || i >= g.n[k]) {
    atomicExch(g.err, (int)T3F_ERR_ARG);
    i = i < 0 ? 0 : g.n[k] - 1;
  }
  return i;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  __syncthreads();
  return s;
}

// Forward: values and / or loss partials.
template <int R>
__global__ void __launch_bounds__(kGatherThreads) k_gather_fwd(const __grid_constant__ GatherArgs g) {
  extern __shared__ __align__(16) float sm[];
  __shared__ double red[kGatherThreads / 32];
  __shared__ __align__(8) uint64_t bar;
  float* Ls = sm;
  // slices R^2 + 4 floats apart: the random slice indices of a warp's tuples fall on
  // different banks
  constexpr int SS = R * R + 4;
  float* landing = sm + g.d * g.nmax * SS;  // 16-byte aligned (SS is a multiple of 4)
  bar_init(&bar);
  if (!stage_object_tma<R>(Ls, SS, landing, g.L, g.Lnfl, g.Loff, g.rl, g.n, g.d, g.nmax, &bar, 0u) &&
      threadIdx.x == 0)
    atomicExch(g.err, (int)T3F_ERR_TIMEOUT);
  __syncthreads();
  double lsum = 0.0;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < g.N;
       t += (long long)gridDim.x * blockDim.x) {
    float l[R];
#pragma unroll
    for (int a = 0; a < R; ++a) l[a] = a == 0 ? 1.0f : 0.0f;
    for (int k = 0; k < g.d; ++k) {
      const int i = load_index(g, k, t);
      const float* S = Ls + (k * g.nmax + i) * SS;
      float nl[R];
#pragma unroll
      for (int b = 0; b < R; ++b) nl[b] = 0.0f;
#pragma unroll
      for (int a = 0; a < R; ++a) {
#pragma unroll
        for (int b = 0; b < R; b += 4) {
          const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
          nl[b] = fmaf(l[a], s4.x, nl[b]);
          nl[b + 1] = fmaf(l[a], s4.y, nl[b + 1]);
          nl[b + 2] = fmaf(l[a], s4.z, nl[b + 2]);
          nl[b + 3] = fmaf(l[a], s4.w, nl[b + 3]);
        }
      }
#pragma unroll
      for (int b = 0; b < R; ++b) l[b] = nl[b];
    }
    const float x = l[0];
    if (g.vals) g.vals[t] = x;
    if (g.loss_part) {
      const double res = (double)x - (double)g.y[t];
      lsum += 0.5 * res * res;
    }
  }
  if (g.loss_part) {
    const double s = block_sum(lsum, red);
    if (threadIdx.x == 0) g.loss_part[blockIdx.x] = s;
  }
}

// Adjoint (Euclidean or Riemannian): per-CTA partial gradients (+ loss partials).
template <int R>
__global__ void __launch_bounds__(kGatherThreads) k_gather_bwd(const __grid_constant__ GatherArgs g) {
  extern __shared__ float sm[];
  __shared__ double red[kGatherThreads / 32];
  constexpr int SS = R * R + 4;          // slice stride (distinct banks for random slices)
  const int SL = g.d * g.nmax * SS;      // staged floats per core set
  const int GS = R * R + 1;              // odd slice stride of the accumulator
  float* Ls = sm;
  float* Rs = g.same ? Ls : Ls + SL;
  float* acc = Ls + (g.same ? SL : 2 * SL);  // d * nmax * GS
  float* sfx = acc + g.d * g.nmax * GS;      // [d][R][blockDim]: suffix at interface k+1
  // both objects land in the accumulator region (zeroed afterwards), one after the other
  __shared__ __align__(8) uint64_t bar;
  bar_init(&bar);
  bool ok = stage_object_tma<R>(Ls, SS, acc, g.L, g.Lnfl, g.Loff, g.rl, g.n, g.d, g.nmax, &bar, 0u);
  __syncthreads();
  if (!g.same) {
    ok &= stage_object_tma<R>(Rs, SS, acc, g.Rg, g.Rnfl, g.Roff, g.rr, g.n, g.d, g.nmax, &bar, 1u);
    __syncthreads();
  }
  if (!ok && threadIdx.x == 0) atomicExch(g.err, (int)T3F_ERR_TIMEOUT);
  for (int e = threadIdx.x; e < g.d * g.nmax * GS; e += blockDim.x) acc[e] = 0.0f;
  __syncthreads();
  const int tid = threadIdx.x, nth = blockDim.x;
  double lsum = 0.0;
  for (long long t0 = (long long)blockIdx.x * nth; t0 < g.N; t0 += (long long)gridDim.x * nth) {
    const long long t = t0 + tid;
    const bool active = t < g.N;
    if (active) {
      // suffix chain through the right cores
      float rho[R];
#pragma unroll
      for (int a = 0; a < R; ++a) rho[a] = a == 0 ? 1.0f : 0.0f;
      for (int k = g.d - 1; k >= 1; --k) {
#pragma unroll
        for (int a = 0; a < R; ++a) sfx[(k * R + a) * nth + tid] = rho[a];
        const int i = load_index(g, k, t);
        const float* S = Rs + (k * g.nmax + i) * SS;
        float nr[R];
#pragma unroll
        for (int a = 0; a < R; ++a) {
          float s = 0.0f;
#pragma unroll
          for (int b = 0; b < R; b += 4) {
            const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
            s = fmaf(s4.x, rho[b], s);
            s = fmaf(s4.y, rho[b + 1], s);
            s = fmaf(s4.z, rho[b + 2], s);
            s = fmaf(s4.w, rho[b + 3], s);
          }
          nr[a] = s;
        }
#pragma unroll
        for (int a = 0; a < R; ++a) rho[a] = nr[a];
      }
#pragma unroll
      for (int a = 0; a < R; ++a) sfx[a * nth + tid] = rho[a];
      const int i0 = load_index(g, 0, t);
      // X(i_t) = row 0 of the first suffix core's slice times the suffix at interface 1
      const float* S0 = Rs + i0 * SS;
      float x = 0.0f;
#pragma unroll
      for (int b = 0; b < R; ++b) x = fmaf(S0[b], rho[b], x);
      float wt;
      if (g.w) {
        wt = g.w[t];
      } else {
        const double res = (double)x - (double)g.y[t];
        lsum += 0.5 * res * res;
        wt = (float)res;
      }
      // prefix walk with the scatter of w l_k rho_{k+1}^T into slice i_k of core k
      float l[R];
#pragma unroll
      for (int a = 0; a < R; ++a) l[a] = a == 0 ? wt : 0.0f;  // carries the weight
      for (int k = 0; k < g.d; ++k) {
        const int i = (k == 0) ? i0 : load_index(g, k, t);
        float r1[R];
#pragma unroll
        for (int b = 0; b < R; ++b) r1[b] = sfx[(k * R + b) * nth + tid];
        const int ra = g.rl[k], rb = g.rr[k + 1];
        float* A = acc + (k * g.nmax + i) * GS;
#pragma unroll
        for (int a = 0; a < R; ++a) {
          if (a < ra) {
#pragma unroll
            for (int b = 0; b < R; ++b)
              if (b < rb) atomicAdd(A + a * R + b, l[a] * r1[b]);
          }
        }
        if (k + 1 < g.d) {
          const float* S = Ls + (k * g.nmax + i) * SS;
          float nl[R];
#pragma unroll
          for (int b = 0; b < R; ++b) nl[b] = 0.0f;
#pragma unroll
          for (int a = 0; a < R; ++a) {
#pragma unroll
            for (int b = 0; b < R; b += 4) {
              const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
              nl[b] = fmaf(l[a], s4.x, nl[b]);
              nl[b + 1] = fmaf(l[a], s4.y, nl[b + 1]);
              nl[b + 2] = fmaf(l[a], s4.z, nl[b + 2]);
              nl[b + 3] = fmaf(l[a], s4.w, nl[b + 3]);
            }
          }
#pragma unroll
          for (int b = 0; b < R; ++b) l[b] = nl[b];
        }
      }
    }
  }
  __syncthreads();
  // write this CTA's partial gradient in the compact layout
  float* out = g.grad_part + (long long)blockIdx.x * g.gsize;
  for (int k = 0; k < g.d; ++k) {
    const int ra = g.rl[k], rb = g.rr[k + 1], nk = g.n[k];
    for (int e = tid; e < ra * nk * rb; e += nth) {
      const int b = e % rb, i = (e / rb) % nk, a = e / (rb * nk);
      out[g.goff[k] + e] = acc[(k * g.nmax + i) * GS + a * R + b];
    }
  }
  if (g.loss_part) {
    const double s = block_sum(lsum, red);
    if (threadIdx.x == 0) g.loss_part[blockIdx.x] = s;
  }
}

// Bucketed adjoint (the main path for ranks <= 8). Per chunk of T tuples, 2 T threads:
//  (1) a deterministic counting sort of the chunk's tuples by slice, for every core (warp
//      match + per-warp prefix sums; each thread of a tuple takes every other core), giving each
//      tuple its bucket position at core k; the next chunk's indices are fetched meanwhile;
//  (2) R = 8: both chains step core by core in bucket order, T threads each: the thread of row p at
//      core k reads l_k (rho_{k+1}), multiplies it by its slice -- the same slice for the neighbouring
//      rows of its bucket, so a warp reads three or four slices instead of 32 random ones -- and
//      writes the result to its tuple's row in the order of core k + 1 (k - 1). R = 4: the two threads of
//      a tuple walk its chains through their own slices and store every partial in bucket order (a
//      step is 16 multiply-adds, less than the barrier it would need);
//  (3) thread per item (core k, slice s, part): a persistent R x R register accumulator
//      adds w l_k rho_{k+1}^T over the item's share of the bucket; consecutive lanes read
//      consecutive bucket rows.
// The per-CTA partial is summed in a fixed order by a second kernel; the parts of a slice within one CTA
// are summed within each warp and then by shared-memory atomics (by atomics alone, all to one address, that
// took 35 of the 60 us of a call on 100 tuples at d = 4, n = 8, r = 8).
// Bound by shared-memory wavefronts (a chain step reads R^2 slice values per tuple for as many
// multiply-adds). 10^6 tuples, d = 10, n = 10, r = 8: 529 us with one thread per tuple walking both
// chains through its own slices, 422 us with the chains on two threads (shared-memory pipe 71 %
// busy, 5.8 wavefronts a request), 390 us in bucket order (65 %); with two sets of slices (the Riemannian
// form) 591 -> 462 -> 433 us. r = 4, 1.5 10^6 tuples: 284 us with one thread per tuple, 365 in bucket order
// with half the tuples in flight, now 236.
struct CompletionArgs {
  GatherArgs g;
  int T;                      // tuples per chunk (half of blockDim.x)
  int NB;                     // buckets per core (nmax + 1; the last holds invalid tuples)
  int region;                 // floats of the RH / LW region
  int parts[T3F_MAX_D];       // items per slice at core k
  int item0[T3F_MAX_D + 1];   // first item of core k
};

template <int R>
__global__ void __launch_bounds__(512) k_completion(const __grid_constant__ CompletionArgs ca) {
  extern __shared__ __align__(16) float sm[];
  __shared__ double red[16];
  const GatherArgs& g = ca.g;
  const int d = g.d, nmax = g.nmax, T = ca.T, NB = ca.NB;
  constexpr int SS = R * R + 4;  // padded slice stride (breaks same-bank slices)
  constexpr int H = R / 4;       // float4 planes of a rank vector
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = T >> 5, nwarps = blockDim.x >> 5;
  const int grp = tid >= T ? 1 : 0, tt = tid - grp * T, tw = tt >> 5;  // chain (0 suffix, 1 prefix), tuple / row, its warp
  const int SL = d * nmax * SS;
  float* Ls = sm;
  float* Rs = g.same ? Ls : Ls + SL;
  float4* RH = reinterpret_cast<float4*>(Ls + (g.same ? SL : 2 * SL));  // [d - 1][H][T]: rho_{k+1} of core k
  float4* LW = RH + (size_t)(d - 1) * H * T;                               // [d - 1][H][T]: l of core k + 1
  float* Wt = reinterpret_cast<float*>(RH) + ca.region;                    // [T] weights
  int* IN = reinterpret_cast<int*>(Wt + T);                                // [d][T] the next chunk's indices
  unsigned short* WC = reinterpret_cast<unsigned short*>(IN + (size_t)d * T);  // [d][NB][NW]
  unsigned short* BO = WC + (size_t)d * NB * NW;                               // [d][NB] bucket starts
  unsigned char* IDX = reinterpret_cast<unsigned char*>(BO + (size_t)d * NB);  // [d][T] slice of a tuple
  unsigned char* POS = IDX + (size_t)d * T;   // [d][T] rank among its warp's, then bucket row of a tuple
  unsigned char* TID = POS + (size_t)d * T;   // [d][T] tuple of a bucket row
  unsigned char* SLC = TID + (size_t)d * T;   // [d][T] slice of a bucket row

  // stage the cores as zero-padded R x R slices with stride SS: the whole object(s) land in
  // the RH / LW region (not used before the first chunk) through one TMA bulk copy each
  __shared__ __align__(8) uint64_t bar;
  bar_init(&bar);
  float* landL = reinterpret_cast<float*>(RH);
  float* landR = landL + ((raw_bytes(g.L, g.Lnfl) + 15) / 16) * 4;
  if (tid == 0) {
    tma_expect(&bar, raw_bytes(g.L, g.Lnfl) + (g.same ? 0u : raw_bytes(g.Rg, g.Rnfl)));
    tma_copy(landL, g.L, g.Lnfl, &bar);
    if (!g.same) tma_copy(landR, g.Rg, g.Rnfl, &bar);
  }
  // this thread's indices of the chunk at base (read back by this thread only)
  auto fetch = [&](long long base) {
    const long long t = base + tt;
    const bool ok = t < g.N;
    for (int k = grp; k < d; k += 2) {
      const int* src = g.idx + (ok ? (long long)k * g.N + t : 0);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(smem_u32(IN + k * T + tt)), "l"(src),
                   "r"(ok ? 4 : 0));
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  fetch((long long)blockIdx.x * T);
  if (!bar_wait(smem_u32(&bar), 0u) && tid == 0) atomicExch(g.err, (int)T3F_ERR_TIMEOUT);
  stage_from_raw<R>(Ls, SS, landL + raw_delta(g.L), g.Loff, g.rl, g.n, d, nmax);
  if (!g.same) stage_from_raw<R>(Rs, SS, landR + raw_delta(g.Rg), g.Roff, g.rr, g.n, d, nmax);
  // this thread's item (core ik, slice is, part ip) of the accumulation phase
  int ik = -1, is = 0, ip = 0, np = 1;
  for (int k = 0; k < d; ++k)
    if (tid >= ca.item0[k] && tid < ca.item0[k + 1]) {
      ik = k;
      is = (tid - ca.item0[k]) / ca.parts[k];
      ip = (tid - ca.item0[k]) % ca.parts[k];
      np = ca.parts[k];
    }
  float acc[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) acc[a][b] = 0.0f;
  bool used = false;  // the item has had a tuple
  double lsum = 0.0;
  __syncthreads();

  for (long long base = (long long)blockIdx.x * T; base < g.N; base += (long long)gridDim.x * T) {
    const long long t = base + tt;
    const bool valid = t < g.N;
    const int nv = (int)min((long long)T, g.N - base);  // valid tuples: the first nv rows of every core
    float yt = 0.0f;
    if (grp == 0 && valid) yt = g.w ? __ldg(g.w + t) : __ldg(g.y + t);
    // (1) counting sort by slice (the counts of a (core, warp) belong to that warp)
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    for (int k = grp; k < d; k += 2) {
      int sl = nmax;
      if (valid) {
        sl = IN[k * T + tt];
        if (sl < 0 || sl >= g.n[k]) {
          atomicExch(g.err, (int)T3F_ERR_ARG);
          sl = sl < 0 ? 0 : g.n[k] - 1;
        }
      }
      for (int b = lane; b < NB; b += 32) WC[(k * NB + b) * NW + tw] = 0;
      const unsigned m = __match_any_sync(0xffffffffu, sl);
      const int rank = __popc(m & ((1u << lane) - 1u));
      IDX[k * T + tt] = (unsigned char)sl;
      POS[k * T + tt] = (unsigned char)rank;
      __syncwarp();
      if (rank == 0) WC[(k * NB + sl) * NW + tw] = (unsigned short)__popc(m);
    }
    fetch(base + (long long)gridDim.x * T);
    __syncthreads();  // counts complete; the previous chunk's accumulation is done
    if (grp == 0) Wt[tt] = yt;
    for (int k = warp; k < d; k += nwarps) {  // a warp per core: scan over the slices
      int carry = 0;
      for (int b0 = 0; b0 < NB; b0 += 32) {
        const int b = b0 + lane;
        unsigned short* wc = WC + (size_t)(k * NB + min(b, NB - 1)) * NW;
        int tot = 0;
        if (b < NB)
          for (int w = 0; w < NW; ++w) tot += wc[w];
        int inc = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += v;
        }
        int run = carry + inc - tot;
        if (b < NB) {
          BO[k * NB + b] = (unsigned short)run;
          for (int w = 0; w < NW; ++w) {
            const int c = wc[w];
            wc[w] = (unsigned short)run;
            run += c;
          }
        }
        carry += __shfl_sync(0xffffffffu, inc, 31);
      }
    }
    __syncthreads();
    if constexpr (R == 4) {
      // (2) the tuple's chains; p = its row in the bucket order of core k
      if (valid) {
        float v[R];
#pragma unroll
        for (int a = 0; a < R; ++a) v[a] = a == 0 ? 1.0f : 0.0f;
        if (grp == 0) {
          for (int k = d - 1; k >= 0; --k) {
            const int sl = IDX[k * T + tt];
            const float* S = Rs + (k * nmax + sl) * SS;
            if (k < d - 1) {
              const int p = WC[(k * NB + sl) * NW + tw] + POS[k * T + tt];
#pragma unroll
              for (int h = 0; h < H; ++h)
                RH[((size_t)k * H + h) * T + p] = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
            }
            if (k == 0) {
              float x = 0.0f;
#pragma unroll
              for (int b = 0; b < R; ++b) x = fmaf(S[b], v[b], x);
              v[0] = x;
              break;
            }
            float nr[R];
#pragma unroll
            for (int a = 0; a < R; ++a) {
              float acc1 = 0.0f;
#pragma unroll
              for (int b = 0; b < R; b += 4) {
                const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
                acc1 = fmaf(s4.x, v[b], acc1);
                acc1 = fmaf(s4.y, v[b + 1], acc1);
                acc1 = fmaf(s4.z, v[b + 2], acc1);
                acc1 = fmaf(s4.w, v[b + 3], acc1);
              }
              nr[a] = acc1;
            }
#pragma unroll
            for (int a = 0; a < R; ++a) v[a] = nr[a];
          }
          float wt = yt;
          if (!g.w) {
            const double res = (double)v[0] - (double)yt;
            lsum += 0.5 * res * res;
            wt = (float)res;
          }
          Wt[tt] = wt;
        } else {
          for (int k = 0; k < d; ++k) {
            const int sl = IDX[k * T + tt];
            const int p = WC[(k * NB + sl) * NW + tw] + POS[k * T + tt];
            TID[k * T + p] = (unsigned char)tt;
            if (k > 0)
#pragma unroll
              for (int h = 0; h < H; ++h)
                LW[((size_t)(k - 1) * H + h) * T + p] = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
            if (k + 1 == d) break;
            const float* S = Ls + (k * nmax + sl) * SS;
            float nl[R];
#pragma unroll
            for (int b = 0; b < R; ++b) nl[b] = 0.0f;
#pragma unroll
            for (int a = 0; a < R; ++a) {
#pragma unroll
              for (int b = 0; b < R; b += 4) {
                const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
                nl[b] = fmaf(v[a], s4.x, nl[b]);
                nl[b + 1] = fmaf(v[a], s4.y, nl[b + 1]);
                nl[b + 2] = fmaf(v[a], s4.z, nl[b + 2]);
                nl[b + 3] = fmaf(v[a], s4.w, nl[b + 3]);
              }
            }
#pragma unroll
            for (int b = 0; b < R; ++b) v[b] = nl[b];
          }
        }
      }
    } else {
      for (int k = grp; k < d; k += 2) {
        const int sl = IDX[k * T + tt], p = WC[(k * NB + sl) * NW + tw] + POS[k * T + tt];
        POS[k * T + tt] = (unsigned char)p;
        TID[k * T + p] = (unsigned char)tt;
        SLC[k * T + p] = (unsigned char)sl;
      }
      __syncthreads();
      // (2) the chains, row tt of each core in turn
      for (int q = 0; q + 1 < d; ++q) {
        if (tt < nv) {
          if (grp == 0) {
            const int k = d - 1 - q;
            const float* S = Rs + (k * nmax + SLC[k * T + tt]) * SS;
            const int p = POS[(k - 1) * T + TID[k * T + tt]];
            float v[R], nr[R];
            if (q == 0) {
#pragma unroll
              for (int a = 0; a < R; ++a) nr[a] = S[a * R];
            } else {
#pragma unroll
              for (int h = 0; h < H; ++h) {
                const float4 r4 = RH[((size_t)k * H + h) * T + tt];
                v[4 * h] = r4.x; v[4 * h + 1] = r4.y; v[4 * h + 2] = r4.z; v[4 * h + 3] = r4.w;
              }
#pragma unroll
              for (int a = 0; a < R; ++a) {
                float acc1 = 0.0f;
#pragma unroll
                for (int b = 0; b < R; b += 4) {
                  const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
                  acc1 = fmaf(s4.x, v[b], acc1);
                  acc1 = fmaf(s4.y, v[b + 1], acc1);
                  acc1 = fmaf(s4.z, v[b + 2], acc1);
                  acc1 = fmaf(s4.w, v[b + 3], acc1);
                }
                nr[a] = acc1;
              }
            }
#pragma unroll
            for (int h = 0; h < H; ++h)
              RH[((size_t)(k - 1) * H + h) * T + p] = make_float4(nr[4 * h], nr[4 * h + 1], nr[4 * h + 2], nr[4 * h + 3]);
          } else {
            const int k = q;
            const float* S = Ls + (k * nmax + SLC[k * T + tt]) * SS;
            const int p = POS[(k + 1) * T + TID[k * T + tt]];
            float v[R], nl[R];
            if (q == 0) {
#pragma unroll
              for (int b = 0; b < R; ++b) nl[b] = S[b];
            } else {
#pragma unroll
              for (int h = 0; h < H; ++h) {
                const float4 l4 = LW[((size_t)(k - 1) * H + h) * T + tt];
                v[4 * h] = l4.x; v[4 * h + 1] = l4.y; v[4 * h + 2] = l4.z; v[4 * h + 3] = l4.w;
              }
#pragma unroll
              for (int b = 0; b < R; ++b) nl[b] = 0.0f;
#pragma unroll
              for (int a = 0; a < R; ++a) {
#pragma unroll
                for (int b = 0; b < R; b += 4) {
                  const float4 s4 = *reinterpret_cast<const float4*>(S + a * R + b);
                  nl[b] = fmaf(v[a], s4.x, nl[b]);
                  nl[b + 1] = fmaf(v[a], s4.y, nl[b + 1]);
                  nl[b + 2] = fmaf(v[a], s4.z, nl[b + 2]);
                  nl[b + 3] = fmaf(v[a], s4.w, nl[b + 3]);
                }
              }
            }
#pragma unroll
            for (int h = 0; h < H; ++h)
              LW[((size_t)k * H + h) * T + p] = make_float4(nl[4 * h], nl[4 * h + 1], nl[4 * h + 2], nl[4 * h + 3]);
          }
        }
        __syncthreads();
      }
      // the value (from the suffix cores), residual and weight of row tt of the first core
      if (grp == 0 && tt < nv) {
        const float* S = Rs + SLC[tt] * SS;
        const int o = TID[tt];
        float x = S[0];
        if (d > 1) {
          x = 0.0f;
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const float4 r4 = RH[(size_t)h * T + tt];
            const float4 s4 = *reinterpret_cast<const float4*>(S + 4 * h);
            x = fmaf(s4.x, r4.x, x);
            x = fmaf(s4.y, r4.y, x);
            x = fmaf(s4.z, r4.z, x);
            x = fmaf(s4.w, r4.w, x);
          }
        }
        if (!g.w) {
          const double res = (double)x - (double)Wt[o];
          lsum += 0.5 * res * res;
          Wt[o] = (float)res;
        }
      }
    }
    __syncthreads();
    // (3) accumulation: this thread's item over its share of the bucket (l = 1 before the first
    // core, rho = 1 after the last)
    if (ik >= 0) {
      const int p0 = BO[ik * NB + is], p1 = BO[ik * NB + is + 1];
      used = used || p0 + ip < p1;
      const unsigned char* tb = TID + (size_t)ik * T;
      const float4* lw = LW + (size_t)(ik - 1) * H * T;
      const float4* rh = RH + (size_t)ik * H * T;
      if (ik == 0) {
        for (int p = p0 + ip; p < p1; p += np) {
          const float w = Wt[tb[p]];
          if (d == 1) {
            acc[0][0] += w;
            continue;
          }
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const float4 b4 = rh[(size_t)h * T + p];
            acc[0][4 * h] = fmaf(w, b4.x, acc[0][4 * h]);
            acc[0][4 * h + 1] = fmaf(w, b4.y, acc[0][4 * h + 1]);
            acc[0][4 * h + 2] = fmaf(w, b4.z, acc[0][4 * h + 2]);
            acc[0][4 * h + 3] = fmaf(w, b4.w, acc[0][4 * h + 3]);
          }
        }
      } else if (ik == d - 1) {
        for (int p = p0 + ip; p < p1; p += np) {
          const float w = Wt[tb[p]];
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const float4 a4 = lw[(size_t)h * T + p];
            acc[4 * h][0] = fmaf(w, a4.x, acc[4 * h][0]);
            acc[4 * h + 1][0] = fmaf(w, a4.y, acc[4 * h + 1][0]);
            acc[4 * h + 2][0] = fmaf(w, a4.z, acc[4 * h + 2][0]);
            acc[4 * h + 3][0] = fmaf(w, a4.w, acc[4 * h + 3][0]);
          }
        }
      } else {
        for (int p = p0 + ip; p < p1; p += np) {
          const float w = Wt[tb[p]];
          float lv[R], rv[R];
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const float4 a4 = lw[(size_t)h * T + p];
            const float4 b4 = rh[(size_t)h * T + p];
            lv[4 * h] = w * a4.x; lv[4 * h + 1] = w * a4.y; lv[4 * h + 2] = w * a4.z; lv[4 * h + 3] = w * a4.w;
            rv[4 * h] = b4.x; rv[4 * h + 1] = b4.y; rv[4 * h + 2] = b4.z; rv[4 * h + 3] = b4.w;
          }
#pragma unroll
          for (int a = 0; a < R; ++a)
#pragma unroll
            for (int b = 0; b < R; ++b) acc[a][b] = fmaf(lv[a], rv[b], acc[a][b]);
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  // sum the parts of every (core, slice) in shared memory, then write the CTA's partial
  float* cacc = reinterpret_cast<float*>(RH);  // d * nmax * R * R floats (fits the region)
  for (int e = tid; e < d * nmax * R * R; e += blockDim.x) cacc[e] = 0.0f;
  __syncthreads();
  if (const int lanes = __popc(__ballot_sync(0xffffffffu, used))) {
    // the parts of a slice sit on neighbouring lanes: their sum within the warp ends in the lane of the first
    // (a warp with a few tuples adds them directly)
    const int left = ik < 0 ? 1 : np - ip;  // lanes of this slice from here on
    int most = 1;
    if (lanes > 4)
      for (int k = 0; k < d; ++k) most = max(most, min(ca.parts[k], 32));
    for (int o = 1; o < most; o <<= 1) {
      const bool on = o < left && lane + o < 32;
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) {
          const float v = __shfl_down_sync(0xffffffffu, acc[a][b], o);
          if (on) acc[a][b] += v;
        }
    }
    if (ik >= 0 && (most == 1 || lane == 0 || ip == 0)) {
      float* dst = cacc + (ik * nmax + is) * R * R;
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b)
          if (acc[a][b] != 0.0f) atomicAdd(dst + a * R + b, acc[a][b]);
    }
  }
  __syncthreads();
  float* out = g.grad_part + (long long)blockIdx.x * g.gsize;
  for (int k = 0; k < d; ++k) {
    const int ra = g.rl[k], rb = g.rr[k + 1], nk = g.n[k];
    for (int e = tid; e < ra * nk * rb; e += blockDim.x) {
      const int b = e % rb, i = (e / rb) % nk, a = e / (rb * nk);
      out[g.goff[k] + e] = cacc[(k * nmax + i) * R * R + a * R + b];
    }
  }
  if (g.loss_part) {
    double v = lsum;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (tid == 0) {
      double s2 = 0.0;
      for (int i = 0; i < nwarps; ++i) s2 += red[i];
      g.loss_part[blockIdx.x] = s2;
    }
  }
}

// Sum of the per-CTA partials in a fixed order: a block owns 32 elements, its eight rows of 32
// threads each sum every eighth partial and are then summed in order (one thread per element
// over all partials left 21 of 608 blocks with 300 dependent reads each: 32 us, now 5 us). One
// more block sums the loss partials where there is a loss.
__global__ void __launch_bounds__(256) k_reduce_partials(const float* part, int nparts, long long size, float* out,
                                                         const double* lpart, double* loss) {
  __shared__ float sm[8][33];
  __shared__ double red[8];
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  const long long blocks = (size + 31) / 32;
  if (blockIdx.x == blocks) {
    double s = 0.0;
    for (int p = threadIdx.x; p < nparts; p += 256) s += lpart[p];
    s = block_sum(s, red);
    if (threadIdx.x == 0) *loss = s;
    return;
  }
  const long long e = (long long)blockIdx.x * 32 + lane;
  float s = 0.0f;
  if (e < size)
#pragma unroll 4
    for (int p = row; p < nparts; p += 8) s += part[(long long)p * size + e];
  sm[row][lane] = s;
  __syncthreads();
  if (row == 0 && e < size) {
#pragma unroll
    for (int r = 1; r < 8; ++r) s += sm[r][lane];
    out[e] = s;
  }
}

__global__ void k_reduce_loss(const double* part, int nparts, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int p = threadIdx.x; p < nparts; p += blockDim.x) s += part[p];
  s = block_sum(s, red);
  if (threadIdx.x == 0) *out = s;
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------

static int pick_R(int rmax) {
  if (rmax <= 4) return 4;
  if (rmax <= 8) return 8;
  if (rmax <= 16) return 16;
  return 0;
}

static int gather_grid(long long N, int maxCtas) {
  long long g = (N + kGatherThreads - 1) / kGatherThreads;
  if (g > maxCtas) g = maxCtas;
  return (int)(g < 1 ? 1 : g);
}

// SM count of the current device, looked up once per device index.
static int num_sms() { return device_sm_count(); }

struct GatherLayout {
  int R;
  int grid;
  size_t smem;
  size_t loss_off, grad_off, total;
  // bucketed adjoint
  int bucketed, T, NB, region;
  int parts[T3F_MAX_D];
  int item0[T3F_MAX_D + 1];
};

// Floats of the RH / LW region: both chains' vectors, the landing zone of the packed objects and the
// final sums of the parts all use it.
static long long completion_region(const TTV& L, const TTV& Rv, int R, int T, bool same) {
  const long long nl = L.off[L.d - 1] + L.osz[L.d - 1], nr = same ? 0 : Rv.off[Rv.d - 1] + Rv.osz[Rv.d - 1];
  long long f = std::max(2LL * (L.d - 1) * R * T, (long long)L.d * L.nmax * R * R);
  f = std::max(f, nl + nr + 16);  // each rounded out to 16 bytes on both sides
  return (f + 3) & ~3LL;
}

static size_t completion_smem(const TTV& L, const TTV& Rv, int R, int T, bool same) {
  const size_t SS = (size_t)R * R + 4, d = L.d;
  const size_t NB = L.nmax + 1, NW = T / 32;
  size_t b = sizeof(float) * ((same ? 1 : 2) * d * L.nmax * SS + (size_t)completion_region(L, Rv, R, T, same) + T);
  b += sizeof(int) * d * T;                              // IN
  b += sizeof(unsigned short) * (d * NB * NW + d * NB);  // WC, BO (counts <= T)
  b += 4 * d * T;                                        // IDX, POS, TID, SLC
  return (b + 15) & ~(size_t)15;
}

// Choose the bucketed adjoint when its items fit one CTA and its buffers fit shared memory: the
// largest chunk T <= 256 of one CTA per SM, or the largest of two (one CTA's barrier waits overlap the
// other's chains; up to 256 threads at the 128 registers of R = 8, 512 at the 64 of R = 4) where that keeps
// as many tuples in flight, or for R = 4 of four on the same condition. 1.5 10^6 tuples, r = 4: d = 10, n = 10
// two CTAs of 256 tuples 252 us, four of 128 236; d = 30, n = 4 two CTAs of fewer tuples than one holds
// 1255 us, one 986.
static bool plan_completion(const TTV& L, const TTV& Rv, bool same, int R, GatherLayout* lay) {
  if (R > 8 || L.nmax > 254) return false;
  const int d = L.d;
  // boundary cores take one item per slice, interior cores share the rest of the 2 T threads evenly
  int bnd = 0, inner = 0;
  for (int k = 0; k < d; ++k) {
    if (k == 0 || k == d - 1) bnd += L.n[k];
    else inner += L.n[k];
  }
  // the largest chunk of at most `most` tuples that leaves room for `ctas` CTAs on an SM, 0 where none does
  auto best = [&](int ctas, int most) {
    const size_t cap = ctas == 1 ? 220 * 1024 : (228 * 1024 - ctas * 1400) / ctas;
    for (int T = most; T >= 64; T -= 32)
      if (completion_smem(L, Rv, R, T, same) <= cap && bnd + inner <= 2 * T) return T;
    return 0;
  };
  const int T1 = best(1, 256), T2 = best(2, R == 4 ? 256 : 128), T4 = R == 4 ? best(4, 128) : 0;
  if (!T1) return false;
  const bool two = T2 > 0 && 2 * T2 >= T1, four = two && T4 > 0 && 2 * T4 >= T2;
  const int T = four ? T4 : two ? T2 : T1;
  const int P2 = inner ? (2 * T - bnd) / inner : 1;
  int it = 0;
  for (int k = 0; k < d; ++k) {
    lay->item0[k] = it;
    lay->parts[k] = (k == 0 || k == d - 1) ? 1 : P2;
    it += L.n[k] * lay->parts[k];
  }
  lay->item0[d] = it;
  lay->bucketed = four ? 4 : two ? 2 : 1;  // CTAs per SM
  lay->T = T;
  lay->NB = L.nmax + 1;
  lay->region = (int)completion_region(L, Rv, R, T, same);
  lay->smem = completion_smem(L, Rv, R, T, same);
  return true;
}

static GatherLayout gather_layout(const TTV& L, const TTV& Rv, long long N, bool bwd, bool same) {
  GatherLayout lay{};
  lay.R = pick_R(L.rmax > Rv.rmax ? L.rmax : Rv.rmax);
  const int R = lay.R ? lay.R : 16;
  const int nmax = L.nmax;
  if (!bwd) {
    // padded slices + the TMA landing zone of the packed object (rounded out to 16 bytes)
    const long long nfl = L.off[L.d - 1] + L.osz[L.d - 1];
    lay.smem = sizeof(float) * (size_t)L.d * nmax * (R * R + 4) + (size_t)((nfl * 4 + 12 + 15) / 16) * 16;
    lay.grid = gather_grid(N, num_sms() * 8);
  } else if (lay.R && plan_completion(L, Rv, same, R, &lay)) {
    long long g = (N + lay.T - 1) / lay.T;
    if (g > (long long)num_sms() * lay.bucketed) g = (long long)num_sms() * lay.bucketed;
    lay.grid = (int)(g < 1 ? 1 : g);
  } else {
    lay.smem = sizeof(float) * ((same ? 1 : 2) * (size_t)L.d * nmax * (R * R + 4) + (size_t)L.d * nmax * (R * R + 1) +
                                (size_t)L.d * R * kGatherThreads);
    lay.grid = gather_grid(N, num_sms() * 2);
  }
  long long gsize = 0;
  for (int k = 0; k < L.d; ++k) gsize += (long long)L.r[k] * L.n[k] * Rv.r[k + 1];
  lay.loss_off = kWsHeader;
  lay.grad_off = lay.loss_off + align256(sizeof(double) * lay.grid);
  lay.total = lay.grad_off + (bwd ? align256(sizeof(float) * gsize * lay.grid) : 0);
  return lay;
}

size_t ws_gather(const TTV& X, long long N, bool bwd) {
  return gather_layout(X, X, N, bwd, true).total;
}
size_t ws_rgather(const TTV& U, const TTV& V, long long N) {
  return gather_layout(U, V, N, true, false).total;
}

static void fill_args(GatherArgs* g, const TTV& L, const TTV& Rv) {
  g->d = L.d;
  g->nmax = L.nmax;
  for (int k = 0; k <= L.d; ++k) {
    g->rl[k] = L.r[k];
    g->rr[k] = Rv.r[k];
  }
  long long go = 0;
  for (int k = 0; k < L.d; ++k) {
    g->n[k] = L.n[k];
    g->Loff[k] = L.off[k];
    g->Roff[k] = Rv.off[k];
    g->goff[k] = go;
    go += (long long)L.r[k] * L.n[k] * Rv.r[k + 1];
  }
  g->gsize = go;
  g->L = static_cast<const float*>(L.p);
  g->Rg = static_cast<const float*>(Rv.p);
  g->Lnfl = L.off[L.d - 1] + L.osz[L.d - 1];
  g->Rnfl = Rv.off[Rv.d - 1] + Rv.osz[Rv.d - 1];
}

template <int R>
static t3f_status launch_fwd(const GatherArgs& g, const GatherLayout& lay, cudaStream_t s) {
  auto kern = k_gather_fwd<R>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lay.smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<lay.grid, kGatherThreads, lay.smem, s>>>(g);
  return launch_status();
}

template <int R>
static t3f_status launch_completion(const GatherArgs& g, const GatherLayout& lay, cudaStream_t s) {
  CompletionArgs ca;
  memset(&ca, 0, sizeof(ca));
  ca.g = g;
  ca.T = lay.T;
  ca.NB = lay.NB;
  ca.region = lay.region;
  for (int k = 0; k < g.d; ++k) ca.parts[k] = lay.parts[k];
  for (int k = 0; k <= g.d; ++k) ca.item0[k] = lay.item0[k];
  auto kern = k_completion<R>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lay.smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<lay.grid, 2 * lay.T, lay.smem, s>>>(ca);
  return launch_status();
}

template <int R>
static t3f_status launch_bwd(const GatherArgs& g, const GatherLayout& lay, cudaStream_t s) {
  if (lay.bucketed) return launch_completion<(R <= 4 ? 4 : 8)>(g, lay, s);
  auto kern = k_gather_bwd<R>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lay.smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<lay.grid, kGatherThreads, lay.smem, s>>>(g);
  return launch_status();
}

}  // namespace t3f

using namespace t3f;

extern "C" t3f_status t3f_gather(const t3f_tt* X, const int32_t* idx, int64_t N, const float* y,
                                 float* vals, double* loss, void* ws, size_t ws_bytes,
                                 t3f_stream_t stream) {
  TTV vx;
  T3F_CHECK(make_view(X, &vx, T3F_F32, false));
  if (vx.batch != 1) return T3F_ERR_SHAPE;
  if (N < 0 || (N > 0 && !idx) || (loss && !y && N > 0)) return T3F_ERR_ARG;
  GatherLayout lay = gather_layout(vx, vx, N, false, true);
  if (!lay.R || lay.smem > 227 * 1024) return T3F_ERR_UNSUPPORTED;
  T3F_CHECK(check_ws(ws, ws_bytes, lay.total));
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(ws, 0, sizeof(int32_t), s) != cudaSuccess) return T3F_ERR_CUDA;
  if (N == 0) {
    if (loss && cudaMemsetAsync(loss, 0, sizeof(double), s) != cudaSuccess) return T3F_ERR_CUDA;
    return T3F_OK;
  }
  GatherArgs g;
  memset(&g, 0, sizeof(g));
  fill_args(&g, vx, vx);
  g.same = 1;
  g.N = N;
  g.idx = idx;
  g.y = y;
  g.vals = vals;
  g.err = static_cast<int*>(ws);
  double* lp = reinterpret_cast<double*>(static_cast<char*>(ws) + lay.loss_off);
  g.loss_part = loss ? lp : nullptr;
  t3f_status st;
  switch (lay.R) {
    case 4: st = launch_fwd<4>(g, lay, s); break;
    case 8: st = launch_fwd<8>(g, lay, s); break;
    default: st = launch_fwd<16>(g, lay, s); break;
  }
  T3F_CHECK(st);
  if (loss) {
    k_reduce_loss<<<1, 1024, 0, s>>>(lp, lay.grid, loss);
    T3F_CHECK(launch_status());
  }
  return T3F_OK;
}

extern "C" t3f_status t3f_gather_backward(const t3f_tt* X, const int32_t* idx, int64_t N,
                                          const float* w, const float* y, double* loss,
                                          t3f_tt* dX, int32_t riemannian, const t3f_tt* U,
                                          const t3f_tt* V, void* ws, size_t ws_bytes,
                                          t3f_stream_t stream) {
  TTV vl, vr, vd;
  if (riemannian != 0 && riemannian != 1) return T3F_ERR_ARG;
  if (riemannian) {
    T3F_CHECK(make_view(U, &vl, T3F_F32, false));
    T3F_CHECK(make_view(V, &vr, T3F_F32, false));
    if (vl.batch != 1 || vr.batch != 1 || vl.d != vr.d) return T3F_ERR_SHAPE;
    for (int k = 0; k <= vl.d; ++k)
      if (vl.r[k] != vr.r[k] || (k < vl.d && vl.n[k] != vr.n[k])) return T3F_ERR_SHAPE;
  } else {
    T3F_CHECK(make_view(X, &vl, T3F_F32, false));
    if (vl.batch != 1) return T3F_ERR_SHAPE;
    vr = vl;
  }
  T3F_CHECK(make_view(dX, &vd, T3F_F32, false));
  if (vd.batch != 1 || vd.d != vl.d) return T3F_ERR_SHAPE;
  for (int k = 0; k <= vl.d; ++k)
    if (vd.r[k] != vl.r[k] || (k < vl.d && vd.n[k] != vl.n[k])) return T3F_ERR_SHAPE;
  if (N < 0 || (N > 0 && !idx)) return T3F_ERR_ARG;
  if (N > 0 && !w && !y) return T3F_ERR_ARG;
  if (w && loss) return T3F_ERR_ARG;
  const bool same = !riemannian;
  GatherLayout lay = gather_layout(vl, vr, N, true, same);
  if (!lay.R || lay.smem > 227 * 1024) return T3F_ERR_UNSUPPORTED;
  T3F_CHECK(check_ws(ws, ws_bytes, lay.total));
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(ws, 0, sizeof(int32_t), s) != cudaSuccess) return T3F_ERR_CUDA;
  float* out = static_cast<float*>(vd.p);
  const long long gsize = t3f_packed_size(dX);
  if (N == 0) {
    if (cudaMemsetAsync(out, 0, sizeof(float) * gsize, s) != cudaSuccess) return T3F_ERR_CUDA;
    if (loss && cudaMemsetAsync(loss, 0, sizeof(double), s) != cudaSuccess) return T3F_ERR_CUDA;
    return T3F_OK;
  }
  GatherArgs g;
  memset(&g, 0, sizeof(g));
  fill_args(&g, vl, vr);
  g.same = same ? 1 : 0;
  g.N = N;
  g.idx = idx;
  g.y = y;
  g.w = w;
  g.err = static_cast<int*>(ws);
  double* lp = reinterpret_cast<double*>(static_cast<char*>(ws) + lay.loss_off);
  g.loss_part = (!w && loss) ? lp : nullptr;
  float* gp = reinterpret_cast<float*>(static_cast<char*>(ws) + lay.grad_off);
  g.grad_part = gp;
  t3f_status st;
  switch (lay.R) {
    case 4: st = launch_bwd<4>(g, lay, s); break;
    case 8: st = launch_bwd<8>(g, lay, s); break;
    default: st = launch_bwd<16>(g, lay, s); break;
  }
  T3F_CHECK(st);
  // the compact gradient layout equals the packed layout of a batch-1 descriptor
  float* target = out;
  if (riemannian) {
    // the Riemannian form sums into partial slot 0 (every element is read before it is
    // written) and the gauge projection writes the output from there
    target = gp;
  }
  const bool with_loss = loss && !w;
  k_reduce_partials<<<(unsigned)((g.gsize + 31) / 32 + (with_loss ? 1 : 0)), 256, 0, s>>>(gp, lay.grid, g.gsize, target,
                                                                                        lp, loss);
  T3F_CHECK(launch_status());
  if (riemannian) T3F_CHECK(run_gauge_project(vl, gp, out, s));
  return T3F_OK;
}

// ---------------------------------------------------------------------------------------
// Allocation-free variant of t3f_gather.
//
// Some callers cannot allocate device memory for the workspace: a plugin whose host
// framework owns every byte of device memory through its own pool or a hard memory cap
// (a cudaMalloc there either fails or escapes the host's accounting), or code that must
// not risk the implicit device synchronisation that cudaMalloc/cudaFree can cause. This
// entry point needs no workspace: its scratch (the device error word and the per-CTA loss
// partials) lives in one file-scope device array of T3F_NOALLOC_SCRATCH_BYTES that every
// GPU which loads the library keeps until the process exits.
// ---------------------------------------------------------------------------------------

namespace t3f {

static __device__ __align__(256) unsigned char g_noalloc_scratch[T3F_NOALLOC_SCRATCH_BYTES];

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu[kNoAllocMaxDevices];
static void* g_noalloc_ptr[kNoAllocMaxDevices];

// Device address of the scratch array on the current device. The array's name in host
// code is only a host-side stand-in, so the address is looked up with that device current
// and cached per device. Only a successful lookup is cached: a failed one (for example a
// first call made while a stream is being captured) clears the runtime's pending error and
// is retried by the next call.
static t3f_status noalloc_scratch(void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return T3F_ERR_CUDA;
  }
  if (dev < 0 || dev >= kNoAllocMaxDevices) return T3F_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_noalloc_mu[dev]);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return T3F_ERR_CUDA;
    }
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return T3F_OK;
}

}  // namespace t3f

extern "C" t3f_status t3f_gather_noalloc(const t3f_tt* X, const int32_t* idx, int64_t N,
                                         const float* y, float* vals, double* loss,
                                         t3f_stream_t stream) {
  TTV vx;
  T3F_CHECK(make_view(X, &vx, T3F_F32, false));
  if (N < 0) return T3F_ERR_ARG;
  if (gather_layout(vx, vx, N, false, true).total > (size_t)T3F_NOALLOC_SCRATCH_BYTES)
    return T3F_ERR_WORKSPACE;
  void* scratch = nullptr;
  T3F_CHECK(noalloc_scratch(&scratch));
  // the existing entry point clears the error word and overwrites every partial it reads
  return t3f_gather(X, idx, N, y, vals, loss, scratch, T3F_NOALLOC_SCRATCH_BYTES, stream);
}

// The error word at the start of the shared scratch array: the device-side status of the
// last t3f_gather_noalloc call on this device (an index tuple out of range reads back as
// T3F_ERR_ARG). Synchronises `stream`.
extern "C" t3f_status t3f_gather_noalloc_status(t3f_stream_t stream) {
  void* scratch = nullptr;
  T3F_CHECK(noalloc_scratch(&scratch));
  return t3f_device_status(scratch, stream);
}
