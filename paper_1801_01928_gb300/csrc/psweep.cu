// Register-tiled sweeps for project_sum and its adjoint (paper Section 3.2): one tangent
// point X (orthogonal forms U, V and the gauge-projected cotangent W; batch 1, ranks <= RU)
// against a batch of TT objects Z (ranks <= 8).
//
// Every step of these sweeps has the form
//     T[m][b]     = sum_K CurT[K][m] Zs[K][b]          (K < 8)       "T-step"
//     Next[m][b] += sum_K As[K][m]   T[K][b]           (K < RU)      "accumulate step"
// with, for the left sweep (interfaces 0 -> d), Zs = Z_k[:, i, :], As = A_k[:, i, :]
// (Next = sum_i A_i^T Cur Z_i), and for the right sweep (d -> 0), Zs = Z_k[:, i, :]^T,
// As = A_k[:, i, :]^T (Next = sum_i A_i Cur Z_i^T). The fused ("mixed") sweeps of the
// adjoint carry a second partial:
//     left :  L' = sum_i U_i^T (L Z_i),   P' = sum_i V_i^T (P Z_i) + W_i^T (L Z_i)
//     right:  R' = sum_i V_i (R Z_i^T),   Q' = sum_i U_i (Q Z_i^T) + W_i (R Z_i^T)
// A CTA holds J objects; each object owns SPLIT groups of G = (RU / TM) * (8 / TB) threads and
// group h handles the slices i = h (mod SPLIT). A thread forms a TM x TB block of T, hands it to
// its group through shared memory (a group never leaves its warp, so a warp barrier is enough),
// and accumulates a TM x TB block of Next in registers; at the end of a core the SPLIT partial
// blocks are summed in shared memory. All operands are zero-padded to RU x 8, so boundary cores
// need no special cases.
//
// What bounds it: FP32 multiply-adds against shared-memory operands. A thread reads TM + TB
// floats for TM x TB multiply-adds, so 8 x 8 (one sweep) or 8 x 4 (the fused sweep, whose two
// partials and two T blocks hold 128 registers) where the batch gives a CTA enough objects; a
// CTA of few objects has too few groups that way and takes 4 x 4 with more slices at a time
// (the rule in plan_tiles). Config 5 (1000 objects of rank 8, X of rank 32, d = 20, n = 16): 4 x 4
// blocks with T exchanged behind a block barrier and slices staged line by line took 319 + 358 us
// for the left and right sweeps and 715 + 754 us for the fused ones, now 175 + 177 and 420 + 432 us
// (FP32 at 44 % and 51 % of its measured rate; seven warps on four schedulers and the reduction
// between cores are most of the rest). 100 objects: 230 + 250 -> 49 + 50 us.
#include "t3f_internal.cuh"

namespace t3f {

constexpr int kRZ = 8;

struct PSweepArgs {
  TTV Z;
  const float* A;  // slice-major copies (k_xslices) in the sweep's orientation
  const float* B1;
  const float* B2;
  long long xoff[T3F_MAX_D];  // core k of a copy
  int ra[T3F_MAX_D + 1];
  int dir;
  float* st1;
  float* st2;
  long long ioff[T3F_MAX_D + 1];
  int J, SPLIT;
  int* err;  // device error word (nullable): a bounded wait that ran out
};

template <int TM, int TB>
__device__ __forceinline__ void mul_tile(float (&acc)[TM][TB], const float (&a)[TM], const float (&b)[TB]) {
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TB; ++j) acc[i][j] = a[i] * b[j];
}

template <int TM, int TB>
__device__ __forceinline__ void fma_tile(float (&acc)[TM][TB], const float (&a)[TM], const float (&b)[TB]) {
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TB; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
}

template <int N>
__device__ __forceinline__ void ld_vec(float (&v)[N], const float* p) {
#pragma unroll
  for (int q = 0; q < N; q += 4) {
    const float4 f = *reinterpret_cast<const float4*>(p + q);
    v[q] = f.x;
    v[q + 1] = f.y;
    v[q + 2] = f.z;
    v[q + 3] = f.w;
  }
}

template <int N>
__device__ __forceinline__ void st_vec(float* p, const float (&v)[N]) {
#pragma unroll
  for (int q = 0; q < N; q += 4) *reinterpret_cast<float4*>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
}

// Shared-memory layout of an RU x 8 block (rows m): eight-row blocks 72 floats apart and blocks
// an odd multiple of four floats apart, so that lanes on different row blocks and on different
// objects read and write different banks.
__device__ __forceinline__ int row8(int m) { return m * 8 + (m >> 3) * 8; }
__host__ __device__ constexpr int block8(int RU) { return RU * 8 + RU + 4; }

// Slice-major copies of up to six X-side TTs (batch 1): slice i of core k of set t is one
// contiguous RU x RU block As[K][m] at (t tsize + toff[k] + i RU^2) floats of dst, zero-padded, with
// As[K][m] = X_k[K][i][m] (left orientation) or X_k[m][i][K] (right: bit t of `right`). A batch of
// slices is then one bulk copy for the sweeps and the gradient kernel, issued by one thread (staged
// line by line the copies' address arithmetic was a third of the sweeps' instructions). kXsParts
// blocks per (set, core), each a contiguous range of the output; writes coalesced.
struct XSliceArgs {
  const float* src[6];
  long long soff[T3F_MAX_D], toff[T3F_MAX_D];
  int r[T3F_MAX_D + 1], n[T3F_MAX_D];
  int d, RU;
  unsigned right;
  long long tsize;
  float* dst;
};

constexpr int kXsParts = 8;

__global__ void __launch_bounds__(256) k_xslices(const __grid_constant__ XSliceArgs a) {
  const int part = (int)blockIdx.x % kXsParts, tk = (int)blockIdx.x / kXsParts;
  const int t = tk / a.d, k = tk % a.d;
  const int r0 = a.r[k], r1 = a.r[k + 1], n = a.n[k], RU = a.RU, sz = n * RU * RU;
  const bool right = (a.right >> t) & 1u;
  const float* X = a.src[t] + a.soff[k];
  float* Y = a.dst + (long long)t * a.tsize + a.toff[k];
  const int e1 = (int)(((long long)(part + 1) * sz) / kXsParts);
  for (int e = (int)(((long long)part * sz) / kXsParts) + threadIdx.x; e < e1; e += blockDim.x) {
    const int m = e % RU, K = (e / RU) % RU, i = e / (RU * RU);
    const int row = right ? m : K, col = right ? K : m;
    Y[e] = row < r0 && col < r1 ? __ldg(X + ((long long)row * n + i) * r1 + col) : 0.0f;
  }
}

// thread 0: `bytes` (a multiple of 16) from 16-byte aligned src to dst, completing on bar
__device__ __forceinline__ void ps_bulk(float* dst, const float* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(bytes), "r"((unsigned)__cvta_generic_to_shared(bar))
               : "memory");
}

__device__ __forceinline__ void ps_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)),
               "r"(bytes)
               : "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void ps_bar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)));
}

__device__ __forceinline__ bool ps_bar_wait(uint32_t bar, uint32_t parity) {
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

// One step of the accumulate loop: Next += As[K] (x) T[K] (and the fused pair).
template <bool MIXED, int TM, int TB>
__device__ __forceinline__ void acc_step(float (&acc1)[TM][TB], float (&acc2)[TM][TB], const float* As,
                                         const float* Bs1, const float* Bs2, const float* t1, const float* t2) {
  float tv[TB], av[TM];
  ld_vec(tv, t1);
  ld_vec(av, As);
  fma_tile(acc1, av, tv);
  if (MIXED) {
    ld_vec(av, Bs2);
    fma_tile(acc2, av, tv);
    ld_vec(tv, t2);
    ld_vec(av, Bs1);
    fma_tile(acc2, av, tv);
  }
}

template <int RU, bool MIXED, int TM, int TB>
__global__ void __launch_bounds__(TM * TB > 16 ? 256 : 512) k_psweep(const __grid_constant__ PSweepArgs a) {
  extern __shared__ __align__(16) float sm[];
  constexpr int QB = kRZ / TB;       // column blocks
  constexpr int G = (RU / TM) * QB;  // threads per group (a power of two, at most 32)
  constexpr int TS = RU * kRZ;       // floats of one partial
  constexpr int CS = TS + 4;         // object stride of Cur
  constexpr int BS = block8(RU);     // group stride of T
  constexpr int XS = RU * RU;        // floats of a slice
  const TTV& Z = a.Z;
  const int J = a.J, SP = a.SPLIT, d = Z.d;
  const int nmax = Z.nmax;
  const int ZS = kRZ * nmax * kRZ + 4;  // object stride of the Z cores
  const int tid = threadIdx.x;
  const int grp = tid / G, lg = tid % G;
  const bool live = grp < J * SP;       // the last warp may hold spare threads
  const int gi = live ? grp : 0, h = gi / J, ol = gi % J;
  const int qa = lg / QB, qb = lg % QB;
  constexpr int NX = MIXED ? 3 : 1;
  float* Xs = sm;                                   // [2][NX][SP][RU][RU]
  float* Zc = Xs + (size_t)2 * NX * SP * XS;        // [J][8][nmax][8] (object stride ZS)
  float* C1 = Zc + (size_t)J * ZS;                  // [J][8][RU]  (Cur transposed)
  float* C2 = C1 + (size_t)J * CS;                  // mixed only
  float* T1 = C2 + (MIXED ? (size_t)J * CS : 0);    // [SP][J] blocks of RU x 8
  float* T2 = T1 + (size_t)J * SP * BS;             // mixed only
  const float* Zp = static_cast<const float*>(Z.p);
  __shared__ __align__(8) uint64_t zbar, xbar[2];
  if (tid == 0) {
    ps_bar_init(&zbar);
    ps_bar_init(&xbar[0]);
    ps_bar_init(&xbar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // initial partials: 1 (and 0) at the starting interface
  for (int e = tid; e < J * CS; e += blockDim.x) {
    C1[e] = (e % CS) == 0 ? 1.0f : 0.0f;
    if (MIXED) C2[e] = 0.0f;
  }
  for (int o = tid; o < J; o += blockDim.x) {
    const int j0 = a.dir == 0 ? 0 : d, obj = blockIdx.x * J + o;
    if (obj < Z.batch) {
      a.st1[a.ioff[j0] + obj] = 1.0f;
      if (MIXED) a.st2[a.ioff[j0] + obj] = 0.0f;
    }
  }
  __syncthreads();
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!ps_bar_wait((unsigned)__cvta_generic_to_shared(bar), parity) && tid == 0 && a.err)
      atomicExch(a.err, (int)T3F_ERR_TIMEOUT);
  };
  // thread 0: the next batch of X slices, batch xi (counted over all cores) into buffer xi & 1
  int xs = 0, xb = 0, xi = 0;  // sweep step, batch within its core, running index
  auto issue_x = [&]() {
    if (xs >= d) return;
    const int kx = a.dir == 0 ? xs : d - 1 - xs, xn = Z.n[kx], i0 = xb * SP, ns = min(SP, xn - i0);
    const uint32_t bytes = (uint32_t)ns * XS * 4u;
    float* X0 = Xs + (size_t)(xi & 1) * NX * SP * XS;
    uint64_t* bar = &xbar[xi & 1];
    ps_expect(bar, NX * bytes);
    ps_bulk(X0, a.A + a.xoff[kx] + (long long)i0 * XS, bytes, bar);
    if (MIXED) {
      ps_bulk(X0 + (size_t)SP * XS, a.B1 + a.xoff[kx] + (long long)i0 * XS, bytes, bar);
      ps_bulk(X0 + (size_t)2 * SP * XS, a.B2 + a.xoff[kx] + (long long)i0 * XS, bytes, bar);
    }
    ++xi;
    if ((++xb) * SP >= xn) {
      ++xs;
      xb = 0;
    }
  };
  // this CTA's Z cores of sweep step st as [row][i][col], zero-padded to 8 x n x 8. Cores stored
  // that way (ranks 8 x 8, n_k = nmax, 16-byte aligned blocks) land by one bulk copy per object;
  // the others by zero-filling 4-byte copies of the whole block (waited for with the group count):
  // e = ((o * 8 + row) * n + i) * 8 + col, the quotient by n through an exact 32-bit reciprocal
  auto z_bulk = [&](int k) {
    return Z.r[k] == kRZ && Z.r[k + 1] == kRZ && Z.n[k] == nmax && (Z.off[k] & 3) == 0 && (Z.osz[k] & 3) == 0 &&
           (reinterpret_cast<uintptr_t>(Zp) & 15) == 0;
  };
  auto issue_z = [&](int st) {
    const int k = a.dir == 0 ? st : d - 1 - st;
    if (z_bulk(k)) {
      if (tid == 0) {
        const int nv = min(J, Z.batch - (int)blockIdx.x * J);
        const uint32_t bytes = (uint32_t)Z.osz[k] * 4u;
        ps_expect(&zbar, bytes * (uint32_t)nv);
        for (int o = 0; o < nv; ++o)
          ps_bulk(Zc + (size_t)o * ZS, Zp + core_base(Z, k, blockIdx.x * J + o), bytes, &zbar);
      }
      return;
    }
    const int z0 = Z.r[k], z1 = Z.r[k + 1], n = Z.n[k];
    const unsigned mn = 0xffffffffu / (unsigned)n + 1u;
    for (int e = tid; e < J * kRZ * n * kRZ; e += blockDim.x) {
      const unsigned x = (unsigned)e >> 3, q = n == 1 ? x : __umulhi(x, mn);
      const int col = e & 7, i = (int)(x - q * (unsigned)n), row = (int)(q & 7), o = (int)(q >> 3);
      const int ob = blockIdx.x * J + o;
      const bool ok = ob < Z.batch && row < z0 && col < z1;
      const float* src = ok ? Zp + core_base(Z, k, ob) + ((long long)row * n + i) * z1 + col : Zp;
      const unsigned sa = (unsigned)__cvta_generic_to_shared(Zc + (size_t)o * ZS + (row * nmax + i) * kRZ + col);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(src), "r"(ok ? 4 : 0));
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  if (tid == 0) {
    issue_x();
    issue_x();
  }
  issue_z(0);
  uint32_t zph = 0;
  int bt = 0;  // running batch index: buffer bt & 1, its barrier's phase (bt >> 1) & 1
  for (int s = 0; s < d; ++s) {
    const int k = a.dir == 0 ? s : d - 1 - s;
    const int r0 = a.ra[k], r1 = a.ra[k + 1], z0 = Z.r[k], z1 = Z.r[k + 1], n = Z.n[k];
    if (z_bulk(k)) {
      wait(&zbar, zph);
      zph ^= 1u;
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      __syncthreads();
    }
    float acc1[TM][TB], acc2[TM][TB];
#pragma unroll
    for (int x = 0; x < TM; ++x)
#pragma unroll
      for (int y = 0; y < TB; ++y) {
        acc1[x][y] = 0.0f;
        acc2[x][y] = 0.0f;
      }
    float* tb1 = T1 + (size_t)gi * BS + TB * qb;
    float* tb2 = T2 + (size_t)gi * BS + TB * qb;
    for (int ib = 0; ib * SP < n; ++ib, ++bt) {
      const int i = ib * SP + h;
      const bool on = live && i < n;
      // T-step: T[m][b] = sum_K CurT[K][m] Zs[K][b]; Zs[K][b] = Z[K][i][b] (left), Z[b][i][K] (right)
      if (on) {
        float t1[TM][TB], t2[TM][TB];
        const float* zo = Zc + (size_t)ol * ZS + i * kRZ;
        const float* c1p = C1 + (size_t)ol * CS + TM * qa;
        const float* c2p = C2 + (size_t)ol * CS + TM * qa;
        auto step = [&](int K, const float (&zv)[TB]) {
          float cv[TM];
          ld_vec(cv, c1p + K * RU);
          if (K == 0) mul_tile(t1, cv, zv);
          else fma_tile(t1, cv, zv);
          if (MIXED) {
            ld_vec(cv, c2p + K * RU);
            if (K == 0) mul_tile(t2, cv, zv);
            else fma_tile(t2, cv, zv);
          }
        };
        if (a.dir == 0) {
#pragma unroll
          for (int K = 0; K < kRZ; ++K) {
            float zv[TB];
            ld_vec(zv, zo + K * nmax * kRZ + TB * qb);
            step(K, zv);
          }
        } else {
#pragma unroll
          for (int K4 = 0; K4 < kRZ; K4 += 4) {
            float zr[TB][4];
#pragma unroll
            for (int y = 0; y < TB; ++y) ld_vec(zr[y], zo + (TB * qb + y) * nmax * kRZ + K4);
#pragma unroll
            for (int K = 0; K < 4; ++K) {
              float zv[TB];
#pragma unroll
              for (int y = 0; y < TB; ++y) zv[y] = zr[y][K];
              step(K4 + K, zv);
            }
          }
        }
#pragma unroll
        for (int x = 0; x < TM; ++x) {
          st_vec(tb1 + row8(TM * qa + x), t1[x]);
          if (MIXED) st_vec(tb2 + row8(TM * qa + x), t2[x]);
        }
      }
      __syncwarp();
      wait(&xbar[bt & 1], (bt >> 1) & 1);
      if ((ib + 1) * SP >= n) {
        // last batch: every thread is past its reads of the Z cores, the next core's may land
        __syncthreads();
        if (s + 1 < d) issue_z(s + 1);
      }
      // accumulate step: Next[m][b] += sum_K As[K][m] T[K][b], K below the contracted X rank
      // (r0 left, r1 right; the slices are zero beyond it)
      if (on) {
        const float* As = Xs + ((size_t)(bt & 1) * NX * SP + h) * XS + TM * qa;
        const float* Bs1 = As + (size_t)SP * XS;
        const float* Bs2 = Bs1 + (size_t)SP * XS;
        const int kr = a.dir == 0 ? r0 : r1;
        int K = 0;
        for (; K + 8 <= kr; K += 8) {
          const float *tk1 = tb1 + row8(K), *tk2 = tb2 + row8(K);
#pragma unroll
          for (int u = 0; u < 8; ++u)
            acc_step<MIXED>(acc1, acc2, As + (K + u) * RU, Bs1 + (K + u) * RU, Bs2 + (K + u) * RU, tk1 + 8 * u,
                            tk2 + 8 * u);
        }
        for (; K < kr; ++K)
          acc_step<MIXED>(acc1, acc2, As + K * RU, Bs1 + K * RU, Bs2 + K * RU, tb1 + row8(K), tb2 + row8(K));
      }
      __syncwarp();  // the group's T may be rewritten
      if ((ib + 1) * SP < n) {
        __syncthreads();  // this buffer's batch has been consumed
        if (tid == 0) issue_x();
      }
    }
    // sum the SPLIT partial blocks; the new partial becomes CurT and is stored
    if (live) {
#pragma unroll
      for (int x = 0; x < TM; ++x) {
        st_vec(tb1 + row8(TM * qa + x), acc1[x]);
        if (MIXED) st_vec(tb2 + row8(TM * qa + x), acc2[x]);
      }
    }
    __syncthreads();
    if (tid == 0) issue_x();
    {
      const int jn = a.dir == 0 ? k + 1 : k;
      const int rows = a.dir == 0 ? r1 : r0, cols = a.dir == 0 ? z1 : z0;
      for (int e = tid; e < J * TS / 4; e += blockDim.x) {
        const int b = 4 * (e & 1), m = (e >> 1) % RU, o = e / (TS / 4), ob = blockIdx.x * J + o;
        float v1[4] = {0.0f, 0.0f, 0.0f, 0.0f}, v2[4] = {0.0f, 0.0f, 0.0f, 0.0f}, w[4];
        const size_t q = (size_t)o * BS + row8(m) + b;
        for (int hh = 0; hh < SP; ++hh) {
          ld_vec(w, T1 + q + (size_t)hh * J * BS);
#pragma unroll
          for (int y = 0; y < 4; ++y) v1[y] += w[y];
          if (MIXED) {
            ld_vec(w, T2 + q + (size_t)hh * J * BS);
#pragma unroll
            for (int y = 0; y < 4; ++y) v2[y] += w[y];
          }
        }
        const bool in = ob < Z.batch && m < rows;
        const long long g = a.ioff[jn] + (long long)ob * rows * cols + m * cols + b;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          C1[(size_t)o * CS + (b + y) * RU + m] = v1[y];
          if (MIXED) C2[(size_t)o * CS + (b + y) * RU + m] = v2[y];
          if (in && b + y < cols) {
            a.st1[g + y] = v1[y];
            if (MIXED) a.st2[g + y] = v2[y];
          }
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Assembly of project_sum: Zhat_k[a][i][a'] = sum_j c_j sum_b L_k^{(j)}[a][b] S_i^{(j)}[a'][b],
// S_i = R_{k+1} Z_k[:, i, :]^T. One CTA per (core k, range of objects) keeps the whole
// RU x n x RU partial in registers (an 8 x 8 block per thread) and writes it to the
// workspace; a second kernel sums the ranges.
// ---------------------------------------------------------------------------------------
struct PAssembleArgs {
  TTV Z;
  int ra[T3F_MAX_D + 1];
  const float* L;
  const float* R;
  long long ioff[T3F_MAX_D + 1];
  const float* c;
  int nranges, range;   // objects per range
  float* part;          // [nranges][compact X-shaped]
  long long xoff[T3F_MAX_D];
  long long xsize;
};

constexpr int kAsmChunk = 4;

// row stride 8 with four floats between blocks of four rows: lanes four rows apart read
// different banks
__device__ __forceinline__ int row4(int m) { return m * 8 + (m >> 2) * 4; }

// The products read shared memory: 16 floats per 64 multiply-adds in both, 8 x 8 blocks of the
// result and 4 x 8 blocks of S^T (R's four rows held, Z's eight rows read once, for 256
// multiply-adds). The next chunk's inputs (L, R, Z as stored) arrive by asynchronous copies while
// the 8 x 8 blocks are updated (config 5: 430 -> 195 us). nranges makes d x nranges CTAs fill two
// per SM once (passemble_ranges).
template <int RU>
__global__ void __launch_bounds__(512) k_passemble(const __grid_constant__ PAssembleArgs a) {
  extern __shared__ __align__(16) float sm[];
  const TTV& Z = a.Z;
  const int k = blockIdx.x / a.nranges, rg = blockIdx.x % a.nranges;
  const int r0 = a.ra[k], r1 = a.ra[k + 1], z0 = Z.r[k], z1 = Z.r[k + 1], n = Z.n[k];
  constexpr int RL = RU * 8 + RU;              // R block, rows at row4
  constexpr int LL = block8(RU);               // L block, rows at row8
  const int NC = n * RU;                       // (i, a') columns
  const int ZL = kRZ * Z.nmax * kRZ;           // Z block
  const int tid = threadIdx.x, nth = blockDim.x;
  const int ta = tid % (RU / 8), tc = tid / (RU / 8);   // 8 rows a, 8 columns (i, a')
  float* ST = sm;                                        // [chunk][8][nmax RU]  c_j S^T
  float* Rk = ST + (size_t)kAsmChunk * kRZ * Z.nmax * RU;  // R blocks
  float* Zk = Rk + kAsmChunk * RL;                       // Z blocks
  float* Lb = Zk + (size_t)kAsmChunk * ZL;               // two buffers of L blocks
  const float* Zp = static_cast<const float*>(Z.p);
  float acc[8][8];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) acc[x][y] = 0.0f;
  const int jb = rg * a.range, je = min(Z.batch, jb + a.range);
  const unsigned mn = 0xffffffffu / (unsigned)n + 1u;
  auto cp4 = [](float* dst, const float* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(ok ? 4 : 0));
  };
  auto cp16 = [](float* dst, const float* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(ok ? 16 : 0));
  };
  // full rows of eight on 16-byte boundaries: 16-byte copies
  const bool l16 = z0 == kRZ && ((a.ioff[k] & 3) == 0) && (reinterpret_cast<uintptr_t>(a.L) & 15) == 0;
  const bool r16 = z1 == kRZ && ((a.ioff[k + 1] & 3) == 0) && (reinterpret_cast<uintptr_t>(a.R) & 15) == 0;
  const bool z16 = z1 == kRZ && (Z.off[k] & 3) == 0 && (reinterpret_cast<uintptr_t>(Zp) & 15) == 0;
  auto issue = [&](int j0, int buf) {
    float* Lk = Lb + buf * kAsmChunk * LL;
    const int lw = l16 ? 4 : 1, rw = r16 ? 4 : 1, zw = z16 ? 4 : 1;
    for (int e = tid * lw; e < kAsmChunk * RU * kRZ; e += nth * lw) {
      const int b = e % kRZ, m = (e / kRZ) % RU, o = e / (RU * kRZ), j = j0 + o;
      const bool ok = j < je && m < r0 && b < z0;
      const float* src = ok ? a.L + a.ioff[k] + (long long)j * r0 * z0 + m * z0 + b : a.L;
      if (l16) cp16(Lk + o * LL + row8(m) + b, src, ok);
      else cp4(Lk + o * LL + row8(m) + b, src, ok);
    }
    for (int e = tid * rw; e < kAsmChunk * RU * kRZ; e += nth * rw) {
      const int b = e % kRZ, m = (e / kRZ) % RU, o = e / (RU * kRZ), j = j0 + o;
      const bool ok = j < je && m < r1 && b < z1;
      const float* src = ok ? a.R + a.ioff[k + 1] + (long long)j * r1 * z1 + m * z1 + b : a.R;
      if (r16) cp16(Rk + o * RL + row4(m) + b, src, ok);
      else cp4(Rk + o * RL + row4(m) + b, src, ok);
    }
    for (int e = tid * zw; e < kAsmChunk * kRZ * n * kRZ; e += nth * zw) {
      // quotient by n through an exact 32-bit reciprocal (indices < 2^13)
      const unsigned x = (unsigned)e >> 3, q = n == 1 ? x : __umulhi(x, mn);
      const int col = e & 7, i = (int)(x - q * (unsigned)n), row = (int)(q & 7), o = (int)(q >> 3);
      const int j = j0 + o;
      const bool ok = j < je && row < z0 && col < z1;
      const float* src = ok ? Zp + core_base(Z, k, j) + ((long long)row * n + i) * z1 + col : Zp;
      if (z16) cp16(Zk + o * ZL + (row * n + i) * kRZ + col, src, ok);
      else cp4(Zk + o * ZL + (row * n + i) * kRZ + col, src, ok);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  if (jb < je) issue(jb, 0);
  int buf = 0;
  for (int j0 = jb; j0 < je; j0 += kAsmChunk, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;\n" ::);
    __syncthreads();  // the chunk's inputs have landed; ST and the other L buffer are free
    const float* Lk = Lb + buf * kAsmChunk * LL;
    // S^T[o][b][(i, a')] = c_j sum_delta R[a'][delta] Z[b][i][delta], four a' and eight b per item
    for (int e = tid; e < kAsmChunk * NC / 4; e += nth) {
      const int q = e % (RU / 4), x = e / (RU / 4), o = x / n, i = x - o * n;
      const float cj = j0 + o < je ? a.c[j0 + o] : 0.0f;
      float rr[4][8];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        ld_vec(rr[y], Rk + o * RL + row4(4 * q + y));
#pragma unroll
        for (int t = 0; t < 8; ++t) rr[y][t] *= cj;
      }
#pragma unroll
      for (int b = 0; b < kRZ; ++b) {
        float zz[8], sv[4];
        ld_vec(zz, Zk + o * ZL + (b * n + i) * kRZ);
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          float t = rr[y][0] * zz[0];
#pragma unroll
          for (int u = 1; u < 8; ++u) t = fmaf(rr[y][u], zz[u], t);
          sv[y] = t;
        }
        st_vec(ST + ((size_t)o * kRZ + b) * NC + i * RU + 4 * q, sv);
      }
    }
    __syncthreads();  // S^T is complete; the R and Z blocks are free
    if (j0 + kAsmChunk < je) issue(j0 + kAsmChunk, buf ^ 1);
    if (tc * 8 < NC) {
#pragma unroll 1
      for (int o = 0; o < kAsmChunk; ++o)
#pragma unroll
        for (int b4 = 0; b4 < kRZ; b4 += 4) {
          float lr[8][4];
#pragma unroll
          for (int x = 0; x < 8; ++x) ld_vec(lr[x], Lk + o * LL + row8(8 * ta + x) + b4);
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            float sv[8], lv[8];
            ld_vec(sv, ST + ((size_t)o * kRZ + b4 + b) * NC + 8 * tc);
#pragma unroll
            for (int x = 0; x < 8; ++x) lv[x] = lr[x][b];
            fma_tile(acc, lv, sv);
          }
        }
    }
  }
  // write the partial (compact X-shaped layout of core k)
  if (tc * 8 < NC) {
    float* out = a.part + (long long)rg * a.xsize + a.xoff[k];
    const int i = tc * 8 / RU, ap0 = tc * 8 % RU;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int m = 8 * ta + x;
      if (m >= r0) continue;
#pragma unroll
      for (int y = 0; y < 8; ++y)
        if (ap0 + y < r1) out[((long long)m * n + i) * r1 + ap0 + y] = acc[x][y];
    }
  }
}

// ---------------------------------------------------------------------------------------
// Core gradients of the adjoint: dZ_j^k[:, i, :] = c_j (P_k^T X1_i + L_k^T X2_i) with
// X1_i = V_i R_{k+1}, X2_i = W_i R_{k+1} + U_i Q_{k+1}. Cores are independent, so the grid
// covers (object tile, core); slices are split over SPLIT groups as in the sweeps.
// ---------------------------------------------------------------------------------------
struct PGradFastArgs {
  TTV Z;
  const float *U, *V, *W;  // slice-major copies (k_xslices), right orientation
  long long xoff[T3F_MAX_D];
  int ra[T3F_MAX_D + 1];
  const float *L, *R, *P, *Q;
  long long ioff[T3F_MAX_D + 1];
  const float* c;
  float* dZ;
  float* dc;
  int J, SPLIT, ntiles;
  int* err;
};

// A group of RU / 8 lanes owns one (object, slice): a lane forms the 8 x 8 blocks (rows m) of X1
// and X2 in registers (ten 16-byte reads per 192 multiply-adds), multiplies them with its eight
// rows of P and L in place, and the lanes of the group sum their 8 x 8 results with shuffles, each
// keeping its share of the rows beta: no X1 / X2 buffer and no barrier inside a batch of slices
// (config 5: 629 us with 4 x 4 blocks and a buffer, now 370 us, 58 % of the measured FP32 rate).
template <int RU>
__global__ void __launch_bounds__(256) k_pgrad(const __grid_constant__ PGradFastArgs a) {
  extern __shared__ __align__(16) float sm[];
  constexpr int G = RU / 8, BS = block8(RU);
  const TTV& Z = a.Z;
  const int J = a.J, SP = a.SPLIT;
  const int tile = blockIdx.x % a.ntiles, k = blockIdx.x / a.ntiles;
  const int tid = threadIdx.x;
  const int grp = tid / G, qa = tid % G;
  const int h = grp / J, ol = grp % J;  // (threads = J SPLIT G: whole warps where G > 1 and there are shuffles, 16 at the least)
  const int obj = tile * J + ol;
  const bool valid = obj < Z.batch;
  const int r0 = a.ra[k], r1 = a.ra[k + 1], z0 = Z.r[k], z1 = Z.r[k + 1], n = Z.n[k];
  float* Xs = sm;                                   // [2][3][SP][RU][RU]: V^T, W^T, U^T as [K][m]
  float* Pm0 = Xs + (size_t)6 * SP * RU * RU;       // [4][J] blocks: P_k, L_k (rows m), R_{k+1}, Q_{k+1} (rows K)
  const size_t set = (size_t)J * BS;
  if (k == Z.d - 1 && a.dc && h == 0 && qa == 0 && valid) a.dc[obj] = a.P[a.ioff[Z.d] + obj];
  if (!a.dZ) return;
  __shared__ __align__(8) uint64_t xbar[2];
  if (tid == 0) {
    ps_bar_init(&xbar[0]);
    ps_bar_init(&xbar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // thread 0: slices of batch ib (right orientation: As[K][m] = X_k[m][i][K]) into buffer ib & 1
  auto issue_batch = [&](int ib) {
    const int i0 = ib * SP, ns = min(SP, n - i0);
    if (ns <= 0) return;
    const uint32_t bytes = (uint32_t)ns * RU * RU * 4u;
    float* X0 = Xs + (size_t)(ib & 1) * 3 * SP * RU * RU;
    const long long o = a.xoff[k] + (long long)i0 * RU * RU;
    ps_expect(&xbar[ib & 1], 3 * bytes);
    ps_bulk(X0, a.V + o, bytes, &xbar[ib & 1]);
    ps_bulk(X0 + (size_t)SP * RU * RU, a.W + o, bytes, &xbar[ib & 1]);
    ps_bulk(X0 + (size_t)2 * SP * RU * RU, a.U + o, bytes, &xbar[ib & 1]);
  };
  if (tid == 0) {
    issue_batch(0);
    issue_batch(1);
  }
  for (int e = tid; e < J * RU * kRZ; e += blockDim.x) {
    const int b = e % kRZ, m = (e / kRZ) % RU, o = e / (RU * kRZ), ob = tile * J + o;
    const bool lk = ob < Z.batch && m < r0 && b < z0, rk = ob < Z.batch && m < r1 && b < z1;
    const long long li = a.ioff[k] + (long long)ob * r0 * z0 + m * z0 + b;
    const long long ri = a.ioff[k + 1] + (long long)ob * r1 * z1 + m * z1 + b;
    const size_t q = (size_t)o * BS + row8(m) + b;
    Pm0[q] = lk ? a.P[li] : 0.0f;
    Pm0[set + q] = lk ? a.L[li] : 0.0f;
    Pm0[2 * set + q] = rk ? a.R[ri] : 0.0f;
    Pm0[3 * set + q] = rk ? a.Q[ri] : 0.0f;
  }
  const float cj = valid ? a.c[obj] : 0.0f;
  float* outb = valid ? a.dZ + core_base(Z, k, obj) : nullptr;
  const bool v4 = z1 == kRZ && (Z.off[k] & 3) == 0 && (reinterpret_cast<uintptr_t>(a.dZ) & 15) == 0;
  const float* Pm = Pm0 + (size_t)ol * BS;
  const float *Lm = Pm + set, *Rm = Lm + set, *Qm = Rm + set;
  __syncthreads();
  for (int ib = 0; ib * SP < n; ++ib) {
    if (ib > 0) {
      __syncthreads();  // the other buffer is consumed
      if (tid == 0) issue_batch(ib + 1);
    }
    if (!ps_bar_wait((unsigned)__cvta_generic_to_shared(&xbar[ib & 1]), (ib >> 1) & 1) && tid == 0 && a.err)
      atomicExch(a.err, (int)T3F_ERR_TIMEOUT);
    // a group past the last slice repeats it (its lanes take part in the shuffles) and stores nothing
    const int i = ib * SP + h, hs = min(h, n - 1 - ib * SP);
    float x1[8][8], x2[8][8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        x1[x][y] = 0.0f;
        x2[x][y] = 0.0f;
      }
    const float* Vs = Xs + (size_t)((ib & 1) * 3 * SP + hs) * RU * RU + 8 * qa;
    const float* Ws = Vs + (size_t)SP * RU * RU;
    const float* Us = Ws + (size_t)SP * RU * RU;
    // K below the X rank r1 (the staged slices and R, Q are zero beyond it)
#pragma unroll 2
    for (int K = 0; K < r1; ++K) {
      float rv[8], av[8];
      ld_vec(rv, Rm + row8(K));
      ld_vec(av, Vs + K * RU);
      fma_tile(x1, av, rv);
      ld_vec(av, Ws + K * RU);
      fma_tile(x2, av, rv);
      ld_vec(rv, Qm + row8(K));
      ld_vec(av, Us + K * RU);
      fma_tile(x2, av, rv);
    }
    // dZ_i[beta][b] = c_j sum_m (P[m][beta] X1[m][b] + L[m][beta] X2[m][b]), this lane's rows m
    float z[8][8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) z[x][y] = 0.0f;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      float pv[8];
      ld_vec(pv, Pm + row8(8 * qa + m));
      fma_tile(z, pv, x1[m]);
      ld_vec(pv, Lm + row8(8 * qa + m));
      fma_tile(z, pv, x2[m]);
    }
    // sum over the group: halve the rows kept per exchange
    int beta0 = 0;
    constexpr int KEEP = 8 / G;
    if (G == 4) {
      const bool hi = (qa & 2) != 0;
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 8; ++y) {
          const float got = __shfl_xor_sync(0xffffffffu, hi ? z[x][y] : z[x + 4][y], 2);
          z[x][y] = (hi ? z[x + 4][y] : z[x][y]) + got;
        }
      beta0 += hi ? 4 : 0;
    }
    if (G >= 2) {
      constexpr int H = KEEP;
      const bool hi = (qa & 1) != 0;
#pragma unroll
      for (int x = 0; x < H; ++x)
#pragma unroll
        for (int y = 0; y < 8; ++y) {
          const float got = __shfl_xor_sync(0xffffffffu, hi ? z[x][y] : z[x + H][y], 1);
          z[x][y] = (hi ? z[x + H][y] : z[x][y]) + got;
        }
      beta0 += hi ? H : 0;
    }
    if (i < n && valid)
#pragma unroll
      for (int x = 0; x < KEEP; ++x) {
        const int beta = beta0 + x;
        if (beta >= z0) continue;
        float* o = outb + ((long long)beta * n + i) * z1;
#pragma unroll
        for (int y = 0; y < 8; ++y) z[x][y] *= cj;
        if (v4) {
          st_vec(o, z[x]);
        } else {
#pragma unroll
          for (int y = 0; y < 8; ++y)
            if (y < z1) o[y] = z[x][y];
        }
      }
  }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------

static int pick_RU(int r) { return r <= 8 ? 8 : (r <= 16 ? 16 : (r <= 32 ? 32 : 0)); }

bool psweep_supported(const TTV& X, const TTV& Z) {
  return pick_RU(X.rmax) != 0 && Z.rmax <= kRZ && Z.nmax <= 64;
}

static int sm_count() { return device_sm_count(); }

// Objects per CTA, block shape and slices at a time. With at least four objects per SM a thread
// takes 8 x 8 (8 x 4 fused) if that makes four warps; else 4 x 4 blocks with up to 16 slices at a
// time fill a CTA (100 objects: 1 per CTA, 256 threads instead of 64). Few slices leave few threads: 1000
// objects of d = 8, r = 8, X of rank 16, project_sum and its adjoint with the larger blocks against 4 x 4, us:
// n = 2 119, 94 -> 88, 71; n = 4 125, 105 -> 105, 86; n = 8 (X of rank 8) 146, 99 -> 125, 78.
struct PSweepPlan {
  int J, SP;
  bool big;
  size_t smem;
};

static size_t psweep_smem(int RU, bool mixed, int J, int SP, int nmax) {
  const size_t nx = mixed ? 3 : 1, np = mixed ? 2 : 1;
  const size_t f = 2 * nx * SP * RU * RU + (size_t)J * (kRZ * nmax * kRZ + 4) + np * J * (RU * kRZ + 4) +
                   np * J * SP * block8(RU);
  return f * sizeof(float);
}

static PSweepPlan plan_tiles(int RU, bool mixed, int batch, int nmax) {
  PSweepPlan p;
  int j = (batch + sm_count() - 1) / sm_count();
  p.J = j < 1 ? 1 : (j > 8 ? 8 : j);
  int np2 = 1;
  while (np2 < nmax && np2 < 16) np2 *= 2;
  p.big = j >= 4 && p.J * np2 * (RU / 8) * (mixed ? 2 : 1) >= 128;
  const int G = p.big ? (RU / 8) * (mixed ? 2 : 1) : (RU / 4) * 2;
  const int tmax = p.big ? 256 : 512;
  p.SP = np2;
  while (p.SP > 1 && p.J * p.SP * G > tmax) p.SP /= 2;
  while (p.SP > 1 && psweep_smem(RU, mixed, p.J, p.SP, nmax) > 220 * 1024) p.SP /= 2;
  p.smem = psweep_smem(RU, mixed, p.J, p.SP, nmax);
  return p;
}

template <int RU, bool MIXED, int TM, int TB>
static t3f_status launch_psweep_t(PSweepArgs& a, const PSweepPlan& p, cudaStream_t s) {
  if (p.smem > 227 * 1024) return T3F_ERR_UNSUPPORTED;
  auto kern = k_psweep<RU, MIXED, TM, TB>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  const int G = (RU / TM) * (kRZ / TB);
  const unsigned grid = (unsigned)((a.Z.batch + a.J - 1) / a.J);
  kern<<<grid, (unsigned)((a.J * a.SPLIT * G + 31) & ~31), p.smem, s>>>(a);
  return launch_status();
}

template <int RU>
static t3f_status launch_psweep_r(PSweepArgs& a, const PSweepPlan& p, bool mixed, cudaStream_t s) {
  if (!p.big) return mixed ? launch_psweep_t<RU, true, 4, 4>(a, p, s) : launch_psweep_t<RU, false, 4, 4>(a, p, s);
  return mixed ? launch_psweep_t<RU, true, 8, 4>(a, p, s) : launch_psweep_t<RU, false, 8, 8>(a, p, s);
}

// dir 0: left sweep (A = U [, B1 = V, B2 = W]); dir 1: right sweep (A = V [, B1 = U, B2 = W]).
t3f_status run_psweep(const TTV& X, const TTV& Z, int dir, const float* A, const float* B1, const float* B2,
                      float* st1, float* st2, const long long* ioff, cudaStream_t s, int* err) {
  PSweepArgs a;
  memset(&a, 0, sizeof(a));
  a.err = err;
  a.Z = Z;
  a.A = A;
  a.B1 = B1;
  a.B2 = B2;
  xslices_size(X, a.xoff);
  for (int k = 0; k <= X.d; ++k) {
    a.ra[k] = X.r[k];
    a.ioff[k] = ioff[k];
  }
  a.dir = dir;
  a.st1 = st1;
  a.st2 = st2;
  const int RU = pick_RU(X.rmax);
  const bool mixed = st2 != nullptr;
  const PSweepPlan p = plan_tiles(RU, mixed, Z.batch, Z.nmax);
  a.J = p.J;
  a.SPLIT = p.SP;
  switch (RU) {
    case 8: return launch_psweep_r<8>(a, p, mixed, s);
    case 16: return launch_psweep_r<16>(a, p, mixed, s);
    default: return launch_psweep_r<32>(a, p, mixed, s);
  }
}

long long xslices_size(const TTV& X, long long* toff) {
  const int RU = pick_RU(X.rmax);
  long long o = 0;
  for (int k = 0; k < X.d; ++k) {
    if (toff) toff[k] = o;
    o += (long long)X.n[k] * RU * RU;
  }
  return o;
}

t3f_status run_xslices(const TTV& X, const float* const* srcs, unsigned right, int nsets, float* dst, cudaStream_t s) {
  if (nsets < 1 || nsets > 6 || (reinterpret_cast<uintptr_t>(dst) & 15)) return T3F_ERR_ARG;
  XSliceArgs a;
  memset(&a, 0, sizeof(a));
  for (int t = 0; t < nsets; ++t) a.src[t] = srcs[t];
  a.d = X.d;
  a.RU = pick_RU(X.rmax);
  a.right = right;
  a.dst = dst;
  a.tsize = xslices_size(X, a.toff);
  for (int k = 0; k < X.d; ++k) {
    a.soff[k] = X.off[k];
    a.n[k] = X.n[k];
  }
  for (int k = 0; k <= X.d; ++k) a.r[k] = X.r[k];
  k_xslices<<<(unsigned)(nsets * X.d * kXsParts), 256, 0, s>>>(a);
  return launch_status();
}

int passemble_ranges(const TTV& Z) {
  // (core, range) CTAs for one round of two per SM (320 CTAs over 304 places took two rounds)
  int nr = (2 * sm_count()) / Z.d;
  if (nr > Z.batch) nr = Z.batch;
  return nr < 1 ? 1 : nr;
}

template <int RU>
static t3f_status launch_passemble_t(PAssembleArgs& a, cudaStream_t s) {
  const int threads = ((RU / 8) * a.Z.nmax * (RU / 8) + 31) & ~31;
  if (threads > 512) return T3F_ERR_UNSUPPORTED;
  const size_t smem = sizeof(float) * ((size_t)kAsmChunk * kRZ * a.Z.nmax * RU +
                                       (size_t)kAsmChunk * (2 * block8(RU) + RU * 9 + kRZ * a.Z.nmax * kRZ));
  if (smem > 227 * 1024) return T3F_ERR_UNSUPPORTED;
  auto kern = k_passemble<RU>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<(unsigned)(a.Z.d * a.nranges), threads, smem, s>>>(a);
  return launch_status();
}

t3f_status run_passemble(const TTV& X, const TTV& Z, const float* L, const float* R, const long long* ioff,
                         const float* c, float* part, int nranges, cudaStream_t s) {
  PAssembleArgs a;
  memset(&a, 0, sizeof(a));
  a.Z = Z;
  for (int k = 0; k <= X.d; ++k) {
    a.ra[k] = X.r[k];
    a.ioff[k] = ioff[k];
  }
  a.L = L;
  a.R = R;
  a.c = c;
  a.nranges = nranges;
  a.range = (Z.batch + nranges - 1) / nranges;
  a.part = part;
  long long o = 0;
  for (int k = 0; k < X.d; ++k) {
    a.xoff[k] = o;
    o += X.osz[k];
  }
  a.xsize = o;
  switch (pick_RU(X.rmax)) {
    case 8: return launch_passemble_t<8>(a, s);
    case 16: return launch_passemble_t<16>(a, s);
    default: return launch_passemble_t<32>(a, s);
  }
}

template <int RU>
static t3f_status launch_pgrad_t(PGradFastArgs& a, cudaStream_t s) {
  // 16 objects share a CTA's slices (4 where that would leave SMs without a CTA); the rest of
  // the 256 threads take more slices at a time
  constexpr int G = RU / 8;
  a.J = (long long)((a.Z.batch + 15) / 16) * a.Z.d >= sm_count() ? 16 : 4;
  a.SPLIT = 64 / G / a.J * 4;
  while (a.SPLIT > 4 && a.SPLIT / 2 >= a.Z.nmax) a.SPLIT /= 2;
  auto bytes = [&] { return sizeof(float) * ((size_t)6 * a.SPLIT * RU * RU + (size_t)4 * a.J * block8(RU)); };
  while (a.SPLIT > 4 && bytes() > 220 * 1024) a.SPLIT /= 2;
  const size_t smem = bytes();
  a.ntiles = (a.Z.batch + a.J - 1) / a.J;
  auto kern = k_pgrad<RU>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<(unsigned)(a.ntiles * a.Z.d), (unsigned)(a.J * a.SPLIT * G), smem, s>>>(a);
  return launch_status();
}

t3f_status run_pgrad(const TTV& X, const TTV& Z, const float* U, const float* V, const float* W, const float* L,
                     const float* R, const float* P, const float* Q, const long long* ioff, const float* c, float* dZ,
                     float* dc, int* err, cudaStream_t s) {
  PGradFastArgs a;
  memset(&a, 0, sizeof(a));
  a.Z = Z;
  a.U = U;
  a.V = V;
  a.W = W;
  a.err = err;
  xslices_size(X, a.xoff);
  for (int k = 0; k <= X.d; ++k) {
    a.ra[k] = X.r[k];
    a.ioff[k] = ioff[k];
  }
  a.L = L;
  a.R = R;
  a.P = P;
  a.Q = Q;
  a.c = c;
  a.dZ = dZ;
  a.dc = dc;
  const int RU = pick_RU(X.rmax);
  switch (RU) {
    case 8: return launch_pgrad_t<8>(a, s);
    case 16: return launch_pgrad_t<16>(a, s);
    default: return launch_pgrad_t<32>(a, s);
  }
}

}  // namespace t3f
