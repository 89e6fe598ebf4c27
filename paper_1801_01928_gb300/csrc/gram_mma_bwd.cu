// Tensor-core adjoint of the Gram sweep (cotangent of sum_ab g_ab <A_a, B_b>; paper Section 4
// 'gram', batches of Section 3.1) with TF32 or BF16 operands and FP32 accumulation.
//
// For a pair (a, b) with left partials M_k and right partials R_{k+1} around core k,
//   dA_a^k[:, i, :] = sum_b g_ab M_k B_b^k[:, i, :] R_{k+1}^T,
//   dB_b^k[:, i, :] = sum_a g_ab M_k^T A_a^k[:, i, :] R_{k+1}.
// The two are the same contraction seen from either side of a tile: with x the side whose
// gradient is formed and y the other one,
//   T[(x, xi), (y, et')]  = sum_et gM[(x, xi), (y, et)] Y_y,i[et, et']        (one product per y)
//   dX_x,i[xi, xi']       = sum_(y, et') T[(x, xi), (y, et')] R[(x, xi'), (y, et')]
// where gM holds g_xy M (transposed for x = b) and R the right partials, both as 128 x 128
// operands. The partials come from the adjoint sweeps of the tensor-core forward kernel,
// which store every interface in both orientations, already rounded to the operand type and
// laid out as K-major operands (16-byte core matrices packed along K). A work item is (tile,
// core k, side): two bulk copies bring gM_k and R_{k+1} into shared memory, then every mode
// slice i of core k runs the two products. T lives in tensor memory; TF32 feeds it to the
// second product straight from there (the A operand may sit in tensor memory), BF16 copies it
// to shared memory rounded to BF16. The second product runs over all x at once (N = 128) and
// only its diagonal blocks (x, x) are read: lane (x, xi) adds columns x*RX .. of its row to
// the gradient with atomics (other tiles and items share the objects).
#include <algorithm>
#include <string.h>
#include <vector>

#include "gram_mma.cuh"

namespace t3f {

namespace {

// Roles: warps 0-3 stage the y side's slices, warp 4 copies the partials in and issues the products, warps 5-8 (one per tensor-memory lane quarter) copy T to shared memory (BF16),
// warps 9-12 and 13-16 add the gradient products of even and odd slices to memory, warp 17 fetches
// the next items' tables. Slices, T and the gradient product are double-buffered and the items form a
// ring, so every role runs ahead of the next as far as its buffers allow, across items too.
// What bounds it: latency, an item's loads (64 KB) and a slice's chain of product, copy, product,
// addition; the tensor cores work a quarter of the time. 512 objects of ranks 2 .. 64 in groups of 64,
// BF16: 3291 us with the copy of T and the additions (32 sectors an instruction) on the same four
// warps and a barrier per item; 2397 with the additions coalesced, on warps of their own, and one
// commit a product; 1997 with every lane of a waiting warp polling (one lane and a shuffle: 350 cycles
// a wait more) and the products behind an elected lane; 1664 with the item ring.
constexpr int kGThreads = 576;
constexpr int kGProd = 128;           // staging threads (warps 0-3)
constexpr int kGMmaWarp = 4;
constexpr int kGAddWarp = 9;
constexpr int kGFetchWarp = 17;
constexpr int kGItems = 3;            // items in flight
constexpr uint32_t kGTmemCols = 512;  // T[b] at columns 128 b, the gradient product Q[b] at 256 + 128 b
constexpr uint32_t tmem_q(int b) { return 256u + 128u * (uint32_t)b; }

struct GradTcArgs {
  int mode;                   // 0: uniform batches (items from the block index), 1: work list
  TTV A, B;                   // uniform: the kernel's two sides
  int ntb, ntiles;            // uniform: tiles along B, tile count
  float* outA;                // uniform: gradients of the kernel's A / B side, packed like A / B (nullable)
  float* outB;
  // work-list mode: ragged objects in rank-sorted positions
  const void* cores;
  const long long* off;       // [pos][dmax] element offset of core k
  const int* rk;              // [pos][dmax + 1]
  int dmax;
  const int* nmodes;          // [group][dmax]
  const int* gd;              // [group] d
  const int* items;           // the sweep kernels' tiles: [item][8] group, a0, na, b0, nb, RA, sym, RB
  const int* gitems;          // [item][4]: tile, core, side, 0
  int ngitems;
  int* head;
  float* dX;                  // gradient in the layout of the ragged cores
  // scratch of the adjoint sweeps
  const char* scr;
  const long long* soff;      // work list: slot offset of each tile (in slot orientations)
  long long sstride;          // uniform: slot orientations per tile
  int* err;
  uint32_t smem_bytes;
};

// A work item as its roles read it. x: the objects whose gradient is formed, y: the others.
struct GradItem {
  const char *gm, *rp;            // gM_k and R_{k+1} in the orientation whose rows are the x objects
  int valid, n, nx, RX, RY, side;  // (the arrays' base pointers come from the arguments: known to be global)
  long long ybase[8], xbase[8];
  int yrl[8], yrr[8], xrl[8], xrr[8];
};

struct GradShared {
  uint64_t ldm, ldr;              // copies of gM and of R
  uint64_t ifull[kGItems], iempty[kGItems];  // item ring: fetched / read by every role
  uint64_t sfull[2];              // slice ring: staged
  uint64_t tdone[2];              // T buffers: written, and the slice buffers read
  uint64_t tfree[2], tsfull[2];   // BF16: T buffers copied, their shared-memory copies written
  uint64_t qdone[2], qfree[2];    // gradient product buffers: written (and T, or its copy, read) / added
  uint64_t fin;                   // drain after a timeout
  GradItem it[kGItems];
  uint32_t tmem;
};

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// 32 lanes x 32 consecutive columns, without waiting (tcgen05.wait::ld before use)
__device__ __forceinline__ void tmem_ld32_nw(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

// every lane polls (bounded); the warp goes on together
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}

constexpr uint32_t kGStg = 33;  // row pitch of an epilogue warp's 32 x 32 block

// Shared-memory plan for element size es: gM, R, two slice buffers, (BF16) two shared-memory copies
// of T, and a 32 x 32 block per adding warp.
__host__ __device__ constexpr uint32_t grad_slot(int es) { return 128u * 128u * (uint32_t)es; }
__host__ __device__ constexpr uint32_t grad_slice(int es) { return 128u * 64u * (uint32_t)es; }
__host__ __device__ constexpr uint32_t grad_smem(int es) {
  return 2u * grad_slot(es) + 2u * grad_slice(es) + (es == 2 ? 2u * grad_slot(es) : 0u) + 8u * 32u * kGStg * 4u;
}

__device__ __forceinline__ int rank_class(int r) { return r <= 16 ? 16 : (r <= 32 ? 32 : 64); }

// ---- warp kGFetchWarp: the items of this CTA in order, then one that ends the loop
template <int KIND, typename ST>
__device__ bool grad_fetch(const GradTcArgs& g, GradShared& sh) {
  constexpr uint32_t SLOT = grad_slot(OpT<KIND>::ES);
  const int lane = threadIdx.x & 31;
  long long next = blockIdx.x;  // uniform: every gridDim.x-th item
  for (uint32_t it = 0;; ++it) {
    const uint32_t p = it % kGItems;
    if (it >= kGItems && !warp_wait(su32(&sh.iempty[p]), (it / kGItems - 1u) & 1u)) return false;
    __syncwarp();
    GradItem& I = sh.it[p];
    bool valid;
    int grp = 0, a0, na, b0, nb, RA, RB, k = 0, side = 0, d, t = 0;
    a0 = na = b0 = nb = RA = RB = d = 0;
    if (g.mode == 0) {
      d = g.A.d;
      const long long half = (long long)g.ntiles * d;  // items of one side
      valid = next < half * ((g.outA ? 1 : 0) + (g.outB ? 1 : 0));
      if (valid) {
        side = !g.outA || next >= half ? 1 : 0;
        t = (int)(next % half / d);
        k = (int)(next % d);
        RA = rank_class(g.A.rmax);
        RB = rank_class(g.B.rmax);
        const int TA = 128 / RA, TB = 128 / RB;
        a0 = (t / g.ntb) * TA;
        b0 = (t % g.ntb) * TB;
        na = min(TA, g.A.batch - a0);
        nb = min(TB, g.B.batch - b0);
        next += gridDim.x;
      }
    } else {
      int w = 0;
      if (lane == 0) w = atomicAdd(g.head, 1);
      w = __shfl_sync(0xffffffffu, w, 0);
      valid = w < g.ngitems;
      if (valid) {
        t = g.gitems[w * 4];
        k = g.gitems[w * 4 + 1];
        side = g.gitems[w * 4 + 2];
        const int* im = g.items + t * 8;
        grp = im[0];
        a0 = im[1];
        na = im[2];
        b0 = im[3];
        nb = im[4];
        RA = im[5];
        RB = im[7];
        d = g.gd[grp];
      }
    }
    if (valid) {
      const int x0 = side ? b0 : a0, nx = side ? nb : na, y0 = side ? a0 : b0, ny = side ? na : nb;
      if (lane < 16) {
        const int o = lane & 7, isx = lane >> 3, cnt = isx ? nx : ny, o0 = isx ? x0 : y0;
        long long base = 0;
        int rl = 0, rr = 0;
        if (o < cnt) {
          if (g.mode == 0) {
            const TTV& V = (isx ? side : !side) ? g.B : g.A;
            base = V.off[k] + (long long)(o0 + o) * V.osz[k];
            rl = V.r[k];
            rr = V.r[k + 1];
          } else {
            const int pos = o0 + o;
            base = g.off[(long long)pos * g.dmax + k];
            rl = g.rk[(long long)pos * (g.dmax + 1) + k];
            rr = g.rk[(long long)pos * (g.dmax + 1) + k + 1];
          }
        }
        (isx ? I.xbase : I.ybase)[o] = base;
        (isx ? I.xrl : I.yrl)[o] = rl;
        (isx ? I.xrr : I.yrr)[o] = rr;
      } else if (lane == 16) {
        const char* slots = g.scr + (size_t)(g.mode == 0 ? (long long)t * g.sstride : g.soff[t]) * SLOT;
        I.gm = slots + (size_t)(k * 2 + side) * SLOT;
        I.rp = slots + (size_t)((d + k) * 2 + side) * SLOT;
        I.side = side;
        I.n = g.mode == 0 ? g.A.n[k] : g.nmodes[grp * g.dmax + k];
        I.nx = nx;
        I.RX = side ? RB : RA;
        I.RY = side ? RA : RB;
      }
    }
    if (lane == 16) I.valid = valid ? 1 : 0;
    mbar_arrive(su32(&sh.ifull[p]));
    if (!valid) return true;
  }
}

// The next item of a role, nullptr on a timeout.
__device__ __forceinline__ GradItem* grad_next(GradShared& sh, uint32_t it) {
  const uint32_t p = it % kGItems;
  if (!warp_wait(su32(&sh.ifull[p]), (it / kGItems) & 1u)) return nullptr;
  __syncwarp();
  return &sh.it[p];
}

__device__ __forceinline__ void grad_release(GradShared& sh, uint32_t it) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(su32(&sh.iempty[it % kGItems]));
}

// ---- staging: the slices of the y side (rows et' = right rank, K = et = left rank). gs counts the
// slices of the items before (buffer index and barrier phases continue across items).
template <int KIND, int RY, typename ST>
__device__ bool grad_stage(const GradTcArgs& g, const GradItem& I, char* ysl, GradShared& sh, uint32_t gs) {
  using O = OpT<KIND>;
  constexpr int ES = O::ES, T = 16 / ES, TY = 128 / RY;
  constexpr uint32_t SBOY = (uint32_t)(RY / T) * 128u;  // slice operand of one y: bytes per 8 rows
  constexpr uint32_t YSZ = (uint32_t)RY * RY * ES;      // bytes of one y's slice operand
  constexpr int KGY = RY / T, UPY = TY * RY * KGY / kGProd, USY = kGProd / RY;
  static_assert(UPY * kGProd == TY * RY * KGY, "staging split");
  const int tid = threadIdx.x, sy = tid % RY, uy = tid / RY, n = I.n;
  const ST* const Yp = static_cast<const ST*>(g.mode == 0 ? (I.side ? g.A.p : g.B.p) : g.cores);
  uint32_t py[UPY][T];
  auto load_slice = [&](int i) {
#pragma unroll
    for (int j = 0; j < UPY; ++j) {
      const int w = uy + j * USY, o = w / KGY, c0 = (w % KGY) * T;
      const int rl = I.yrl[o], rr = I.yrr[o], stp = n * rr;
      const ST* ptr = Yp + I.ybase[o] + (long long)c0 * stp + (long long)i * rr + sy;
      const bool rok = sy < rr;
#pragma unroll
      for (int t = 0; t < T; ++t) {
        py[j][t] = (rok && c0 + t < rl) ? ld_raw<ST>(ptr) : 0u;
        ptr += stp;
      }
    }
  };
  load_slice(0);
  for (int i = 0; i < n; ++i) {
    const uint32_t gg = gs + (uint32_t)i, b = gg & 1u;
    if (gg >= 2u && !warp_wait(su32(&sh.tdone[b]), ((gg >> 1) - 1u) & 1u)) return false;
    char* const buf = ysl + b * grad_slice(ES);
#pragma unroll
    for (int j = 0; j < UPY; ++j) {
      const int w = uy + j * USY, o = w / KGY, cg = w % KGY;
      const uint32_t off = (uint32_t)(sy >> 3) * SBOY + (uint32_t)cg * 128u + (uint32_t)(sy & 7) * 16u;
      *reinterpret_cast<uint4*>(buf + o * YSZ + off) = pack_raw<KIND, ST, T>(py[j]);
    }
    async_fence();
    mbar_arrive(su32(&sh.sfull[b]));
    if (i + 1 < n) load_slice(i + 1);
  }
  return true;
}

// ---- BF16: T(i) -> shared memory (rows (x, xi), K = (y, et')), rounded to BF16
__device__ bool grad_copy_t(int n, char* ts, GradShared& sh, uint32_t tmem, uint32_t gs) {
  using O = OpT<1>;
  constexpr uint32_t SLOT = grad_slot(2), SBO = 16u * 128u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, qd = warp & 3, row = qd * 32 + lane;
  for (int i = 0; i < n; ++i) {
    const uint32_t gg = gs + (uint32_t)i, b = gg & 1u;
    if (!warp_wait(su32(&sh.tdone[b]), (gg >> 1) & 1u)) return false;
    if (gg >= 2u && !warp_wait(su32(&sh.qdone[b]), ((gg >> 1) - 1u) & 1u)) return false;
    tc_after();
    char* const dst = ts + b * SLOT;
#pragma unroll
    for (int cc = 0; cc < 128; cc += 64) {
      uint32_t r[2][32];
      tmem_ld32_nw(tmem + b * 128u + ((uint32_t)(qd * 32) << 16) + (uint32_t)cc, r[0]);
      tmem_ld32_nw(tmem + b * 128u + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cc + 32), r[1]);
      tmem_wait_ld();
#pragma unroll
      for (int hh = 0; hh < 8; ++hh) {
        float u[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) u[t] = __uint_as_float(r[hh >> 2][(hh & 3) * 8 + t]);
        *reinterpret_cast<uint4*>(dst + (uint32_t)(row >> 3) * SBO + (uint32_t)((cc + hh * 8) / 8) * 128u +
                                  (uint32_t)(row & 7) * 16u) = O::pack(u);
      }
    }
    async_fence();
    tc_before();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(su32(&sh.tsfull[b]));
      mbar_arrive(su32(&sh.tfree[b]));
    }
  }
  return true;
}

// ---- products of one item. The whole warp walks the loop and one elected lane issues, with the buffer
// index known at compile time.
template <int KIND, int RY, int B>
__device__ __forceinline__ void issue_first(char* sm, GradShared& sh, uint32_t tmem) {
  using O = OpT<KIND>;
  constexpr int ES = O::ES, T = 16 / ES, TY = 128 / RY;
  constexpr uint32_t SBO = (128u / T) * 128u;          // full operand: bytes per 8 rows
  constexpr uint32_t SBOY = (uint32_t)(RY / T) * 128u;
  constexpr uint32_t YSZ = (uint32_t)RY * RY * ES, ID1 = idesc(O::FMT, RY);
  const uint64_t da = sdesc2(su32(sm), 128u, SBO);
  const uint64_t db = sdesc2(su32(sm + 2 * grad_slot(ES) + B * grad_slice(ES)), 128u, SBOY);
  if (elect_one()) {
    // T[(x, xi), (y, et')] = sum_et gM[(x, xi), (y, et)] Y_y,i[et, et'] for every y
#pragma unroll
    for (int y = 0; y < TY; ++y)
#pragma unroll
      for (int kk = 0; kk < RY / O::KI; ++kk)
        mma<KIND>(tmem + B * 128u + (uint32_t)(y * RY), da + (uint32_t)((y * RY + kk * O::KI) / T) * 8u,
                  db + ((uint32_t)y * YSZ + (uint32_t)(kk * O::KI / T) * 128u) / 16u, ID1, kk > 0 ? 1u : 0u);
    mma_commit(su32(&sh.tdone[B]));
  }
}

// T R^T over all x at once (N = 128, K = 128) into Q[B]; only its diagonal blocks (x, x) are read --
// the same products as one N = RX product per x, in 128 / KI instructions instead of TX times as many
template <int KIND, int B>
__device__ __forceinline__ void issue_second(char* sm, GradShared& sh, uint32_t tmem) {
  using O = OpT<KIND>;
  constexpr int ES = O::ES, T = 16 / ES;
  constexpr uint32_t SBO = (128u / T) * 128u, ID2 = idesc(O::FMT, 128);
  const uint64_t db = sdesc2(su32(sm + grad_slot(ES)), 128u, SBO);
  const uint64_t da = sdesc2(su32(sm + (2 + B) * grad_slot(ES) + 2 * grad_slice(ES)), 128u, SBO);
  if (elect_one()) {
#pragma unroll
    for (int kk = 0; kk < 128 / O::KI; ++kk) {
      constexpr uint32_t q = tmem_q(B);
      const uint32_t off = (uint32_t)(kk * O::KI / T) * 8u;
      if constexpr (KIND == 0)
        mma_ts_tf32(tmem + q, tmem + B * 128u + (uint32_t)(kk * O::KI), db + off, ID2, kk > 0 ? 1u : 0u);
      else
        mma<KIND>(tmem + q, da + off, db + off, ID2, kk > 0 ? 1u : 0u);
    }
    mma_commit(su32(&sh.qdone[B]));
  }
}

template <int KIND, int RY>
__device__ bool grad_products(int n, char* sm, GradShared& sh, uint32_t tmem, uint32_t gs, uint32_t ldr_phase) {
  for (int i = 0; i <= n; ++i) {
    if (i < n) {
      const uint32_t gg = gs + (uint32_t)i, b = gg & 1u;
      if (!warp_wait(su32(&sh.sfull[b]), (gg >> 1) & 1u)) return false;
      if (gg >= 2u && !warp_wait(su32(KIND == 0 ? &sh.qdone[b] : &sh.tfree[b]), ((gg >> 1) - 1u) & 1u)) return false;
      tc_after();
      if (b) issue_first<KIND, RY, 1>(sm, sh, tmem);
      else issue_first<KIND, RY, 0>(sm, sh, tmem);
    }
    if (i >= 1) {
      const uint32_t gj = gs + (uint32_t)(i - 1), bj = gj & 1u;
      if (i == 1 && !warp_wait(su32(&sh.ldr), ldr_phase)) return false;
      if (!warp_wait(su32(KIND == 0 ? &sh.tdone[bj] : &sh.tsfull[bj]), (gj >> 1) & 1u)) return false;
      if (gj >= 2u && !warp_wait(su32(&sh.qfree[bj]), ((gj >> 1) - 1u) & 1u)) return false;
      tc_after();
      if (bj) issue_second<KIND, 1>(sm, sh, tmem);
      else issue_second<KIND, 0>(sm, sh, tmem);
    }
  }
  return true;
}

// ---- adding warps: lane quarter qd of the gradient product buffer `set` (slices of that parity).
// The quarter's diagonal blocks go to dX_x[xi, j, :] along the columns, through shared memory: lanes
// along the rows of tensor memory would send every lane's word to its own sector.
template <int KIND, int RX>
__device__ bool grad_add(const GradTcArgs& g, const GradItem& I, float* stg, GradShared& sh, uint32_t tmem,
                         uint32_t it, uint32_t gs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, qd = warp & 3, n = I.n;
  const uint32_t set = (uint32_t)(warp - kGAddWarp) >> 2;
  constexpr int QCOLS = RX < 32 ? 32 : RX;  // columns of the x blocks this quarter's lanes cover
  const int cstart = ((qd * 32) / RX) * RX;
  // the quarter's rows: NB objects (or half of one), rows xi0 .. of them
  constexpr int NB = RX < 32 ? 2 : 1;
  const int xi0 = (qd * 32) % RX;
  int xrl[NB], xrr[NB];  // rows and columns of an object here
  long long xrow[NB];
  float* const outX = g.mode == 0 ? (I.side ? g.outB : g.outA) : g.dX;
#pragma unroll
  for (int o = 0; o < NB; ++o) {
    const int x = (qd * 32) / RX + o;
    xrl[o] = x < I.nx ? min(I.xrl[x] - xi0, 32) : 0;
    xrr[o] = I.xrr[x];
    xrow[o] = I.xbase[x] + (long long)xi0 * n * xrr[o];
  }
  grad_release(sh, it);
  for (int j = (int)((gs ^ set) & 1u); j < n; j += 2) {
    const uint32_t gj = gs + (uint32_t)j;
    if (!warp_wait(su32(&sh.qdone[set]), (gj >> 1) & 1u)) return false;
    tc_after();
#pragma unroll
    for (int h = 0; h < QCOLS / 32; ++h) {
      uint32_t r[32];
      tmem_ld32_nw(tmem + 256u + set * 128u + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cstart + h * 32), r);
      tmem_wait_ld();
      if (h + 1 == QCOLS / 32) {
        tc_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(&sh.qfree[set]));
      }
#pragma unroll
      for (int t = 0; t < 32; ++t) stg[lane * kGStg + t] = __uint_as_float(r[t]);
      __syncwarp();
#pragma unroll
      for (int o = 0; o < NB; ++o) {
        const int wd = min(32, xrr[o] - h * 32);  // columns of this half
        if (wd > 0) {
          const int lg = wd > 1 ? 32 - __clz(wd - 1) : 0;  // 2^lg lanes a row
          const int col = lane & ((1 << lg) - 1), stp = 32 >> lg, r0 = lane >> lg;
          float* dst = outX + xrow[o] + (long long)(r0 * n + j) * xrr[o] + h * 32 + col;
          const long long dstep = (long long)stp * n * xrr[o];
          const float* src = stg + (o * 16 + r0) * kGStg + o * 16 + col;
          const int cnt = col < wd && r0 < xrl[o] ? (xrl[o] - r0 + stp - 1) >> (5 - lg) : 0;
#pragma unroll 8
          for (int q = 0; q < cnt; ++q) {
            atomicAdd(dst, src[q * stp * kGStg]);
            dst += dstep;
          }
        }
      }
      __syncwarp();
    }
  }
  return true;
}

template <int KIND>
__device__ __forceinline__ void grad_setup(GradShared& sh, char* sm, uint32_t bytes) {
  const int tid = threadIdx.x, warp = tid >> 5;
  for (uint32_t e = (uint32_t)tid * 16u; e < bytes; e += kGThreads * 16u)
    *reinterpret_cast<uint4*>(sm + e) = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    auto init = [](uint64_t* b, uint32_t count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count));
    };
    init(&sh.ldm, 1);
    init(&sh.ldr, 1);
    init(&sh.fin, 1);
    for (int b = 0; b < kGItems; ++b) {
      init(&sh.ifull[b], 32);
      init(&sh.iempty[b], kGFetchWarp);  // one arrival of every other warp
    }
    for (int b = 0; b < 2; ++b) {
      init(&sh.sfull[b], kGProd);
      init(&sh.tdone[b], 1);
      init(&sh.tfree[b], 4);
      init(&sh.tsfull[b], 4);
      init(&sh.qdone[b], 1);
      init(&sh.qfree[b], 4);
    }
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sh.tmem)),
                 "r"(kGTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  async_fence();
  tc_before();
  __syncthreads();
  tc_after();
}

// nm, nr: copies of gM and of R that this thread issued.
__device__ __forceinline__ void grad_teardown(const GradTcArgs& g, GradShared& sh, bool failed, uint32_t nm,
                                              uint32_t nr) {
  if (failed) {
    // a wait ran out: report it, then let whatever is still in flight finish (bounded) before
    // the tensor memory is released -- the products through one more commit, the last copies
    if (threadIdx.x == 0 && g.err) atomicExch(g.err, (int)T3F_ERR_TIMEOUT);
    // (the lane that issued the products commits them)
    if ((threadIdx.x >> 5) == kGMmaWarp && elect_one()) {
      mma_commit(su32(&sh.fin));
      mbar_wait(su32(&sh.fin), 0);
      if (nm > 0) mbar_wait(su32(&sh.ldm), (nm - 1u) & 1u);
      if (nr > 0) mbar_wait(su32(&sh.ldr), (nr - 1u) & 1u);
    }
  }
  tc_before();
  __syncthreads();
  tc_after();
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem), "r"(kGTmemCols));
}

#define T3F_GRAD_BY_RANK(R, CALL)                          \
  switch (R) {                                             \
    case 16: { constexpr int RR = 16; ok = CALL; } break;  \
    case 32: { constexpr int RR = 32; ok = CALL; } break;  \
    default: { constexpr int RR = 64; ok = CALL; } break;  \
  }

// Persistent CTAs: the (tile, core, side) items of uniform batches at a fixed stride (they cost the
// same), those of a work list through an atomic counter.
template <int KIND, typename ST>
__global__ void __launch_bounds__(kGThreads, 1) k_gram_tc_grad(const __grid_constant__ GradTcArgs g) {
  extern __shared__ __align__(128) char sm[];
  __shared__ __align__(16) GradShared sh;
  using O = OpT<KIND>;
  constexpr int ES = O::ES;
  constexpr uint32_t SLOT = grad_slot(ES);
  grad_setup<KIND>(sh, sm, g.smem_bytes);
  const int warp = threadIdx.x >> 5;
  const uint32_t tmem = sh.tmem;
  const bool lead = (threadIdx.x & 31) == 0;
  char* const ysl = sm + 2 * SLOT;
  char* const ts = ysl + 2 * grad_slice(ES);
  bool ok = true;
  uint32_t gs = 0, nm = 0, nr = 0;  // slices of the items before, copies issued
  if (warp == kGFetchWarp) {
    ok = grad_fetch<KIND, ST>(g, sh);
  } else {
    for (uint32_t it = 0; ok; ++it) {
      GradItem* const I = grad_next(sh, it);
      if (!I) {
        ok = false;
        break;
      }
      if (!I->valid) break;
      const int n = I->n;
      if (warp < kGMmaWarp) {
        T3F_GRAD_BY_RANK(I->RY, (grad_stage<KIND, RR, ST>(g, *I, ysl, sh, gs)))
        grad_release(sh, it);
      } else if (warp == kGMmaWarp) {
        const int RY = I->RY;
        const char *gm = I->gm, *rp = I->rp;
        grad_release(sh, it);
        // the first products of the last item are complete (its copies of T were awaited, or T
        // itself); the second ones, which read R, are waited for here
        if (lead) {
          expect_tx(su32(&sh.ldm), SLOT);
          bulk_g2s(su32(sm), gm, SLOT, su32(&sh.ldm));
        }
        ++nm;
        if (gs > 0) ok = warp_wait(su32(&sh.qdone[(gs - 1u) & 1u]), ((gs - 1u) >> 1) & 1u);
        if (ok) {
          if (lead) {
            expect_tx(su32(&sh.ldr), SLOT);
            bulk_g2s(su32(sm + SLOT), rp, SLOT, su32(&sh.ldr));
          }
          ++nr;
          ok = warp_wait(su32(&sh.ldm), (nm - 1u) & 1u);
        }
        if (ok) T3F_GRAD_BY_RANK(RY, (grad_products<KIND, RR>(n, sm, sh, tmem, gs, (nr - 1u) & 1u)))
      } else if (warp < kGAddWarp) {
        grad_release(sh, it);
        if constexpr (KIND == 1) ok = grad_copy_t(n, ts, sh, tmem, gs);
      } else {
        float* const stg = reinterpret_cast<float*>(ts + (KIND == 1 ? 2 * SLOT : 0)) + (warp - kGAddWarp) * 32 * kGStg;
        T3F_GRAD_BY_RANK(I->RX, (grad_add<KIND, RR>(g, *I, stg, sh, tmem, it, gs)))
      }
      gs += (uint32_t)n;
    }
  }
  const bool failed = __syncthreads_or(!ok) != 0;
  grad_teardown(g, sh, failed, nm, nr);
}
#undef T3F_GRAD_BY_RANK

template <int KIND, typename ST>
t3f_status launch_grad(const GradTcArgs& g0, int grid, cudaStream_t s) {
  GradTcArgs g = g0;
  g.smem_bytes = grad_smem(OpT<KIND>::ES);
  if (grid <= 0) return T3F_OK;
  auto kern = k_gram_tc_grad<KIND, ST>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem_bytes) != cudaSuccess)
    return T3F_ERR_CUDA;
  kern<<<grid, kGThreads, g.smem_bytes, s>>>(g);
  return launch_status();
}

template <typename F>
t3f_status by_math(int math, int dtype, F&& f) {
  if (math == T3F_MATH_TF32) {
    if (dtype != T3F_F32) return T3F_ERR_DTYPE;
    return f(std::integral_constant<int, 0>{}, (float*)nullptr);
  }
  if (dtype == T3F_BF16) return f(std::integral_constant<int, 1>{}, (__nv_bfloat16*)nullptr);
  return f(std::integral_constant<int, 1>{}, (float*)nullptr);
}

}  // namespace

// sweeps of gram_mma.cu
t3f_status run_gram_mma_sweeps(const TTV& A, const TTV& B, int swap, const float* dG, int ldg, int math, char* scr,
                               long long sstride, int* err, cudaStream_t s);
t3f_status launch_gram_mma_sweeps_list(int math, const void* cores, int dtype, int dmax, const long long* off,
                                       const int* rk, const int* nmodes, const int* items, int nitems, int* head,
                                       const int* gstart, const int* gd, const long long* gout_off, const int* perm,
                                       const float* dout, char* scr, const long long* soff, int* err, cudaStream_t s);

// Slot orientations (128 x 128 operands) one tile of a uniform pair of batches keeps: both
// directions, d interfaces each, two orientations.
long long gram_tc_bwd_slots(const TTV& A) { return 4LL * A.d; }

size_t gram_tc_bwd_tiles(const TTV& A, const TTV& B) {
  const int RA = A.rmax <= 16 ? 16 : (A.rmax <= 32 ? 32 : 64), RB = B.rmax <= 16 ? 16 : (B.rmax <= 32 ? 32 : 64);
  const bool swap = RA > RB;
  const int ra = std::min(RA, RB), rb = std::max(RA, RB);
  const TTV& KA = swap ? B : A;
  const TTV& KB = swap ? A : B;
  return (size_t)((KA.batch + 128 / ra - 1) / (128 / ra)) * (size_t)((KB.batch + 128 / rb - 1) / (128 / rb));
}

// Workspace of the uniform tensor-core adjoint: the error word, then the slots (TF32 size,
// which also covers BF16).
size_t ws_gram_bwd_tc(const TTV& A, const TTV& B) {
  return kWsHeader + gram_tc_bwd_tiles(A, B) * (size_t)gram_tc_bwd_slots(A) * 128u * 128u * 4u;
}

// Uniform tensor-core adjoint: the sweeps into the scratch, then the gradient products.
// dA / dB (nullable) are zeroed here. scr must hold gram_tc_bwd_tiles * gram_tc_bwd_slots
// orientations of 128 x 128 x 4 bytes.
t3f_status run_gram_tc_backward(const TTV& A, const TTV& B, const float* dG, float* dA, float* dB, int math,
                                char* scr, int* err, cudaStream_t s) {
  const int RA = A.rmax <= 16 ? 16 : (A.rmax <= 32 ? 32 : 64), RB = B.rmax <= 16 ? 16 : (B.rmax <= 32 ? 32 : 64);
  const int swap = RA > RB ? 1 : 0;
  const TTV& KA = swap ? B : A;
  const TTV& KB = swap ? A : B;
  if (dA && cudaMemsetAsync(dA, 0, sizeof(float) * (size_t)(A.off[A.d - 1] + (long long)A.batch * A.osz[A.d - 1]), s) != cudaSuccess)
    return T3F_ERR_CUDA;
  if (dB && cudaMemsetAsync(dB, 0, sizeof(float) * (size_t)(B.off[B.d - 1] + (long long)B.batch * B.osz[B.d - 1]), s) != cudaSuccess)
    return T3F_ERR_CUDA;
  if (A.batch == 0 || B.batch == 0) return T3F_OK;
  const long long sstride = gram_tc_bwd_slots(A);
  T3F_CHECK(run_gram_mma_sweeps(KA, KB, swap, dG, B.batch, math, scr, sstride, err, s));
  GradTcArgs g;
  memset(&g, 0, sizeof(g));
  g.mode = 0;
  g.A = KA;
  g.B = KB;
  const int TB = 128 / std::max(RA, RB);
  g.ntb = (KB.batch + TB - 1) / TB;
  g.ntiles = (int)gram_tc_bwd_tiles(A, B);
  g.outA = swap ? dB : dA;
  g.outB = swap ? dA : dB;
  g.scr = scr;
  g.sstride = sstride;
  g.err = err;
  const long long items = (long long)g.ntiles * A.d * 2;
  if (items > 0x7fffffffLL) return T3F_ERR_UNSUPPORTED;
  const long long grid = std::min<long long>(items, device_sm_count());
  return by_math(math, A.dtype, [&](auto kind, auto* st) -> t3f_status {
    using ST = std::remove_pointer_t<decltype(st)>;
    return launch_grad<decltype(kind)::value, ST>(g, (int)grid, s);
  });
}

// Work-list tensor-core adjoint over a ragged collection: the sweeps over the tensor-core tile
// list (both directions), then the (tile, core, side) gradient items. dX must be zeroed.
t3f_status launch_gram_tc_backward_list(int math, const void* cores, int dtype, int dmax, const long long* off,
                                        const int* rk, const int* nmodes, const int* items, int nitems,
                                        const int* gitems, int ngitems, int* heads, const int* gstart,
                                        const int* gd, const long long* gout_off, const int* perm,
                                        const float* dout, float* dX, char* scr, const long long* soff, int* err,
                                        cudaStream_t s) {
  if (nitems <= 0) return T3F_OK;
  T3F_CHECK(launch_gram_mma_sweeps_list(math, cores, dtype, dmax, off, rk, nmodes, items, nitems, heads, gstart, gd,
                                        gout_off, perm, dout, scr, soff, err, s));
  GradTcArgs g;
  memset(&g, 0, sizeof(g));
  g.mode = 1;
  g.cores = cores;
  g.off = off;
  g.rk = rk;
  g.dmax = dmax;
  g.nmodes = nmodes;
  g.gd = gd;
  g.items = items;
  g.gitems = gitems;
  g.ngitems = ngitems;
  g.head = heads + 1;
  g.dX = dX;
  g.scr = scr;
  g.soff = soff;
  g.err = err;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return T3F_ERR_CUDA;
  const int grid = std::max(1, std::min(ngitems, sms));
  return by_math(math, dtype, [&](auto kind, auto* st) -> t3f_status {
    using ST = std::remove_pointer_t<decltype(st)>;
    return launch_grad<decltype(kind)::value, ST>(g, grid, s);
  });
}

}  // namespace t3f
