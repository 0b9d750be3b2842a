// Trailing update of the blocked Cholesky on the 5th-generation tensor cores (tcgen05), FP32
// factors (mixed mode): for nq panel tile columns q in [kb0, kb0 + nq),
//     A(i, j) -= sum_q L(i, q) S_q L(j, q)^T       for jbeg <= j < min(Bc, jend), j <= i < R,
// (S_q: pivot signs of the signed Cholesky, identity for SPD levels)
// batched over all subdomains of a level (Algorithm 1, "factorize the matrices of local saddle
// point problems").  The factorisation runs in 512-wide super-panels of two 256-wide halves:
// after the first half, a rank-256 update (nq = 4) brings the second half's columns up to date;
// after the second half, one rank-512 update (nq = 8) serves every trailing column.  Each
// trailing element is read and written once per 512 columns instead of once per 256 (without its
// output write-back the rank-256 kernel ran 27 % faster): on the 48^3 factorisation the update
// went from 254 to 300 TFLOP/s FP32-equivalent (before the two MMA issuers).
//
// FP32 accuracy from FP16 tensor cores: for the 64 x 256 slab of panel row tile i, every row r
// is scaled by 2^e_r so that its largest entry lies in [2^14, 2^15), and each scaled entry a is
// split into hi = fp16(a) and lo = fp16((a - hi) 2^11) (the scaled low part cannot underflow).
// Then a b = hi_a hi_b + (hi_a lo_b + lo_a hi_b) 2^-11 up to the dropped lo lo term (2^-22
// relative): three FP16 products, 4 bytes per entry (the scheme of Ootomo and Yokota, 2022).
// The output is unscaled exactly by the stored factors 2^-e_i and 2^-e_j.  Indefinite levels
// also get a copy of the parts whose columns carry the pivot signs, read as the B operand, so
// that both operands of every MMA stay FP16.  Measured against FP64 on factor-like data (rows
// spanning four decades): 2-4e-7 of sum |a||b| (three-part BF16 splitting with six products:
// 1.3e-7, FP32 dot: 8e-7).  Accumulating all products in one TMEM accumulator over K = 256
// loses an order of magnitude, so the dominant hi hi product has its own accumulator, which is
// promoted into FP32 registers after every 64-wide panel column; the cross products (2^-11 of
// it) are accumulated over the whole work item.
//
// k_split_panel writes the parts in the exact shared-memory operand image (K-major, 128-byte
// swizzle), so the update moves bytes with cp.async.bulk only.  A work item is a 128 x 128
// output block (row tiles i0, i0+1 by column tiles j, j+1); per panel column q the producer
// warp copies the two parts of the four tiles (64 KB) into one of three shared-memory stages,
// one thread issues the 4 hi hi MMAs (M = N = 128, K = 16) into one of two TMEM accumulators, a
// second thread in another warp the 8 MMAs of the cross products into the item's own
// accumulator (two of those), and eight epilogue warps promote and finally update the output
// tiles.  The two issuers wait independently, so the tensor pipe holds the cross products while
// a promotion is under way; one issuer for all twelve left it idle between commit and wait.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "internal.h"
#include "split.cuh"
#include "tc_items.h"

namespace bddc {

namespace {

constexpr uint32_t kSpinLimit = 1u << 26;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// K-major operand, 128-byte swizzle: rows of 64 16-bit entries (128 B), 8-row atoms of 1024 B
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);   // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;         // stride byte offset: next 8-row atom
  d |= (uint64_t)1 << 46;                   // descriptor version
  d |= (uint64_t)2 << 61;                   // 128-byte swizzle
  return d;
}


__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}


constexpr uint32_t kOpnd = 2 * kTilePart;        // one part of a 128-row operand (16 KB)
constexpr uint32_t kStage2 = 4 * kOpnd;          // A hi, A lo, B hi, B lo (64 KB)
constexpr int kThreads2 = 352;                   // 8 epilogue warps + 2 MMA warps + 1 producer warp
constexpr int kStages2 = 3;                      // shared-memory stages (copies run two steps ahead)
constexpr int kMmaBars = 6;                      // step-completion barriers (two steps sharing one are 6 apart)
constexpr uint32_t kEpiBox = 32 * 128;           // per epilogue warp: one 32 x 32 FP32 output box (4 KB)

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// bounded wait for the completion of a phase (its first test stands alone: the usual case)
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  for (uint32_t spins = 0; spins < kSpinLimit; ++spins)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// position in a ring of N barriers and the parity of its current phase
template <int N>
struct Ring {
  uint32_t k = 0, phase = 0;
  __device__ __forceinline__ void next() {
    if (++k == N) {
      k = 0;
      phase ^= 1u;
    }
  }
};

// 32 columns of this warp's TMEM lanes (lane l: row l), complete on return
__device__ __forceinline__ void tmem_ld32(float (&v)[32], uint32_t taddr) {
  uint32_t* u = (uint32_t*)v;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]),
        "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]),
        "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
      : "r"(taddr)
      : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}


// one block per panel row tile i of every subdomain: ib <= i < R where the launch has output columns
// (ib < Bc); panel_operand: min(ib, Bc) <= i; and the inverse rows reached by the columns below ib
template <int NT>
__global__ void __launch_bounds__(64 * NT) k_split_panel(LevelDev L, int kb0, int ib, int act, int panel_operand,
                                                         uint8_t* __restrict__ split,
                                                         uint8_t* __restrict__ split_signed,
                                                         float* __restrict__ rscale,
                                                         const int64_t* __restrict__ prow_off) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  if (act >= m.Bc || (!panel_operand && !m.nV && ib >= m.Bc)) return;
  const int i = (ib < m.Bc ? ib : m.Bc) + (int)blockIdx.x;
  if (i >= (ib <= m.nIb ? (int)m.Bc : m.R + inverse_rows(m, ib))) return;
  split_row_tile<NT>(L, s, m, i, kb0, split, split_signed, rscale, prow_off);
}

// one block per block row Q of the inverse X of every subdomain's diagonal block (Q < nd): the
// rows of -S_D X, the B operand of the panel solve (its update kernel subtracts A B^T)
__global__ void __launch_bounds__(256) k_split_inverse(LevelDev L, int k0, uint8_t* __restrict__ split, float* __restrict__ rscale,
                                                       const int64_t* __restrict__ prow_off) {
  const int s = blockIdx.y, Q = blockIdx.x;
  const SubMeta m = L.meta[s];
  const int nd = m.Bc - k0 < 4 ? m.Bc - k0 : 4;
  if (Q >= nd) return;
  __shared__ float rm[NB];
  const float* sg = (const float*)L.sgn + m.vec_off + (int64_t)(k0 + Q) * NB;
  if (threadIdx.x < NB) rm[threadIdx.x] = sg[threadIdx.x] < 0.f ? 1.f : -1.f;   // -s_r
  __syncthreads();
  const int c = threadIdx.x >> 6;   // block column of X; zero above the diagonal blocks
  const float* src = c < Q    ? L.xinv + x_tile(m, k0, Q, c)
                     : c == Q ? (const float*)L.dinv + m.dinv_off + (int64_t)(k0 + Q) * NB2
                              : nullptr;
  split_rows<4>(src, rm, prow_off[s] + k0 + Q, split, nullptr, rscale, nullptr);
}

// Persistent: CTA c takes the work items c, c + gridDim.x, ... of the launch (items of all
// subdomains flattened; item_pref[s] = first item of subdomain s).  One global step g per (item, panel
// column).  Roles, in warps of their own: a producer thread requests the copies of each step into
// shared-memory stage g % 3 as soon as the MMAs of step g - 3 have read it; one thread issues the hi hi
// product of each step (4 MMAs) and another the two cross products (8 MMAs); eight epilogue warps
// promote the accumulators and write back each item's output block.
//
// What bounds it.  At 64 KB of operands per step the SM's L2 port (64 B per cycle) allows about 1,024
// cycles per step, the MMAs alone 855 (12 x M = N = 128, K = 16, measured); a step of the one-issuer
// kernel took 2,050.  Its issuing thread spent 740 of them between MMAs: the tensor pipe queues only a
// few, so every barrier wait (150 to 230 cycles of dependent scalar work, even for a phase long complete),
// commit (60 to 90) and address computation left it idle.  Hence
//   - two issuing threads on accumulators of their own (no order between their MMAs is needed): while one
//     waits or commits, the other's MMAs run;
//   - the hi hi product has a TMEM accumulator per step (two, g & 1), promoted into FP32 registers every
//     step; the cross products, 2^-11 smaller, accumulate in TMEM over the whole item (two, item & 1).
//     That halves the epilogue's TMEM reads and additions, and the cross products never wait for the
//     epilogue within an item;
//   - one commit per issuer and step, on a ring of six barriers (g % 6) that the producer and the epilogue
//     wait on: two steps that share a barrier are six apart, more than the three stages let any role
//     run ahead, so a phase is never missed;
//   - items are found in closed form (tc_items.h), and every role walks the subdomains forward.
// The write-back is a TMA reduce-add: each epilogue warp scales its 32 x 64 part of the block into a
// swizzled shared-memory box, 32 columns at a time, and one lane adds the box into the tiles in L2 (the
// output is never read into the SM; every element receives exactly one add per launch, so the result
// does not depend on timing).
// Measured in isolation (n = 16,384, kernel time): rank 512 0.470 -> 0.355 ms (276 -> 365 TFLOP/s FP32-
// equivalent), rank 256 0.320 -> 0.230 ms; of it the MMAs and barriers alone take 0.222 ms, the operand
// copies alone 0.259, and the output's read-modify-write in DRAM 0.158 at the copy bandwidth.
__global__ void __launch_bounds__(kThreads2, 1)
    k_update_tc2(LevelDev L, int nq, int jbeg, int jend, int ibeg, int panel, int act, const uint8_t* __restrict__ split,
                 const uint8_t* __restrict__ split_b, const float* __restrict__ rscale,
                 const int64_t* __restrict__ prow_off, const int64_t* __restrict__ item_pref,
                 const __grid_constant__ CUtensorMap tmap) {
  const int n_sub = (int)L.n_sub;
  const int64_t n_items = item_pref[n_sub];
  if ((int64_t)blockIdx.x >= n_items) return;
  // nq panel tile columns (K = 64 nq) in the split rows; output columns jbeg <= j < min(Bc, jend)

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* stage0 = smem_raw + (base - raw);
  // full: shared-memory stage g % 3 loaded; big / crs: the hi hi / cross products of step g done (stage
  // read, accumulator written); epi: hi hi accumulator g & 1 read; sml: cross accumulator of item & 1 read
  __shared__ __align__(8) uint64_t full_bar[kStages2], big_bar[kMmaBars], crs_bar[kMmaBars], epi_bar[2], sml_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_issued[2], s_requested;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int b = 0; b < kStages2; ++b) mbar_init(&full_bar[b], 1);
    for (int b = 0; b < kMmaBars; ++b) {
      mbar_init(&big_bar[b], 1);
      mbar_init(&crs_bar[b], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&epi_bar[b], 8);
      mbar_init(&sml_bar[b], 8);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_issued[0] = s_issued[1] = 0;
    s_requested = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  // a role's place in the item list: items come in ascending order, so the subdomain only moves forward
  struct Cursor {
    int s = -1;
    int64_t first = 0, next = 0;   // items [first, next) belong to subdomain s
    SubMeta m;
    TcItems t;
    int64_t rbase = 0;
  };
  auto seek = [&](Cursor& c, int64_t it, int& j, int& i0, int& jl) {
    if (it >= c.next) {
      do {
        ++c.s;
        c.first = c.next;
        c.next = item_pref[c.s + 1];
      } while (it >= c.next && c.s + 1 < n_sub);
      c.m = L.meta[c.s];
      c.t = tc_items_of(c.m, jbeg, jend, ibeg, panel, act);
      c.rbase = prow_off[c.s];
    }
    tc_item(c.t, (int)(it - c.first), j, i0, jl);
  };

  // steps of this CTA: its items in order, nq panel columns each; a panel solve's B operand (rows
  // of the inverse of a lower triangular block) is zero beyond block column j - jbeg + 1, so the
  // column pair j, j + 1 takes K steps 0 .. j - jbeg + 1 only
  auto item_nq = [&](int j) { return panel ? min(nq, j - jbeg + 2) : nq; };
  if (warp == 10) {
    // ---- producer: its own thread, so that waiting for a stage never delays the issue of MMAs
    if (lane == 0) {
      bool lost = false;
      Cursor cur;
      uint32_t g = 0;
      Ring<kStages2> st;
      Ring<kMmaBars> rd;   // the step whose MMAs read the stage last
      for (int64_t it = blockIdx.x; it < n_items && !lost; it += gridDim.x) {
        int j, i0, jl;
        seek(cur, it, j, i0, jl);   // before the wait for a stage: overlaps the MMAs still reading it
        const SubMeta& m = cur.m;
        const bool hasA1 = i0 + 1 < cur.t.rend, hasB1 = j + 1 < jl;
        const uint8_t* rowA0 = split + (cur.rbase + i0) * kPanelTiles * (int64_t)kSplitTile;
        const uint8_t* rowA1 = hasA1 ? rowA0 + kPanelTiles * (int64_t)kSplitTile : rowA0;
        const uint8_t* rowB0 = split_b + (cur.rbase + j) * kPanelTiles * (int64_t)kSplitTile;
        const uint8_t* rowB1 = hasB1 ? rowB0 + kPanelTiles * (int64_t)kSplitTile : rowB0;
        const int nqi = item_nq(j);
        for (int q = 0; q < nqi; ++q, ++g) {
          if (g >= (uint32_t)kStages2) {
            if (!mbar_wait(&big_bar[rd.k], rd.phase) || !mbar_wait(&crs_bar[rd.k], rd.phase)) {
              lost = true;
              break;
            }
            rd.next();
          }
          if (q == 0 && !panel)   // the output tiles are read back by the write-back after the last column
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
              for (int c = 0; c < 2; ++c) {
                const int ti = i0 + a, tj = j + c;
                if ((a == 0 || hasA1) && (c == 0 || hasB1) && tile_exists(m, ti, tj))
                  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                                   (const float*)L.tiles + m.tile_off + tile_of(m, ti, tj) * NB2),
                               "r"((uint32_t)(NB2 * 4))
                               : "memory");
              }
          uint8_t* sA = stage0 + st.k * kStage2;   // [A hi | A lo | B hi | B lo], 128 rows each
          uint8_t* sB = sA + 2 * kOpnd;
          uint64_t* bar = &full_bar[st.k];
          mbar_expect_tx(bar, kStage2);
          const int64_t qo = (int64_t)q * kSplitTile;
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            bulk_g2s(sA + p * kOpnd, rowA0 + qo + p * kTilePart, kTilePart, bar);
            bulk_g2s(sA + p * kOpnd + kTilePart, rowA1 + qo + p * kTilePart, kTilePart, bar);
            bulk_g2s(sB + p * kOpnd, rowB0 + qo + p * kTilePart, kTilePart, bar);
            bulk_g2s(sB + p * kOpnd + kTilePart, rowB1 + qo + p * kTilePart, kTilePart, bar);
          }
          st.next();
        }
      }
      s_requested = (int)g;
      if (lost) atomicExch(L.status + 2, 4);
    }
  } else if (warp >= 8) {
    // ---- MMA issuers: one thread each, warp 8 the hi hi product, warp 9 the cross products
    if (lane == 0) {
      const bool big = warp == 8;
      uint64_t* done_bar = big ? big_bar : crs_bar;
      // c FP32, a and b FP16, both K-major, N = 128, M = 128
      const uint32_t idesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
      const uint64_t desc0 = desc_sw128(base);   // operand at stage 0; the start address counts 16-byte units
      auto mma = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
        asm volatile(
            "{\n .reg .pred pp;\n setp.ne.b32 pp, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pp;\n}\n" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc));
      };
      constexpr uint64_t kA1 = kOpnd >> 4, kB0 = 2 * (kOpnd >> 4), kB1 = 3 * (kOpnd >> 4);   // A lo, B hi, B lo
      bool ok = true;
      Cursor cur;
      uint32_t g = 0, n = 0;   // n: items of this CTA so far
      Ring<kStages2> st;
      Ring<kMmaBars> dn;
      for (int64_t it = blockIdx.x; it < n_items && ok; it += gridDim.x, ++n) {
        int nqi = nq;
        if (panel) {
          int j, i0, jl;
          seek(cur, it, j, i0, jl);
          nqi = item_nq(j);
        }
        const uint32_t acc_small = tmem + 256u + 128u * (n & 1u);
        // the cross accumulator of item n - 2 is read before the first product of item n
        if (!big && n >= 2) ok = mbar_wait(&sml_bar[n & 1u], ((n >> 1) - 1) & 1u);
        for (int q = 0; q < nqi && ok; ++q) {
          const uint64_t d = desc0 + (uint64_t)(st.k * (kStage2 >> 4));
          if (big) {
            const uint32_t b = g & 1u;
            if (g >= 2) ok = mbar_wait(&epi_bar[b], ((g >> 1) - 1) & 1u);   // hi hi of step g - 2 is read
            ok = mbar_wait(&full_bar[st.k], st.phase) && ok;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma(tmem + 128u * b, d + 2 * kk, d + kB0 + 2 * kk, kk > 0);   // hi hi
          } else {
            ok = mbar_wait(&full_bar[st.k], st.phase);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma(acc_small, d + kA1 + 2 * kk, d + kB0 + 2 * kk, q > 0 || kk > 0);   // lo hi
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma(acc_small, d + 2 * kk, d + kB1 + 2 * kk, 1u);                      // hi lo
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(&done_bar[dn.k]))
                       : "memory");
          ++g;
          st.next();
          dn.next();
        }
      }
      s_issued[big ? 0 : 1] = (int)g;
      if (!ok) atomicExch(L.status + 2, 4);
    }
  } else {
    // ---- epilogue warps: warp w reads TMEM lanes 32 (w & 3) .. +31 (output rows) and columns
    // 64 (w >> 2) .. +63
    bool lost = false;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const uint32_t col0 = 64u * (uint32_t)(warp >> 2);
    const int erow = 32 * (warp & 3) + lane;
    uint8_t* box = stage0 + kStages2 * kStage2 + warp * kEpiBox;   // 1024-byte aligned
    Cursor cur;
    uint32_t g = 0, n = 0;
    Ring<kMmaBars> dn;
    for (int64_t it = blockIdx.x; it < n_items && !lost; it += gridDim.x, ++n) {
      int j, i0, jl;
      seek(cur, it, j, i0, jl);
      const SubMeta& m = cur.m;
      const bool hasA1 = i0 + 1 < cur.t.rend, hasB1 = j + 1 < jl;
      const int ti = erow < 64 ? i0 : i0 + 1;
      const int tj = col0 < 64 ? j : j + 1;
      const bool ok = (erow < 64 || hasA1) && (col0 < 64 || hasB1) && tile_exists(m, ti, tj);
      // negated row factor: the tiles receive x + (-(acc sa) f), which equals x - (acc sa) f
      const float sa = ok ? -rscale[(cur.rbase + ti) * NB + (erow & 63)] : 0.f;
      float racc[64];
#pragma unroll
      for (int c = 0; c < 64; ++c) racc[c] = 0.f;
      const int nqi = item_nq(j);
      for (int q = 0; q < nqi; ++q, ++g) {
        const uint32_t b = g & 1u;
        lost = __any_sync(0xffffffffu, !mbar_wait(&big_bar[dn.k], dn.phase));
        if (q + 1 == nqi) lost = __any_sync(0xffffffffu, !mbar_wait(&crs_bar[dn.k], dn.phase)) || lost;
        if (lost) break;
        dn.next();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[32];
          tmem_ld32(v, tmem + lane_base + 128u * b + col0 + 32u * h);
#pragma unroll
          for (int c = 0; c < 32; ++c) racc[32 * h + c] += v[c];
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&epi_bar[b]);
      }
      if (lost) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // the item's cross products
        float v[32];
        tmem_ld32(v, tmem + lane_base + 256u + 128u * (n & 1u) + col0 + 32u * h);
#pragma unroll
        for (int c = 0; c < 32; ++c) racc[32 * h + c] += v[c] * (1.f / 2048.f);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&sml_bar[n & 1u]);
      if (ok) {   // warp-uniform: the warp's 32 rows and 64 columns lie in one output tile
        const float4* sb = (const float4*)(rscale + (cur.rbase + tj) * NB);
        // row of the warp's first output row in the [rows][64] view of the tile buffer
        const int y = (int)((m.tile_off + tile_of(m, ti, tj) * NB2) / NB) + (32 * (warp & 3) & 63);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          // the previous reduce-add out of this warp's box has read it
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int u = 8 * hh + k;
            const float4 f = __ldg(sb + u);   // both factors are powers of two: the products are exact
            float4 x;
            x.x = (racc[4 * u + 0] * sa) * f.x;
            x.y = (racc[4 * u + 1] * sa) * f.y;
            x.z = (racc[4 * u + 2] * sa) * f.z;
            x.w = (racc[4 * u + 3] * sa) * f.w;
            // 128-byte swizzle: 16-byte chunk k of box row r sits at chunk k ^ (r & 7)
            *(float4*)(box + lane * 128 + ((k ^ (lane & 7)) << 4)) = x;
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            if (panel)   // a panel solve writes its tiles (their old contents are the split A operand)
              asm volatile(
                  "cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                      (uint64_t)&tmap),
                  "r"(32 * hh), "r"(y), "r"(smem_u32(box))
                  : "memory");
            else
              asm volatile(
                  "cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                      (uint64_t)&tmap),
                  "r"(32 * hh), "r"(y), "r"(smem_u32(box))
                  : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        }
      }
    }
    // the reduce-adds are complete (and the boxes free) before the CTA ends, also on the error path
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (lost && lane == 0) atomicExch(L.status + 2, 4);
  }
  __syncthreads();
  // copies requested but never consumed (a wait gave up) may still be landing in shared memory:
  // wait (bounded) for them before the CTA exits
  if (tid == 0)
    for (int c = max(0, s_requested - kStages2); c < s_requested; ++c)
      mbar_wait(&full_bar[c % kStages2], (uint32_t)(c / kStages2) & 1u);
  // before the accumulators are released no MMA may still be running (also on the error path): the last
  // commit of each issuer covers every MMA it issued
  for (int k = 0; k < 2; ++k)
    if (s_issued[k] > 0)
      mbar_wait(&(k == 0 ? big_bar : crs_bar)[(s_issued[k] - 1) % kMmaBars], (uint32_t)((s_issued[k] - 1) / kMmaBars) & 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

}  // namespace

void launch_split_panel(const LevelDev& L, int kb0, int nt, int ib, int act, int rows, uint8_t* split,
                        uint8_t* split_signed, float* rscale, const int64_t* prow_off, cudaStream_t st,
                        int panel_operand) {
  if (L.n_sub <= 0 || rows <= 0) return;
  note_launch();
  const dim3 grid((unsigned)rows, (unsigned)L.n_sub);
  if (nt == 8)
    k_split_panel<8><<<grid, 512, 0, st>>>(L, kb0, ib, act, panel_operand, split, split_signed, rscale, prow_off);
  else
    k_split_panel<4><<<grid, 256, 0, st>>>(L, kb0, ib, act, panel_operand, split, split_signed, rscale, prow_off);
}

void launch_split_inverse(const LevelDev& L, int k0, uint8_t* split, float* rscale,
                          const int64_t* prow_off, cudaStream_t st) {
  if (L.n_sub <= 0) return;
  note_launch();
  k_split_inverse<<<dim3(4, (unsigned)L.n_sub), 256, 0, st>>>(L, k0, split, rscale, prow_off);
}

void launch_update_tc2(const LevelDev& L, int nq, int jbeg, int jend, int ibeg, int panel, int act, int grid,
                       const uint8_t* split,
                       const uint8_t* split_b, const float* rscale, const int64_t* prow_off,
                       const int64_t* item_pref, const TensorMap128& tmap, cudaStream_t st) {
  if (grid <= 0 || L.n_sub <= 0 || nq <= 0 || nq > kPanelTiles) return;
  const size_t dyn = kStages2 * kStage2 + 8 * kEpiBox + 1024;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_update_tc2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    attr = true;
  }
  note_launch();
  CUtensorMap m;
  static_assert(sizeof(CUtensorMap) == sizeof(TensorMap128), "tensor map size");
  std::memcpy(&m, &tmap, sizeof(m));
  k_update_tc2<<<(unsigned)grid, kThreads2, dyn, st>>>(L, nq, jbeg, jend, ibeg, panel, act, split, split_b, rscale, prow_off,
                                                        item_pref, m);
}

int make_tile_tmap(TensorMap128* map, float* tiles, int64_t tile_elems) {
  using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeTiled encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return (int)CUDA_ERROR_NOT_FOUND;
    encode = (EncodeTiled)fn;
  }
  const int64_t rows = tile_elems / NB;
  if (rows <= 0 || rows >= ((int64_t)1 << 31)) return (int)CUDA_ERROR_INVALID_VALUE;   // int32 box coordinates
  const cuuint64_t dims[2] = {(cuuint64_t)NB, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)NB * sizeof(float)};
  const cuuint32_t box[2] = {32, 32};
  const cuuint32_t estr[2] = {1, 1};
  CUtensorMap m;
  const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, tiles, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return (int)r;
  std::memcpy(map, &m, sizeof(m));
  return 0;
}

}  // namespace bddc
