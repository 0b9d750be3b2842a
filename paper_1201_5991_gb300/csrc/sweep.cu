// Streaming triangular sweeps with the tiled factors, batched over all subdomains of a level:
// forward y = S L^{-1} b and backward L^T x = y over the interior block rows (the discrete
// Dirichlet problems of the Schur operator, Sec. 2) or over the interface block rows (the
// constrained Neumann problem of Eq. sub_cor, restricted to the interface; factors that hold the
// interface inverse apply that instead, trmv.cu).  S holds the pivot
// signs of the signed Cholesky (identity for SPD levels), so the pair solves L S L^T x = b.
//
// Design (GB300): the sweep is bound by reading the factor from HBM once.  A persistent grid
// of 2 CTAs per SM takes block-row tasks (subdomain s, block row i) from a global counter in
// dependency order (all subdomains' first rows, then their second rows, ...).  A task
// streams its row of NB x NB tiles (forward) or its column of tiles (backward) into a ring of
// shared-memory stages with cp.async.bulk, completion tracked by mbarriers, while the solution
// blocks it depends on are published by other CTAs in a publication buffer that is filled with
// all-ones words before the launch: a block is ready when none of its words is all-ones any
// more (every word is written once, atomically, and no arithmetic result has that NaN bit
// pattern: NaN results are canonical, and a computed all-ones word is published as the
// canonical NaN).  The consumer polls the data itself, one L2 round trip instead of a flag
// acquire followed by the data load, and the producer needs no fence.  A task only waits for
// tasks handed out before it, so the scheme cannot deadlock whatever the residency.  Every wait
// is bounded; a timeout sets status[2] and the kernel finishes without waiting further (the host
// reports BDDC_ERR_TIMEOUT).  A wait for a published block that gives up stages the block as it
// is and goes on, so every tile copy is still consumed and no access leaves the task's own rows;
// a tile wait that gives up drains the ring before exit.
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"
#include "pdl.cuh"
#include "reduce.cuh"

namespace bddc {

namespace {

constexpr int kThreads = 256;
constexpr int kYSlots = 16;          // solution blocks staged in shared memory at a time
constexpr long long kSpinLimit = 1ll << 24;
constexpr long long kProbeSpins = 32;   // publication wait limit of the timeout probe

__device__ __forceinline__ int64_t tile_index(int i, int j, int Bc) {
  return i < Bc ? ((int64_t)i * (i + 1) / 2 + j) : ((int64_t)Bc * (Bc + 1) / 2 + (int64_t)(i - Bc) * Bc + j);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
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

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// publication words: relaxed (coherent at L2) loads and stores; all-ones = not yet written
__device__ __forceinline__ bool pub_ld2(const float* p, float2& v) {
  uint32_t a, b;
  asm volatile("ld.relaxed.gpu.global.v2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p) : "memory");
  v = make_float2(__uint_as_float(a), __uint_as_float(b));
  return a != 0xFFFFFFFFu && b != 0xFFFFFFFFu;
}
__device__ __forceinline__ bool pub_ld2(const double* p, double2& v) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  v = make_double2(__longlong_as_double((long long)a), __longlong_as_double((long long)b));
  return a != ~0ull && b != ~0ull;
}
__device__ __forceinline__ void pub_st(float* p, float x) {
  uint32_t a = __float_as_uint(x);
  if (a == 0xFFFFFFFFu) a = 0x7FFFFFFFu;
  asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(a) : "memory");
}
__device__ __forceinline__ void pub_st(double* p, double x) {
  unsigned long long a = (unsigned long long)__double_as_longlong(x);
  if (a == ~0ull) a = 0x7FFFFFFFFFFFFFFFull;
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}

template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
  using type = float2;
};
template <>
struct Vec2<double> {
  using type = double2;
};

// One task: (subdomain, block row).  Forward consumes tiles (i, B0..i-1) then D_i^{-1};
// backward consumes tiles (B1-1..i+1, i) then D_i^{-1}.
// GRP (interior sweeps of levels that keep the inverses X_D of their 256-wide diagonal blocks
// D = [g0, g0 + 4)): row g0 + Q consumes the tiles left of its block, publishes its remaining right-hand side
// r'_Q (p2), and then y_Q = sum_{P <= Q} X_QP r'_P (backward: X_PQ^T, P >= Q) with the other rows' r'.  The rows of
// a block no longer wait for one another's solutions: two dependent L2 round trips per four block rows
// instead of four.  It matters where the chain bounds the sweep: 8 subdomains of 81 interior block rows
// took 1.3 us per row, 100 us for bytes of 47.  NR right-hand sides are solved together
// (column r at vec + r * vstride): every factor tile is streamed from HBM once per task and
// applied to all of them from shared memory.
template <typename T, int S, bool BWD, int NR, bool GRP>
__global__ void __launch_bounds__(kThreads, 2)
    k_sweep(LevelDev L, T* __restrict__ vec, int64_t vstride, const int2* __restrict__ tasks, int ntasks, int part,
            int* __restrict__ ctrl, T* pub, T* pub2) {
  using V2 = typename Vec2<T>::type;
  constexpr int YS = NR == 1 ? kYSlots : (NR == 2 ? 8 : 4);   // solution blocks staged at a time
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* stage = (T*)smem_raw;                       // S tiles of NB*NB
  __shared__ __align__(8) uint64_t full[S];
  __shared__ __align__(16) T ybuf[YS][NR][NB];
  __shared__ T red[kThreads / 32][NR][NB];
  __shared__ __align__(16) T rhs[NR][NB];
  __shared__ T s_sg[NB];                         // pivot signs of the task's block row (indefinite)
  __shared__ int s_task;
  __shared__ int s_rdy[kYSlots];                 // poll result per candidate block
  int* counter = ctrl;
  int* status = L.status;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int k = 0; k < S; ++k) mbar_init(&full[k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  constexpr int NV = 8 * NR, NC = NV < 32 ? 1 : NV / 32;   // row sums (lane_sums)
  const int f0 = lane_sum_index<NV>(lane);
  const bool writer = lane_sum_writer<NV>(lane);
  uint32_t cons = 0;     // tiles consumed by this CTA (ring position and phase)
  uint32_t issued = 0;   // tiles issued (thread 0)
  bool lost = false;     // a tile wait gave up: drain before exit
  for (;;) {
    if (tid == 0) s_task = atomicAdd(counter, 1) + 1;   // the counter starts at -1 (all ones)
    __syncthreads();
    const int t = s_task;
    if (t >= ntasks) break;
    const int sub = tasks[t].x, i = tasks[t].y;
    const SubMeta m = L.meta[sub];
    if (!BWD && L.indefinite && tid < NB) s_sg[tid] = ((const T*)L.sgn)[m.vec_off + (int64_t)i * NB + tid];
    // interior part: the block rows that hold interior DOFs (padding identity block rows, whose
    // rows and columns of L are unit vectors and whose right-hand sides are zero, are skipped)
    const int B0 = part == 0 ? 0 : m.nIb, B1 = part == 0 ? (m.nI + NB - 1) / NB : m.Bc;
    const int g0 = GRP ? (i & ~3) : i, g1 = GRP ? (g0 + 4 < B1 ? g0 + 4 : B1) : i + 1;   // the row's diagonal block
    const int nL = BWD ? (B1 - g1) : (g0 - B0);           // factor tiles beside the diagonal block
    const int ntile = BWD ? (B1 - i) : (i - B0 + 1);      // and its inverse's tiles, D_i^{-1} last
    const T* tiles = (const T*)L.tiles + m.tile_off;
    const T* dinv = (const T*)L.dinv + m.dinv_off + (int64_t)i * NB2;
    T* v = vec + m.vec_off;
    T* pv = pub + m.vec_off;   // this subdomain's published blocks (same layout as v)
    T* p2 = GRP ? pub2 + m.vec_off : nullptr;   // and remaining right-hand sides
    auto tile_src = [&](int k) -> const T* {
      if (k == ntile - 1) return dinv;
      const int j = BWD ? (B1 - 1 - k) : (B0 + k);
      if (GRP && k >= nL) return (const T*)L.xinv + (BWD ? x_tile(m, g0, j - g0, i - g0) : x_tile(m, g0, i - g0, j - g0));
      return BWD ? tiles + tile_index(j, i, m.Bc) * NB2 : tiles + tile_index(i, j, m.Bc) * NB2;
    };
    // the task's own right-hand side block depends on no other task: read it into rhs now, off
    // the chain of dependent rows (the diagonal step subtracts the updates in place)
    for (int e = tid; e < NR * NB; e += kThreads) rhs[e / NB][e % NB] = __ldcg(v + (e / NB) * vstride + i * NB + e % NB);
    __syncthreads();
    // prologue: fill the ring
    if (tid == 0) {
      const int pre = ntile < S ? ntile : S;
      for (int k = 0; k < pre; ++k) {
        const uint32_t slot = (cons + k) % S;
        mbar_expect_tx(&full[slot], (uint32_t)(NB2 * sizeof(T)));
        bulk_g2s(stage + slot * NB2, tile_src(k), (uint32_t)(NB2 * sizeof(T)), &full[slot]);
      }
      issued += pre;
    }
    T acc[NR][8];        // forward: rows warp + 8 r, this lane's two columns, every right-hand side
    T accc[NR][2];       // backward: this lane's two columns, summed over the warp's rows
#pragma unroll
    for (int q = 0; q < NR; ++q)
#pragma unroll
      for (int r = 0; r < 8; ++r) acc[q][r] = (T)0;
#pragma unroll
    for (int q = 0; q < NR; ++q) accc[q][0] = accc[q][1] = (T)0;
    int staged_end = 0;   // tiles [staged_begin, staged_end) have their solution block in ybuf
    for (int k = 0; k < ntile; ++k) {
      if (k == nL) {
        // the factor's part is complete: the remaining right-hand side of the row
        if (!BWD) {
          lane_sums<NV>(&acc[0][0], lane);   // N = 8 NR values per lane: value 8 q + r is row warp + 8 r of column q
          if (writer)
#pragma unroll
            for (int c = 0; c < NC; ++c) rhs[(f0 + c) / 8][warp + 8 * ((f0 + c) % 8)] -= (&acc[0][0])[c];
          if constexpr (GRP)
#pragma unroll
            for (int q = 0; q < NR; ++q)
#pragma unroll
              for (int r = 0; r < 8; ++r) acc[q][r] = (T)0;
          __syncthreads();
        } else {
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            red[warp][q][2 * lane] = accc[q][0];
            red[warp][q][2 * lane + 1] = accc[q][1];
            accc[q][0] = accc[q][1] = (T)0;
          }
          __syncthreads();
          for (int e = tid; e < NR * NB; e += kThreads) {
            const int q = e / NB, c = e % NB;
            T a = (T)0;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) a += red[w][q][c];
            rhs[q][c] -= a;
          }
          __syncthreads();
        }
        if (GRP && g1 - g0 > 1 && i != (BWD ? g0 : g1 - 1))
          for (int e = tid; e < NR * NB; e += kThreads)
            pub_st(p2 + (e / NB) * vstride + i * NB + e % NB, rhs[e / NB][e % NB]);
      }
      if (k < ntile - 1 && k >= staged_end) {
        // wait until the next solution blocks are published, then stage up to YS of them: warp w
        // polls blocks k + w and k + w + 8 (all their words at once), writes the ready ones into
        // ybuf, and the consecutive ready blocks from k are staged
        const int upto = k < nL ? nL : ntile - 1;   // factor tiles, then the inverse's
        const int want = upto - k < YS ? upto - k : YS;
        const T* pb = k < nL ? pv : p2;
        int cnt = 0;
        long long spins = 0;
        for (;;) {
          __syncthreads();   // every thread has read s_rdy of the previous poll
          for (int b = warp; b < want; b += kThreads / 32) {
            const int j = BWD ? (B1 - 1 - (k + b)) : (B0 + k + b);
            V2 y[NR];
            bool ok = true;
#pragma unroll
            for (int q = 0; q < NR; ++q) ok &= pub_ld2(pb + q * vstride + j * NB + 2 * lane, y[q]);
            // the timeout probe waits for a word that nothing sets (status[3]) instead
            if (L.wait_probe) ok = ld_acquire(status + 3) != 0;
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
              V2 sg = {(T)1, (T)1};
              if (!BWD && L.indefinite && k < nL)   // solved rows hold S_j y_j: the update needs y_j
                sg = *(const V2*)((const T*)L.sgn + m.vec_off + (int64_t)j * NB + 2 * lane);
#pragma unroll
              for (int q = 0; q < NR; ++q) {
                y[q].x *= sg.x;
                y[q].y *= sg.y;
                *(V2*)&ybuf[(k + b) % YS][q][2 * lane] = y[q];
              }
            }
            if (lane == 0) s_rdy[b] = ok ? 1 : 0;
          }
          __syncthreads();
          cnt = 0;
          while (cnt < want && s_rdy[cnt]) ++cnt;
          if (cnt > 0) break;
          if (++spins > (L.wait_probe ? kProbeSpins : kSpinLimit)) {
            if (tid == 0) atomicExch(status + 2, 1);
            cnt = 1;   // stage the block as it is and go on (error path)
            break;
          }
          __nanosleep(64);
        }
        staged_end = k + cnt;
      }
      // wait for the tile
      const uint32_t slot = cons % S, parity = (cons / S) & 1u;
      {
        long long spins = 0;
        while (!mbar_try_wait(&full[slot], parity)) {
          if (++spins > kSpinLimit) {
            if (tid == 0) atomicExch(status + 2, 2);
            lost = true;
            break;
          }
        }
      }
      const T* tl = stage + slot * NB2;
      if (k < ntile - 1) {
        const int ys = k % YS;
        if (!BWD) {
          V2 a[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) a[r] = *(const V2*)(tl + (warp + 8 * r) * NB + 2 * lane);
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            const V2 yv = *(const V2*)(&ybuf[ys][q][2 * lane]);
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[q][r] += a[r].x * yv.x + a[r].y * yv.y;
          }
        } else {
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int row = warp + 8 * r;
            const V2 a = *(const V2*)(tl + row * NB + 2 * lane);
#pragma unroll
            for (int q = 0; q < NR; ++q) {
              const T x = ybuf[ys][q][row];
              accc[q][0] += a.x * x;
              accc[q][1] += a.y * x;
            }
          }
        }
      } else {
        // the diagonal tile's inverse on the row's own right-hand side: D_i^{-1} (forward), D_i^{-T} (backward).
        // The sums over the lanes end a link of the dependency chain; as one butterfly per value
        // they bound the forward sweep where the factor is small or FP64 (64 subdomains of 6^3
        // elements, FP64 interior: 166 us against 54 us for the backward sweep).  Whole calls with
        // lane_sums instead: FP64 24^3 elasticity 84.6 -> 73.9 ms, FP32 solve of 24^3 (8 subdomains)
        // 18.3 -> 15.5 ms, FP64 operator on 8 columns (48^3) 9.61 -> 7.94 ms, same bits
        if (!BWD) {
          const bool signed_rows = L.indefinite != 0;   // forward output is S L^{-1} b
          V2 a[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) a[r] = *(const V2*)(tl + (warp + 8 * r) * NB + 2 * lane);
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            const V2 rv = *(const V2*)(&rhs[q][2 * lane]);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              const T d = a[r].x * rv.x + a[r].y * rv.y;
              acc[q][r] = GRP ? acc[q][r] + d : d;
            }
          }
          lane_sums<NV>(&acc[0][0], lane);
          if (writer)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
              const int q = (f0 + c) / 8, row = warp + 8 * ((f0 + c) % 8);
              const T yv = (&acc[0][0])[c];
              const T out = signed_rows ? yv * s_sg[row] : yv;
              v[q * vstride + i * NB + row] = out;
              pub_st(pv + q * vstride + i * NB + row, out);
            }
        } else {
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int row = warp + 8 * r;
            const V2 a = *(const V2*)(tl + row * NB + 2 * lane);
#pragma unroll
            for (int q = 0; q < NR; ++q) {
              accc[q][0] += a.x * rhs[q][row];
              accc[q][1] += a.y * rhs[q][row];
            }
          }
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            red[warp][q][2 * lane] = accc[q][0];
            red[warp][q][2 * lane + 1] = accc[q][1];
          }
          __syncthreads();
          for (int e = tid; e < NR * NB; e += kThreads) {
            const int q = e / NB, c = e % NB;
            T a = (T)0;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) a += red[w][q][c];
            v[q * vstride + i * NB + c] = a;
            pub_st(pv + q * vstride + i * NB + c, a);
          }
        }
      }
      __syncthreads();   // every thread is done with this stage
      ++cons;
      if (tid == 0 && k + S < ntile) {
        const uint32_t ns = (cons + S - 1) % S;   // the slot just released
        mbar_expect_tx(&full[ns], (uint32_t)(NB2 * sizeof(T)));
        bulk_g2s(stage + ns * NB2, tile_src(k + S), (uint32_t)(NB2 * sizeof(T)), &full[ns]);
        ++issued;
      }
    }
  }
  // After a lost tile wait, copies may still be in flight into this CTA's shared memory:
  // wait (bounded) for the last phase issued on every slot before the CTA exits.
  if (tid == 0 && lost) {
    for (uint32_t c = (issued > (uint32_t)S ? issued - S : 0u); c < issued; ++c) {
      long long spins = 0;
      while (!mbar_try_wait(&full[c % S], (c / S) & 1u) && ++spins < kSpinLimit) {
      }
    }
  }
}

}  // namespace

// Task lists and the scratch buffer live in the level (see capi.cpp).  scratch: two task counters (forward,
// backward) in its first 64 bytes, then the publication buffers of either direction (solutions, with GRP also the
// remaining right-hand sides), n_vec NR words of T each; one
// memset to all ones resets what a launch uses (counters start at -1).  A pair resets both directions at
// once and its backward sweep is launched over the forward sweep's end (pdl.cuh): per pair one memset
// instead of four, each 1.5 to 2 us between short sweeps.
template <typename T, int S, int NR, bool GRP>
void launch_sweep_s(const LevelDev& L, T* vec, const int2* const* tasks, const int* ntasks, int part, int which,
                    void* scratch, int grid_max, cudaStream_t st) {
  const size_t dyn = (size_t)S * NB2 * sizeof(T);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_sweep<T, S, false, NR, GRP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    cudaFuncSetAttribute(k_sweep<T, S, true, NR, GRP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    attr = true;
  }
  const size_t words = (size_t)L.n_vec * NR, dir = words * (GRP ? 2 : 1);   // published words per direction
  int* ctrl = (int*)scratch;
  T* pub = (T*)((char*)scratch + 64);
  cudaMemsetAsync(scratch, 0xFF, 64 + sizeof(T) * dir * (which == 2 ? 2 : 1), st);
  if (which != 1) {
    note_launch();
    k_sweep<T, S, false, NR, GRP><<<ntasks[0] < grid_max ? ntasks[0] : grid_max, kThreads, dyn, st>>>(
        L, vec, L.n_vec, tasks[0], ntasks[0], part, ctrl, pub, pub + words);
  }
  if (which == 2) {
    note_launch();
    launch_pdl(k_sweep<T, S, true, NR, GRP>, ntasks[1] < grid_max ? ntasks[1] : grid_max, kThreads, dyn, st, L, vec,
               (int64_t)L.n_vec, tasks[1], ntasks[1], part, ctrl + 1, pub + dir, pub + dir + words);
  } else if (which == 1) {
    note_launch();
    k_sweep<T, S, true, NR, GRP><<<ntasks[1] < grid_max ? ntasks[1] : grid_max, kThreads, dyn, st>>>(
        L, vec, L.n_vec, tasks[1], ntasks[1], part, ctrl, pub, pub + words);
  }
}

template <typename T, int S, int NR>
void launch_sweep_g(const LevelDev& L, T* vec, const int2* const* tasks, const int* ntasks, int part, int which,
                    void* scratch, int grid_max, cudaStream_t st) {
  // Any number of columns, so that a column of a block has the arithmetic of a single one.  It pays up to two columns,
  // where the chain of block rows counts: 24^3 solve (8 subdomains) 8.41 -> 7.50 ms, tetrahedra 11.4 -> 10.9, 48^3
  // (bound by HBM) as before.  With eight columns the tiles' products bound the sweep and the extra exchange
  // costs up to 1 %: FP64 operator on 8 columns (48^3) 6.11 -> 6.16 ms, 64^3 with 16 loads 444.6 -> 448.3.
  if constexpr (sizeof(T) == 4) {
    if (part == 0 && L.x_kept) {   // the inverses of the 256-wide diagonal blocks are at hand
      launch_sweep_s<T, S, NR, true>(L, vec, tasks, ntasks, part, which, scratch, grid_max, st);
      return;
    }
  }
  launch_sweep_s<T, S, NR, false>(L, vec, tasks, ntasks, part, which, scratch, grid_max, st);
}

template <typename T, int S>
void launch_sweep_nr(const LevelDev& L, T* vec, const int2* const* tasks, const int* ntasks, int part, int which,
                     void* scratch, int grid_max, int nr, cudaStream_t st) {
  // right-hand sides in groups of up to 8 (FP32) / 4 (FP64), each group one launch over the factor
  constexpr int kMaxNR = sizeof(T) == 4 ? 8 : 4;
  for (int r0 = 0; r0 < nr;) {
    const int left = nr - r0;
    const int g = left >= kMaxNR ? kMaxNR : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    T* v = vec + (int64_t)r0 * L.n_vec;
    if (g == 8)
      launch_sweep_g<T, S, (sizeof(T) == 4 ? 8 : 4)>(L, v, tasks, ntasks, part, which, scratch, grid_max, st);
    else if (g == 4)
      launch_sweep_g<T, S, 4>(L, v, tasks, ntasks, part, which, scratch, grid_max, st);
    else if (g == 2)
      launch_sweep_g<T, S, 2>(L, v, tasks, ntasks, part, which, scratch, grid_max, st);
    else
      launch_sweep_g<T, S, 1>(L, v, tasks, ntasks, part, which, scratch, grid_max, st);
    r0 += g;
  }
}

// deep: the longer tile ring (FP32: 6 stages, FP64: 3); shallow: FP32 4, FP64 2.  nr columns of length n_vec
// at vec.
template <typename T>
void launch_sweep(const LevelDev& L, T* vec, const int2* const* tasks, const int* ntasks, int part, int which,
                  void* scratch, int grid_max, int deep, cudaStream_t st, int nr) {
  if (ntasks[which == 1 ? 1 : 0] <= 0 || nr <= 0) return;
  if (sizeof(T) == 4) {
    if (deep)
      launch_sweep_nr<T, 6>(L, vec, tasks, ntasks, part, which, scratch, grid_max, nr, st);
    else
      launch_sweep_nr<T, 4>(L, vec, tasks, ntasks, part, which, scratch, grid_max, nr, st);
  } else {
    if (deep)
      launch_sweep_nr<T, 3>(L, vec, tasks, ntasks, part, which, scratch, grid_max, nr, st);
    else
      launch_sweep_nr<T, 2>(L, vec, tasks, ntasks, part, which, scratch, grid_max, nr, st);
  }
}

template void launch_sweep<float>(const LevelDev&, float*, const int2* const*, const int*, int, int, void*, int, int,
                                  cudaStream_t, int);
template void launch_sweep<double>(const LevelDev&, double*, const int2* const*, const int*, int, int, void*, int, int,
                                   cudaStream_t, int);

}  // namespace bddc
