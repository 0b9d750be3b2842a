// Dense per-subdomain kernels, batched over all subdomains of a level.
//
//  * Partial Cholesky of the augmented matrix [A_i; C_i], A_i = K_i + rho C_i^T C_i
//    (right-looking, NB x NB tiles): gives L_i (A_i = L_i L_i^T) and Y_i = C_i L_i^{-T}.
//    With the local order (interior, interface) the leading block of L_i factors K_II
//    ("prepare interior correction", Algorithm 1) and the trailing block factors the
//    constrained Neumann problem of Eq. psi_def / Eq. sub_cor restricted to the interface.
//  * G_i = Y_i Y_i^T = C_i A_i^{-1} C_i^T (FP64), its Cholesky factor and inverse;
//    Psi_i = A_i^{-1} C_i^T G_i^{-1} (so C_i Psi_i = I and K_i Psi_i = -C_i^T Lambda_i with
//    Lambda_i = R - G_i^{-1}), K_Ci = Psi_i^T K_i Psi_i = -Lambda_i = G_i^{-1} - R, where
//    R = diag(rho c_rho) (rho on the rows that augment A_i, 0 on Stokes pressure rows).
#include "internal.h"
#include "pdl.cuh"
#include "reduce.cuh"

namespace bddc {

namespace {

__device__ __forceinline__ int64_t tile_index(int i, int j, int Bc) {
  return i < Bc ? ((int64_t)i * (i + 1) / 2 + j) : ((int64_t)Bc * (Bc + 1) / 2 + (int64_t)(i - Bc) * Bc + j);
}

template <typename T>
__device__ __forceinline__ T* tile_ptr(const SubMeta& m, void* base, int i, int j) {
  return (T*)base + m.tile_off + tile_index(i, j, m.Bc) * NB2;
}

__device__ __forceinline__ void flag_breakdown(int* status, int sub) {
  atomicExch(status + 0, 1);
  atomicMin(status + 1, sub);
}

constexpr int LDS = NB + 4;   // k-major shared tile stride (multiple of 4 for vector loads)

template <typename T>
__device__ __forceinline__ void load_kmajor(T* s, const T* __restrict__ g) {
  // s[m * LDS + r] = g[r * NB + m]
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
    const int r = t / NB, m = t % NB;
    s[m * LDS + r] = g[t];
  }
}

// 16-byte aligned vectors of four entries (global or shared memory)
template <typename T>
__device__ __forceinline__ void load4(T (&v)[4], const T* p);
template <>
__device__ __forceinline__ void load4<float>(float (&v)[4], const float* p) {
  const float4 a = *(const float4*)p;
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
}
template <>
__device__ __forceinline__ void load4<double>(double (&v)[4], const double* p) {
  const double2 a = *(const double2*)p, b = *(const double2*)(p + 2);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}
template <typename T>
__device__ __forceinline__ void store4(T* p, const T (&v)[4]);
template <>
__device__ __forceinline__ void store4<float>(float* p, const float (&v)[4]) {
  *(float4*)p = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void store4<double>(double* p, const double (&v)[4]) {
  *(double2*)p = make_double2(v[0], v[1]);
  *(double2*)(p + 2) = make_double2(v[2], v[3]);
}

// acc[i][j] += sum_m A[4ty+i][m] * B[4tx+j][m] with both operands k-major in shared memory
template <typename T>
__device__ __forceinline__ void gemm_nt_4x4(const T* As, const T* Bs, T acc[4][4], int tx, int ty) {
#pragma unroll 8
  for (int m = 0; m < NB; ++m) {
    T a[4], b[4];
    load4(a, As + m * LDS + 4 * ty);   // LDS and the tile offsets keep these 16-byte aligned
    load4(b, Bs + m * LDS + 4 * tx);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * b[j];
  }
}

// ---- step k, part 1: factor the diagonal tile and invert it -------------------------------
// One CTA of 256 threads; smem_raw holds 2 NB (NB + 1) entries of T.  Called by k_potrf_diag and,
// for the next block column of a panel, by the in-panel update kernel right after it has updated
// that diagonal tile (so that the factorisation of a panel's later diagonal tiles overlaps the
// rest of the previous step's update instead of taking a launch of its own).
template <typename T>
__device__ void factor_diag_tile(const LevelDev& L, const SubMeta& m, int s, int k, unsigned char* smem_raw) {
  T(*A)[NB + 1] = (T(*)[NB + 1])smem_raw;                 // the tile, then its factor L
  T(*X)[NB + 1] = (T(*)[NB + 1])(smem_raw + sizeof(T) * NB * (NB + 1));   // L^{-1}
  __shared__ int bad;
  T* g = tile_ptr<T>(m, L.tiles, k, k);
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
    const int r = t / NB, c = t % NB;
    A[r][c] = c <= r ? g[t] : (T)0;
  }
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  __shared__ T sg[NB];
  __shared__ T dd[NB];   // pivots as used by the elimination (1 where a pivot failed)
  // Right-looking elimination on the unscaled columns: at column j every entry below the pivot
  // is updated as a_ic -= (a_ij / d_j) a_cj (d_j = a_jj after the updates of the columns before
  // j), which equals l_ij s_j l_cj with l_ij = a_ij / (s_j sqrt|d_j|), s_j = sign d_j; the columns
  // are scaled to L afterwards.  Blocked by panels of 16 columns, with three barriers per panel:
  //   (a1) warp 0 eliminates inside the 16 x 16 diagonal block from registers: lane i + 16 h holds row i's
  //        columns of parity h, column j and its pivot come by shuffle (from shared memory, each
  //        step was a chain of up to eight dependent reads and writes);
  //   (a2) one thread per row below it applies the panel's 16 eliminations to its 16 panel
  //        entries and keeps the multipliers a_ij / d_j (in X, unused until the inverse);
  //   (b)  the trailing block takes a_rc -= sum_j (a_rj / d_j) a_cj over the panel columns, 2 x 2 entries per
  //        thread, the blocks on and below the diagonal only.
  // Every entry receives the same updates in the same order (j ascending) as column by column.
  // The chain of diagonal tiles is the critical path of the factorisation (one CTA per subdomain): FP32 38 -> 25 us
  // per tile with the factor and the inverse, FP64 160 -> 150 (bound by its dependent divisions and products).
  {
    constexpr int PW = 16;
    T(*F)[PW + 1] = (T(*)[PW + 1])(&X[0][0]);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int p0 = 0; p0 < NB; p0 += PW) {
      if (warp == 0) {
        const int i = lane & 15, half = lane >> 4;
        T a[PW / 2];   // row i, columns 2 q + half (above the diagonal: never read by another row)
#pragma unroll
        for (int q = 0; q < PW / 2; ++q) a[q] = A[p0 + i][p0 + 2 * q + half];
#pragma unroll
        for (int j = 0; j < PW; ++j) {
          const T v = __shfl_sync(0xffffffffu, a[j >> 1], ((j & 1) << 4) | i);   // a_ij
          T d = __shfl_sync(0xffffffffu, v, j);
          // a failed pivot (flagged below from the same value) continues as 1, as in the scaling
          if (L.indefinite ? !(fabs(d) > (T)1e-30) : !(d > (T)0)) d = (T)1;
          if (lane == 0) dd[p0 + j] = d;
          const T f = v / d;
#pragma unroll
          for (int q = j >> 1; q < PW / 2; ++q) {
            const T vc = __shfl_sync(0xffffffffu, v, 2 * q + half);   // a_cj, c = 2 q + half
            if (2 * q + half > j) a[q] -= f * vc;
          }
        }
#pragma unroll
        for (int q = 0; q < PW / 2; ++q)
          if (2 * q + half <= i) A[p0 + i][p0 + 2 * q + half] = a[q];
      }
      __syncthreads();
      const int nb = NB - p0 - PW;   // rows below the diagonal block
      if (tid < nb) {
        const int i = p0 + PW + tid;
        T a[PW];
#pragma unroll
        for (int jj = 0; jj < PW; ++jj) a[jj] = A[i][p0 + jj];
#pragma unroll
        for (int jj = 0; jj < PW; ++jj) {
          const T f = a[jj] / dd[p0 + jj];
#pragma unroll
          for (int c = jj + 1; c < PW; ++c) a[c] -= f * A[p0 + c][p0 + jj];
          F[tid][jj] = f;   // last, so that the next column's reads run beside its division
        }
#pragma unroll
        for (int jj = 0; jj < PW; ++jj) A[i][p0 + jj] = a[jj];
      }
      __syncthreads();
      const int nt = nb / 2;   // block rows nt - 1 - u and u together hold nt + 1 blocks
      for (int e = tid; e < nt / 2 * (nt + 1); e += blockDim.x) {
        const int u = e / (nt + 1), q = e % (nt + 1);
        const int r = 2 * (q < nt - u ? nt - 1 - u : u), c = 2 * (q < nt - u ? q : q - (nt - u));
        T* A0 = &A[p0 + PW + r][p0 + PW + c];
        T* A1 = A0 + NB + 1;
        T s00 = A0[0], s01 = A0[1], s10 = A1[0], s11 = A1[1];
#pragma unroll
        for (int jj = 0; jj < PW; ++jj) {
          const T f0 = F[r][jj], f1 = F[r + 1][jj];
          const T v0 = A[p0 + PW + c][p0 + jj], v1 = A[p0 + PW + c + 1][p0 + jj];
          s00 -= f0 * v0;
          s01 -= f0 * v1;
          s10 -= f1 * v0;
          s11 -= f1 * v1;
        }
        A0[0] = s00;
        if (c < r) A0[1] = s01;
        A1[0] = s10;
        A1[1] = s11;
      }
      __syncthreads();
    }
  }
  if (threadIdx.x < NB) {
    const int j = threadIdx.x;
    T d = A[j][j];
    T sj = (T)1;
    bool b = false;
    if (L.indefinite) {
      if (!(fabs(d) > (T)1e-30)) {
        b = true;
        d = (T)1;
      }
      if (d < (T)0) {
        sj = (T)-1;
        d = -d;
      }
    } else if (!(d > (T)0)) {
      b = true;
      d = (T)1;
    }
    if (b) bad = 1;
    sg[j] = sj;
    X[0][j] = sqrt(d);   // pivots, kept in the first row of X until the inverse is formed
  }
  __syncthreads();
  for (int t = threadIdx.x; t < NB / 2 * (NB - 1); t += blockDim.x) {   // rows NB - 1 - u and u: NB - 1 entries
    const int u = t / (NB - 1), q = t % (NB - 1);
    const int r = q < NB - 1 - u ? NB - 1 - u : u, c = q < NB - 1 - u ? q : q - (NB - 1 - u);
    A[r][c] /= X[0][c] * sg[c];
  }
  __syncthreads();
  if (threadIdx.x < NB) A[threadIdx.x][threadIdx.x] = X[0][threadIdx.x];
  __syncthreads();
  if (threadIdx.x < NB) ((T*)L.sgn)[m.vec_off + (int64_t)k * NB + threadIdx.x] = sg[threadIdx.x];
  if (threadIdx.x == 0 && bad) flag_breakdown(L.status, s);
  // X = L^{-1} by 16 x 16 blocks: the four diagonal blocks X_PP = L_PP^{-1} by forward
  // substitution (half a warp each, one lane per column, in registers), then the blocks below the diagonal by
  // their distance d = Q - P: X_QP = -X_QQ (sum_{P <= K < Q} L_QK X_KP), the inner sum into a
  // scratch block first (3 - d + 1 blocks per distance, one entry per thread and block).
  {
    constexpr int PW = 16;
    __shared__ T Tq[3][PW][PW + 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp < 2) {
      const int p0 = PW * (2 * warp + (lane >> 4)), c = lane & 15;
      T x[PW];
#pragma unroll
      for (int i = 0; i < PW; ++i) {
        T part = (T)0;   // x[q] = 0 above the column's own row
#pragma unroll
        for (int q = 0; q < i; ++q) part += A[p0 + i][p0 + q] * x[q];
        x[i] = i < c ? (T)0 : (i == c ? (T)1 : -part) / A[p0 + i][p0 + i];
      }
#pragma unroll
      for (int i = 0; i < PW; ++i) X[p0 + i][p0 + c] = x[i];
    }
    __syncthreads();
    for (int dist = 1; dist < 4; ++dist) {
      const int nblk = 4 - dist;
      for (int e = tid; e < nblk * PW * PW; e += blockDim.x) {   // T = sum_K L_QK X_KP
        const int bq = e / (PW * PW), r = (e / PW) % PW, c = e % PW;
        const int P = bq, Q = bq + dist;
        T acc = (T)0;
        for (int K = P; K < Q; ++K)
#pragma unroll
          for (int q = 0; q < PW; ++q) acc += A[PW * Q + r][PW * K + q] * X[PW * K + q][PW * P + c];
        Tq[bq][r][c] = acc;
      }
      __syncthreads();
      for (int e = tid; e < nblk * PW * PW; e += blockDim.x) {   // X_QP = -X_QQ T
        const int bq = e / (PW * PW), r = (e / PW) % PW, c = e % PW;
        const int P = bq, Q = bq + dist;
        T acc = (T)0;
        for (int q0 = 0; q0 <= r; q0 += 4)   // X_QQ is zero above its diagonal
#pragma unroll
          for (int q = q0; q < q0 + 4; ++q) acc += X[PW * Q + r][PW * Q + q] * Tq[bq][q][c];
        X[PW * Q + r][PW * P + c] = -acc;
      }
      __syncthreads();
    }
  }
  T* dv = (T*)L.dinv + m.dinv_off + (int64_t)k * NB2;
  for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
    const int r = t / NB, c = t % NB;
    dv[t] = c <= r ? X[r][c] : (T)0;
    g[t] = A[r][c];
  }
}

template <typename T>
__global__ void k_potrf_diag(LevelDev L, int k) {
  const int s = blockIdx.x;
  const SubMeta m = L.meta[s];
  if (k >= m.Bc) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  factor_diag_tile<T>(L, m, s, k, smem_raw);
}

// ---- step k, part 2: panel L(i,k) = A(i,k) L_kk^{-T} for i = k+1 .. R-1 --------------------
// rlim > 0: only the rows of the diagonal block, i < min(rlim, Bc) (the rows below it are solved
// on the tensor cores with the block's inverse)
template <typename T>
__global__ void k_trsm_panel(LevelDev L, int k, int rlim) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int i = k + 1 + blockIdx.x;
  const int ilim = rlim > 0 ? (rlim < m.Bc ? rlim : m.Bc) : (k < m.nIb ? (int)m.Bc : (int)m.R);   // see k_syrk_update
  if (k >= m.Bc || i >= ilim) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* As = (T*)smem_raw;
  T* Xs = As + NB * LDS;
  T* g = tile_ptr<T>(m, L.tiles, i, k);
  load_kmajor(As, g);
  load_kmajor(Xs, (const T*)L.dinv + m.dinv_off + (int64_t)k * NB2);
  __syncthreads();
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  T acc[4][4] = {};
  gemm_nt_4x4(As, Xs, acc, tx, ty);
  __syncthreads();
  const T* sk = (const T*)L.sgn + m.vec_off + (int64_t)k * NB;   // L(i,k) = A(i,k) L_kk^{-T} S_k
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    T v[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) v[b] = acc[a][b] * sk[4 * tx + b];
    store4(g + (4 * ty + a) * NB + 4 * tx, v);
  }
}

// The same panel by blocks of 16 rows, for launches with fewer 64 x 64 tiles than SMs: an FP64 tile takes
// one SM 131,000 cycles of FP64 products, so the coarsest level's panels (one subdomain, 3,345 DOFs: 52
// tiles at most) ran on a third of the chip, 72 us per step.
template <typename T>
__global__ void __launch_bounds__(256) k_trsm_panel16(LevelDev L, int k, int rlim) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int i = k + 1 + (int)(blockIdx.x >> 2), r0 = 16 * (blockIdx.x & 3);
  const int ilim = rlim > 0 ? (rlim < m.Bc ? rlim : m.Bc) : (k < m.nIb ? (int)m.Bc : (int)m.R);
  if (k >= m.Bc || i >= ilim) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Xs = (T*)smem_raw;             // k-major inverse of the diagonal tile
  T* As = Xs + NB * LDS;            // 16 rows of the panel tile
  T* g = tile_ptr<T>(m, L.tiles, i, k) + r0 * NB;
  load_kmajor(Xs, (const T*)L.dinv + m.dinv_off + (int64_t)k * NB2);
  for (int t = threadIdx.x; t < 16 * NB; t += 256) As[t] = g[t];
  __syncthreads();
  const int tx = threadIdx.x % 16, r = threadIdx.x / 16;
  T acc[4] = {};
#pragma unroll 8
  for (int q = 0; q < NB; ++q) {
    const T a = As[r * NB + q];
    T x[4];
    load4(x, Xs + q * LDS + 4 * tx);
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[b] += a * x[b];
  }
  const T* sk = (const T*)L.sgn + m.vec_off + (int64_t)k * NB;
#pragma unroll
  for (int b = 0; b < 4; ++b) acc[b] *= sk[4 * tx + b];
  store4(g + r * NB + 4 * tx, acc);
}

// ---- inverse of a sub-panel's 256 x 256 diagonal block (FP32, the tensor-core panel solve) ----
// X = L_D^{-1} for the block D = [k0, k0 + nd) (nd = min(4, Bc - k0)): X_QQ = L_QQ^{-1} (the stored
// inverse of the diagonal tile) and X_QP = -X_QQ sum_{P <= K < Q} L_QK X_KP for P < Q.  Block row
// Q needs the tiles L_QK (K < Q) and the rows of X above it, so it is formed during step k0 + Q of
// the block's factorisation, by blocks of that step's in-block update launch (next to the one that
// factors tile Q + 1).  One CTA of 256 threads takes 16 columns c0 .. c0 + 15 of X_QP (thread:
// row r, columns cg .. cg + 3), the sums in ascending K and t; X_QP is stored as a row-major tile
// at x_tile(k0, Q, P) (the diagonal tiles X_QQ are read from the inverses).
__device__ void xinv_row_part(const LevelDev& L, const SubMeta& m, int k0, int Q, int P, int c0,
                              unsigned char* smem_raw) {
  float(*Ls)[NB + 1] = (float(*)[NB + 1])smem_raw;                               // L_QK, then L_QQ^{-1}
  float(*Xk)[16] = (float(*)[16])(smem_raw + sizeof(float) * NB * (NB + 1));     // X_KP(:, c0 ..)
  float(*Ts)[16] = (float(*)[16])(smem_raw + sizeof(float) * NB * (NB + 1 + 16));
  const int tid = threadIdx.x, r = tid >> 2, cg = 4 * (tid & 3);
  const float* dinv = (const float*)L.dinv + m.dinv_off;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int K = P; K < Q; ++K) {   // T = sum_K L_QK X_KP
    const float* lq = tile_ptr<float>(m, L.tiles, k0 + Q, k0 + K);
    const float* xk = K == P ? dinv + (int64_t)(k0 + P) * NB2 : L.xinv + x_tile(m, k0, K, P);
    for (int e = tid; e < NB2; e += blockDim.x) Ls[e >> 6][e & 63] = lq[e];
    for (int e = tid; e < NB * 16; e += blockDim.x) Xk[e >> 4][e & 15] = xk[(e >> 4) * NB + c0 + (e & 15)];
    __syncthreads();
#pragma unroll 8
    for (int t = 0; t < NB; ++t) {
      const float a = Ls[r][t];
      const float4 x = *(const float4*)&Xk[t][cg];
      acc[0] += a * x.x;
      acc[1] += a * x.y;
      acc[2] += a * x.z;
      acc[3] += a * x.w;
    }
    __syncthreads();
  }
  *(float4*)&Ts[r][cg] = make_float4(acc[0], acc[1], acc[2], acc[3]);
  const float* dQ = dinv + (int64_t)(k0 + Q) * NB2;   // X_QP = -L_QQ^{-1} T (lower triangular)
  for (int e = tid; e < NB2; e += blockDim.x) Ls[e >> 6][e & 63] = dQ[e];
  __syncthreads();
  float y[4] = {0.f, 0.f, 0.f, 0.f};
  for (int t = 0; t <= r; ++t) {
    const float a = Ls[r][t];
    const float4 x = *(const float4*)&Ts[t][cg];
    y[0] += a * x.x;
    y[1] += a * x.y;
    y[2] += a * x.z;
    y[3] += a * x.w;
  }
  float* dst = L.xinv + x_tile(m, k0, Q, P) + r * NB + c0 + cg;
  *(float4*)dst = make_float4(-y[0], -y[1], -y[2], -y[3]);
}

// ---- step k, part 3: trailing update A(i,j) -= L(i,k) L(j,k)^T, k < j <= i, j < min(Bc, jmax) --
// fuse_next: the block that updates the next diagonal tile (k+1, k+1) (always block 0 of its
// subdomain) factors and inverts it right away, and step k+1 launches no k_potrf_diag.
// rlim > 0: only rows i < min(rlim, Bc) (the diagonal block of a sub-panel).  xinv (FP32 panel
// solves): the blocks n_upd .. n_upd + 4 xq - 1 of the grid form block row xq = k - k0 of the
// inverse of the diagonal block [k0, k0 + 4) (block column P = e / 4, columns 16 (e % 4) ..).
template <typename T>
__global__ void k_syrk_update(LevelDev L, int k, int jmax, int fuse_next, int rlim, int n_upd, int xinv,
                              int k0) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  if ((int)blockIdx.x >= n_upd) {
    if constexpr (sizeof(T) == 4) {
      const int e = (int)blockIdx.x - n_upd, Q = k - k0;
      extern __shared__ __align__(16) unsigned char smem_raw[];
      if (xinv && Q < m.Bc - k0) xinv_row_part(L, m, k0, Q, e >> 2, 16 * (e & 3), smem_raw);
    }
    return;
  }
  if (k >= m.Bc) return;
  const int jend = jmax < m.Bc ? jmax : m.Bc;
  // constraints touch interface DOFs only, so the constraint rows are zero in interior columns k < nIb
  // (a fifth of the trailing tiles of 64 subdomains of 6^3 elements)
  const int ilim = rlim > 0 ? (rlim < m.Bc ? rlim : m.Bc) : (k < m.nIb ? (int)m.Bc : (int)m.R);
  int t = blockIdx.x, j = k + 1, i = -1;
  for (; j < jend; ++j) {
    const int cnt = ilim - j;
    if (t < cnt) {
      i = j + t;
      break;
    }
    t -= cnt;
  }
  if (i < 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* As = (T*)smem_raw;
  T* Bs = As + NB * LDS;
  load_kmajor(As, tile_ptr<T>(m, L.tiles, i, k));
  load_kmajor(Bs, tile_ptr<T>(m, L.tiles, j, k));
  __syncthreads();
  if (L.indefinite) {   // A(i,j) -= L(i,k) S_k L(j,k)^T: fold S_k into the k-major B operand
    const T* sk = (const T*)L.sgn + m.vec_off + (int64_t)k * NB;
    for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) Bs[(t / NB) * LDS + (t % NB)] *= sk[t / NB];
    __syncthreads();
  }
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  T acc[4][4] = {};
  gemm_nt_4x4(As, Bs, acc, tx, ty);
  T* c = tile_ptr<T>(m, L.tiles, i, j);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    T v[4];
    load4(v, c + (4 * ty + a) * NB + 4 * tx);
#pragma unroll
    for (int b = 0; b < 4; ++b) v[b] -= acc[a][b];
    store4(c + (4 * ty + a) * NB + 4 * tx, v);
  }
  if (fuse_next && i == k + 1 && j == k + 1) {   // block-uniform
    __syncthreads();   // the updated tile is in global memory, visible to the whole block
    factor_diag_tile<T>(L, m, s, k + 1, smem_raw);
  }
}

// ---- G = Y_G Y_G^T in FP64, Cholesky, inverse; K_C = G^{-1} - rho I ----------------------
// FP64 levels: one warp per entry (a, b), a >= b, of one subdomain's G; lanes stride over the interface
// columns (contiguous inside a tile row), FP64 products, fixed-order warp reduction
__global__ void k_gram(LevelDev L) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int nc = m.nc;
  const int pair = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (pair >= nc * nc) return;
  const int a = pair / nc, b = pair % nc;
  if (b > a) return;
  const double* ya = tile_ptr<double>(m, L.tiles, m.Bc + a / NB, m.nIb) + (a % NB) * NB;
  const double* yb = tile_ptr<double>(m, L.tiles, m.Bc + b / NB, m.nIb) + (b % NB) * NB;
  const double* sG = (const double*)L.sgn + m.vec_off + (int64_t)m.nIb * NB;   // G = Y S Y^T
  double acc = 0.0;
  for (int c = lane; c < m.nGb * NB; c += 32) {
    const int64_t o = (int64_t)(c / NB) * NB2 + (c % NB);
    acc += (double)ya[o] * (double)sG[c] * (double)yb[o];
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    double* G = L.Ginv + m.g_off;
    G[a * nc + b] = acc;
    G[b * nc + a] = acc;
  }
}

// ---- FP32 factors: G and Z = Y^T G^{-1} with sums in three FP32 parts -------------------------
// The FP64 units give 2 products per cycle and SM, so these two products (n_G n_c^2 each) were bound by
// them, with one warp or thread per entry and few blocks where n_c is large: 48^3 elasticity (n_c <= 78)
// 1.5 + 1.4 ms per set-up, 64 k-means subdomains (n_c <= 258) 15 + 22 ms.  The factor's entries are FP32, so
// a product a b is p + e exactly (e = fma(a, b, -p)), and a sum is kept as three unevaluated FP32 parts:
// p goes into the first, what its addition rounds off and e into the second, what those additions round
// off into the third, each by two-sum (Knuth; Dekker).  Only the additions into the third part round, at
// 2^-72 of the sum: 22 FP32 operations per product at 128 lanes per cycle, and the sum comes out as exact as FP64
// holds it.  With two parts (10 operations) the second rounds at every addition, and the error grows with the
// length: root mean square relative to the sum for 64 / 1,024 / 6,016 squares 2^-46 / 2^-42 / 2^-40, where FP64 (32
// lanes, then a tree) keeps 2^-53.6 / 2^-53 / 2^-50 and three parts 2^-54.2 at any of them.
// One block per 32 x 32 part of the result, both operands k-major in shared memory, 2 x 2 entries per thread: bound
// by the FP32 operations, with 64 x 64 parts there were too few blocks (48^3: 192 of them for 152 SMs) and more
// padding (n_c = 78 took 128 columns, now 96).  48^3 set-up and solve: pairs 96.2 ms, three parts by 64 x 64 97.7,
// by 32 x 32 96.4; 64 k-means subdomains 157.4 / 159.6 / 159.2.  Y is scaled by 2^k, G^{-1} by 2^-2k with 4^k about rho (G is at most 1 / rho), exactly, so that the small
// parts stay above FP32's least numbers whatever the unit of the moduli.
struct Sum3 {
  float hi, mid, lo;
};

__device__ __forceinline__ float two_sum(float& s, float x) {   // s + x rounded into s; returns what was lost
  const float t = __fadd_rn(s, x);
  const float b = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
  s = t;
  return err;
}

__device__ __forceinline__ void add3(Sum3& s, float p, float e) {   // s += p + e
  float r = two_sum(s.hi, p);
  const float l = two_sum(r, e);
  s.lo = __fadd_rn(s.lo, __fadd_rn(l, two_sum(s.mid, r)));
}

__device__ __forceinline__ double value3(const Sum3& s) { return (double)s.hi + ((double)s.mid + (double)s.lo); }

__device__ __forceinline__ int gram_exponent(const LevelDev& L, int s) {
  const double rho = L.rho[s];
  const int k = rho > 0.0 && rho < 1e300 ? ilogb(rho) / 2 : 0;
  return min(max(k, -60), 60);
}

constexpr int GB = 32;       // edge of a block's part of the result
constexpr int LDG = GB + 2;   // k-major stride: two-way bank conflicts in the transposing stores

// block (a, b), b <= a, of G = Y_G S Y_G^T
__global__ void __launch_bounds__(256) k_gram_f32(LevelDev L) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  int ab = 0, t = blockIdx.x;
  while (t > ab) t -= ++ab;   // row block ab, column block t
  const int r0 = GB * ab, c0 = GB * t, nc = m.nc;
  if (r0 >= nc) return;
  __shared__ __align__(16) float As[NB][LDG], Bs[NB][LDG];
  const float* sG = (const float*)L.sgn + m.vec_off + (int64_t)m.nIb * NB;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16, ex = gram_exponent(L, s);
  const float sc = ldexpf(1.f, ex);
  Sum3 acc[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = {0.f, 0.f, 0.f};
  for (int c = 0; c < m.nGb; ++c) {
    const float* ya = tile_ptr<float>(m, L.tiles, m.Bc + r0 / NB, m.nIb + c) + (r0 % NB) * NB;
    const float* yb = tile_ptr<float>(m, L.tiles, m.Bc + c0 / NB, m.nIb + c) + (c0 % NB) * NB;
#pragma unroll
    for (int u = 0; u < GB * NB / 256; ++u) {
      const int e = threadIdx.x + 256 * u, r = e / NB, k = e % NB;
      As[k][r] = sc * ya[e];
      Bs[k][r] = sG[c * NB + k] * (sc * yb[e]);   // S = +-1: exact
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < NB; ++k) {
      const float2 av = *(const float2*)&As[k][2 * ty], bv = *(const float2*)&Bs[k][2 * tx];
      const float a[2] = {av.x, av.y}, b[2] = {bv.x, bv.y};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float p = __fmul_rn(a[i], b[j]);
          add3(acc[i][j], p, __fmaf_rn(a[i], b[j], -p));
        }
    }
    __syncthreads();
  }
  double* G = L.Ginv + m.g_off;
  double* G0 = L.G ? L.G + m.g_off : nullptr;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = r0 + 2 * ty + i, c = c0 + 2 * tx + j;
      if (r >= nc || c >= nc || c > r) continue;   // the diagonal blocks' upper halves mirror the lower
      const double v = ldexp(value3(acc[i][j]), -2 * ex);
      G[(int64_t)r * nc + c] = v;
      G[(int64_t)c * nc + r] = v;
      if (G0) {   // kept: Ginv is inverted in place
        G0[(int64_t)r * nc + c] = v;
        G0[(int64_t)c * nc + r] = v;
      }
    }
}

// rows 32 jb .. of Z = Y_G^T G^{-1}, columns 32 qb ..: G^{-1} as an FP32 pair (gh + gl, 2^-49); Z is rounded to FP32
__global__ void __launch_bounds__(256) k_psi_rhs_f32(LevelDev L) {
  const int j = blockIdx.x / (NB / GB), h0 = GB * (blockIdx.x % (NB / GB)), q0 = GB * blockIdx.y, s = blockIdx.z;
  const SubMeta m = L.meta[s];
  const int nc = m.nc;
  if (j >= m.nGb || q0 >= nc) return;
  __shared__ __align__(16) float Ys[NB][GB], Gh[NB][GB], Gl[NB][GB];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16, ex = gram_exponent(L, s);
  const float sc = ldexpf(1.f, ex);
  const double scg = ldexp(1.0, -2 * ex);
  const double* Gi = L.Ginv + m.g_off;
  Sum3 acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = {0.f, 0.f, 0.f};
  for (int p0 = 0; p0 < nc; p0 += NB) {
    const float* y = tile_ptr<float>(m, L.tiles, m.Bc + p0 / NB, m.nIb + j) + h0;
    const int pn = min(NB, nc - p0);
#pragma unroll
    for (int u = 0; u < GB * NB / 256; ++u) {
      const int e = threadIdx.x + 256 * u, p = e / GB, c = e % GB, gq = q0 + c;
      Ys[p][c] = sc * y[p * NB + c];
      const double g = p < pn && gq < nc ? scg * Gi[(int64_t)(p0 + p) * nc + gq] : 0.0;
      const float h = (float)g;
      Gh[p][c] = h;
      Gl[p][c] = (float)(g - (double)h);
    }
    __syncthreads();
#pragma unroll 4
    for (int p = 0; p < pn; ++p) {
      const float2 av = *(const float2*)&Ys[p][2 * ty], hv = *(const float2*)&Gh[p][2 * tx], lv = *(const float2*)&Gl[p][2 * tx];
      const float a[2] = {av.x, av.y}, h[2] = {hv.x, hv.y}, l[2] = {lv.x, lv.y};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float v = __fmul_rn(a[i], h[k]);
          add3(acc[i][k], v, __fmaf_rn(a[i], l[k], __fmaf_rn(a[i], h[k], -v)));
        }
    }
    __syncthreads();
  }
  float* Z = (float*)L.psi + m.psi_off;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int q = q0 + 2 * tx + k;
      if (q < nc) Z[(int64_t)(j * NB + h0 + 2 * ty + i) * nc + q] = (float)ldexp(value3(acc[i][k]), ex);
    }
}

// G^{-1} by Gauss-Jordan elimination with partial pivoting (indefinite levels), FP64, one block
// per subdomain; W (the K_C buffer) holds the eliminated copy of G.
__device__ void gauss_jordan_inverse(double* G, double* W, int n, int* bad) {
  __shared__ int piv_row;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    W[t] = G[t];
    G[t] = (t / n == t % n) ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    if (threadIdx.x == 0) {
      int best = j;
      double bv = fabs(W[j * n + j]);
      for (int i = j + 1; i < n; ++i)
        if (fabs(W[i * n + j]) > bv) {
          bv = fabs(W[i * n + j]);
          best = i;
        }
      if (!(bv > 0.0)) *bad = 1;
      piv_row = best;
    }
    __syncthreads();
    const int pr = piv_row;
    if (pr != j)
      for (int c = threadIdx.x; c < n; c += blockDim.x) {
        double a = W[j * n + c], b = W[pr * n + c];
        W[j * n + c] = b;
        W[pr * n + c] = a;
        a = G[j * n + c];
        b = G[pr * n + c];
        G[j * n + c] = b;
        G[pr * n + c] = a;
      }
    __syncthreads();
    const double inv = W[j * n + j] != 0.0 ? 1.0 / W[j * n + j] : 0.0;
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      W[j * n + c] *= inv;
      G[j * n + c] *= inv;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
      const int i = t / n, c = t % n;
      if (i == j) continue;
      const double f = W[i * n + j];
      if (c != j) W[i * n + c] -= f * W[j * n + c];
      G[i * n + c] -= f * G[j * n + c];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      if (i != j) W[i * n + j] = 0.0;
    __syncthreads();
  }
}

__global__ void k_small_chol_inv(LevelDev L) {
  const int s = blockIdx.x;
  const SubMeta m = L.meta[s];
  const int n = m.nc;
  if (n == 0) return;
  if (L.indefinite) {
    __shared__ int badi;
    if (threadIdx.x == 0) badi = 0;
    __syncthreads();
    double* G = L.Ginv + m.g_off;
    double* W = L.KC + m.g_off;
    gauss_jordan_inverse(G, W, n, &badi);
    __syncthreads();
    if (threadIdx.x == 0 && badi) flag_breakdown(L.status, s);
    const double rho = L.rho[s];
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
      const int a = t / n, b = t % n;
      W[t] = G[t] - (a == b ? rho * L.c_rho[m.c_off + a] : 0.0);   // K_C = G^{-1} - R
    }
    return;
  }
  double* G = L.Ginv + m.g_off;   // in: G (full), out: G^{-1}
  double* W = L.KC + m.g_off;     // scratch for L^{-1}, then K_C
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    if (threadIdx.x == 0) {
      double d = G[j * n + j];
      if (!(d > 0.0)) {
        bad = 1;
        d = 1.0;
      }
      G[j * n + j] = sqrt(d);
    }
    __syncthreads();
    const double piv = G[j * n + j];
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) G[i * n + j] /= piv;
    __syncthreads();
    const int w = n - 1 - j;
    for (int t = threadIdx.x; t < w * w; t += blockDim.x) {
      const int i = j + 1 + t / w, c = j + 1 + t % w;
      if (c <= i) G[i * n + c] -= G[i * n + j] * G[c * n + j];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && bad) flag_breakdown(L.status, s);
  // W = L^{-1} (lower), one column per thread
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    for (int r = 0; r < c; ++r) W[r * n + c] = 0.0;
    W[c * n + c] = 1.0 / G[c * n + c];
    for (int i = c + 1; i < n; ++i) {
      double acc = 0.0;
      for (int q = c; q < i; ++q) acc += G[i * n + q] * W[q * n + c];
      W[i * n + c] = -acc / G[i * n + i];
    }
  }
  __syncthreads();
  // G^{-1} = W^T W
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int a = t / n, b = t % n;
    double acc = 0.0;
    for (int q = (a > b ? a : b); q < n; ++q) acc += W[q * n + a] * W[q * n + b];
    G[t] = acc;   // safe: G's lower part (the factor) is no longer read
  }
  __syncthreads();
  const double rho = L.rho[s];
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int a = t / n, b = t % n;
    W[t] = G[t] - (a == b ? rho * L.c_rho[m.c_off + a] : 0.0);   // K_C = G^{-1} - R
  }
}

// ---- G^{-1} and K_C of SPD levels with many constraints per subdomain (max n_c > 96) ----------
// k_small_chol_inv works on one SM per subdomain, whose FP64 units give two products per cycle: n_c = 258
// took 10 ms, with one thread per column of L^{-1}.  Here only the Cholesky factorisation (n_c^3 / 6
// products) stays on one SM, by panels of 16 columns in shared memory; the inverse of the factor takes a
// warp per column and the product W^T W a thread per entry, over the whole chip.

constexpr int kPanelMaxNc = 1600;   // its panel of 16 columns takes 213 KB of shared memory

// G = L L^T in place; the strictly upper part receives L^T (its rows are the columns of L)
__global__ void __launch_bounds__(1024) k_gram_potrf(LevelDev L) {
  constexpr int PW = 16;
  const int s = blockIdx.x;
  const SubMeta m = L.meta[s];
  const int n = m.nc, tid = threadIdx.x;
  if (n == 0) return;
  double* G = L.Ginv + m.g_off;
  extern __shared__ __align__(16) double panel[];   // [n][PW + 1]: rows p0 .. of the panel
  __shared__ double diag[PW][PW + 1];
  __shared__ int bad;
  if (tid == 0) bad = 0;
  for (int p0 = 0; p0 < n; p0 += PW) {
    const int w = min(PW, n - p0), rows = n - p0 - w;
    __syncthreads();
    for (int e = tid; e < w * w; e += blockDim.x) diag[e / w][e % w] = G[(int64_t)(p0 + e / w) * n + p0 + e % w];
    __syncthreads();
    if (tid < 32) {   // the diagonal block, one lane per row
      for (int j = 0; j < w; ++j) {
        double d = diag[j][j];
        if (!(d > 0.0)) {
          if (tid == 0) bad = 1;
          d = 1.0;
        }
        const double piv = sqrt(d);
        __syncwarp();
        if (tid == j) diag[j][j] = piv;
        if (tid > j && tid < w) diag[tid][j] /= piv;
        __syncwarp();
        if (tid > j && tid < w)
          for (int c = j + 1; c <= tid; ++c) diag[tid][c] -= diag[tid][j] * diag[c][j];
        __syncwarp();
      }
    }
    __syncthreads();
    for (int e = tid; e < w * w; e += blockDim.x) {
      const int r = e / w, c = e % w;
      if (c <= r) {
        G[(int64_t)(p0 + r) * n + p0 + c] = diag[r][c];
        if (c < r) G[(int64_t)(p0 + c) * n + p0 + r] = diag[r][c];
      }
    }
    for (int r = tid; r < rows; r += blockDim.x) {   // L(i, panel) = A(i, panel) L_D^{-T}
      const int i = p0 + w + r;
      double* row = panel + r * (PW + 1);
      for (int j = 0; j < w; ++j) {
        double a = G[(int64_t)i * n + p0 + j];
        for (int c = 0; c < j; ++c) a -= row[c] * diag[j][c];
        row[j] = a / diag[j][j];
      }
      for (int j = 0; j < w; ++j) {
        G[(int64_t)i * n + p0 + j] = row[j];
        G[(int64_t)(p0 + j) * n + i] = row[j];
      }
    }
    __syncthreads();
    for (int64_t e = tid; e < (int64_t)rows * rows; e += blockDim.x) {
      const int r = (int)(e / rows), c = (int)(e % rows);
      if (c > r) continue;
      double* g = G + (int64_t)(p0 + w + r) * n + p0 + w + c;
      double a = *g;
      for (int j = 0; j < w; ++j) a -= panel[r * (PW + 1) + j] * panel[c * (PW + 1) + j];
      *g = a;
    }
  }
  __syncthreads();
  if (tid == 0 && bad) flag_breakdown(L.status, s);
}

// W = L^{-1} into the K_C buffer, column c per warp: w_q = b_q / l_qq, b_i -= l_iq w_q for i > q (row q of the
// upper part of G holds column q of L); b in shared memory
__global__ void __launch_bounds__(128) k_gram_linv(LevelDev L, int max_nc) {
  const int s = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const SubMeta m = L.meta[s];
  const int n = m.nc, c = blockIdx.x * 4 + warp;
  if (c >= n) return;
  extern __shared__ __align__(16) double bs[];
  double* b = bs + (int64_t)warp * max_nc;
  const double* G = L.Ginv + m.g_off;
  double* W = L.KC + m.g_off;
  for (int i = lane; i < n; i += 32) b[i] = i == c ? 1.0 : 0.0;
  __syncwarp();
  for (int q = c; q < n; ++q) {
    const double w = b[q] / G[(int64_t)q * n + q];
    const double* lq = G + (int64_t)q * n;
    for (int i = q + 1 + lane; i < n; i += 32) b[i] -= lq[i] * w;
    __syncwarp();
    if (lane == 0) b[q] = w;
    __syncwarp();
  }
  for (int i = lane; i < n; i += 32) W[(int64_t)i * n + c] = b[i];
}

// G^{-1} = W^T W: one thread per entry (a, b), b <= a
__global__ void __launch_bounds__(256) k_gram_inverse(LevelDev L) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int n = m.nc;
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (t >= (int64_t)n * n) return;
  const int a = (int)(t / n), b = (int)(t % n);
  if (b > a) return;
  const double* W = L.KC + m.g_off;
  double acc = 0.0;
  for (int q = a; q < n; ++q) acc += W[(int64_t)q * n + a] * W[(int64_t)q * n + b];
  double* G = L.Ginv + m.g_off;
  G[(int64_t)a * n + b] = acc;
  G[(int64_t)b * n + a] = acc;
}

// K_C = G^{-1} - R
__global__ void __launch_bounds__(256) k_gram_kc(LevelDev L) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int n = m.nc;
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (t >= (int64_t)n * n) return;
  const int a = (int)(t / n), b = (int)(t % n);
  L.KC[m.g_off + t] = L.Ginv[m.g_off + t] - (a == b ? L.rho[s] * L.c_rho[m.c_off + a] : 0.0);
}

// FP64 levels: Z = Y_G^T G^{-1}, written into the Psi buffer (rows: interface padded positions)
__global__ void k_psi_rhs(LevelDev L) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int nc = m.nc;
  if (nc == 0) return;
  const int rows = m.nGb * NB;
  const int64_t total = (int64_t)rows * nc;
  const double* Gi = L.Ginv + m.g_off;
  double* Z = (double*)L.psi + m.psi_off;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(t / nc), q = (int)(t % nc);
    const int jb = m.nIb + c / NB, cc = c % NB;
    double acc = 0.0;
    for (int p = 0; p < nc; ++p) {
      const double y = tile_ptr<double>(m, L.tiles, m.Bc + p / NB, jb)[(p % NB) * NB + cc];
      acc += y * Gi[p * nc + q];
    }
    Z[t] = acc;   // Z = Y^T G^{-1}
  }
}

// Psi_G = L_GG^{-T} Z, right-looking over the interface block rows from the bottom: at step t,
// block row i = Bc - 1 - t of every subdomain is final once X_i = D_i^T Z_i (D_i the stored inverse
// of the diagonal tile), and every block row j < i above it receives Z_j -= L(i, j)^T X_i.  The
// updates of a step are independent (one CTA per (j, subdomain, 16 columns)), so a step is one
// wide launch instead of a per-CTA chain of dependent tiles.
template <typename T>
__global__ void __launch_bounds__(256) k_psi_final(LevelDev L, int t) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int i = m.Bc - 1 - t, c0 = 16 * blockIdx.x, nc = m.nc;
  if (i < m.nIb || c0 >= nc) return;
  __shared__ T Ds[NB][NB + 1];
  __shared__ __align__(16) T Zs[NB][16];
  const T* dv = (const T*)L.dinv + m.dinv_off + (int64_t)i * NB2;
  T* Zi = (T*)L.psi + m.psi_off + (int64_t)(i - m.nIb) * NB * nc;
  for (int e = threadIdx.x; e < NB2; e += blockDim.x) Ds[e / NB][e % NB] = dv[e];
  for (int e = threadIdx.x; e < NB * 16; e += blockDim.x) {
    const int r = e / 16, q = e % 16;
    Zs[r][q] = c0 + q < nc ? Zi[(int64_t)r * nc + c0 + q] : (T)0;
  }
  __syncthreads();
  const int r = threadIdx.x >> 2, q4 = 4 * (threadIdx.x & 3);
  T x[4] = {};
#pragma unroll 8
  for (int mm = 0; mm < NB; ++mm) {   // X_i = D_i^T Z_i
    const T d = Ds[mm][r];
#pragma unroll
    for (int b = 0; b < 4; ++b) x[b] += d * Zs[mm][q4 + b];
  }
#pragma unroll
  for (int b = 0; b < 4; ++b)
    if (c0 + q4 + b < nc) Zi[(int64_t)r * nc + c0 + q4 + b] = x[b];
}

template <typename T>
__global__ void __launch_bounds__(256) k_psi_update(LevelDev L, int t) {
  const int s = blockIdx.y;
  const SubMeta m = L.meta[s];
  const int i = m.Bc - 1 - t, j = m.nIb + (int)blockIdx.x, c0 = 16 * blockIdx.z, nc = m.nc;
  if (j >= i || c0 >= nc) return;
  __shared__ T Ls[NB][NB + 1];
  __shared__ __align__(16) T Xs[NB][16];
  const T* lt = (const T*)L.tiles + m.tile_off + tile_index(i, j, m.Bc) * NB2;
  const T* Xi = (const T*)L.psi + m.psi_off + (int64_t)(i - m.nIb) * NB * nc;
  T* Zj = (T*)L.psi + m.psi_off + (int64_t)(j - m.nIb) * NB * nc;
  for (int e = threadIdx.x; e < NB2; e += blockDim.x) Ls[e / NB][e % NB] = lt[e];
  for (int e = threadIdx.x; e < NB * 16; e += blockDim.x) {
    const int r = e / 16, q = e % 16;
    Xs[r][q] = c0 + q < nc ? Xi[(int64_t)r * nc + c0 + q] : (T)0;
  }
  __syncthreads();
  const int c = threadIdx.x >> 2, q4 = 4 * (threadIdx.x & 3);
  T acc[4] = {};
#pragma unroll 8
  for (int r = 0; r < NB; ++r) {   // (L(i, j)^T X_i)[c] = sum_r L(i, j)[r][c] X_i[r]
    const T l = Ls[r][c];
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[b] += l * Xs[r][q4 + b];
  }
#pragma unroll
  for (int b = 0; b < 4; ++b)
    if (c0 + q4 + b < nc) Zj[(int64_t)c * nc + c0 + q4 + b] -= acc[b];
}

// v_G -= Y_G^T G^{-1} Y_G v_G  (the constraint part of Eq. sub_cor): t = Y_G v and the final
// update stream the constraint block rows of the factor (k_rows_matvec / k_cols_matvec below);
// mu = G^{-1} t takes one warp per row of G^{-1}.
__global__ void k_cc_mu(LevelDev L, const int32_t* __restrict__ crow_sub, int64_t total_rows,
                        const double* __restrict__ t, double* __restrict__ mu) {
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (g >= total_rows) return;
  t += (int64_t)blockIdx.y * total_rows;
  mu += (int64_t)blockIdx.y * total_rows;
  const int s = crow_sub[g];
  const SubMeta m = L.meta[s];
  const int p = (int)(g - m.c_off);
  const double* Gi = L.Ginv + m.g_off + (int64_t)p * m.nc;
  double acc = 0.0;
  for (int q = lane; q < m.nc; q += 32) acc += Gi[q] * t[m.c_off + q];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) mu[g] = acc;
}

// out_p = z_C[R_Ci p] - sum_q G_pq t_q: one warp per constraint row, its row of G read once for NR columns
template <int NR>
__global__ void k_coarse_coef(LevelDev L, const int32_t* __restrict__ crow_sub, int64_t total_rows,
                              const double* zC, const double* t, double* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (g >= total_rows) return;
  const int s = crow_sub[g];
  const SubMeta& m = L.meta[s];
  const int nc = m.nc;
  const int64_t c_off = m.c_off;
  const double* G = L.G + m.g_off + (g - c_off) * nc;
  double acc[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) acc[k] = 0.0;
  for (int q = lane; q < nc; q += 32) {
    const double a = G[q];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] += a * t[(int64_t)k * total_rows + c_off + q];
  }
  lane_sums<NR>(acc, lane);
  if (lane_sum_writer<NR>(lane)) {
    const int k = lane_sum_index<NR>(lane);
    out[(int64_t)k * total_rows + g] = zC[(int64_t)k * L.n_coarse + L.sub_coarse[g]] - acc[0];
  }
}

// identity tiles of the inverse rows
__global__ void k_unit_rows(LevelDev L) {
  const SubMeta m = L.meta[blockIdx.y];
  const int r = blockIdx.x;
  if (r >= m.nV) return;
  float* t = (float*)L.tiles + m.tile_off + tile_of(m, m.R + r, m.nIb + r) * NB2;
  if (threadIdx.x < NB) t[threadIdx.x * NB + threadIdx.x] = 1.f;
}

// ---- products with Y_G and Psi_G^T, both held as ncb x nGb tiles of NB x NB per subdomain ----
// MODE 0: M = Y_G, the constraint block rows of the factor (the forward sweep left S L^{-1} r in
// the vector, so its entries are multiplied by the pivot signs S first); MODE 1: M = Psi_G^T
// (psiT).  Row p of M belongs to coarse DOF p of the subdomain, column c to interface position c.
template <typename T>
struct Pair;
template <>
struct Pair<float> {
  using type = float2;
};
template <>
struct Pair<double> {
  using type = double2;
};

template <typename T, int MODE>
__device__ __forceinline__ const T* m_tile(const LevelDev& L, const SubMeta& m, int rb, int j) {
  if (MODE == 0) return tile_ptr<T>(m, L.tiles, m.Bc + rb, m.nIb + j);
  return (const T*)L.psiT + m.psiT_off + ((int64_t)rb * m.nGb + j) * NB2;
}

// Row products over four tile columns: block (z, rb, s) adds the columns 4z .. 4z+3 of the
// coarse rows rb NB .. rb NB + 63 of subdomain s for NR right-hand sides (column q at
// vec + q n_vec) and writes part[(q sum_nc + c_off + p) zmax + z] (zero where the subdomain has
// no such tile columns).  Warp w takes the rows w, w+8, .., lane l the columns 2l, 2l+1 of every
// tile, so each tile row is one coalesced 256-byte read; rows past nc are not read.
template <typename T, int NR, int MODE>
__global__ void __launch_bounds__(256) k_rows_matvec(LevelDev L, const T* vec, double* __restrict__ part,
                                                     int zmax, int64_t sum_nc) {
  pdl_wait();
  pdl_trigger();
  using V2 = typename Pair<T>::type;
  const int z = blockIdx.x, rb = blockIdx.y, s = blockIdx.z;
  const SubMeta m = L.meta[s];
  if (rb >= m.ncb) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = 4 * z, j1 = min(m.nGb, j0 + 4);
  __shared__ __align__(16) T xs[NR][4][NB];
  const T* v = vec + m.vec_off + (int64_t)m.nIb * NB;
  const T* sg = (const T*)L.sgn + m.vec_off + (int64_t)m.nIb * NB;
  for (int e = threadIdx.x; e < NR * 4 * NB; e += blockDim.x) {
    const int q = e / (4 * NB), jj = (e / NB) % 4, c = e % NB;
    const int j = j0 + jj;
    T x = (T)0;
    if (j < j1) {
      x = v[(int64_t)q * L.n_vec + (int64_t)j * NB + c];
      if (MODE == 0 && L.indefinite) x *= sg[(int64_t)j * NB + c];
    }
    xs[q][jj][c] = x;
  }
  __syncthreads();
  const int rows = min(NB, m.nc - rb * NB);
  T acc[NR][8];
#pragma unroll
  for (int q = 0; q < NR; ++q)
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[q][r] = (T)0;
  for (int j = j0; j < j1; ++j) {
    const T* t = m_tile<T, MODE>(L, m, rb, j) + 2 * lane;
    V2 xv[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) xv[q] = *(const V2*)&xs[q][j - j0][2 * lane];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int row = warp + 8 * r;
      if (row < rows) {
        const V2 a = __ldg((const V2*)(t + row * NB));
#pragma unroll
        for (int q = 0; q < NR; ++q) acc[q][r] += a.x * xv[q].x + a.y * xv[q].y;
      }
    }
  }
  constexpr int NV = 8 * NR, NC = NV < 32 ? 1 : NV / 32;
  lane_sums<NV>(&acc[0][0], lane);
  if (lane_sum_writer<NV>(lane))
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int f = lane_sum_index<NV>(lane) + k, q = f / 8, row = warp + 8 * (f % 8);
      if (row < rows) part[((int64_t)q * sum_nc + m.c_off + rb * NB + row) * zmax + z] = (double)(&acc[0][0])[k];
    }
}

// out[q sum_nc + g] = sum_{z < zmax} part[(q sum_nc + g) zmax + z], in order
__global__ void k_sum_parts(const double* __restrict__ part, int zmax, int64_t total, double* __restrict__ out) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= total) return;
  const int64_t o = (int64_t)blockIdx.y * total + g;
  double t = 0.0;
  for (int z = 0; z < zmax; ++z) t += part[o * zmax + z];
  out[o] = t;
}

// Column products: block (j, s) makes v[nIb NB + j NB + c] += sign sum_p M[p][j NB + c] zsub_p
// for the 64 positions of interface tile column j and NR right-hand sides (zsub column q at
// zsub + q sum_nc, per-subdomain coarse vectors); the eight warps' partial sums are added in a
// fixed order.
template <typename T, int NR, int MODE>
__global__ void __launch_bounds__(256) k_cols_matvec(LevelDev L, T* __restrict__ vec, const double* zsub,
                                                     int64_t sum_nc, T sign) {
  pdl_wait();
  pdl_trigger();
  using V2 = typename Pair<T>::type;
  const int j = blockIdx.x, s = blockIdx.y;
  const SubMeta m = L.meta[s];
  if (j >= m.nGb || m.nc == 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ T zs[NR][NB];
  __shared__ T red[8][NR][NB];
  T acc[NR][2];
#pragma unroll
  for (int q = 0; q < NR; ++q) acc[q][0] = acc[q][1] = (T)0;
  for (int rb = 0; rb < m.ncb; ++rb) {
    const int rows = min(NB, m.nc - rb * NB);
    __syncthreads();
    for (int e = threadIdx.x; e < NR * NB; e += blockDim.x) {
      const int q = e / NB, p = e % NB;
      zs[q][p] = p < rows ? (T)zsub[(int64_t)q * sum_nc + m.c_off + rb * NB + p] : (T)0;
    }
    __syncthreads();
    const T* t = m_tile<T, MODE>(L, m, rb, j) + 2 * lane;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int row = warp + 8 * r;
      if (row < rows) {
        const V2 a = __ldg((const V2*)(t + row * NB));
#pragma unroll
        for (int q = 0; q < NR; ++q) {
          const T zq = zs[q][row];
          acc[q][0] += a.x * zq;
          acc[q][1] += a.y * zq;
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    red[warp][q][2 * lane] = acc[q][0];
    red[warp][q][2 * lane + 1] = acc[q][1];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NR * NB; e += blockDim.x) {
    const int q = e / NB, c = e % NB;
    T a = (T)0;
#pragma unroll
    for (int w = 0; w < 8; ++w) a += red[w][q][c];
    T* v = vec + (int64_t)q * L.n_vec + m.vec_off + (int64_t)m.nIb * NB + (int64_t)j * NB + c;
    *v = *v + sign * a;
  }
}

// psiT tile (rb, j)[p][c] = Psi_G[(j NB + c) nc + rb NB + p], zero outside nG x nc (set-up)
template <typename T>
__global__ void k_psi_transpose(LevelDev L) {
  const int j = blockIdx.x, rb = blockIdx.y, s = blockIdx.z;
  const SubMeta m = L.meta[s];
  if (j >= m.nGb || rb >= m.ncb) return;
  const T* P = (const T*)L.psi + m.psi_off;
  T* out = (T*)L.psiT + m.psiT_off + ((int64_t)rb * m.nGb + j) * NB2;
  __shared__ T ts[NB][NB + 1];
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    const int c = e / NB, p = e % NB;
    const int gc = j * NB + c, gp = rb * NB + p;
    ts[c][p] = (gc < m.nG && gp < m.nc) ? P[(int64_t)gc * m.nc + gp] : (T)0;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) out[e] = ts[e % NB][e / NB];
}

// ---- explicit inverse of the coarsest factor (FP32 copy, mixed form) ------------------------
// W = A_C^{-1} = L^{-T} S L^{-1} of the single-subdomain coarsest level, whose block rows are all
// "interior" (identity padding past the last DOF).  CTA c substitutes the identity columns
// c CW .. c CW + CW - 1 through the tiled factor: forward y_i = D_i (e_i - sum_{j<i} L_ij y_j),
// t = S y, backward x_i = D_i^T (t_i - sum_{j>i} L_ji^T x_j), with D_i the stored inverses of the
// diagonal tiles (the same steps as the sweeps, in the same precision).  Column q of the result is
// kept at W + (c CW + q) npad, so W is stored column after column.  The forward solution is zero above the
// column's own block b0, and A_C^{-1} is symmetric, so only the blocks i >= b0 are computed (a third of
// the products) and k_coarse_mirror fills in the rest.  Each product of a tile with a 64 x CW block runs from
// shared memory, the tile k-major, one row x 4 columns per thread; the next tile is in registers meanwhile.
// Bound by the chain of tiles of the first column block (nb^2 of them, about 1 us each), hence narrow blocks
// of columns: 3,345 coarse DOFs take 5.6 ms (14.6 ms with 53 blocks of 64 columns through every block row).
constexpr int CW = 16;

__global__ void __launch_bounds__(256) k_coarse_inverse(LevelDev L, float* __restrict__ W) {
  const SubMeta m = L.meta[0];
  const int nb = m.Bc;
  const int64_t npad = (int64_t)nb * NB;
  const int c0 = blockIdx.x * CW;
  if (c0 >= npad) return;
  const int b0 = c0 / NB;
  __shared__ __align__(16) float As[NB][NB + 4];   // tile, k-major: As[k][r]
  __shared__ __align__(16) float Bs[NB][CW + 4];   // 64 x CW block: Bs[k][c]
  const int tid = threadIdx.x;
  const int cg = tid % (CW / 4), r = tid / (CW / 4);   // columns 4 cg .. +3 of row r
  float* Wc = W + (int64_t)c0 * npad;              // this CTA's columns, each of npad entries
  const float* tiles = (const float*)L.tiles + m.tile_off;
  const float* dinv = (const float*)L.dinv + m.dinv_off;
  const float* sgn = (const float*)L.sgn + m.vec_off;
  float4 ta[4], tb;   // the next tile and block
  auto fetch_tile = [&](const float* t) {
#pragma unroll
    for (int u = 0; u < 4; ++u) ta[u] = __ldg((const float4*)t + tid + 256 * u);
  };
  auto fetch_block = [&](int blk) {   // 16 columns x 64 rows: column tid / 16, rows 4 (tid % 16) ..
    tb = *(const float4*)(Wc + (int64_t)(tid >> 4) * npad + (int64_t)blk * NB + 4 * (tid & 15));
  };
  auto put_tile = [&](bool transpose) {   // As[k][r] = t[r][k] (transpose) or t[k][r]
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = tid + 256 * u, a = q >> 4, b = 4 * (q & 15);
      if (transpose) {
        As[b][a] = ta[u].x;
        As[b + 1][a] = ta[u].y;
        As[b + 2][a] = ta[u].z;
        As[b + 3][a] = ta[u].w;
      } else {
        *(float4*)&As[a][b] = ta[u];
      }
    }
  };
  auto put_block = [&]() {
    const int c = tid >> 4, k = 4 * (tid & 15);
    Bs[k][c] = tb.x;
    Bs[k + 1][c] = tb.y;
    Bs[k + 2][c] = tb.z;
    Bs[k + 3][c] = tb.w;
  };
  auto mma = [&](float (&acc)[4]) {
#pragma unroll 16
    for (int k = 0; k < NB; ++k) {
      const float a = As[k][r];
      const float4 b = *(const float4*)&Bs[k][4 * cg];
      acc[0] += a * b.x;
      acc[1] += a * b.y;
      acc[2] += a * b.z;
      acc[3] += a * b.w;
    }
  };
  auto store_block = [&](int blk, const float (&v)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) Wc[(int64_t)(4 * cg + q) * npad + (int64_t)blk * NB + r] = v[q];
  };
  // forward: y_i = D_i (e_i - sum_{b0 <= j < i} L_ij y_j)
  for (int i = b0; i < nb; ++i) {
    float acc[4] = {};
    const float* row = tiles + (int64_t)i * (i + 1) / 2 * NB2;
    __syncthreads();   // the blocks stored so far are visible to the whole CTA
    if (b0 < i) {
      fetch_tile(row + (int64_t)b0 * NB2);
      fetch_block(b0);
    }
    for (int j = b0; j < i; ++j) {
      put_tile(true);
      put_block();
      __syncthreads();
      if (j + 1 < i) {
        fetch_tile(row + (int64_t)(j + 1) * NB2);
        fetch_block(j + 1);
      } else {
        fetch_tile(dinv + (int64_t)i * NB2);
      }
      mma(acc);
      __syncthreads();
    }
    if (b0 == i) fetch_tile(dinv + (int64_t)i * NB2);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      Bs[r][4 * cg + q] = ((int64_t)i * NB + r == c0 + 4 * cg + q ? 1.f : 0.f) - acc[q];
    put_tile(true);
    __syncthreads();
    float y[4] = {};
    mma(y);
    store_block(i, y);
  }
  __syncthreads();
  // t = S y (pivot signs of the signed factor; all +1 on SPD levels)
  for (int e = tid; e < NB * CW; e += 256) {
    const int c = e / NB;
    for (int64_t row = (int64_t)b0 * NB + e % NB; row < npad; row += NB) Wc[(int64_t)c * npad + row] *= sgn[row];
  }
  // backward: x_i = D_i^T (t_i - sum_{j>i} L_ji^T x_j), i >= b0
  for (int i = nb - 1; i >= b0; --i) {
    float acc[4] = {};
    __syncthreads();
    if (i + 1 < nb) {
      fetch_tile(tiles + ((int64_t)(i + 1) * (i + 2) / 2 + i) * NB2);
      fetch_block(i + 1);
    }
    for (int j = i + 1; j < nb; ++j) {
      put_tile(false);
      put_block();
      __syncthreads();
      if (j + 1 < nb) {
        fetch_tile(tiles + ((int64_t)(j + 1) * (j + 2) / 2 + i) * NB2);
        fetch_block(j + 1);
      } else {
        fetch_tile(dinv + (int64_t)i * NB2);
        fetch_block(i);
      }
      mma(acc);
      __syncthreads();
    }
    if (i + 1 == nb) {
      fetch_tile(dinv + (int64_t)i * NB2);
      fetch_block(i);
    }
    put_tile(false);
    put_block();
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) Bs[r][4 * cg + q] -= acc[q];   // this thread's own entries
    __syncthreads();
    float x[4] = {};
    mma(x);
    store_block(i, x);
  }
}

// the blocks above every column's own: W(i, j) = W(j, i), one 64 x 64 block (j > i) per CTA
__global__ void __launch_bounds__(256) k_coarse_mirror(float* __restrict__ W, int64_t npad) {
  const int i = blockIdx.x, j = blockIdx.y;
  if (i >= j) return;
  __shared__ float t[NB][NB + 1];
  for (int e = threadIdx.x; e < NB2; e += 256)   // columns of block i, rows of block j
    t[e / NB][e % NB] = W[((int64_t)i * NB + e / NB) * npad + (int64_t)j * NB + e % NB];
  __syncthreads();
  for (int e = threadIdx.x; e < NB2; e += 256)
    W[((int64_t)j * NB + e / NB) * npad + (int64_t)i * NB + e % NB] = t[e % NB][e / NB];
}

// z = W x for nr columns (x: columns of n_vec, padded local positions 0 .. npad-1; z: level DOFs); one warp
// per output row, lanes along the row (coalesced), FP32 sums in a fixed order.
template <int NR>
__global__ void k_coarse_apply(const float* __restrict__ W, int64_t npad, const float* x,
                               double* __restrict__ z, const int32_t* __restrict__ loc2glob, int64_t n_vec,
                               int64_t n_dof) {
  pdl_wait();
  pdl_trigger();
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= npad) return;
  const int64_t c0 = (int64_t)blockIdx.y * NR;
  const float* w = W + row * npad;
  float acc[NR];
#pragma unroll
  for (int q = 0; q < NR; ++q) acc[q] = 0.f;
  for (int64_t c = 4 * lane; c < npad; c += 128) {
    const float4 a = *(const float4*)(w + c);
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const float4 b = *(const float4*)(x + (c0 + q) * n_vec + c);
      acc[q] += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
    }
  }
  lane_sums<NR>(acc, lane);
  const int32_t g = loc2glob[row];
  if (lane_sum_writer<NR>(lane) && g >= 0) z[(c0 + lane_sum_index<NR>(lane)) * n_dof + g] = (double)acc[0];
}

}  // namespace

void launch_coarse_inverse(const LevelDev& L, int64_t npad, float* W, cudaStream_t st) {
  if (npad <= 0) return;
  note_launch();
  k_coarse_inverse<<<(unsigned)((npad + CW - 1) / CW), 256, 0, st>>>(L, W);
  const unsigned nb = (unsigned)(npad / NB);
  if (nb > 1) {
    note_launch();
    k_coarse_mirror<<<dim3(nb, nb), 256, 0, st>>>(W, npad);
  }
}

void launch_coarse_apply(const float* W, int64_t npad, const float* x, double* z, const int32_t* loc2glob,
                         int64_t n_vec, int64_t n_dof, int nr, cudaStream_t st) {
  if (npad <= 0 || nr <= 0) return;
  const unsigned gx = (unsigned)((npad + 7) / 8);
  for (int r0 = 0; r0 < nr;) {
    const int left = nr - r0;
    const int g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    const int ng = left / g;
    const float* xs = x + (int64_t)r0 * n_vec;
    double* zs = z + (int64_t)r0 * n_dof;
    note_launch();
    if (g == 8)
      launch_pdl(k_coarse_apply<8>, dim3(gx, ng), 256, 0, st, W, npad, xs, zs, loc2glob, n_vec, n_dof);
    else if (g == 4)
      launch_pdl(k_coarse_apply<4>, dim3(gx, ng), 256, 0, st, W, npad, xs, zs, loc2glob, n_vec, n_dof);
    else if (g == 2)
      launch_pdl(k_coarse_apply<2>, dim3(gx, ng), 256, 0, st, W, npad, xs, zs, loc2glob, n_vec, n_dof);
    else
      launch_pdl(k_coarse_apply<1>, dim3(gx, ng), 256, 0, st, W, npad, xs, zs, loc2glob, n_vec, n_dof);
    r0 += ng * g;
  }
}

template <typename T>
void launch_potrf_step(const LevelDev& L, int k, int max_R, int max_tiles, int jmax, cudaStream_t st, int skip_diag,
                       int fuse_next, int rlim, int xinv, int k0) {
  const unsigned ns = (unsigned)L.n_sub;
  const size_t sm = 2 * NB * LDS * sizeof(T);
  const size_t sm_diag = 2 * NB * (NB + 1) * sizeof(T);
  static bool attr = false;   // opt in to more than 48 KB of dynamic shared memory once
  if (!attr) {
    cudaFuncSetAttribute(k_potrf_diag<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_diag);
    cudaFuncSetAttribute(k_trsm_panel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    cudaFuncSetAttribute(k_trsm_panel16<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    cudaFuncSetAttribute(k_syrk_update<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    attr = true;
  }
  static_assert(2 * NB * LDS >= 2 * NB * (NB + 1), "the update's shared memory holds the diagonal factorisation");
  if (!skip_diag) { note_launch(); k_potrf_diag<T><<<ns, 256, sm_diag, st>>>(L, k); }
  const int panel = (rlim > 0 && rlim < max_R ? rlim : max_R) - k - 1;
  if (panel > 0) {
    note_launch();
    if (sizeof(T) == 8 && (int64_t)panel * ns < 152)
      k_trsm_panel16<T><<<dim3((unsigned)panel * 4, ns), 256, sm, st>>>(L, k, rlim);
    else
      k_trsm_panel<T><<<dim3((unsigned)panel, ns), 256, sm, st>>>(L, k, rlim);
  }
  static_assert(sizeof(float) * NB * (NB + 1 + 32) <= 2 * NB * LDS * sizeof(float), "block inverse shared memory");
  const int xq = xinv && sizeof(T) == 4 ? k - k0 : 0;   // block row of the diagonal block's inverse
  if (max_tiles > 0 || xq > 0) {
    note_launch();
    k_syrk_update<T><<<dim3((unsigned)(max_tiles + 4 * xq), ns), 256, sm, st>>>(L, k, jmax, fuse_next, rlim, max_tiles,
                                                                               xinv, k0);
  }
}

void launch_gram_f32(const LevelDev& L, int max_nc, cudaStream_t st) {
  const unsigned nb = (unsigned)((max_nc + GB - 1) / GB);
  note_launch();
  k_gram_f32<<<dim3(nb * (nb + 1) / 2, (unsigned)L.n_sub), 256, 0, st>>>(L);
}

void launch_psi_rhs_f32(const LevelDev& L, int max_nGb, int max_nc, cudaStream_t st) {
  note_launch();
  k_psi_rhs_f32<<<dim3((unsigned)max_nGb * (NB / GB), (unsigned)((max_nc + GB - 1) / GB), (unsigned)L.n_sub), 256, 0,
                  st>>>(L);
}

void launch_gram_chol(const LevelDev& L, int precision_fp32, int max_nc, cudaStream_t st) {
  const unsigned ns = (unsigned)L.n_sub;
  if (precision_fp32) {
    launch_gram_f32(L, max_nc, st);
  } else {
    note_launch();
    const unsigned gx = (unsigned)(((int64_t)max_nc * max_nc + 7) / 8);
    k_gram<<<dim3(gx, ns), 256, 0, st>>>(L);
  }
  // one pass per subdomain where n_c is small (its four launches would be longer) or G indefinite, and where the
  // panel of 16 columns does not fit
  if (L.indefinite || max_nc <= 96 || max_nc > kPanelMaxNc) {
    note_launch();
    k_small_chol_inv<<<ns, 256, 0, st>>>(L);
    return;
  }
  const size_t sm = sizeof(double) * 17 * (size_t)max_nc, smw = sizeof(double) * 4 * (size_t)max_nc;
  // the limits of the largest n_c at every set-up: the attribute is one per device, other threads launch with it, and
  // one set to this level's need could fall below theirs
  cudaFuncSetAttribute(k_gram_potrf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(double) * 17 * kPanelMaxNc));
  cudaFuncSetAttribute(k_gram_linv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(double) * 4 * kPanelMaxNc));
  const unsigned ge = (unsigned)(((int64_t)max_nc * max_nc + 255) / 256);
  { note_launch(); k_gram_potrf<<<ns, 1024, sm, st>>>(L); }
  { note_launch(); k_gram_linv<<<dim3((unsigned)((max_nc + 3) / 4), ns), 128, smw, st>>>(L, max_nc); }
  { note_launch(); k_gram_inverse<<<dim3(ge, ns), 256, 0, st>>>(L); }
  { note_launch(); k_gram_kc<<<dim3(ge, ns), 256, 0, st>>>(L); }
}

template <typename T>
void launch_psi(const LevelDev& L, int max_nGb, int max_nc, cudaStream_t st) {
  const unsigned ns = (unsigned)L.n_sub;
  if (max_nc <= 0 || max_nGb <= 0) return;
  if constexpr (sizeof(T) == 4) {
    launch_psi_rhs_f32(L, max_nGb, max_nc, st);
  } else {
    note_launch();
    k_psi_rhs<<<dim3(16, ns), 256, 0, st>>>(L);
  }
  const unsigned chunks = (unsigned)((max_nc + 15) / 16);
  for (int t = 0; t < max_nGb; ++t) {   // block row Bc - 1 - t of every subdomain, bottom up
    { note_launch(); k_psi_final<T><<<dim3(chunks, ns), 256, 0, st>>>(L, t); }
    if (max_nGb - 1 - t > 0)
      { note_launch(); k_psi_update<T><<<dim3((unsigned)(max_nGb - 1 - t), ns, chunks), 256, 0, st>>>(L, t); }
  }
}

// The solve-phase launches below take nr right-hand sides: local vectors of n_vec, per-subdomain
// coarse vectors of sum nc entries per column.
template <typename T, int MODE>
void rows_matvec(const LevelDev& L, const T* vec, double* part, int64_t sum_nc, int max_nGb, int max_ncb,
                 cudaStream_t st, int nr) {
  const int zmax = rows_zmax(max_nGb);
  const dim3 grid((unsigned)zmax, (unsigned)max_ncb, (unsigned)L.n_sub);
  constexpr int kMaxNR = sizeof(T) == 4 ? 8 : 4;
  for (int r0 = 0; r0 < nr;) {
    const int left = nr - r0;
    const int g = left >= kMaxNR ? kMaxNR : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    const T* v = vec + (int64_t)r0 * L.n_vec;
    double* pt = part + (int64_t)r0 * sum_nc * zmax;
    note_launch();
    if (g == 8)
      k_rows_matvec<T, (sizeof(T) == 4 ? 8 : 4), MODE><<<grid, 256, 0, st>>>(L, v, pt, zmax, sum_nc);
    else if (g == 4)
      k_rows_matvec<T, 4, MODE><<<grid, 256, 0, st>>>(L, v, pt, zmax, sum_nc);
    else if (g == 2)
      k_rows_matvec<T, 2, MODE><<<grid, 256, 0, st>>>(L, v, pt, zmax, sum_nc);
    else
      k_rows_matvec<T, 1, MODE><<<grid, 256, 0, st>>>(L, v, pt, zmax, sum_nc);
    r0 += g;
  }
}

template <typename T, int MODE>
void cols_matvec(const LevelDev& L, T* vec, const double* zsub, int64_t sum_nc, int max_nGb, T sign, cudaStream_t st,
                 int nr) {
  const dim3 grid((unsigned)max_nGb, (unsigned)L.n_sub);
  constexpr int kMaxNR = sizeof(T) == 4 ? 8 : 4;
  for (int r0 = 0; r0 < nr;) {
    const int left = nr - r0;
    const int g = left >= kMaxNR ? kMaxNR : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    T* v = vec + (int64_t)r0 * L.n_vec;
    const double* zz = zsub + (int64_t)r0 * sum_nc;
    note_launch();
    if (g == 8)
      k_cols_matvec<T, (sizeof(T) == 4 ? 8 : 4), MODE><<<grid, 256, 0, st>>>(L, v, zz, sum_nc, sign);
    else if (g == 4)
      k_cols_matvec<T, 4, MODE><<<grid, 256, 0, st>>>(L, v, zz, sum_nc, sign);
    else if (g == 2)
      k_cols_matvec<T, 2, MODE><<<grid, 256, 0, st>>>(L, v, zz, sum_nc, sign);
    else
      k_cols_matvec<T, 1, MODE><<<grid, 256, 0, st>>>(L, v, zz, sum_nc, sign);
    r0 += g;
  }
}

template <typename T>
void launch_constraint_corr(const LevelDev& L, T* vec, const int32_t* crow_sub, int64_t total_rows, double* t,
                            double* mu, double* part, int max_nGb, int max_ncb, cudaStream_t st, int nr) {
  if (total_rows <= 0 || max_nGb <= 0) return;
  rows_matvec<T, 0>(L, vec, part, total_rows, max_nGb, max_ncb, st, nr);
  const int zmax = rows_zmax(max_nGb);
  note_launch();
  k_sum_parts<<<dim3((unsigned)((total_rows + 255) / 256), (unsigned)nr), 256, 0, st>>>(part, zmax, total_rows, t);
  const unsigned g = (unsigned)((total_rows + 7) / 8);
  { note_launch(); k_cc_mu<<<dim3(g, nr), 256, 0, st>>>(L, crow_sub, total_rows, t, mu); }
  cols_matvec<T, 0>(L, vec, mu, total_rows, max_nGb, (T)-1, st, nr);
}

template <typename T>
void launch_psi_t_apply(const LevelDev& L, const T* vec, double* part, int64_t sum_nc, int max_nGb, int max_ncb,
                        cudaStream_t st, int nr) {
  if (sum_nc <= 0 || max_nGb <= 0) return;
  rows_matvec<T, 1>(L, vec, part, sum_nc, max_nGb, max_ncb, st, nr);
}

template <typename T>
void launch_psi_apply_add(const LevelDev& L, const double* zc_sub, int64_t sum_nc, T* vec, int max_nGb, int max_ncb,
                          cudaStream_t st, int nr) {
  if (sum_nc <= 0 || max_nGb <= 0) return;
  (void)max_ncb;
  cols_matvec<T, 1>(L, vec, zc_sub, sum_nc, max_nGb, (T)1, st, nr);
}

void launch_coarse_coef(const LevelDev& L, const int32_t* crow_sub, int64_t sum_nc, const double* zC, const double* t,
                        double* out, cudaStream_t st, int nr) {
  if (sum_nc <= 0) return;
  const unsigned gx = (unsigned)((sum_nc + 7) / 8);
  for (int r0 = 0; r0 < nr;) {
    const int left = nr - r0, g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    const double *z = zC + (int64_t)r0 * L.n_coarse, *tt = t + (int64_t)r0 * sum_nc;
    double* o = out + (int64_t)r0 * sum_nc;
    note_launch();
    if (g == 8)
      launch_pdl(k_coarse_coef<8>, gx, 256, 0, st, L, crow_sub, sum_nc, z, tt, o);
    else if (g == 4)
      launch_pdl(k_coarse_coef<4>, gx, 256, 0, st, L, crow_sub, sum_nc, z, tt, o);
    else if (g == 2)
      launch_pdl(k_coarse_coef<2>, gx, 256, 0, st, L, crow_sub, sum_nc, z, tt, o);
    else
      launch_pdl(k_coarse_coef<1>, gx, 256, 0, st, L, crow_sub, sum_nc, z, tt, o);
    r0 += g;
  }
}

void launch_unit_rows(const LevelDev& L, int max_nGb, cudaStream_t st) {
  if (max_nGb <= 0 || L.n_sub <= 0) return;
  note_launch();
  k_unit_rows<<<dim3((unsigned)max_nGb, (unsigned)L.n_sub), NB, 0, st>>>(L);
}

template <typename T>
void launch_psi_transpose(const LevelDev& L, int max_nGb, int max_ncb, cudaStream_t st) {
  if (max_nGb <= 0 || max_ncb <= 0) return;
  note_launch();
  k_psi_transpose<T><<<dim3((unsigned)max_nGb, (unsigned)max_ncb, (unsigned)L.n_sub), 256, 0, st>>>(L);
}

#define INST(T)                                                                                 \
  template void launch_potrf_step<T>(const LevelDev&, int, int, int, int, cudaStream_t, int, int, int, int, int); \
  template void launch_psi<T>(const LevelDev&, int, int, cudaStream_t);                          \
  template void launch_constraint_corr<T>(const LevelDev&, T*, const int32_t*, int64_t, double*, double*, double*, \
                                         int, int, cudaStream_t, int);                                     \
  template void launch_psi_t_apply<T>(const LevelDev&, const T*, double*, int64_t, int, int, cudaStream_t, int);   \
  template void launch_psi_apply_add<T>(const LevelDev&, const double*, int64_t, T*, int, int, cudaStream_t, int); \
  template void launch_psi_transpose<T>(const LevelDev&, int, int, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace bddc
