// Vector kernels of the solve phase: interface gather/scatter with weights (r_i = E_i^T r,
// z = sum E_i z_i, Sec. 2), FP64 sparse products with K_i, coarse gather/scatter with R_Ci,
// deterministic FP64 reductions and the device-side PCG recurrences, and the element
// contraction of the adjoint gradient.
//
// All sums run in a fixed order (ascending subdomain for the interface / coarse sums, a
// fixed grid and tree for the dot products), so results are bit-reproducible.
#include "internal.h"
#include "pdl.cuh"
#include "reduce.cuh"

namespace bddc {

namespace {

// Several right-hand sides: blockIdx.y selects the column; every vector of a block stores its
// columns one after another with its own length as the stride (local vectors n_vec, interface
// vectors n_iface, level vectors n_dof, coarse vectors n_coarse, per-subdomain coarse vectors sum nc).
template <typename T>
__global__ void k_gather_iface(LevelDev L, const double* x, int weighted, T* __restrict__ loc) {
  pdl_wait();
  pdl_trigger();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.n_vec) return;
  x += (int64_t)blockIdx.y * L.n_iface;
  loc += (int64_t)blockIdx.y * L.n_vec;
  const int32_t g = L.loc2iface[p];
  double v = 0.0;
  if (g >= 0) v = weighted ? L.w[p] * x[g] : x[g];
  loc[p] = (T)v;
}

// Sum v0 (and v1) over the block, then over the blocks of column blockIdx.y: every block writes its partial
// sums, the last one to finish adds them in block order.  True in that block (all threads), totals in s0, s1.
__device__ bool sum_over_grid(double v0, double v1, bool two, double* __restrict__ partial, int* cnt, double& s0,
                              double& s1) {
  __shared__ double red[2][8];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto block_sum = [&](double a, double b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      if (two) b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
      red[0][warp] = a;
      red[1][warp] = b;
    }
    __syncthreads();
    s0 = s1 = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      s0 += red[0][w];
      if (two) s1 += red[1][w];
    }
    __syncthreads();
  };
  block_sum(v0, v1);
  const int nb = gridDim.x;
  double* p0 = partial + (int64_t)blockIdx.y * 2 * nb;
  if (threadIdx.x == 0) {
    p0[blockIdx.x] = s0;
    if (two) p0[nb + blockIdx.x] = s1;
    __threadfence();
    last = atomicAdd(cnt + blockIdx.y, 1) == nb - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    a += __ldcg(p0 + i);
    if (two) b += __ldcg(p0 + nb + i);
  }
  block_sum(a, b);
  if (threadIdx.x == 0) cnt[blockIdx.y] = 0;
  return true;
}

// scal layout (see capi.cpp): 0 rz, 1 pq, 2 alpha, 3 beta, 4 rz_new, 5 rr, 6 gg, 7 iteration, 8 frozen.  The scalar step of
// the recurrence that follows the sums (one thread); frozen columns keep alpha = beta = 0.
__device__ void pcg_step(const FusedDot& dot, double s0, double s1) {
  double* S = dot.scal + 16 * blockIdx.y;
  const bool frozen = S[8] != 0.0;
  if (dot.mode == 1) {
    S[1] = s0;
    S[2] = !frozen && s0 != 0.0 ? S[0] / s0 : 0.0;
  } else {
    S[4] = s0;
    const double num = dot.flexible ? -S[2] * s1 : s0;   // z . (r - r_old) = -alpha z . q
    S[3] = !frozen && S[0] != 0.0 ? num / S[0] : 0.0;
    if (!frozen) S[0] = s0;
  }
}

// the sums of a fused scatter over its outputs y[g] and the scalar step
__device__ void fused_dot(const FusedDot& dot, int64_t g, int64_t n, double y) {
  double v0 = 0.0, v1 = 0.0, s0, s1;
  if (g < n) {
    const int64_t o = (int64_t)blockIdx.y * n + g;
    v0 = dot.a[o] * y;
    if (dot.mode == 2) v1 = dot.b[o] * y;
  }
  if (sum_over_grid(v0, v1, dot.mode == 2, dot.partial, dot.cnt, s0, s1) && threadIdx.x == 0) pcg_step(dot, s0, s1);
}

// sum of term(p) over the occurrences of interface DOF g, ascending subdomain: one 16-byte load instead of
// the list's bounds and entries, so that the terms' loads are one step away (most DOFs have two occurrences)
template <typename F>
__device__ __forceinline__ double sum_occurrences(const LevelDev& L, int64_t g, F&& term) {
  const int4 o = __ldg(L.iface_occ4 + g);
  const double a = o.x >= 0 ? term((int64_t)o.x) : 0.0, b = o.y >= 0 ? term((int64_t)o.y) : 0.0;
  const double c = o.z >= 0 ? term((int64_t)o.z) : 0.0, d = o.w >= 0 ? term((int64_t)o.w) : 0.0;
  double s = a;
  if (o.y >= 0) s += b;
  if (o.z >= 0) s += c;
  if (o.w >= 0) s += d;
  if (o.w == -2)
    for (int64_t q = L.iface_ptr[g] + 3; q < L.iface_ptr[g + 1]; ++q) s += term(L.iface_occ[q]);
  return s;
}

template <typename T>
__global__ void __launch_bounds__(256) k_scatter_iface(LevelDev L, const T* loc, int weighted,
                                                       double* __restrict__ y, FusedDot dot) {
  pdl_wait();
  pdl_trigger();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double s = 0.0;
  if (g < L.n_iface) {
    loc += (int64_t)blockIdx.y * L.n_vec;
    s = sum_occurrences(L, g, [&](int64_t p) { return weighted ? L.w[p] * (double)loc[p] : (double)loc[p]; });
    y[(int64_t)blockIdx.y * L.n_iface + g] = s;
  }
  if (dot.mode) fused_dot(dot, g, L.n_iface, s);
}

// inner operator, before its FP32 product: blocks below nv gather loc = R_i x, the others take one
// constraint row per warp: t = rho c_rho (C_i R_i x); NR columns per pass over the index lists
template <int NR>
__global__ void __launch_bounds__(256) k_inner_gather(LevelDev L, const double* x, float* __restrict__ loc,
                                                      int nv, const int32_t* __restrict__ crow_sub, int64_t total_rows,
                                                      double* __restrict__ t) {
  pdl_wait();
  pdl_trigger();
  if ((int)blockIdx.x < nv) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= L.n_vec) return;
    const int32_t g = L.loc2iface[p];
#pragma unroll
    for (int k = 0; k < NR; ++k) loc[k * L.n_vec + p] = g >= 0 ? (float)x[k * L.n_iface + g] : 0.f;
    return;
  }
  const int64_t r = (int64_t)(blockIdx.x - nv) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= total_rows) return;
  const int s = crow_sub[r];
  const double rq = L.rho[s] * L.c_rho[r];
  const int32_t* l2i = L.loc2iface + L.meta[s].vec_off;
  double acc[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) acc[k] = 0.0;
  if (rq != 0.0)
    for (int64_t e = L.c_ptr[r] + lane; e < L.c_ptr[r + 1]; e += 32) {
      const double c = L.c_val[e];
      const int32_t g = l2i[L.c_pos[e]];
#pragma unroll
      for (int k = 0; k < NR; ++k) acc[k] += c * x[k * L.n_iface + g];
    }
  lane_sums<NR>(acc, lane);
  if (lane_sum_writer<NR>(lane)) t[lane_sum_index<NR>(lane) * total_rows + r] = rq * acc[0];
}

// y = sum R_i^T (loc - C_i^T t): distinct constraint rows touch disjoint positions (each local DOF lies in
// one glob and has one component)
__global__ void __launch_bounds__(256) k_inner_scatter(LevelDev L, const float* loc,
                                                       const double* t, int64_t total_rows,
                                                       double* __restrict__ y, FusedDot dot) {
  pdl_wait();
  pdl_trigger();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double s = 0.0;
  if (g < L.n_iface) {
    loc += (int64_t)blockIdx.y * L.n_vec;
    t += (int64_t)blockIdx.y * total_rows;
    s = sum_occurrences(L, g, [&](int64_t p) {
      const int32_t r = L.crow[p];
      const double v = (double)loc[p], c = L.cval[p];
      return r >= 0 ? v - t[r] * c : v;
    });
    y[(int64_t)blockIdx.y * L.n_iface + g] = s;
  }
  if (dot.mode) fused_dot(dot, g, L.n_iface, s);
}

__global__ void k_constraint_positions(LevelDev L, const int32_t* __restrict__ crow_sub, int64_t total_rows) {
  const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= total_rows) return;
  const int64_t off = L.meta[crow_sub[r]].vec_off;
  for (int64_t e = L.c_ptr[r] + lane; e < L.c_ptr[r + 1]; e += 32) {
    L.crow[off + L.c_pos[e]] = (int32_t)r;
    L.cval[off + L.c_pos[e]] = L.c_val[e];
  }
}

// part: 0 interior positions only, 1 interface only, 2 all
template <typename T>
__global__ void k_gather_glob(LevelDev L, const double* __restrict__ x, int part, T* __restrict__ loc) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.n_vec) return;
  x += (int64_t)blockIdx.y * L.n_dof;
  loc += (int64_t)blockIdx.y * L.n_vec;
  const int32_t g = L.loc2glob[p];
  const bool is_if = L.loc2iface[p] >= 0;
  double v = 0.0;
  if (g >= 0 && (part == 2 || (part == 0 && !is_if) || (part == 1 && is_if))) v = x[g];
  loc[p] = (T)v;
}

template <typename T>
__global__ void k_scatter_interior(LevelDev L, const T* __restrict__ loc, double* __restrict__ y) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.n_vec) return;
  const int32_t g = L.loc2glob[p];
  if (g >= 0 && L.loc2iface[p] < 0) y[(int64_t)blockIdx.y * L.n_dof + g] = (double)loc[(int64_t)blockIdx.y * L.n_vec + p];
}

__global__ void k_scatter_interior_diff(LevelDev L, const double* __restrict__ a, const double* __restrict__ b,
                                        double* __restrict__ y) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.n_vec) return;
  const int32_t g = L.loc2glob[p];
  const int64_t o = (int64_t)blockIdx.y * L.n_vec + p;
  if (g >= 0 && L.loc2iface[p] < 0) y[(int64_t)blockIdx.y * L.n_dof + g] = a[o] - b[o];
}

// y[row] = beta*y[row] + alpha * (K_i x)[row] for the rows of a list (interior rows, interface rows or all rows
// of every subdomain) and NR right-hand sides.  A group of LR lanes takes a row: its entries are read once
// for all columns, and the FP64 units, which bound the product (2 operations per cycle and SM: 27 M entries
// take 47 us, as long as their 12 bytes each from HBM), spend few additions on the sums over the lanes.
// Sixteen lanes and one column at a time spent as many on those sums as on the products and read the matrix
// once per column: 48^3, 8 columns 700 us.
template <int NR, int LR>
__global__ void __launch_bounds__(256) k_spmv(LevelDev L, const int64_t* __restrict__ rows, int64_t nrows,
                                              const double* x, double* __restrict__ y, double alpha,
                                              double beta, const int32_t* __restrict__ row_sub) {
  pdl_wait();
  pdl_trigger();
  const int64_t g = ((int64_t)blockIdx.x * 256 + threadIdx.x) / LR;
  const int l = threadIdx.x % LR;
  const bool valid = g < nrows;
  const int64_t row = rows[valid ? g : 0];
  const double* xs = x + L.meta[row_sub[row]].vec_off;
  double acc[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) acc[k] = 0.0;
  if (valid) {
    const int64_t q1 = L.row_ptr[row + 1];
    constexpr int U = NR == 1 ? 4 : 2;   // entries in flight per lane
    int64_t q = L.row_ptr[row] + l;
    for (; q + (U - 1) * LR < q1; q += U * LR) {
      double v[U];
      int c[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v[u] = __ldg(L.val + q + u * LR);
        c[u] = __ldg(L.col + q + u * LR);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < NR; ++k) acc[k] += v[u] * xs[(int64_t)k * L.n_vec + c[u]];
    }
    for (; q < q1; q += LR) {
      const double v = __ldg(L.val + q);
      const int c = __ldg(L.col + q);
#pragma unroll
      for (int k = 0; k < NR; ++k) acc[k] += v * xs[(int64_t)k * L.n_vec + c];
    }
  }
#pragma unroll
  for (int k = 0; k < NR; ++k) {
#pragma unroll
    for (int o = LR / 2; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
  }
  if (valid) {
#pragma unroll
    for (int k = 0; k < NR; ++k)
      if (l == k % LR) {
        double* yr = y + (int64_t)k * L.n_vec + row;
        *yr = (beta == 0.0 ? 0.0 : beta * *yr) + alpha * acc[k];
      }
  }
}

template <typename Tin, typename Tout>
__global__ void k_convert(const Tin* in, Tout* __restrict__ out, int64_t n) {
  pdl_wait();
  pdl_trigger();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (Tout)in[i];
}

template <typename T>
__global__ void k_add_to_double(double* __restrict__ y, const T* x, int64_t n) {
  pdl_wait();
  pdl_trigger();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] += (double)x[i];
}

__global__ void k_axpy(double* __restrict__ y, const double* x, double a, int64_t n) {
  pdl_wait();
  pdl_trigger();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] += a * x[i];
}

// One warp per coarse DOF, which owns its per-subdomain rows: 4 rows at a time, 8 lanes along each row's parts
// (a thread per DOF summed up to 120 parts in a chain of loads).
__global__ void k_coarse_gather(LevelDev L, const double* part, int zmax, double* __restrict__ rc_sub,
                                int64_t sum_nc, double* __restrict__ rC, float* __restrict__ v32,
                                const int32_t* __restrict__ v32_pos, int64_t n_v32) {
  pdl_wait();
  pdl_trigger();
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (g >= L.n_coarse) return;
  part += (int64_t)blockIdx.y * sum_nc * zmax;
  rc_sub += (int64_t)blockIdx.y * sum_nc;
  const int64_t o1 = L.cinv_ptr[g + 1];
  double s = 0.0;
  for (int64_t o0 = L.cinv_ptr[g]; o0 < o1; o0 += 4) {
    const int64_t o = o0 + (lane >> 3);
    const int64_t r = o < o1 ? L.cinv_occ[o] : -1;
    double t = 0.0;
    if (r >= 0)
      for (int z = lane & 7; z < zmax; z += 8) t += part[r * zmax + z];
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) t += __shfl_xor_sync(0xffffffffu, t, h);
    if (r >= 0 && (lane & 7) == 0) rc_sub[r] = t;
    t += __shfl_xor_sync(0xffffffffu, t, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    s += t;
  }
  if (lane == 0) {
    rC[(int64_t)blockIdx.y * L.n_coarse + g] = s;
    if (v32) v32[(int64_t)blockIdx.y * n_v32 + v32_pos[g]] = (float)s;
  }
}

__global__ void k_coarse_scatter(const int32_t* __restrict__ sub_coarse, int64_t total, const double* __restrict__ zC,
                                 int64_t n_coarse, double* __restrict__ zc_sub) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < total) zc_sub[(int64_t)blockIdx.y * total + t] = zC[(int64_t)blockIdx.y * n_coarse + sub_coarse[t]];
}

// deterministic dot: fixed grid, per-block tree, then a single block over the partials
__global__ void k_dot_partial(const double* __restrict__ a, const double* __restrict__ b, int64_t n,
                              double* __restrict__ partial) {
  __shared__ double red[256];
  a += (int64_t)blockIdx.y * n;
  b += (int64_t)blockIdx.y * n;
  partial += (int64_t)blockIdx.y * gridDim.x;
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += a[i] * b[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_dot_final(const double* __restrict__ partial, int nblk, double* __restrict__ out, int ostride) {
  __shared__ double red[256];
  partial += (int64_t)blockIdx.x * nblk;
  out += (int64_t)blockIdx.x * ostride;
  double s = 0.0;
  for (int i = threadIdx.x; i < nblk; i += 256) s += partial[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

__global__ void __launch_bounds__(256) k_pcg_xr(double* __restrict__ x, double* __restrict__ r,
                                                const double* p, const double* q,
                                                double* __restrict__ scal, int64_t n, double* __restrict__ partial,
                                                int* cnt, KrylovStore ks, double* mail) {
  pdl_wait();
  pdl_trigger();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double rr = 0.0, s0, s1;
  const double a = scal[16 * blockIdx.y + 2];
  const int slot = ks.cap > 0 && a != 0.0 ? ks.cnt[blockIdx.y] : ks.cap;
  if (i < n) {
    const int64_t o = (int64_t)blockIdx.y * n + i;
    const double pv = p[o], qv = q[o];
    x[o] += a * pv;
    const double v = r[o] - a * qv;
    r[o] = v;
    rr = v * v;
    if (slot < ks.cap) {
      const int64_t k = ((int64_t)blockIdx.y * ks.cap + slot) * n + i;
      ks.p[k] = (float)pv;
      ks.q[k] = (float)qv;
    }
  }
  if (sum_over_grid(rr, 0.0, false, partial, cnt, s0, s1) && threadIdx.x == 0) {
    double* S = scal + 16 * blockIdx.y;
    S[5] = s0;
    S[7] += 1.0;   // iteration number
    double* box = mail + 4 * blockIdx.y;
    box[0] = s0;
    box[1] = a;
    box[2] = S[3];
    __threadfence_system();
    *(volatile long long*)(box + 3) = (long long)S[7];
    if (slot < ks.cap) {   // every block has read its count (this one is the last)
      ks.d[(int64_t)blockIdx.y * ks.cap + slot] = scal[16 * blockIdx.y + 1];
      ks.cnt[blockIdx.y] = slot + 1;
    }
  }
}

// coef[(k cap + v)(kProjBlocks + 1) + b] = slice b of p_v . g of column k
__global__ void __launch_bounds__(256) k_project_dot(KrylovStore ks, const double* __restrict__ g, int64_t n,
                                                     double* __restrict__ coef) {
  const int v = blockIdx.y, k = blockIdx.z;
  if (v >= ks.cnt[k]) return;
  __shared__ double red[8];
  const float* p = ks.p + ((int64_t)k * ks.cap + v) * n;
  g += (int64_t)k * n;
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += (double)p[i] * g[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += red[w];
    coef[((int64_t)k * ks.cap + v) * (kProjBlocks + 1) + blockIdx.x] = s;
  }
}

// c_v into slot kProjBlocks of its row; one thread per (v, column)
__global__ void k_project_coef(KrylovStore ks, double* __restrict__ coef) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
  if (v >= ks.cnt[k]) return;
  double* c = coef + ((int64_t)k * ks.cap + v) * (kProjBlocks + 1);
  double s = 0.0;
  for (int b = 0; b < kProjBlocks; ++b) s += c[b];
  const double d = ks.d[(int64_t)k * ks.cap + v];
  c[kProjBlocks] = d > 0.0 ? s / d : 0.0;
}

__global__ void __launch_bounds__(256) k_project_apply(KrylovStore ks, const double* __restrict__ g,
                                                       double* __restrict__ x, double* __restrict__ r, int64_t n,
                                                       const double* __restrict__ coef) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int k = blockIdx.y, m = ks.cnt[k];
  if (i >= n) return;
  const float* p = ks.p + (int64_t)k * ks.cap * n + i;
  const float* q = ks.q + (int64_t)k * ks.cap * n + i;
  const double* c = coef + (int64_t)k * ks.cap * (kProjBlocks + 1) + kProjBlocks;
  double xs = 0.0, rs = g[(int64_t)k * n + i];
#pragma unroll 4
  for (int v = 0; v < m; ++v) {
    const double cv = c[(int64_t)v * (kProjBlocks + 1)];
    xs += cv * (double)p[(int64_t)v * n];
    rs -= cv * (double)q[(int64_t)v * n];
  }
  x[(int64_t)k * n + i] = xs;
  r[(int64_t)k * n + i] = rs;
}

__global__ void k_pcg_p(double* __restrict__ p, const double* z, const double* scal,
                        int64_t n) {
  pdl_wait();
  pdl_trigger();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t o = (int64_t)blockIdx.y * n;
  p[o + i] = z[o + i] + scal[16 * blockIdx.y + 3] * p[o + i];
}

// grad[e] = -(1/coef_e) * sum_k lam_k,e^T K_e u_k,e ; one warp per element
__global__ void k_grad_contract(int64_t n_elems, int ne, const double* __restrict__ ke,
                                const int32_t* __restrict__ slot_elem, const double* __restrict__ coef,
                                const int32_t* __restrict__ conn, int ndof, const double* __restrict__ lam,
                                const double* __restrict__ u, int nrhs, int64_t n_full, double* __restrict__ grad) {
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (slot >= n_elems) return;
  const int64_t e = slot_elem[slot];
  const double* K = ke + slot * (int64_t)ne * ne;
  const int32_t* cn = conn + e * (int64_t)(ne / ndof);
  auto dof = [&](int a) { return (int64_t)cn[a / ndof] * ndof + a % ndof; };
  double acc = 0.0;
  for (int k = 0; k < nrhs; ++k) {
    const double* lk = lam + (int64_t)k * n_full;
    const double* uk = u + (int64_t)k * n_full;
    for (int a = lane; a < ne; a += 32) {
      double t = 0.0;
      for (int b = 0; b < ne; ++b) t += K[a * ne + b] * uk[dof(b)];
      acc += lk[dof(a)] * t;
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) grad[e] = -acc / coef[e];
}

__global__ void k_expand_free(const double* __restrict__ xf, const int64_t* __restrict__ free_of_full,
                              int64_t n_full, int nrhs, int64_t n_free, double* __restrict__ xfull) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_full * nrhs) return;
  const int64_t k = i / n_full, j = i % n_full;
  const int64_t f = free_of_full[j];
  xfull[i] = f >= 0 ? xf[k * n_free + f] : 0.0;
}

// dst[dst_off[k] + t] = src[src_off[k] + t], t < len[k]; one block per segment
__global__ void k_copy_segments(const double* __restrict__ src, const int64_t* __restrict__ src_off,
                                double* __restrict__ dst, const int64_t* __restrict__ dst_off,
                                const int64_t* __restrict__ len, int64_t n) {
  const int64_t k = blockIdx.x;
  if (k >= n) return;
  for (int64_t t = threadIdx.x; t < len[k]; t += blockDim.x) dst[dst_off[k] + t] = src[src_off[k] + t];
}

// g[k] = f[idx[k]] - t[k] (column blockIdx.y; f has columns of length fstride)
__global__ void k_iface_rhs(double* __restrict__ g, const double* __restrict__ f, int64_t fstride,
                            const int64_t* __restrict__ idx, const double* __restrict__ t, int64_t n) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t o = (int64_t)blockIdx.y * n;
  if (k < n) g[o + k] = f[(int64_t)blockIdx.y * fstride + idx[k]] - t[o + k];
}

// u[idx[k]] = v[k] (column blockIdx.y; u has columns of length ustride)
__global__ void k_put_indexed(double* __restrict__ u, int64_t ustride, const int64_t* __restrict__ idx,
                              const double* __restrict__ v, int64_t n) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) u[(int64_t)blockIdx.y * ustride + idx[k]] = v[(int64_t)blockIdx.y * n + k];
}

// BiCGstab (right preconditioned) device scalars; layout: 0 rho, 1 alpha, 2 omega, 3 rho_new,
// 4 rh.v, 5 t.s, 6 t.t, 7 beta.  A zero denominator (breakdown) yields 0, which the host sees as
// a stalled residual.
__global__ void k_bicg_scalars(double* S, int stage) {
  if (threadIdx.x != 0) return;
  if (stage == 3) {          // start: rho = alpha = omega = 1
    S[0] = S[1] = S[2] = 1.0;
  } else if (stage == 0) {   // beta = (rho_new / rho) (alpha / omega)
    S[7] = (S[0] != 0.0 && S[2] != 0.0) ? (S[3] / S[0]) * (S[1] / S[2]) : 0.0;
    S[0] = S[3];
  } else if (stage == 1) {   // alpha = rho / (rh . v)
    S[1] = S[4] != 0.0 ? S[0] / S[4] : 0.0;
  } else {                   // omega = (t . s) / (t . t)
    S[2] = S[6] != 0.0 ? S[5] / S[6] : 0.0;
  }
}

// p = r + beta (p - omega v)
__global__ void k_bicg_p(double* __restrict__ p, const double* __restrict__ r, const double* __restrict__ v,
                         const double* __restrict__ S, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = r[i] + S[7] * (p[i] - S[2] * v[i]);
}

// s = r - alpha v
__global__ void k_bicg_s(double* __restrict__ sv, const double* __restrict__ r, const double* __restrict__ v,
                         const double* __restrict__ S, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) sv[i] = r[i] - S[1] * v[i];
}

// x += alpha ph + omega sh ; r = s - omega t
__global__ void k_bicg_xr(double* __restrict__ x, double* __restrict__ r, const double* __restrict__ ph,
                          const double* __restrict__ sh, const double* __restrict__ sv, const double* __restrict__ t,
                          const double* __restrict__ S, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  x[i] += S[1] * ph[i] + S[2] * sh[i];
  r[i] = sv[i] - S[2] * t[i];
}

// ---- flexible GMRES building blocks (fixed-order, reproducible) ----
// partial[i * nblk + b] = sum over the grid-stride slice b of V_i . w, for i < nv (grid nblk x nv)
__global__ void k_multidot_partial(const double* __restrict__ V, int64_t ldv, const double* __restrict__ w, int64_t n,
                                   double* __restrict__ partial) {
  __shared__ double red[256];
  const double* v = V + (int64_t)blockIdx.y * ldv;
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += v[i] * w[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = red[0];
}

// out[i] = sum_b partial[i * nblk + b]; one block per i
__global__ void k_multidot_final(const double* __restrict__ partial, int nblk, double* __restrict__ out) {
  __shared__ double red[256];
  const double* p = partial + (int64_t)blockIdx.x * nblk;
  double s = 0.0;
  for (int i = threadIdx.x; i < nblk; i += 256) s += p[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

// w += alpha sum_{i < nv} c_i V_i, i ascending
__global__ void k_combine(double* __restrict__ w, const double* __restrict__ V, int64_t ldv, int nv,
                          const double* __restrict__ c, double alpha, int64_t n) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  double acc = 0.0;
  for (int i = 0; i < nv; ++i) acc += c[i] * V[(int64_t)i * ldv + k];
  w[k] += alpha * acc;
}

// dst = src / sqrt(*nrm2) (dst = 0 when the norm vanishes: lucky breakdown)
__global__ void k_scale_by_norm(double* __restrict__ dst, const double* __restrict__ src,
                                const double* __restrict__ nrm2, int64_t n) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double s = *nrm2 > 0.0 ? 1.0 / sqrt(*nrm2) : 0.0;
  dst[k] = src[k] * s;
}

inline unsigned nblocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

template <typename T>
void launch_gather_iface(const LevelDev& L, const double* x, int weighted, T* loc, cudaStream_t st, int nr,
                         int after_kernel) {
  if (L.n_vec > 0) { note_launch(); launch_pdl_if(after_kernel, k_gather_iface<T>, dim3(nblocks(L.n_vec, 256), nr), 256, 0, st, L, x, weighted, loc); }
}
template <typename T>
void launch_scatter_iface(const LevelDev& L, const T* loc, int weighted, double* y, cudaStream_t st, int nr,
                          const FusedDot& dot, int after_kernel) {
  if (L.n_iface > 0) { note_launch(); launch_pdl_if(after_kernel, k_scatter_iface<T>, dim3(nblocks(L.n_iface, 256), nr), 256, 0, st, L, loc, weighted, y, dot); }
}
void launch_inner_gather(const LevelDev& L, const double* x, float* loc, const int32_t* crow_sub, int64_t total_rows,
                         double* t, cudaStream_t st, int nr) {
  if (L.n_vec <= 0) return;
  const unsigned nv = nblocks(L.n_vec, 256), nb = nv + nblocks(total_rows, 8);
  for (int r0 = 0; r0 < nr;) {
    const int left = nr - r0, g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    const double* xs = x + (int64_t)r0 * L.n_iface;
    float* ls = loc + (int64_t)r0 * L.n_vec;
    double* ts = t + (int64_t)r0 * total_rows;
    note_launch();
    if (g == 8)
      k_inner_gather<8><<<nb, 256, 0, st>>>(L, xs, ls, (int)nv, crow_sub, total_rows, ts);
    else if (g == 4)
      k_inner_gather<4><<<nb, 256, 0, st>>>(L, xs, ls, (int)nv, crow_sub, total_rows, ts);
    else if (g == 2)
      k_inner_gather<2><<<nb, 256, 0, st>>>(L, xs, ls, (int)nv, crow_sub, total_rows, ts);
    else
      k_inner_gather<1><<<nb, 256, 0, st>>>(L, xs, ls, (int)nv, crow_sub, total_rows, ts);
    r0 += g;
  }
}
void launch_inner_scatter(const LevelDev& L, const float* loc, const double* t, int64_t total_rows, double* y,
                          cudaStream_t st, int nr, const FusedDot& dot) {
  if (L.n_iface <= 0) return;
  note_launch();
  launch_pdl(k_inner_scatter, dim3(nblocks(L.n_iface, 256), nr), 256, 0, st, L, loc, t, total_rows, y, dot);
}
void launch_constraint_positions(const LevelDev& L, const int32_t* crow_sub, int64_t total_rows, cudaStream_t st) {
  if (total_rows > 0) { note_launch(); k_constraint_positions<<<nblocks(total_rows, 8), 256, 0, st>>>(L, crow_sub, total_rows); }
}
template <typename T>
void launch_gather_glob(const LevelDev& L, const double* x, int part, T* loc, cudaStream_t st, int nr) {
  if (L.n_vec > 0) { note_launch(); k_gather_glob<T><<<dim3(nblocks(L.n_vec, 256), nr), 256, 0, st>>>(L, x, part, loc); }
}
template <typename T>
void launch_scatter_interior(const LevelDev& L, const T* loc, double* y, cudaStream_t st, int nr) {
  if (L.n_vec > 0) { note_launch(); k_scatter_interior<T><<<dim3(nblocks(L.n_vec, 256), nr), 256, 0, st>>>(L, loc, y); }
}
void launch_scatter_interior_diff(const LevelDev& L, const double* a, const double* b, double* y, cudaStream_t st,
                                  int nr) {
  if (L.n_vec > 0) { note_launch(); k_scatter_interior_diff<<<dim3(nblocks(L.n_vec, 256), nr), 256, 0, st>>>(L, a, b, y); }
}
template <int NR>
void launch_spmv_nr(const LevelDev& L, const int64_t* rows, int64_t nrows, const double* x, double* y, double alpha,
                    double beta, const int32_t* row_sub, cudaStream_t st, int after_kernel) {
  constexpr int LR = 4;
  note_launch();
  launch_pdl_if(after_kernel, k_spmv<NR, LR>, nblocks(nrows * LR, 256), 256, 0, st, L, rows, nrows, x, y, alpha, beta, row_sub);
}
void launch_spmv_rows(const LevelDev& L, const int64_t* rows, int64_t nrows, const double* x, double* y, double alpha,
                      double beta, const int32_t* row_sub, cudaStream_t st, int nr, int after_kernel) {
  if (nrows <= 0) return;
  for (int r0 = 0; r0 < nr;) {   // columns in groups of 8, 4, 2, 1: one pass over the matrix each
    const int left = nr - r0, g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    const double* xs = x + (int64_t)r0 * L.n_vec;
    double* ys = y + (int64_t)r0 * L.n_vec;
    if (g == 8)
      launch_spmv_nr<8>(L, rows, nrows, xs, ys, alpha, beta, row_sub, st, after_kernel);
    else if (g == 4)
      launch_spmv_nr<4>(L, rows, nrows, xs, ys, alpha, beta, row_sub, st, after_kernel);
    else if (g == 2)
      launch_spmv_nr<2>(L, rows, nrows, xs, ys, alpha, beta, row_sub, st, after_kernel);
    else
      launch_spmv_nr<1>(L, rows, nrows, xs, ys, alpha, beta, row_sub, st, after_kernel);
    r0 += g;
    after_kernel = kAfterKernel;
  }
}
template <typename Tin, typename Tout>
void launch_convert(const Tin* in, Tout* out, int64_t n, cudaStream_t st, int after_kernel) {
  if (n > 0) { note_launch(); launch_pdl_if(after_kernel, k_convert<Tin, Tout>, nblocks(n, 256), 256, 0, st, in, out, n); }
}
template <typename T>
void launch_add_to_double(double* y, const T* x, int64_t n, cudaStream_t st, int after_kernel) {
  if (n > 0) { note_launch(); launch_pdl_if(after_kernel, k_add_to_double<T>, nblocks(n, 256), 256, 0, st, y, x, n); }
}
void launch_axpy_loc(double* y, const double* x, double a, int64_t n, cudaStream_t st, int after_kernel) {
  if (n > 0) { note_launch(); launch_pdl_if(after_kernel, k_axpy, nblocks(n, 256), 256, 0, st, y, x, a, n); }
}
void launch_coarse_gather(const LevelDev& L, const double* part, int zmax, double* rc_sub, int64_t sum_nc, double* rC,
                          float* v32, const int32_t* v32_pos, int64_t n_v32, cudaStream_t st, int nr) {
  if (L.n_coarse <= 0) return;
  note_launch();
  launch_pdl(k_coarse_gather, dim3(nblocks(L.n_coarse, 8), nr), 256, 0, st, L, part, zmax, rc_sub, sum_nc, rC, v32, v32_pos, n_v32);
}
void launch_coarse_scatter_n(const int32_t* sub_coarse, int64_t total, const double* zC, int64_t n_coarse,
                             double* zc_sub, cudaStream_t st, int nr) {
  if (total > 0) { note_launch(); k_coarse_scatter<<<dim3(nblocks(total, 256), nr), 256, 0, st>>>(sub_coarse, total, zC, n_coarse, zc_sub); }
}
void launch_dot(const double* a, const double* b, int64_t n, double* partial, int nblk, double* out, cudaStream_t st,
                int nr, int ostride) {
  { note_launch(); k_dot_partial<<<dim3(nblk, nr), 256, 0, st>>>(a, b, n, partial); }
  { note_launch(); k_dot_final<<<nr, 256, 0, st>>>(partial, nblk, out, ostride); }
}
void launch_pcg_update_x_r(double* x, double* r, const double* p, const double* q, double* scal, int64_t n,
                           double* partial, int* cnt, const KrylovStore& ks, double* mail, cudaStream_t st, int nr) {
  if (n > 0) { note_launch(); launch_pdl(k_pcg_xr, dim3(nblocks(n, 256), nr), 256, 0, st, x, r, p, q, scal, n, partial, cnt, ks, mail); }
}
void launch_project(const KrylovStore& ks, const double* g, double* x, double* r, int64_t n, double* coef,
                    cudaStream_t st, int nr) {
  if (n <= 0 || ks.cap <= 0) return;
  note_launch();
  k_project_dot<<<dim3(kProjBlocks, ks.cap, nr), 256, 0, st>>>(ks, g, n, coef);
  note_launch();
  k_project_coef<<<dim3(nblocks(ks.cap, 128), nr), 128, 0, st>>>(ks, coef);
  note_launch();
  k_project_apply<<<dim3(nblocks(n, 256), nr), 256, 0, st>>>(ks, g, x, r, n, coef);
}
void launch_pcg_update_p(double* p, const double* z, const double* scal, int64_t n, cudaStream_t st, int nr) {
  if (n > 0) { note_launch(); launch_pdl(k_pcg_p, dim3(nblocks(n, 256), nr), 256, 0, st, p, z, scal, n); }
}
void launch_grad_contract_slots(int64_t n_elems, int ne, const double* ke, const int32_t* slot_elem, const double* coef,
                                const int32_t* conn, int ndof, const double* lam, const double* u, int nrhs,
                                int64_t n_full, double* grad, cudaStream_t st) {
  if (n_elems > 0)
    { note_launch(); k_grad_contract<<<nblocks(n_elems, 8), 256, 0, st>>>(n_elems, ne, ke, slot_elem, coef, conn, ndof, lam, u,
                                                          nrhs, n_full, grad); }
}
void launch_expand_free(const double* xf, const int64_t* free_of_full, int64_t n_full, int nrhs, int64_t n_free,
                        double* xfull, cudaStream_t st) {
  if (n_full > 0)
    { note_launch(); k_expand_free<<<nblocks(n_full * nrhs, 256), 256, 0, st>>>(xf, free_of_full, n_full, nrhs, n_free, xfull); }
}

void launch_copy_segments(const double* src, const int64_t* src_off, double* dst, const int64_t* dst_off,
                          const int64_t* len, int64_t n, cudaStream_t st) {
  if (n > 0) { note_launch(); k_copy_segments<<<(unsigned)n, 256, 0, st>>>(src, src_off, dst, dst_off, len, n); }
}
void launch_iface_rhs(double* g, const double* f, int64_t fstride, const int64_t* idx, const double* t, int64_t n,
                      cudaStream_t st, int nr) {
  if (n > 0) { note_launch(); k_iface_rhs<<<dim3(nblocks(n, 256), nr), 256, 0, st>>>(g, f, fstride, idx, t, n); }
}
void launch_put_indexed(double* u, int64_t ustride, const int64_t* idx, const double* v, int64_t n, cudaStream_t st,
                        int nr) {
  if (n > 0) { note_launch(); k_put_indexed<<<dim3(nblocks(n, 256), nr), 256, 0, st>>>(u, ustride, idx, v, n); }
}

void launch_multidot(const double* V, int64_t ldv, int nv, const double* w, int64_t n, double* partial, int nblk,
                     double* out, cudaStream_t st) {
  if (nv <= 0) return;
  note_launch();
  k_multidot_partial<<<dim3(nblk, nv), 256, 0, st>>>(V, ldv, w, n, partial);
  note_launch();
  k_multidot_final<<<nv, 256, 0, st>>>(partial, nblk, out);
}
void launch_combine(double* w, const double* V, int64_t ldv, int nv, const double* c, double alpha, int64_t n,
                    cudaStream_t st) {
  if (n > 0 && nv > 0) { note_launch(); k_combine<<<nblocks(n, 256), 256, 0, st>>>(w, V, ldv, nv, c, alpha, n); }
}
void launch_scale_by_norm(double* dst, const double* src, const double* nrm2, int64_t n, cudaStream_t st) {
  if (n > 0) { note_launch(); k_scale_by_norm<<<nblocks(n, 256), 256, 0, st>>>(dst, src, nrm2, n); }
}

void launch_bicg_scalars(double* S, int stage, cudaStream_t st) {
  note_launch();
  k_bicg_scalars<<<1, 32, 0, st>>>(S, stage);
}
void launch_bicg_p(double* p, const double* r, const double* v, const double* S, int64_t n, cudaStream_t st) {
  if (n > 0) { note_launch(); k_bicg_p<<<nblocks(n, 256), 256, 0, st>>>(p, r, v, S, n); }
}
void launch_bicg_s(double* sv, const double* r, const double* v, const double* S, int64_t n, cudaStream_t st) {
  if (n > 0) { note_launch(); k_bicg_s<<<nblocks(n, 256), 256, 0, st>>>(sv, r, v, S, n); }
}
void launch_bicg_xr(double* x, double* r, const double* ph, const double* sh, const double* sv, const double* t,
                    const double* S, int64_t n, cudaStream_t st) {
  if (n > 0) { note_launch(); k_bicg_xr<<<nblocks(n, 256), 256, 0, st>>>(x, r, ph, sh, sv, t, S, n); }
}

#define INST(T)                                                                             \
  template void launch_gather_iface<T>(const LevelDev&, const double*, int, T*, cudaStream_t, int, int); \
  template void launch_scatter_iface<T>(const LevelDev&, const T*, int, double*, cudaStream_t, int, const FusedDot&, int); \
  template void launch_gather_glob<T>(const LevelDev&, const double*, int, T*, cudaStream_t, int);  \
  template void launch_scatter_interior<T>(const LevelDev&, const T*, double*, cudaStream_t, int);  \
  template void launch_add_to_double<T>(double*, const T*, int64_t, cudaStream_t, int);
INST(float)
INST(double)
#undef INST
template void launch_convert<double, float>(const double*, float*, int64_t, cudaStream_t, int);
template void launch_convert<float, double>(const float*, double*, int64_t, cudaStream_t, int);
template void launch_convert<double, double>(const double*, double*, int64_t, cudaStream_t, int);

}  // namespace bddc
