// Global control variate g_x = Q(phi) h_x, Q = sum_i q_i phi(r_i) = rho . phi,
// with h a fixed field of the charge set (no phi dependence).  Its Stein term
//   T g = sum_x (dg_x/dphi_x - g_x (A phi)_x) = h . rho - Q (A h) . phi
// has mean 0 under exp(-H_L) for any h (integration by parts).  With
// h = -G rho it equals Q^2 - rho.G.rho, so e - T g = rho.G.rho - P: the far
// pairs' part of the variance of the Eq. (nsum2) sample is gone and only that
// of P = sum_i (q_i phi_i)^2 is left.  h comes from red/black SOR on
// A h = -rho (sor.cu, once per charge set); the estimator stays unbiased whatever the
// solver's residual, which only sets how much variance is removed.
//
// A second, local term removes most of the variance of P: g^P_x =
// sum_i q_i^2 phi(r_i) k(x - r_i), k a fixed kernel of radius R (the
// Dirichlet Green function of the (2R+1)^3 cube at its centre, restricted to
// the box), has Stein term
//   T g^P = k(0) sum_i q_i^2 - sum_i q_i^2 phi(r_i) w_i,
//   w_i = sum_d k(d) (A phi)(r_i + d)   (d over the cube, r_i + d in the box);
// with k = G(., r_i) it would equal sum q^2 G_ii - P, so e - T g - T g^P would
// be E_lat exactly.  Mean 0 for any k, like T g.
//
// Exactness: h is rounded to the fixed-point grid 2^-k (h~, k as large as lets
// 13 max|h~| 2^k stay below 2^24), so v = A h~ is a multiple of 2^-k below
// 2^24 2^-k in magnitude and exact in FP32; h~ . rho is formed in FP64.  Thus
// E[T g] = 0 holds for the h~ actually used.  The per-sample v . phi adds FP32
// products in FP32 over 16 sites and those partial sums in FP64.
#include <algorithm>
#include <cmath>

#include "charge_local.cuh"
#include "device_common.cuh"
#include "internal.h"
#include "sor.cuh"

namespace coulps {
namespace {

constexpr int kGcvThreads = 256;

__device__ __forceinline__ double nat_at(const double *u, int Lx, int Ly, int Lz, int x, int y,
                                         int z) {
  if (x < 0 || y < 0 || z < 0 || x >= Lx || y >= Ly || z >= Lz) return 0.0;
  return u[((size_t)z * Ly + y) * Lx + x];
}

__device__ __forceinline__ void block_sum2(double a, double b, double *out) {
  __shared__ double red[2][kGcvThreads / 32];
  a = warp_sum(a);
  b = warp_sum(b);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    red[0][wid] = a;
    red[1][wid] = b;
  }
  __syncthreads();
  if (wid == 0) {
    a = lane < kGcvThreads / 32 ? red[0][lane] : 0.0;
    b = lane < kGcvThreads / 32 ? red[1][lane] : 0.0;
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) {
      out[0] = a;
      out[1] = b;
    }
  }
}

// per block four doubles: sum (A u + rho)^2, sum rho^2, max |u|, 0
__global__ void gcv_check_kernel(const double *__restrict__ u, const double *__restrict__ rho,
                                 int Lx, int Ly, int Lz, double *__restrict__ partials) {
  const int64_t n = (int64_t)Lx * Ly * Lz;
  double r2 = 0.0, b2 = 0.0, mx = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % Lx), y = (int)((i / Lx) % Ly), z = (int)(i / ((int64_t)Lx * Ly));
    const double S = nat_at(u, Lx, Ly, Lz, x - 1, y, z) + nat_at(u, Lx, Ly, Lz, x + 1, y, z) +
                     nat_at(u, Lx, Ly, Lz, x, y - 1, z) + nat_at(u, Lx, Ly, Lz, x, y + 1, z) +
                     nat_at(u, Lx, Ly, Lz, x, y, z - 1) + nat_at(u, Lx, Ly, Lz, x, y, z + 1);
    const double r = 6.0 * u[i] - S + rho[i];
    r2 += r * r;
    b2 += rho[i] * rho[i];
    mx = fmax(mx, fabs(u[i]));
  }
  block_sum2(r2, b2, partials + 4 * blockIdx.x);
  __syncthreads();
  // block max of mx through the same tree (max is order-free)
  __shared__ double m[kGcvThreads / 32];
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) m[wid] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kGcvThreads / 32; ++w) mx = fmax(mx, m[w]);
    partials[4 * blockIdx.x + 2] = mx;
    partials[4 * blockIdx.x + 3] = 0.0;
  }
}

// res[1] = |A u + rho| / |rho|, res[2] = max |u|
__global__ void gcv_check_sums_kernel(const double *__restrict__ partials, int nblk,
                                      double *__restrict__ res) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double r2 = 0.0, b2 = 0.0, mx = 0.0;
  for (int b = 0; b < nblk; ++b) {
    r2 += partials[4 * b + 0];
    b2 += partials[4 * b + 1];
    mx = fmax(mx, partials[4 * b + 2]);
  }
  res[1] = b2 > 0.0 ? sqrt(r2 / b2) : 0.0;
  res[2] = mx;
}

// h~ = round(u 2^k) 2^-k (an FP32 value), per block h~ . rho
__global__ void gcv_quantize_kernel(const double *__restrict__ u, const double *__restrict__ rho,
                                    int64_t n, double scale, double inv_scale,
                                    float *__restrict__ h32, double *__restrict__ partials) {
  double hr = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float h = (float)(rint(u[i] * scale) * inv_scale);
    h32[i] = h;
    hr += (double)h * rho[i];
  }
  block_sum2(hr, 0.0, partials + 2 * blockIdx.x);
}

__global__ void gcv_c0_kernel(const double *__restrict__ partials, int nblk,
                              double *__restrict__ res) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double hr = 0.0;
  for (int b = 0; b < nblk; ++b) hr += partials[2 * b];
  res[0] = hr;
}

// Where element e of a chain's storage lies in v.  FP32 fields: within each
// whole run of 512 elements (32 chunks of 16), the four quads of the chunk that
// lane l sums (gcv_eval_kernel: chunk 8 (l % 4) + l / 4) lie 32 quads apart, in
// the lanes' order, so that a warp's loads are contiguous.
__host__ __device__ __forceinline__ size_t v_place(size_t e, size_t chain_elems, bool f32) {
  if (!f32 || (e | 511) >= chain_elems) return e;
  const size_t chunk = (e >> 4) & 31, lane = 4 * (chunk & 7) + (chunk >> 3);
  return (e & ~(size_t)511) | ((e & 12) << 5) | (lane << 2) | (e & 3);
}

// v = A h~ (exact in FP32, see above), in the field's per-chain layout
// (colour-split, padded rows; padding and the x >= Lx tail stay 0), permuted
// by v_place
__global__ void gcv_v_kernel(const float *__restrict__ h32, Geometry g, float *__restrict__ v) {
  const int64_t n = (int64_t)g.Lx * g.Ly * g.Lz;
  const int Lx = g.Lx, Ly = g.Ly, Lz = g.Lz;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % Lx), y = (int)((i / Lx) % Ly), z = (int)(i / ((int64_t)Lx * Ly));
    auto at = [&](int xx, int yy, int zz) -> double {
      if (xx < 0 || yy < 0 || zz < 0 || xx >= Lx || yy >= Ly || zz >= Lz) return 0.0;
      return (double)h32[((size_t)zz * Ly + yy) * Lx + xx];
    };
    const double val = 6.0 * (double)h32[i] - at(x - 1, y, z) - at(x + 1, y, z) - at(x, y - 1, z) -
                       at(x, y + 1, z) - at(x, y, z - 1) - at(x, y, z + 1);
    const int c = (x + y + z) & 1;
    const size_t e = (size_t)c * g.colour_elems + ((size_t)z * Ly + y) * g.W + (x >> 1);
    v[v_place(e, g.chain_elems, g.precision == COULPS_F32)] = (float)val;
  }
}

// One launch for both sums, a chain's blocks one after another in the grid: the
// local term's charge neighbourhoods are then read while the chain is still in
// L2 from its v . phi.
//
// v . phi: a lane adds the products of 16 consecutive elements in FP32, those
// sums in FP64.  A warp loads its 512 elements in four contiguous pieces, four
// lanes a chunk of 16 at a time, and four lanes then exchange quads so that each
// has one chunk (a lane loading its own 64 bytes made 16 cache line accesses per
// load, and those, not DRAM, were the time; through shared memory by bulk
// copies 113 us, its barriers and v's latency in the way).
//
// Local term: charge_local.cuh, up to kEvalCharges charges of a chain a warp, or a
// warp a charge (gcv_direct).
//
// Measured, evaluation of 128^3 x 64 chains, 4096 charges (cold L2, the finish
// kernel included): R = 1 313 -> 243 us, R = 0 144 -> 116.  v . phi is near its
// DRAM time (77); the local term is bound by its accesses to L1.
constexpr int kEvalTile = 4096;  // elements a block takes at a time
constexpr int kEvalWarps = kGcvThreads / 32;
template <typename T> constexpr int kEvalCharges = sizeof(T) == 4 ? 16 : 8;

struct EvalArgs {
  const void *field;
  const float *v;
  const uint32_t *idx;
  const double *q;
  int64_t n_q;
  const float *kt;  // kernel values, then the points (gcv_points)
  int R, per;       // per: charges of a warp
  int n_pts;
  int nblk, nblk_p;
  double *partials, *ppart;
};

__device__ __forceinline__ float4 pick(bool c, const float4 &x, const float4 &y) {
  return make_float4(c ? x.x : y.x, c ? x.y : y.y, c ? x.z : y.z, c ? x.w : y.w);
}
__device__ __forceinline__ float4 swap_lanes(const float4 &x, int mask) {
  return make_float4(__shfl_xor_sync(0xffffffffu, x.x, mask), __shfl_xor_sync(0xffffffffu, x.y, mask),
                     __shfl_xor_sync(0xffffffffu, x.z, mask), __shfl_xor_sync(0xffffffffu, x.w, mask));
}
// Four lanes' 4 x 4 quads transposed: lane l % 4 = j holds x[i] = quad j of chunk
// i before, quads x[0 .. 3] of chunk j after.
__device__ __forceinline__ void transpose_quads(float4 (&x)[4], int lane) {
#pragma unroll
  for (int b = 1; b <= 2; b *= 2) {
    const bool up = lane & b;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i & b) continue;
      const float4 got = swap_lanes(pick(up, x[i], x[i + b]), b);
      x[i] = pick(up, got, x[i]);
      x[i + b] = pick(up, x[i + b], got);
    }
  }
}

__device__ __forceinline__ float dot16(const float4 (&w)[4], const float4 (&x)[4]) {
  float a = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    a = fmaf(w[j].x, x[j].x, a);
    a = fmaf(w[j].y, x[j].y, a);
    a = fmaf(w[j].z, x[j].z, a);
    a = fmaf(w[j].w, x[j].w, a);
  }
  return a;
}

template <typename T>
__device__ __forceinline__ void eval_dot(const Geometry &g, const EvalArgs &A, int chain) {
  const T *f = reinterpret_cast<const T *>(A.field) + (size_t)chain * g.chain_elems;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t stride = (int64_t)A.nblk * kGcvThreads;
  double s = 0.0, Q = 0.0;
  if constexpr (sizeof(T) == 4) {
    const int64_t n512 = (int64_t)g.chain_elems / 512, n16 = (int64_t)g.chain_elems / 16;
    for (int64_t k = (int64_t)blockIdx.x * (kGcvThreads / 32) + (tid >> 5); k < n512;
         k += (int64_t)A.nblk * (kGcvThreads / 32)) {
      const float4 *x4 = reinterpret_cast<const float4 *>(f) + 128 * k + lane;
      const float4 *w4 = reinterpret_cast<const float4 *>(A.v) + 128 * k + lane;
      float4 x[4], w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = x4[32 * j];
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = __ldg(w4 + 32 * j);
      transpose_quads(x, lane);
      s += (double)dot16(w, x);
    }
    for (int64_t k = n512 * 32 + (int64_t)blockIdx.x * kGcvThreads + tid; k < n16; k += stride) {
      float4 w[4], x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[j] = reinterpret_cast<const float4 *>(f)[4 * k + j];
        w[j] = reinterpret_cast<const float4 *>(A.v)[4 * k + j];
      }
      s += (double)dot16(w, x);
    }
    for (int64_t e = n16 * 16 + (int64_t)blockIdx.x * kGcvThreads + tid;
         e < (int64_t)g.chain_elems; e += stride)
      s += (double)(A.v[e] * (float)f[e]);
  } else {
    for (int64_t e = (int64_t)blockIdx.x * kGcvThreads + tid; e < (int64_t)g.chain_elems;
         e += stride)
      s += (double)A.v[e] * (double)f[e];
  }
  for (int64_t i = (int64_t)blockIdx.x * kGcvThreads + tid; i < A.n_q; i += stride)
    Q += A.q[i] * (double)f[A.idx[i]];
  block_sum2(s, Q, A.partials + 2 * ((size_t)chain * A.nblk + blockIdx.x));
}

template <typename T>
__device__ __forceinline__ void eval_local(const Geometry &g, const EvalArgs &A, int chain, int pb,
                                           unsigned char *smem) {
  const T *f = reinterpret_cast<const T *>(A.field) + (size_t)chain * g.chain_elems;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  LocalSums<T> local(smem, kEvalWarps, kEvalCharges<T>, A.R, A.n_pts, A.kt);
  const LocalBox<T> box{f, g.colour_elems, g.Lx, g.Ly, g.Lz, g.W};
  const int64_t i0 = ((int64_t)pb * kEvalWarps + wid) * A.per;
  const int n = (int)max((int64_t)0, min((int64_t)A.per, A.n_q - i0));
  // lane j: site of charge i0 + j from its storage offset
  int sx = 0, sy = 0, sz = 0;
  double qq = 0.0;
  if (lane < n) {
    const uint32_t e = A.idx[i0 + lane], ce = (uint32_t)g.colour_elems;
    const int c = e >= ce ? 1 : 0;
    const uint32_t r = e - (c ? ce : 0u), row = r / (uint32_t)g.W;
    sz = (int)(row / (uint32_t)g.Ly);
    sy = (int)(row - (uint32_t)sz * (uint32_t)g.Ly);
    sx = 2 * (int)(r - row * (uint32_t)g.W) + ((c + sy + sz) & 1);
    const double qi = A.q[i0 + lane];
    qq = qi * qi * (double)f[e];
  }
  for (int j = 0; j < n; j += 2) {
    const int k = min(j + 1, n - 1);
    const int x0 = __shfl_sync(0xffffffffu, sx, j), x1 = __shfl_sync(0xffffffffu, sx, k);
    const int y0 = __shfl_sync(0xffffffffu, sy, j), y1 = __shfl_sync(0xffffffffu, sy, k);
    const int z0 = __shfl_sync(0xffffffffu, sz, j), z1 = __shfl_sync(0xffffffffu, sz, k);
    local.pair(box, box, x0, y0, z0, x1, y1, z1, j, k, lane);
  }
  const int each = 32 / A.per;
  const double w = local.sum(A.per, n, lane);
  double contrib = __shfl_sync(0xffffffffu, qq, lane / each) * w;
  if (lane % each != 0) contrib = 0.0;
  __shared__ double red[kEvalWarps];
  contrib = warp_sum(contrib);
  if (lane == 0) red[wid] = contrib;
  __syncthreads();
  if (tid == 0) {
    double sum = 0.0;
    for (int k = 0; k < kEvalWarps; ++k) sum += red[k];
    A.ppart[(size_t)chain * A.nblk_p + pb] = sum;
  }
}

// The local term by a warp per charge (direct_sum).
template <typename T>
__device__ __forceinline__ void eval_direct(const Geometry &g, const EvalArgs &A, int chain, int pb) {
  const T *f = reinterpret_cast<const T *>(A.field) + (size_t)chain * g.chain_elems;
  const LocalBox<T> box{f, g.colour_elems, g.Lx, g.Ly, g.Lz, g.W};
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t i = (int64_t)pb * kEvalWarps + wid;
  double contrib = 0.0;
  if (i < A.n_q) {
    const uint32_t e = A.idx[i], ce = (uint32_t)g.colour_elems;
    const int c = e >= ce ? 1 : 0;
    const uint32_t r = e - (c ? ce : 0u), row = r / (uint32_t)g.W;
    const int z = (int)(row / (uint32_t)g.Ly), y = (int)(row - (uint32_t)z * (uint32_t)g.Ly),
              x = 2 * (int)(r - row * (uint32_t)g.W) + ((c + y + z) & 1);
    const double qi = A.q[i];
    contrib = qi * qi * (double)f[e] * direct_sum(box, x, y, z, A.R, A.kt, lane);
  }
  __shared__ double red[kEvalWarps];
  if (lane == 0) red[wid] = contrib;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int k = 0; k < kEvalWarps; ++k) sum += red[k];
    A.ppart[(size_t)chain * A.nblk_p + pb] = sum;
  }
}

// (direct: five CTAs per SM, 48 registers; with four FP64 96^3 x 16, 200 charges,
// R = 2 takes 100 instead of 88 us, 128^3 x 2, R = 4 59 instead of 47)
template <typename T, bool DIRECT>
__global__ void __launch_bounds__(kGcvThreads, DIRECT ? 5 : 4)
    gcv_eval_kernel(const Geometry g, const EvalArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int pb = (int)blockIdx.x - A.nblk;
  if (pb < 0)
    eval_dot<T>(g, A, blockIdx.y);
  else if (DIRECT)
    eval_direct<T>(g, A, blockIdx.y, pb);
  else
    eval_local<T>(g, A, blockIdx.y, pb, smem);
}

template <typename T>
cudaError_t launch_eval(const Geometry &g, const EvalArgs &A, bool direct, cudaStream_t s) {
  const dim3 grid(A.nblk + A.nblk_p, g.n_chains);
  if (direct || A.nblk_p == 0) {
    gcv_eval_kernel<T, true><<<grid, kGcvThreads, 0, s>>>(g, A);
    return cudaGetLastError();
  }
  const size_t smem = local_bytes<T>(kEvalWarps, kEvalCharges<T>, A.R, A.n_pts);
  const cudaError_t e = raise_smem((const void *)gcv_eval_kernel<T, false>, smem);
  if (e != cudaSuccess) return e;
  gcv_eval_kernel<T, false><<<grid, kGcvThreads, smem, s>>>(g, A);
  return cudaGetLastError();
}

// warp per chain: fixed-order sums, then
// T g + T g^P = h~ . rho - Q s + cP - sum_i q_i^2 phi_i w_i
__global__ void gcv_finish_kernel(const double *__restrict__ partials, int nblk,
                                  const double *__restrict__ ppart, int nblk_p, int n_chains,
                                  const double *__restrict__ c0, double cP,
                                  double *__restrict__ tg) {
  const int chain = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (chain >= n_chains) return;
  double s = 0.0, Q = 0.0, p = 0.0;
  for (int b = lane; b < nblk; b += 32) {
    s += partials[2 * ((size_t)chain * nblk + b) + 0];
    Q += partials[2 * ((size_t)chain * nblk + b) + 1];
  }
  for (int b = lane; b < nblk_p; b += 32) p += ppart[(size_t)chain * nblk_p + b];
  s = warp_sum(s);
  Q = warp_sum(Q);
  p = warp_sum(p);
  if (lane == 0) tg[chain] = *c0 - Q * s + cP - p;
}

}  // namespace

// Sites of the cube of radius R and their neighbours, by row, then by parity of
// x: packed offsets from the corner of the (2R + 3)^3 box.
std::vector<int> gcv_points(int R) {
  const int d = 2 * R + 3;
  std::vector<int> out;
  for (int z = 0; z < d; ++z)
    for (int y = 0; y < d; ++y)
      for (int parity = 0; parity < 2; ++parity)
        for (int x = parity; x < d; x += 2) {
          const int faces = (x == 0 || x == d - 1) + (y == 0 || y == d - 1) + (z == 0 || z == d - 1);
          if (faces <= 1) out.push_back(x | y << 8 | z << 16);
        }
  return out;
}

// v . phi blocks of a chain: eight tiles each, at most 64; more where the
// chains alone would not fill the GPU (4 blocks on each of 152 SMs)
int gcv_blocks(const Geometry &g) {
  const int64_t tiles = std::max<int64_t>(1, (int64_t)g.chain_elems / kEvalTile);
  const int64_t b = std::min<int64_t>(64, (tiles + 7) / 8);
  return (int)std::max<int64_t>(b, std::min<int64_t>(tiles, 608 / g.n_chains));
}

cudaError_t gcv_solve(const Geometry &g, int64_t n_q, const int32_t *sites, const double *q,
                      double *rho_nat, double *u_nat, float *h32, float *v_layout,
                      double *scratch, int nblk_red, int n_iter, double *res,
                      const Allocator &alloc, cudaStream_t s) {
  const int64_t n = (int64_t)g.Lx * g.Ly * g.Lz;
  const int threads = 256;
  const int blocks = (int)((n + threads - 1) / threads > 4096 ? 4096 : (n + threads - 1) / threads);
  std::vector<SorBox> boxes{sor_box(g.Lx, g.Ly, g.Lz, 0, 0)};
  std::vector<SorCharge> charges;
  sor_charges(boxes[0], n_q, sites, q, charges);
  cudaError_t e = sor_solve(boxes, charges, n_iter, u_nat, rho_nat, alloc, s);
  if (e != cudaSuccess) return e;
  gcv_check_kernel<<<nblk_red, kGcvThreads, 0, s>>>(u_nat, rho_nat, g.Lx, g.Ly, g.Lz, scratch);
  gcv_check_sums_kernel<<<1, 32, 0, s>>>(scratch, nblk_red, res);
  double hres[3] = {0, 0, 0};
  if ((e = cudaMemcpyAsync(hres, res, sizeof(hres), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaStreamSynchronize(s)) != cudaSuccess)
    return e;
  // largest k with 13 max|u| 2^k < 2^24 (v = A h~ then fits 24 bits exactly)
  int k = 0;
  if (hres[2] > 0.0) {
    k = (int)std::floor(std::log2((16777216.0 - 1.0) / (13.0 * hres[2])));
    if (k > 60) k = 60;
    if (k < -60) k = -60;
  }
  const double scale = std::ldexp(1.0, k), inv_scale = std::ldexp(1.0, -k);
  gcv_quantize_kernel<<<nblk_red, kGcvThreads, 0, s>>>(u_nat, rho_nat, n, scale, inv_scale, h32,
                                                       scratch);
  gcv_c0_kernel<<<1, 32, 0, s>>>(scratch, nblk_red, res);
  if ((e = cudaMemsetAsync(v_layout, 0, sizeof(float) * g.chain_elems, s)) != cudaSuccess) return e;
  gcv_v_kernel<<<blocks, threads, 0, s>>>(h32, g, v_layout);
  return cudaGetLastError();
}

// Whether a warp takes one charge for itself (eval_direct).  What the shared
// neighbourhoods save, accesses to L1, counts only where there are charges enough to
// fill the GPU, and their shared memory leaves an SM few warps from R = 4 (FP32) or 2
// (FP64) on, also for v . phi.  Evaluation hot / cold, us, neighbourhoods against
// direct: 64^3 x 4, 200 charges, R = 2 14.5 / 19.1 against 12.4 / 16.0; 128^3 x 64,
// 1000 charges, R = 1 133 / 143 against 145 / 152, R = 4 604 / 612 against 388 / 393;
// FP64 96^3 x 16, 1000 charges, R = 4 409 / 416 against 258 / 261, R = 1, 4096 charges
// 126 / 135 against 158 / 160.
static bool gcv_direct(const Geometry &g, int R, int64_t n_q) {
  const int64_t n = n_q * g.n_chains;
  if (g.precision == COULPS_F32) return R >= 4 || n < ((int64_t)12000 << R);
  return R >= 2 || n < 10000;
}

cudaError_t gcv_eval(const Geometry &g, const void *field, const float *v_layout,
                     const uint32_t *idx, const double *q, int64_t n_q, double *partials,
                     int nblk, const double *c0, const float *kt, int R, double cP,
                     double *ppart, double *tg, cudaStream_t s) {
  EvalArgs A;
  A.field = field;
  A.v = v_layout;
  A.idx = idx;
  A.q = q;
  A.n_q = n_q;
  A.kt = kt;
  A.R = R;
  A.nblk = nblk;
  A.partials = partials;
  A.ppart = ppart;
  A.nblk_p = 0;
  A.per = 1;
  const int m = 2 * R + 1;
  A.n_pts = m * m * (m + 6);
  const bool direct = R > 0 && gcv_direct(g, R, n_q);
  if (R > 0 && n_q > 0) {
    // neighbourhoods: as many charges a warp as leave 32 warps for each of 152 SMs (evaluation of
    // 128^3 x 4 chains, 4096 charges, 16 / 32 / 64 warps: 39.6 / 37.5 / 47.7 us; 40^3 x
    // 64, 500 charges 39.6 / 43.7 / 47.7)
    const int most = g.precision == COULPS_F32 ? kEvalCharges<float> : kEvalCharges<double>;
    while (!direct && 2 * A.per <= most && n_q * g.n_chains / (2 * A.per) >= 32 * 152) A.per *= 2;
    const int per_block = A.per * (kGcvThreads / 32);
    A.nblk_p = (int)((n_q + per_block - 1) / per_block);
  }
  const cudaError_t e = g.precision == COULPS_F32 ? launch_eval<float>(g, A, direct, s)
                                                  : launch_eval<double>(g, A, direct, s);
  if (e != cudaSuccess) return e;
  gcv_finish_kernel<<<(g.n_chains + 7) / 8, 256, 0, s>>>(partials, nblk, ppart, A.nblk_p,
                                                        g.n_chains, c0, A.nblk_p > 0 ? cP : 0.0,
                                                        tg);
  return cudaGetLastError();
}

}  // namespace coulps
