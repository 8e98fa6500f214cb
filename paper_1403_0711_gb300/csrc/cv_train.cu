// Training kernels of the localized learned control variate: the memory-bound
// steps between the convolutions and the batched products of the divergence.
//
// The gradients pass through BF16 roundings (dh and da, where the convolutions
// take them), and a sum formed in another order moves values across them: the
// whole pass on tensor-core contractions was 14 times as fast as the framework
// operations and as close to FP64, but its gradients were 1e-4 away from
// theirs.  So these kernels keep every rounding and every order of addition of
// the operations that they stand for, and are bitwise them.
//
//   pack_weights  the convolutions' packed BF16 weights from FP32 weights in
//                 device memory (through the host each of a pass's eight cost a
//                 copy in either direction and a wait)
//   act           a = tanh h (BF16) and s = 1 - a^2 (rounded to BF16, held in
//                 FP32), and their backward dh = ((da - ds a) - ds a) (1 - a^2)
//   gather        the 27 neighbours of the sites next to R in the layout of the
//                 batched product, left[m][n][16 c + ...][27 e]: the framework's
//                 27 gathers, their concatenation and a transposing copy
//   scatter       its transpose: every site's up to 27 contributions added in
//                 the order o = 26 .. 0 in which the 27 gathers' backwards run
//
// Measured, a whole pass on 256 samples of 14^3 (R = 8^3): 16.5 -> 7.2 ms.
#include <algorithm>
#include <cstdint>

#include <cuda_bf16.h>

#include "device_common.cuh"
#include "internal.h"

namespace coulps {
namespace {

constexpr int kTrThreads = 256;

// w[16][16][27] -> 27 blocks of 256 BF16 in the tensor core's order (see
// coulps_cv_pack_weights)
__global__ void cv_pack_weights_kernel(const float *__restrict__ w,
                                       __nv_bfloat16 *__restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 27 * 256) return;
  const int o = i >> 8, co = (i >> 4) & 15, ci = i & 15;
  out[o * 256 + (co / 8) * 64 + (ci / 8) * 128 + (co % 8) * 8 + ci % 8] =
      __float2bfloat16_rn(w[(co * 16 + ci) * 27 + o]);
}

// 4 values per thread.  The framework's operations round after each step: the
// products and differences here must not contract into fma, where theirs do not.
__global__ void __launch_bounds__(kTrThreads)
    cv_act_forward_kernel(const float4 *__restrict__ h, uint2 *__restrict__ a,
                          float4 *__restrict__ s, int64_t n4) {
  const int64_t i = (int64_t)blockIdx.x * kTrThreads + threadIdx.x;
  if (i >= n4) return;
  const float4 v = h[i];
  const float x[4] = {v.x, v.y, v.z, v.w};
  __align__(8) __nv_bfloat16 ta[4];
  float ts[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float t = tanhf(x[k]);
    ta[k] = __float2bfloat16_rn(t);
    ts[k] = __bfloat162float(__float2bfloat16_rn(__fsub_rn(1.f, __fmul_rn(t, t))));
  }
  a[i] = *reinterpret_cast<const uint2 *>(ta);
  s[i] = make_float4(ts[0], ts[1], ts[2], ts[3]);
}

// dh from h, da (BF16) and ds (either may be null: no gradient)
__global__ void __launch_bounds__(kTrThreads)
    cv_act_backward_kernel(const float4 *__restrict__ h, const uint2 *__restrict__ da,
                           const float4 *__restrict__ ds, float4 *__restrict__ dh, int64_t n4) {
  const int64_t i = (int64_t)blockIdx.x * kTrThreads + threadIdx.x;
  if (i >= n4) return;
  const float4 v = h[i];
  const float x[4] = {v.x, v.y, v.z, v.w};
  float d[4] = {0.f, 0.f, 0.f, 0.f}, g[4];
  if (ds) {
    const float4 w = ds[i];
    d[0] = w.x; d[1] = w.y; d[2] = w.z; d[3] = w.w;
  }
  __align__(8) __nv_bfloat16 b[4];
  *reinterpret_cast<uint2 *>(b) = da ? da[i] : make_uint2(0, 0);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float t = tanhf(x[k]);
    const float p = __fmul_rn(-d[k], t);
    const float tot = __fadd_rn(__fadd_rn(__bfloat162float(b[k]), p), p);
    g[k] = __fmul_rn(tot, fmaf(-t, t, 1.f));
  }
  dh[i] = make_float4(g[0], g[1], g[2], g[3]);
}

struct RegionBox {
  int nb, ex, ey, ez;        // samples [n][z][y][x][16]
  int x0, y0, z0, nx, ny, nz;  // sites q: a box of E
};

// left[q][n][c][e] = s[n][q + e][c], 0 outside E.  One CTA: one q, 8 samples,
// turned from site rows to [c][e] rows in shared memory.
constexpr int kGaN = 8;
__global__ void __launch_bounds__(kTrThreads)
    cv_gather_kernel(const float4 *__restrict__ s, const RegionBox r, float *__restrict__ left) {
  __shared__ __align__(16) float buf[kGaN][432];
  const int q = blockIdx.x, n0 = blockIdx.y * kGaN;
  const int nn = min(kGaN, r.nb - n0);
  const int x = r.x0 + q % r.nx, y = r.y0 + q / r.nx % r.ny, z = r.z0 + q / (r.nx * r.ny);
  for (int i = threadIdx.x; i < nn * 108; i += kTrThreads) {
    const int c4 = i & 3, e = (i >> 2) % 27, n = i / 108;
    const int xx = x + e % 3 - 1, yy = y + e / 3 % 3 - 1, zz = z + e / 9 - 1;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (xx >= 0 && yy >= 0 && zz >= 0 && xx < r.ex && yy < r.ey && zz < r.ez)
      v = __ldg(s + ((((int64_t)(n0 + n) * r.ez + zz) * r.ey + yy) * r.ex + xx) * 4 + c4);
    buf[n][(4 * c4) * 27 + e] = v.x;
    buf[n][(4 * c4 + 1) * 27 + e] = v.y;
    buf[n][(4 * c4 + 2) * 27 + e] = v.z;
    buf[n][(4 * c4 + 3) * 27 + e] = v.w;
  }
  __syncthreads();
  float4 *out = reinterpret_cast<float4 *>(left + ((int64_t)q * r.nb + n0) * 432);
  const float4 *src = reinterpret_cast<const float4 *>(&buf[0][0]);
  for (int i = threadIdx.x; i < nn * 108; i += kTrThreads) __stcs(out + i, src[i]);
}

// ds[n][p][c] = sum over o = 26 .. 0 of dleft[p - o][n][c][o].  In o's descending
// order p - o ascends in (z, y, x), so a CTA, one sample and nc channels, runs
// through the q in order and adds each one's 27 nc values to its sums of the
// sites p = q + o in shared memory; thread (c, o) holds the next kScAhead values
// in registers, as the loop's own steps are only a barrier apart.
constexpr int kScAhead = 8;
__global__ void cv_scatter_kernel(const float *__restrict__ dleft, const RegionBox r, int nc,
                                  float *__restrict__ ds) {
  extern __shared__ float acc[];  // [site of the box grown by one][c]
  const int n = blockIdx.x, c0 = blockIdx.y * nc;
  const int px0 = max(r.x0 - 1, 0), py0 = max(r.y0 - 1, 0), pz0 = max(r.z0 - 1, 0);
  const int pnx = min(r.x0 + r.nx + 1, r.ex) - px0, pny = min(r.y0 + r.ny + 1, r.ey) - py0,
            pnz = min(r.z0 + r.nz + 1, r.ez) - pz0;
  const int np = pnx * pny * pnz, nq = r.nx * r.ny * r.nz;
  for (int i = threadIdx.x; i < np * nc; i += blockDim.x) acc[i] = 0.f;
  const int t = threadIdx.x, c = t / 27, o = t % 27;
  const bool on = t < 27 * nc;
  const int dx = o % 3 - 1, dy = o / 3 % 3 - 1, dz = o / 9 - 1;
  const float *src = dleft + (int64_t)n * 432 + c0 * 27 + t;
  const int64_t step = (int64_t)r.nb * 432;
  float v[kScAhead];
#pragma unroll
  for (int k = 0; k < kScAhead; ++k) v[k] = on && k < nq ? __ldcs(src + k * step) : 0.f;
  int x = r.x0, y = r.y0, z = r.z0;
  __syncthreads();
  for (int q0 = 0; q0 < nq; q0 += kScAhead) {
#pragma unroll
    for (int k = 0; k < kScAhead; ++k) {
      const int q = q0 + k;
      if (q < nq) {  // the same for every thread
        const int xx = x + dx - px0, yy = y + dy - py0, zz = z + dz - pz0;
        if (on && xx >= 0 && yy >= 0 && zz >= 0 && xx < pnx && yy < pny && zz < pnz) {
          float *at = acc + ((zz * pny + yy) * pnx + xx) * nc + c;
          *at = __fadd_rn(*at, v[k]);
        }
        const int qn = q + kScAhead;
        v[k] = on && qn < nq ? __ldcs(src + qn * step) : 0.f;
        if (++x == r.x0 + r.nx) {
          x = r.x0;
          if (++y == r.y0 + r.ny) {
            y = r.y0;
            ++z;
          }
        }
        __syncthreads();
      }
    }
  }
  for (int i = t; i < r.ex * r.ey * r.ez * nc; i += blockDim.x) {
    const int cc = i % nc, s = i / nc;
    const int xx = s % r.ex - px0, yy = s / r.ex % r.ey - py0, zz = s / (r.ex * r.ey) - pz0;
    const bool in = xx >= 0 && yy >= 0 && zz >= 0 && xx < pnx && yy < pny && zz < pnz;
    ds[((int64_t)n * r.ex * r.ey * r.ez + s) * 16 + c0 + cc] =
        in ? acc[((zz * pny + yy) * pnx + xx) * nc + cc] : 0.f;
  }
}

bool region_box(int nb, const int32_t *e, const int32_t *lo, const int32_t *hi, RegionBox *r) {
  if (nb < 1 || !e || !lo || !hi) return false;
  for (int k = 0; k < 3; ++k)
    if (e[k] < 1 || lo[k] < 0 || hi[k] > e[k] || lo[k] >= hi[k]) return false;
  if ((int64_t)e[0] * e[1] * e[2] > 0x7fffffff / 16) return false;
  *r = RegionBox{nb, e[0], e[1], e[2], lo[0], lo[1], lo[2], hi[0] - lo[0], hi[1] - lo[1],
                 hi[2] - lo[2]};
  return true;
}

// Channels per CTA of the scatter: the most of 8, 4, 2, 1 whose sums fit shared
// memory twice per SM (8 where they do: 55 KB for 12^3 sites), else once.
int scatter_channels(const RegionBox &r) {
  const int64_t np = (int64_t)(r.nx + 2) * (r.ny + 2) * (r.nz + 2);
  for (int nc = 8; nc >= 1; nc /= 2)
    if (np * nc * 4 <= (nc == 1 ? 220 : 110) * 1024) return nc;
  return 0;
}

}  // namespace
}  // namespace coulps

using namespace coulps;

extern "C" {

int coulps_cv_pack_weights_dev(const float *w, void *out_bf16, void *stream) {
  if (!w || !out_bf16) return COULPS_EINVAL;
  cv_pack_weights_kernel<<<27, 256, 0, (cudaStream_t)stream>>>(
      w, reinterpret_cast<__nv_bfloat16 *>(out_bf16));
  return cudaGetLastError() == cudaSuccess ? COULPS_OK : COULPS_ECUDA;
}

int coulps_cv_act_forward(const float *h, void *a_bf16, float *s, int64_t n, void *stream) {
  if (!h || !a_bf16 || !s || n < 0 || n % 4) return COULPS_EINVAL;
  if (((reinterpret_cast<uintptr_t>(h) | reinterpret_cast<uintptr_t>(s)) & 15) ||
      (reinterpret_cast<uintptr_t>(a_bf16) & 7))
    return COULPS_EINVAL;
  if (n == 0) return COULPS_OK;
  cv_act_forward_kernel<<<(unsigned)((n / 4 + kTrThreads - 1) / kTrThreads), kTrThreads, 0,
                          (cudaStream_t)stream>>>(
      reinterpret_cast<const float4 *>(h), reinterpret_cast<uint2 *>(a_bf16),
      reinterpret_cast<float4 *>(s), n / 4);
  return cudaGetLastError() == cudaSuccess ? COULPS_OK : COULPS_ECUDA;
}

int coulps_cv_act_backward(const float *h, const void *da_bf16, const float *ds, float *dh,
                           int64_t n, void *stream) {
  if (!h || !dh || n < 0 || n % 4) return COULPS_EINVAL;
  if (((reinterpret_cast<uintptr_t>(h) | reinterpret_cast<uintptr_t>(ds) |
        reinterpret_cast<uintptr_t>(dh)) & 15) ||
      (reinterpret_cast<uintptr_t>(da_bf16) & 7))
    return COULPS_EINVAL;
  if (n == 0) return COULPS_OK;
  cv_act_backward_kernel<<<(unsigned)((n / 4 + kTrThreads - 1) / kTrThreads), kTrThreads, 0,
                           (cudaStream_t)stream>>>(
      reinterpret_cast<const float4 *>(h), reinterpret_cast<const uint2 *>(da_bf16),
      reinterpret_cast<const float4 *>(ds), reinterpret_cast<float4 *>(dh), n / 4);
  return cudaGetLastError() == cudaSuccess ? COULPS_OK : COULPS_ECUDA;
}

int coulps_cv_region_gather(const float *s, float *left, int nb, const int32_t *e,
                            const int32_t *lo, const int32_t *hi, void *stream) {
  RegionBox r;
  if (!s || !left || !region_box(nb, e, lo, hi, &r)) return COULPS_EINVAL;
  if ((reinterpret_cast<uintptr_t>(s) | reinterpret_cast<uintptr_t>(left)) & 15)
    return COULPS_EINVAL;
  if ((nb + kGaN - 1) / kGaN > 65535) return COULPS_EINVAL;
  cv_gather_kernel<<<dim3(r.nx * r.ny * r.nz, (nb + kGaN - 1) / kGaN), kTrThreads, 0,
                     (cudaStream_t)stream>>>(reinterpret_cast<const float4 *>(s), r, left);
  return cudaGetLastError() == cudaSuccess ? COULPS_OK : COULPS_ECUDA;
}

int coulps_cv_region_scatter(const float *dleft, float *ds, int nb, const int32_t *e,
                             const int32_t *lo, const int32_t *hi, void *stream) {
  RegionBox r;
  if (!dleft || !ds || !region_box(nb, e, lo, hi, &r)) return COULPS_EINVAL;
  const int nc = scatter_channels(r);
  if (nc == 0) return COULPS_EUNSUPPORTED;
  const int smem = (r.nx + 2) * (r.ny + 2) * (r.nz + 2) * nc * 4;
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(cv_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           224 * 1024) != cudaSuccess) {
    cudaGetLastError();
    return COULPS_ECUDA;
  }
  cv_scatter_kernel<<<dim3(nb, 16 / nc), (27 * nc + 31) / 32 * 32, smem, (cudaStream_t)stream>>>(
      dleft, r, nc, ds);
  return cudaGetLastError() == cudaSuccess ? COULPS_OK : COULPS_ECUDA;
}

}  // extern "C"
