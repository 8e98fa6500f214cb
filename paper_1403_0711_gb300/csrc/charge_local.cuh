// The local term's sums over charge neighbourhoods, w_i = sum_d k(d) (A phi)(r_i + d)
// over the cube of radius R around charge i inside its box, shared by the global
// control variate of a lattice and of a batch.
//
// A warp takes up to `per` charges, two at a time: it loads the cube's sites and
// their neighbours once each (gcv_points: sorted by row and colour, a cache line
// access for each such pair; seven loads per point of the cube made three times as
// many, and these are what a kernel of them spends its time on), then lane t
// computes k(d) (A phi)(r_i + d) for points t, t + 32, ... of the cube, in the
// field's precision, and leaves its share in shared memory; then 32 / per lanes add
// each charge's shares in FP64 (a butterfly sum per charge was six FP64-unit
// instructions a charge, one lane per charge 54 a warp, and that unit has two lanes
// per clock).
#pragma once

#include "device_common.cuh"

namespace coulps {

// a chain's (system's) field: colour 0 at f, colour 1 ce elements on
template <typename T>
struct LocalBox {
  const T *f;
  size_t ce;
  int Lx, Ly, Lz, W;
};

// phi at a site, 0 outside the box
template <typename T>
__device__ __forceinline__ T box_phi(const LocalBox<T> &b, int x, int y, int z) {
  if ((unsigned)x >= (unsigned)b.Lx || (unsigned)y >= (unsigned)b.Ly || (unsigned)z >= (unsigned)b.Lz)
    return T(0);
  return b.f[((x + y + z) & 1 ? b.ce : (size_t)0) + ((size_t)z * b.Ly + y) * b.W + (x >> 1)];
}

// w of the charge at (x, y, z) in every lane, by a warp for itself: lane t takes the
// points t, t + 32, .. of the cube and loads each with its six neighbours.  No shared
// memory and no charge waits for another: for few charges, and for FP64 and cubes so
// large that their neighbourhoods leave an SM few warps.
template <typename T>
__device__ __forceinline__ double direct_sum(const LocalBox<T> &b, int x, int y, int z, int R,
                                             const float *kt, int lane) {
  const int m = 2 * R + 1, m3 = m * m * m;
  T w = T(0);
  for (int t = lane; t < m3; t += 32) {
    const int xx = x + t % m - R, yy = y + (t / m) % m - R, zz = z + t / (m * m) - R;
    if ((unsigned)xx >= (unsigned)b.Lx || (unsigned)yy >= (unsigned)b.Ly ||
        (unsigned)zz >= (unsigned)b.Lz)
      continue;
    const T Ap = T(6) * box_phi(b, xx, yy, zz) - box_phi(b, xx - 1, yy, zz) -
                 box_phi(b, xx + 1, yy, zz) - box_phi(b, xx, yy - 1, zz) -
                 box_phi(b, xx, yy + 1, zz) - box_phi(b, xx, yy, zz - 1) -
                 box_phi(b, xx, yy, zz + 1);
    w += (T)__ldg(kt + t) * Ap;
  }
  return warp_sum((double)w);
}

// Shared memory of a CTA of `warps` warps with at most `charges` charges a warp:
// per warp the neighbourhoods of two charges ((2R + 3)^3 each) and the lanes'
// shares [charge][33], then the cube's points (offsets in such a neighbourhood),
// the kernel's values and the neighbourhood's points.
template <typename T>
__host__ __device__ __forceinline__ size_t local_bytes(int warps, int charges, int R, int n_pts) {
  const int m = 2 * R + 1;
  return warps * (2 * (m + 2) * (m + 2) * (m + 2) + charges * 33) * sizeof(T) +
         4 * (size_t)(2 * m * m * m + n_pts);
}

template <typename T>
struct LocalSums {
  int R, n_pts;
  T *near, *share;  // this warp's
  int *pt, *all;
  float *kv;

  // Every thread of the CTA; ends with a barrier.  kt: kernel values, then points.
  __device__ __forceinline__ LocalSums(unsigned char *smem, int warps, int charges, int R_,
                                       int n_pts_, const float *kt)
      : R(R_), n_pts(n_pts_) {
    const int m = 2 * R + 1, m3 = m * m * m, d = m + 2, own = 2 * d * d * d + charges * 33;
    near = reinterpret_cast<T *>(smem) + (threadIdx.x >> 5) * own;
    share = near + 2 * d * d * d;
    pt = reinterpret_cast<int *>(reinterpret_cast<T *>(smem) + warps * own);
    kv = reinterpret_cast<float *>(pt + m3);
    all = reinterpret_cast<int *>(kv + m3);
    for (int t = threadIdx.x; t < m3; t += blockDim.x) {
      pt[t] = (t % m + 1) + ((t / m) % m + 1) * d + (t / (m * m) + 1) * d * d;
      kv[t] = kt[t];
    }
    for (int t = threadIdx.x; t < n_pts; t += blockDim.x)
      all[t] = reinterpret_cast<const int *>(kt + m3)[t];
    __syncthreads();
  }

  // phi at a point of the neighbourhood (packed offsets from its corner x, y, z),
  // 0 outside the box
  __device__ __forceinline__ T phi(const LocalBox<T> &b, int x, int y, int z, int o) const {
    const int xx = x + (o & 255), yy = y + ((o >> 8) & 255), zz = z + (o >> 16);
    const bool in = (unsigned)xx < (unsigned)b.Lx && (unsigned)yy < (unsigned)b.Ly &&
                    (unsigned)zz < (unsigned)b.Lz;
    const size_t at = ((xx + yy + zz) & 1 ? b.ce : (size_t)0) +
                      ((size_t)zz * b.Ly + yy) * b.W + (xx >> 1);
    return in ? b.f[at] : T(0);
  }

  __device__ __forceinline__ void shares(const LocalBox<T> &b, int x, int y, int z, const T *v,
                                         T *out, int lane) const {
    const int m = 2 * R + 1, m3 = m * m * m, d = m + 2;
    T wl = T(0);
    for (int t = lane; t < m3; t += 32) {
      const int dx = t % m, dy = (t / m) % m, dz = t / (m * m);
      const T *c = v + pt[t];
      const T Ap = T(6) * c[0] - c[-1] - c[1] - c[-d] - c[d] - c[-d * d] - c[d * d];
      if ((unsigned)(x - R + dx) < (unsigned)b.Lx && (unsigned)(y - R + dy) < (unsigned)b.Ly &&
          (unsigned)(z - R + dz) < (unsigned)b.Lz)
        wl += (T)kv[t] * Ap;
    }
    out[lane] = wl;
  }

  // The warp's charges j and k (k == j: one) at these sites.
  __device__ __forceinline__ void pair(const LocalBox<T> &b0, const LocalBox<T> &b1, int x0, int y0,
                                       int z0, int x1, int y1, int z1, int j, int k, int lane) {
    const int R1 = R + 1, d = 2 * R + 3, d3 = d * d * d;
#pragma unroll 3
    for (int t = lane; t < n_pts; t += 32) {
      const int o = all[t], at = (o & 255) + ((o >> 8) & 255) * d + (o >> 16) * d * d;
      const T p0 = phi(b0, x0 - R1, y0 - R1, z0 - R1, o);
      const T p1 = k > j ? phi(b1, x1 - R1, y1 - R1, z1 - R1, o) : T(0);
      near[at] = p0;
      near[d3 + at] = p1;
    }
    __syncwarp();
    shares(b0, x0, y0, z0, near, share + j * 33, lane);
    if (k > j) shares(b1, x1, y1, z1, near + d3, share + k * 33, lane);
    __syncwarp();
  }

  // w of charge lane / (32 / per) in each of its lanes (per: a power of two, n
  // charges made)
  __device__ __forceinline__ double sum(int per, int n, int lane) const {
    const int m = 2 * R + 1, m3 = m * m * m, each = 32 / per, j = lane / each;
    double w = 0.0;
    if (j < n)
      for (int l = lane % each, k = min(32, m3); l < k; l += each) w += (double)share[j * 33 + l];
    for (int o = each >> 1; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    return w;
  }
};

}  // namespace coulps
