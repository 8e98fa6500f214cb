// What the fused pass and the pass pair do with one quad (four consecutive
// sites of one colour in a row): load, store, update and masking, in packed
// pairs.
#pragma once

#include "device_common.cuh"
#include "tile_march.cuh"

namespace coulps {
namespace tile {

template <typename T>
__device__ __forceinline__ Quad<T> qzero() {
  Quad<T> q;
  q.a = pset(T(0));
  q.b = pset(T(0));
  return q;
}

template <typename T>
__device__ __forceinline__ Quad<T> qload(const T *p);
template <>
__device__ __forceinline__ Quad<float> qload<float>(const float *p) {
  const float4 f = *reinterpret_cast<const float4 *>(p);
  Quad<float> q;
  q.a = make_float2(f.x, f.y);
  q.b = make_float2(f.z, f.w);
  return q;
}
template <>
__device__ __forceinline__ Quad<double> qload<double>(const double *p) {
  Quad<double> q;
  q.a = reinterpret_cast<const double2 *>(p)[0];
  q.b = reinterpret_cast<const double2 *>(p)[1];
  return q;
}

template <typename T>
__device__ __forceinline__ void qstore(T *p, const Quad<T> &q);
template <>
__device__ __forceinline__ void qstore<float>(float *p, const Quad<float> &q) {
  *reinterpret_cast<float4 *>(p) = make_float4(q.a.x, q.a.y, q.b.x, q.b.y);
}
template <>
__device__ __forceinline__ void qstore<double>(double *p, const Quad<double> &q) {
  reinterpret_cast<double2 *>(p)[0] = q.a;
  reinterpret_cast<double2 *>(p)[1] = q.b;
}

// The heatbath deviates of two quads (two stages' Philox words): FP32 as
// four packed pairs with one branch per thread for the rare tail words; FP64
// word by word.
template <typename T> struct StageNoise;
template <> struct StageNoise<float> {
  __device__ __forceinline__ static void of(uint4 wa, uint4 wb, Quad<float> &na,
                                            Quad<float> &nb) {
    const uint32_t w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
    float2 o[4];
    hb_noise_pairs_f32<4>(w, o);
    na.a = o[0];
    na.b = o[1];
    nb.a = o[2];
    nb.b = o[3];
  }
};
template <> struct StageNoise<double> {
  __device__ __forceinline__ static void of(uint4 wa, uint4 wb, Quad<double> &na,
                                            Quad<double> &nb) {
    na.a = make_double2(hb_noise_f64(wa.x), hb_noise_f64(wa.y));
    na.b = make_double2(hb_noise_f64(wa.z), hb_noise_f64(wa.w));
    nb.a = make_double2(hb_noise_f64(wb.x), hb_noise_f64(wb.y));
    nb.b = make_double2(hb_noise_f64(wb.z), hb_noise_f64(wb.w));
  }
};

// The new values of a quad.  zm, zp: the other colour's quad on planes
// z -+ 1; ym, yp: rows y -+ 1; c: same row and plane; e: the x neighbour
// outside c (the previous quad's last site for an even row, the next quad's
// first for an odd row; 0 beyond the box); r: the site's value before the
// pass (over-relaxation) or the heatbath deviates.  Sums in the order of the
// half-sweep kernel: S = ((zm + zp) + (ym + yp)) + (c + xs), then
// S/3 - old or S/6 + deviate by one fma.
template <typename T, bool OR>
__device__ __forceinline__ Quad<T> update(const Quad<T> &zm, const Quad<T> &zp, const Quad<T> &ym,
                                          const Quad<T> &yp, const Quad<T> &c, bool odd, T e,
                                          const Quad<T> &r) {
  using P2 = typename Pair2<T>::type;
  P2 xa, xb;
  xa.x = odd ? c.a.y : e;
  xa.y = odd ? c.b.x : c.a.x;
  xb.x = odd ? c.b.y : c.a.y;
  xb.y = odd ? e : c.b.x;
  Quad<T> S, v;
  S.a = padd(padd(padd(zm.a, zp.a), padd(ym.a, yp.a)), padd(c.a, xa));
  S.b = padd(padd(padd(zm.b, zp.b), padd(ym.b, yp.b)), padd(c.b, xb));
  if (OR) {
    const P2 third = pset(Coef<T>::third);
    v.a = pfma(S.a, third, pneg2(r.a));
    v.b = pfma(S.b, third, pneg2(r.b));
  } else {
    const P2 sixth = pset(Coef<T>::sixth);
    v.a = pfma(S.a, sixth, r.a);
    v.b = pfma(S.b, sixth, r.b);
  }
  return v;
}

// Zero what is not a site of the box: the whole quad when `valid` is false
// (a ghost row or plane), else the lanes past x = Lx - 1 (bit i of pm: site i
// of the quad).
template <typename T>
__device__ __forceinline__ void mask(Quad<T> &v, bool valid, uint32_t pm) {
  if (!valid) v = qzero<T>();
  if (pm) {
    if (pm & 1u) v.a.x = T(0);
    if (pm & 2u) v.a.y = T(0);
    if (pm & 4u) v.b.x = T(0);
    if (pm & 8u) v.b.y = T(0);
  }
}

}  // namespace tile
}  // namespace coulps
