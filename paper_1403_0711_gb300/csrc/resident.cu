// Resident sweeps of small lattices: one thread-block cluster holds a whole
// chain in its CTAs' shared memory and runs any number of compound sweeps (and
// their samples) in one launch.
//
// What this replaces: the z-march kernels read and write the field once per
// launch, and a compound sweep is 4 to 6 launches.  A chain of 1e5 sites is
// then bound by launches and their tails, not by its work.
//
// Work split.  CTA r of the cluster's C owns planes [z0, z1), both colours, in
// shared memory, with a halo plane at either end and a row of zeros above and
// below every plane (the phi = 0 ghosts).  Within a half-sweep a thread owns V
// same-colour sites of a row (FP32: a quad, one Philox call; FP64: one site,
// so that the few FP64 lanes of every scheduler are fed even by a 16^3 box)
// and marches a short run of planes, keeping planes z - 1, z, z + 1 of the
// other colour in registers.  A thread that writes the first or last plane of
// its CTA also stores it into the neighbour's halo (distributed shared
// memory), and one cluster barrier ends the half-sweep: it makes the halos
// visible and says that the neighbours no longer read what the next half-sweep
// overwrites.  The deviates of a thread's first run do not depend on the field
// and are formed between the barrier's arrive and wait.
//
// Samples.  kMeasWarps further warps per CTA form Q and P while the others
// sweep: colour 0's charges during the sweep's last half-sweep (which writes
// colour 1), colour 1's during the next sweep's first; the sums go to CTA 0,
// whose last warp adds them in a fixed order one half-sweep later and records
// the sample another one later.  So a measured sweep costs no extra barrier
// (only the last one of a launch does) and each of these chains of dependent
// FP64 instructions has a half-sweep to itself.
//
// The arithmetic per site is that of the half-sweep kernel (the same sums in
// the same order, the same fma, Philox words and deviates), so fields are
// bitwise those of the march kernels.
//
// Every wait here is a hardware barrier of the cluster or the block; every
// CTA of a cluster runs the same number of them.
//
// What bounds it: with few groups per thread the barrier and the latency
// between two (0.5 us per half-sweep with a cluster); in FP32 with many, shared
// memory (5 16-byte loads and a store per quad and reflection) and the draw's
// instructions; in FP64 the FP64 instructions.  Measured, us per measured
// compound sweep, march kernels -> this one: FP64 16^3 x 1 heatbath only 38.6
// -> 2.7 (85 with the earlier deviate); 1:3: FP32 16^3 x 1 31 -> 4.7, 61 x 47 x
// 53 x 12 45 -> 22, 64^3 x 64 163 -> 112; FP64 32^3 x 1 112 -> 28.  Forms tried on
// the way (FP64 16^3, heatbath only): one form of sweep, the sample recorded
// from cross-warp sums by one thread 5.2; statistics in registers and deviates
// by warps of their own 3.9; recorder and gather warps apart 2.7.
#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "tile_march.cuh"

namespace coulps {
namespace {

using namespace tile;

constexpr int kMeasWarps = 4;    // the last one records
constexpr int kGatherWarps = 3;  // at most, the others gather
constexpr int kMeasThreads = 32 * kMeasWarps;
constexpr int kMaxSweepThreads = 512;
constexpr int kResEntries = 4;  // charges a measuring thread keeps in registers
// "Single" form: every sweeping thread has one group of V sites for the whole
// launch (CTAs of at most kSingleThreads groups per colour).
constexpr int kSingleThreads = 256;

// Shared memory: partial sums [CTA][measuring warp][2] (used in CTA 0), the
// chain's batch sums and the load's mbarrier, then (single form) the deviates of the next heatbath
// half-sweep by colour, then the planes.
constexpr int kResParts = kMaxCluster * kGatherWarps;
constexpr int kResBar = (2 * kResParts + kStatStride) * 8;
constexpr int kResHeaderBytes = (kResBar + 8 + 127) / 128 * 128;
constexpr int kResDrawBytes = 2 * kSingleThreads * 16;  // 2 colours x 4 floats (or 1 double)

// Plane copies by the TMA unit (16-byte aligned addresses and sizes: a row is a
// multiple of 16 bytes).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_store(void *dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
               :: "l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store_wait() {
  asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// (the warp's lanes may have diverged: the barriers are of whole warps)
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of shared-memory address `a` in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t a, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
  return d;
}
__device__ __forceinline__ void st_remote(uint32_t a, const float (&v)[4]) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3])
               : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, const double (&v)[1]) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v[0]) : "memory");
}

template <typename T, int V> struct Group;
template <> struct Group<float, 4> {
  __device__ __forceinline__ static void ld(const float *p, float (&v)[4]) { ld_quad(p, v); }
  __device__ __forceinline__ static void st(float *p, const float (&v)[4]) { st_quad(p, v); }
};
template <> struct Group<double, 1> {
  __device__ __forceinline__ static void ld(const double *p, double (&v)[1]) { v[0] = *p; }
  __device__ __forceinline__ static void st(double *p, const double (&v)[1]) { *p = v[0]; }
};

// S / 6 + deviate or S / 3 - old of V sites, from the other colour's M, C, P
// (planes z - 1, z, z + 1), ym, yp and the x neighbour e beyond C.
__device__ __forceinline__ void neighbour_sum(const float (&M)[4], const float (&C)[4],
                                              const float (&P)[4], const float (&ym)[4],
                                              const float (&yp)[4], float e, bool odd,
                                              float2 (&S)[2]) {
  float xs[4];
  x_neighbours(odd, e, C, xs);
#pragma unroll
  for (int h = 0; h < 2; ++h)
    S[h] = padd(padd(padd(pair_of(M, h), pair_of(P, h)), padd(pair_of(ym, h), pair_of(yp, h))),
                padd(pair_of(C, h), pair_of(xs, h)));
}
__device__ __forceinline__ void update(const float2 (&S)[2], float coef, const float (&add)[4],
                                       float (&u)[4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 r = pfma(S[h], pset(coef), pair_of(add, h));
    u[2 * h] = r.x;
    u[2 * h + 1] = r.y;
  }
}

template <int V> struct Draw;
template <> struct Draw<4> {
  __device__ __forceinline__ static void of(uint4 w, int, float (&n)[4]) {
    float2 p[2];
    QuadNoise2<float>::of(w, p);
    n[0] = p[0].x; n[1] = p[0].y; n[2] = p[1].x; n[3] = p[1].y;
  }
};
template <> struct Draw<1> {
  __device__ __forceinline__ static void of(uint4 w, int h, double (&n)[1]) {
    const int k = h & 3;
    n[0] = hb_noise_f64(k == 0 ? w.x : (k == 1 ? w.y : (k == 2 ? w.z : w.w)));
  }
};

// A sample's sums, here and in resident_sample_kernel: the same order, and
// explicit roundings, so that a contraction does not depend on the kernel.
__device__ __forceinline__ void add_charge(double q, double phi, double &sq, double &sp) {
  const double t = __dmul_rn(q, phi);
  sq = __dadd_rn(sq, t);
  sp = __fma_rn(t, t, sp);
}
// sums of a warp whose first `n` lanes hold something
__device__ __forceinline__ void add_lanes(uint32_t n, double &a, double &b) {
  for (uint32_t o = 16; o > 0; o >>= 1)
    if (o < n) {
      a = __dadd_rn(a, __shfl_xor_sync(0xffffffffu, a, o));
      b = __dadd_rn(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
}
// the n measuring warps' sums, by a warp
__device__ __forceinline__ void add_parts(const double *part, int n, int lane, double &Q, double &P) {
  Q = P = 0.0;
  for (int r = lane; r < n; r += 32) {
    Q = __dadd_rn(Q, part[2 * r]);
    P = __dadd_rn(P, part[2 * r + 1]);
  }
  add_lanes((uint32_t)n, Q, P);
}
// e = Q^2 - P into a chain's running sums `st` and batch sums, and the log
__device__ __forceinline__ void record_sums(const ResidentArgs &a, int chain, double Q, double P,
                                            double *st, double *batch) {
  const double e = __fma_rn(Q, Q, -P);
  const int64_t n = (int64_t)st[kStatN];
  if (a.log != nullptr && n < a.log_cap) {
    double *row = a.log + 3 * ((size_t)n * a.n_chains + chain);
    row[0] = Q;
    row[1] = P;
    row[2] = e;
  }
  record_value(st, batch, e, a.err);
}

template <typename T, int V, bool SINGLE>
__global__ void __launch_bounds__(kMaxSweepThreads + kMeasThreads, 1)
    resident_kernel(const ResidentArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  double *part = reinterpret_cast<double *>(smem);
  double *st = part + 2 * kResParts;
  T *draws = reinterpret_cast<T *>(smem + kResHeaderBytes);
  T *planes = reinterpret_cast<T *>(smem + kResHeaderBytes + (SINGLE ? kResDrawBytes : 0));
  const int tid = threadIdx.x;
  // warps: sweeping, then (single form) as many drawing, then measuring
  const int n_sweep_thr = ((int)blockDim.x - kMeasThreads) / (SINGLE ? 2 : 1);
  const int C = a.cluster;
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int chain = (int)blockIdx.x / C;
  const int Lx = a.Lx, Ly = a.Ly, Lz = a.Lz, W = a.W;
  const int z0 = (int)((int64_t)Lz * rank / C), nz = (int)((int64_t)Lz * (rank + 1) / C) - z0;
  const int plane = (Ly + 2) * W;                    // with its two ghost rows
  const int colour_s = ((Lz + C - 1) / C + 2) * plane;  // the same in every CTA
  T *field = reinterpret_cast<T *>(a.field) + (size_t)chain * a.chain_elems;
  const PhiloxKeys &K = *reinterpret_cast<const PhiloxKeys *>(a.round_keys);
  const bool measure = a.stats != nullptr;

  // ---- load: planes z0 - 1 .. z0 + nz of both colours, ghosts as 0.  The rows
  // of a plane lie one after another here and in the field: one bulk copy each
  // (a loop over 16-byte loads, with its divisions, and a like store made a
  // launch of one sweep of 64^3 x 30 chains 72 us, heatbath only; now 51).
  const int in_lo = z0 > 0 ? 0 : 1, in_hi = z0 + nz < Lz ? nz + 2 : nz + 1;  // planes in the box
  const uint32_t plane_bytes = (uint32_t)(Ly * W) * (uint32_t)sizeof(T);
  const uint32_t bar_load = smem_addr(smem + kResBar);
  bool loaded = true;
  {
    if (tid == 0) {
      mbar_init(bar_load, 1);
      fence_mbar_init();
      mbar_arrive_expect_tx(bar_load, 2u * (uint32_t)(in_hi - in_lo) * plane_bytes);
      for (int c = 0; c < 2; ++c)
        for (int p = in_lo; p < in_hi; ++p)
          bulk_load(smem_addr(planes + c * colour_s + p * plane + W),
                    field + (size_t)c * a.colour_elems + (size_t)(z0 - 1 + p) * Ly * W, plane_bytes,
                    bar_load);
    }
    constexpr int kPer = 16 / (int)sizeof(T);  // elements per 16 bytes
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p = 0; p < nz + 2; ++p) {
      const bool in = p >= in_lo && p < in_hi;
      for (int c = 0; c < 2; ++c) {
        float4 *q = reinterpret_cast<float4 *>(planes + c * colour_s + p * plane);
        const int W16 = W / kPer, rows = in ? 2 : Ly + 2, last = (Ly + 1) * W16;
        for (int i = tid; i < rows * W16; i += blockDim.x)
          q[in && i >= W16 ? last + i - W16 : i] = zero;
      }
    }
    if (measure && rank == 0) {
      for (int i = tid; i < kStatStride; i += blockDim.x)
        st[i] = a.stats[(size_t)chain * kStatStride + i];
      for (int i = tid; i < 2 * kResParts; i += blockDim.x) part[i] = 0.0;
    }
    __syncthreads();  // the mbarrier is initialised
    loaded = mbar_wait_bounded(bar_load, 0u);
    if (!loaded && tid == 0) atomicOr(a.err, kErrTimeout);
  }
  uint32_t pass = *a.pass_ptr;
  auto barrier = [&]() {
    if (C > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  // lanes across a row, then rows; row index = run * Ly + y, a run being
  // a.run consecutive planes (drawing threads: the sweeping thread's place)
  const int place_id = SINGLE && tid >= n_sweep_thr ? tid - n_sweep_thr : tid;
  const int lanes = V == 4 ? a.Wq : (Lx + 1) / 2;
  const int tx = place_id % lanes, row0 = place_id / lanes, step = n_sweep_thr / lanes;
  const int n_rows = (nz + a.run - 1) / a.run * Ly;
  const int first = tx * V;  // the thread's first site index h of a row
  const bool worker = row0 < step;
  const int y_first = row0 % Ly, run_first = row0 / Ly;
  const bool has_first = worker && row0 < n_rows;
  auto draw = [&](int c, int y, int z, T (&n)[V]) {
    const uint32_t quad = ((uint32_t)z * (uint32_t)Ly + (uint32_t)y) * (uint32_t)a.Wq +
                          (uint32_t)(first >> 2);
    const uint4 w = philox4x32_10(make_uint4(quad, pass, (uint32_t)chain, (uint32_t)c), K);
    Draw<V>::of(w, first, n);
  };
  const int n_pass = a.n_hb + a.n_or, n_half = 2 * n_pass;
  const bool drawing = SINGLE && tid >= n_sweep_thr && tid < 2 * n_sweep_thr;
  if (drawing && has_first && a.n_hb > 0) {  // for the first half-sweep
    T n[V];
    draw(0, y_first, z0 + run_first, n);
    Group<T, V>::st(draws + place_id * V, n);
  }
  barrier();

  if (drawing) {
    // ----------------------------------------------------------- drawing
    // the deviates of half-sweep hs + 1 while the sweeping warps do hs
    for (int s = 0; s < a.n_sweeps; ++s)
      for (int hs = 0; hs < n_half; ++hs) {
        const int nh = hs + 1 < n_half ? hs + 1 : 0;
        if (hs & 1) ++pass;
        if ((nh >> 1) < a.n_hb && has_first) {
          T n[V];
          draw(nh & 1, y_first, z0 + run_first, n);
          Group<T, V>::st(draws + ((nh & 1) * n_sweep_thr + place_id) * V, n);
        }
        barrier();
      }
    if (measure) barrier();  // the last sample's (see below)
  } else if (tid < n_sweep_thr) {
    // ---------------------------------------------------------- sweeping
    uint32_t pad[2] = {0u, 0u};  // sites at or past Lx, by row parity
#pragma unroll
    for (int i = 0; i < V; ++i)
#pragma unroll
      for (int p = 0; p < 2; ++p)
        if (2 * (first + i) + p >= Lx) pad[p] |= 1u << i;
    const bool lo_ok = first > 0, hi_ok = first + V < W;
    const uint32_t sbase = smem_addr(planes);
    const uint32_t below = C > 1 && rank > 0 ? map_rank(sbase, rank - 1) : 0u;
    const uint32_t above = C > 1 && rank < C - 1 ? map_rank(sbase, rank + 1) : 0u;
    // the plane after the last of the CTA below (its upper halo)
    const int nz_below =
        rank > 0 ? z0 - (int)((int64_t)Lz * (rank - 1) / C) : 0;

    if constexpr (SINGLE) {
      // this thread's sites in registers, its places fixed
      const int z = z0 + run_first, p = run_first + 1;
      const int off = p * plane + (y_first + 1) * W + first;
      T own[2][V];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int i = 0; i < V; ++i) own[c][i] = has_first ? planes[c * colour_s + off + i] : T(0);
      const int odd0 = (y_first + z) & 1;
      const uint32_t to_below =
          below && p == 1 ? below + (uint32_t)((off + nz_below * plane) * (int)sizeof(T)) : 0u;
      const uint32_t to_above =
          above && p == nz ? above + (uint32_t)((off - p * plane) * (int)sizeof(T)) : 0u;
      for (int s = 0; s < a.n_sweeps; ++s)
        for (int ps = 0; ps < n_pass; ++ps) {
          const bool orx = ps >= a.n_hb;
          const T coef = orx ? Coef<T>::third : Coef<T>::sixth;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            if (has_first) {
              const T *o = planes + (c ^ 1) * colour_s + off;
              const bool odd = (odd0 ^ c) != 0;
              T M[V], P[V], ym[V], yp[V], add[V], u[V];
              Group<T, V>::ld(o - plane, M);
              Group<T, V>::ld(o + plane, P);
              Group<T, V>::ld(o - W, ym);
              Group<T, V>::ld(o + W, yp);
              const T e = (odd ? hi_ok : lo_ok) ? o[odd ? V : -1] : T(0);
              if (orx) {
#pragma unroll
                for (int i = 0; i < V; ++i) add[i] = -own[c][i];
              } else {
                Group<T, V>::ld(draws + (c * n_sweep_thr + tid) * V, add);
              }
              if constexpr (V == 4) {
                float2 S[2];
                neighbour_sum(M, own[c ^ 1], P, ym, yp, e, odd, S);
                update(S, coef, add, u);
              } else {
                u[0] = fma(((M[0] + P[0]) + (ym[0] + yp[0])) + (own[c ^ 1][0] + e), coef, add[0]);
              }
              const uint32_t pm = odd ? pad[1] : pad[0];
#pragma unroll
              for (int i = 0; i < V; ++i) {
                if ((pm >> i) & 1u) u[i] = T(0);
                own[c][i] = u[i];
              }
              Group<T, V>::st(planes + c * colour_s + off, u);
              const uint32_t cs = (uint32_t)(c * colour_s * (int)sizeof(T));
              if (to_below) st_remote(to_below + cs, u);
              if (to_above) st_remote(to_above + cs, u);
            }
            barrier();
          }
        }
    } else {
    T pre[V];
#pragma unroll
    for (int i = 0; i < V; ++i) pre[i] = T(0);
    if (has_first && a.n_hb > 0) draw(0, y_first, z0 + run_first * a.run, pre);

    const int dy = step % Ly, dr = step / Ly;
    for (int s = 0; s < a.n_sweeps; ++s) {
      for (int hs = 0; hs < n_half; ++hs) {
        const int c = hs & 1;
        const bool orx = (hs >> 1) >= a.n_hb;
        const T *oth = planes + (c ^ 1) * colour_s;
        T *own = planes + c * colour_s;
        bool at_first = true;
        if (worker) {
          int y = y_first, run = run_first;
          for (int row = row0; row < n_rows; row += step) {
            const int p0 = run * a.run + 1, p1 = min(p0 + a.run, nz + 1);  // local planes
            int off = p0 * plane + (y + 1) * W + first;
            T M[V], Cc[V];
            Group<T, V>::ld(oth + off - plane, M);
            Group<T, V>::ld(oth + off, Cc);
            for (int p = p0; p < p1; ++p, off += plane) {
              const int z = z0 + p - 1;
              const int par = (c + y + z) & 1;
              const bool odd = par != 0;
              T P[V], ym[V], yp[V], u[V];
              Group<T, V>::ld(oth + off + plane, P);
              Group<T, V>::ld(oth + off - W, ym);
              Group<T, V>::ld(oth + off + W, yp);
              const T e = (odd ? hi_ok : lo_ok) ? oth[off + (odd ? V : -1)] : T(0);
              T add[V];
              if (orx) {
                Group<T, V>::ld(own + off, add);
#pragma unroll
                for (int i = 0; i < V; ++i) add[i] = -add[i];
              } else if (at_first) {
#pragma unroll
                for (int i = 0; i < V; ++i) add[i] = pre[i];
              } else {
                draw(c, y, z, add);
              }
              at_first = false;
              const T coef = orx ? Coef<T>::third : Coef<T>::sixth;
              if constexpr (V == 4) {
                float2 S[2];
                neighbour_sum(M, Cc, P, ym, yp, e, odd, S);
                update(S, coef, add, u);
              } else {
                u[0] = fma(((M[0] + P[0]) + (ym[0] + yp[0])) + (Cc[0] + e), coef, add[0]);
              }
              const uint32_t pm = par ? pad[1] : pad[0];
              if (pm) {
#pragma unroll
                for (int i = 0; i < V; ++i)
                  if ((pm >> i) & 1u) u[i] = T(0);
              }
              Group<T, V>::st(own + off, u);
              if (p == 1 && below)
                st_remote(below + (uint32_t)((c * colour_s + (nz_below + 1) * plane +
                                              (off - p * plane)) * (int)sizeof(T)), u);
              if (p == nz && above)
                st_remote(above + (uint32_t)((c * colour_s + (off - p * plane)) *
                                             (int)sizeof(T)), u);
#pragma unroll
              for (int i = 0; i < V; ++i) {
                M[i] = Cc[i];
                Cc[i] = P[i];
              }
            }
            y += dy;
            run += dr;
            if (y >= Ly) {
              y -= Ly;
              ++run;
            }
          }
        }
        if (C > 1) cluster_arrive();
        // the first deviates of the next half-sweep while the others arrive
        if (c == 1) ++pass;
        const int nh = hs + 1 < n_half ? hs + 1 : 0;
        if ((nh >> 1) < a.n_hb && has_first)
          draw(nh & 1, y_first, z0 + run_first * a.run, pre);
        if (C > 1)
          cluster_wait();
        else
          __syncthreads();
      }
    }
    }
    if (measure) barrier();  // the last sample's (see below)
  } else {
    // ---------------------------------------------------------- measuring
    const int mt = tid - ((int)blockDim.x - kMeasThreads), lane = mt & 31, wid = mt >> 5;
    if (wid == kMeasWarps - 1) {
      // the recorder (works in CTA 0): the slots' sum during half-sweep 1, the
      // running statistics, in lane 0's registers, during the one after
      const bool on = measure && rank == 0;
      double run_st[kStatBatch0];
#pragma unroll
      for (int i = 0; i < kStatBatch0; ++i) run_st[i] = on ? st[i] : 0.0;
      double Q = 0.0, P = 0.0;
      bool pending = false;
      auto sum = [&]() {
        add_parts(part, C * a.meas_warps, lane, Q, P);
        pending = true;
      };
      auto record = [&]() {
        if (lane == 0 && pending) record_sums(a, chain, Q, P, run_st, st + kStatBatch0);
        pending = false;
      };
      const int at_half = n_half > 2 ? 2 : 0;
      for (int s = 0; s < a.n_sweeps; ++s)
        for (int hs = 0; hs < n_half; ++hs) {
          if (on && hs == at_half) record();
          if (on && hs == 1 && s > 0) sum();
          barrier();
        }
      if (measure) {
        if (on) record();
        barrier();
        if (on) {
          sum();
          record();
          if (lane == 0)
#pragma unroll
            for (int i = 0; i < kStatBatch0; ++i) st[i] = run_st[i];
        }
      }
    } else {
      // gathering warp w takes the entries w * 32 + lane, then those
      // a.meas_warps warps further on; warps past those only keep the barriers
      const uint32_t stride = 32u * (uint32_t)a.meas_warps;
      uint32_t e0 = 0, e1 = 0, top = 0;
      uint32_t at[kResEntries];
      double q[kResEntries];
      auto place = [&](uint32_t ent) -> uint32_t {  // element of `planes`
        const uint32_t o = ent & ~kGatherColourBit, c = ent >> 31;
        const uint32_t row = o / (uint32_t)W, h = o - row * (uint32_t)W;
        const uint32_t z = row / (uint32_t)Ly, y = row - z * (uint32_t)Ly;
        return (c * (uint32_t)colour_s + (z - (uint32_t)z0 + 1u) * (uint32_t)plane +
                (y + 1u) * (uint32_t)W + h) | (ent & kGatherColourBit);
      };
      if (measure && wid < a.meas_warps) {
        e0 = a.g_off[z0] + (uint32_t)(32 * wid);
        e1 = a.g_off[z0 + nz];
        top = e1 > e0 ? e1 - e0 : 0u;  // lanes with entries: the first `top`
        e0 += (uint32_t)lane;
      }
#pragma unroll
      for (int k = 0; k < kResEntries; ++k) {
        const uint32_t e = e0 + (uint32_t)k * stride;
        at[k] = 0u;
        q[k] = 0.0;
        if (e < e1) {
          at[k] = place(a.g_ent[e]);
          q[k] = a.g_q[e];
        }
      }
      double sq = 0.0, sp = 0.0;
      auto add_colour = [&](uint32_t c) {
#pragma unroll
        for (int k = 0; k < kResEntries; ++k) {
          const uint32_t e = e0 + (uint32_t)k * stride;
          if (e < e1 && (at[k] >> 31) == c)
            add_charge(q[k], (double)planes[at[k] & ~kGatherColourBit], sq, sp);
        }
        for (uint32_t e = e0 + (uint32_t)kResEntries * stride; e < e1; e += stride) {
          const uint32_t ent = a.g_ent[e];
          if ((ent >> 31) == c)
            add_charge(a.g_q[e], (double)planes[place(ent) & ~kGatherColourBit], sq, sp);
        }
      };
      // this warp's sums to CTA 0's shared memory (the slots of warps without
      // charges stay the zeros written at the start)
      const int slot = rank * a.meas_warps + wid;
      const uint32_t to = smem_addr(part) + 16u * (uint32_t)slot;
      const uint32_t to_cta0 = C > 1 ? map_rank(to, 0u) : 0u;
      auto send = [&]() {
        if (top == 0u) return;
        add_lanes(top, sq, sp);
        if (lane == 0) {
          if (C > 1) {
            const double vq[1] = {sq}, vp[1] = {sp};
            st_remote(to_cta0, vq);
            st_remote(to_cta0 + 8u, vp);
          } else {
            part[2 * slot] = sq;
            part[2 * slot + 1] = sp;
          }
        }
        sq = sp = 0.0;
      };
      for (int s = 0; s < a.n_sweeps; ++s)
        for (int hs = 0; hs < n_half; ++hs) {
          if (hs == 0 && s > 0) {
            add_colour(1u);
            send();
          }
          if (hs == n_half - 1) add_colour(0u);
          barrier();
        }
      if (measure) {
        add_colour(1u);
        send();
        barrier();
      }
    }
  }
  // no CTA leaves while another may still store into it; the statistics are
  // final, and the planes visible to the bulk stores, after this barrier
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  barrier();

  // ---- store this CTA's planes and the statistics.  After a load that never
  // came the field stays as it was.
  if (tid == 0) {
    if (!loaded) loaded = mbar_wait_bounded(bar_load, 0u);  // no copy in flight at the end
    else {
      for (int c = 0; c < 2; ++c)
        for (int p = 0; p < nz; ++p)
          bulk_store(field + (size_t)c * a.colour_elems + (size_t)(z0 + p) * Ly * W,
                     smem_addr(planes + c * colour_s + (p + 1) * plane + W), plane_bytes);
      bulk_store_wait();
    }
  }
  if (measure && rank == 0)
    for (int i = tid; i < kStatStride; i += blockDim.x)
      a.stats[(size_t)chain * kStatStride + i] = st[i];
}

// One sample of every chain from the fields in memory, bitwise the resident
// kernel's: its warps' charges, their order and its additions.  For runs of so
// few sweeps that the march kernels make them sooner.  A CTA per chain, bound by
// its chain of dependent loads and sums; with 8 warps instead of 16 the sums of 12
// measuring warps take two rounds and a sweep 40.2 instead of 38.0 us (40^3 x 100).
constexpr int kSampleThreads = 512;
template <typename T>
__global__ void __launch_bounds__(kSampleThreads) resident_sample_kernel(const ResidentArgs a) {
  __shared__ double part[2 * kResParts];
  const int chain = blockIdx.x, lane = threadIdx.x & 31;
  const T *f = reinterpret_cast<const T *>(a.field) + (size_t)chain * a.chain_elems;
  const int slots = a.cluster * a.meas_warps;
  const uint32_t stride = 32u * (uint32_t)a.meas_warps;
  for (int s = threadIdx.x >> 5; s < slots; s += kSampleThreads / 32) {
    const int rank = s / a.meas_warps, w = s - rank * a.meas_warps;
    const int z0 = (int)((int64_t)a.Lz * rank / a.cluster),
              z1 = (int)((int64_t)a.Lz * (rank + 1) / a.cluster);
    const uint32_t first = a.g_off[z0] + (uint32_t)(32 * w), e1 = a.g_off[z1];
    double sq = 0.0, sp = 0.0;
    for (uint32_t c = 0; c < 2; ++c)
      for (uint32_t e0 = first + (uint32_t)lane; e0 < e1; e0 += 4u * stride) {
        // four charges' loads at a time, added in order
        double q[4], phi[4];
        bool in[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t e = e0 + (uint32_t)k * stride;
          const uint32_t ent = e < e1 ? a.g_ent[e] : 0u;
          in[k] = e < e1 && (ent >> 31) == c;
          q[k] = in[k] ? a.g_q[e] : 0.0;
          phi[k] = in[k] ? (double)f[(size_t)c * a.colour_elems + (ent & ~kGatherColourBit)] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (in[k]) add_charge(q[k], phi[k], sq, sp);
      }
    add_lanes(e1 > first ? e1 - first : 0u, sq, sp);
    if (lane == 0) {
      part[2 * s] = sq;
      part[2 * s + 1] = sp;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double Q, P;
    add_parts(part, slots, lane, Q, P);
    double *st = a.stats + (size_t)chain * kStatStride;
    if (lane == 0) record_sums(a, chain, Q, P, st, st + kStatBatch0);
  }
}

size_t resident_smem(const Geometry &g, int C, bool single) {
  return (size_t)kResHeaderBytes + (single ? kResDrawBytes : 0) +
         2 * (size_t)((g.Lz + C - 1) / C + 2) * (g.Ly + 2) * g.W * g.es;
}

// threads of a CTA
int resident_block(const ResidentPlan &p) {
  return (p.single ? 2 : 1) * p.threads + kMeasThreads;
}

template <typename T, int V, bool SINGLE>
cudaError_t launch_t(const Geometry &g, const ResidentPlan &p, const ResidentArgs &a,
                     cudaStream_t s) {
  auto kfn = resident_kernel<T, V, SINGLE>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(g.n_chains * p.cluster));
  cfg.blockDim = dim3((unsigned)resident_block(p));
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)p.cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kfn, a);
}

template <typename T, int V, bool SINGLE>
int active_clusters_t(const ResidentPlan &p) {
  auto kfn = resident_kernel<T, V, SINGLE>;
  static bool configured = false;
  if (!configured) {
    if (cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResMaxSmem) !=
            cudaSuccess ||
        cudaFuncSetAttribute(kfn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    configured = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.cluster);
  cfg.blockDim = dim3((unsigned)resident_block(p));
  cfg.dynamicSmemBytes = p.smem;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)p.cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kfn, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace

bool resident_shape(const Geometry &g, int C, ResidentPlan *p) {
  if (C < 1 || C > kMaxCluster || C > g.Lz) return false;
  const bool f32 = g.precision == COULPS_F32;
  const int lanes = f32 ? g.Wq : (g.Lx + 1) / 2;
  const int nz = (g.Lz + C - 1) / C;
  const int64_t items = (int64_t)nz * g.Ly * lanes;
  p->cluster = C;
  p->single = items <= kSingleThreads;
  p->smem = resident_smem(g, C, p->single);
  if (p->smem > kResMaxSmem) return false;
  const int64_t rows = std::min<int64_t>((int64_t)nz * g.Ly, std::max(1, kMaxSweepThreads / lanes));
  p->threads = (int)std::min<int64_t>(kMaxSweepThreads, (rows * lanes + 31) / 32 * 32);
  // planes per march: the fewest thread-steps, a march's start (two planes
  // loaded and not used again) counted as half a step
  const int step = p->threads / lanes;
  p->run = 1;
  p->steps = 0.0;
  for (int r = 1; r <= nz; ++r) {
    const int n_runs = (nz + r - 1) / r;
    const double c = (double)(((int64_t)n_runs * g.Ly + step - 1) / step) * (r + 0.5);
    if (r == 1 || c < p->steps) {
      p->steps = c;
      p->run = r;
    }
  }
  return true;
}

int resident_per_sm(const ResidentPlan &p) {
  return std::min(2048 / resident_block(p), (int)(228 * 1024 / (p.smem + 1024)));
}

bool resident_active(const Geometry &g, ResidentPlan *p) {
  const bool f32 = g.precision == COULPS_F32;
  if (p->single)
    p->active = f32 ? active_clusters_t<float, 4, true>(*p) : active_clusters_t<double, 1, true>(*p);
  else
    p->active =
        f32 ? active_clusters_t<float, 4, false>(*p) : active_clusters_t<double, 1, false>(*p);
  return p->active > 0;
}

// Barriers (0.55 us a half-sweep with a cluster, 0.33 without) and thread-steps
// (FP32: 512 threads share the schedulers and shared memory) or sites (FP64:
// bound by the FP64 instructions, 16 per draw and update, 6 per reflection),
// in as many waves as the clusters need.
double resident_time(const Geometry &g, const ResidentPlan &p, int n_hb, int n_or) {
  const int waves = (g.n_chains + p.active - 1) / p.active;
  const int n_half = 2 * (n_hb + n_or);
  const double barrier = p.cluster > 1 ? 0.55 : 0.33;
  double work;
  if (g.precision == COULPS_F32) {
    const double load = std::max(0.35, p.threads / (double)kMaxSweepThreads);
    work = p.steps * load * (1.5 * n_hb + 0.5 * n_or);
  } else {
    const double sites = (double)((g.Lz + p.cluster - 1) / p.cluster) * g.Ly * ((g.Lx + 1) / 2);
    work = sites * (9.0e-3 * n_hb + 4.2e-3 * n_or);
  }
  return waves * (n_half * barrier + work);
}

// one measuring warp where each CTA has few charges
static int measuring_warps(const ResidentPlan &p, int64_t n_q) {
  return n_q <= 16 * (int64_t)p.cluster ? 1 : kGatherWarps;
}

cudaError_t launch_resident_sample(const Geometry &g, const ResidentPlan &p, ResidentArgs a,
                                   int64_t n_q, cudaStream_t s) {
  a.cluster = p.cluster;
  a.meas_warps = measuring_warps(p, n_q);
  if (g.precision == COULPS_F32)
    resident_sample_kernel<float><<<g.n_chains, kSampleThreads, 0, s>>>(a);
  else
    resident_sample_kernel<double><<<g.n_chains, kSampleThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_resident(const Geometry &g, const ResidentPlan &p, ResidentArgs a, int64_t n_q,
                            cudaStream_t s) {
  a.cluster = p.cluster;
  a.run = p.run;
  a.meas_warps = measuring_warps(p, n_q);
  const bool f32 = g.precision == COULPS_F32;
  if (p.single)
    return f32 ? launch_t<float, 4, true>(g, p, a, s) : launch_t<double, 1, true>(g, p, a, s);
  return f32 ? launch_t<float, 4, false>(g, p, a, s) : launch_t<double, 1, false>(g, p, a, s);
}

}  // namespace coulps
