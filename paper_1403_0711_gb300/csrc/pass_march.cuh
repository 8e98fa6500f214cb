// One tile of a fused pass (both half-sweeps of one pass in a single z-march
// from a source copy of the field to a destination copy; see pass_fused.cu for
// the design), shared by the single-lattice pass kernel and the many-system
// kernel.  A CTA may march several tiles of different systems in a row: the
// ring's mbarrier phases run on from tile to tile (`gbase`).
#pragma once

#include <type_traits>

#include "device_common.cuh"
#include "internal.h"
#include "march_quad.cuh"
#include "tile_march.cuh"

namespace coulps {
namespace tile {

// Ring depth of the fused pass (slots of one colour-1 box and one colour-0
// box); at most 8 (mbarriers at 0 .. 63 of the header, abort flag at 64).
// Measured per over-relaxation pass, 128^3 x 64 chains / 512^3: 204 / 204 us with
// 4 slots, 183 / 175 with 6, 179 / 227 with 8 (a CTA less per SM).
constexpr int kPassStages = 6;
static_assert(kPassStages <= 8, "mbarriers must end before the abort flag");

struct PassLayout {
  int c1_bytes;    // colour-1 box: (TY + 4) rows x W
  int c0_bytes;    // colour-0 box: (TY + 2) rows x W (over-relaxation only)
  int slot_bytes;  // both, each rounded to 128 bytes
  int new_bytes;   // one plane of new colour-0 rows: (TY + 2) x W
  int total;       // header + kPassStages slots + 2 new planes
};

__host__ __device__ inline PassLayout pass_layout(int TY, int W, int es, bool orx) {
  PassLayout L;
  L.c1_bytes = (TY + 4) * W * es;
  L.c0_bytes = orx ? (TY + 2) * W * es : 0;
  L.slot_bytes = round_up_int(L.c1_bytes, 128) + round_up_int(L.c0_bytes, 128);
  L.new_bytes = round_up_int((TY + 2) * W * es, 128);
  L.total = kHeaderBytes + kPassStages * L.slot_bytes + 2 * L.new_bytes;
  return L;
}

// The tile: TY rows from y0 and planes [z0, z0 + nz) of one chain (or
// system), read through tm_c1 / tm_c0 (4th coordinates map_c1 / map_c0) and
// written to dst (colour 0) and dst + colour_elems (colour 1), element
// (z Ly + y) W + h.  Philox counter words: quad, pass, rng_id, colour.  With
// GATHER, g_off points at the tile column's plane offsets (entries of plane
// z: [g_off[z], g_off[z + 1])).
//
// march_pass reads a tile through accessors of these names.  PassTile
// stores them (the many-system kernel fills one per tile of its work list);
// the one-tile-per-CTA kernel answers from its parameters and block index at
// the point of use, which measured 8% fewer instructions than a stored job
// (the compiler then shares the address arithmetic of the two colours and
// keeps the origin out of registers).
template <typename T>
struct PassTile {
  // the CTA may have whole warps past the tile's rows (one block size for
  // tiles of every system): they skip the stages
  static constexpr bool kIdleWarps = true;
  const CUtensorMap *tm_c1_, *tm_c0_;
  int map_c1_, map_c0_;
  T *dst_;
  size_t colour_elems_;
  int Lx_, Ly_, Lz_, W_, Wq_, QW_, TY_;
  int y0_, z0_, nz_;
  uint32_t rng_id_, pass_;
  const uint32_t *g_off_, *g_ent_;
  const double *g_q_;
  COULPS_FIELD(const CUtensorMap *, tm_c1) COULPS_FIELD(const CUtensorMap *, tm_c0)
  COULPS_FIELD(int, map_c1) COULPS_FIELD(int, map_c0)
  COULPS_FIELD(T *, dst) COULPS_FIELD(size_t, colour_elems)
  COULPS_FIELD(int, Lx) COULPS_FIELD(int, Ly) COULPS_FIELD(int, Lz) COULPS_FIELD(int, W)
  COULPS_FIELD(int, Wq) COULPS_FIELD(int, QW) COULPS_FIELD(int, TY)
  COULPS_FIELD(int, y0) COULPS_FIELD(int, z0) COULPS_FIELD(int, nz)
  COULPS_FIELD(uint32_t, rng_id) COULPS_FIELD(uint32_t, pass)
  COULPS_FIELD(const uint32_t *, g_off) COULPS_FIELD(const uint32_t *, g_ent)
  COULPS_FIELD(const double *, g_q)
};

// Shared-memory header of a pass CTA: kPassStages mbarriers and the abort
// flag; done once per CTA.
__device__ __forceinline__ void pass_ring_init(unsigned char *smem) {
  if (threadIdx.x == 0) {
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    for (int k = 0; k < kPassStages; ++k) mbar_init(smem_addr(&bars[k]), 1);
    *reinterpret_cast<volatile int *>(smem + 64) = 0;
    fence_mbar_init();
  }
  __syncthreads();
}

// Runs the tile; with GATHER adds this thread's share of Q and P over the
// tile's charges to (sq, sp).  `gbase` counts the ring planes this CTA has
// streamed before (phases continue from there) and is advanced past this
// tile's.  Returns false if a bounded wait gave up (the error word is set and
// no copy is left in flight).  Threads past the tile's (TY + 2) x QW quads
// only take part in the barriers.
template <typename T, bool OR, bool GATHER, typename Job>
__device__ bool march_pass(const Job &a, const PhiloxKeys &K, unsigned char *smem, int *err,
                           int &gbase, double &sq, double &sp) {
  const PassLayout lay = pass_layout(a.TY(), a.W(), (int)sizeof(T), OR);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + 64);
  const int gb = gbase;
  // ring slot of plane j, as a byte offset; the colour-0 box lies c0_off in
  auto slot_at = [&](int j) {
    return (uint32_t)(kHeaderBytes + ((gb + j) % kPassStages) * lay.slot_bytes);
  };
  auto at = [&](uint32_t off) { return reinterpret_cast<T *>(smem + off); };
  const uint32_t c0_off = (uint32_t)round_up_int(lay.c1_bytes, 128);

  const int W = a.W(), TY = a.TY(), QW = a.QW(), Lz = a.Lz();
  const int y0 = a.y0(), z0 = a.z0(), nz = a.nz();
  const int tid = threadIdx.x;
  const int rows = TY + 2;
  // this thread: quad qx of row r (y = y0 - 1 + r; rows 0 and TY + 1 are the
  // halo of stage 0); lanes past the last row alias its addresses for their
  // loads and store nothing
  const int qx = tid % QW;
  const bool lane_ok = tid < rows * QW;
  const int r = lane_ok ? tid / QW : rows - 1;
  const int y = y0 - 1 + r;
  const bool live = lane_ok && y >= 0 && y < a.Ly() && qx < a.Wq();
  const bool own_row = live && r >= 1 && r <= TY;  // a row of this tile: written out
  const bool warp_in0 = (tid & ~31) < rows * QW;
  const int n_ring = nz + 4;  // colour-1 planes z0 - 2 .. z0 + nz + 1
  T *dst0 = a.dst();
  T *dst1 = dst0 + a.colour_elems();
  const uint32_t pass = a.pass();

  if (tid == 0) {
    prefetch_tensormap(a.tm_c1());
    if (OR) prefetch_tensormap(a.tm_c0());
  }
  // ring plane j: colour 1 at z0 - 2 + j; with it (j >= 2) colour 0 at z0 - 3 + j
  auto issue = [&](int j) {
    const uint32_t bar = smem_addr(&bars[(gb + j) % kPassStages]);
    const bool own = OR && j >= 2;
    mbar_arrive_expect_tx(bar, lay.c1_bytes + (own ? lay.c0_bytes : 0));
    const uint32_t slot = smem_addr(at(slot_at(j)));
    tma_load_4d(slot, a.tm_c1(), 0, y0 - 2, z0 - 2 + j, a.map_c1(), bar);
    if (own) tma_load_4d(slot + c0_off, a.tm_c0(), 0, y0 - 1, z0 - 3 + j, a.map_c0(), bar);
  };
  auto wait_plane = [&](int j) -> bool {
    return mbar_wait_bounded(smem_addr(&bars[(gb + j) % kPassStages]),
                             (uint32_t)(((gb + j) / kPassStages) & 1));
  };
  int issued = 0;
  if (tid == 0)
    for (; issued < min(kPassStages, n_ring); ++issued) issue(issued);
  // fused gather: this tile's charge range, and this thread's first entry,
  // loaded while the first planes arrive (used once the tile is written)
  uint32_t g_e = 0u, g_e1 = 0u, g_ent0 = 0u;
  double g_q0 = 0.0;
  if (GATHER) {
    g_e = a.g_off()[z0] + (uint32_t)tid;
    g_e1 = a.g_off()[z0 + nz];
    if (g_e < g_e1) {
      g_ent0 = a.g_ent()[g_e];
      g_q0 = a.g_q()[g_e];
    }
  }
  // lanes of the quad past x = Lx - 1 (kept at 0), for row parity 0 and 1
  uint32_t pad0 = 0u, pad1 = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (2 * (4 * qx + i) >= a.Lx()) pad0 |= 1u << i;
    if (2 * (4 * qx + i) + 1 >= a.Lx()) pad1 |= 1u << i;
  }
  // the whole warp is inside the box and has no padding lanes
  const bool warp_full = __all_sync(0xffffffffu, live && pad0 == 0u && pad1 == 0u);
  const bool lo_ok = qx > 0, hi_ok = 4 * qx + 4 < W;
  // byte offsets: row r of the colour-0 box and of the buffers; the colour-1
  // box holds it one row further
  const uint32_t wb = (uint32_t)W * (uint32_t)sizeof(T);
  const uint32_t o_r = (uint32_t)r * wb + (uint32_t)(4 * qx) * (uint32_t)sizeof(T);
  const uint32_t bb = (uint32_t)lay.new_bytes;
  const uint32_t b_r = (uint32_t)(kHeaderBytes + kPassStages * lay.slot_bytes) + o_r;
  const size_t plane_elems = (size_t)a.Ly() * W;
  const size_t row_off = (size_t)(y < 0 ? 0 : y) * W + 4 * qx;
  // Philox counter word 0 of the quad at plane p: (p Ly + y) Wq + qx
  const uint32_t qrow = (uint32_t)y * (uint32_t)a.Wq() + (uint32_t)qx;
  const uint32_t qplane = (uint32_t)a.Ly() * (uint32_t)a.Wq();
  const uint32_t rng = a.rng_id();

  {
    const bool ok = wait_plane(0) && wait_plane(1);
    if (!ok) {
      atomicOr(err, kErrTimeout);
      *abort_flag = 1;
    }
  }
  __syncthreads();
  bool aborted = *abort_flag != 0;
  int done = 1;  // ring planes 0 .. done waited for by every thread

  // windows of the quad's three planes: old colour 1 (P), new colour 0 (N)
  Quad<T> P0 = qzero<T>(), P1 = qzero<T>(), P2 = qzero<T>();
  Quad<T> N0 = qzero<T>(), N1 = qzero<T>(), N2 = qzero<T>();
  if (!aborted) {
    P0 = qload<T>(at(slot_at(0) + o_r + wb));
    P1 = qload<T>(at(slot_at(1) + o_r + wb));
  }

  // What advances from step to step: this thread's row in the ring slots of
  // planes s + 1 and s + 2, the mbarrier of plane s + 2 and its parity, the
  // buffer, the row parity, the output pointer of stage 0's plane.
  const uint32_t ring_o = (uint32_t)kHeaderBytes + o_r;
  const uint32_t ring_end = ring_o + (uint32_t)(kPassStages * lay.slot_bytes);
  uint32_t n1 = slot_at(1) + o_r, n2 = slot_at(2) + o_r;
  const uint32_t bar0 = smem_addr(bars);
  uint32_t bar_n = bar0 + 8u * (uint32_t)((gb + 2) % kPassStages);
  uint32_t par_n = (uint32_t)(((gb + 2) / kPassStages) & 1);
  uint32_t w_r = b_r;                  // the buffer row the step writes (the other is read)
  const uint32_t b_sum = 2u * b_r + bb;
  bool odd = ((y + z0 - 1) & 1) != 0;  // the same row parity for both stages
  T *out = dst0 + (ptrdiff_t)(z0 - 1) * (ptrdiff_t)plane_elems + row_off;  // plane f
  const ptrdiff_t out1 = (ptrdiff_t)a.colour_elems() - (ptrdiff_t)plane_elems;

  // Step s, stage 0 at plane f = z0 - 1 + s and stage 1 at f - 1, with the
  // windows' names rotated by the caller.  At entry: P0, P1 = old colour 1 at
  // f - 1, f (P2 loaded here: f + 1); N0, N1 = new colour 0 at f - 2, f - 1
  // (N2 made here: f).  Ring planes s, s + 1 have arrived; s + 2 is waited
  // for here.  The deviates and stage 0 read no other warp's work of this
  // step and come before its one barrier, so that a warp through the previous
  // step goes on with them; stage 1 reads the previous step's buffer after
  // it.  STEADY: s >= 3.
  auto step = [&](auto steady, int s, Quad<T> &P0, Quad<T> &P1, Quad<T> &P2, Quad<T> &N0,
                  Quad<T> &N1, Quad<T> &N2) -> bool {
    constexpr bool STEADY = decltype(steady)::value;
    const int f = z0 - 1 + s;
    const bool e_ok = odd ? hi_ok : lo_ok;
    const uint32_t eo = odd ? 4u * (uint32_t)sizeof(T) : 0u - (uint32_t)sizeof(T);
    // nothing to zero in either stage
    const bool fast = warp_full && (STEADY || f >= 0) && f < Lz;
    bool got = mbar_wait_bounded(bar_n, par_n);
    // a warp makes the heatbath deviates and stage 0 whole or not at all
    if (!OR) got = __all_sync(0xffffffffu, got);
    if (!got) {
      atomicOr(err, kErrTimeout);
      *abort_flag = 1;
    }
    Quad<T> n0 = qzero<T>(), n1_dev = qzero<T>();
    if (got && (!Job::kIdleWarps || warp_in0)) {
      if (!OR) {
        const uint4 w0 =
            philox4x32_10(make_uint4((uint32_t)f * qplane + qrow, pass, rng, 0u), K);
        const uint4 w1 =
            philox4x32_10(make_uint4((uint32_t)(f - 1) * qplane + qrow, pass, rng, 1u), K);
        StageNoise<T>::of(w0, w1, n0, n1_dev);
      }
      // ---- stage 0: colour 0 at plane f (ring only)
      P2 = qload<T>(at(n2 + wb));
      const Quad<T> ym = qload<T>(at(n1)), yp = qload<T>(at(n1 + 2u * wb));
      const T e = e_ok ? *at(n1 + wb + eo) : T(0);
      if (OR) n0 = qload<T>(at(n2 + c0_off));
      N2 = update<T, OR>(P0, P2, ym, yp, P1, odd, e, n0);
      if (!fast) mask(N2, live && f >= 0 && f < Lz, odd ? pad1 : pad0);
    }
    __syncthreads();
    if (*abort_flag) return false;
    done = s + 2;
    // ring plane s was last read in the previous step: refill its slot
    if (tid == 0 && issued < n_ring) issue(issued++);
    if (lane_ok) qstore(at(w_r), N2);
    // the tile's planes: s = 1 .. nz
    if (own_row && (STEADY || s >= 1) && s <= nz) qstore(out, N2);
    // ---- stage 1: colour 1 at plane f - 1 (old value: P0)
    if ((STEADY || s >= 2) && own_row) {
      const uint32_t br = b_sum - w_r;
      const Quad<T> ym = qload<T>(at(br - wb)), yp = qload<T>(at(br + wb));
      const T e = e_ok ? *at(br + eo) : T(0);
      Quad<T> v = update<T, OR>(N0, N2, ym, yp, N1, odd, e, OR ? P0 : n1_dev);
      if (!fast) mask(v, true, odd ? pad1 : pad0);
      qstore(out + out1, v);
    }
    n1 = n2;
    n2 += (uint32_t)lay.slot_bytes;
    if (n2 == ring_end) n2 = ring_o;
    bar_n += 8u;
    if (bar_n == bar0 + 8u * kPassStages) {
      bar_n = bar0;
      par_n ^= 1u;
    }
    w_r = b_sum - w_r;
    odd = !odd;
    out += plane_elems;
    return true;
  };

  const int n_steps = nz + 2;
  using First = std::integral_constant<bool, false>;
  using Steady = std::integral_constant<bool, true>;
  if (!aborted)
    aborted = !(step(First(), 0, P0, P1, P2, N0, N1, N2) &&
                step(First(), 1, P1, P2, P0, N1, N2, N0) &&
                step(First(), 2, P2, P0, P1, N2, N0, N1));
#pragma unroll 1
  for (int s = 3; s < n_steps && !aborted; s += 3) {
    if (!step(Steady(), s, P0, P1, P2, N0, N1, N2)) { aborted = true; break; }
    if (s + 1 >= n_steps) break;
    if (!step(Steady(), s + 1, P1, P2, P0, N1, N2, N0)) { aborted = true; break; }
    if (s + 2 >= n_steps) break;
    if (!step(Steady(), s + 2, P2, P0, P1, N2, N0, N1)) { aborted = true; break; }
  }
  if (aborted && tid == 0) {
    // leave no copy in flight into this CTA's shared memory
    for (int k = done + 1; k < issued; ++k)
      if (!wait_plane(k)) break;
  }
  gbase = gb + n_ring;
  if (GATHER) {
    __syncthreads();  // this CTA's stores of the last step are visible to all its threads
    if (!aborted) {
      // both colours of the tile are still in L2; an entry holds its site's
      // colour and offset within the colour's array
      double tq = 0.0, tp = 0.0;
      for (uint32_t e = g_e; e < g_e1; e += blockDim.x) {
        const uint32_t ent = e == g_e ? g_ent0 : a.g_ent()[e];
        const double qe = e == g_e ? g_q0 : a.g_q()[e];
        const uint32_t at = ent & ~kGatherColourBit;
        const T val = (ent & kGatherColourBit) ? dst1[at] : dst0[at];
        const double t = qe * (double)val;
        tq += t;
        tp += t * t;
      }
      sq += tq;
      sp += tp;
    }
  }
  return !aborted;
}

}  // namespace tile
}  // namespace coulps
