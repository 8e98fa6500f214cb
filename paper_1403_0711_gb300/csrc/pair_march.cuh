// One tile of a pass pair (two passes in one z-march from a source copy of
// the field to a destination copy, four stages one plane apart; see
// pass_pair.cu for the design), shared by the single-lattice pair kernel and
// the many-system kernel.  A CTA may march several tiles of different
// systems in a row: the ring's mbarrier phases run on from tile to tile
// (`gbase`).
#pragma once

#include <type_traits>

#include "device_common.cuh"
#include "internal.h"
#include "march_quad.cuh"
#include "tile_march.cuh"

namespace coulps {
namespace tile {

// Ring depth: one CTA per SM streams the pair, so several planes (tens of KB)
// must be in flight to cover DRAM latency (measured at 128^3 x 64 chains,
// over-relaxation pairs: 270 us per launch with 4 slots, 258 with 6, 262 with 8;
// a compound sweep on two streams 668, 651, 651).
constexpr int kPairStages = 8;
// header: kPairStages (<= 12) mbarriers at 0, abort flag at 96, block reduction at 128
constexpr int kPairAbort = 96;
static_assert(kPairStages <= 12, "mbarriers must end before the abort flag");

// The stages' buffers (3 stages x 2 planes of (TY + 6) x W) lie quad by quad:
// the six values of one quad side by side and 16 bytes of padding, so that a
// stage's buffer is an immediate offset of the quad's one address and eight
// lanes' 16-byte accesses (pitch 28 words, FP64 52 words) fall on different
// banks.  Over-relaxation pair of 128^3 x 64 chains / 16^3 x 512 chains:
// 262 / 18.0 us; planes at a distance known only at run time 264 / 18.1; at a
// fixed 8192 bytes 258 / 28.4 (the small tile then loses CTAs per SM).
constexpr int pair_quad_pitch(int es) { return 6 * 4 * es + 16; }

struct PairLayout {
  int c1_bytes;   // colour-1 box: (TY + 8) rows x W
  int c0_bytes;   // colour-0 box: (TY + 6) rows x W (pass A over-relaxation only)
  int slot_bytes;
  int total;      // header + ring slots + 3 stages x 2 planes
};

__host__ __device__ inline PairLayout pair_layout(int TY, int W, int es, bool a_or) {
  PairLayout L;
  L.c1_bytes = (TY + 8) * W * es;
  L.c0_bytes = a_or ? (TY + 6) * W * es : 0;
  L.slot_bytes = round_up_int(L.c1_bytes, 128) + round_up_int(L.c0_bytes, 128);
  L.total = kHeaderBytes + kPairStages * L.slot_bytes + (TY + 6) * (W / 4) * pair_quad_pitch(es);
  return L;
}

// The tile: TY rows from y0 and planes [z0, z0 + nz) of one chain (or
// system), read through tm_c1 (TY + 8 rows) / tm_c0 (TY + 6 rows) with 4th
// coordinates map_c1 / map_c0, written to dst (colour 0) and dst +
// colour_elems (colour 1), element (z Ly + y) W + h.  Philox counter words:
// quad, pass (pass A; B is pass + 1), rng_id, colour.  With GATHER, g_off
// points at the tile column's plane offsets (entries of plane z:
// [g_off[z], g_off[z + 1])).  march_pair reads a tile through accessors of
// these names, as march_pass does (pass_march.cuh): PairTile stores them for
// the many-system kernel, the one-tile-per-CTA kernel reads its parameters.
template <typename T>
struct PairTile {
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

// Shared-memory header of a pair CTA: kPairStages mbarriers and the abort
// flag; done once per CTA.
__device__ __forceinline__ void pair_ring_init(unsigned char *smem) {
  if (threadIdx.x == 0) {
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    for (int k = 0; k < kPairStages; ++k) mbar_init(smem_addr(&bars[k]), 1);
    *reinterpret_cast<volatile int *>(smem + kPairAbort) = 0;
    fence_mbar_init();
  }
  __syncthreads();
}

// Runs the tile; with GATHER adds this thread's share of Q and P over the
// tile's charges to (sq, sp).  `gbase` counts the ring planes this CTA has
// streamed before and is advanced past this tile's.  Returns false if a
// bounded wait gave up (the error word is set and no copy is left in flight).
// With Job::kIdleWarps, warps with no row of the tile only take part in the
// barriers.
template <typename T, bool A_OR, bool B_OR, bool GATHER, typename Job>
__device__ bool march_pair(const Job &a, const PhiloxKeys &K, unsigned char *smem, int *err,
                           int &gbase, double &sq, double &sp) {
  const PairLayout lay = pair_layout(a.TY(), a.W(), (int)sizeof(T), A_OR);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kPairAbort);
  const int gb = gbase;
  // ring slot of plane j, as a byte offset
  auto slot_at = [&](int j) {
    return (uint32_t)(kHeaderBytes + ((gb + j) % kPairStages) * lay.slot_bytes);
  };
  auto at = [&](uint32_t off) { return reinterpret_cast<T *>(smem + off); };
  const uint32_t c0_off = (uint32_t)round_up_int(lay.c1_bytes, 128);  // colour-0 box in a slot

  const int W = a.W(), TY = a.TY(), QW = a.QW(), Ly = a.Ly(), Lz = a.Lz();
  const int y0 = a.y0(), z0 = a.z0(), nz = a.nz();
  const int tid = threadIdx.x;
  const int rows = TY + 6;
  // this thread: quad qx of row r (y = y0 - 3 + r); lanes past the last row
  // (block rounded up to whole warps) alias the last row's addresses for
  // their loads and store nothing (their stores would race with that row's)
  const int qx = tid % QW;
  const bool lane_ok = tid < rows * QW;
  const int r = lane_ok ? tid / QW : rows - 1;
  const int y = y0 - 3 + r;
  const bool live = lane_ok && y >= 0 && y < Ly && qx < a.Wq();
  const bool own_row = live && r >= 3 && r < TY + 3;  // a row of this tile: written out
  // rows of this warp, for skipping a stage that has none of them
  const int wr_lo = (tid & ~31) / QW, wr_hi = (tid | 31) / QW;
  bool warp_in[4];  // warp_in[0]: the warp has a row of the tile at all
#pragma unroll
  for (int k = 0; k < 4; ++k) warp_in[k] = wr_hi >= k && wr_lo <= rows - 1 - k;

  // byte offsets: row r in a colour-0 box = row r + 1 in the colour-1 box less
  // one row, and this quad's buffers (and its row neighbours', clamped for
  // rows no stage reads)
  constexpr uint32_t kQ = (uint32_t)(4 * sizeof(T)), kPitch = pair_quad_pitch((int)sizeof(T));
  const uint32_t wb = (uint32_t)W * (uint32_t)sizeof(T);
  const uint32_t o_r = (uint32_t)r * wb + (uint32_t)qx * kQ;
  const uint32_t bw = (uint32_t)QW * kPitch;
  const uint32_t b_r = (uint32_t)(kHeaderBytes + kPairStages * lay.slot_bytes) +
                       (uint32_t)r * bw + (uint32_t)qx * kPitch;
  const uint32_t b_m = r > 0 ? b_r - bw : b_r, b_p = r + 1 < rows ? b_r + bw : b_r;
  const bool lo_ok = qx > 0, hi_ok = 4 * qx + 4 < W;
  uint32_t pad0 = 0u, pad1 = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (2 * (4 * qx + i) >= a.Lx()) pad0 |= 1u << i;
    if (2 * (4 * qx + i) + 1 >= a.Lx()) pad1 |= 1u << i;
  }
  // the whole warp is inside the box and has no padding lanes
  const bool warp_full = __all_sync(0xffffffffu, live && pad0 == 0u && pad1 == 0u);
  T *dst0 = a.dst();
  T *dst1 = dst0 + a.colour_elems();
  const size_t plane_elems = (size_t)Ly * W;
  const size_t row_off = (size_t)(y < 0 ? 0 : y) * W + 4 * qx;
  const uint32_t pass_a = a.pass();
  const uint32_t pass_b = pass_a + 1u;
  const uint32_t rng = a.rng_id();
  // Philox counter word 0 of the quad at plane p: (p Ly + y) Wq + qx
  const uint32_t qrow = (uint32_t)y * (uint32_t)a.Wq() + (uint32_t)qx;
  const uint32_t qplane = (uint32_t)Ly * (uint32_t)a.Wq();

  const int n_ring = nz + 8;  // colour-1 planes z0 - 4 .. z0 + nz + 3
  if (tid == 0) {
    prefetch_tensormap(a.tm_c1());
    if (A_OR) prefetch_tensormap(a.tm_c0());
  }
  // ring plane j: colour 1 at z0 - 4 + j, with it (j >= 2) colour 0 at z0 - 5 + j
  auto issue = [&](int j) {
    const uint32_t bar = smem_addr(&bars[(gb + j) % kPairStages]);
    const bool own = A_OR && j >= 2;
    mbar_arrive_expect_tx(bar, lay.c1_bytes + (own ? lay.c0_bytes : 0));
    const uint32_t slot = smem_addr(at(slot_at(j)));
    tma_load_4d(slot, a.tm_c1(), 0, y0 - 4, z0 - 4 + j, a.map_c1(), bar);
    if (own) tma_load_4d(slot + c0_off, a.tm_c0(), 0, y0 - 3, z0 - 5 + j, a.map_c0(), bar);
  };
  auto wait_plane = [&](int j) -> bool {
    return mbar_wait_bounded(smem_addr(&bars[(gb + j) % kPairStages]),
                             (uint32_t)(((gb + j) / kPairStages) & 1));
  };
  int issued = 0;
  if (tid == 0)
    for (; issued < min(kPairStages, n_ring); ++issued) issue(issued);
  // fused gather: this CTA's charge range, and this thread's first entry,
  // loaded while the first planes arrive (used once the tile is written)
  uint32_t g_e = 0u, g_e1 = 0u, g_ent0 = 0u;
  double g_q0 = 0.0;
  if (GATHER) {
    const uint32_t *g_off = a.g_off();
    g_e = g_off[z0] + (uint32_t)tid;
    g_e1 = g_off[z0 + nz];
    if (g_e < g_e1) {
      g_ent0 = a.g_ent()[g_e];
      g_q0 = a.g_q()[g_e];
    }
  }
  {
    const bool ok = wait_plane(0) && wait_plane(1);
    if (!ok) {
      atomicOr(err, kErrTimeout);
      *abort_flag = 1;
    }
  }
  __syncthreads();
  bool aborted = *abort_flag != 0;
  int done = 1;  // ring planes 0 .. done completed for every thread

  // windows, per stage, of the quad's three planes (see the step): old colour
  // 1 (P), colour 0 after A (Q), colour 1 after A (R), colour 0 after B (U)
  Quad<T> P0 = qzero<T>(), P1 = qzero<T>(), P2 = qzero<T>();
  Quad<T> Q0 = qzero<T>(), Q1 = qzero<T>(), Q2 = qzero<T>();
  Quad<T> R0 = qzero<T>(), R1 = qzero<T>(), R2 = qzero<T>();
  Quad<T> U0 = qzero<T>(), U1 = qzero<T>(), U2 = qzero<T>();
  if (!aborted) {
    P0 = qload<T>(at(slot_at(0) + o_r + wb));
    P1 = qload<T>(at(slot_at(1) + o_r + wb));
  }

  // What advances from step to step: this thread's row in the ring slots of
  // planes s + 1 and s + 2, the mbarrier of plane s + 2 and its parity, the
  // buffers' parity, the row parity, the output pointer of stage 2's plane.
  const uint32_t ring_o = (uint32_t)kHeaderBytes + o_r;
  const uint32_t ring_end = ring_o + (uint32_t)(kPairStages * lay.slot_bytes);
  uint32_t n1 = slot_at(1) + o_r, n2 = slot_at(2) + o_r;
  const uint32_t bar0 = smem_addr(bars);
  uint32_t bar_n = bar0 + 8u * (uint32_t)((gb + 2) % kPairStages);
  uint32_t par_n = (uint32_t)(((gb + 2) / kPairStages) & 1);
  uint32_t tog = 0u;  // kQ in odd steps: what the step writes
  bool odd = ((y + z0 - 3) & 1) != 0;  // the same row parity for all four stages
  T *out = dst0 + (ptrdiff_t)(z0 - 5) * (ptrdiff_t)plane_elems + row_off;  // plane f - 2
  const ptrdiff_t out3 = (ptrdiff_t)a.colour_elems() - (ptrdiff_t)plane_elems;

  // Step s with the windows' names rotated by the caller.  At entry:
  // P0, P1 = old colour 1 at f - 1, f (P2 loaded here: f + 1); Q0, Q1 =
  // colour 0 after A at f - 2, f - 1 (Q2 made here: f); R0, R1 = colour 1
  // after A at f - 3, f - 2 (R2: f - 1); U0, U1 = colour 0 after B at f - 4,
  // f - 3 (U2: f - 2).  Ring planes s, s + 1 have arrived; s + 2 is waited
  // for here.
  //
  // What needs no other warp's rows of this step -- the heatbath deviates
  // (Philox words and erfc^-1) of every stage and the whole of stage 0,
  // which reads only the ring -- comes before the step's one barrier, so a
  // warp that finished the previous step early goes on with it while the
  // others finish.  After the barrier (all warps are through the previous
  // step: its buffer writes are visible and the buffers it read are free)
  // stages 1 .. 3 read the previous step's buffers and write this step's.
  //
  // STEADY: s >= 6, all four stages run and stage 3's plane is the tile's.
  auto step = [&](auto steady, int s, Quad<T> &P0, Quad<T> &P1, Quad<T> &P2, Quad<T> &Q0,
                  Quad<T> &Q1, Quad<T> &Q2, Quad<T> &R0, Quad<T> &R1, Quad<T> &R2, Quad<T> &U0,
                  Quad<T> &U1, Quad<T> &U2) -> bool {
    constexpr bool STEADY = decltype(steady)::value;
    const int f = z0 - 3 + s;
    const bool e_ok = odd ? hi_ok : lo_ok;
    const uint32_t eo = odd ? kQ : 0u - (uint32_t)sizeof(T);
    const uint32_t beo = odd ? kPitch : 3u * (uint32_t)sizeof(T) - kPitch;
    // nothing to zero in any stage: the warp is inside the box and without
    // padding lanes, and so are planes f - 3 .. f
    const bool fast = warp_full && f >= 3 && f < Lz;
    bool got = mbar_wait_bounded(bar_n, par_n);
    // a warp makes the heatbath deviates and stage 0 whole or not at all
    if (!A_OR || !B_OR) got = __all_sync(0xffffffffu, got);
    if (!got) {
      atomicOr(err, kErrTimeout);
      *abort_flag = 1;
    }
    Quad<T> nA0 = qzero<T>(), nA1 = qzero<T>(), nB0 = qzero<T>(), nB1 = qzero<T>();
    if (got && (!Job::kIdleWarps || warp_in[0])) {
      if (!A_OR) {
        const uint4 w0 = philox4x32_10(
            make_uint4((uint32_t)f * qplane + qrow, pass_a, rng, 0u), K);
        const uint4 w1 = philox4x32_10(
            make_uint4((uint32_t)(f - 1) * qplane + qrow, pass_a, rng, 1u), K);
        StageNoise<T>::of(w0, w1, nA0, nA1);
      }
      if (!B_OR && (STEADY || s >= 4)) {
        const uint4 w2 = philox4x32_10(
            make_uint4((uint32_t)(f - 2) * qplane + qrow, pass_b, rng, 0u), K);
        const uint4 w3 = philox4x32_10(
            make_uint4((uint32_t)(f - 3) * qplane + qrow, pass_b, rng, 1u), K);
        StageNoise<T>::of(w2, w3, nB0, nB1);
      }
      // ---- stage 0: colour 0 of pass A at plane f (ring only)
      P2 = qload<T>(at(n2 + wb));
      const Quad<T> ym = qload<T>(at(n1)), yp = qload<T>(at(n1 + 2u * wb));
      const T e = e_ok ? *at(n1 + wb + eo) : T(0);
      Quad<T> r0 = nA0;
      if (A_OR) r0 = qload<T>(at(n2 + c0_off));
      Q2 = update<T, A_OR>(P0, P2, ym, yp, P1, odd, e, r0);
      if (!fast) mask(Q2, live && f >= 0 && f < Lz, odd ? pad1 : pad0);
    }
    __syncthreads();
    if (*abort_flag) return false;
    done = s + 2;
    // ring plane s was last read in the previous step: refill its slot
    if (tid == 0 && issued < n_ring) issue(issued++);
    // stage k's plane goes to buffer k of this step's parity; stage k + 1 reads
    // buffer k of the other one
    const uint32_t w_r = b_r + tog, d = kQ - tog;
    const uint32_t r_m = b_m + d, r_p = b_p + d, r_e = b_r + d + beo;
    if (lane_ok) qstore(at(w_r), Q2);
    // ---- stage 1: colour 1 of pass A at plane f - 1 (old value: P0)
    if ((STEADY || s >= 2) && warp_in[1]) {
      const Quad<T> ym = qload<T>(at(r_m)), yp = qload<T>(at(r_p));
      const T e = e_ok ? *at(r_e) : T(0);
      R2 = update<T, A_OR>(Q0, Q2, ym, yp, Q1, odd, e, A_OR ? P0 : nA1);
      if (!fast) mask(R2, live && f >= 1 && f - 1 < Lz, odd ? pad1 : pad0);
      if (lane_ok) qstore(at(w_r + 2u * kQ), R2);
    }
    // ---- stage 2: colour 0 of pass B at plane f - 2 (old value: Q0)
    if ((STEADY || s >= 4) && warp_in[2]) {
      const Quad<T> ym = qload<T>(at(r_m + 2u * kQ)), yp = qload<T>(at(r_p + 2u * kQ));
      const T e = e_ok ? *at(r_e + 2u * kQ) : T(0);
      U2 = update<T, B_OR>(R0, R2, ym, yp, R1, odd, e, B_OR ? Q0 : nB0);
      if (!fast) mask(U2, live && f >= 2 && f - 2 < Lz, odd ? pad1 : pad0);
      if (lane_ok) qstore(at(w_r + 4u * kQ), U2);
      // the tile's planes: s = 5 .. nz + 4
      if (own_row && (STEADY || s >= 5) && s < nz + 5) qstore(out, U2);
    }
    // ---- stage 3: colour 1 of pass B at plane f - 3 (old value: R0)
    if ((STEADY || s >= 6) && warp_in[3]) {
      const Quad<T> ym = qload<T>(at(r_m + 4u * kQ)), yp = qload<T>(at(r_p + 4u * kQ));
      const T e = e_ok ? *at(r_e + 4u * kQ) : T(0);
      Quad<T> v = update<T, B_OR>(U0, U2, ym, yp, U1, odd, e, B_OR ? R0 : nB1);
      if (!fast) mask(v, true, odd ? pad1 : pad0);
      if (own_row) qstore(out + out3, v);
    }
    n1 = n2;
    n2 += (uint32_t)lay.slot_bytes;
    if (n2 == ring_end) n2 = ring_o;
    bar_n += 8u;
    if (bar_n == bar0 + 8u * kPairStages) {
      bar_n = bar0;
      par_n ^= 1u;
    }
    tog ^= kQ;
    odd = !odd;
    out += plane_elems;
    return true;
  };

  const int n_steps = nz + 6;
  using First = std::integral_constant<bool, false>;
  using Steady = std::integral_constant<bool, true>;
  int s = 0;
#pragma unroll 1
  for (; s < 6 && !aborted; s += 3)
    aborted = !(step(First(), s, P0, P1, P2, Q0, Q1, Q2, R0, R1, R2, U0, U1, U2) &&
                step(First(), s + 1, P1, P2, P0, Q1, Q2, Q0, R1, R2, R0, U1, U2, U0) &&
                step(First(), s + 2, P2, P0, P1, Q2, Q0, Q1, R2, R0, R1, U2, U0, U1));
#pragma unroll 1
  for (; s < n_steps && !aborted; s += 3) {
    if (!step(Steady(), s, P0, P1, P2, Q0, Q1, Q2, R0, R1, R2, U0, U1, U2)) { aborted = true; break; }
    if (s + 1 >= n_steps) break;
    if (!step(Steady(), s + 1, P1, P2, P0, Q1, Q2, Q0, R1, R2, R0, U1, U2, U0)) { aborted = true; break; }
    if (s + 2 >= n_steps) break;
    if (!step(Steady(), s + 2, P2, P0, P1, Q2, Q0, Q1, R2, R0, R1, U2, U0, U1)) { aborted = true; break; }
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
      for (uint32_t e = g_e; e < g_e1; e += blockDim.x) {
        const uint32_t ent = e == g_e ? g_ent0 : a.g_ent()[e];
        const double qe = e == g_e ? g_q0 : a.g_q()[e];
        const uint32_t at = ent & ~kGatherColourBit;
        const T val = (ent & kGatherColourBit) ? dst1[at] : dst0[at];
        const double t = qe * (double)val;
        sq += t;
        sp += t * t;
      }
    }
  }
  return !aborted;
}


}  // namespace tile
}  // namespace coulps
