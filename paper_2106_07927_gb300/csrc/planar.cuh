// Path aggregation and disparity selection on path planes: the route for P2 <= 255.
//
// With C(p,d) the matching cost, Eq. (sgm_path) is L_r(p,d) = C(p,d) + U_r(p,d) with
//   U_r(p,d) = min(L_r(q,d), L_r(q,d-1) + P1, L_r(q,d+1) + P1, m(q) + P2) - m(q) <= P2,
// so U_r fits a byte when P2 <= 255 and S(p,d) = R C(p,d) + sum_r U_r(p,d) <= 4080 for R <= 8.
// The U_r are stored as planes of bytes laid out as the cost volume, and the selection stage reads
// the planes once and adds them up. Nothing is accumulated with atomics: eight passes of adds into
// a 2-byte S run at the rate the L2 reduces at, which measured 2.8 TB/s into 480 MB and 4.0-4.4
// TB/s into 60 MB, against 6.3 TB/s for plain stores of half the bytes, and S need not be cleared.
//
// Pairs of opposite directions. Where two values fit a byte (2 P2 <= 255) a direction and its
// opposite share one plane: their two warps, side by side in one block, walk the same lines from
// both ends. Up to the middle each stores its U; they meet at a barrier; past it each adds its U to
// the other's, which it reads ahead with the costs (the most recently stored first, so much of it
// is still in the L2). The selection then reads 4 planes instead of 8. 5 bytes per disparity
// estimate are held (volume of sums: 3), 9 when P2 is 128 .. 255.
//
// Pair order. The volumes keep a pixel's D bytes together, but byte 2 i + s holds disparity
// i + s D/2 (i < D/2, s = 0, 1). Unpacking two bytes gives the word (L(i), L(i + D/2)) of two
// 16-bit values, and the words of disparities i - 1 and i + 1 are the neighbouring words as they
// stand: no byte permute is needed to pair a value with its neighbours (the natural order takes
// one per word), only the words at a lane's ends come from the neighbouring lanes, and at the two
// ends of the range the halves of the opposite end are put beside a sentinel.
// What bounds it (1242 x 375, D = 128, 8 paths): bytes. The stage reads the cost 8 times and writes
// 8 planes' worth, plus the other directions' halves, 20 bytes per disparity estimate (16 when not
// paired), at 7.7 TB/s through the L2; the selection reads 5 (9) from DRAM. Aggregation and
// selection together take 0.206 ms paired, 0.210 ms with 8 planes, and took 0.249 ms with atomic
// adds into S; at 1920 x 1080, D = 256: 2.03, 2.09 and 3.46 ms.
#pragma once
#include <type_traits>

#include "aggregate.cuh"
#include "common.cuh"

namespace r2t {

__device__ __forceinline__ uint32_t vmin3(uint32_t a, uint32_t b, uint32_t c) {
  return __vimin3_u16x2(a, b, c);
}
// min(a + b, c) per half
__device__ __forceinline__ uint32_t vaddmin(uint32_t a, uint32_t b, uint32_t c) {
  return __viaddmin_u16x2(a, b, c);
}

// Word exchange of a group of nl lanes holding consecutive words: the lanes to read the word
// before a lane's first one and after its last one from, and the byte selectors that keep it
// (0x3210) or, at the ends of the range, put the half that belongs there beside the sentinel
// (the last word's low half d = D/2 - 1 precedes the high half of word 0; the first word's high
// half d = D/2 follows the low half of the last word).
struct Ends {
  int up, dn;
  uint32_t sel_up, sel_dn;
  __device__ __forceinline__ Ends(int lane, int lig, int nl, bool in) {
    const int base = lane - lig;
    up = !in ? lane : base + (lig == 0 ? nl - 1 : lig - 1);
    dn = !in ? lane : base + (lig == nl - 1 ? 0 : lig + 1);
    sel_up = lig == 0 ? 0x1054u : 0x3210u;
    sel_dn = lig == nl - 1 ? 0x5432u : 0x3210u;
  }
  __device__ __forceinline__ uint32_t prev(uint32_t last) const {
    return __byte_perm(__shfl_sync(0xffffffffu, last, up), kSent, sel_up);
  }
  __device__ __forceinline__ uint32_t next(uint32_t first) const {
    return __byte_perm(__shfl_sync(0xffffffffu, first, dn), kSent, sel_dn);
  }
};

// The kernels' blocks are one pair of warps, the two opposite directions of the same lines. (Blocks
// of several pairs that met at barriers numbered at run time held all 16 of a block's barriers each,
// which left 4 blocks to an SM.)
constexpr int kPairThreads = 64;

// Two opposite directions share a plane.
__host__ __device__ inline bool planar_paired(const Method& mt) { return 2 * mt.P2 <= 255; }
__host__ __device__ inline int planar_planes(const Method& mt) {
  return planar_paired(mt) ? mt.num_paths / 2 : mt.num_paths;
}

// ------------------------------------------------------------------------------- rows
// Costs of a row (and the other direction's U) are copied to shared memory a chunk of pixels at a
// time (one contiguous run), three chunks ahead.
constexpr int kRowStages = 4, kRowChunk = 8;
// Ring of one warp of 32 / lpl chains: what their D takes, since it decides how many blocks of both
// kernels share an SM (803 x 601, D = 144: 350 -> 314 us a call against rings for full lanes; chunks of
// 4 pixels at D > 128: 2513 x 122, D = 240 380 -> 415).
__host__ __device__ inline int planar_ring_smem(int D, int lpl) {
  return 2 * kRowStages * kRowChunk * (32 / lpl) * D;
}
// Byte of a pixel where the lane with number lig of a chain starts, NW words a lane (0 for a lane past
// the chain's words, whose reads are not used).
__host__ __device__ inline int planar_lane_at(int lig, int NW, int D) {
  return lig < D / (2 * NW) ? lig * 2 * NW : 0;
}
// Pixel at which the two directions of a row meet when they share a plane.
__host__ __device__ inline int planar_row_mid(int W) { return (W / 2) & ~(kRowChunk - 1); }
// Warps of one direction: 32 / lanes rows each.
__host__ __device__ inline int planar_row_warps(int H, int lpl) {
  const int cpw = 32 / lpl;
  return (H + cpw - 1) / cpw;
}

template <int NW>
struct PairBytes {};  // a lane's 2 NW bytes of one pixel
template <>
struct PairBytes<1> {
  typedef uint32_t T;
  static __device__ __forceinline__ T load(uint32_t a) {
    unsigned short r;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(r) : "r"(a));
    return r;
  }
  static __device__ __forceinline__ void unpack(T r, uint32_t (&c)[1]) {
    c[0] = __byte_perm(r, 0u, 0x4140);
  }
  static __device__ __forceinline__ T pack(const uint32_t (&u)[1]) {
    return __byte_perm(u[0], 0u, 0x4420);
  }
  static __device__ __forceinline__ void add(T& a, T b) { a += b; }
  static __device__ __forceinline__ void store(uint8_t* p, T v) {
    *reinterpret_cast<unsigned short*>(p) = (unsigned short)v;
  }
};
template <>
struct PairBytes<2> {
  typedef uint32_t T;
  static __device__ __forceinline__ T load(uint32_t a) {
    T r;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(a));
    return r;
  }
  static __device__ __forceinline__ void unpack(T r, uint32_t (&c)[2]) { unpack4(r, c[0], c[1]); }
  static __device__ __forceinline__ T pack(const uint32_t (&u)[2]) {
    return __byte_perm(u[0], u[1], 0x6420);
  }
  static __device__ __forceinline__ void add(T& a, T b) { a += b; }
  static __device__ __forceinline__ void store(uint8_t* p, T v) {
    *reinterpret_cast<uint32_t*>(p) = v;
  }
};
template <>
struct PairBytes<4> {
  typedef uint2 T;
  static __device__ __forceinline__ T load(uint32_t a) {
    T r;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "r"(a));
    return r;
  }
  static __device__ __forceinline__ void unpack(T r, uint32_t (&c)[4]) {
    unpack4(r.x, c[0], c[1]);
    unpack4(r.y, c[2], c[3]);
  }
  static __device__ __forceinline__ T pack(const uint32_t (&u)[4]) {
    return make_uint2(__byte_perm(u[0], u[1], 0x6420), __byte_perm(u[2], u[3], 0x6420));
  }
  static __device__ __forceinline__ void add(T& a, T b) {
    a.x += b.x;
    a.y += b.y;
  }
  static __device__ __forceinline__ void store(uint8_t* p, T v) {
    *reinterpret_cast<uint2*>(p) = v;
  }
};

// Chains of one warp with few words per lane: groups of LPL lanes, lane member lig owns words
// [lig NW, (lig + 1) NW). FULL: D == 2 NW LPL. The chain of one step, L -> neighbour shuffle -> L, is
// its cost: the group minimum (one redux.sync when a chain takes the whole warp) runs beside it.
template <int NW, int LPL, bool FULL>
struct LongChain {
  typedef PairBytes<NW> PB;
  Ends ends;
  bool owns;  // the lane holds words of its chain
  uint32_t L[NW], mm;
  __device__ __forceinline__ LongChain(int lane, int D)
      : ends(lane, lane % LPL, FULL ? LPL : D / (2 * NW), FULL || lane % LPL < D / (2 * NW)),
        owns(FULL || lane % LPL < D / (2 * NW)) {
    restart();
  }
  // the next step starts a line of the path: L = C
  __device__ __forceinline__ void restart() {
#pragma unroll
    for (int k = 0; k < NW; k++) L[k] = 0;
    mm = 0;
  }
  // One step with the costs raw; returns the lane's bytes of U.
  __device__ __forceinline__ typename PB::T step(typename PB::T raw, uint32_t P1P1,
                                                 uint32_t P2P2) {
    uint32_t cst[NW], U[NW], Ln[NW];
    PB::unpack(raw, cst);
    const uint32_t up = ends.prev(L[NW - 1]), dn = ends.next(L[0]);
    const uint32_t mP2 = mm + P2P2;
    uint32_t lmin = 0;
#pragma unroll
    for (int k = 0; k < NW; k++) {
      const uint32_t t =
          vmin2(k == 0 ? up : L[(k + NW - 1) % NW], k == NW - 1 ? dn : L[(k + 1) % NW]) + P1P1;
      U[k] = vmin3(t, L[k], mP2) - mm;  // halves >= m(q): no borrow
      Ln[k] = U[k] + cst[k];
      lmin = k == 0 ? Ln[0] : vmin2(lmin, Ln[k]);
    }
#pragma unroll
    for (int k = 0; k < NW; k++) L[k] = Ln[k];
    lmin = halves_min(lmin);
    if (!FULL) lmin = owns ? lmin : 0xFFFFFFFFu;
    mm = group_min<LPL>(lmin);
    return PB::pack(U);
  }
};

// Rows y0 .. y0 + 32 / LPL - 1 in one direction, one per group of LPL lanes. ring: planar_ring_smem
// bytes of this warp. The two directions meet at pixel `mid` (a multiple of the
// chunk) when they share a plane.
template <int NW, int LPL, bool FULL, bool BACK>
__device__ __forceinline__ void planar_rows(const Problem& pb, const Method& mt, int y0,
                                            uint8_t* ring) {
  typedef PairBytes<NW> PB;
  constexpr int CPW = 32 / LPL, G = kRowChunk;
  const int lane = threadIdx.x & 31, c = lane / LPL, lig = lane % LPL;
  const int W = pb.W, D = FULL ? 2 * NW * LPL : pb.D;
  const int y = y0 + c;
  LongChain<NW, LPL, FULL> chain(lane, D);
  const bool valid = y < pb.H, active = valid && chain.owns;
  const int at = planar_lane_at(lig, NW, D);
  const bool paired = planar_paired(mt);
  const int64_t row = (int64_t)(valid ? y : 0) * W * D;
  const uint32_t slot_bytes = (uint32_t)(CPW * G * D);
  const uint32_t other = kRowStages * slot_bytes;  // the other direction's U behind the costs
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)(c * G * D);
  const uint32_t P1P1 = (uint32_t)mt.P1 * 0x10001u, P2P2 = (uint32_t)mt.P2 * 0x10001u;
  uint8_t* const plane =
      reinterpret_cast<uint8_t*>(pb.agg) + (BACK && !paired ? pb.plane : 0) + row;
  const uint8_t* const cost = pb.cost + row;
  const int64_t nde = (int64_t)W * pb.H * D;  // extent of the volumes (range checks)
  (void)nde;

  // pixels [q0, q1), walked from q1 - 1 down when BACK; add: onto the other direction's U
  auto walk = [&](int q0, int q1, auto add_) {
    constexpr bool add = decltype(add_)::value;
    const int len = q1 - q0, nch = (len + G - 1) / G;
    // chunk k: n pixels from p
    auto first = [&](int k, int n) { return BACK ? q1 - k * G - n : q0 + k * G; };
    auto copy = [&](int k) {
      if (k < nch) {
        const int n = min(G, len - k * G), pieces = n * D / 16;
        const int64_t o = (int64_t)first(k, n) * D;
        const uint32_t dst = ring_s + (uint32_t)(k & (kRowStages - 1)) * slot_bytes;
#pragma unroll
        for (int v = 0; v < NW; v++) {  // pieces <= D / 2 <= NW LPL
          const int i = 16 * (lig + LPL * v);
          if (valid && i < 16 * pieces) {
            if (R2T_CHECKED(pb, cost + o + i, 16, pb.cost, nde, 1))
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i),
                           "l"(cost + o + i)
                           : "memory");
            if (add && R2T_CHECKED(pb, plane + o + i, 16, pb.agg, planar_planes(mt) * nde, 1))
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + other + i),
                           "l"(plane + o + i)
                           : "memory");
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto step = [&](typename PB::T raw, typename PB::T oth, uint8_t* out) {
      typename PB::T u = chain.step(raw, P1P1, P2P2);
      if (add) PB::add(u, oth);  // bytes add without a carry
      if (active && R2T_CHECKED(pb, out, 2 * NW, pb.agg, planar_planes(mt) * nde, 2))
        PB::store(out, u);
    };
#pragma unroll
    for (int k = 0; k < kRowStages - 1; k++) copy(k);
    for (int k = 0; k < nch; k++) {
      __syncwarp();  // every lane is done with the slot refilled below
      copy(k + kRowStages - 1);
      asm volatile("cp.async.wait_group 3;" ::: "memory");
      __syncwarp();
      const int n = min(G, len - k * G);
      const uint32_t slot = ring_s + (uint32_t)(k & (kRowStages - 1)) * slot_bytes +
                            (uint32_t)(at + (BACK ? (n - 1) * D : 0));
      uint8_t* out = plane + (int64_t)(first(k, n) + (BACK ? n - 1 : 0)) * D + at;
      if (n == G) {
        typename PB::T raw[G], oth[G];
#pragma unroll
        for (int u = 0; u < G; u++) raw[u] = PB::load(slot + (BACK ? -u : u) * D);
#pragma unroll
        for (int u = 0; u < G; u++) {
          oth[u] = typename PB::T();
          if (add) oth[u] = PB::load(slot + other + (BACK ? -u : u) * D);
        }
#pragma unroll
        for (int u = 0; u < G; u++) step(raw[u], oth[u], out + (BACK ? -u : u) * (int64_t)D);
      } else {
        for (int u = 0; u < n; u++) {
          const uint32_t a = slot + (BACK ? -u : u) * D;
          typename PB::T oth = typename PB::T();
          if (add) oth = PB::load(a + other);
          step(PB::load(a), oth, out + (BACK ? -u : u) * (int64_t)D);
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
  };
  const int mid = planar_row_mid(W);
  if (paired) {
    walk(BACK ? mid : 0, BACK ? W : mid, std::false_type());
    __syncthreads();
    walk(BACK ? 0 : mid, BACK ? mid : W, std::true_type());
  } else {
    walk(0, W, std::false_type());
  }
}

// ------------------------------------------------------------------------------- sheared columns
// The sheared chains of aggregate.cuh on planes, in one of two shapes (planar_shear_dpl):
// - planar_shear: NL = D / 16 lanes per chain, 8 words (16 disparities, 16 bytes of each volume) per
//   lane; groups of any number of lanes share a warp (D = 144: three chains of 9 lanes). A lane
//   copies its own 16 cost bytes of a step to shared memory 6 steps ahead and stores its own 16
//   bytes of U, so the lanes of a warp never wait for each other's copies; adjacent chains sit on
//   adjacent pixels, so both are contiguous over the warp. The fewest instructions per estimate.
// - planar_long: one chain per warp, as the row paths. The shortest step, for small images.
constexpr int kPlanarRing = 8;
constexpr int kShearGroup = 2;                          // steps between two tests for a wrap
constexpr int kShearAhead = kPlanarRing - kShearGroup;  // steps from a cost copy to its use
__host__ __device__ inline int planar_shear_smem() { return kPlanarRing * 1024; }  // of one warp
// Pairs of warps: the two opposite directions of a group of adjacent chains, or of one chain.
__host__ __device__ inline int planar_shear_pairs(int W, int D, int num_paths) {
  const int ch = 32 / (D / 16);
  return shear_kinds(num_paths) / 2 * ((W + ch - 1) / ch);
}
__host__ __device__ inline int planar_long_pairs(int W, int num_paths) {
  return shear_kinds(num_paths) / 2 * W;
}
// Words per lane of the one-chain-per-warp shape.
__host__ __device__ inline int planar_long_words(int D) { return D <= 64 ? 1 : (D <= 128 ? 2 : 4); }
// Shape of a launch over pairs of that many chains in all (setting shear_dpl): 8 for one chain per
// warp, 16 otherwise. The line lies where the warps of the 16-disparity shape leave most schedulers
// with one or none, so that a step's latency decides, unless the rows' chains, which run beside, are
// the longer ones (W > 2 H) and only the work counts. us per call with one chain per warp and with 16
// disparities per lane, 8 paths: 160x120, D = 32 (960 chains) 38, 44; 320x375, D = 64 (1920) 65, 77, D
// = 128 84, 94, D = 224 137, 128; 413x307, D = 48 (2478) 83, 80; 640x480, D = 64 (3840) 138, 132;
// W > 2 H: 320x120, D = 32 (1920) 43, 40, D = 256 65, 53; 4 paths: 413x375, D = 144 (826) equal;
// 640x375, D = 64 (1280) 0.90 of the other, D = 144 147, 123; 1000x375, D = 128 (2000) 148, 146, D =
// 256 265, 247. Tall pairs of large D would gain from it past the line too (413x900, D = 256, 2478
// chains 397, 528); D between 160 and 240 lose up to 8 % of a call at it (320x375).
// wmin: the smallest width among them (a chunk of the one-chain-per-warp walk wraps around the image
// edge at most once); flat: one of them has W > 2 H.
constexpr int64_t kLongChains = 2200;
inline int planar_shear_dpl(int64_t chains, int wmin, bool flat) {
  return wmin >= kRowChunk && !flat && chains <= kLongChains ? 8 : 16;
}

// Minimum over the NL lanes of a group of a value whose halves are equal. Any NL: rotations by
// 1, 2, 3 and then by multiples of 4 lanes (overlaps do no harm to a minimum).
template <int NL>
struct GroupMin {
  int s1, s2, s3, s4, s8, s12;
  __device__ __forceinline__ GroupMin(int lane, int lig, bool in) {
    const int base = lane - lig;
    auto at = [&](int k) { return in ? base + (lig + k) % NL : lane; };
    s1 = at(1);
    s2 = at(2);
    s3 = at(3);
    s4 = at(4);
    s8 = at(8);
    s12 = at(12);
  }
  static __device__ __forceinline__ uint32_t g(uint32_t v, int s) {
    return __shfl_sync(0xffffffffu, v, s);
  }
  __device__ __forceinline__ uint32_t operator()(uint32_t v) const {
    if constexpr ((NL & (NL - 1)) == 0) {
      return group_min<NL>(v);
    } else {
      if constexpr (NL == 3) {
        v = vmin3(v, g(v, s1), g(v, s2));
      } else {
        const uint32_t a = g(v, s1), b = g(v, s2), e = g(v, s3);
        v = vmin2(vmin3(v, a, b), e);
      }
      if constexpr (NL > 12) {
        const uint32_t a = g(v, s4), b = g(v, s8), e = g(v, s12);
        v = vmin2(vmin3(v, a, b), e);
      } else if constexpr (NL > 8) {
        v = vmin3(v, g(v, s4), g(v, s8));
      } else if constexpr (NL > 4) {
        v = vmin2(v, g(v, s4));
      }
      return v;
    }
  }
};

// One direction (back: the upward one) of pair `item`: adjacent chains of one kind. Groups of GS
// steps in which no chain of the warp wraps around the image edge (nor its copies, PF steps ahead)
// and which are not among the last rows of the walk take the fast path; te is the first step of
// the next group that does not. Steps are counted from the start of each of the walk's two parts.
template <int NL>
__device__ __forceinline__ void planar_shear(const Problem& pb, const Method& mt, int item,
                                             bool back, uint8_t* ring) {
  constexpr int NP = 8, LB = 16, D = LB * NL, CH = 32 / NL;
  constexpr int GS = kShearGroup, KS = kPlanarRing, PF = kShearAhead;
  constexpr int SLOT = 1024, OTHER = 512;  // costs, then the other direction's U
  const int lane = threadIdx.x & 31, c = lane / NL, lig = lane - c * NL;
  const bool in = c < CH;
  const int W = pb.W, H = pb.H;
  const int ng = (W + CH - 1) / CH;
  const int kp = item / ng;  // kinds 2 kp (down) and 2 kp + 1 (up)
  const int j = (item - kp * ng) * CH + c;
  const int sh = kp == 0 ? 0 : (kp == 1 ? 1 : -1);
  const bool paired = planar_paired(mt);
  const int dy = back ? -1 : 1, dx = back ? -sh : sh;
  const int ystart = back ? H - 1 : 0;
  const Ends ends(lane, lig, NL, in);
  const GroupMin<NL> gmin(lane, lig, in);
  const uint32_t P1P1 = (uint32_t)mt.P1 * 0x10001u, P2P2 = (uint32_t)mt.P2 * 0x10001u;
  const uint32_t own = (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)(LB * lane);
  // offsets into a volume, modulo 2^32 (planar volumes are smaller, see layout.h)
  const uint32_t stride = (uint32_t)((dy * W + dx) * D);
  const uint32_t wrap = (uint32_t)(dx * W * D);  // taken off where a chain wraps around the edge
  const int64_t nde = (int64_t)W * H * D;        // extent of the volumes (range checks)
  (void)nde;
  constexpr int kNever = 0x40000000;
  const uint8_t* const cost = pb.cost;
  uint8_t* const plane = reinterpret_cast<uint8_t*>(pb.agg) +
                         (int64_t)(paired ? 1 + kp : 2 + 2 * kp + (back ? 1 : 0)) * pb.plane;
  const bool act = in && j < W;
  int x = act ? (j + sh * ystart) % W : 0;
  if (x < 0) x += W;
  uint32_t wo = (uint32_t)(((int64_t)ystart * W + x) * D + LB * lig);  // offset of the next store
  int tw = !act || dx == 0 ? kNever : (dx > 0 ? W - x : x + 1);  // step of the chain's next wrap
  uint32_t L[NP], mm = 0;
#pragma unroll
  for (int k = 0; k < NP; k++) L[k] = 0;
  // n steps; add: onto the other direction's U
  auto walk = [&](int n, auto add_) {
    constexpr bool add = decltype(add_)::value;
    uint32_t ro = wo;  // offset of the next cost copy, and the step of its next wrap
    int tr = tw;
    auto fetch = [&](uint32_t o, uint32_t slot) {
      if (act && R2T_CHECKED(pb, cost + o, LB, pb.cost, nde, 3))
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot), "l"(cost + o)
                     : "memory");
      if (add && act && R2T_CHECKED(pb, plane + o, LB, pb.agg, planar_planes(mt) * nde, 3))
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot + OTHER),
                     "l"(plane + o)
                     : "memory");
    };
    auto copy_step = [&](int t) {  // any step (past the last one: nothing)
      if (t < n) {
        if (tr == t) {
          ro -= wrap;
          tr += W;
        }
        fetch(ro, own + (uint32_t)((t & (KS - 1)) * SLOT));
        ro += stride;
      }
    };
    // one step from the values La to Lb (a group's steps return to the same registers)
    auto step = [&](uint32_t slot, uint32_t o, const uint32_t (&La)[NP], uint32_t (&Lb)[NP]) {
      const uint4 raw = lds128(slot);
      uint4 oth = make_uint4(0, 0, 0, 0);
      if (add) oth = lds128(slot + OTHER);
      const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w}, ow[4] = {oth.x, oth.y, oth.z, oth.w};
      const uint32_t up = ends.prev(La[NP - 1]), dn = ends.next(La[0]);
      const uint32_t mP2 = mm + P2P2;
      uint32_t lm = 0, u[4];
#pragma unroll
      for (int k = 0; k < NP; k += 2) {
        uint32_t c0, c1;
        unpack4(rw[k / 2], c0, c1);
        const uint32_t t0 = vmin2(k == 0 ? up : La[(k + NP - 1) % NP], La[k + 1]) + P1P1;
        const uint32_t t1 = vmin2(La[k], k + 2 < NP ? La[(k + 2) % NP] : dn) + P1P1;
        const uint32_t u0 = vmin3(t0, La[k], mP2) - mm;  // halves >= m(q): no borrow
        const uint32_t u1 = vmin3(t1, La[k + 1], mP2) - mm;
        Lb[k] = u0 + c0;
        Lb[k + 1] = u1 + c1;
        lm = k == 0 ? vmin2(Lb[0], Lb[1]) : vmin3(lm, Lb[k], Lb[k + 1]);
        u[k / 2] = __byte_perm(u0, u1, 0x6420);
        if (add) u[k / 2] += ow[k / 2];  // bytes add without a carry
      }
      if (act && R2T_CHECKED(pb, plane + o, LB, pb.agg, planar_planes(mt) * nde, 4)) {
        const uint4 v = make_uint4(u[0], u[1], u[2], u[3]);
        // bytes that this kernel does not read again leave the L2 first
        if (add || !paired)
          __stcs(reinterpret_cast<uint4*>(plane + o), v);
        else
          *reinterpret_cast<uint4*>(plane + o) = v;
      }
      mm = gmin(halves_min(lm));
    };
    // first step of the next group with an event, from a group's first step t on
    const int tail = n < PF + GS ? 0 : (n - PF) & ~(GS - 1);  // its copies reach past the end
    auto next_event = [&](int t) {
      const int e =
          (int)__reduce_min_sync(0xffffffffu, (unsigned)max(min(tw, tr - PF), 0)) & ~(GS - 1);
      return max(min(e, tail), t);
    };

#pragma unroll
    for (int s = 0; s < PF; s++) {
      copy_step(s);
      if (s % GS == GS - 1) asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int te = next_event(0);
    uint32_t rs = 0;  // ring offset of step t
    for (int t = 0; t < n; t += GS) {
      const uint32_t slot = own + rs, ahead = own + ((rs + PF * SLOT) & (KS * SLOT - 1));
      rs = (rs + GS * SLOT) & (KS * SLOT - 1);
      uint32_t M[NP];
      if (t < te) {
        fetch(ro, ahead);
        fetch(ro + stride, ahead + SLOT);
        ro += GS * stride;
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 3;" ::: "memory");
        step(slot, wo, L, M);
        step(slot + SLOT, wo + stride, M, L);
        wo += GS * stride;
      } else {
#pragma unroll
        for (int u = 0; u < GS; u++) copy_step(t + PF + u);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 3;" ::: "memory");
        for (int u = 0; u < GS && t + u < n; u++) {
          if (tw == t + u) {  // a new line of the path enters: L = C
#pragma unroll
            for (int k = 0; k < NP; k++) L[k] = 0;
            mm = 0;
            wo -= wrap;
            tw += W;
          }
          step(slot + (uint32_t)(u * SLOT), wo, L, M);
#pragma unroll
          for (int k = 0; k < NP; k++) L[k] = M[k];
          wo += stride;
        }
        te = next_event(t + GS);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    tw -= tw == kNever ? 0 : n;
  };
  if (paired) {
    const int n0 = back ? H - H / 2 : H / 2;  // the two directions meet in the middle
    walk(n0, std::false_type());
    __syncthreads();
    walk(H - n0, std::true_type());
  } else {
    walk(H, std::false_type());
  }
}

// One direction of sheared chain `item` (all chains of kind pair 0, then of 1 and 2), the whole warp
// on one chain. Costs are copied kRowChunk steps at a time, three chunks ahead, each lane the same
// 16-byte pieces of every chunk. W >= kRowChunk. ring: planar_ring_smem bytes of this warp.
template <int NW, bool FULL>
__device__ __forceinline__ void planar_long(const Problem& pb, const Method& mt, int item,
                                            bool back, uint8_t* ring) {
  typedef PairBytes<NW> PB;
  constexpr int G = kRowChunk;
  const int lane = threadIdx.x & 31;
  const int W = pb.W, H = pb.H, D = FULL ? 64 * NW : pb.D;
  const int kp = item / W;  // kinds 2 kp (down) and 2 kp + 1 (up)
  const int j = item - kp * W;
  const int sh = kp == 0 ? 0 : (kp == 1 ? 1 : -1);
  const bool paired = planar_paired(mt);
  const int dy = back ? -1 : 1, dx = back ? -sh : sh;
  const int ystart = back ? H - 1 : 0;
  LongChain<NW, 32, FULL> chain(lane, D);
  const int at = planar_lane_at(lane, NW, D);
  const uint32_t P1P1 = (uint32_t)mt.P1 * 0x10001u, P2P2 = (uint32_t)mt.P2 * 0x10001u;
  const uint32_t slot_bytes = (uint32_t)(G * D);
  const uint32_t other = kRowStages * slot_bytes;  // the other direction's U behind the costs
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
  // offsets into a volume, modulo 2^32 (planar volumes are smaller, see layout.h)
  const uint32_t stride = (uint32_t)((dy * W + dx) * D);
  const uint32_t wrap = (uint32_t)(dx * W * D);  // taken off where the chain wraps around the edge
  const int64_t nde = (int64_t)W * H * D;        // extent of the volumes (range checks)
  (void)nde;
  const uint8_t* const cost = pb.cost;
  uint8_t* const plane = reinterpret_cast<uint8_t*>(pb.agg) +
                         (int64_t)(paired ? 1 + kp : 2 + 2 * kp + (back ? 1 : 0)) * pb.plane;
  const int ppx = D / 16;  // 16-byte pieces of a pixel; G ppx <= 32 NW of a chunk
  int pu[NW], pq[NW];      // the lane's pieces: step in the chunk, piece of the pixel
#pragma unroll
  for (int v = 0; v < NW; v++) {
    pu[v] = (lane + 32 * v) / ppx;
    pq[v] = (lane + 32 * v) - pu[v] * ppx;
  }
  int x = (j + sh * ystart) % W;  // column of the next step
  if (x < 0) x += W;
  uint32_t wo = (uint32_t)(((int64_t)ystart * W + x) * D);  // and its offset
  auto wrapped = [&](int& xx, uint32_t& o) {  // xx in (-W, 2 W)
    if (xx >= W || xx < 0) {
      xx -= dx * W;
      o -= wrap;
    }
  };
  bool fresh = false;  // the next step starts a line
  // n steps; add: onto the other direction's U
  auto walk = [&](int n, auto add_) {
    constexpr bool add = decltype(add_)::value;
    const int nch = (n + G - 1) / G;
    int px[NW];  // column and offset of the lane's pieces of the next chunk to copy
    uint32_t po[NW];
#pragma unroll
    for (int v = 0; v < NW; v++) {
      px[v] = x + dx * pu[v];
      po[v] = wo + pu[v] * stride;
      wrapped(px[v], po[v]);
      po[v] += 16 * pq[v];
    }
    auto copy = [&](int k) {
      const uint32_t dst = ring_s + (uint32_t)(k & (kRowStages - 1)) * slot_bytes;
#pragma unroll
      for (int v = 0; v < NW; v++) {
        if (pu[v] < G && k * G + pu[v] < n) {
          const uint32_t a = dst + 16 * (lane + 32 * v), o = po[v];
          if (R2T_CHECKED(pb, cost + o, 16, pb.cost, nde, 3))
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(cost + o)
                         : "memory");
          if (add && R2T_CHECKED(pb, plane + o, 16, pb.agg, planar_planes(mt) * nde, 3))
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a + other),
                         "l"(plane + o)
                         : "memory");
        }
        px[v] += G * dx;
        po[v] += G * stride;
        wrapped(px[v], po[v]);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto step = [&](typename PB::T raw, typename PB::T oth, uint32_t o) {
      typename PB::T u = chain.step(raw, P1P1, P2P2);
      if (add) PB::add(u, oth);  // bytes add without a carry
      uint8_t* const out = plane + o + at;
      if (chain.owns && R2T_CHECKED(pb, out, 2 * NW, pb.agg, planar_planes(mt) * nde, 4))
        PB::store(out, u);
    };
#pragma unroll
    for (int k = 0; k < kRowStages - 1; k++) copy(k);
    for (int k = 0; k < nch; k++) {
      __syncwarp();  // every lane is done with the slot refilled below
      copy(k + kRowStages - 1);
      asm volatile("cp.async.wait_group 3;" ::: "memory");
      __syncwarp();
      const uint32_t slot = ring_s + (uint32_t)(k & (kRowStages - 1)) * slot_bytes +
                            (uint32_t)at;
      const int m = min(G, n - k * G);
      const int last = x + G * dx;
      if (m == G && !fresh && last < W && last >= 0) {  // no line starts in or after the chunk
        typename PB::T raw[G], oth[G];
#pragma unroll
        for (int u = 0; u < G; u++) raw[u] = PB::load(slot + u * D);
#pragma unroll
        for (int u = 0; u < G; u++) {
          oth[u] = typename PB::T();
          if (add) oth[u] = PB::load(slot + other + u * D);
        }
#pragma unroll
        for (int u = 0; u < G; u++) {
          step(raw[u], oth[u], wo);
          wo += stride;
        }
        x = last;
      } else {
        for (int u = 0; u < m; u++) {
          if (fresh) chain.restart();
          const uint32_t a = slot + u * D;
          typename PB::T oth = typename PB::T();
          if (add) oth = PB::load(a + other);
          step(PB::load(a), oth, wo);
          wo += stride;
          x += dx;
          fresh = x >= W || x < 0;
          wrapped(x, wo);
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
  };
  if (paired) {
    const int n0 = back ? H - H / 2 : H / 2;  // the two directions meet in the middle
    walk(n0, std::false_type());
    __syncthreads();
    walk(H - n0, std::true_type());
  } else {
    walk(H, std::false_type());
  }
}

// ------------------------------------------------------------------------------- selection
// Sum of the planes, D^L and the tile's share of D^R for T consecutive pixels of a row. The sums,
// times 16, are put in shared memory in natural order, two to a word, at a pitch of D/2 + 1 words
// (odd: both the pixels' rows and the diagonals of D^R are read without bank conflicts). Word k of
// pixel p holds d = 2k and 2k + 1: along the diagonal p = t + 2k its low halves belong to target
// x' = t and its high halves to t - 1. A thread scans one pixel's words (D^L) or one diagonal
// (D^R), 16 words at a time with the word's number in the low 4 bits of each half, so one
// instruction adds the number and takes the minimum of two sums; the least key has the least
// sum and, among equal ones, the smallest d.
// Pixels of a tile: whole blocks of 16 words along a diagonal, at most T and at most 29 KB of sums, past
// which the SM has too little left for the L1, which holds the loads in flight. Stage us with 32, 64,
// 96, 128 pixels, 4 planes, 1281 x 720: D = 64 98, 68, 61, 55; D = 128 121, 100, 100, 115; D = 160 147,
// 129, 152, 154; D = 224 182, 166, 174, 184; D = 256 195, 215, 219, -; 1920 x 1080: D = 128 260, 221,
// 219, 234; D = 256 430, 461, 466, -; 8 planes: D = 128 430, 397, 385, 406; D = 256 794, 797, 842, -.
// From 320 x 240 to 1920 x 1080 and 700 x 2000 the choice is within 4 % of the best of 32 .. 256 for D
// >= 64 (within the clock's 2 us on the small ones). Below it T is the bound, and 256 pixels would
// take 0.8 of the stage at D = 16.
__host__ __device__ inline int planar_wta_px(int D, int T) {
  const int cap = (29500 / (4 * (D / 2 + 1))) & ~31;
  return T < cap ? T : cap;
}
__host__ __device__ inline size_t planar_wta_smem(int D, int T) {
  return (size_t)T * (D / 2 + 1) * 4 + (size_t)(T + D) * 8;
}

// A word no sum can be (S = 0xFFF, and adding a word's number does not carry).
constexpr uint32_t kNoSum = 0xFFF0FFF0u;

// Keys S << 8 | d of a scanned block of words k = kb + j: low halves are d = 2k, high ones 2k + 1.
__device__ __forceinline__ void block_keys(uint32_t acc, int kb, uint32_t& lo, uint32_t& hi) {
  const uint32_t l = acc & 0xFFFFu, h = acc >> 16;  // S << 4 | j
  lo = min(lo, ((l & 0xFFF0u) << 4) | (uint32_t)(2 * (kb + (int)(l & 15u)) & 255));
  hi = min(hi, ((h & 0xFFF0u) << 4) | (uint32_t)((2 * (kb + (int)(h & 15u)) + 1) & 255));
}

template <int R>  // planes; paths: how often the cost counts
__device__ __forceinline__ void planar_wta_tile(const Problem& pb, int paths, int item,
                                                uint8_t* smem, int T) {
  const int W = pb.W, D = pb.D, h = D / 2, pitch = h + 1;
  const int ntx = (W + T - 1) / T;
  // rows from both edges of the image inwards: the walks ended at the edges, so the planes' last
  // stored bytes may still be in the L2
  const int yi = item / ntx, x0 = (item - yi * ntx) * T;
  const int y = (yi & 1) ? pb.H - 1 - (yi >> 1) : yi >> 1;
  const int n = min(T, W - x0);
  const int64_t rowbase = (int64_t)y * W;
  uint32_t* S = reinterpret_cast<uint32_t*>(smem);
  uint32_t* klo = S + T * pitch;
  uint32_t* khi = klo + T + D;
  const int ppx = D / 16;
  {
    const int64_t base = (rowbase + x0) * D;
    const uint8_t* cost = pb.cost + base;
    const uint8_t* pl = reinterpret_cast<const uint8_t*>(pb.agg) + base;
    // exact i / ppx for i < 2^16 (2^32 / 1 does not fit: D = 16 takes i itself)
    const uint32_t inv = (uint32_t)((0xFFFFFFFFull + ppx) / ppx);
    for (int i = threadIdx.x; i < n * ppx; i += blockDim.x) {
      uint4 cw = make_uint4(0, 0, 0, 0), u[R];
      if (R2T_CHECKED(pb, cost + 16 * (int64_t)i, 16, pb.cost, pb.plane, 6))
        cw = __ldcs(reinterpret_cast<const uint4*>(cost) + i);
#pragma unroll
      for (int r = 0; r < R; r++) {
        u[r] = make_uint4(0, 0, 0, 0);
        if (R2T_CHECKED(pb, pl + r * pb.plane + 16 * (int64_t)i, 16, pb.agg, R * pb.plane, 6))
          u[r] = __ldcs(reinterpret_cast<const uint4*>(pl + r * pb.plane) + i);
      }
      const int px = ppx == 1 ? i : (int)__umulhi((uint32_t)i, inv), q = i - px * ppx;
      uint32_t* o = S + px * pitch + 4 * q;
      auto sum = [&](uint32_t cword, auto&& get, int j) {
        // bytes d, d + h, d + 1, d + 1 + h: the even bytes and the odd bytes are natural pairs
        uint32_t e = (cword & 0x00FF00FFu) * paths, f = __byte_perm(cword, 0u, 0x4341) * paths;
#pragma unroll
        for (int r = 0; r < R; r++) {
          const uint32_t w = get(r);
          e += w & 0x00FF00FFu;
          f += __byte_perm(w, 0u, 0x4341);
        }
        o[j] = e << 4;
        o[h / 2 + j] = f << 4;
      };
      sum(cw.x, [&](int r) { return u[r].x; }, 0);
      sum(cw.y, [&](int r) { return u[r].y; }, 1);
      sum(cw.z, [&](int r) { return u[r].z; }, 2);
      sum(cw.w, [&](int r) { return u[r].w; }, 3);
    }
  }
  for (int i = n * pitch + threadIdx.x; i < T * pitch; i += blockDim.x) S[i] = kNoSum;
  __syncthreads();
  // diagonals t = x0 - D + 1 + i; those of t < 0 have no target
  const int nd = n + D - 1;
  for (int i = threadIdx.x; i < n + nd; i += blockDim.x) {
    uint32_t lo, hi;
    if (i < n) {
      lo = hi = 0xFFFFFFFFu;
      const uint32_t* w = S + i * pitch;
      for (int kb = 0; kb < h; kb += 16, w += 16) {
        uint32_t acc = 0xFFFFFFFFu;
#pragma unroll
        for (int j = 0; j < 8; j++) acc = vaddmin(w[j], j * 0x10001u, acc);
        if (kb + 16 <= h) {  // h is a multiple of 8
#pragma unroll
          for (int j = 8; j < 16; j++) acc = vaddmin(w[j], j * 0x10001u, acc);
        }
        block_keys(acc, kb, lo, hi);
      }
      const int d = (int)(min(lo, hi) & 0xFFu);
      const int64_t p = rowbase + x0 + i;
      if (R2T_CHECKED(pb, pb.dl + p, 2, pb.dl, 2 * (int64_t)W * pb.H, 7)) pb.dl[p] = (uint16_t)d;
      if (pb.dlf) {
        float v = (float)d;
        if (d >= 1 && d <= D - 2) {
          const uint16_t* s = reinterpret_cast<const uint16_t*>(S + i * pitch) + d;
          const int s0 = s[0] >> 4, a = (s[-1] >> 4) - s0, b = (s[1] >> 4) - s0;
          v = __fadd_rn(v, __fdiv_rn((float)(a - b), (float)(2 * (a + b))));
        }
        if (R2T_CHECKED(pb, pb.dlf + p, 4, pb.dlf, 4 * (int64_t)W * pb.H, 7)) pb.dlf[p] = v;
      }
    } else {
      const int j = i - n, t = j - (D - 1);  // relative to x0
      lo = hi = 0xFFFFFFFFu;
      if (x0 + t >= 0) {
        // pixels p = t mod 2, + 2, ... of the tile, 16 at a time: words k = (p - t) / 2
        const int par = t & 1;
        int kb = (par - t) / 2;
        const uint32_t* w = S + par * pitch + kb;
        const int step = 2 * pitch + 1;
        for (int p = par; p < T; p += 32, kb += 16, w += 16 * step) {
          if (kb <= -16 || kb >= h) continue;
          uint32_t acc = 0xFFFFFFFFu;
          if (kb >= 0 && kb + 16 <= h) {
#pragma unroll
            for (int j = 0; j < 16; j++) acc = vaddmin(w[j * step], j * 0x10001u, acc);
          } else {
#pragma unroll
            for (int j = 0; j < 16; j++)
              if ((unsigned)(kb + j) < (unsigned)h)
                acc = vaddmin(w[j * step], j * 0x10001u, acc);
          }
          block_keys(acc, kb, lo, hi);
        }
      }
      klo[j] = lo;
      khi[j] = hi;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < nd; j += blockDim.x) {
    const int x = x0 - (D - 1) + j;
    if (x < 0) continue;
    const uint32_t k = min(klo[j], j + 1 < nd ? khi[j + 1] : 0xFFFFFFFFu);
    if (k >= 0xFFF00u) continue;
    if (!R2T_CHECKED(pb, pb.kr + rowbase + x, 4, pb.kr, 4 * (int64_t)W * pb.H, 9)) continue;
    if (x >= x0 && min(x + D - 1, W - 1) < x0 + n)
      pb.kr[rowbase + x] = k;
    else
      atomicMin(&pb.kr[rowbase + x], k);
  }
}

}  // namespace r2t
