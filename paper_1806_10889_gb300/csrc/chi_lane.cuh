// K_chi, sum-tree form: the intracellular module chi (arXiv 1806.10889,
// Sec. II-A1) over a work list of cells, G = 1..32 lanes of a warp per cell.
//
// Every cell keeps a tree of propensity sums.  With up to four lanes per cell
// a node has four children: the voxel totals are the leaves, S_{LV-1}[q] the
// total of the four voxels of quad q, S_l[i] that of four entries of S_{l+1};
// S_1 has four entries.  With eight lanes and more the upper nodes are as wide
// as the cell's lanes (8 or 16): a lane holds the prefix before its child, one
// compare, ballot and population count find the child (11 instructions for 3 or
// 4 bits, 26 for 2 in a four-ary node), the root's prefixes stay in registers,
// and an update is one predicated addition per lane.  An event descends from the
// root in the direct method's voxel-major order, finds the channel inside the
// voxel in closed form, changes one or two voxels and adds the two differences
// along their paths: 250 to 500 instructions, the most of which no lane can take
// off another.  The segmented kernel (chi_seg.cuh) finds a voxel with ballots and
// scans over 8 to 32 lanes, and its event loop (600 to 900 instructions) serves
// one to four cells; here an instruction serves up to 32 (G = 1).
//
// What the G lanes of a cell share out is the work that does not depend on
// the state: lane j of the cell draws the random numbers of event j of the
// next G (about 360 instructions), and computes its waiting time (120).  The
// waiting time only decides where the cell stops.  So the G events are applied
// first, the total propensity A before each kept by its lane, then all G
// waiting times are computed at once and added in order (by a scan of integers
// while the time's exponent stays the same); the events past the end of the
// step are undone (at most G a cell and step, on the counts only: the sums are
// not used again).  With few warps on an SM a helper warp beside each draws a
// batch ahead of it.
//
// Bound (one GB300, from ncu).  Few cells: the event chain -- one warp alone
// issues every 3.9 cycles, 260 instructions and 1,010 cycles an event with G =
// 32 (2,530 cycles in the segmented kernel; 371 and 1,320 with four-ary nodes
// and the times added one by one).  Cells of up to 256 voxels that fill the
// chip: issue (34 and 40 warp instructions an event with G = 1, 8x8 and 16x16
// voxels, 44 to 48% of the peak; 171 and 227 segmented) beside their scattered
// accesses (57% of the L1 wavefronts).  Larger ones that do: shared memory
// holds 8 warps an SM, 6 cycles an instruction of which 2.3 wait for the
// scattered leaves (43 instructions and 147 DRAM bytes an event, 1.4 TB/s; a
// dependent read and write a lane reaches 25 G/s in DRAM, an event makes two).
// Chi ms per step, segmented -> this kernel: 2x2 cells of 8x8 voxels 2.9 ->
// 1.10, 64x64 of 16x16 21.1 -> 9.1, 48x48 of 32x32 77.5 -> 31.0, 256x256 of 8x8
// 33.4 -> 7.9, 256x256 of 32x32 611 -> 130.
//
// Template parameters: MODEL 0 Notch-Delta without in-voxel binding (k_in =
// k_off = 0), 1 Notch-Delta, 2 promoter; LV the levels of the tree (V <= 4^LV,
// LV = 3, 4, 5); LEAF where the voxels live (chi_lane.h): shared memory (20
// bytes a voxel and the sums: the shortest chain); planes there, 16-bit counts
// and no totals (6 bytes a voxel: two to four times the cells; four lanes
// recompute the totals of the chosen quad, one each); or a scratch array with
// the upper sums in shared memory, so that hundreds of cells fit on an SM --
// records, total and packed counts of a voxel side by side, a quad one aligned
// 64-byte block; or sectors, 32 bytes a quad with its sum and 16-bit counts,
// the four quads under a shared sum one 128-byte line that an event reads
// whole, the four totals of the chosen quad recomputed, the sum and the changed
// count of one or two quads written (256x256 cells of 32x32 voxels, one state:
// 186 ms with records and 490 DRAM bytes an event, 136 when sectors took their
// place; later 122 and 147 bytes, against 132 with 32 bits a voxel and the sums of
// all four quads recomputed, 260 instructions more); G lanes per cell; HELP blocks
// an SM with a helper warp, 0: none.
//
// Planes against records: 48x48 cells of 32x32 voxels 44.2 -> 31.0 ms, 76x76 of
// 16x16 13.8 -> 11.1, 113x113 of them 19.8 -> 15.9 (an event's two dependent
// accesses to L2, 400 cycles each and more under load, become shared memory's 30).
//
// Limits.  Counts below the tissue's `small` keep every total below 2^52
// unchecked, and R below kLaneHill reads the Hill table unchecked.  With
// shared leaves a cell past either goes on with exact checks.  A packed cell
// (20 or 16 bits a count) goes on with limits of its own, taken from its largest
// counts when it is loaded and again when one is met (pick_limits; the event
// loop compares with them all the same, so that this costs a running tissue
// nothing).  Only where there are none -- counts past their field, R past the
// Hill table, totals near 2^52 -- it is left untouched and goes to the redo list,
// which the launcher runs through the segmented kernel from the same state and
// random streams.  Cells past `small` (hops at 100 and 600 D a voxel), redone and
// with their own limits: 256x180 of 16x16 voxels 55.5 -> 9.5 ms, 48x48 of 32x32
// 28.2 -> 6.9, 256x256 of 8x8 40.8 -> 8.6; with 2,500 R a voxel 54.1 -> 10.5 and,
// 128x160 of 32x32, 63.0 -> 10.0.
#pragma once
#include "chi_lane.h"
#include "early_launch.cuh"
#include "pair_end.h"
#include "tissue_dev.cuh"

namespace tsg {

namespace {

// Rates of the cell a lane runs, in registers.
template <int MODEL>
struct LaneRates {
  uint64_t hD, hN, hR, gD, gN, gR, kN;  // promoter: kN unused
  uint64_t k_in, k_off, tD, kd;         // MODEL 1: k_in, k_off; MODEL 2: k_in (k_a), tD, kd
  const uint64_t* hill;
  uint32_t small;
  __device__ __forceinline__ void load(const QRates& q) {
    hD = q.hopD;
    hN = q.hopN;
    hR = q.hopR;
    gD = q.gD;
    gN = q.gN;
    gR = q.gR;
    kN = q.kN;
    k_in = MODEL ? q.k_in : 0ull;
    k_off = MODEL == 1 ? q.k_off : 0ull;
    tD = MODEL == 2 ? q.tD : 0ull;
    kd = MODEL == 2 ? q.kd : 0ull;
    hill = q.hill;
    small = q.small;
  }
};

// Hill(R) from the table; counts past it are computed (their view is read
// from memory: never in a running tissue).
__device__ __forceinline__ uint64_t lane_hill(const uint64_t* hill, const TissueView* tv,
                                              uint32_t R) {
  return R < kHillTab ? __ldg(hill + R) : hill_direct(tv->q, R);
}

// Total propensity of a voxel with nn neighbours, modulo 2^64 (exact while
// the counts are below `small`; larger ones are checked by exact_ovf).
template <int MODEL>
__device__ __forceinline__ uint64_t lane_total(const LaneRates<MODEL>& q, const TissueView* tv,
                                               uint32_t D, uint32_t N, uint32_t R, uint32_t nn,
                                               bool centre) {
  uint64_t a = (q.gD + q.hD * nn) * D + (q.gN + q.hN * nn) * N;
  if (MODEL == 2) {
    const uint32_t F = static_cast<uint32_t>(centre) - R;
    a += q.tD * F + q.kd * R + q.k_in * (static_cast<uint64_t>(N) * F);
  } else {
    a += (q.gR + q.k_off + q.hR * nn) * R + lane_hill(q.hill, tv, R) + q.kN;
    if (MODEL == 1) a += q.k_in * (static_cast<uint64_t>(D) * N);
  }
  return a;
}

// Whether a voxel's total (or one of its products) reaches 2^52, for a voxel
// holding a count of `small` or more.
template <int MODEL>
__device__ __noinline__ bool exact_ovf(const TissueView* tv, uint32_t D, uint32_t N, uint32_t R,
                                       uint32_t nn, bool centre) {
  const QRates& q = tv->q;
  if ((D | N | R) < q.small) return false;
  uint64_t a, X;
  if (MODEL == 2) {
    const uint32_t F = static_cast<uint32_t>(centre) - R;
    a = q.tD * F + q.kd * R;
    X = static_cast<uint64_t>(N) * F;
  } else {
    a = hill_q(q, R) + q.kN;
    X = static_cast<uint64_t>(D) * N;
  }
  bool ovf = false;
  a += mul_lim(q.gD + q.hopD * nn, D, ovf);
  a += mul_lim(q.gN + q.hopN * nn, N, ovf);
  a += mul_lim(q.gR + q.hopR * nn, R, ovf);
  a += mul_lim(q.k_in, X, ovf);
  a += mul_lim(q.k_off, R, ovf);
  return ovf || (a >> 52) != 0ull;
}

// Limits of a cell's counts of D, N and R.
struct Limits {
  uint32_t D, N, R;
};

// The limits of a cell with packed counts, from the largest it holds: while every
// count stays below them, no total reaches 2^52, no count leaves its field
// (`most`) and no R the Hill table (most_r).  As a rule that is the tissue's
// `small`.  A cell past it gets limits of its own: records, compared by their
// bits, the next power of two each; else one for D and N and one for R, the
// largest counts times what 2^52 leaves room for (a total grows at most with
// the square of that; in single precision, 3% below).  False where there are
// none: the cell goes to the redo list.
template <int MODEL, int LEAF>
__device__ __forceinline__ bool pick_limits(const TissueView* tv, Limits m, Limits& l) {
  constexpr uint32_t most = LEAF == kLeafRecords ? kWordCount : kHalfCount;
  constexpr uint32_t most_r = MODEL == 2               ? most
                              : LEAF == kLeafRecords ? kHillTab
                                                     : kHillTab - 1u;
  const QRates& q = tv->q;
  if (LEAF != kLeafRecords) m.D = m.N = max(m.D, m.N);
  l.D = l.N = min(q.small, most);
  l.R = min(q.small, most_r);
  if (max(m.D, m.N) < l.D && m.R < l.R) return true;
  if (max(m.D, m.N) >= most || m.R >= most_r) return false;
  auto up = [](uint32_t x) { return LEAF == kLeafRecords ? 2u << (31 - __clz(x | 1)) : x + 1u; };
  l = Limits{up(m.D), up(m.N), up(m.R)};
  const float fD = static_cast<float>(l.D), fN = static_cast<float>(l.N);
  float a = __ull2float_rn(q.gD + 4u * q.hopD) * fD + __ull2float_rn(q.gN + 4u * q.hopN) * fN;
  if (MODEL == 2) {
    a += __ull2float_rn(q.tD + q.kd) + __ull2float_rn(q.k_in) * fN;
  } else {
    a += __ull2float_rn(q.gR + q.k_off + 4u * q.hopR) * static_cast<float>(l.R) +
         __ull2float_rn(__ldg(q.hill) + q.kN);  // the table falls with R
    if (MODEL == 1) a += __ull2float_rn(q.k_in) * (fD * fN);
  }
  float f = 0x1.fp51f / a;
  if (!(f >= 1.0f)) return false;
  if (LEAF != kLeafRecords) {
    f = fminf(MODEL == 1 ? sqrtf(f) : f, 64.0f) * 0.99f;
    l.D = l.N = min(most, max(l.D, static_cast<uint32_t>(fD * f)));
    l.R = min(most_r, max(l.R, static_cast<uint32_t>(static_cast<float>(l.R) * f)));
  }
  return true;
}

// Whether the event that changed v (and u) took a count past its maximum or
// a total past its limit (shared leaves).
template <int MODEL>
__device__ __noinline__ bool past_limits(const TissueView* tv, const int32_t* cp, uint32_t ps,
                                         const unsigned char* lut, uint32_t v, uint32_t u,
                                         uint32_t centre) {
  bool o = false;
  for (int k = 0; k < 2; ++k) {
    const uint32_t x = k ? u : v;
    const uint32_t D = static_cast<uint32_t>(cp[x]), N = static_cast<uint32_t>(cp[ps + x]);
    const uint32_t R = static_cast<uint32_t>(cp[2u * ps + x]);
    o |= exact_ovf<MODEL>(tv, D, N, R, lut[x] >> 4, MODEL == 2 && x == centre);
    o |= max(D, max(N, R)) > static_cast<uint32_t>(kCountMax);
  }
  return o;
}

// What the two warps of a block with a helper exchange.
struct LaneExchange {
  uint64_t Em[2][32], Rb[2][32];
  int Ek[2][32];
  uint32_t stream[2][32][7];  // step, cell, word 3, key, next event, whether new
  uint32_t home[32][6];       // the cell's step, number, word 3, key, tissue
  PairEnd end;
  int swap, pad;
};
static_assert(sizeof(LaneExchange) == kExchangeBytes, "chi_lane.h");

__device__ __forceinline__ void pair_barrier() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

// The child of a node that r falls into: k = the number of leading children
// whose running sum is at most r; r becomes the remainder inside it.  WIDE
// compares with the three running sums at once (the shorter chain, for few
// warps); otherwise the half first, then the child in it (fewer instructions).
template <bool WIDE>
__device__ __forceinline__ uint32_t pick_child(uint64_t s0, uint64_t s1, uint64_t s2, uint64_t& r) {
  const uint64_t p1 = s0 + s1;
  if (WIDE) {
    const uint64_t p2 = p1 + s2;
    const bool c0 = r >= s0, c1 = r >= p1, c2 = r >= p2;
    r -= c2 ? p2 : c1 ? p1 : c0 ? s0 : 0ull;
    return c2 ? 3u : c1 ? 2u : c0 ? 1u : 0u;
  }
  const bool up = r >= p1;
  r -= up ? p1 : 0ull;
  const uint64_t t = up ? s2 : s0;
  const bool second = r >= t;
  r -= second ? t : 0ull;
  return (up ? 2u : 0u) + (second ? 1u : 0u);
}

struct U64x4 {
  uint64_t a, b, c, d;
};

// 32 bytes of the scratch array with one load.
__device__ __forceinline__ U64x4 load4(const uint64_t* p) {
  U64x4 r;
  asm volatile("ld.global.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(r.a), "=l"(r.b), "=l"(r.c), "=l"(r.d)
               : "l"(p)
               : "memory");
  return r;
}

__device__ __forceinline__ void store4(uint64_t* p, const U64x4& x) {
  asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};"
               :
               : "l"(p), "l"(x.a), "l"(x.b), "l"(x.c), "l"(x.d)
               : "memory");
}

// Sectors: the counts of a quad's four voxels, 16 bits each.
__device__ __forceinline__ uint64_t pack4(const uint32_t* c) {
  return static_cast<uint64_t>((c[0] & 0xFFFFu) | (c[1] << 16)) |
         (static_cast<uint64_t>((c[2] & 0xFFFFu) | (c[3] << 16)) << 32);
}
__device__ __forceinline__ uint32_t field16(uint64_t w, uint32_t k) {
  const uint32_t h = (k & 2u) ? static_cast<uint32_t>(w >> 32) : static_cast<uint32_t>(w);
  return (k & 1u) ? h >> 16 : h & 0xFFFFu;
}
__device__ __forceinline__ uint4 unpack4(uint64_t w) {
  return make_uint4(field16(w, 0), field16(w, 1), field16(w, 2), field16(w, 3));
}

__device__ __forceinline__ void add64(uint64_t* p, uint64_t x) {
  atomicAdd(reinterpret_cast<unsigned long long*>(p), static_cast<unsigned long long>(x));
}

// A voxel of the scratch array in one word: D in bits 0..19, N in 20..39, R
// in 40..59, the neighbour mask in 60..63.
__device__ __forceinline__ uint64_t pack_voxel(uint32_t D, uint32_t N, uint32_t R, uint32_t mask) {
  return D | (static_cast<uint64_t>(N) << 20) | (static_cast<uint64_t>(R | (mask << 20)) << 40);
}
__device__ __forceinline__ uint32_t word_D(uint64_t w) {
  return static_cast<uint32_t>(w) & 0xFFFFFu;
}
__device__ __forceinline__ uint32_t word_N(uint64_t w) {
  return static_cast<uint32_t>(w >> 20) & 0xFFFFFu;
}
__device__ __forceinline__ uint32_t word_R(uint64_t w) {
  return static_cast<uint32_t>(w >> 40) & 0xFFFFFu;
}
__device__ __forceinline__ uint32_t word_mask(uint64_t w) {
  return static_cast<uint32_t>(w >> 60);
}
// The change of a word by one molecule of species s.
__device__ __forceinline__ uint64_t word_unit(uint32_t s) {
  const uint32_t lo = s == 0u ? 1u : s == 1u ? 1u << 20 : 0u, hi = s == 2u ? 1u << 8 : 0u;
  return (static_cast<uint64_t>(hi) << 32) | lo;
}

// tau in units of the last place of a binary64 t with exponent field te, rounded
// to nearest; `tie` when it lies half-way, or when tau is not below 2^53 of
// them (t and tau both >= 0; sums below 2^63 stay exact).
__device__ __forceinline__ uint64_t ulps_of(double tau, int te, bool& tie) {
  const uint64_t b = static_cast<uint64_t>(__double_as_longlong(tau));
  const int sh = te - static_cast<int>(b >> 52);
  const uint64_t m = b == 0ull ? 0ull : ((b & ((1ull << 52) - 1ull)) | (1ull << 52));
  if (sh <= 0) {
    tie = sh < 0;
    return m;
  }
  if (sh > 54) return 0ull;  // below half a unit
  const uint64_t half = 1ull << (sh - 1), up = m + half;
  tie = (up & ((half << 1) - 1ull)) == 0ull && m != 0ull;
  return up >> sh;
}

// Event codes of the undo log.
constexpr uint32_t kEvBind = 5u, kEvRelease = 6u, kEvHop = 8u;  // 0..4: channel; 8 + species: hop

// The child of a lane-wide node that r falls into: lane l of the cell holds the
// exclusive prefix x of child l (of R, from lane `base` on), so the child is
// the last whose prefix is at most r (children of sum 0 share their prefix
// with the next and are passed over).
template <int R>
__device__ __forceinline__ uint32_t pick_lane(uint64_t x, uint64_t& r, int base) {
  const unsigned b = __ballot_sync(kFull, r >= x) >> base;
  const int k = __popc((b | 1u) & ((1u << R) - 1u)) - 1;
  r -= __shfl_sync(kFull, x, base + k);
  return static_cast<uint32_t>(k);
}

// Registers: shared leaves 168 (12 warps an SM; beyond, more lanes' worth of cells
// take records); one lane per cell of more than 256 voxels as many as it wants, 130
// to 151 (shared memory holds 8 warps an SM anyway); with a helper of HELP blocks an SM 168 (six,
// 12 warps) or 128 (eight); else 128, so that 14 to 16 warps fit an SM.
template <int MODEL, int LV, int LEAF, int G, int HELP>
__global__ void __launch_bounds__(HELP || G == 1 ? 64 : 32, HELP                  ? HELP
                                                            : LEAF == kLeafShared ? 12
                                                            : G > 1               ? 14
                                                            : LV == 5             ? 4
                                                                                  : 7)
    k_chi_lane(const LaneArgs p) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool ONE = G == 1;
  // rates read from shared memory by every event rather than held in registers:
  // MODEL 0 then fits 128 of them but for four words (the others gain nothing)
  constexpr bool kLean = MODEL == 0 && LEAF == kLeafShared && HELP == 8;
  // Lane-wide nodes (8 lanes per cell and more): the root's prefixes, one a
  // lane, in registers; below it one level of nodes of RAD prefixes in shared
  // memory, down to voxels (VMID), quads or (FOUR) four quads.
  constexpr bool WIDE = G >= 8;
  constexpr uint32_t RAD = G >= 16 ? 16u : 8u;
  constexpr uint32_t RV = (1u << (2 * LV)) / RAD;  // voxels under a root entry
  constexpr bool MID = WIDE && RV > 4u;
  constexpr uint32_t MV = MID ? RV / RAD : 1u;     // ... under an entry of the level below
  constexpr bool VMID = MID && MV == 1u, FOUR = MID && MV == 16u;
  constexpr uint32_t kMid = RAD, kFour = RAD + RAD * RAD;
  static_assert(!VMID || LEAF == kLeafShared, "voxel prefixes: shared leaves");
  static_assert(ONE ? LEAF != kLeafShared : LEAF != kLeafSectors,
                "one lane per cell: leaves in the scratch array; sectors: one lane per cell");
  constexpr bool PLN = LEAF == kLeafPlanes;   // 16-bit counts in shared memory, no voxel totals
  static_assert(!PLN || G == 4 || (MID && MV == 4u), "planes: sums down to quads");
  constexpr bool REC = LEAF != kLeafShared;   // counts in a packed range (else: scratch array)
  constexpr bool SEC = LEAF == kLeafSectors;  // ... as counts and quad sums, no voxel totals
  constexpr uint32_t NQ = 1u << (2 * (LV - 1));  // quads of a full tree
  // the levels of sums in shared memory: down to the quads' (sectors: down to
  // those of four quads)
  constexpr int SL = SEC ? LV - 2 : LV - 1;
  const int lane = threadIdx.x & 31;
  int wib = threadIdx.x >> 5;
  const uint32_t slot = static_cast<uint32_t>(lane) / G, sl = static_cast<uint32_t>(lane) % G;
  constexpr uint32_t slots = 32u / G;
  const int base_lane = lane - static_cast<int>(sl);
  const uint32_t li = sl % RAD;  // this lane's entry of a lane-wide node
  const bool lead = sl == 0u;
  const uint32_t V = p.V, n = p.n, nq = (V + 3u) >> 2;
  const uint32_t ps = nq * 4u;  // distance between the planes of D, N and R (shared leaves)
  const uint32_t centre = MODEL == 2 ? (n >> 1) * n + (n >> 1) : 0u;
  const bool vec = (V & 3u) == 0u;
  const uint32_t warps = HELP ? 1u : blockDim.x >> 5;  // that run cells

  // The index i of an array of n (checked build: `oob` when it is out of range).
  [[maybe_unused]] bool oob = false;
#define IX(i, n) TSG_IDX(i, n, oob)
  // offsets u - v of the m-th existing direction for each neighbour mask, then
  // (shared leaves) the voxels' masks: bits 0..3, and their number: bits 4..6
  int16_t* hop_off = reinterpret_cast<int16_t*>(smem);
  LaneExchange* ex = reinterpret_cast<LaneExchange*>(smem + p.lut_bytes - sizeof(LaneExchange));
  if (HELP && threadIdx.x == 0) {
    unsigned w;
    asm volatile("mov.u32 %0, %%warpid;" : "=r"(w));
    // every other pair of blocks the other way round, so that the warps that run
    // cells spread over the SM's four schedulers (one half of them otherwise:
    // 64x64 cells 9.3 -> 12.2 ms)
    ex->swap = static_cast<int>((w >> 2) & 1u);
    ex->end.clear();
  }
  unsigned char* lut = smem + 128;
  for (uint32_t i = threadIdx.x; i < 64u; i += blockDim.x) {
    uint32_t b = i >> 2;
    for (uint32_t k = i & 3u; k > 0u; --k) b &= b - 1u;
    const int d = __ffs(static_cast<int>(b)) - 1;
    hop_off[IX(i, 64)] = static_cast<int16_t>(d < 0    ? 0
                                      : d == 0 ? -1
                                      : d == 1 ? 1
                                      : d == 2 ? -static_cast<int>(n)
                                               : static_cast<int>(n));
  }
  const uint32_t nl = (nq + 3u) >> 2;  // lines of four quads (sectors)
  [[maybe_unused]] const uint32_t lut_n = SEC ? nl * 16u : nq * 4u;
  for (uint32_t v = threadIdx.x; v < (SEC ? nl * 16u : nq * 4u); v += blockDim.x) {
    const uint32_t vy = v / n, vx = v - vy * n;
    const uint32_t m = static_cast<uint32_t>(vx > 0) | (static_cast<uint32_t>(vx < n - 1) << 1) |
                       (static_cast<uint32_t>(vy > 0) << 2) |
                       (static_cast<uint32_t>(vy < n - 1) << 3);
    lut[IX(v, lut_n)] = static_cast<unsigned char>(m | (__popc(m) << 4));
  }
  __syncthreads();
  early_launch();
  if (kChecked) {  // the parts of shared memory and of the scratch array
    uint32_t bytes;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(bytes));
    const uint32_t cell = 48u + 8u * lane_sum_words(LV, LEAF, G) + (PLN ? 6u : REC ? 0u : 20u) * ps;
    const uint64_t words = SEC ? 16u * nl : 8u * nq;
    if (128u + lut_n + (HELP ? kExchangeBytes : 0u) > p.lut_bytes || cell > p.cell_stride ||
        p.lut_bytes + warps * slots * p.cell_stride > bytes ||
        (REC && !PLN && gridDim.x * warps * slots * words > p.scratch_words)) {
      if (threadIdx.x == 0) atomicOr(p.views[0].err, kErrBounds);
      return;  // the whole block
    }
  }

  // The helper warp: draws for the events after those in hand, a batch ahead.
  // Per phase (one barrier of both warps) it takes the new cells' streams and
  // leaves the draws for the next phase; buffers and streams alternate.
  if (HELP) wib ^= ex->swap;
  if (HELP && wib == 1) {
    uint32_t hs[5] = {}, he = 0;
    for (uint32_t ph = 0;; ph ^= 1u) {
      pair_barrier();
      if (ex->end.reached(ph)) return;
      const uint32_t* d = ex->stream[ph][slot];
      if (d[6]) {
#pragma unroll
        for (int k = 0; k < 5; ++k) hs[k] = d[k];
        he = d[5];
      } else {
        he += G;
      }
      uint64_t m_, r_;
      int k_;
      draw_event(he + G + sl, hs[0], hs[1], hs[2], hs[3], hs[4], m_, k_, r_);
      ex->Em[ph ^ 1u][lane] = m_;
      ex->Rb[ph ^ 1u][lane] = r_;
      ex->Ek[ph ^ 1u][lane] = k_;
    }
  }
  uint32_t phase = 0;
  uint32_t* home = HELP ? ex->home[slot] : nullptr;

  // A cell's shared memory: the rates {g, h} of D, N and R, the sums, and with
  // shared leaves the voxel totals (the tree's last level) and the counts.
  unsigned char* warp_cells =
      smem + p.lut_bytes + static_cast<size_t>(wib) * slots * p.cell_stride;
  unsigned char* cs = warp_cells + slot * p.cell_stride;
  const ulonglong2* rates = reinterpret_cast<const ulonglong2*>(cs);
  uint64_t* tree = reinterpret_cast<uint64_t*>(cs + 48);
  constexpr uint32_t kCnt = lane_sum_words(LV, LEAF, G);  // shared leaves: the voxel totals
  int32_t* cp = reinterpret_cast<int32_t*>(tree + kCnt + ps);
  // a cell's scratch: 2 words per voxel, its total and its counts (records);
  // or 4 words per quad, its sum and its counts of D, N and R (sectors)
  uint16_t* hp = reinterpret_cast<uint16_t*>(tree + kCnt);  // planes: the counts
  const uint32_t rec_words = SEC ? 16u * nl : 8u * nq;
  uint64_t* warp_rec =
      REC && !PLN ? p.scratch + (static_cast<size_t>(blockIdx.x) * warps + wib) * slots * rec_words
          : nullptr;
  uint64_t* rec = warp_rec + static_cast<size_t>(slot) * rec_words;
  [[maybe_unused]] const uint32_t tree_n = kCnt + (REC ? 0u : ps);  // words of `tree`

  LaneRates<MODEL> q{};
  const TissueView* tv = p.views + (p.items ? p.items[0].x : 0u);
  q.hill = tv->q.hill;
  bool have = false, done = false;
  int started = 0;
  uint32_t e_next = 0xFFFFFFFFu;  // the event the helper's next draws start with
  uint32_t cell = 0, vidx = 0, step = 0, word3 = 0, key0 = 0, key1 = 0, e0 = 0;
  uint64_t A = 0, over_mask = 0;
  uint64_t X1 = 0;  // lane-wide nodes: the root's prefix of entry li
  uint32_t lim_dn = 0, lim_r = 0;  // sectors: the counts' limits
  double tnow = 0.0;
  int err = 0;
  // records: the bits a count has once it reaches its limit (a power of two)
  auto set_limits = [&](const Limits& l) {
    auto bits = [](uint32_t x) { return 0xFFFFFu & ~(x - 1u); };
    over_mask = pack_voxel(bits(l.D), bits(l.N), bits(l.R), 0u);
    lim_dn = l.D;
    lim_r = l.R;
  };
  auto warp_max = [](const Limits& m) {
    return Limits{__reduce_max_sync(kFull, m.D), __reduce_max_sync(kFull, m.N),
                  __reduce_max_sync(kFull, m.R)};
  };
  uint32_t lim = 0;
  bool big = false;  // shared leaves: the cell holds, or held, a D or N of `small` or an R of
                     // `lim` or more

  // Cells of up to 64 voxels, one lane each: every lane loads its first cell, at the
  // same time as the others theirs (one after another, as below, a warp's 32 take
  // 50 us: 140x140 cells of 2x2 voxels at dt 0.001 126 us a step, 91 so).
  if (ONE && LV == 3) {
    const uint32_t it = (blockIdx.x * warps + wib) * slots + static_cast<uint32_t>(lane);
    started = 1;
    if (it < p.n_items) {
      const uint2 w = p.items ? p.items[it] : make_uint2(0u, it);
      const TissueView* ntv = p.views + w.x;
      if (kChecked && (ntv->V != V || w.y >= ntv->width * ntv->height)) {
        atomicOr(ntv->err, kErrBounds);
      } else {
        q.load(ntv->q);
        const int32_t* g = ntv->counts + static_cast<size_t>(w.y) * 3u * V;
        ulonglong2* rt = reinterpret_cast<ulonglong2*>(cs);
        rt[0] = make_ulonglong2(q.gD, q.hD);
        rt[1] = make_ulonglong2(q.gN, q.hN);
        rt[2] = make_ulonglong2(q.gR + (MODEL == 1 ? q.k_off : 0ull), q.hR);
        bool bad_state = false;
        Limits top{0, 0, 0};
        uint64_t four = 0;
        A = 0;
#pragma unroll 1
        for (uint32_t qi = 0; qi < NQ; ++qi) {
          uint64_t S = 0;
          if (qi < nq) {
            uint32_t d[4] = {0, 0, 0, 0}, m[4] = {0, 0, 0, 0}, r[4] = {0, 0, 0, 0};
            if (vec) {
              const uint4 x = reinterpret_cast<const uint4*>(g)[IX(qi, V / 4u)];
              const uint4 y = reinterpret_cast<const uint4*>(g + V)[IX(qi, V / 4u)];
              const uint4 z = reinterpret_cast<const uint4*>(g + 2u * V)[IX(qi, V / 4u)];
              d[0] = x.x, d[1] = x.y, d[2] = x.z, d[3] = x.w;
              m[0] = y.x, m[1] = y.y, m[2] = y.z, m[3] = y.w;
              r[0] = z.x, r[1] = z.y, r[2] = z.z, r[3] = z.w;
            } else {
#pragma unroll
              for (uint32_t i = 0; i < 4u; ++i)
                if (4u * qi + i < V) {
                  d[i] = static_cast<uint32_t>(g[IX(4u * qi + i, 3u * V)]);
                  m[i] = static_cast<uint32_t>(g[IX(V + 4u * qi + i, 3u * V)]);
                  r[i] = static_cast<uint32_t>(g[IX(2u * V + 4u * qi + i, 3u * V)]);
                }
            }
            ulonglong2* o = reinterpret_cast<ulonglong2*>(rec) + 4u * IX(qi, rec_words / 8u);
#pragma unroll
            for (uint32_t i = 0; i < 4u; ++i) {
              const uint32_t v = 4u * qi + i;
              uint64_t a = 0, wd = 0;
              if (v < V) {
                const uint32_t mk = lut[IX(v, lut_n)];
                const bool ctr = MODEL == 2 && v == centre;
                bad_state = bad_state || (MODEL == 2 && r[i] > static_cast<uint32_t>(ctr));
                top = Limits{max(top.D, d[i]), max(top.N, m[i]), max(top.R, r[i])};
                wd = pack_voxel(d[i], m[i], r[i] & 0xFFFFFu, mk & 15u);
                a = lane_total<MODEL>(q, ntv, d[i], m[i], r[i], mk >> 4, ctr);
              }
              o[i] = make_ulonglong2(a, wd);
              S += a;
            }
          }
          tree[IX(level_off(2) + qi, tree_n)] = S;
          four += S;
          if ((qi & 3u) == 3u) {
            tree[IX(qi >> 2, tree_n)] = four;
            A += four;
            four = 0;
          }
        }
        Limits nlim{1, 1, 1};
        const bool past = !pick_limits<MODEL, LEAF>(ntv, top, nlim);
        err = bad_state ? kErrState : past ? kErrNarrow : 0;
        set_limits(nlim);
        if (kChecked && oob) err = kErrBounds;
        oob = false;
        tv = ntv;
        step = *ntv->step + p.step_off;
        cell = w.y;
        word3 = ntv->tissue_id | (kTagChi << 24);
        key0 = static_cast<uint32_t>(ntv->seed);
        key1 = static_cast<uint32_t>(ntv->seed >> 32);
        vidx = w.x;
        if (HELP) {
          home[0] = step;
          home[1] = cell;
          home[2] = word3;
          home[3] = key0;
          home[4] = key1;
          home[5] = vidx;
        }
        have = true;
      }
    }
    __syncwarp();
  }

  for (;;) {
    // ---- slots without a cell take the next work items, one after another --
    unsigned want = __ballot_sync(kFull, !have && !done && lead);
    const bool loads = want != 0u;  // uniform
    while (want) {
      const int src = __ffs(want) - 1;
      want &= want - 1u;
      const uint32_t sc = static_cast<uint32_t>(src) / G;
      // the first item by position, further ones by the counter (never read when
      // one wave takes all)
      const uint32_t places = gridDim.x * warps * slots;
      uint32_t it = (blockIdx.x * warps + wib) * slots + sc;
      if (__shfl_sync(kFull, started, src)) {
        it = p.n_items;
        if (places < p.n_items) {
          if (lane == src) it = places + atomicAdd(p.counter, 1u);
          it = __shfl_sync(kFull, it, src);
        }
      }
      if (slot == sc) started = 1;
      if (it >= p.n_items) {
        if (slot == sc) done = true;
        continue;
      }
      const uint2 w = p.items ? p.items[it] : make_uint2(0u, it);
      const TissueView* ntv = p.views + w.x;
      if (kChecked && (ntv->V != V || w.y >= ntv->width * ntv->height)) {
        if (lane == 0) atomicOr(ntv->err, kErrBounds);
        continue;
      }
      LaneRates<MODEL> nr;
      nr.load(ntv->q);
      const int32_t* g = ntv->counts + static_cast<size_t>(w.y) * 3u * V;
      unsigned char* ncs = warp_cells + sc * p.cell_stride;
      uint64_t* ntree = reinterpret_cast<uint64_t*>(ncs + 48);
      int32_t* ncp = reinterpret_cast<int32_t*>(ntree + kCnt + ps);
      uint64_t* nrec = warp_rec + static_cast<size_t>(sc) * rec_words;
      if (lane < 3)
        reinterpret_cast<ulonglong2*>(ncs)[lane] =
            lane == 0   ? make_ulonglong2(nr.gD, nr.hD)
            : lane == 1 ? make_ulonglong2(nr.gN, nr.hN)
                        : make_ulonglong2(nr.gR + (MODEL == 1 ? nr.k_off : 0ull), nr.hR);
      bool ovf = false, bad_state = false, nbig = false;
      Limits top{0, 0, 0};  // packed counts: the largest
      uint64_t total = 0, pair = 0;
      for (uint32_t k = 0; k < (NQ + 31u) / 32u; ++k) {
        const uint32_t qi = static_cast<uint32_t>(lane) + 32u * k;
        uint64_t S = 0, a[4] = {0ull, 0ull, 0ull, 0ull};
        if (qi < nq) {
          uint32_t d[4] = {0, 0, 0, 0}, m[4] = {0, 0, 0, 0}, r[4] = {0, 0, 0, 0};
          if (vec) {
            const uint4 x = reinterpret_cast<const uint4*>(g)[IX(qi, V / 4u)];
            const uint4 y = reinterpret_cast<const uint4*>(g + V)[IX(qi, V / 4u)];
            const uint4 z = reinterpret_cast<const uint4*>(g + 2u * V)[IX(qi, V / 4u)];
            d[0] = x.x, d[1] = x.y, d[2] = x.z, d[3] = x.w;
            m[0] = y.x, m[1] = y.y, m[2] = y.z, m[3] = y.w;
            r[0] = z.x, r[1] = z.y, r[2] = z.z, r[3] = z.w;
          } else {
#pragma unroll
            for (uint32_t i = 0; i < 4u; ++i)
              if (4u * qi + i < V) {
                d[i] = static_cast<uint32_t>(g[IX(4u * qi + i, 3u * V)]);
                m[i] = static_cast<uint32_t>(g[IX(V + 4u * qi + i, 3u * V)]);
                r[i] = static_cast<uint32_t>(g[IX(2u * V + 4u * qi + i, 3u * V)]);
              }
          }
          uint64_t wd[4];
#pragma unroll
          for (uint32_t i = 0; i < 4u; ++i) {
            const uint32_t v = 4u * qi + i;
            wd[i] = 0ull;
            if (v < V) {
              const uint32_t mk = lut[IX(v, lut_n)], nn = mk >> 4;
              const bool ctr = MODEL == 2 && v == centre;
              if (MODEL == 2 && r[i] > static_cast<uint32_t>(ctr)) bad_state = true;
              if (REC) {
                top = Limits{max(top.D, d[i]), max(top.N, m[i]), max(top.R, r[i])};
              } else {
                if (MODEL != 2 && r[i] >= kLaneHill) nbig = true;
                if ((d[i] | m[i] | r[i]) >= nr.small) {
                  nbig = true;
                  ovf |= exact_ovf<MODEL>(ntv, d[i], m[i], r[i], nn, ctr);
                }
              }
              if (REC) {
                wd[i] = pack_voxel(d[i], m[i], r[i] & 0xFFFFFu, mk & 15u);
              }
              a[i] = lane_total<MODEL>(nr, ntv, d[i], m[i], r[i], nn, ctr);
            }
            S += a[i];
          }
          if (SEC) {
            store4(nrec + 4u * IX(qi, rec_words / 4u), U64x4{S, pack4(d), pack4(m), pack4(r)});
          } else if (PLN) {
            uint64_t* o = ntree + kCnt;
            o[IX(qi, 3u * nq)] = pack4(d);
            o[IX(nq + qi, 3u * nq)] = pack4(m);
            o[IX(2u * nq + qi, 3u * nq)] = pack4(r);
          } else if (REC) {
            ulonglong2* o = reinterpret_cast<ulonglong2*>(nrec) + 4u * IX(qi, rec_words / 8u);
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = make_ulonglong2(a[i], wd[i]);
          } else {
            ulonglong2* o = reinterpret_cast<ulonglong2*>(ntree + kCnt) + 2u * IX(qi, nq);
            o[0] = make_ulonglong2(a[0], a[1]);
            o[1] = make_ulonglong2(a[2], a[3]);
            reinterpret_cast<uint4*>(ncp)[IX(qi, nq)] = make_uint4(d[0], d[1], d[2], d[3]);
            reinterpret_cast<uint4*>(ncp + ps)[IX(qi, nq)] = make_uint4(m[0], m[1], m[2], m[3]);
            reinterpret_cast<uint4*>(ncp + 2u * ps)[IX(qi, nq)] =
                make_uint4(r[0], r[1], r[2], r[3]);
          }
        } else if (SEC && qi < 4u * nl) {
          store4(nrec + 4u * IX(qi, rec_words / 4u), U64x4{0ull, 0ull, 0ull, 0ull});
        }
        // the sums above the quads (entries past the last quad are zero)
        if (WIDE) {
          constexpr uint32_t W = RV / 4u;  // quads under a root entry
          uint64_t I = S;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint64_t x = __shfl_up_sync(kFull, I, o);
            if (lane >= o) I += x;
          }
          const uint64_t E = I - S;
          const uint64_t first = __shfl_sync(kFull, E, lane & ~static_cast<int>(W - 1u));
          if (qi < NQ) {
            if (qi % W == 0u) ntree[IX(qi / W, tree_n)] = total + first;
            if (VMID) {
              uint64_t x = E - first;
#pragma unroll
              for (uint32_t i = 0; i < 4u; ++i) {
                ntree[IX(kMid + 4u * qi + i, tree_n)] = x;
                x += a[i];
              }
            } else if (FOUR) {
              if (qi % 4u == 0u) ntree[IX(kMid + qi / 4u, tree_n)] = E - first;
              ntree[IX(kFour + qi, tree_n)] = S;
            } else if (MID) {
              ntree[IX(kMid + qi, tree_n)] = E - first;
            }
          }
          total += __shfl_sync(kFull, I, 31);
          continue;
        }
        if (!SEC && qi < NQ) ntree[IX(level_off(LV - 1) + qi, tree_n)] = S;
        uint64_t x = S + __shfl_xor_sync(kFull, S, 1);
        x += __shfl_xor_sync(kFull, x, 2);
        if (qi < NQ && (lane & 3) == 0) ntree[IX(level_off(LV - 2) + (qi >> 2), tree_n)] = x;
        x += __shfl_xor_sync(kFull, x, 4);
        x += __shfl_xor_sync(kFull, x, 8);
        if (LV >= 4 && (lane & 15) == 0)
          ntree[IX(level_off(LV >= 4 ? LV - 3 : 1) + (qi >> 4), tree_n)] = x;
        x += __shfl_xor_sync(kFull, x, 16);
        if (LV == 5) {
          pair = (k & 1u) ? pair + x : x;
          if ((k & 1u) && lane == 0) ntree[IX(k >> 1, tree_n)] = pair;
        }
        total += x;
      }
      const bool any_ovf = __any_sync(kFull, ovf), any_bad = __any_sync(kFull, bad_state);
      nbig = __any_sync(kFull, nbig);
      Limits nlim{1, 1, 1};
      if (REC) nbig = !pick_limits<MODEL, LEAF>(ntv, warp_max(top), nlim);
      const bool out_of_range = kChecked && __any_sync(kFull, oob);
      oob = false;
      __syncwarp();
      if (slot == sc) {
        if (WIDE) X1 = ntree[IX(li, tree_n)];
        q = nr;
        tv = ntv;
        step = *ntv->step + p.step_off;
        cell = w.y;
        word3 = ntv->tissue_id | (kTagChi << 24);
        key0 = static_cast<uint32_t>(ntv->seed);
        key1 = static_cast<uint32_t>(ntv->seed >> 32);
        vidx = w.x;
        if (HELP && lead) {
          home[0] = step;
          home[1] = cell;
          home[2] = word3;
          home[3] = key0;
          home[4] = key1;
          home[5] = vidx;
        }
        A = total;
        tnow = 0.0;
        e0 = 0;
        e_next = 0xFFFFFFFFu;
        big = nbig;
        lim = min(nr.small, kLaneHill);
        err = any_bad ? kErrState : any_ovf ? kErrOverflow : (REC && nbig) ? kErrNarrow : 0;
        if (out_of_range) err = kErrBounds;
        have = true;
        if (REC) set_limits(nlim);
      }
    }
    __syncwarp();
    if (__all_sync(kFull, done)) {
      if (HELP) {
        if (lane == 0) ex->end.announce(phase);
        __syncwarp();
        pair_barrier();
      }
      break;
    }

    // ---- draws: lane j of a cell, event e0 + j -----------------------------
    uint64_t Em = 0, Rb = 0;
    int Ek = 0;
    const uint64_t* bits = nullptr;  // helper: the batch's random bits
    if (HELP) {
      const bool fresh = have && e0 != e_next;  // a new cell, or a batch cut short
      if (lead) {
        uint32_t* d = ex->stream[phase][slot];
        if (fresh) {
#pragma unroll
          for (int k = 0; k < 5; ++k) d[k] = home[k];
          d[5] = e0;
        }
        d[6] = fresh ? 1u : 0u;
      }
      __syncwarp();
      pair_barrier();
      if (__any_sync(kFull, fresh)) {
        uint64_t m_, r_;
        int k_;
        draw_event(e0 + sl, home[0], home[1], home[2], home[3], home[4], m_, k_, r_);
        if (fresh) {
          ex->Em[phase][lane] = m_;
          ex->Ek[phase][lane] = k_;
          ex->Rb[phase][lane] = r_;
        }
        __syncwarp();
      }
      bits = ex->Rb[phase] + base_lane;
      e_next = e0 + G;
    } else {
      draw_event(e0 + sl, step, cell, word3, key0, key1, Em, Ek, Rb);
    }

    // ---- G events of every cell, the whole warp in step --------------------
    bool run = have && err == 0;
    bool paused = false;    // shared leaves: a count reached its limit for the first time
    const bool slow = !REC && __any_sync(kFull, run && big);
    uint32_t m = 0;         // events applied
    uint64_t Aj = 0;        // the total propensity before this lane's event
    uint32_t log = 0;       // this lane's event: v, u, code
    uint64_t Rn = HELP ? bits[0] : ONE ? Rb : __shfl_sync(kFull, Rb, base_lane);  // the next event's random bits
    // No more events than are likely left in the step (A (dt - t) are expected), so
    // that a short one does not undo most of its batch.  A whole warp on a cell asks
    // before every batch (2x2 cells of 8x8 voxels, dt 1e-9: 34 -> 22 us a step), 8 and
    // 16 lanes on small cells, which have the fewest events, after a load (40x40 of
    // 4x4, dt 1e-5: 34 -> 27 us; larger cells: 2% slower with the promoter model).
    uint32_t batch = G;
    if (G == 32 || (LV == 3 && WIDE && loads)) {
      const float left = __double2float_rn(p.dt - tnow) * (__ull2float_rn(A) * 0x1p-32f);
      const uint32_t few =
          left < 32.0f ? static_cast<uint32_t>(left + 3.0f * sqrtf(left)) + 3u : 32u;
      // uniform, for the compiler too
      batch = min(static_cast<uint32_t>(G), __reduce_max_sync(kFull, have || G == 32 ? few : 0u));
    }
    for (uint32_t i = 0; i < batch; ++i) {
      [[maybe_unused]] const bool ran = run;
      const uint64_t R64 = Rn;
      if (!ONE)
        Rn = HELP ? bits[(i + 1u) % G]
                  : __shfl_sync(kFull, Rb, base_lane + static_cast<int>((i + 1u) % G));
      uint64_t r = __umul64hi(R64, A);
      // descent to a quad
      uint32_t idx = 0, kv = 0, pv = 0;
      uint64_t xm = 0;
      if (WIDE) {
        kv = pick_lane<RAD>(X1, r, base_lane);
        idx = kv;
        if (MID) {
          xm = tree[IX(kMid + kv * RAD + li, tree_n)];
          pv = pick_lane<RAD>(xm, r, base_lane);
          idx = kv * RAD + pv;
        }
        if (FOUR) {
          const ulonglong2* nd =
              reinterpret_cast<const ulonglong2*>(tree + kFour) + 2u * IX(idx, 64);
          const ulonglong2 x = nd[0], y = nd[1];
          idx = 4u * idx + pick_child<!ONE>(x.x, x.y, y.x, r);
        }
      } else {
#pragma unroll
        for (uint32_t l = 1; l <= SL; ++l) {
          const ulonglong2* nd = reinterpret_cast<const ulonglong2*>(tree + level_off(l)) +
                                 2u * IX(idx, 1 << (2u * (l - 1u)));
          const ulonglong2 x = nd[0], y = nd[1];
          idx = 4u * idx + pick_child<!ONE>(x.x, x.y, y.x, r);
        }
      }
      U64x4 sec{};  // sectors: the quad's sum and its counts of D, N and R
      if (SEC) {
        idx = min(idx, nl - 1u);
        const uint64_t* line = rec + 16u * IX(idx, nl);
        const U64x4 x0 = load4(line), x1 = load4(line + 4), x2 = load4(line + 8),
                    x3 = load4(line + 12);
        const uint32_t k = pick_child<false>(x0.a, x1.a, x2.a, r);
        idx = 4u * idx + k;
        sec.a = k == 0u ? x0.a : k == 1u ? x1.a : k == 2u ? x2.a : x3.a;
        sec.b = k == 0u ? x0.b : k == 1u ? x1.b : k == 2u ? x2.b : x3.b;
        sec.c = k == 0u ? x0.c : k == 1u ? x1.c : k == 2u ? x2.c : x3.c;
        sec.d = k == 0u ? x0.d : k == 1u ? x1.d : k == 2u ? x2.d : x3.d;
      }
      // never past the cell's quads (or voxels), whatever the sums hold
      if (kChecked && run && idx >= (VMID ? 4u * nq : nq)) err |= kErrBounds;
      idx = min(idx, (VMID ? 4u * nq : nq) - 1u);
      // the voxel, its total, counts and neighbours
      uint64_t a_v, w_v = 0;
      uint32_t v, D, N, R, mask, nn;
      if (SEC) {
        const uint32_t mk4 = *reinterpret_cast<const uint32_t*>(lut + 4u * IX(idx, lut_n / 4u));
        uint64_t a[4];
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) {
          const uint32_t Dj = field16(sec.b, j), Nj = field16(sec.c, j), Rj = field16(sec.d, j);
          const uint32_t nj = (mk4 >> (8u * j + 4u)) & 7u;
          uint64_t t = (q.gD + q.hD * nj) * Dj + (q.gN + q.hN * nj) * Nj;
          if (MODEL == 2) {
            const uint32_t F = static_cast<uint32_t>(4u * idx + j == centre) - Rj;
            t += q.tD * F + q.kd * Rj + q.k_in * (static_cast<uint64_t>(Nj) * F);
          } else {
            // R < kHillTab in a cell that runs; the mask is for idle lanes
            t += (q.gR + q.k_off + q.hR * nj) * Rj +
                 __ldg(q.hill + IX(Rj & (kHillTab - 1u), kHillTab)) + q.kN;
            if (MODEL == 1) t += q.k_in * (static_cast<uint64_t>(Dj) * Nj);
          }
          a[j] = t;
        }
        const uint32_t k = pick_child<false>(a[0], a[1], a[2], r);
        a_v = k == 0u ? a[0] : k == 1u ? a[1] : k == 2u ? a[2] : a[3];
        v = 4u * idx + k;
        D = field16(sec.b, k);
        N = field16(sec.c, k);
        R = field16(sec.d, k);
        const uint32_t mk = (mk4 >> (8u * k)) & 0xFFu;
        mask = mk & 15u;
        nn = mk >> 4;
      } else if (PLN) {
        // lane j of every four computes the quad's voxel j; the prefixes find v
        const uint32_t vj = 4u * idx + (sl & 3u);
        const uint32_t Dj = hp[IX(vj, 3u * ps)], Nj = hp[IX(ps + vj, 3u * ps)],
                       Rj = hp[IX(2u * ps + vj, 3u * ps)];
        const uint32_t mk = lut[IX(vj, lut_n)], nj = mk >> 4;
        uint64_t t = (q.gD + q.hD * nj) * Dj + (q.gN + q.hN * nj) * Nj;
        if (MODEL == 2) {
          const uint32_t Fj = static_cast<uint32_t>(vj == centre) - Rj;
          t += q.tD * Fj + q.kd * Rj + q.k_in * (static_cast<uint64_t>(Nj) * Fj);
        } else {
          // R < kHillTab in a cell that runs; the mask is for idle lanes
          t += (q.gR + q.k_off + q.hR * nj) * Rj +
               __ldg(q.hill + IX(Rj & (kHillTab - 1u), kHillTab)) + q.kN;
          if (MODEL == 1) t += q.k_in * (static_cast<uint64_t>(Dj) * Nj);
        }
        uint64_t in = t;
        uint64_t z = __shfl_up_sync(kFull, in, 1, 4);
        if (sl & 3u) in += z;
        z = __shfl_up_sync(kFull, in, 2, 4);
        if (sl & 2u) in += z;
        const uint64_t ex4 = in - t;
        const unsigned b4 = __ballot_sync(kFull, r >= ex4) >> base_lane;
        const int k = __popc((b4 | 1u) & 15u) - 1;
        r -= __shfl_sync(kFull, ex4, base_lane + k);
        a_v = __shfl_sync(kFull, t, base_lane + k);
        const uint32_t dn = __shfl_sync(kFull, Dj | (Nj << 16), base_lane + k);
        const uint32_t rm = __shfl_sync(kFull, Rj | (mk << 16), base_lane + k);
        v = 4u * idx + static_cast<uint32_t>(k);
        D = dn & 0xFFFFu;
        N = dn >> 16;
        R = rm & 0xFFFFu;
        mask = (rm >> 16) & 15u;
        nn = rm >> 20;
      } else if (REC) {
        const U64x4 x = load4(rec + 8u * IX(idx, nq));
        const U64x4 y = load4(rec + 8u * IX(idx, nq) + 4u);
        const uint32_t k = pick_child<!ONE>(x.a, x.c, y.a, r);
        a_v = k == 0u ? x.a : k == 1u ? x.c : k == 2u ? y.a : y.c;
        w_v = k == 0u ? x.b : k == 1u ? x.d : k == 2u ? y.b : y.d;
        v = 4u * idx + k;
        D = word_D(w_v);
        N = word_N(w_v);
        R = word_R(w_v);
        mask = word_mask(w_v);
        nn = __popc(mask);
      } else {
        v = idx;
        if (!VMID) {
          const ulonglong2* nd =
              reinterpret_cast<const ulonglong2*>(tree + kCnt) + 2u * IX(idx, nq);
          const ulonglong2 x = nd[0], y = nd[1];
          v = 4u * idx + pick_child<!ONE>(x.x, x.y, y.x, r);
        }
        a_v = tree[IX(kCnt + v, tree_n)];
        D = static_cast<uint32_t>(cp[IX(v, 3u * ps)]);
        N = static_cast<uint32_t>(cp[IX(ps + v, 3u * ps)]);
        R = static_cast<uint32_t>(cp[IX(2u * ps + v, 3u * ps)]);
        const uint32_t mk = lut[IX(v, lut_n)];
        mask = mk & 15u;
        nn = mk >> 4;
      }
      // nothing left to happen (A = 0); else never while the sums are
      // consistent (voxels past V have total 0)
      if (run && r >= a_v) {
        run = false;
        err |= A != 0ull ? kErrInternal : 0;
      }

      // channel: hops are the last but the in-voxel bindings in channel order
      const bool ctr = MODEL == 2 && v == centre;
      const uint32_t F = MODEL == 2 ? static_cast<uint32_t>(ctr) - R : 0u;
      // F is 0 or 1
      const uint64_t y17 = MODEL == 2 ? (F ? q.k_in * N : 0ull)
                           : MODEL    ? q.k_in * (static_cast<uint64_t>(D) * N)
                                      : 0ull;
      const uint64_t y18 = MODEL == 1 ? q.k_off * R : 0ull;
      const uint64_t UD = (kLean ? rates[0].y : q.hD) * D, UN = (kLean ? rates[1].y : q.hN) * N;
      const uint64_t UR = MODEL == 2 ? 0ull : (kLean ? rates[2].y : q.hR) * R;
      const uint64_t HD = UD * nn, H2 = HD + UN * nn, H3 = MODEL == 2 ? H2 : H2 + UR * nn;
      const uint64_t top = a_v - y17 - y18, y = top - H3;
      const bool hop = r >= y && (MODEL == 0 || r < top);
      const uint64_t z0 = r - y;
      const bool z1 = z0 >= HD, z2 = MODEL != 2 && z0 >= H2;
      uint32_t s = z2 ? 2u : z1 ? 1u : 0u;  // the species a hop or a MODEL 0 channel changes
      bool gain = false;                    // ... and whether by +1 at v
      uint32_t code = kEvHop + s, u = v;
      int dD = 0, dN = 0, dR = 0;           // MODEL 1, 2: the changes at v
      bool several = false;                 // ... of more than one species
      if (hop) {
        const uint64_t unit = z2 ? UR : z1 ? UN : UD, unit2 = unit + unit;
        const uint64_t z3 = z0 - (z2 ? H2 : z1 ? HD : 0ull);
        const bool b2 = z3 >= unit2;
        const uint64_t z4 = z3 - (b2 ? unit2 : 0ull);
        const int off = hop_off[IX((mask << 2) + (b2 ? 2u : 0u) + (z4 >= unit ? 1u : 0u), 64)];
        u = v + static_cast<uint32_t>(off);
        if (kChecked && run && u >= V) err |= kErrBounds;
        u = min(u, V - 1u);
        if (MODEL) {
          dD = s == 0u ? -1 : 0;
          dN = s == 1u ? -1 : 0;
          dR = s == 2u ? -1 : 0;
        }
      } else {
        const uint64_t gDD = (kLean ? rates[0].x : q.gD) * D, gNN = (kLean ? rates[1].x : q.gN) * N;
        uint64_t c0, c1;
        if (MODEL == 2) {
          c0 = F ? q.tD : 0ull;
          c1 = c0 + (R ? q.kd : 0ull);
        } else {
          c1 = y - (kLean ? rates[2].x * R - y18 : q.gR * R) - gNN - gDD;
          c0 = c1 - (kLean ? tv->q.kN : q.kN);
        }
        const uint64_t c2 = c1 + gDD, c3 = c2 + gNN;
        const uint32_t ch = static_cast<uint32_t>(r >= c0) + static_cast<uint32_t>(r >= c1) +
                            static_cast<uint32_t>(r >= c2) + static_cast<uint32_t>(r >= c3);
        code = ch;
        s = ch == 4u ? 2u : (ch & 1u);  // D, N, D, N, R
        gain = ch <= 1u;
        if (MODEL) {
          dD = ch == 0u ? 1 : ch == 2u ? -1 : 0;
          dN = ch == 1u ? 1 : ch == 3u ? -1 : 0;
          dR = ch == 4u ? -1 : (MODEL == 2 && ch == 1u) ? -1 : 0;
          several = (MODEL == 2 && ch == 1u) || r >= top;
          if (r >= top) {
            const bool rel = MODEL == 1 && r >= top + y17;  // R -> D + N
            code = rel ? kEvRelease : kEvBind;
            dD = MODEL == 2 ? 0 : rel ? 1 : -1;
            dN = rel ? 1 : -1;
            dR = rel ? -1 : 1;
          }
        }
      }
      const bool move = run && hop;
      // lane-wide nodes: u's entry in each, and what is there
      const uint32_t ku = u / RV, pu = u / MV % RAD;
      uint64_t xu = 0, fq = 0;
      if (MID) xu = tree[IX(kMid + ku * RAD + li, tree_n)];
      if (FOUR) fq = tree[IX(kFour + ((sl & 1u) ? u >> 2 : v >> 2), tree_n)];
      // differences of the totals of v and u
      const ulonglong2 gh = rates[IX(s, 3)];
      uint64_t dv, du = 0;
      uint32_t nc = 0, newmax = 0;
      {
        // one molecule of s more or less: a voxel's total is affine in D and in
        // N (R's Hill term follows below)
        uint64_t c = gh.x + gh.y * nn;
        if (MODEL == 1) c += s == 2u ? 0ull : q.k_in * (s == 0u ? N : D);
        if (MODEL == 2) c += s == 1u && F ? q.k_in : 0ull;
        dv = gain ? c : 0ull - c;
      }
      if (MODEL == 0) {
        nc = (s == 0u ? D : s == 1u ? N : R) + (gain ? 1u : 0xFFFFFFFFu);
        newmax = nc;
      } else {
        newmax = (D + dD) | (N + dN) | (R + dR);
        // binding, unbinding: two or three species change (not for lanes without a
        // cell: what they read can send the Hill term to its slow path)
        if (several && run) dv = lane_total<MODEL>(q, tv, D + dD, N + dN, R + dR, nn, ctr) - a_v;
      }
      uint32_t cu = 0;
      uint64_t a_u = 0, w_u = 0;  // records: u's total and word; sectors: its quad's sum and counts
      if (SEC) {
        const uint64_t* uq = rec + 4u * IX(u >> 2, rec_words / 4u);
        a_u = uq[0];
        w_u = uq[1u + s];
        cu = field16(w_u, u & 3u) + 1u;
        if (hop) {
          du = gh.x + gh.y * (lut[IX(u, lut_n)] >> 4);
          if (MODEL == 1 && s < 2u) du += q.k_in * field16(uq[2u - s], u & 3u);
          if (MODEL == 2 && s == 1u)
            du += q.k_in * (static_cast<uint32_t>(u == centre) - field16(uq[3], u & 3u));
        }
      } else if (PLN) {
        cu = hp[IX(s * ps + u, 3u * ps)] + 1u;
        if (hop) {
          du = gh.x + gh.y * (lut[IX(u, lut_n)] >> 4);
          if (MODEL == 1 && s < 2u) du += q.k_in * hp[IX((1u - s) * ps + u, 3u * ps)];
          if (MODEL == 2 && s == 1u)
            du += q.k_in * (static_cast<uint32_t>(u == centre) - hp[IX(2u * ps + u, 3u * ps)]);
        }
      } else if (REC) {
        const ulonglong2 x = reinterpret_cast<const ulonglong2*>(rec)[IX(u, rec_words / 2u)];
        a_u = x.x;
        w_u = x.y;
        if (hop) {
          du = gh.x + gh.y * static_cast<uint32_t>(__popc(word_mask(w_u)));
          if (MODEL == 1) du += s == 2u ? 0ull : q.k_in * (s == 0u ? word_N(w_u) : word_D(w_u));
          if (MODEL == 2 && s == 1u)
            du += q.k_in * (static_cast<uint32_t>(u == centre) - word_R(w_u));
        }
      } else {
        cu = static_cast<uint32_t>(cp[IX(s * ps + u, 3u * ps)]) + 1u;
        if (WIDE) a_u = tree[IX(kCnt + u, tree_n)];
        if (hop) {
          du = gh.x + gh.y * (lut[IX(u, lut_n)] >> 4);
          if (MODEL == 1 && s < 2u)
            du += q.k_in * static_cast<uint32_t>(cp[IX((1u - s) * ps + u, 3u * ps)]);
          if (MODEL == 2 && s == 1u)
            du += q.k_in * (static_cast<uint32_t>(u == centre) -
                            static_cast<uint32_t>(cp[IX(2u * ps + u, 3u * ps)]));
          newmax |= cu;
        }
      }
      // R changes the Hill term, here and where it arrives
      if (MODEL != 2 && s == 2u && run && !several) {
        // (records: the event that leaves the table reads its end; its cell is redone)
        const uint32_t Ru = !hop                       ? 1u
                            : LEAF == kLeafRecords ? min(word_R(w_u) + 1u, kHillTab - 1u)
                                                   : cu;
        if (!slow) {  // every count is inside the table
          dv += __ldg(q.hill + IX(R - 1u, kHillTab)) -
                __ldg(q.hill + IX(R, kHillTab));
          const uint64_t d = __ldg(q.hill + IX(Ru, kHillTab)) -
                             __ldg(q.hill + IX(Ru - 1u, kHillTab));
          if (hop) du += d;
        } else {
          dv += lane_hill(q.hill, tv, R - 1u) - lane_hill(q.hill, tv, R);
          if (hop) du += lane_hill(q.hill, tv, Ru) - lane_hill(q.hill, tv, Ru - 1u);
        }
      }
      // the sums along both paths.  Lane-wide nodes: every lane its entry, where
      // it comes after v's or u's.  Otherwise, one lane: all reads, then all
      // stores; more: lane pairs take the levels, the even lane v's entry, the
      // odd lane u's (v's adds both differences where the paths share the entry).
      if (WIDE) {
        const bool same = kv == ku;
        const uint64_t dvm = li > pv ? dv : 0ull, dum = li > pu ? du : 0ull;
        xm += dvm + (same ? dum : 0ull);
        xu += dum;
        if (run) X1 += (li > kv ? dv : 0ull) + (li > ku ? du : 0ull);
        __syncwarp();
        if (run) {
          if (MID && sl < RAD) {
            tree[IX(kMid + kv * RAD + li, tree_n)] = xm;
            if (!same) tree[IX(kMid + ku * RAD + li, tree_n)] = xu;
          }
          if (FOUR && sl < 2u) {
            const bool sq = (v >> 2) == (u >> 2);
            if (sl == 0u) tree[IX(kFour + (v >> 2), tree_n)] = fq + dv + (sq ? du : 0ull);
            else if (!sq) tree[IX(kFour + (u >> 2), tree_n)] = fq + du;
          }
          if (!REC) {
            if (sl == 0u) tree[IX(kCnt + v, tree_n)] = a_v + dv;
            if (sl == 1u && hop) tree[IX(kCnt + u, tree_n)] = a_u + du;
          }
        }
      } else if (ONE) {
        if (run) {
          // v's entries, then u's: one may be the other
#pragma unroll
          for (int side = 0; side < 2; ++side) {
            uint64_t x[SL];
#pragma unroll
            for (uint32_t l = 1; l <= SL; ++l)
              x[l - 1] = tree[IX(level_off(l) + ((side ? u : v) >> (2u * (LV - l))), tree_n)];
#pragma unroll
            for (uint32_t l = 1; l <= SL; ++l)
              tree[IX(level_off(l) + ((side ? u : v) >> (2u * (LV - l))), tree_n)] =
                  x[l - 1] + (side ? du : dv);
          }
        }
      } else {
        const bool odd = sl & 1u;
        const uint32_t me = odd ? u : v, other = odd ? v : u;
        const uint64_t dme = odd ? du : dv, dot = odd ? 0ull : du;
        __syncwarp();
        // level LV of the tree: the voxel totals themselves (shared leaves)
        constexpr uint32_t kTasks = 2u * (REC ? SL : LV);
        for (uint32_t t = sl; t < kTasks; t += G) {
          const uint32_t l = (t >> 1) + 1u;
          const uint32_t i1 = me >> (2u * (LV - l)), i2 = other >> (2u * (LV - l));
          uint64_t* at = tree + IX(level_off(l) + i1, tree_n);
          const bool same = i1 == i2;
          if (run && !(odd && same)) *at += dme + (same ? dot : 0ull);
        }
      }
      // the two voxels
      if (SEC) {
        // the quad's sum and the changed species' counts, here and at u
        const uint64_t at = 1ull << (16u * (v & 3u)), to = hop ? 1ull << (16u * (u & 3u)) : 0ull;
        const bool same = (v >> 2) == (u >> 2);
        uint64_t* vq = rec + 4u * IX(v >> 2, rec_words / 4u);
        const uint64_t w = (s == 0u ? sec.b : s == 1u ? sec.c : sec.d) + (gain ? at : 0ull - at);
        if (run && (ONE || sl == 0u)) {
          vq[0] = sec.a + dv + (same ? du : 0ull);
          if (MODEL != 0 && several) {
            vq[1] = sec.b + (dD > 0 ? at : dD < 0 ? 0ull - at : 0ull);
            vq[2] = sec.c + (dN > 0 ? at : 0ull - at);
            vq[3] = sec.d + (dR > 0 ? at : 0ull - at);
          } else {
            vq[1u + s] = w + (same ? to : 0ull);
          }
        }
        if (move && !same && (ONE || sl == 1u)) {
          uint64_t* uq = rec + 4u * IX(u >> 2, rec_words / 4u);
          uq[0] = a_u + du;
          uq[1u + s] = w_u + to;
        }
        const uint32_t lim_s = s == 2u ? lim_r : lim_dn;
        bool over = hop && cu >= lim_s;
        if (MODEL == 0) over = over || nc >= lim_s;
        else over = over || max(D + dD, N + dN) >= lim_dn || R + dR >= lim_r;
        if (run && over) err |= kErrNarrow;
      } else if (PLN) {
        if (run && lead) {
          if (MODEL == 0) {
            hp[IX(s * ps + v, 3u * ps)] = static_cast<uint16_t>(nc);
          } else {
            if (dD) hp[IX(v, 3u * ps)] = static_cast<uint16_t>(D + dD);
            if (dN) hp[IX(ps + v, 3u * ps)] = static_cast<uint16_t>(N + dN);
            if (dR) hp[IX(2u * ps + v, 3u * ps)] = static_cast<uint16_t>(R + dR);
          }
          if (hop) hp[IX(s * ps + u, 3u * ps)] = static_cast<uint16_t>(cu);
        }
        const uint32_t lim_s = s == 2u ? lim_r : lim_dn;
        bool over = hop && cu >= lim_s;
        if (MODEL == 0) over = over || nc >= lim_s;
        else over = over || max(D + dD, N + dN) >= lim_dn || R + dR >= lim_r;
        if (run && over) err |= kErrNarrow;
      } else if (REC) {
        const uint64_t one = word_unit(s);
        const uint64_t wv2 = MODEL == 0 ? (gain ? w_v + one : w_v - one)
                                        : pack_voxel(D + dD, N + dN, R + dR, mask);
        const uint64_t wu2 = w_u + one;
        if (run && (ONE || sl == 0u)) {
          reinterpret_cast<ulonglong2*>(rec)[IX(v, rec_words / 2u)] =
              make_ulonglong2(a_v + dv, wv2);
        }
        if (move && (ONE || sl == 1u)) {
          reinterpret_cast<ulonglong2*>(rec)[IX(u, rec_words / 2u)] =
              make_ulonglong2(a_u + du, wu2);
        }
        if (run && (((wv2 | (hop ? wu2 : 0ull)) & over_mask) != 0ull)) err |= kErrNarrow;
      } else {
        if (run && lead) {
          if (MODEL == 0) {
            cp[IX(s * ps + v, 3u * ps)] = static_cast<int32_t>(nc);
          } else {
            if (dD) cp[IX(v, 3u * ps)] = static_cast<int32_t>(D + dD);
            if (dN) cp[IX(ps + v, 3u * ps)] = static_cast<int32_t>(N + dN);
            if (dR) cp[IX(2u * ps + v, 3u * ps)] = static_cast<int32_t>(R + dR);
          }
          if (hop) cp[IX(s * ps + u, 3u * ps)] = static_cast<int32_t>(cu);
        }
      }
      if (!ONE) __syncwarp();
      if (sl == i) {
        Aj = A;
        log = v | (u << 10) | (code << 20);
      }
      if (run) {
        A += dv + du;
        m = i + 1u;
        if (REC) {
          run = err == 0;
        } else if (!big && newmax >= (MODEL == 2 || (MODEL == 0 && s != 2u) ? q.small : lim)) {
          big = paused = true;  // its limits are checked below, the next batch's in it
          run = false;
        }
      }
      if (slow) {  // cells past those limits: checked exactly
        if (run && big &&
            past_limits<MODEL>(tv, cp, ps, lut, IX(v, lut_n), IX(u, lut_n), centre)) {
          err |= kErrOverflow;
          run = false;
        }
        if (!ONE) __syncwarp();
      }
      if (kChecked) {  // an index of the event out of range, on any of the cell's lanes
        const unsigned bad = __ballot_sync(kFull, oob && ran) >> base_lane;
        if (bad & (G == 32 ? kFull : (1u << (G & 31)) - 1u)) {
          err |= kErrBounds;
          run = false;
        }
        oob = false;
      }
    }
    if (!REC && __any_sync(kFull, paused)) {
      const uint32_t last = ONE ? log : __shfl_sync(kFull, log, base_lane + static_cast<int>(m ? m - 1u : 0u));
      if (paused && past_limits<MODEL>(tv, cp, ps, lut, IX(last & 1023u, lut_n),
                                       IX((last >> 10) & 1023u, lut_n), centre)) {
        err |= kErrOverflow;
        paused = false;
      }
      __syncwarp();
    }

    // ---- the waiting times of the applied events, added in order -----------
    if (HELP) {
      Em = ex->Em[phase][lane];
      Ek = ex->Ek[phase][lane];
      phase ^= 1u;
    }
    const double tau = tau_from(F53{Em, Ek}, Ek < 0 || Aj == 0ull, Aj | (Aj == 0ull));
    uint32_t fired = 0;
    if (ONE) {
      const double tn = __dadd_rn(tnow, tau);
      if (m && before(tn, p.dt)) {
        tnow = tn;
        fired = 1;
      }
    } else {
      // Lane j's time after event j.  While t stays in one binade a binary64
      // sum t + tau is t's bits plus tau rounded to t's last place (ties
      // apart), whatever t is: the rounded taus are integers, and a scan adds
      // them.  Otherwise one addition after the other.
      const uint64_t tb = static_cast<uint64_t>(__double_as_longlong(tnow));
      bool tie = false;
      const uint64_t ulps = ulps_of(tau, static_cast<int>(tb >> 52), tie);
      uint64_t sum = ulps;
#pragma unroll
      for (int o = 1; o < G; o <<= 1) {
        const uint64_t x = __shfl_up_sync(kFull, sum, o, G);
        if (static_cast<int>(sl) >= o) sum += x;
      }
      double mine = __longlong_as_double(static_cast<long long>(tb + sum));
      const bool same = ((tb + sum) >> 52) == (tb >> 52) && !tie && tb != 0ull;
      if (!__all_sync(kFull, same || !have)) {
        double t = tnow;
#pragma unroll
        for (uint32_t j = 0; j < static_cast<uint32_t>(G); ++j) {
          t = __dadd_rn(t, __shfl_sync(kFull, tau, base_lane + static_cast<int>(j)));
          if (sl == j) mine = t;
        }
      }
      // times only grow, so the events that fire are the leading ones
      const unsigned late = __ballot_sync(kFull, !(sl < m && before(mine, p.dt))) >> base_lane;
      fired = min(static_cast<uint32_t>(G), static_cast<uint32_t>(__ffs(static_cast<int>(late))) - 1u);
      const double tl = __shfl_sync(kFull, mine, base_lane + static_cast<int>(fired ? fired - 1u : 0u));
      if (fired) tnow = tl;
    }
    if (fired < m) err &= ~(kErrOverflow | kErrNarrow);  // the event that met a limit did not fire
    const uint32_t e = e0 + fired;
    if (have && fired == batch && e >= 0xFFFFFFFFu - 32u) err |= kErrEventIndex;
    bool fin = have && (err != 0 || fired < m || (m < batch && !paused));
    e0 = e;
    unsigned out = __ballot_sync(kFull, fin && lead);
    if (out) {
      if (REC) {
        // cells that met a limit: other limits, from what they hold now, the whole
        // warp one cell at a time
        unsigned met = __ballot_sync(kFull, fin && lead && (err & kErrNarrow) && m);
        if (met) __syncwarp();  // the counts that other lanes wrote
        for (; met; met &= met - 1u) {
          const uint32_t sc = static_cast<uint32_t>(__ffs(met) - 1) / G;
          const uint64_t* words =
              PLN ? reinterpret_cast<const uint64_t*>(warp_cells + sc * p.cell_stride + 48) + kCnt
                  : warp_rec + static_cast<size_t>(sc) * rec_words;
          Limits now{0, 0, 0}, next{1, 1, 1};
#pragma unroll 1
          for (uint32_t i = lane; i < V; i += 32u) {
            uint32_t D, N, R;
            if (LEAF == kLeafRecords) {
              const uint64_t w = words[IX(2u * i + 1u, rec_words)];
              D = word_D(w), N = word_N(w), R = word_R(w);
            } else {
              const uint64_t* x = SEC ? words + 4u * IX(i >> 2, rec_words / 4u) + 1u
                                      : words + IX(i >> 2, nq);
              const uint32_t dist = SEC ? 1u : nq, k = i & 3u;
              D = field16(x[0], k), N = field16(x[dist], k), R = field16(x[2u * dist], k);
            }
            now = Limits{max(now.D, D), max(now.N, N), max(now.R, R)};
          }
          now = warp_max(now);
          if (slot == sc && pick_limits<MODEL, LEAF>(tv, now, next)) {
            set_limits(next);
            err &= ~kErrNarrow;
            fin = err != 0;
          }
        }
      }
      // undo the events past the end of the step (counts only), every lane its
      // own: the changes commute
      if (fin && sl >= fired && sl < m) {
        const uint32_t v = log & 1023u, u = (log >> 10) & 1023u, code = log >> 20;
        int cD = 0, cN = 0, cR = 0;  // back at v
        if (code == kEvBind || code == kEvRelease) {
          cN = code == kEvBind ? 1 : -1;
          cD = MODEL != 2 ? cN : 0;
          cR = -cN;
        } else {
          const uint32_t s = code >= kEvHop ? code - kEvHop : code == 4u ? 2u : (code & 1u);
          const int c = code <= 1u ? -1 : 1;
          cD = s == 0u ? c : 0;
          cN = s == 1u ? c : 0;
          cR = s == 2u || (MODEL == 2 && code == 1u) ? 1 : 0;
        }
        const uint32_t su = code - kEvHop;  // hops: the species taken back from u
        if (SEC) {
          uint64_t* w = rec + 4u * IX(v >> 2, rec_words / 4u) + 1u;
          const uint32_t sh = 16u * (v & 3u);
          if (cD) add64(w, static_cast<uint64_t>(static_cast<int64_t>(cD)) << sh);
          if (cN) add64(w + 1, static_cast<uint64_t>(static_cast<int64_t>(cN)) << sh);
          if (cR) add64(w + 2, static_cast<uint64_t>(static_cast<int64_t>(cR)) << sh);
          if (code >= kEvHop)
            add64(rec + IX(4u * (u >> 2) + 1u + su, rec_words), 0ull - (1ull << (16u * (u & 3u))));
        } else if (PLN) {
          // whole 32-bit words: the sum of all changes is in range, so carries
          // between the halves cancel
          auto add16 = [&](uint32_t at, int c) {
            atomicAdd(reinterpret_cast<uint32_t*>(hp) + IX(at >> 1, 3u * ps / 2u),
                      static_cast<uint32_t>(c) << (16u * (at & 1u)));
          };
          if (cD) add16(v, cD);
          if (cN) add16(ps + v, cN);
          if (cR) add16(2u * ps + v, cR);
          if (code >= kEvHop) add16(su * ps + u, -1);
        } else if (REC) {
          add64(rec + IX(2u * v + 1u, rec_words),
                word_unit(0) * static_cast<uint64_t>(static_cast<int64_t>(cD)) +
                    word_unit(1) * static_cast<uint64_t>(static_cast<int64_t>(cN)) +
                    word_unit(2) * static_cast<uint64_t>(static_cast<int64_t>(cR)));
          if (code >= kEvHop) add64(rec + IX(2u * u + 1u, rec_words), 0ull - word_unit(su));
        } else {
          if (cD) atomicAdd(cp + IX(v, 3u * ps), cD);
          if (cN) atomicAdd(cp + IX(ps + v, 3u * ps), cN);
          if (cR) atomicAdd(cp + IX(2u * ps + v, 3u * ps), cR);
          if (code >= kEvHop) atomicAdd(cp + IX(su * ps + u, 3u * ps), -1);
        }
      }
      __syncwarp();
      if (REC && fin && lead && (err & kErrNarrow)) {
        // left as it was, for the 32-bit pass
        p.redo[IX(atomicAdd(p.redo_n, 1u), p.n_items)] =
            make_uint2(HELP ? home[5] : vidx, HELP ? home[1] : cell);
      } else if (fin && lead) {
        const uint32_t cells = kChecked ? tv->width * tv->height : 0u;
        const uint32_t c = IX(HELP ? home[1] : cell, cells);
        tv->ev_last[c] = e;
        tv->t_last[c] = tnow;
        tv->ev_total[c] += e;
        if (err) atomicOr(tv->err, err);
      }
      // the counts back to the state array, the whole warp one cell at a time
      out = __ballot_sync(kFull, fin && lead && !(REC && (err & (kErrNarrow | kErrState))));
      while (out) {
        const int src = __ffs(out) - 1;
        out &= out - 1u;
        const uint32_t sc = static_cast<uint32_t>(src) / G;
        const uint32_t c = HELP ? ex->home[sc][1] : __shfl_sync(kFull, cell, src);
        const uint32_t vi = HELP ? ex->home[sc][5] : __shfl_sync(kFull, vidx, src);
        int32_t* g = p.views[vi].counts + static_cast<size_t>(c) * 3u * V;
        if (SEC) {
          const uint64_t* from = warp_rec + static_cast<size_t>(sc) * rec_words;
          if (vec) {
            for (uint32_t i = lane; i < nq; i += 32u) {
              const U64x4 x = load4(from + 4u * IX(i, rec_words / 4u));
              reinterpret_cast<uint4*>(g)[IX(i, V / 4u)] = unpack4(x.b);
              reinterpret_cast<uint4*>(g + V)[IX(i, V / 4u)] = unpack4(x.c);
              reinterpret_cast<uint4*>(g + 2u * V)[IX(i, V / 4u)] = unpack4(x.d);
            }
          } else {
            for (uint32_t i = lane; i < V; i += 32u)
              for (uint32_t sp = 0; sp < 3u; ++sp)
                g[IX(sp * V + i, 3u * V)] =
                    static_cast<int32_t>(field16(from[IX(4u * (i >> 2) + 1u + sp, rec_words)],
                                                 i & 3u));
          }
        } else if (PLN) {
          const uint64_t* from =
              reinterpret_cast<const uint64_t*>(warp_cells + sc * p.cell_stride + 48) + kCnt;
          for (uint32_t sp = 0; sp < 3u; ++sp) {
            if (vec) {
              for (uint32_t i = lane; i < nq; i += 32u)
                reinterpret_cast<uint4*>(g + sp * V)[IX(i, V / 4u)] =
                    unpack4(from[IX(sp * nq + i, 3u * nq)]);
            } else {
              for (uint32_t i = lane; i < V; i += 32u)
                g[IX(sp * V + i, 3u * V)] =
                    static_cast<int32_t>(field16(from[IX(sp * nq + (i >> 2), 3u * nq)], i & 3u));
            }
          }
        } else if (REC) {
          const uint64_t* from = warp_rec + static_cast<size_t>(sc) * rec_words;
          if (vec) {
            for (uint32_t i = lane; i < nq; i += 32u) {
              const uint64_t* at = from + 8u * IX(i, rec_words / 8u);
              const U64x4 x = load4(at), y = load4(at + 4u);
              const U64x4 w{x.b, x.d, y.b, y.d};
              reinterpret_cast<uint4*>(g)[IX(i, V / 4u)] =
                  make_uint4(word_D(w.a), word_D(w.b), word_D(w.c), word_D(w.d));
              reinterpret_cast<uint4*>(g + V)[IX(i, V / 4u)] =
                  make_uint4(word_N(w.a), word_N(w.b), word_N(w.c), word_N(w.d));
              reinterpret_cast<uint4*>(g + 2u * V)[IX(i, V / 4u)] =
                  make_uint4(word_R(w.a), word_R(w.b), word_R(w.c), word_R(w.d));
            }
          } else {
            for (uint32_t i = lane; i < V; i += 32u) {
              const uint64_t w = from[IX(2u * i + 1u, rec_words)];
              g[IX(i, 3u * V)] = static_cast<int32_t>(word_D(w));
              g[IX(V + i, 3u * V)] = static_cast<int32_t>(word_N(w));
              g[IX(2u * V + i, 3u * V)] = static_cast<int32_t>(word_R(w));
            }
          }
        } else {
          const int32_t* from = reinterpret_cast<const int32_t*>(
              reinterpret_cast<const uint64_t*>(warp_cells + sc * p.cell_stride + 48) + kCnt + ps);
          for (uint32_t sp = 0; sp < 3u; ++sp) {
            if (vec) {
              for (uint32_t i = lane; i < nq; i += 32u)
                reinterpret_cast<int4*>(g + sp * V)[IX(i, V / 4u)] =
                    reinterpret_cast<const int4*>(from + sp * ps)[IX(i, nq)];
            } else {
              for (uint32_t i = lane; i < V; i += 32u)
                g[IX(sp * V + i, 3u * V)] = from[IX(sp * ps + i, 3u * ps)];
            }
          }
        }
      }
      if (kChecked && oob) {
        atomicOr(tv->err, kErrBounds);
        oob = false;
      }
      __syncwarp();
      if (fin) {
        have = false;
        err = 0;
        A = 0;
      }
    }
  }
}

#undef IX

// The instantiations the launch plan picks from.
template <int MODEL>
ChiLaneKernel lane_instance(uint32_t V, int leaf, uint32_t G, uint32_t helper) {
  const int lv = V <= 64 ? 3 : V <= 256 ? 4 : 5;
#define LANE_CASE(L, F, N, H) \
  if (lv == L && leaf == F && G == N && helper == H) return k_chi_lane<MODEL, L, F, N, H>
  LANE_CASE(3, kLeafShared, 32, 6);
  LANE_CASE(3, kLeafShared, 32, 0);
  LANE_CASE(3, kLeafShared, 16, 6);
  LANE_CASE(3, kLeafShared, 16, 0);
  LANE_CASE(3, kLeafShared, 8, 6);
  if constexpr (MODEL != 1) LANE_CASE(3, kLeafShared, 8, 8);
  LANE_CASE(3, kLeafShared, 8, 0);
  LANE_CASE(3, kLeafShared, 4, 0);
  LANE_CASE(3, kLeafRecords, 1, 8);
  LANE_CASE(3, kLeafRecords, 1, 6);
  LANE_CASE(3, kLeafRecords, 1, 0);
  LANE_CASE(4, kLeafShared, 32, 6);
  LANE_CASE(4, kLeafShared, 32, 0);
  LANE_CASE(4, kLeafShared, 16, 6);
  LANE_CASE(4, kLeafShared, 16, 0);
  LANE_CASE(4, kLeafShared, 8, 6);
  if constexpr (MODEL != 1) LANE_CASE(4, kLeafShared, 8, 8);
  LANE_CASE(4, kLeafShared, 8, 0);
  LANE_CASE(4, kLeafShared, 4, 0);
  LANE_CASE(4, kLeafRecords, 4, 0);
  LANE_CASE(4, kLeafSectors, 1, 8);
  LANE_CASE(4, kLeafSectors, 1, 6);
  LANE_CASE(4, kLeafSectors, 1, 0);
  LANE_CASE(5, kLeafShared, 32, 6);
  LANE_CASE(5, kLeafShared, 16, 6);
  LANE_CASE(5, kLeafPlanes, 16, 6);
  LANE_CASE(5, kLeafPlanes, 16, 8);
  LANE_CASE(5, kLeafPlanes, 16, 0);
  LANE_CASE(4, kLeafPlanes, 8, 0);
  LANE_CASE(4, kLeafPlanes, 4, 0);
  LANE_CASE(3, kLeafPlanes, 4, 0);
  LANE_CASE(5, kLeafRecords, 16, 0);
  LANE_CASE(5, kLeafRecords, 8, 0);
  LANE_CASE(5, kLeafSectors, 1, 6);
  LANE_CASE(5, kLeafSectors, 1, 0);
#undef LANE_CASE
  return nullptr;
}

}  // namespace

}  // namespace tsg
