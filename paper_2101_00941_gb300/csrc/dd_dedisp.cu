// Tiled brute-force dedispersion for sm_103a (Sec. 2.1 "dedispersion of data"; the sum is the
// plain definition y[i][j] = sum_c x_d[c][j + s[i][c]], computed exactly in integers).
//
// One CTA owns a tile of D consecutive DM trials x TT output samples of one range and walks the
// channels in stages of kNG groups of eight channels. Tile shapes (the plan picks one by the
// launch's estimated work, or times them all): 64 x 512 or 128 x 256 with 16 warps (128 registers
// per thread, 64 accumulators per lane), 64 x 512 with 32 warps (64 registers, 32 accumulators:
// twice the warps on the same tables and shared memory), and 64 x 256 or 32 x 256 with 16 warps,
// two CTAs per SM. Bound by the shared-memory pipe (71% busy) and instruction issue (58%): 1216
// trials x 65536 outputs x 4096 channels take 6.3 ms (uint8; 8.5 before the class chains, the
// packed sums, the 128-trial tile and leaner stages, 6.8 with the first two of them alone).
//
//   * Delay classes. For an 8-channel group the tile's trials fall into a few classes by the
//     relative delays (r0..r7) of the eight channels. A class shares one sequence of sums
//        S_p[u] = x[c0][a+u+r0] + .. + x[c7][a+u+r7]
//     that each of its trials reads at its own base offset, stored as "pair words"
//        Z_p[u] = S_p[u] | S_p[u+1] << 16
//     (exact in 16-bit lanes: two groups' sums stay below 2^16 for d <= 16). The even and odd
//     pair words are kept in two planes, so a lane that owns outputs 2m and 2m+1 of a trial
//     reads one word, and consecutive lanes read consecutive words. The classes depend on the
//     delay table only, so the plan computes them once (tiled_plan, below) as one table per
//     (trial tile, stage), together with a balanced split of the stage's word building over the
//     warps; the kernel never searches for them.
//   * Class chains. Sorted by their delay sums, a group's classes differ from their neighbours
//     by about one channel moved by one sample (about 7 classes and 7 such steps per group on
//     the 4096-channel plan). A warp therefore sums all eight channels for the first class of
//     its share only and reaches each further class by the steps x[r + 1] - x[r] of the moved
//     channels, in the same packed 16-bit lanes (exact: the arithmetic is modulo 2^32 and each
//     class's own sums fit their lanes).
//   * TMA brings each stage's 16 channel rows (one 3-D tensor copy: every row from the same
//     128-byte segment on, so each lands contiguous) and its class table into shared memory
//     NS - 1 stages ahead (NS = 4 staging buffers, or 3 where 4 do not fit shared memory);
//     completion is tracked by mbarriers with bounded waits.
//   * The main loop adds, per (trial, output pair), the two groups' pair words to a packed
//     accumulator with one three-input add: one 32-bit shared-memory load per sixteen
//     channel-adds, for uint8 and uint16 (decimated) data alike. Every TiledArgs::flush stages,
//     before a 16-bit lane can overflow, two DP2As add the packed sums to the 32-bit outputs.
//
// Software pipeline, one __syncthreads per stage s:
//     TMA for stage s+NS-1 | build the words of stage s+1 | accumulate stage s
// Words are built from 32-bit loads and funnel shifts; the eight-channel sums are formed in SWAR
// lanes (bytes split into 16-bit lanes for uint8 data). Where a class's rows start in a stage
// buffer is known at plan time up to the copy's phase within its first segment, one value per
// stage and tile, which the build adds to the plan's offsets. Exact
// moments (S1, 128-bit S2) of every series are added in the epilogue with integer atomics, so
// the search needs no second statistics pass.
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>

#include "dd_internal.h"

namespace ddk {

namespace {

constexpr int kMaxTileTrials = 128;        // trials per tile: 128, 64 or 32
constexpr int kFusedTrials = 64;           // ... of the fused form
constexpr int kThreads = 512;               // threads of the 16-warp shapes
constexpr int kWarps = kThreads / 32;
constexpr int kMaxWarps = 32;
constexpr int kG = 8;                       // channels per group (one delay class)
constexpr int kNG = 2;                      // groups per stage
constexpr int kRows = kG * kNG;             // channel rows per stage
constexpr int kMaxNStage = 4;               // staging buffers (rows + class table), at most
constexpr int kMaxCls = 24;                 // classes per group of a 128-trial tile
constexpr int kMaxCls64 = 16;               // ... of a smaller one
constexpr int kMaxSteps = 3;                // channel steps between chained classes
constexpr int kMaxLinks = 32;               // chain links (classes and in-between steps) per group
constexpr int kBlock = 31;                  // build units stored per 32-lane block
constexpr int kSegBytes = 128;              // inner extent of a staged-row copy (tensor map)
constexpr size_t kSmemLimit = 226 * 1024;   // dynamic shared memory a CTA may plan for: 227 KB
                                            // less the persistent form's static 1 KB
constexpr size_t kSmemLimit2 = 110 * 1024;  // ... when two CTAs share an SM

// CTAs per SM a tile shape is compiled for (its register budget: 65536 / (NT x CTAs)).
__host__ __device__ constexpr int tile_ctas(int D, int TT, int NT) {
  return (NT == 1024 || D * TT == 64 * 512) ? 1 : 2;
}

// Entry of trial t of a tile in a stage's word offsets for a CTA of W warps with tpw trials per warp:
// warp t mod W reads its trials t, t + W, ... as tpw consecutive entries.
__host__ __device__ constexpr int trial_slot(int t, int W, int tpw) { return (t % W) * tpw + t / W; }

// One link of a group's chain: a delay class, or a step between two classes that are several
// channel steps apart (un = 0: it stores nothing). A group's classes share a frame of pair words:
// frame word v of a class is the sum that a trial of smallest delay b in the class uses for
// output v - (b - F), F being the group's smallest delay. A unit is 4 (uint8) or 2 (uint16)
// consecutive frame words; the class stores units ulo .. ulo + un - 1. Row offsets are byte
// offsets within the stage buffer for frame word 0, before the copy's phase is added. step: the
// channel step that leads here from the preceding link, the row offset of x[r] of x[r + 1] - x[r]
// with the step's sign in the top two bits (01: add, 11: subtract); 0 for the first link of a
// chain.
struct ClsLink {
  uint32_t off[kG];
  uint32_t step;
  int32_t ev, od;  // byte offset of frame word 0's place in the even plane, word 1's in the odd
  uint32_t range;  // ulo | un << 16
  __host__ __device__ uint32_t ulo() const { return range & 0xFFFFu; }
  __host__ __device__ uint32_t un() const { return range >> 16; }
};
static_assert(sizeof(ClsLink) == 48, "read as three 16-byte words");
constexpr uint32_t kStepOff = 0x0000FFFFu, kStepAdd = 0x40000000u, kStepSub = 0xC0000000u;

// A build task: units u0 .. u0 + 30 of a run of chained links of one group. link: byte offset of
// the first link in the stage's table | (links - 1) << 16.
struct BuildTask {
  uint32_t link, u0;
};

// A stage's table: this head, the byte offset of each trial's sequence in the stage's words
// (uint32 [kNG][trials per tile], entry trial_slot(t); 0: no trial), the links (group 0's, then
// group 1's) and the build tasks. Warp w runs the tasks of wtask[w].
struct StageTab {
  uint32_t wtask[kMaxWarps];  // byte offset of the first task in the table | tasks << 16
  uint8_t nlink[kNG];
  uint8_t pad[6];
  int32_t xmin;  // smallest delay of the stage's rows for the tile's first trial
  int32_t pad1;
};
static_assert(sizeof(StageTab) % 16 == 0, "class tables are copied in 16-byte units");
// where the links of a table for D trials start
__host__ __device__ constexpr uint32_t links_at(int D) {
  return (uint32_t)sizeof(StageTab) + 4u * kNG * (uint32_t)D;
}
constexpr int kMaxRun = 16;

__host__ __device__ constexpr size_t align16(size_t v) { return (v + 15) & ~size_t(15); }

struct SmemLayout {
  size_t raw, z, tab, mbar, total;
};

// The mbarriers come first, at the same place for every tile shape and range (a persistent CTA
// re-initialises them between tiles of different ranges); the staged rows start 128-byte aligned.
__host__ __device__ inline SmemLayout smem_layout(int es, int row_slot, int zcap, int pitch,
                                                  int nst) {
  SmemLayout L;
  L.mbar = 0;
  size_t off = 128;
  L.raw = off;
  off = align16(off + (size_t)nst * kRows * row_slot * es);
  L.z = off;
  off = align16(off + (size_t)2 * zcap * 4);
  L.tab = off;
  off = align16(off + (size_t)pitch * nst);
  L.total = off;
  return L;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

template <int OFF>  // 32-bit shared-memory load at a byte address + OFF
__device__ __forceinline__ uint32_t lds(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
  return v;
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait for a stage with a bound: at most 2 s and 2^26 polls; false if it ran out.
__device__ bool mbar_wait_bounded(unsigned long long* bar, uint32_t parity) {
  const unsigned long long t0 = globaltimer_ns();
  for (int it = 0; it < (1 << 26); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255) == 255 && globaltimer_ns() - t0 > 2000000000ull) return false;
  }
  return false;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// First row segment of a stage's copy: every row is copied from the segment holding sample
// m0 + j0 + xmin on, xmin being the smallest delay of the stage's rows.
template <typename T>
__device__ __forceinline__ int64_t first_seg(const TiledArgs& a, int64_t j0, int32_t xmin) {
  constexpr int SEG = kSegBytes / (int)sizeof(T);  // elements per segment
  return (a.m0 + j0 + xmin) / SEG;
}

__device__ __forceinline__ int32_t stage_xmin(const TiledArgs& a, int stage, int nstages,
                                              int tile) {
  if (stage >= nstages) return 0;
  return __ldg(&reinterpret_cast<const StageTab*>(
                    a.tabs + ((size_t)tile * nstages + stage) * a.tab_pitch)->xmin);
}

// Issue of one stage by one thread: one tensor copy of the stage's 16 rows (segments
// [first_seg, first_seg + nseg) of each; rows past the padded channels read as zeros) and one
// bulk copy of its class table, after arming the stage's mbarrier with their bytes.
template <typename T>
__device__ __forceinline__ void issue_stage(const TiledArgs& a, int stage, int nstages,
                                            T* raw_buf, unsigned char* tab_buf,
                                            unsigned long long* bar, int32_t xmin, int64_t j0,
                                            int tile) {
  const uint32_t row_bytes = (uint32_t)a.row_slot * (uint32_t)sizeof(T);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  mbar_arrive_expect_tx(bar, kRows * row_bytes + (uint32_t)a.tab_pitch);
  const int32_t seg = (int32_t)first_seg<T>(a, j0, xmin);
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(raw_buf)),
      "l"(reinterpret_cast<uint64_t>(&a.rows)), "r"(0), "r"(seg), "r"(stage * kRows),
      "r"(smem_addr(bar))
      : "memory");
  bulk_g2s(tab_buf, a.tabs + ((size_t)tile * nstages + stage) * a.tab_pitch,
           (uint32_t)a.tab_pitch, bar);
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr));
  return v;
}

template <typename T>
struct Word;

// The two row words holding a lane's samples of one channel: off is the row offset (a step's sign
// may sit above bit 29), base the stage buffer's shared address plus the copy's phase and one word
// per unit. The sum's low two bits and its low five bits times eight are the byte and the funnel
// shift; a shared address has 18 bits. Returns 8 x the sum (shift amounts are taken modulo 32).
__device__ __forceinline__ uint32_t row_words(uint32_t base, uint32_t off, uint32_t& w0,
                                              uint32_t& w1) {
  const uint32_t at = base + off, addr = at & 0x3FFFCu;
  w0 = lds<0>(addr);
  w1 = lds<4>(addr);
  return at << 3;
}

// uint8 data. Unit u covers pair words 4u .. 4u + 3, i.e. the eight-channel sums
// S[4u .. 4u + 4] (one more than its words, which the last pair word needs). A channel's two row
// words are funnel-shifted to the unit's first sample; bytes are split into even/odd 16-bit lanes
// so that eight channels add without carries (8 x 255 < 2^16). The fifth sum is the next unit's
// first one, S[4(u + 1)]: the next lane's, taken with one shuffle. So a block of 32 lanes stores
// 31 units (lanes 0 .. 30); lane 31 computes the next block's first unit only to hand its first
// sum to lane 30. The pair words go to the class's even plane (4u, 4u + 2) and odd plane (4u + 1,
// 4u + 3); lanes take consecutive units, so every load and store is free of bank conflicts.
template <>
struct Word<uint8_t> {
  static constexpr int kUnit = 4;  // pair words per unit
  uint32_t e = 0, o = 0;           // samples (0, 2) and (1, 3) in 16-bit lanes
  __device__ __forceinline__ void add(uint32_t base, uint32_t off) {
    uint32_t w0, w1;
    const uint32_t w8 = row_words(base, off, w0, w1);
    const uint32_t a = __funnelshift_r(w0, w1, w8);  // samples 0..3 in bytes 0..3
    e += a & 0x00FF00FFu;
    o += __byte_perm(a, 0, 0x4341);
  }
  // one channel's samples r .. r + 3 replaced by r + 1 .. r + 4 (sign 1) or the reverse (-1)
  __device__ __forceinline__ void step(uint32_t base, uint32_t off, int sign) {
    uint32_t w0, w1;
    const uint32_t w8 = row_words(base, off, w0, w1);
    const uint32_t a = __funnelshift_r(w0, w1, w8);
    const uint32_t x4 = __funnelshift_r(w1, w1, w8);               // sample 4 in byte 0
    const uint32_t a02 = a & 0x00FF00FFu, a13 = __byte_perm(a, 0, 0x4341);
    const uint32_t a24 = __byte_perm(a, x4, 0x0402) & 0x00FF00FFu;  // samples 2, 4
    e += (a13 - a02) * (uint32_t)sign;
    o += (a24 - a13) * (uint32_t)sign;
  }
  __device__ __forceinline__ void emit(uint32_t ev, uint32_t od, uint32_t v, uint32_t n) const {
    const uint32_t nx = __shfl_down_sync(0xffffffffu, e, 1);  // low half: S4 (next unit's S0)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.lt.u32 p, %6, %7;\n\t"
        "@p st.shared.v2.u32 [%0], {%2, %3};\n\t"
        "@p st.shared.v2.u32 [%1], {%4, %5};\n\t}" ::"r"(ev),
        "r"(od), "r"(__byte_perm(e, o, 0x5410)),   // S0 | S1 << 16
        "r"(__byte_perm(e, o, 0x7632)),            // S2 | S3 << 16
        "r"(__byte_perm(o, e, 0x7610)),            // S1 | S2 << 16
        "r"(__byte_perm(o, nx, 0x5432)),           // S3 | S4 << 16
        "r"(v), "r"(n)
        : "memory");
  }
};

// uint16 data. Unit u covers pair words 2u, 2u + 1 (sums S[2u .. 2u + 2], the third the next
// lane's first) from two row words per channel; 16-bit lanes add eight channels without carries
// (8 x 255 x d < 2^16).
template <>
struct Word<uint16_t> {
  static constexpr int kUnit = 2;
  uint32_t e = 0;  // samples 0, 1
  __device__ __forceinline__ void add(uint32_t base, uint32_t off) {
    uint32_t w0, w1;
    const uint32_t w8 = row_words(base, off, w0, w1);
    e += __funnelshift_r(w0, w1, w8);
  }
  __device__ __forceinline__ void step(uint32_t base, uint32_t off, int sign) {
    uint32_t w0, w1;
    const uint32_t w8 = row_words(base, off, w0, w1);
    const uint32_t a = __funnelshift_r(w0, w1, w8);
    const uint32_t x2 = __funnelshift_r(w1, w1, w8);  // sample 2 in the low half
    e += (__byte_perm(a, x2, 0x5432) - a) * (uint32_t)sign;
  }
  __device__ __forceinline__ void emit(uint32_t ev, uint32_t od, uint32_t v, uint32_t n) const {
    const uint32_t nx = __shfl_down_sync(0xffffffffu, e, 1);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.lt.u32 p, %4, %5;\n\t"
        "@p st.shared.u32 [%0], %2;\n\t"
        "@p st.shared.u32 [%1], %3;\n\t}" ::"r"(ev),
        "r"(od), "r"(e),                  // S0 | S1 << 16
        "r"(__byte_perm(e, nx, 0x5432)),  // S1 | S2 << 16
        "r"(v), "r"(n)
        : "memory");
  }
};

// Add one pair word's two packed sums to the two outputs it serves.
__device__ __forceinline__ void pair_add(uint32_t z, uint32_t& even, uint32_t& odd) {
  even = __dp2a_lo(z, 0x0001u, even);  // + low half
  odd = __dp2a_lo(z, 0x0100u, odd);    // + high half
}

// Build one warp's share of a stage's pair words: per task (a run of chained links, one block
// of 31 units; lane l takes unit 31 * block + l) the eight channels of the first class, then per
// further link the channel step that leads to it. Every lane runs every unit (the shuffle needs
// them all); lanes 0 .. 30 store the units inside the class's own range. Loads of lanes past the
// staged rows stay inside the CTA's shared memory (the rows are followed by the word planes).
// The loop counts come from warp reductions, which the compiler knows to be the same in every
// lane: the loops then need no divergence bookkeeping.
template <typename T>
__device__ __forceinline__ void build_stage(uint32_t tabp, uint32_t rawb, uint32_t zb,
                                            uint32_t pos, int warp, int lane) {
  constexpr uint32_t SEG = kSegBytes / sizeof(T);
  constexpr uint32_t ZU = 4u * (Word<T>::kUnit / 2);  // plane bytes per unit
  uint32_t wt;
  asm volatile("ld.shared.u32 %0, [%1];"
               : "=r"(wt)
               : "r"(tabp + (uint32_t)offsetof(StageTab, wtask) + 4u * warp));
  const uint32_t xmin = lds<offsetof(StageTab, xmin)>(tabp);
  const uint32_t base0 =
      rawb + ((pos + xmin) & (SEG - 1)) * (uint32_t)sizeof(T) + 4u * (uint32_t)lane;
  const uint32_t zl0 = zb + ZU * (uint32_t)lane;
  const uint32_t us0 = lane < kBlock ? (uint32_t)lane : 0x80000000u;  // lane 31 stores nothing
  uint32_t tp = tabp + (wt & 0xFFFFu);
  for (uint32_t left = __reduce_max_sync(0xffffffffu, wt >> 16); left > 0; --left, tp += 8) {
    uint32_t tl, u0;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(tl), "=r"(u0) : "r"(tp));
    uint32_t n = __reduce_max_sync(0xffffffffu, tl >> 16);
    uint32_t cp = tabp + (tl & 0xFFFFu);
    const uint32_t us = us0 + u0, base = base0 + 4u * u0, zl = zl0 + ZU * u0;
    Word<T> w;
    const uint4 a = lds128(cp), b = lds128(cp + 16);
    uint4 lk = lds128(cp + 32);
    w.add(base, a.x);
    w.add(base, a.y);
    w.add(base, a.z);
    w.add(base, a.w);
    w.add(base, b.x);
    w.add(base, b.y);
    w.add(base, b.z);
    w.add(base, b.w);
    // the next link's record is loaded before this one's stores
#pragma unroll 1
    for (; n >= 2; n -= 2, cp += 2u * (uint32_t)sizeof(ClsLink)) {
      const uint4 l1 = lds128(cp + 32 + sizeof(ClsLink));
      w.emit(zl + lk.y, zl + lk.z, us - (lk.w & 0xFFFFu), lk.w >> 16);
      w.step(base, l1.x, (int32_t)l1.x >> 30);
      lk = lds128(cp + 32 + 2 * sizeof(ClsLink));
      w.emit(zl + l1.y, zl + l1.z, us - (l1.w & 0xFFFFu), l1.w >> 16);
      w.step(base, lk.x, (int32_t)lk.x >> 30);
    }
    w.emit(zl + lk.y, zl + lk.z, us - (lk.w & 0xFFFFu), lk.w >> 16);
    if (n) {
      lk = lds128(cp + 32 + sizeof(ClsLink));
      w.step(base, lk.x, (int32_t)lk.x >> 30);
      w.emit(zl + lk.y, zl + lk.z, us - (lk.w & 0xFFFFu), lk.w >> 16);
    }
  }
}

// ---- search fused into the tile (Sec. 2.2 boxcars over the series the tile has just summed)
//
// Per trial the warp forms the tile's inclusive prefix sums P[j] (uint32, relative to the tile's
// start: exact differences since every boxcar sum is < 2^31) in a shared-memory row, preceded by
// the `hist` prefix sums of the previous tile in this tile's frame (P[m] = -(sum of the previous
// tile's outputs after m), m = -hist .. -1). Then B_w[j] = P[j] - P[j - w] for every width, and
// per peak block the largest B_w + 1 (0: no valid sample) and its earliest sample are stored.
// Valid samples: inside the window, j >= w - 1 in the window (the boxcars of Sec. 2.2 reading),
// and, in the first tile of a segment (no previous tile), boxcars inside the tile only; the
// others are k_fused_edges' work.

// L2 evict-last access policy for the tail buffers: rewritten every tile and read back one tile
// later, while the streamed channel rows pass through L2 in between.
__device__ __forceinline__ uint64_t l2_keep_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint32_t ld_keep(const uint32_t* p, uint64_t pol) {
  uint32_t v;
  asm volatile("ld.global.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ void st_keep(uint32_t* p, uint32_t v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(pol) : "memory");
}

// Largest key over aligned groups of B lanes (B a power of two <= 32) and, for the group's
// first lane, the group's earliest lane holding it.
__device__ __forceinline__ uint32_t group_max(uint32_t key, int B, int lane, int* first) {
  uint32_t mx = key;
  if (B == 32) {
    mx = __reduce_max_sync(0xffffffffu, key);
  } else {
    for (int o = B >> 1; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  const uint32_t bal = __ballot_sync(0xffffffffu, key == mx);
  const uint32_t gm = B == 32 ? 0xffffffffu : ((1u << B) - 1u);
  *first = __ffs((bal >> (lane & ~(B - 1))) & gm) - 1;
  return mx;
}

// Head and tail buffers of CTA (trial tile bx, segment seg): [64][hist] each.
__device__ __forceinline__ uint32_t* fused_edge(const FusedArgs& f, int ntx, int bx, int seg) {
  return f.edge + ((size_t)seg * ntx + bx) * 2 * kFusedTrials * (size_t)f.hist;
}

// A warp's prefix-sum row is padded by four words after every 16, so that lanes reading 16-byte
// chunks 16 samples apart touch every bank once: place of entry j, and of the first entry of
// 4-entry chunk c.
__host__ __device__ constexpr int fused_row_words(int hp) { return (hp + 512) / 4 * 5; }
__device__ __forceinline__ int row_at(int j) { return j + 4 * (j >> 4); }
__device__ __forceinline__ int chunk_at(int c) { return 4 * c + 4 * (c >> 2); }

// d = p - the sixteen entries from M entries past chunk x on (of the lane's part e of a row).
template <int M>
__device__ __forceinline__ void row_diffs(const uint32_t (&p)[16], const uint32_t* e, int x,
                                          uint32_t (&d)[16]) {
  uint4 v[5];
#pragma unroll
  for (int i = 0; i < (M ? 5 : 4); ++i)
    v[i] = *reinterpret_cast<const uint4*>(e + chunk_at(x + i));
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint4 c = v[(i + M) / 4];
    const int r = (i + M) % 4;
    d[i] = p[i] - (r == 0 ? c.x : r == 1 ? c.y : r == 2 ? c.z : c.w);
  }
}

// Peak blocks of 16 or 32 samples: lane l takes samples 16 l .. 16 l + 15 of the tile, their
// prefix sums in registers, and per width reads the 16 earlier ones in four or five aligned
// 16-byte loads. Samples are visited in order, so the first of the largest sums wins; the two
// halves of a 32-sample block meet by one shuffle. About 80 instructions per width and trial,
// where one 4-byte load and a tie rule per sample and width took 330 at a quarter of the issue
// rate (113 us a tile of 64 trials x 512 samples x 9 widths, about 55 so).
template <bool INTERIOR>
__device__ __forceinline__ void fused_blocks(const FusedArgs& f, const uint32_t* E, int64_t rowk,
                                             int64_t j0, int64_t nout, bool first, int lane) {
  const int Bk = f.block, nw = f.nw, jl0 = 16 * lane;
  uint32_t p[16];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint4 v = *reinterpret_cast<const uint4*>(E + 20 * lane + 4 * i);
    p[4 * i] = v.x, p[4 * i + 1] = v.y, p[4 * i + 2] = v.z, p[4 * i + 3] = v.w;
  }
  const int64_t left = nout - j0 - jl0;  // window samples from this lane's first on
  const int hi = (int)(left < 0 ? 0 : (left > 16 ? 16 : left));
  const bool keep = hi > 0 && (Bk == 16 || (lane & 1) == 0);
  const int64_t blk = (j0 + jl0) / Bk;
#pragma unroll 1
  for (int k = 0; k < nw; ++k) {
    const int w = f.wd[k], m = (-w) & 3, x = -((w + m) >> 2);
    const uint32_t* e = E + 20 * lane;
    uint32_t d[16];
    if (m == 0) row_diffs<0>(p, e, x, d);  // uniform
    else if (m == 1) row_diffs<1>(p, e, x, d);
    else if (m == 2) row_diffs<2>(p, e, x, d);
    else row_diffs<3>(p, e, x, d);
    if (!INTERIOR) {  // keys: 1 + the sum, 0 for a sample outside the window or the segment
      const int64_t back = w - 1 - (j0 + jl0);
      int lo = (int)(back < 0 ? 0 : (back > 16 ? 16 : back));
      if (first) lo = max(lo, w - 1 - jl0);
#pragma unroll
      for (int i = 0; i < 16; ++i) d[i] = i >= lo && i < hi ? d[i] + 1u : 0u;
    }
    // the largest and its first place: four quarters, then the quarters in order
    uint32_t best[4];
    int off[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      best[i] = d[4 * i];
      off[i] = 4 * i;
#pragma unroll
      for (int q = 1; q < 4; ++q)
        if (d[4 * i + q] > best[i]) best[i] = d[4 * i + q], off[i] = 4 * i + q;
    }
#pragma unroll
    for (int i = 1; i < 4; i += 2)
      if (best[i] > best[i - 1]) best[i - 1] = best[i], off[i - 1] = off[i];
    if (best[2] > best[0]) best[0] = best[2], off[0] = off[2];
    uint32_t key = best[0] + (INTERIOR ? 1u : 0u);
    int at = off[0];
    if (Bk == 32) {  // the odd lane holds the block's second half
      const uint32_t ok = __shfl_xor_sync(0xffffffffu, key, 1);
      const int oa = __shfl_xor_sync(0xffffffffu, at, 1);
      if (ok > key) key = ok, at = oa + 16;
    }
    if (keep) {
      const int64_t idx = (rowk + k) * f.nblk + blk;
      f.key[idx] = key;
      f.off[idx] = (uint8_t)(key ? at : 0);
    }
  }
}

template <int TT, int W, int kTPW, int KT>
__device__ __forceinline__ void fused_search(const TiledArgs& a, const FusedArgs& f,
                                             const uint32_t (&acc)[kTPW][KT],
                                             unsigned char* smem, int bx, int by, bool first,
                                             int trial0, int ntr, int64_t j0, int warp,
                                             int lane) {
  constexpr int KP = KT / 2;
  const int hist = f.hist, HP = f.hp, Bk = f.block, nw = f.nw;
  const int wmax = f.wd[nw - 1];
  const int ntx = (a.n_trials + kFusedTrials - 1) / kFusedTrials;
  const int seg = by / f.seg_tiles;
  uint32_t* head = fused_edge(f, ntx, bx, seg);
  uint32_t* tail = head + kFusedTrials * (size_t)hist;
  static_assert(TT == 512, "sixteen samples a lane");
  uint32_t* E = reinterpret_cast<uint32_t*>(smem + f.e_off) +
                (size_t)warp * fused_row_words(HP) + HP / 4 * 5;
  const int64_t nout = a.nout;
  const uint64_t pol = l2_keep_policy();
#pragma unroll
  for (int q = 0; q < kTPW; ++q) {  // unrolled: acc stays in registers
    const int t = warp + W * q;
    if (t >= ntr) break;  // uniform in the warp; later q only larger
    uint32_t* tl = tail + (size_t)t * hist;
    uint32_t hv[16];  // hist <= 512; independent loads, all in flight before the scan
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int i = lane + 32 * r;
      hv[r] = (!first && i < hist) ? ld_keep(tl + i, pol) : 0u;
    }
    // inclusive prefix sums of the tile; lane l holds outputs 2(l + 32k) and 2(l + 32k) + 1
    uint32_t carry = 0;
#pragma unroll
    for (int k = 0; k < KP; ++k) {
      const uint32_t ev = acc[q][2 * k], od = acc[q][2 * k + 1];
      uint32_t incl = ev + od;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      const uint32_t po = carry + incl;
      *reinterpret_cast<uint2*>(E + row_at(2 * (lane + 32 * k))) = make_uint2(po - od, po);
      carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    // the previous tile's prefix sums in this tile's frame (none before a segment's first tile:
    // no valid boxcar reads them there)
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int i = lane + 32 * r;
      if (i < hist) E[row_at(i - hist)] = hv[r];
    }
    __syncwarp();
    if (first && seg > 0) {
      uint32_t* hd = head + (size_t)t * hist;
      for (int i = lane; i < hist; i += 32) hd[i] = E[row_at(i)];
    }
    // this tile's last prefix sums in the next tile's frame (P[TT + m] - P[TT - 1])
    for (int i = lane; i < hist; i += 32)
      st_keep(tl + i, E[row_at(TT - hist + i)] - carry, pol);
    const int64_t rowk = (int64_t)(trial0 + t) * nw;
    const bool interior = j0 >= wmax - 1 && !first && j0 + TT <= nout;
    if (Bk >= 16) {
      if (interior) fused_blocks<true>(f, E, rowk, j0, nout, first, lane);
      else fused_blocks<false>(f, E, rowk, j0, nout, first, lane);
      __syncwarp();  // the row is rewritten for the warp's next trial
      continue;
    }
    // smaller blocks: a lane takes a whole one and visits its samples from (lane mod Bk) on,
    // keeping per width the largest key and, on ties, the earliest sample
#pragma unroll 1
    for (int b = lane; b < TT / Bk; b += 32) {
      const int64_t jb = j0 + (int64_t)b * Bk;  // the block's first window sample
#pragma unroll 1
      for (int k = 0; k < nw; ++k) {
        const int w = f.wd[k];
        uint32_t best = 0;
        int boff = 32;
        for (int i = 0; i < Bk; ++i) {
          const int o = (i + lane) & (Bk - 1), jl = b * Bk + o;
          const int64_t jg = j0 + jl;
          const bool valid =
              interior || (jg < nout && jg >= w - 1 && (!first || jl >= w - 1));
          const uint32_t key = valid ? E[row_at(jl)] + 1u - E[row_at(jl - w)] : 0u;
          const bool take = key > best || (key == best && o < boff);
          best = take ? key : best;
          boff = take ? o : boff;
        }
        if (jb < nout) {
          const int64_t idx = (rowk + k) * f.nblk + jb / Bk;
          f.key[idx] = best;
          f.off[idx] = (uint8_t)(best ? boff : 0);
        }
      }
    }
    __syncwarp();  // the row is rewritten for the warp's next trial
  }
  // the rows overlay the staging buffers that the next tile's tensor copies fill
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Boxcars of a segment's first tile that start in the previous segment: per (boundary, trial),
// width w, samples j < w - 1 of the tile, B = head[j] - tail[hist + j - w], merged into the
// block's record (these samples precede every sample the fused pass saw in the block, so they
// win ties). CTA (4 x trial tile + quarter, boundary) takes 16 trials of the trial tile, one per
// warp; a warp first copies its trial's head and tail into shared memory (independent loads, all
// in flight), then works from there.
constexpr int kEdgeTrials = 16;

__global__ void __launch_bounds__(512) k_fused_edges(const __grid_constant__ TiledArgs a,
                                                     const __grid_constant__ FusedArgs f) {
  extern __shared__ __align__(16) uint32_t edge_rows[];  // [16 warps][2][hist]
  const int bx = blockIdx.x / 4, quarter = blockIdx.x % 4, seg = blockIdx.y + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t J = (int64_t)seg * f.seg_tiles * 512;
  if (J >= a.nout) return;
  const int ntx = gridDim.x / 4;
  const int hist = f.hist, Bk = f.block;
  const int t = quarter * kEdgeTrials + warp;  // trial within the trial tile
  const int trial = bx * kFusedTrials + t;
  if (trial >= a.n_trials) return;  // warp-uniform; no barrier follows
  const uint32_t* hd = fused_edge(f, ntx, bx, seg) + (size_t)t * hist;
  const uint32_t* tl =
      fused_edge(f, ntx, bx, seg - 1) + kFusedTrials * (size_t)hist + (size_t)t * hist;
  uint32_t* H = edge_rows + (size_t)warp * 2 * hist;
  uint32_t* T = H + hist;
#pragma unroll 4
  for (int i = lane; i < hist; i += 32) {
    H[i] = __ldcg(hd + i);
    T[i] = __ldcg(tl + i);
  }
  __syncwarp();
  for (int k = 0; k < f.nw; ++k) {
    const int w = f.wd[k];
    for (int jb = 0; jb < w - 1; jb += 32) {
      const int jl = jb + lane;
      const int64_t jg = J + jl;
      const bool valid = jl < w - 1 && jg < a.nout;
      const uint32_t key = valid ? H[jl] + 1u - T[hist + jl - w] : 0u;
      int fo;
      const uint32_t mx = group_max(key, Bk, lane, &fo);
      if ((lane & (Bk - 1)) == 0 && jg < a.nout && mx != 0) {
        const int64_t idx = ((int64_t)trial * f.nw + k) * f.nblk + jg / Bk;
        if (mx >= f.key[idx]) {
          f.key[idx] = mx;
          f.off[idx] = (uint8_t)fo;
        }
      }
    }
  }
}

// A tile's outputs: the series (if `store`) and the exact moments. Lane l of warp v holds outputs
// 2(l + 32k) and 2(l + 32k) + 1 of trials v, v + W, ... of the tile.
template <int W, int kTPW, int KT>
__device__ __forceinline__ void store_tile(const uint32_t (&acc)[kTPW][KT], int32_t* y,
                                           int64_t y_stride, Moments* mom, int64_t nout,
                                           int trial0, int ntr, int64_t j0, int warp, int lane,
                                           bool store) {
  constexpr int KP = KT / 2;
#pragma unroll
  for (int q = 0; q < kTPW; ++q) {
    const int t = warp + W * q;
    if (t < ntr) {
      int32_t* yr = y + (int64_t)(trial0 + t) * y_stride;
      unsigned long long s1 = 0, lo = 0, hi = 0;
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        const int64_t j = j0 + 2 * (lane + 32 * k);
        if (!store) {
        } else if (j + 1 < nout) {
          *reinterpret_cast<int2*>(yr + j) = make_int2((int32_t)acc[q][2 * k],
                                                       (int32_t)acc[q][2 * k + 1]);
        } else if (j < nout) {
          yr[j] = (int32_t)acc[q][2 * k];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (j + h < nout) {
            const uint32_t v = acc[q][2 * k + h];
            s1 += v;
            const unsigned long long sq = (unsigned long long)v * v;
            lo += sq;
            hi += (lo < sq) ? 1ull : 0ull;
          }
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, off);
        const unsigned long long olo = __shfl_xor_sync(0xffffffffu, lo, off);
        const unsigned long long ohi = __shfl_xor_sync(0xffffffffu, hi, off);
        const unsigned long long nlo = lo + olo;
        hi = hi + ohi + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
      }
      if (lane == 0) {
        Moments* m = mom + trial0 + t;
        atomicAdd(&m->s1, s1);
        const unsigned long long old = atomicAdd(&m->s2lo, lo);
        atomicAdd(&m->s2hi, hi + ((old + lo < old) ? 1ull : 0ull));
      }
    }
  }
}

// Words 32k + lane of N trials' sequences in both groups (or, both = false, in the first) added
// to the packed sums of trials q0 ..; tc: shared address of the trials' word offsets, zs: of the
// stage's words at the lane.
template <int D, int KP, int N, int kTPW>
__device__ __forceinline__ void add_words(uint32_t zs, uint32_t tc, bool both, int q0,
                                          uint32_t (&pk)[kTPW][KP]) {
  uint32_t zp[N], zq[N];  // N trials' words in group 0 and 1
  if constexpr (N == 4) {
    const uint4 e = lds128(tc), f = lds128(tc + 4 * D);
    zp[0] = zs + e.x, zp[1] = zs + e.y, zp[2] = zs + e.z, zp[3] = zs + e.w;
    zq[0] = zs + f.x, zq[1] = zs + f.y, zq[2] = zs + f.z, zq[3] = zs + f.w;
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      zp[q] = zs + lds<0>(tc + 4 * q);
      zq[q] = zs + lds<4 * D>(tc + 4 * q);
    }
  }
  if (both) {
#pragma unroll
    for (int k = 0; k < KP; ++k)
#pragma unroll
      for (int q = 0; q < N; ++q)
        pk[q0 + q][k] += lds<0>(zp[q] + 128 * k) + lds<0>(zq[q] + 128 * k);
  } else {
#pragma unroll
    for (int k = 0; k < KP; ++k)
#pragma unroll
      for (int q = 0; q < N; ++q) pk[q0 + q][k] += lds<0>(zp[q] + 128 * k);
  }
}

template <typename T, int TT, int NS, int D, int NT, bool FUSED = false>
__device__ __forceinline__ bool tile_body(const TiledArgs& a, int bx, int by,
                                          unsigned char* smem, bool reuse,
                                          const FusedArgs* f = nullptr, bool first = false) {
  constexpr int KT = TT / 32;       // outputs per lane and trial
  constexpr int KP = TT / 64;       // pair words per lane and trial
  constexpr int W = NT / 32;        // warps
  constexpr int kTPW = D / W;       // trials per warp
  const SmemLayout SL = smem_layout(sizeof(T), a.row_slot, a.zcap, a.tab_pitch, NS);
  T* raw = reinterpret_cast<T*>(smem + SL.raw);
  uint32_t* Zbuf = reinterpret_cast<uint32_t*>(smem + SL.z);
  unsigned char* tab = smem + SL.tab;
  uint32_t sraw = smem_addr(raw), sz = smem_addr(Zbuf), stab = smem_addr(tab);
  asm volatile("" : "+r"(sraw), "+r"(sz), "+r"(stab));  // worked out once, not per use
  const uint32_t pos = (uint32_t)(a.m0 + (int64_t)by * TT);  // ring column of the tile (mod 2^32)
  unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem + SL.mbar);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int trial0 = bx * D;
  const int ntr = min(D, a.n_trials - trial0);
  const int64_t j0 = (int64_t)by * TT;
  const int ngroups = a.cpad / kG;
  const int nstages = (ngroups + kNG - 1) / kNG;
  const size_t stage_elems = (size_t)kRows * a.row_slot;

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      if (reuse) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(&mbar[s]))
                              : "memory");
      mbar_init(&mbar[s], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // stages whose copies have been issued: NS in the prologue, then one per iteration s >= 1
  // (the same count in every thread)
  int issued = min(NS, nstages);
  int32_t xmin_next = 0;  // first delay of the next stage to issue (issuing thread)
  if (tid == NT - 32) {
    for (int s = 0; s < NS && s < nstages; ++s)
      issue_stage<T>(a, s, nstages, raw + (size_t)s * stage_elems, tab + s * a.tab_pitch, &mbar[s],
                     stage_xmin(a, s, nstages, bx), j0, bx);
    xmin_next = stage_xmin(a, NS, nstages, bx);
  }
  bool ok0 = mbar_wait_bounded(&mbar[0], 0);
  if (ok0) build_stage<T>(stab, sraw, sz, pos, warp, lane);
  bool aborted = __syncthreads_or(!ok0);
  int s_abort = 0;  // first stage whose copies may still be in flight

  uint32_t acc[kTPW][KT];
#pragma unroll
  for (int q = 0; q < kTPW; ++q)
#pragma unroll
    for (int k = 0; k < KT; ++k) acc[q][k] = 0;
  uint32_t pk[kTPW][KP];  // packed sums of the stages since the last flush
#pragma unroll
  for (int q = 0; q < kTPW; ++q)
#pragma unroll
    for (int k = 0; k < KP; ++k) pk[q][k] = 0;
  int left = a.flush;  // stages until the packed sums go to the 32-bit outputs
  const uint32_t raw_step = (uint32_t)(stage_elems * sizeof(T)), tab_step = (uint32_t)a.tab_pitch;
  // of stage s: staging buffer; of stage s + 1: staging buffer, its rows and table, barrier parity
  int b0 = 0, b1 = 1;
  uint32_t tcur = stab, rnext = sraw + raw_step, tnext = stab + tab_step, par1 = 0;
  uint32_t zcur = sz, znext = sz + a.zcap * 4u;  // word buffers of stages s and s + 1
  const uint32_t zrow = (uint32_t)sizeof(StageTab) + 4u * kTPW * warp;
  const int lone = (ngroups & 1) ? nstages - 1 : nstages;  // the stage holding one group

  for (int s = 0; s < nstages && !aborted; ++s) {
    // (1) TMA for stage s + NS - 1 into the buffers stage s - 1 used (its words were built
    //     during stage s - 2 and its table last read by the accumulation of stage s - 1)
    if (s >= 1 && s + NS - 1 < nstages) {
      if (tid == NT - 32) {
        const int b2 = b0 == 0 ? NS - 1 : b0 - 1;
        issue_stage<T>(a, s + NS - 1, nstages, raw + (size_t)b2 * stage_elems,
                       tab + b2 * a.tab_pitch, &mbar[b2], xmin_next, j0, bx);
        xmin_next = stage_xmin(a, s + NS, nstages, bx);
      }
      issued = s + NS;
    }
    bool ok = true;
    if (s + 1 < nstages) ok = mbar_try_wait(&mbar[b1], par1) || mbar_wait_bounded(&mbar[b1], par1);
    // (2) pair words of stage s + 1, and
    // (3) accumulation of stage s: lane l of the warp reads, for each of its trials, pair word
    //     l + 32k of the trial's plane in both groups (outputs 2(l + 32k) and 2(l + 32k) + 1).
    // Every warp builds first: with every second warp accumulating first, so that the two phases'
    // pipes overlap, the launch above took 7.40 ms against 6.38.
    if (ok && s + 1 < nstages) build_stage<T>(tnext, rnext, znext, pos, warp, lane);
    {
      const uint32_t zs = zcur + 4u * lane, tc = tcur + zrow;
      constexpr int N = kTPW < 4 ? kTPW : 4;  // trials at a time: eight row addresses
#pragma unroll
      for (int q = 0; q < kTPW; q += N) add_words<D, KP, N>(zs, tc + 4u * q, s != lone, q, pk);
    }
    if (--left == 0 || s + 1 == nstages) {  // uniform
      left = a.flush;
#pragma unroll
      for (int k = 0; k < KP; ++k)
#pragma unroll
        for (int q = 0; q < kTPW; ++q) {
          pair_add(pk[q][k], acc[q][2 * k], acc[q][2 * k + 1]);
          pk[q][k] = 0;
        }
    }
    b0 = b1;
    tcur = tnext;
    if (++b1 == NS) {
      b1 = 0;
      par1 ^= 1u;
      rnext = sraw;
      tnext = stab;
    } else {
      rnext += raw_step;
      tnext += tab_step;
    }
    const uint32_t zt = zcur;
    zcur = znext;
    znext = zt;
    if (__syncthreads_or(!ok)) {
      aborted = true;
      s_abort = s + 1;
    }
  }

  if (aborted) {
    if (tid == 0) {
      atomicOr(a.err, 1);
      // let every copy still in flight land before the CTA's shared memory goes away
      for (int s = s_abort; s < issued; ++s)
        mbar_wait_bounded(&mbar[s % NS], (uint32_t)((s / NS) & 1));
    }
    return false;
  }

  store_tile<W, kTPW, KT>(acc, a.y, a.y_stride, a.mom, a.nout, trial0, ntr, j0, warp, lane,
                          !FUSED || f->keep_series);
  if constexpr (FUSED)
    fused_search<TT, W, kTPW, KT>(a, *f, acc, smem, bx, by, first, trial0, ntr, j0, warp, lane);
  return true;
}

// One launch per range: CTA (x, y) runs trial tile x, time tile y.
template <typename T, int TT, int NS, int D, int NT>
__global__ void __launch_bounds__(NT, tile_ctas(D, TT, NT))
    k_dedisp_tiled(const __grid_constant__ TiledArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];  // tensor copies land 128-aligned
  tile_body<T, TT, NS, D, NT>(a, blockIdx.x, blockIdx.y, smem, false);
}

// Persistent form: one CTA per SM takes tiles from a device work list that spans many ranges of
// many plans (beams), until the list is exhausted. Segment k of the list holds every tile of
// descriptor seg_desc[k] (trial tiles fastest, as the per-range grid orders them), items
// seg_first[k] .. seg_first[k + 1] - 1. The shared-memory arrangement of each tile follows its
// own descriptor; the launch provides the largest any descriptor needs.
template <typename T, int TT, int NS, int D, int NT>
__global__ void __launch_bounds__(NT, 1) k_dedisp_persistent(const __grid_constant__ PersistArgs p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ long long item_s;
  const int64_t total = p.seg_first[p.nseg];
  bool reuse = false;
  for (;;) {
    if (threadIdx.x == 0) item_s = (long long)atomicAdd(p.counter, 1ull);
    __syncthreads();
    const int64_t item = item_s;
    if (item >= total) break;  // uniform
    int lo = 0, hi = p.nseg - 1;  // the segment holding the item
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (p.seg_first[mid] <= item) lo = mid; else hi = mid - 1;
    }
    const TiledArgs& a = p.descs[p.seg_desc[lo]];
    // the tensor map was written to global memory by a copy: acquire it for the tensor proxy
    // before the tile's first copy uses it
    if (threadIdx.x == NT - 32)
      asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&a.rows)
                   : "memory");
    const int64_t local = item - p.seg_first[lo];
    const int ntx = (a.n_trials + D - 1) / D;
    if (!tile_body<T, TT, NS, D, NT>(a, (int)(local % ntx), (int)(local / ntx), smem, reuse))
      break;  // a bounded wait ran out (uniform): the error bit is set
    reuse = true;
  }
}

// Fused form: CTA (x, y) runs trial tile x over time tiles y * seg_tiles .. (y + 1) * seg_tiles
// - 1 in order, each tile's search reading the previous tile's prefix sums (FusedArgs).
template <typename T, int NS>
__global__ void __launch_bounds__(512, 1)
    k_dedisp_fused(const __grid_constant__ TiledArgs a, const __grid_constant__ FusedArgs f) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int ntt = (int)((a.nout + 511) / 512);
  const int y0 = blockIdx.y * f.seg_tiles, y1 = min(ntt, y0 + f.seg_tiles);
  for (int y = y0; y < y1; ++y)
    if (!tile_body<T, 512, NS, 64, 512, true>(a, blockIdx.x, y, smem, y > y0, &f, y == y0))
      break;  // a bounded wait ran out (uniform): the error bit is set
}

// ---- staged direct kernel: ranges without shared delay classes (coarse channels, whose
// neighbouring trials differ by several samples within a group, or decimation above x16)
//
// CTA (x, y): 64 trials x 512 outputs, 16 warps, warp v the trials v, v + 16, ... of the tile as in
// the tiled kernel. Per stage of kSC channels the rows' windows (512 samples plus the tile's delay
// spread) come to shared memory by 16-byte asynchronous copies, are turned once into single-channel
// pair words x[v] | x[v + 1] << 16 in an even and an odd plane, and every trial adds the words of
// its own offset: one 32-bit shared-memory load per two channel-adds, conflict free, into packed
// 16-bit sums that go to the 32-bit outputs before they can overflow. Bound by the shared-memory
// pipe at 64 channel-adds per SM-clock; reading each trial's samples through the read-only cache
// with funnel shifts (k_dedisp_direct) was bound by instruction issue at about half of that (256
// channels of 1.6 MHz, 800 trials x 131072 at x1 and 400 at x2: 5.47 -> 3.00 ms, 1.1e13 channel-adds
// per second).
// Copies of stage s + 2, words of stage s + 1 and sums of stage s share one barrier per stage.
// Where the tiles are too few for the chip, blockIdx.z takes a share of the channels and the
// shares' sums are added to a zeroed series.
constexpr int kSC = 8;        // channels per stage
constexpr int kStTrials = 64, kStOut = 512;

struct StagedLayout {
  size_t z, off, total;
  int row;  // bytes of a staged row
};

// Where a staged row's copy starts in its ring row (bytes; at: ring column of the tile's first
// sample at the tile's smallest delay). Every copy takes a whole staged row (StagedLayout::row),
// as long as the widest trial tile of the range needs, from there: a tile of few trials that
// starts at the largest delay, with few outputs left, copies up to frame + 32 samples past the
// data, and the plan's ring rows are that long (staged_slack).
__host__ __device__ inline int64_t staged_copy_start(int64_t at, int es) {
  return at * es & ~(int64_t)15;
}

// frame: pair words per channel, a multiple of 8; the raw rows come first
__host__ __device__ inline StagedLayout staged_layout(int es, int frame) {
  StagedLayout L;
  L.row = (int)align16((size_t)(frame + 16) * es);
  L.z = (size_t)2 * kSC * L.row;
  L.off = L.z + (size_t)2 * kSC * frame * 4;
  L.total = L.off + (size_t)2 * kStTrials * kSC * 4;
  return L;
}

template <typename T>
__global__ void __launch_bounds__(512, 1) k_dedisp_staged(const StagedArgs a) {
  constexpr int es = (int)sizeof(T);
  constexpr int kTPW = kStTrials / 16, KT = kStOut / 32, KP = kStOut / 64;
  extern __shared__ __align__(1024) unsigned char smem[];
  const StagedLayout SL = staged_layout(es, a.frame);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int trial0 = blockIdx.x * kStTrials;
  const int ntr = min(kStTrials, a.n_trials - trial0);
  const int64_t j0 = (int64_t)blockIdx.y * kStOut;
  const int all = a.cpad / kSC;  // stages; this CTA's: sb .. sb + nstages - 1
  const int sb = (int)((int64_t)all * blockIdx.z / gridDim.z);
  const int nstages = (int)((int64_t)all * (blockIdx.z + 1) / gridDim.z) - sb;
  uint32_t sraw = smem_addr(smem);
  asm volatile("" : "+r"(sraw));
  const uint32_t sz = sraw + (uint32_t)SL.z, soff = sraw + (uint32_t)SL.off;
  const uint32_t zbytes = (uint32_t)(kSC * a.frame * 4);
  // the tile's smallest delays
  const int32_t* first = a.shifts + (int64_t)trial0 * a.cpad + sb * kSC;

  // copies: 64 threads per row
  const int crow = tid >> 6, cchunk = tid & 63;
  auto copy_rows = [&](int s, int32_t sfirst) {
    const int64_t byte = staged_copy_start(a.m0 + j0 + sfirst, es);
    const unsigned char* src = static_cast<const unsigned char*>(a.xd) +
                               (int64_t)((sb + s) * kSC + crow) * a.xd_stride * es + byte;
    const uint32_t dst = sraw + (uint32_t)((s & 1) * kSC + crow) * (uint32_t)SL.row;
    for (int c = 16 * cchunk; c < SL.row; c += 16 * 64)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + c), "l"(src + c)
                   : "memory");
  };
  // offsets: thread (trial, channel); byte offset of the trial's words in the stage's planes
  const int ot = tid >> 3, oc = tid & 7;
  auto offset = [&](int32_t st, int32_t sf) {
    const int ph = (int)(((a.m0 + j0 + sf) * es & 15) / es);
    const int o = (ot < ntr ? st - sf : 0) + ph;
    return (uint32_t)(oc * a.frame * 4 + (o & 1) * a.frame * 2 + (o >> 1) * 4);
  };
  const int32_t* myrow = a.shifts + (int64_t)(trial0 + min(ot, ntr - 1)) * a.cpad + sb * kSC + oc;
  auto build = [&](int s) {
    // each warp half a channel's units: one row word per unit and the next one
    const int ch = warp >> 1;
    const uint32_t row = sraw + (uint32_t)((s & 1) * kSC + ch) * (uint32_t)SL.row;
    const uint32_t ev = sz + (s & 1) * zbytes + (uint32_t)(ch * a.frame * 4);
    const uint32_t od = ev + (uint32_t)a.frame * 2;
    constexpr int U = 4 / es;  // samples per row word
    for (int u = (warp & 1) * 32 + lane; u * U < a.frame; u += 64) {
      const uint32_t w0 = lds<0>(row + 4 * u), w1 = lds<4>(row + 4 * u);
      if constexpr (es == 1) {
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(ev + 8 * u),
                     "r"(__byte_perm(w0, 0, 0x4140)), "r"(__byte_perm(w0, 0, 0x4342))
                     : "memory");
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(od + 8 * u),
                     "r"(__byte_perm(w0, 0, 0x4241)),
                     "r"(__byte_perm(__funnelshift_r(w0, w1, 24), 0, 0x4140))
                     : "memory");
      } else {
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(ev + 4 * u), "r"(w0) : "memory");
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(od + 4 * u), "r"(__byte_perm(w0, w1, 0x5432))
                     : "memory");
      }
    }
  };
  auto put_offset = [&](int s, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(soff + (uint32_t)((s & 1) * 512 + tid) * 4u),
                 "r"(v)
                 : "memory");
  };

  // prologue: rows of stages 0 and 1, words and offsets of stage 0
  copy_rows(0, __ldg(first + crow));
  if (nstages > 1) copy_rows(1, __ldg(first + kSC + crow));
  put_offset(0, offset(__ldg(myrow), __ldg(first + oc)));
  int32_t nst = 0, nsf = 0, ncf = 0;  // delays for the next offsets and the next copy
  if (nstages > 1) nst = __ldg(myrow + kSC), nsf = __ldg(first + kSC + oc);
  if (nstages > 2) ncf = __ldg(first + 2 * kSC + crow);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  build(0);
  __syncthreads();

  uint32_t acc[kTPW][KT], pk[kTPW][KP];
#pragma unroll
  for (int q = 0; q < kTPW; ++q) {
#pragma unroll
    for (int k = 0; k < KT; ++k) acc[q][k] = 0;
#pragma unroll
    for (int k = 0; k < KP; ++k) pk[q][k] = 0;
  }
  int left = a.flush;
  for (int s = 0; s < nstages; ++s) {
    if (s + 2 < nstages) {
      copy_rows(s + 2, ncf);  // into the rows of stage s, whose words are built
      if (s + 3 < nstages) ncf = __ldg(first + (s + 3) * kSC + crow);
    }
    if (s + 1 < nstages) {
      put_offset(s + 1, offset(nst, nsf));
      if (s + 2 < nstages)
        nst = __ldg(myrow + (s + 2) * kSC), nsf = __ldg(first + (s + 2) * kSC + oc);
      build(s + 1);
    }
    const uint32_t zs = sz + (s & 1) * zbytes + 4u * lane;
#pragma unroll
    for (int q = 0; q < kTPW; ++q) {
      const uint32_t ob = soff + (uint32_t)((s & 1) * 512 + (warp + 16 * q) * kSC) * 4u;
      const uint4 oa = lds128(ob), oz = lds128(ob + 16);
      const uint32_t zp[kSC] = {zs + oa.x, zs + oa.y, zs + oa.z, zs + oa.w,
                                zs + oz.x, zs + oz.y, zs + oz.z, zs + oz.w};
      if (a.flush > 0) {
#pragma unroll
        for (int c = 0; c < kSC; c += 2)
#pragma unroll
          for (int k = 0; k < KP; ++k)
            pk[q][k] += lds<0>(zp[c] + 128 * k) + lds<0>(zp[c + 1] + 128 * k);
      } else {  // eight channels' sum does not fit a 16-bit lane
#pragma unroll 1
        for (int c = 0; c < kSC; ++c) {
          const uint32_t z = zs + lds<0>(ob + 4 * c);
#pragma unroll
          for (int k = 0; k < KP; ++k)
            pair_add(lds<0>(z + 128 * k), acc[q][2 * k], acc[q][2 * k + 1]);
        }
      }
    }
    if (a.flush > 0 && (--left == 0 || s + 1 == nstages)) {
      left = a.flush;
#pragma unroll
      for (int k = 0; k < KP; ++k)
#pragma unroll
        for (int q = 0; q < kTPW; ++q) {
          pair_add(pk[q][k], acc[q][2 * k], acc[q][2 * k + 1]);
          pk[q][k] = 0;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  if (gridDim.z > 1) {  // moments follow from the complete series
#pragma unroll
    for (int q = 0; q < kTPW; ++q) {
      const int t = warp + 16 * q;
      if (t >= ntr) continue;
      int32_t* yr = a.y + (int64_t)(trial0 + t) * a.y_stride;
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        const int64_t j = j0 + 2 * (lane + 32 * k);
        if (j < a.nout) atomicAdd(yr + j, (int32_t)acc[q][2 * k]);
        if (j + 1 < a.nout) atomicAdd(yr + j + 1, (int32_t)acc[q][2 * k + 1]);
      }
    }
    return;
  }
  store_tile<16, kTPW, KT>(acc, a.y, a.y_stride, a.mom, a.nout, trial0, ntr, j0, warp, lane, true);
}

template <typename T, int TT, int NS, int D, int NT>
cudaError_t launch_tiled_t(const TiledArgs& a, cudaStream_t st) {
  const SmemLayout SL = smem_layout(sizeof(T), a.row_slot, a.zcap, a.tab_pitch, NS);
  dim3 grid((unsigned)((a.n_trials + D - 1) / D), (unsigned)((a.nout + TT - 1) / TT));
  k_dedisp_tiled<T, TT, NS, D, NT><<<grid, NT, SL.total, st>>>(a);
  return cudaGetLastError();
}

// Ranges sharing an instance need different amounts of shared memory, so the instance is
// allowed the device's opt-in maximum once (a launch still only reserves what it asks for).
template <typename T, int TT, int NS, int D, int NT>
cudaError_t prepare_t(size_t smem) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  if (smem > (size_t)optin) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(k_dedisp_tiled<T, TT, NS, D, NT>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  // the whole unified L1 as shared memory, so that two CTAs of a two-CTA shape fit an SM
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_dedisp_tiled<T, TT, NS, D, NT>,
                             cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
  return e;
}

}  // namespace

namespace {

// Costs of a build task, for dealing tasks to warps: its set-up with the eight channels of its
// first class, each link's store, each channel step. In instructions they would be about 100, 16,
// 18 (uint8) and 80, 13, 14 (uint16); a task's set-up is a chain of dependent shared-memory reads
// that a warp waits for, and counting it more than twice measured best (1216 trials x 65536 outputs x
// 4096 channels, ms a run, uint8 / uint16: 6.37 / 4.01 with the instruction counts, 6.31 / 3.94
// with 130 and 110, 6.29 / 3.92 with 170 and 140, 6.28 / 3.91 with these).
struct BuildCost {
  int base, emit, step;
};
constexpr BuildCost kCostU8{230, 16, 18}, kCostU16{190, 13, 14};

// Deal a stage's build work to W warps: per group and block of 31 units, the chain of links,
// from and to classes that store units in the block, cut where the plan breaks the chain
// (link without a step) and where a warp has its share. The share is the smallest, found by
// bisection, with which W warps suffice. Returns it.
int deal_work(StageTab& st, const ClsLink* cls, int D, std::vector<BuildTask>& tasks, int W,
              const BuildCost& C) {
  const int first[kNG + 1] = {0, st.nlink[0], st.nlink[0] + st.nlink[1]};
  const uint32_t l0 = links_at(D), t0 = l0 + (uint32_t)(first[kNG] * sizeof(ClsLink));
  int nblk[kNG] = {0, 0};
  for (int gl = 0; gl < kNG; ++gl)
    for (int p = first[gl]; p < first[gl + 1]; ++p)
      nblk[gl] = std::max(nblk[gl], (int)(cls[p].ulo() + cls[p].un() + kBlock - 1) / kBlock);
  auto stores = [&](int p, int b) {
    return cls[p].un() && (int)cls[p].ulo() < (b + 1) * kBlock &&
           (int)(cls[p].ulo() + cls[p].un()) > b * kBlock;
  };
  // deal with a given share; returns the warps used
  auto deal = [&](int share, bool out) {
    int w = 0, load = 0, nt = 0;
    if (out) {
      tasks.clear();
      std::memset(st.wtask, 0, sizeof st.wtask);
    }
    for (int gl = 0; gl < kNG; ++gl)
      for (int b = 0; b < nblk[gl]; ++b) {
        int p = first[gl];
        while (p < first[gl + 1]) {
          if (!stores(p, b)) {
            ++p;
            continue;
          }
          if (load > 0 && load + C.base + C.emit > share) {
            ++w;
            load = 0;
          }
          // a run from p: extend while the links chain and fit the share
          load += C.base + C.emit;
          int last = p, cost = 0;
          for (int q = p + 1; q < first[gl + 1] && cls[q].step && q < p + kMaxRun; ++q) {
            cost += C.step + C.emit;
            if (load + cost > share) break;
            if (stores(q, b)) {
              load += cost;
              cost = 0;
              last = q;
            }
          }
          if (out) {
            if (st.wtask[w] == 0) st.wtask[w] = t0 + (uint32_t)(nt * sizeof(BuildTask));
            st.wtask[w] += 1u << 16;
            tasks.push_back({(uint32_t)(l0 + p * sizeof(ClsLink)) | (uint32_t)(last - p) << 16,
                             (uint32_t)(b * kBlock)});
          }
          ++nt;
          p = last + 1;
        }
      }
    return w + 1;
  };
  int lo = C.base + C.emit, hi = lo;
  while (deal(hi, false) > W) {
    lo = hi;
    hi *= 2;
  }
  while (hi - lo > 8) {
    const int mid = (lo + hi) / 2;
    if (deal(mid, false) > W) lo = mid; else hi = mid;
  }
  deal(hi, true);
  return hi;
}

// Tasks of a stage, and where they lie in its table for D trials.
int stage_tasks(const StageTab& st) {
  int n = 0;
  for (int w = 0; w < kMaxWarps; ++w) n += (int)(st.wtask[w] >> 16);
  return n;
}

const ClsLink* table_links(const uint8_t* tab, int D) {
  return reinterpret_cast<const ClsLink*>(tab + links_at(D));
}

const BuildTask* table_tasks(const uint8_t* tab, int D) {
  const StageTab& st = *reinterpret_cast<const StageTab*>(tab);
  return reinterpret_cast<const BuildTask*>(table_links(tab, D) + st.nlink[0] + st.nlink[1]);
}

// Self-test of the bounded wait above: one thread arms a fresh mbarrier that nothing ever
// completes and waits on it; when the bound runs out it records the error bit, as the tiled
// kernel does for a copy that never lands.
__global__ void k_wait_selftest(int32_t* err) {
  __shared__ unsigned long long bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait_bounded(&bar, 0)) atomicOr(err, 1);
  }
}

}  // namespace

cudaError_t launch_wait_selftest(int32_t* err, cudaStream_t st) {
  k_wait_selftest<<<1, 32, 0, st>>>(err);
  return cudaGetLastError();
}

// Host: the shared-memory work of one row of time tiles, instruction by instruction as
// k_dedisp_tiled issues it (one wavefront per warp-wide access: the kernel's loads and stores are
// free of bank conflicts; a 64-bit store of 32 lanes is two wavefronts). Per (trial tile, stage):
//   accumulation : every warp loads, for its kTPW trials and TT / 64 pair-word columns, one word
//                  per group present (trials past the range's end load too), plus the trials'
//                  zstart entries;
//   build        : per task its descriptor, the first class's eight row offsets and two row words
//                  per channel; per link its record, its step's two row words and the two plane
//                  stores;
//   copies       : the tensor copy of the 16 staged rows and the bulk copy of the stage table.
static void tiled_smem_work(TiledPlan& P, int ntiles, int nstages, int ngroups, bool u16) {
  const int W = P.threads / 32;
  const int KP = P.tt / 64, kTPW = P.trials / W;
  const int sts_per_class = u16 ? 2 : 4;
  int64_t lsu = 0, bytes = 0;
  for (int ti = 0; ti < ntiles; ++ti)
    for (int s = 0; s < nstages; ++s) {
      const uint8_t* tp = P.tabs.data() + ((size_t)ti * nstages + s) * P.tab_pitch;
      const StageTab& st = *reinterpret_cast<const StageTab*>(tp);
      const int ng = std::min(kNG, ngroups - s * kNG);
      lsu += (int64_t)W * kTPW * KP * ng;             // accumulation words
      lsu += (int64_t)W * ng * ((kTPW + 3) / 4);      // zstart entries (four a load)
      lsu += 2 * W;                                   // wtask, xmin
      for (int t = 0; t < stage_tasks(st); ++t) {
        const int n = (int)(table_tasks(tp, P.trials)[t].link >> 16);  // links after the first
        lsu += 3 + 2 * kG;                            // descriptor, row offsets, row words
        lsu += (int64_t)(n + 1) * (1 + sts_per_class) + 2 * n;
      }
      bytes += (int64_t)kRows * P.row_slot * (u16 ? 2 : 1) + P.tab_pitch;
    }
  P.lsu_wavefronts = lsu;
  P.copy_bytes = bytes;
}

// Host: delay classes of every (trial tile, stage) of one range, as the kernel reads them.
// Classes of a group are sorted by their relative delays' sum, which makes neighbours differ by
// few channel steps (on the 4096- and 8192-channel plans within 2% of a nearest-neighbour chain);
// where two or three steps separate neighbours, links that store nothing go between them, and
// where more do, the chain breaks. A class's zlen = un x unit
// pair words start at a multiple of 4 within the stage, groups one after another, the even plane
// in the first zlen / 2 words and the odd plane after it. A trial whose sequence starts o words
// into its class reads plane (o mod 2) from word o / 2 on. Fails (ok = false) where the kernel's
// limits do not hold: a 16-bit lane holds the sum of two groups' eight channels of values up to
// 255 x decimation, so decimation must stay at or below 16; delays must be monotone in the trial
// within a channel; classes, tasks and the staged rows must fit their fixed-size tables and
// shared memory.
namespace {

// A stage's table with room for every link, and what the plan needs to know of it.
struct StagePlan {
  StageTab st;
  uint32_t zstart[kNG][kMaxTileTrials];
  ClsLink cls[kNG * kMaxLinks];
  std::vector<BuildTask> tasks;
  int words, links;  // pair words and links used
  int share;         // the largest warp's build work (BuildCost units)
};

bool plan_stage(const int32_t* tab, int t0, int n, int cpad, int s, bool u16, int tt, int D,
                int W, int row_slot, StagePlan& F) {
  const int U = u16 ? Word<uint16_t>::kUnit : Word<uint8_t>::kUnit;
  const int ngroups = cpad / kG;
  const uint32_t es = u16 ? 2 : 1;
  std::memset(&F.st, 0, sizeof F.st);
  std::memset(F.zstart, 0, sizeof F.zstart);
  std::memset(F.cls, 0, sizeof F.cls);
  StageTab& st = F.st;
  int32_t xmin = INT32_MAX;
  for (int c = s * kRows; c < std::min(cpad, (s + 1) * kRows); ++c)
    xmin = std::min(xmin, tab[(int64_t)t0 * cpad + c]);
  st.xmin = xmin;
  int words = 0, nl = 0;  // words and links of the groups before
  for (int gl = 0; gl < kNG && s * kNG + gl < ngroups; ++gl) {
    const int g = s * kNG + gl;
    int b[kMaxTileTrials], cls_of[kMaxTileTrials];
    int32_t ckey[kMaxCls][kG];
    int cmin[kMaxCls], cmax[kMaxCls], csum[kMaxCls];
    int ncls = 0, prev = 0, f0 = INT32_MAX;
    const int nl0 = nl;
    for (int i = 0; i < n; ++i) {
      const int32_t* sv = tab + (int64_t)(t0 + i) * cpad + kG * g;
      b[i] = *std::min_element(sv, sv + kG);
      f0 = std::min(f0, b[i]);
      int32_t key[kG];
      int sum = 0;
      for (int q = 0; q < kG; ++q) {
        const int64_t r = (int64_t)sv[q] - b[i];
        if (r > 32767) return false;
        key[q] = (int32_t)r;
        sum += (int)r;
      }
      int p = 0;
      while (p < ncls && !(csum[p] == sum && std::equal(key, key + kG, ckey[p]))) ++p;
      if (p == ncls) {
        if (ncls == (D > 64 ? kMaxCls : kMaxCls64)) return false;
        std::copy(key, key + kG, ckey[ncls]);
        cmin[ncls] = cmax[ncls] = b[i];
        csum[ncls] = sum;
        ++ncls;
      } else {
        cmin[p] = std::min(cmin[p], b[i]);
        cmax[p] = std::max(cmax[p], b[i]);
      }
      cls_of[i] = p;
    }
    int order[kMaxCls], zoff[kMaxCls], zlens[kMaxCls], ulos[kMaxCls];
    for (int p = 0; p < ncls; ++p) order[p] = p;
    std::stable_sort(order, order + ncls, [&](int x, int y) { return csum[x] < csum[y]; });
    for (int k = 0; k < ncls; ++k) {
      const int p = order[k];
      const int ulo = (cmin[p] - f0) / U;
      if (ulo > 32767 || cmax[p] - f0 + tt > 65535) return false;
      int un = (cmax[p] - f0 + tt + U - 1) / U - ulo;
      if (u16) un += un & 1;  // 16-byte aligned classes
      zoff[p] = words;
      zlens[p] = un * U;
      ulos[p] = ulo;
      int32_t key[kG];  // walks from the preceding class to this one
      std::copy(ckey[k > 0 ? prev : p], ckey[k > 0 ? prev : p] + kG, key);
      auto at_row = [&](int q, int r) {
        return es * (uint32_t)((gl * kG + q) * row_slot + f0 + r - xmin);
      };
      int dist = 0;
      for (int q = 0; q < kG; ++q) dist += std::abs(ckey[p][q] - key[q]);
      if (k == 0 || dist > kMaxSteps || nl - nl0 + dist + ncls - k - 1 > kMaxLinks) {
        std::copy(ckey[p], ckey[p] + kG, key);  // a chain starts here
        for (int q = 0; q < kG; ++q) F.cls[nl].off[q] = at_row(q, key[q]);
        ++nl;
      }
      for (int q = 0; q < kG; ++q)
        while (key[q] != ckey[p][q]) {
          const bool up = ckey[p][q] > key[q];
          F.cls[nl].step = (up ? kStepAdd : kStepSub) | at_row(q, up ? key[q] : key[q] - 1);
          key[q] += up ? 1 : -1;
          for (int c = 0; c < kG; ++c) F.cls[nl].off[c] = at_row(c, key[c]);
          ++nl;
        }
      ClsLink& e = F.cls[nl - 1];
      e.ev = 4 * (words - ulo * U / 2);
      e.od = e.ev + 2 * zlens[p];
      e.range = (uint32_t)ulo | (uint32_t)un << 16;
      prev = p;
      words += zlens[p];
      if (words > 32767) return false;
    }
    for (int i = 0; i < n; ++i) {
      const int p = cls_of[i], o = b[i] - f0 - ulos[p] * U;
      F.zstart[gl][trial_slot(i, W, D / W)] =
          4u * (uint32_t)(zoff[p] + (o % 2) * (zlens[p] / 2) + o / 2);
    }
    st.nlink[gl] = (uint8_t)(nl - nl0);
  }
  F.words = words;
  F.links = nl;
  F.share = deal_work(st, F.cls, D, F.tasks, W, u16 ? kCostU16 : kCostU8);
  return true;
}

bool shape_exists(int tt, int D, int nt) {
  return (tt == 512 && D == 64 && (nt == 512 || nt == 1024)) ||
         (tt == 256 && (D == 128 || D == 64 || D == 32) && nt == 512);
}

}  // namespace

double tiled_cost(const int32_t* tab, int ntr, int cpad, int decimation, int tt, int D, int nt,
                  int64_t nout, int sms) {
  if (decimation < 1 || kRows * 255 * decimation > 65535 || cpad % kG || !shape_exists(tt, D, nt))
    return -1.0;
  const int nstages = (cpad / kG + kNG - 1) / kNG, ntiles = (ntr + D - 1) / D;
  const int W = nt / 32;
  StagePlan F;
  double sum = 0;
  int count = 0;
  for (int a = 0; a < std::min(ntiles, 4); ++a)
    for (int b = 0; b < std::min(nstages, 16); ++b) {
      const int ti = (int)((int64_t)a * ntiles / std::min(ntiles, 4));
      const int s = (int)((int64_t)b * nstages / std::min(nstages, 16));
      if (!plan_stage(tab, ti * D, std::min(D, ntr - ti * D), cpad, s, decimation > 1, tt, D, W, 0,
                      F))
        return -1.0;
      sum += F.share;
      ++count;
    }
  // the rest of a stage, per warp: kTPW x KP words (two loads and an add each) and about 100
  // instructions of waits, addresses and barrier
  const double stage = sum / count + (D / W) * (tt / 64) * 3 + 100;
  const int64_t ctas = ntiles * ((nout + tt - 1) / tt), slots = (int64_t)sms * tile_ctas(D, tt, nt);
  return stage * nstages * (double)((ctas + slots - 1) / slots) * tile_ctas(D, tt, nt);
}

TiledPlan tiled_plan(const int32_t* tab, int ntr, int cpad, int decimation, int tt, int D,
                     int nt) {
  TiledPlan P;
  P.ok = false;
  const bool u16 = decimation > 1;
  if (decimation < 1 || kRows * 255 * decimation > 65535 || cpad % kG) return P;
  if (!shape_exists(tt, D, nt)) return P;
  const int es = u16 ? 2 : 1, W = nt / 32;
  const int ngroups = cpad / kG, nstages = (ngroups + kNG - 1) / kNG;
  const int ntiles = (ntr + D - 1) / D;
  // staged rows: a stage's common copy window runs from the smallest first-trial delay to the
  // largest last-trial delay of its channels
  int64_t spread = 0, span = 0;
  for (int ti = 0; ti < ntiles; ++ti) {
    const int t0 = ti * D, n = std::min(D, ntr - t0);
    const int32_t* a = tab + (int64_t)t0 * cpad;
    const int32_t* z = tab + (int64_t)(t0 + n - 1) * cpad;
    for (int i = 1; i < n; ++i) {
      bool down = false;
      for (int c = 0; c < cpad; ++c)
        down |= a[(int64_t)i * cpad + c] < a[(int64_t)(i - 1) * cpad + c];
      if (down) return P;
    }
    for (int c0 = 0; c0 < cpad; c0 += kRows) {
      int32_t xmin = INT32_MAX, xmax = 0;
      for (int c = c0; c < std::min(cpad, c0 + kRows); ++c) {
        xmin = std::min(xmin, a[c]);
        xmax = std::max(xmax, z[c]);
        spread = std::max<int64_t>(spread, z[c] - a[c]);
      }
      span = std::max<int64_t>(span, (int64_t)xmax - xmin);
    }
  }
  if (spread > 65536) return P;
  const int SEG = kSegBytes / es;
  P.tt = tt;
  P.trials = D;
  P.threads = nt;
  P.ctas = tile_ctas(D, tt, nt);
  P.flush = 65535 / (kRows * 255 * decimation);
  // staged row: the stage's window (span + tt samples) from up to SEG - 1 samples into its
  // first segment, and 32 samples the word-wise build may read past the last word it uses
  P.nseg = (int)std::min<int64_t>((span + tt + 32 + 2 * SEG - 2) / SEG, 256);
  if (P.nseg > 255) return P;
  P.row_slot = P.nseg * SEG;
  // a stage buffer's byte offsets fit 16 bits (ClsLink's fields count on it)
  if ((size_t)kRows * P.row_slot * es > 65535) return P;

  // the tables, each as long as its links: host threads take runs of trial tiles
  struct Part {
    std::vector<uint8_t> bytes;
    std::vector<uint32_t> len;
    int words = 0;
    bool ok = true, nomem = false;
  };
  const int want = std::min(ntiles, (int)std::min<int64_t>((int64_t)ntiles * nstages / 256 + 1, 8));
  const int hw = (int)std::thread::hardware_concurrency();
  const int nth = std::max(1, std::min(want, hw));
  std::vector<Part> parts(nth);
  auto run = [&](int k) {
    Part& q = parts[k];
    try {
      StagePlan F;
      const int a = (int)((int64_t)ntiles * k / nth), z = (int)((int64_t)ntiles * (k + 1) / nth);
      q.len.reserve((size_t)(z - a) * nstages);
      q.bytes.reserve((size_t)(z - a) * nstages * (links_at(D) + 24 * sizeof(ClsLink)));
      for (int ti = a; ti < z && q.ok; ++ti)
        for (int s = 0; s < nstages && q.ok; ++s) {
          q.ok = plan_stage(tab, ti * D, std::min(D, ntr - ti * D), cpad, s, u16, tt, D, W,
                            P.row_slot, F);
          if (!q.ok) break;
          const size_t zlen = 4 * (size_t)D, links = F.links * sizeof(ClsLink);
          const size_t tasks = F.tasks.size() * sizeof(BuildTask);
          const size_t at = q.bytes.size(), len = align16(links_at(D) + links + tasks);
          q.bytes.resize(at + len);
          uint8_t* to = q.bytes.data() + at;
          std::memcpy(to, &F.st, sizeof(StageTab));
          for (int gl = 0; gl < kNG; ++gl)
            std::memcpy(to + sizeof(StageTab) + gl * zlen, F.zstart[gl], zlen);
          std::memcpy(to + links_at(D), F.cls, links);
          std::memcpy(to + links_at(D) + links, F.tasks.data(), tasks);
          q.len.push_back((uint32_t)len);
          q.words = std::max(q.words, F.words);
        }
    } catch (const std::bad_alloc&) {
      q.nomem = true;
    }
  };
  {
    std::vector<std::thread> th;
    th.reserve(nth);
    int k = 1;
    try {
      for (; k < nth; ++k) th.emplace_back(run, k);
    } catch (const std::system_error&) {  // no more threads: this one does the rest
    }
    run(0);
    for (; k < nth; ++k) run(k);
    for (auto& t : th) t.join();
  }
  size_t most = 0;
  int zcap = 4;
  for (const Part& q : parts) {
    if (q.nomem) throw std::bad_alloc();
    if (!q.ok) return P;
    for (uint32_t l : q.len) most = std::max<size_t>(most, l);
    zcap = std::max(zcap, q.words);
  }
  P.zcap = (zcap + 3) / 4 * 4;
  P.tab_pitch = (int)most;
  P.tab_bytes = most * ntiles * nstages;
  P.tabs.resize(P.tab_bytes);
  uint8_t* to = P.tabs.data();
  for (const Part& q : parts) {
    const uint8_t* from = q.bytes.data();
    for (uint32_t l : q.len) {
      std::memcpy(to, from, l);
      from += l;
      to += most;
    }
  }
  // as many staging buffers as fit (4, else 3: a copy is then issued two stages ahead)
  const size_t limit = P.ctas == 2 ? kSmemLimit2 : kSmemLimit;
  for (int nst = kMaxNStage; nst >= 3 && !P.ok; --nst) {
    P.nstage = nst;
    P.smem = smem_layout(es, P.row_slot, P.zcap, P.tab_pitch, nst).total;
    P.ok = P.smem <= limit;
  }
  if (P.ok) tiled_smem_work(P, ntiles, nstages, ngroups, u16);
  return P;
}

// Instances: uint8/uint16 data x 4/3 staging buffers x the tile shapes (outputs, trials,
// threads): 512 x 64 with 512 or 1024 threads, 256 x 128, 256 x 64 and 256 x 32 with 512.
#define DD_TILED_SHAPES(X, T, U16)                                                  \
  X(T, U16, 512, 4, 64, 512) X(T, U16, 512, 3, 64, 512) X(T, U16, 512, 4, 64, 1024) \
  X(T, U16, 512, 3, 64, 1024) X(T, U16, 256, 4, 64, 512) X(T, U16, 256, 3, 64, 512) \
  X(T, U16, 256, 4, 128, 512) X(T, U16, 256, 3, 128, 512)                           \
  X(T, U16, 256, 4, 32, 512) X(T, U16, 256, 3, 32, 512)
#define DD_TILED_INSTANCES(X) DD_TILED_SHAPES(X, uint8_t, 0) DD_TILED_SHAPES(X, uint16_t, 1)
// The persistent form exists for the 64 x 512 and 128 x 256 tiles with 16 warps, the shapes a
// plan chooses between.
#define DD_PERSIST_INSTANCES(X)                                                   \
  X(uint8_t, 0, 256, 4, 128, 512) X(uint8_t, 0, 256, 3, 128, 512)                 \
  X(uint16_t, 1, 256, 4, 128, 512) X(uint16_t, 1, 256, 3, 128, 512)               \
  X(uint8_t, 0, 512, 4, 64, 512) X(uint8_t, 0, 512, 3, 64, 512)                   \
  X(uint16_t, 1, 512, 4, 64, 512) X(uint16_t, 1, 512, 3, 64, 512)

// Host: plan one range and verify the tables against the delay table they were built from,
// independently of how they were built, by running the build's address arithmetic. Returns the
// number of violations of:
//   - the stage's copy start is the smallest first-trial delay of its rows, and every read of
//     every trial stays inside the staged row;
//   - the tasks, run as the kernel runs them (a first link's row offsets, then the steps),
//     visit links at exactly their own row offsets, and store every unit of every class
//     exactly once; class word ranges are 16-byte aligned and do not overlap;
//   - every trial's tt / 2 pair words lie inside one plane of a class of its group, and the frame
//     word they stand for adds, in every channel of the group, the sample at the trial's delay;
//   - a task's loads, phase included, end inside the CTA's shared memory.
int64_t tiled_plan_check(const int32_t* tab, int ntr, int cpad, int decimation, int tt, int D,
                         int* ok) {
  const TiledPlan P = tiled_plan(tab, ntr, cpad, decimation, tt, D, kThreads);
  *ok = P.ok ? 1 : 0;
  if (!P.ok) return 0;
  const bool u16 = decimation > 1;
  const int U = u16 ? 2 : 4, es = u16 ? 2 : 1, SEG = kSegBytes / es;
  const int ngroups = cpad / kG, nstages = (ngroups + kNG - 1) / kNG;
  const int ntiles = (ntr + D - 1) / D;
  const SmemLayout L = smem_layout(es, P.row_slot, P.zcap, P.tab_pitch, P.nstage);
  int64_t bad = (P.tab_pitch % 16) != 0;
  bad += (int64_t)P.flush * kRows * 255 * decimation > 65535 || P.flush < 1;
  for (int ti = 0; ti < ntiles; ++ti) {
    const int t0 = ti * D, n = std::min(D, ntr - t0);
    for (int s = 0; s < nstages; ++s) {
      const uint8_t* tp = P.tabs.data() + ((size_t)ti * nstages + s) * P.tab_pitch;
      const StageTab& st = *reinterpret_cast<const StageTab*>(tp);
      const ClsLink* cls = table_links(tp, D);
      const BuildTask* task = table_tasks(tp, D);
      const uint32_t* zst = reinterpret_cast<const uint32_t*>(tp + sizeof(StageTab));
      const int ncls = st.nlink[0] + st.nlink[1];
      const size_t tasks0 = (const uint8_t*)task - tp;
      bad += tasks0 + stage_tasks(st) * sizeof(BuildTask) > (size_t)P.tab_pitch;
      int32_t xmin = INT32_MAX;
      for (int c = s * kRows; c < std::min(cpad, (s + 1) * kRows); ++c)
        xmin = std::min(xmin, tab[(int64_t)t0 * cpad + c]);
      bad += st.xmin != xmin;
      for (int t = t0; t < t0 + n; ++t)
        for (int c = s * kRows; c < std::min(cpad, (s + 1) * kRows); ++c)
          bad += (int64_t)tab[(int64_t)t * cpad + c] - xmin + tt + 32 + SEG - 1 > P.row_slot;
      std::vector<std::vector<int>> stored(ncls);  // units of each class, times stored
      std::vector<int> words(P.zcap, 0);           // classes holding each word
      for (int p = 0; p < ncls; ++p) {
        stored[p].assign(cls[p].un(), 0);
        const int z0 = cls[p].ev / 4 + (int)cls[p].ulo() * U / 2, zlen = (int)cls[p].un() * U;
        if (zlen == 0) continue;  // a step between classes
        bad += z0 % 4 != 0 || zlen % 4 != 0 || cls[p].od != cls[p].ev + 2 * zlen;
        if (z0 < 0 || z0 + zlen > P.zcap) {
          ++bad;
          continue;
        }
        for (int v = z0; v < z0 + zlen; ++v) bad += words[v]++ != 0;
      }
      for (int w = 0, t = 0; w < kWarps; ++w) {  // the warps' tasks follow one another
        bad += (st.wtask[w] >> 16) && (st.wtask[w] & 0xFFFFu) != tasks0 + t * sizeof(BuildTask);
        t += (int)(st.wtask[w] >> 16);
      }
      for (int w = kWarps; w < kMaxWarps; ++w) bad += st.wtask[w] != 0;
      for (int t = 0; t < stage_tasks(st); ++t) {
        const int p0 = (int)((task[t].link & 0xFFFFu) - links_at(D)) / (int)sizeof(ClsLink);
        const int np = (int)(task[t].link >> 16) + 1, u0 = (int)task[t].u0;
        bad += (task[t].link & 0xFFFFu) != links_at(D) + p0 * sizeof(ClsLink);
        const int gl = p0 >= st.nlink[0];
        if (p0 + np > (gl ? ncls : (int)st.nlink[0])) {
          ++bad;
          continue;
        }
        uint32_t off[kG];
        std::copy(cls[p0].off, cls[p0].off + kG, off);
        for (int p = p0; p < p0 + np; ++p) {
          if (p > p0) {
            const uint32_t sw = cls[p].step, at = sw & kStepOff;
            const bool up = (sw & ~kStepOff) == kStepAdd;
            bad += !up && (sw & ~kStepOff) != kStepSub;
            int hit = 0;
            for (int q = 0; q < kG && !hit; ++q)
              if (off[q] == (up ? at : at + es)) {
                off[q] = up ? at + es : at;
                ++hit;
              }
            bad += hit != 1;
          }
          bad += !std::equal(off, off + kG, cls[p].off);
          for (int l = 0; l < kBlock; ++l) {
            const int v = u0 + l - (int)cls[p].ulo();
            if (v >= 0 && v < (int)cls[p].un()) bad += stored[p][v]++ != 0;
          }
          // lane 31's second row word at the largest phase
          for (int q = 0; q < kG; ++q)
            bad += L.raw + (size_t)(P.nstage - 1) * kRows * P.row_slot * es +
                       4u * (uint32_t)(u0 + 31) + cls[p].off[q] + (SEG - 1) * es + 8 >
                   L.total;
        }
      }
      for (const auto& v : stored)
        for (int k : v) bad += k != 1;
      int p1 = 0;
      for (int gl = 0; gl < kNG && s * kNG + gl < ngroups; ++gl) {
        const int c0 = (s * kNG + gl) * kG, g0 = p1;
        p1 += st.nlink[gl];
        for (int i = 0; i < n; ++i) {
          const uint32_t zb = zst[gl * D + trial_slot(i, kWarps, D / kWarps)];
          bad += zb % 4 != 0;
          const int z = (int)zb / 4;
          int p = g0, v = -1;
          for (; p < p1; ++p) {
            const int zo = cls[p].ev / 4 + (int)cls[p].ulo() * U / 2;
            const int half = (int)cls[p].un() * U / 2;
            if (zo <= z && z + tt / 2 <= zo + half) {
              v = (int)cls[p].ulo() * U + 2 * (z - zo);  // even plane
              break;
            }
            if (zo + half <= z && z + tt / 2 <= zo + 2 * half) {
              v = (int)cls[p].ulo() * U + 2 * (z - zo - half) + 1;  // odd plane
              break;
            }
          }
          if (p == p1) {
            ++bad;
            continue;
          }
          for (int q = 0; q < kG; ++q)
            bad += (int64_t)cls[p].off[q] / es + v !=
                   (int64_t)(gl * kG + q) * P.row_slot +
                       tab[(int64_t)(t0 + i) * cpad + c0 + q] - xmin;
        }
      }
    }
  }
  return bad;
}

cudaError_t launch_tiled_persistent(const PersistArgs& p, int is_u16, int tt, int nstage, int D,
                                    int nt, size_t smem, int ctas, cudaStream_t st) {
  if (p.nseg <= 0 || ctas <= 0) return cudaSuccess;
  if (smem > kSmemLimit) return cudaErrorInvalidValue;
  // The limit set is the largest any plan may need, not this launch's: it is state of the function
  // on the device, and another host thread's batch must not find it lowered.
#define DD_PERSIST(T, U16, TT, NS, DT, NTH)                                     \
  if (is_u16 == U16 && tt == TT && nstage == NS && D == DT && nt == NTH) {       \
    cudaError_t e = cudaFuncSetAttribute(k_dedisp_persistent<T, TT, NS, DT, NTH>, \
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                         (int)kSmemLimit);                      \
    if (e != cudaSuccess) return e;                                             \
    k_dedisp_persistent<T, TT, NS, DT, NTH><<<ctas, NTH, smem, st>>>(p);        \
    return cudaGetLastError();                                                  \
  }
  DD_PERSIST_INSTANCES(DD_PERSIST)
#undef DD_PERSIST
  return cudaErrorInvalidValue;
}

cudaError_t prepare_tiled(int is_u16, int tt, int nstage, int D, int nt, size_t smem) {
#define DD_PREPARE(T, U16, TT, NS, DT, NTH)                                     \
  if (is_u16 == U16 && tt == TT && nstage == NS && D == DT && nt == NTH) \
    return prepare_t<T, TT, NS, DT, NTH>(smem);
  DD_TILED_INSTANCES(DD_PREPARE)
#undef DD_PREPARE
  return cudaErrorInvalidValue;
}

namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

}  // namespace

cudaError_t make_ring_map(CUtensorMap* map, const void* ring, int is_u16, int64_t stride,
                          int32_t cpad, int nseg) {
  const int es = is_u16 ? 2 : 1;
  const int64_t seg = kSegBytes / es;
  if ((stride * es) % kSegBytes || nseg < 1 || nseg > 255 || cpad < 1 ||
      (reinterpret_cast<uintptr_t>(ring) & 15))
    return cudaErrorInvalidValue;
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)seg, (cuuint64_t)(stride / seg), (cuuint64_t)cpad};
  const cuuint64_t strides[2] = {(cuuint64_t)kSegBytes, (cuuint64_t)(stride * es)};
  const cuuint32_t box[3] = {(cuuint32_t)seg, (cuuint32_t)nseg, (cuuint32_t)kRows};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r =
      fn(map, is_u16 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
         const_cast<void*>(ring), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

bool fused_smem(int is_u16, int row_slot, int zcap, int pitch, int nstage, int hp,
                int32_t* e_off, size_t* smem) {
  const SmemLayout L = smem_layout(is_u16 ? 2 : 1, row_slot, zcap, pitch, nstage);
  const size_t rows = (size_t)kWarps * fused_row_words(hp) * sizeof(uint32_t);
  size_t total = L.total, off = L.raw;
  if (L.tab - L.raw < rows) {  // the staging area is too small: the rows go after it
    off = L.total;
    total = L.total + rows;
  }
  if (total > kSmemLimit) return false;
  *e_off = (int32_t)off;
  *smem = total;
  return true;
}

namespace {

template <typename T, int NS>
cudaError_t prepare_fused_t() {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_dedisp_fused<T, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin);
  return e;
}

}  // namespace

cudaError_t prepare_fused(int is_u16, int nstage, size_t smem) {
  if (smem > kSmemLimit) return cudaErrorInvalidValue;
  const cudaError_t e = cudaFuncSetAttribute(k_fused_edges,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)((512 / 32) * 2 * 512 * sizeof(uint32_t)));
  if (e != cudaSuccess) return e;
  if (!is_u16 && nstage == 4) return prepare_fused_t<uint8_t, 4>();
  if (!is_u16 && nstage == 3) return prepare_fused_t<uint8_t, 3>();
  if (is_u16 && nstage == 4) return prepare_fused_t<uint16_t, 4>();
  if (is_u16 && nstage == 3) return prepare_fused_t<uint16_t, 3>();
  return cudaErrorInvalidValue;
}

int fused_segments(int ntx, int ntt, int sms, int smax) {
  int best = 1;
  int64_t best_cost = -1;
  for (int s = 1; s <= std::min(ntt, std::max(1, smax)); ++s) {
    const int seg = (ntt + s - 1) / s;
    const int used = (ntt + seg - 1) / seg;  // segments that get tiles
    const int64_t waves = ((int64_t)ntx * used + sms - 1) / sms;
    const int64_t cost = waves * seg;
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = used;
    }
  }
  return best;
}

cudaError_t launch_fused(const TiledArgs& a, const FusedArgs& f, int is_u16, size_t smem,
                         cudaStream_t st) {
  if (a.nout <= 0 || a.n_trials <= 0) return cudaSuccess;
  const int ntx = (a.n_trials + kFusedTrials - 1) / kFusedTrials;
  const int ntt = (int)((a.nout + 511) / 512);
  if (f.nsegs < 1 || (int64_t)f.nsegs * f.seg_tiles < ntt ||
      (int64_t)(f.nsegs - 1) * f.seg_tiles >= ntt || f.hist < 1 || f.hist > 512 ||
      f.hp < f.hist || f.nw < 1 || f.wd[f.nw - 1] != f.hist)
    return cudaErrorInvalidValue;
  const dim3 grid((unsigned)ntx, (unsigned)f.nsegs);
  if (!is_u16 && a.nstage == 4) k_dedisp_fused<uint8_t, 4><<<grid, 512, smem, st>>>(a, f);
  else if (!is_u16 && a.nstage == 3) k_dedisp_fused<uint8_t, 3><<<grid, 512, smem, st>>>(a, f);
  else if (is_u16 && a.nstage == 4) k_dedisp_fused<uint16_t, 4><<<grid, 512, smem, st>>>(a, f);
  else if (is_u16 && a.nstage == 3) k_dedisp_fused<uint16_t, 3><<<grid, 512, smem, st>>>(a, f);
  else return cudaErrorInvalidValue;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || f.nsegs < 2) return e;
  const size_t esmem = (size_t)(512 / 32) * 2 * f.hist * sizeof(uint32_t);
  k_fused_edges<<<dim3((unsigned)ntx * 4, (unsigned)(f.nsegs - 1)), 512, esmem, st>>>(a, f);
  return cudaGetLastError();
}

int staged_plan(const int32_t* tab, int ntr, int cpad, int decimation, int* frame) {
  if (cpad % kSC) return 0;
  int64_t spread = 0;
  for (int t0 = 0; t0 < ntr; t0 += kStTrials) {
    const int n = std::min(kStTrials, ntr - t0);
    for (int i = 0; i < n; ++i)
      for (int c = 0; c < cpad; ++c) {
        const int64_t o = (int64_t)tab[(int64_t)(t0 + i) * cpad + c] - tab[(int64_t)t0 * cpad + c];
        if (o < 0) return 0;
        spread = std::max(spread, o);
      }
  }
  // a row may start up to 15 samples before the tile's first one
  const int64_t f = (spread + 15 + kStOut + 7) / 8 * 8;
  if (f > 4096) return 0;
  const int es = decimation > 1 ? 2 : 1;
  if (staged_layout(es, (int)f).total > kSmemLimit) return 0;
  *frame = (int)f;
  return 1;
}

int64_t staged_slack(int frame) { return frame + 32; }

// Host: walk the staged kernel's launch over a window of nout outputs from ring column m0 on, in
// ring rows of row_len elements, with the kernel's own copy arithmetic. Returns the number of
// violations of:
//   - every 16-byte copy of every row lies inside the ring row;
//   - the copied bytes hold every sample the tile's trials add;
//   - every trial's pair words lie inside their plane of the frame.
int64_t staged_plan_check(const int32_t* tab, int ntr, int cpad, int decimation, int frame,
                          int64_t m0, int64_t nout, int64_t row_len) {
  const int es = decimation > 1 ? 2 : 1;
  const StagedLayout L = staged_layout(es, frame);
  const int64_t ring_row = row_len * es;
  int64_t bad = ring_row % 16 != 0 || L.row % 16 != 0 || frame % 8 != 0;
  for (int t0 = 0; t0 < ntr; t0 += kStTrials)
    for (int64_t j0 = 0; j0 < nout; j0 += kStOut)
      for (int c = 0; c < cpad; ++c) {
        const int64_t byte = staged_copy_start(m0 + j0 + tab[(int64_t)t0 * cpad + c], es);
        const int64_t end = byte + L.row;
        bad += byte < 0 || byte % 16 != 0 || end > ring_row;
        const int64_t left = std::min<int64_t>(kStOut, nout - j0);
        for (int t = t0; t < std::min(ntr, t0 + kStTrials); ++t) {
          const int64_t first = m0 + j0 + tab[(int64_t)t * cpad + c];
          const int64_t o = first - byte / es;  // the trial's first word
          bad += first * es < byte || (first + left) * es > end;
          bad += o < 0 || o / 2 + kStOut / 2 > frame / 2;
        }
      }
  return bad;
}

cudaError_t prepare_staged(int is_u16) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  return is_u16 ? cudaFuncSetAttribute(k_dedisp_staged<uint16_t>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, optin)
                : cudaFuncSetAttribute(k_dedisp_staged<uint8_t>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
}

cudaError_t launch_staged(const StagedArgs& a, int is_u16, int sms, cudaStream_t st,
                          int* launches) {
  *launches = 0;
  if (a.nout <= 0 || a.n_trials <= 0) return cudaSuccess;
  dim3 grid((unsigned)((a.n_trials + kStTrials - 1) / kStTrials),
            (unsigned)((a.nout + kStOut - 1) / kStOut), 1);
  // shares of at least four stages while the chip has room for them
  const int64_t ctas = (int64_t)grid.x * grid.y;
  if (2 * ctas <= sms) grid.z = (unsigned)std::max<int64_t>(1, std::min<int64_t>(sms / ctas, a.cpad / kSC / 4));
  const size_t smem = staged_layout(is_u16 ? 2 : 1, a.frame).total;
  cudaError_t e = cudaSuccess;
  if (grid.z > 1)
    e = cudaMemset2DAsync(a.y, a.y_stride * sizeof(int32_t), 0, a.nout * sizeof(int32_t),
                          a.n_trials, st);
  if (e != cudaSuccess) return e;
  if (is_u16) k_dedisp_staged<uint16_t><<<grid, 512, smem, st>>>(a);
  else k_dedisp_staged<uint8_t><<<grid, 512, smem, st>>>(a);
  *launches = 1;
  e = cudaGetLastError();
  if (e == cudaSuccess && grid.z > 1) {
    e = launch_moments(a.y, a.n_trials, a.nout, a.y_stride, a.mom, st);
    *launches = 2;
  }
  return e;
}

cudaError_t launch_tiled(const TiledArgs& a, int is_u16, int tt, int D, int nt,
                         cudaStream_t st) {
  if (a.nout <= 0 || a.n_trials <= 0) return cudaSuccess;
#define DD_LAUNCH(T, U16, TT, NS, DT, NTH)                                        \
  if (is_u16 == U16 && tt == TT && a.nstage == NS && D == DT && nt == NTH) \
    return launch_tiled_t<T, TT, NS, DT, NTH>(a, st);
  DD_TILED_INSTANCES(DD_LAUNCH)
#undef DD_LAUNCH
  return cudaErrorInvalidValue;
}

}  // namespace ddk
