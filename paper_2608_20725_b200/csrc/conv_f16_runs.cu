// fp16-input / fp32-accumulate im2win convolution with the window tensor brought in as contiguous runs.  It needs no
// alignment of planes, strips or images and takes every stride: the layers whose plane pitch is no multiple of 16
// bytes, which conv_f16_mat.cu and conv_f16_raw.cu cannot bring in with tiled copies, and the 3x3 layers of stride 1 on which it
// is the faster one (runs_before_tiled in api.cu).
//
// Columns.  In the im2win tensor the s*Kh elements of columns i*s .. i*s + s - 1 of a strip are contiguous, so a
// convolution of stride s is one of stride 1 on columns s times as tall: virtual column i holds e = t*Kh + u
// (t < min(s, Kw)), E = min(s, Kw)*Kh of them, and the kernel is G = ceil(Kw/s) virtual columns wide; filter elements
// with g*s + t >= Kw are zeros (3x3 with stride 2: a third more products, but every element is staged once and from
// one run).  A GEMM row is a virtual position q = (n*Ho + ho)*Wq + i, Wq = ceil(Wp/s); S[row][64 k2] is staged once per k2-block and
// the MMAs of virtual kernel column g read the view that starts g rows further down.
//
// Order of k2.  A unit of eight k2 (16 bytes of S) is eight channels at one e: unit j = octet * E + e (up to four
// channels: four channels at two e).  The places of a row's elements in the eight channel planes are then the same
// for every unit but for one uniform offset -- also where planes start at different phases of 16 bytes, because
// eight planes further the phase repeats -- and a unit costs a thread eight 2-byte shared loads, four packs and one
// store.
//
// Raw copies.  The columns a tile needs of one channel are one contiguous run per image it touches.  An untiled bulk copy
// brings a run from the 16-byte boundary below to the one above into a ring of raw slots (`octs` octets of channels
// each); or, where 1, 2 or 4 channel planes are a multiple of 16 bytes and a tile touches at most two images, a tiled copy brings
// the same run of every first, second or fourth channel of an octet (a copy costs the copy engine about 100 cycles, whatever
// its size).  Gathering with 2-byte global loads instead (conv_f16_shift.cu) makes every load instruction
// touch 32 rows s*Kh elements apart: three or more L1 wavefronts each, and a round trip to memory per batch.
//
// Above 128 channels two CTAs form a pair (M = 256, cta_group::2): each stages its own position tile and half of the filter,
// and the second CTA's MMA warp tells the leader that its half of a filter slot has arrived.
//
// Where tiles are so few that SMs would be left over, the CTAs of a cluster share a tile's k2-blocks and add their accumulators up
// (SPLIT; see choose_split for when and what it gives).  A part may begin and end within a raw slot, which then two CTAs copy.
//
// What bounds it: no single pipe.  With the read-back, the S stores, the MMAs and the output stores all left out, what remains
// (copies, hand-offs, the staging warps' arithmetic) still takes four fifths of the time: 86 of 109 us for 3x3 on 64 channels at
// 56x56, batch 128.  Measured: 3x3 stride 2 on 256 -> 512 channels at 28x28, batch 128, 140 us with the gathering kernel,
// 112 with a unit at a time, no pairs and two S stages, now 88 (670 TFLOP/s); 3x3 on 256 channels at 28x28, batch 64, 70 -> 58;
// 64 -> 128 channels at 112x112, batch 64, 256 -> 194; 5x5 stride 2 on 37 -> 75 channels at 45x61, batch 13, 27 (gathering) and 13.
// Eight staging warps: twelve or sixteen, with four epilogue warps, gave 111 and 117 us where eight gave 113, and 115 and 125 us
// where eight gave 103.
#include <cuda_fp16.h>
#include <cuda.h>
#include <stdlib.h>
#include <string.h>

#define IM2WIN_INLINE_SLOW_WAIT      // (a call beside the epilogue's live sums costs spills)
#include "common.cuh"
#include "launch.cuh"
#include "ptx_sm100.cuh"

namespace im2win {
namespace {

using namespace ptx;

constexpr int TILE_M = 128;
constexpr int KB = 64;
constexpr int MAX_A = 4, MAX_RAW = 8, MAX_B = 16, MAX_ACC = 8;
constexpr int MAX_SEG = 6;                    // images a tile may touch
constexpr int kRunsSmem = 226 * 1024;
constexpr int STAGING_WARPS = 8;
constexpr int THREADS = 32 * (STAGING_WARPS + 4 + 8);   // staging; MMA, filter copies, two raw-copy warps; epilogue

// n / d for n below 2^31: (n * mul) >> shift with mul = floor(2^shift / d) + 1, shift = 31 + ceil(log2 d).
struct FastDiv {
  uint32_t mul, shift;
  __device__ __forceinline__ uint32_t operator()(uint32_t n) const { return (uint32_t)(((uint64_t)n * mul) >> shift); }
};
FastDiv fast_div(uint32_t d) {
  uint32_t l = 0;
  while (((uint64_t)1 << l) < d) ++l;
  return {(uint32_t)((((uint64_t)1 << (31 + l)) / d) + 1), 31 + l};
}

struct alignas(64) RunsParams {
  CUtensorMap map;                            // window tensor in rows of `planes` channel planes (tiled raw copies)
  const unsigned char* __restrict__ win;
  const unsigned char* __restrict__ fp;       // packed filter: shared-memory images, see pack_f16_runs_kernel
  float* __restrict__ y;
  uint32_t* status;
  int64_t img_bytes, chan_bytes, win_bytes;   // of one image, one channel plane, the whole window tensor
  uint32_t VQ;
  FastDiv div_wq, div_ho;
  int32_t C, Wp, Wq, Ho, Wo, HoWo, Co, Kh, Kw, s;
  int32_t E, G, units, num_kb, nks_last;      // units: of eight k2
  int32_t quad;                               // 1: up to four channels, a unit is four channels at two e
  int32_t foreign;                            // 1: zero filter elements meet elements that are not of the window
  int32_t halo, region, octs, raw_slot, a_stage;
  int32_t bn, ntn, nwork, sa, sr, sb, slot_bytes, resident;
  int32_t teams;                              // of staging warps, a divisor of sr
  int32_t cols;                               // kernel columns in a filter slot
  int32_t ntm;                                // position tiles
  int32_t planes;                             // the least number of channel planes that is a multiple of 16 bytes; 0: bulk copies
  int32_t seg_bytes;                          // tiled copies: from image to image of a tile in a raw slot
  int32_t split;                              // CTAs of a cluster that share the k2-blocks of a tile
};

__device__ __forceinline__ uint32_t ld_shared_u16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
constexpr int ES = 2;                         // bytes of an element
constexpr int REGS_STAGING = 96, REGS_MISC = 64, REGS_EPILOGUE = 112;   // 2*96 + 64 + 2*112 = 5*96

// Where the rows of a tile lie: image n0 + g of the tile is a run of its own, [start, end) in elements of a channel
// plane, at byte seg_off(g) of a channel's region in a raw slot.
struct TileRuns {
  uint32_t n0, n1;
  int32_t start0, end1;                                     // first element of image n0, end in image n1
};
__device__ __forceinline__ int run_size(int elems) { return (elems * ES + 30) & ~15; }
__device__ __forceinline__ void split_q(const RunsParams& q, uint32_t vq, uint32_t& n, int& ho, int& i) {
  const uint32_t sg = q.div_wq(vq);
  i = (int)(vq - sg * (uint32_t)q.Wq);
  n = q.div_ho(sg);
  ho = (int)(sg - n * (uint32_t)q.Ho);
}
__device__ __forceinline__ TileRuns tile_runs(const RunsParams& q, uint32_t q0) {
  TileRuns r;
  int ho, i;
  split_q(q, q0, r.n0, ho, i);
  r.start0 = (ho * q.Wp + i * q.s) * q.Kh;
  uint32_t ql = q0 + TILE_M + q.halo - 1;
  if (ql >= q.VQ) ql = q.VQ - 1;
  split_q(q, ql, r.n1, ho, i);
  // (all s columns of the last virtual column: where s does not divide Wp some lie in the next strip or plane.  Only
  // zero filter elements meet them, but they have to be numbers)
  r.end1 = (ho * q.Wp + (i + 1) * q.s) * q.Kh;
  return r;
}

// The outputs y[i * ystride], i < which <= 16 (MASK: those whose bit i of `which` is set), that came out infinite or NaN although a zero filter element may have met an
// infinity or NaN from outside their window (RunsParams::foreign): in fp32 FMAs, k ascending, from the window at x and
// rows i of the filter image at f.  Sixteen sums at a time keep the loads of the filter (the same address in every lane) in
// flight; they end early once all are NaN.  (A function of its own: expanded beside the epilogue it costs spills.)
template <bool MASK>
__device__ __noinline__ void exact_outputs(const unsigned char* __restrict__ x, const unsigned char* __restrict__ f, float* y,
                                           int64_t ystride, int64_t chan_bytes, int C, int Kh, int Kw, int s, int E, int g_step,
                                           int j_step, int quad, int which) {
  auto not_finite = [](float v) { return !(fabsf(v) <= 3.4028234663852886e38f); };
  bool any = false;
  auto mine = [&](int i) { return MASK ? (which >> i & 1) != 0 : i < which; };
  for (int i = 0; MASK ? i < 16 : i < which; ++i) any |= mine(i) && not_finite(y[i * ystride]);
  if (!any) return;
  float acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.f;
  bool open = true;
#pragma unroll 1
  for (int c = 0; c < C && open; ++c, x += chan_bytes) {
    int g = 0, t = 0;                                      // kernel column v = g * s + t
#pragma unroll 1
    for (int v = 0; v < Kw; ++v) {
#pragma unroll 1
      for (int u = 0; u < Kh; ++u) {
        const int e = t * Kh + u;
        const int j = quad ? e >> 1 : (c >> 3) * E + e, at = quad ? (e & 1) * 4 + c : c & 7;      // unit, place in it
        const unsigned char* fj = f + (int64_t)(j >> 3) * j_step + (int64_t)g * g_step + at * ES;
        const float xv = __half2float(*reinterpret_cast<const __half*>(x + (v * Kh + u) * ES));
#pragma unroll
        for (int i = 0; i < 16; ++i)                       // (rows up to the next multiple of 16 exist)
          acc[i] = fmaf(xv, __half2float(*reinterpret_cast<const __half*>(fj + i * 128 + (((j & 7) ^ (i & 7)) << 4))), acc[i]);
      }
      if (++t == s) { t = 0; ++g; }
    }
    open = false;
#pragma unroll
    for (int i = 0; i < 16; ++i) open |= acc[i] == acc[i];
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float* p = y + i * ystride;
    if (mine(i) && not_finite(*p)) *p = acc[i];
  }
}

// The MMAs of COLS kernel columns, straight-line: a lone lane pays for every branch and address computation between them.
template <int NKS, int COLS, bool PAIR>
__device__ __forceinline__ void issue_columns(uint32_t d, uint32_t a, uint32_t b, uint32_t b_step, uint32_t idesc, uint32_t more) {
#pragma unroll
  for (int g = 0; g < COLS; ++g, b += b_step)              // next view: one row (128 bytes) further down
#pragma unroll
    for (int j = 0; j < NKS; ++j) {
      const uint32_t acc = g == 0 && j == 0 ? more : 1u;
      if (PAIR) umma_f16_ab_pair(d, a + 8 * g + 2 * j, kSmemDescHiSw128, b + 2 * j, kSmemDescHiSw128, idesc, acc);
      else umma_f16_lohi(d, a + 8 * g + 2 * j, b + 2 * j, idesc, acc);
    }
}
template <int COLS, bool PAIR>
__device__ __forceinline__ void issue_slot(int nks, uint32_t d, uint32_t a, uint32_t b, uint32_t b_step, uint32_t idesc, uint32_t more) {
  if (nks == KB / 16) issue_columns<KB / 16, COLS, PAIR>(d, a, b, b_step, idesc, more);
  else if (nks == 3) issue_columns<3, COLS, PAIR>(d, a, b, b_step, idesc, more);
  else if (nks == 2) issue_columns<2, COLS, PAIR>(d, a, b, b_step, idesc, more);
  else issue_columns<1, COLS, PAIR>(d, a, b, b_step, idesc, more);
}

// The work items of a CTA: items first, first + step, ...; an item is a channel tile of one position tile, or of two for a
// CTA pair (of an odd number of position tiles the last is staged by both and stored by one).
struct Walk {
  int first, step, rank, pair;
  __device__ __forceinline__ int tile(const RunsParams& q, int w) const { return pair ? 2 * (w / q.ntn) + rank : w / q.ntn; }
  __device__ __forceinline__ uint32_t start(const RunsParams& q, int w) const {
    const int mt = tile(q, w);
    return (uint32_t)(mt < q.ntm ? mt : q.ntm - 1) * TILE_M;
  }
};

// Where channel x of an octet lies in a raw slot: tiled copies bring every `planes`-th channel at a time.
__device__ __forceinline__ int slot_row(const RunsParams& q, int x) {
  if (q.planes <= 1) return x;
  return q.planes == 2 ? (x & 1) * 4 + (x >> 1) : (x & 3) * 2 + (x >> 2);
}

// The staging warps: raw runs -> S, thread = row (or two neighbouring rows).
//   HALVES     an element at a time: any alignment
//   WORDS      two elements of a row at a time: E even and every row on a 4-byte boundary (strides of 2)
//   ROW_PAIRS  rows 2t and 2t + 1 of a 3-high kernel at stride 1 are six neighbouring elements, read as three words: images
//              of an even number of virtual columns, so that no pair lies in two images
//   UNITS      an element and a unit at a time, both warpgroups on every slot: any layer (stage_units)
// The kernel is compiled for each by itself: small layers pay for code that is skipped (in one kernel for all, 8 to 9 us where
// a kernel of UNITS alone takes 6 to 7).
enum StagingMode { HALVES, WORDS, ROW_PAIRS, UNITS };
constexpr int group_of(int mode) { return mode == WORDS ? 6 : 3; }

// The part of the reduction a CTA does: k2-blocks, units and raw slots (of the first and the last slot maybe not every unit).
struct Part {
  int kb0, kb1, j0, j1, slot0, slot1;
};
__device__ __forceinline__ Part part_of(const RunsParams& q, int rank) {
  const int per_slot = q.quad ? q.units : q.octs * q.E;
  Part p;
  p.kb0 = q.num_kb * rank / q.split;
  p.kb1 = q.num_kb * (rank + 1) / q.split;
  p.j0 = 8 * p.kb0;
  p.j1 = 8 * p.kb1 < q.units ? 8 * p.kb1 : q.units;
  p.slot0 = p.j0 / per_slot;
  p.slot1 = (p.j1 + per_slot - 1) / per_slot;
  return p;
}

struct StagingBarriers {
  uint32_t a_full0, a_empty0, raw_full0, raw_empty0;        // (a_full0 in a pair: the leader's, wherever it lies)
};

// Place of the first element of virtual position vq in channel x of a slot's octet: byte inside the raw slot.
__device__ __forceinline__ void locate_row(const RunsParams& q, const TileRuns& tr, int plane, uint32_t vq, bool quad, uint32_t (&rb)[8]) {
  uint32_t off = 0, phase = 0;
  if (vq < q.VQ) {                                           // dead rows read whatever lies at the start: they are dropped
    uint32_t n;
    int ho, i;
    split_q(q, vq, n, ho, i);
    const int g = (int)(n - tr.n0), start = g == 0 ? tr.start0 : 0;
    if (q.planes) off = g * q.seg_bytes;
    else if (g > 0) off = run_size(plane - tr.start0) + (g - 1) * run_size(plane);
    off += ((ho * q.Wp + i * q.s) * q.Kh - start) * ES;
    phase = (uint32_t)((int64_t)n * q.img_bytes + (int64_t)start * ES);
  }
#pragma unroll
  for (int x = 0; x < 8; ++x) rb[x] = off + slot_row(q, x) * q.region + ((phase + (uint32_t)x * (uint32_t)q.chan_bytes) & 15u);
  if (quad) {
#pragma unroll
    for (int x = 0; x < 4; ++x) rb[4 + x] = rb[x] + ES;
  }
}

// A team of warps covers the rows of the tile and takes every `teams`-th slot as a whole; all loads of up to GROUP units
// are in flight together, and the slot is given back before the wait for a free S stage.  (A unit at a time, both
// warpgroups on every slot, took 87 instructions and 560 cycles a unit: 3x3 stride 2 on 256 -> 512 channels at 28x28, batch
// 128, 121 us.)
template <int MODE, bool PAIR, bool SPLIT>
__device__ __forceinline__ void stage_tiles(const RunsParams& q, const Walk& walk, const Part& part, uint32_t a_ring, uint32_t raw_ring,
                                            const StagingBarriers& b, int warp, int lane, volatile uint32_t* abort_flag) {
  auto arrive_full = [&](int stage) {
    if (PAIR) mbar_arrive_cluster(b.a_full0 + 8 * stage);
    else mbar_arrive(b.a_full0 + 8 * stage);
  };
  constexpr int ROWS = MODE == ROW_PAIRS ? 2 : 1;
  constexpr int TEAM = 4 / ROWS;
  constexpr int GROUP = MODE == WORDS ? 6 : 3;              // units in flight
  const int team = warp / TEAM, row = ((warp % TEAM) * 32 + lane) * ROWS;
  const int plane = (q.Ho * q.Wp + q.Wq * q.s - q.Wp) * q.Kh;     // (up to the end of the last virtual column)
  const int per_oct = q.E, nocts = q.units / q.E, octs = q.octs;
  const int nslots = SPLIT ? part.slot1 - part.slot0 : (nocts + octs - 1) / octs;      // (`next` counts from the part's first slot)
  auto swizzled = [](int r) { return (uint32_t)(r * 128 + ((r & 7) << 4)); };
  // (lanes 4 to 7 of eight store the second row of a pair first: the eight meet eight bank groups)
  const int second = ROWS == 2 ? (lane >> 2) & 1 : 0;
  const uint32_t dst0 = swizzled(row + second), dst1 = ROWS == 2 ? swizzled(row + 1 - second) : 0u;
  // rows below the tile: lane -> (row, unit of the group); one warp of the team has them, another one from slot to slot
  bool ok = true;
  // The number of teams divides the number of slots, so that a slot's fills all belong to one team.  It has waited for the one
  // before when it waits for the next, whose parity then is not that of two fills ago.  (With slots that go from team to team
  // that one may not have landed yet: copies of different slots land in any order.)
  const int teams = q.teams;
  int sa = 0, sr = team, next = team < teams ? team : 1 << 30;    // (next: this team's next slot of the tile)
  uint32_t pa = 0, pr = 0;
  uint32_t turn = 0;
  for (int w = walk.first; w < q.nwork && ok; w += walk.step) {
    const uint32_t q0 = walk.start(q, w);
    const TileRuns tr = tile_runs(q, q0);
    auto locate = [&](int r, uint32_t (&at)[8]) { locate_row(q, tr, plane, q0 + r, false, at); };
    uint32_t rb[8], hb[8];
    locate(row, rb);
    const int he = q.halo > 0 ? lane / q.halo : GROUP, hrow = TILE_M + lane - he * q.halo;
    if (he < GROUP) {
      locate(hrow, hb);
#pragma unroll
      for (int x = 0; x < 8; ++x) hb[x] += he * ES;
    }
    int kb = 0;                                              // S stage this warp is at, and whether it may write to it
    bool held = false;
    auto go_to = [&](int target) {
      while (ok && !(held && kb == target)) {
        if (!held) {
          ok = mbar_wait(b.a_empty0 + 8 * sa, pa ^ 1u, abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          held = true;
        } else {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) arrive_full(sa);
          if (++sa == q.sa) { sa = 0; pa ^= 1u; }
          ++kb;
          held = false;
        }
      }
    };
    for (; next < nslots && ok; next += teams, ++turn) {
      ok = mbar_wait(b.raw_full0 + 8 * sr, pr, abort_flag, q.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      uint32_t src = raw_ring + sr * q.raw_slot;
      const bool halo_turn = q.halo > 0 && (int)(turn % TEAM) == warp % TEAM;
      const int slot = SPLIT ? part.slot0 + next : next;
      const int here = nocts - slot * octs < octs ? nocts - slot * octs : octs;
      int j = slot * octs * per_oct;                                // unit
      for (int o = 0; o < here && ok; ++o, src += 8u * q.region) {
        for (int e0 = 0; e0 < per_oct && ok; e0 += GROUP) {
          const int n = per_oct - e0 < GROUP ? per_oct - e0 : GROUP;
          const uint32_t at = src + e0 * ES;
          uint32_t p[GROUP * ROWS][4], hp[4] = {};
          if constexpr (MODE == WORDS || MODE == ROW_PAIRS) {
            uint32_t v[3][8];                                // (beyond the octet's last unit: place 0 again)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              const uint32_t from = MODE == ROW_PAIRS || 2 * i < n ? at + 4 * i : at;
#pragma unroll
              for (int x = 0; x < 8; ++x) v[i][x] = ld_shared_u32(from + rb[x]);
            }
#pragma unroll
            for (int i = 0; i < 6; ++i)
#pragma unroll
              for (int x = 0; x < 4; ++x)
                p[i][x] = __byte_perm(v[i / 2][2 * x], v[i / 2][2 * x + 1], (i & 1) ? 0x7632 : 0x5410);
          } else {
            uint32_t v[GROUP][8];
#pragma unroll
            for (int i = 0; i < GROUP; ++i) {
              const uint32_t from = i < n ? at + i * ES : at;
#pragma unroll
              for (int x = 0; x < 8; ++x) v[i][x] = ld_shared_u16(from + rb[x]);
            }
#pragma unroll
            for (int i = 0; i < GROUP; ++i)
#pragma unroll
              for (int x = 0; x < 4; ++x) p[i][x] = __byte_perm(v[i][2 * x], v[i][2 * x + 1], 0x5410);
          }
          if (halo_turn && he < n) {
#pragma unroll
            for (int x = 0; x < 4; ++x)
              hp[x] = __byte_perm(ld_shared_u16(at + hb[2 * x]), ld_shared_u16(at + hb[2 * x + 1]), 0x5410);
          }
          if (o == here - 1 && e0 + GROUP >= per_oct) {      // everything of the slot is in registers
            __syncwarp();
            if (lane == 0) mbar_arrive(b.raw_empty0 + 8 * sr);
          }
#pragma unroll
          for (int i = 0; i < GROUP; ++i) {
            if (i >= n) break;
            if (SPLIT && (j + i < part.j0 || j + i >= part.j1)) continue;      // (another CTA's)
            go_to(((j + i) >> 3) - part.kb0);
            if (!ok) break;
            const uint32_t stage = a_ring + sa * q.a_stage, ch = (uint32_t)((j + i) & 7) << 4;
            if constexpr (ROWS == 2) {
              const uint32_t (&r0)[4] = p[i], (&r1)[4] = p[3 + i];
              st_shared16(stage + (dst0 ^ ch), second ? r1[0] : r0[0], second ? r1[1] : r0[1], second ? r1[2] : r0[2], second ? r1[3] : r0[3]);
              st_shared16(stage + (dst1 ^ ch), second ? r0[0] : r1[0], second ? r0[1] : r1[1], second ? r0[2] : r1[2], second ? r0[3] : r1[3]);
            } else {
              st_shared16(stage + (dst0 ^ ch), p[i][0], p[i][1], p[i][2], p[i][3]);
            }
            if (halo_turn && he == i) st_shared16(stage + (swizzled(hrow) ^ ch), hp[0], hp[1], hp[2], hp[3]);
          }
          j += n;
        }
      }
      sr += teams;
      if (sr >= q.sr) { sr -= q.sr; pr ^= 1u; }
    }
    if (team < teams) next -= nslots;
    go_to(part.kb1 - part.kb0 - 1);
    if (!ok) break;
    if ((q.units & 1) != 0 && part.kb1 == q.num_kb && team == 0) {                   // zeros up to the end of the MMA's last step
      const uint32_t stage = a_ring + sa * q.a_stage, ch = (uint32_t)(q.units & 7) << 4;
      st_shared16(stage + (dst0 ^ ch), 0u, 0u, 0u, 0u);
      if (ROWS == 2) st_shared16(stage + (dst1 ^ ch), 0u, 0u, 0u, 0u);
      if (warp == 0 && lane < q.halo) st_shared16(stage + (swizzled(TILE_M + lane) ^ ch), 0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) arrive_full(sa);
    if (++sa == q.sa) { sa = 0; pa ^= 1u; }
  }
}

// The form for layers that give the teams too little to share out (see plan_f16_runs) or have more rows below a tile than a warp
// can read for a group of units.  Warpgroup wg takes every second unit; every warp passes every stage and every slot in order, so no wait by phase
// parity can run ahead.
template <bool PAIR, bool SPLIT>
__device__ __forceinline__ void stage_units(const RunsParams& q, const Walk& walk, const Part& part, uint32_t a_ring, uint32_t raw_ring,
                                            const StagingBarriers& b, int warp, int lane, volatile uint32_t* abort_flag) {
  const int wg = warp >> 2, row = (warp & 3) * 32 + lane;
  const int plane = (q.Ho * q.Wp + q.Wq * q.s - q.Wp) * q.Kh;     // (up to the end of the last virtual column)
  const int per_slot = q.quad ? q.units : q.octs * q.E;
  const uint32_t oct_step = 8u * q.region - (uint32_t)(q.E - 1) * ES, unit_step = q.quad ? 2u * ES : ES;
  bool ok = true;
  int sa = 0, sr = 0;
  uint32_t pa = 0, pr = 0;
  for (int w = walk.first; w < q.nwork && ok; w += walk.step) {
    const uint32_t q0 = walk.start(q, w);
    const TileRuns tr = tile_runs(q, q0);
    uint32_t rb[8], hb[8];
    locate_row(q, tr, plane, q0 + row, q.quad, rb);
    if (lane < q.halo) locate_row(q, tr, plane, q0 + TILE_M + lane, q.quad, hb);
    uint32_t src = 0;                                        // of the current unit; inside the slot: its number, and its e
    int in_slot = SPLIT ? part.j0 - part.slot0 * per_slot : 0, e = 0;
    bool enter = true;                                       // the next unit is the first one of a slot
    for (int kb = part.kb0; kb < part.kb1 && ok; ++kb) {
      ok = mbar_wait(b.a_empty0 + 8 * sa, pa ^ 1u, abort_flag, q.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const uint32_t stage = a_ring + sa * q.a_stage;
      const int n_units = q.units - 8 * kb < 8 ? q.units - 8 * kb : 8;
      for (int ch = 0; ch < n_units; ++ch) {
        if (enter) {
          ok = mbar_wait(b.raw_full0 + 8 * sr, pr, abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          src = raw_ring + sr * q.raw_slot;
          e = 0;
          if (SPLIT && in_slot > 0) {                        // (the part starts within a slot)
            const int o = q.quad ? 0 : in_slot / q.E;
            e = in_slot - o * q.E;
            src += 8u * q.region * o + unit_step * e;
          }
          enter = false;
        }
        if ((ch & 1) == wg) {
          auto unit = [&](const uint32_t (&at)[8], int srow) {
            uint32_t v[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) v[x] = ld_shared_u16(src + at[x]);
            st_shared16(stage + srow * 128 + ((ch ^ (srow & 7)) << 4), v[0] | (v[1] << 16), v[2] | (v[3] << 16),
                        v[4] | (v[5] << 16), v[6] | (v[7] << 16));
          };
          unit(rb, row);
          // the rows below the tile: lanes of one of the warpgroup's warps, another one from unit to unit
          if ((ch >> 1) == (warp & 3) && lane < q.halo) unit(hb, TILE_M + lane);
        }
        if (++in_slot == per_slot || 8 * kb + ch == part.j1 - 1) {
          __syncwarp();
          if (lane == 0) mbar_arrive(b.raw_empty0 + 8 * sr);
          if (++sr == q.sr) { sr = 0; pr ^= 1u; }
          in_slot = 0;
          enter = true;
        }
        ++e;
        src += e == q.E ? oct_step : unit_step;
        if (e == q.E) e = 0;
      }
      if (!ok) break;
      if ((n_units & 1) != 0 && wg == 1) {                   // zeros up to the end of the MMA's last step
        st_shared16(stage + row * 128 + ((n_units ^ (row & 7)) << 4), 0u, 0u, 0u, 0u);
        if (lane < q.halo) st_shared16(stage + (TILE_M + lane) * 128 + ((n_units ^ (lane & 7)) << 4), 0u, 0u, 0u, 0u);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(b.a_full0 + 8 * sa);
        else mbar_arrive(b.a_full0 + 8 * sa);
      }
      if (++sa == q.sa) { sa = 0; pa ^= 1u; }
    }
  }
}

template <int BNMAX, bool PAIR, int MODE, bool SPLIT>
__global__ void __launch_bounds__(THREADS, 1) conv_f16_runs_kernel(const __grid_constant__ RunsParams q) {
  constexpr int NACC = 512 / BNMAX, ACC_LOG = NACC == 2 ? 1 : (NACC == 4 ? 2 : 3);      // ring of accumulators in tensor memory
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bars[2 * (MAX_A + MAX_RAW + MAX_B + MAX_ACC)];
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile uint32_t abort_flag;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t a_ring = smem_u32(smem);
  const uint32_t b_ring = a_ring + q.sa * q.a_stage;
  const uint32_t raw_ring = b_ring + q.sb * q.slot_bytes;
  const uint32_t a_full0 = smem_u32(&bars[0]), a_empty0 = a_full0 + 8 * MAX_A;
  const uint32_t raw_full0 = a_empty0 + 8 * MAX_A, raw_empty0 = raw_full0 + 8 * MAX_RAW;
  const uint32_t b_full0 = raw_empty0 + 8 * MAX_RAW, b_empty0 = b_full0 + 8 * MAX_B;
  const uint32_t acc_full0 = b_empty0 + 8 * MAX_B, acc_empty0 = acc_full0 + 8 * MAX_ACC;
  const int rank = PAIR ? (int)cluster_ctarank() : 0;
  // (SPLIT: the cluster has one item, this CTA that part of its reduction)
  const int share = SPLIT ? (int)cluster_ctarank() : 0;
  const Walk walk = {SPLIT ? (int)blockIdx.x / q.split : (PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x),
                     SPLIT ? q.nwork : (PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x), rank, PAIR};
  const Part part = SPLIT ? part_of(q, share) : Part{0, q.num_kb, 0, q.units, 0, 0};   // (unsplit the slots are counted where they are used)
  // the leader's barriers that both CTAs of a pair arrive on
  const uint32_t a_full_dst = PAIR ? mapa_shared(a_full0, 0) : a_full0;
  const uint32_t b_full_dst = PAIR ? mapa_shared(b_full0, 0) : b_full0;
  const uint32_t acc_empty_dst = PAIR ? mapa_shared(acc_empty0, 0) : acc_empty0;
  bool met = false;                                        // SPLIT: this warp has been at the cluster's barriers
  const int b_rows = PAIR ? q.bn / 2 : q.bn;               // filter rows (channels) this CTA holds of a kernel column

  if (threadIdx.x == 0) {
    abort_flag = 0u;
    for (int i = 0; i < MAX_A; ++i) { mbar_init(a_full0 + 8 * i, PAIR ? 2 * STAGING_WARPS : STAGING_WARPS); mbar_init(a_empty0 + 8 * i, 1); }
    for (int i = 0; i < MAX_RAW; ++i) { mbar_init(raw_full0 + 8 * i, 1); mbar_init(raw_empty0 + 8 * i, MODE == UNITS ? STAGING_WARPS : (MODE == ROW_PAIRS ? 2 : 4)); }
    // (the leader's b_full: its own copy and word from the other CTA's)
    for (int i = 0; i < MAX_B; ++i) { mbar_init(b_full0 + 8 * i, PAIR && rank == 0 ? 2 : 1); mbar_init(b_empty0 + 8 * i, 1); }
    for (int i = 0; i < MAX_ACC; ++i) { mbar_init(acc_full0 + 8 * i, 1); mbar_init(acc_empty0 + 8 * i, PAIR ? 16 : 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == STAGING_WARPS) {
    if (PAIR) tmem_alloc_pair(smem_u32(&tmem_base_slot), 512);
    else tmem_alloc(smem_u32(&tmem_base_slot), 512);
  }
  // The raw ring starts as zeros: places no copy fills (channels beyond C in the last octet) meet zero filter
  // elements, but they have to be numbers.
  for (int i = threadIdx.x * 16; i < q.sr * q.raw_slot; i += THREADS * 16) st_shared16(raw_ring + i, 0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();                             // the peer's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_acc = tmem_base_slot;
  wait_for_previous_kernel();

  if (warp < STAGING_WARPS) {
    // ---------------- staging: raw runs -> S ------------------------------------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_STAGING));
    const StagingBarriers b = {a_full_dst, a_empty0, raw_full0, raw_empty0};
    if constexpr (MODE == UNITS) stage_units<PAIR, SPLIT>(q, walk, part, a_ring, raw_ring, b, warp, lane, &abort_flag);
    else stage_tiles<MODE, PAIR, SPLIT>(q, walk, part, a_ring, raw_ring, b, warp, lane, &abort_flag);
  } else if (warp < STAGING_WARPS + 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_MISC));
    if (warp == STAGING_WARPS && rank == 0) {
      // ---------------- MMA issuer (the leader of a pair) -----------------------------------------------------------------------
      const bool leader = elect_one();
      const uint32_t a_lo0 = smem_desc_lo(a_ring), b_lo0 = smem_desc_lo(b_ring);
      const uint32_t idesc = instr_desc_f16(PAIR ? 2 * TILE_M : TILE_M, q.bn), b_step = (uint32_t)b_rows * 8u;
      bool ok = true;
      int sa = 0, slot = 0;
      uint32_t pa = 0, pb = 0, ac = 0;                       // ... tiles so far
      // A wait for a barrier that is already complete costs 200 cycles and more while the shared-memory pipe is busy, and
      // the tensor pipe runs dry meanwhile: every barrier is looked at ahead of the instructions issued before it is
      // needed, and waited for only where that look came too early.
      uint32_t a_seen = 0, b_seen = 0, acc_seen = 0;
      // (testing aid: the commit of the first tile left out; looked up while its first stage is on its way)
      uint32_t drop = blockIdx.x == 0 ? *reinterpret_cast<volatile uint32_t*>(q.status + 2) : 0u;
      // (in a pair the other CTA arrives on all three kinds: cluster scope)
      auto need = [&](uint32_t bar, uint32_t parity, uint32_t seen) {
        return mbar_wait_unless_seen<PAIR>(bar, parity, seen, &abort_flag, q.status);
      };
      auto look = [&](uint32_t bar, uint32_t parity) { return PAIR ? mbar_test_wait_cluster(bar, parity) : mbar_test_wait(bar, parity); };
      auto commit = [&](uint32_t bar) {
        if (PAIR) umma_commit_pair(bar);
        else umma_commit(bar);
      };
      for (int w = walk.first; w < q.nwork && ok; w += walk.step, ++ac) {
        const int ab = ac & (NACC - 1);
        ok = need(acc_empty0 + 8 * ab, ((ac >> ACC_LOG) & 1) ^ 1, acc_seen);
        if (!ok) break;
        const uint32_t d = tmem_acc + ab * BNMAX;
        uint32_t more = 0u;                                  // the tile's first instruction clears the accumulator
        const bool fetch_b = !q.resident || w == walk.first;          // (a resident filter is complete after the first tile)
        if (q.resident) slot = 0;
        for (int kb = part.kb0; kb < part.kb1 && ok; ++kb) {
          const int nks = kb == q.num_kb - 1 ? q.nks_last : KB / 16;
          ok = need(a_full0 + 8 * sa, pa, a_seen);
          if (!ok) break;
          tc_fence_after();
          uint32_t a_view = a_lo0 + (uint32_t)(sa * (q.a_stage >> 4));
          int nsa = sa + 1;
          uint32_t npa = pa;
          if (nsa == q.sa) { nsa = 0; npa ^= 1u; }
          for (int g = 0; g < q.G; g += q.cols, a_view += 8u * q.cols) {
            const bool last_unit = g + q.cols == q.G, last = kb + 1 == part.kb1 && last_unit;
            int nslot = slot + 1;
            uint32_t npb = pb;
            if (nslot == q.sb) { nslot = 0; if (!q.resident) npb ^= 1u; }
            if (fetch_b) {
              ok = need(b_full0 + 8 * slot, pb, b_seen);
              if (!ok) break;
              b_seen = look(b_full0 + 8 * nslot, npb);
            }
            if (last) acc_seen = look(acc_empty0 + 8 * ((ac + 1) & (NACC - 1)), (((ac + 1) >> ACC_LOG) & 1) ^ 1);
            if (last_unit) a_seen = look(a_full0 + 8 * nsa, npa);
            const uint32_t b_lo = b_lo0 + (uint32_t)(slot * (q.slot_bytes >> 4));
            if (leader) {
              if (q.cols == 3) issue_slot<3, PAIR>(nks, d, a_view, b_lo, b_step, idesc, more);
              else if (q.cols == 2) issue_slot<2, PAIR>(nks, d, a_view, b_lo, b_step, idesc, more);
              else issue_slot<1, PAIR>(nks, d, a_view, b_lo, b_step, idesc, more);
              if (!q.resident) commit(b_empty0 + 8 * slot);
              if (last_unit) commit(a_empty0 + 8 * sa);
              if (last && drop != kDebugDropArrive) commit(acc_full0 + 8 * ab);
            }
            __syncwarp();
            slot = nslot;
            pb = npb;
            more = 1u;
          }
          sa = nsa;
          pa = npa;
        }
        drop = 0u;
      }
    } else if (warp == STAGING_WARPS) {
      // ---------------- the pair's other CTA: word to the leader that its half of a filter slot has arrived --------
      bool ok = true;
      int slot = 0;
      uint32_t pb = 0;
      const int slots = q.num_kb * q.G / q.cols;
      for (int w = walk.first; w < q.nwork && ok; w += walk.step) {
        for (int u = 0; u < slots; ++u) {
          ok = mbar_wait(b_full0 + 8 * slot, pb, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (lane == 0) mbar_arrive_cluster(b_full_dst + 8 * slot);
          __syncwarp();
          if (++slot == q.sb) { slot = 0; pb ^= 1u; }
        }
        if (q.resident) break;
      }
    } else if (warp == STAGING_WARPS + 1) {
      // ---------------- filter copies ----------------------------------------------------------------------
      const bool leader = elect_one();
      bool ok = true;
      int slot = 0;
      uint32_t pb = 0;
      const int slots = (part.kb1 - part.kb0) * q.G / q.cols, column = q.bn * 128;       // bytes of a kernel column's image
      for (int w = walk.first; w < q.nwork && ok; w += walk.step) {
        const unsigned char* src = q.fp + (int64_t)(w % q.ntn) * slots * q.cols * column + rank * b_rows * 128;
        if (SPLIT) src = q.fp + ((int64_t)(w % q.ntn) * q.num_kb + part.kb0) * q.G * column;
        for (int u = 0; u < slots; ++u, src += q.cols * column) {
          ok = mbar_wait(b_empty0 + 8 * slot, pb ^ 1u, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (leader) {
            mbar_arrive_expect_tx(b_full0 + 8 * slot, (uint32_t)q.slot_bytes);
            if (PAIR) {
              for (int c = 0; c < q.cols; ++c)
                bulk_load(b_ring + slot * q.slot_bytes + c * b_rows * 128, src + c * column, (uint32_t)b_rows * 128u, b_full0 + 8 * slot);
            } else {
              bulk_load(b_ring + slot * q.slot_bytes, src, (uint32_t)q.slot_bytes, b_full0 + 8 * slot);
            }
          }
          __syncwarp();
          if (++slot == q.sb) { slot = 0; pb ^= 1u; }
        }
        if (q.resident) break;                               // the whole filter is in place
      }
      if (!ok) for (int i = 0; i < 64; ++i) __nanosleep(1000);   // copies in flight must land first
    } else {
      // ---------------- raw copies: two warps, every second slot each --------------------------------------------------------------------------
      bool ok = true;
      int sr = 0;
      uint32_t pr = 0, sc = warp & 1;
      const int plane = (q.Ho * q.Wp + q.Wq * q.s - q.Wp) * q.Kh;
      const int per_slot = q.quad ? 4 : 8 * q.octs, slot1 = SPLIT ? part.slot1 : (q.quad ? 1 : (q.C + per_slot - 1) / per_slot);
      for (int w = walk.first; w < q.nwork && ok; w += walk.step) {
        const TileRuns tr = tile_runs(q, walk.start(q, w));
        const int nseg = (int)(tr.n1 - tr.n0) + 1;
        // Copy `it` of a slot: one channel of one image.  From slot to slot only its source moves: per_slot planes further a
        // run starts at the same phase of 16 bytes.  (Worked out per slot, a slot's eight copies cost their warp 1270 cycles.)
        const int items = nseg * per_slot;
        auto run_of = [&](int it, int64_t& from, uint32_t& size, uint32_t& to) {
          const int g = it / per_slot, c = it - g * per_slot;
          const int start = g == 0 ? tr.start0 : 0, end = g == nseg - 1 ? tr.end1 : plane;
          const int64_t b0 = (int64_t)(tr.n0 + g) * q.img_bytes + (int64_t)c * q.chan_bytes + (int64_t)start * ES;
          from = b0 & ~(int64_t)15;
          size = (uint32_t)(((b0 + (int64_t)(end - start) * ES + 15) & ~(int64_t)15) - from);
          to = raw_ring + c * q.region + (g == 0 ? 0 : run_size(plane - tr.start0) + (g - 1) * run_size(plane));
        };
        int64_t from0 = 0;
        uint32_t size0 = 0, to0 = 0, total = 0;
        // Tiled copies: lane -> image, octet of the slot and class of its channels; from slot to slot only the row moves.
        int tx = 0, ty = 0, to = 0, oct = 0;
        const int boxes = nseg * q.octs * q.planes;
        if (q.planes) {
          const int g = lane / (q.octs * q.planes), rest = lane - g * q.octs * q.planes, o = rest / q.planes, r = rest - o * q.planes;
          tx = (int)((r * q.chan_bytes + (int64_t)(g == 0 ? tr.start0 : 0) * ES) >> 4) * 2;         // in 8-byte elements, even
          ty = (int)(((int64_t)(tr.n0 + g) * q.C + 8 * o) / q.planes);
          to = o < q.octs ? g * q.seg_bytes + (8 * o + r * (8 / q.planes)) * q.region : 0;
          oct = o;
        } else if (MODE != UNITS) {
          if (lane < items) {
            run_of(lane, from0, size0, to0);
            total = size0;
          }
          for (int it = lane + 32; it < items; it += 32) {
            int64_t from;
            uint32_t size, to;
            run_of(it, from, size, to);
            total += size;
          }
          total = __reduce_add_sync(0xffffffffu, total);
        }
        // bytes behind the first slot's last run, up to the next 16-byte boundary, that are still of the tensor
        const int64_t spare = q.win_bytes - 15 - ((int64_t)tr.n1 * q.img_bytes + (per_slot - 1) * q.chan_bytes + (int64_t)tr.end1 * ES);
        for (int sl = part.slot0; sl < slot1; ++sl, ++sc) {
          if (sc & 1) {
            if (++sr == q.sr) { sr = 0; pr ^= 1u; }
            continue;
          }
          ok = mbar_wait(raw_empty0 + 8 * sr, pr ^ 1u, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (q.planes) {
            const int here = (q.C + 7) / 8 - sl * q.octs < q.octs ? (q.C + 7) / 8 - sl * q.octs : q.octs;     // octets
            if (lane == 0) mbar_arrive_expect_tx(raw_full0 + 8 * sr, (uint32_t)(nseg * here * 8 * q.region));
            __syncwarp();
            if (lane < boxes && oct < here)
              tma_load_2d(raw_ring + sr * q.raw_slot + to, &q.map, tx, ty + sl * q.octs * (8 / q.planes), raw_full0 + 8 * sr);
            __syncwarp();
            if (++sr == q.sr) { sr = 0; pr ^= 1u; }
            continue;
          }
          const int64_t ahead = (int64_t)sl * per_slot * q.chan_bytes;
          if (MODE != UNITS && (sl + 1) * per_slot <= q.C && ahead <= spare) {
            const uint32_t bar = raw_full0 + 8 * sr, slot = sr * q.raw_slot;
            const unsigned char* win = q.win + ahead;
            if (lane == 0) mbar_arrive_expect_tx(bar, total);
            __syncwarp();
            if (lane < items) bulk_load(to0 + slot, win + from0, size0, bar);
            for (int it = lane + 32; it < items; it += 32) {
              int64_t from;
              uint32_t size, to;
              run_of(it, from, size, to);
              bulk_load(to + slot, win + from, size, bar);
            }
            __syncwarp();
            if (++sr == q.sr) { sr = 0; pr ^= 1u; }
            continue;
          }
          // a slot that is not full or may reach the end of the tensor, or one of few (UNITS: not worth working out ahead)
          const uint32_t bar = raw_full0 + 8 * sr;
          const int c0 = sl * per_slot, nc = q.C - c0 < per_slot ? q.C - c0 : per_slot;
          int seg_off = 0;
          for (int g = 0; g < nseg; ++g) {
            const int start = g == 0 ? tr.start0 : 0, end = g == nseg - 1 ? tr.end1 : plane;
            for (int c = lane; c < nc; c += 32) {
              const int64_t b0 = (int64_t)(tr.n0 + g) * q.img_bytes + (int64_t)(c0 + c) * q.chan_bytes + (int64_t)start * ES;
              const int64_t from = b0 & ~(int64_t)15;
              const int64_t stop = b0 + (int64_t)(end - start) * ES;
              int64_t to = (stop + 15) & ~(int64_t)15;
              const uint32_t dst = raw_ring + sr * q.raw_slot + c * q.region + seg_off;
              if (to > q.win_bytes) {                        // the tensor ends here: its last bytes by hand, zeros beyond
                to = q.win_bytes & ~(int64_t)15;
                for (int64_t b = to; b < stop; b += 2)
                  asm volatile("st.shared.u16 [%0], %1;" ::"r"(dst + (uint32_t)(b - from)),
                               "h"(b < q.win_bytes ? *reinterpret_cast<const uint16_t*>(q.win + b) : (uint16_t)0) : "memory");
              }
              if (to > from) {
                mbar_expect_tx(bar, (uint32_t)(to - from));
                bulk_load(dst, q.win + from, (uint32_t)(to - from), bar);
              }
            }
            seg_off += run_size(end - start);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar);
          if (++sr == q.sr) { sr = 0; pr ^= 1u; }
        }
      }
      if (!ok) for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ---------------------------------------------------------------------------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_EPILOGUE));
    const int lq = warp & 3, h = (warp - STAGING_WARPS - 4) >> 2;           // tensor-memory quadrant; which channels
    bool ok = true;
    uint32_t ac = 0;
    auto arrive_empty = [&](int ab) {
      if (PAIR) mbar_arrive_cluster(acc_empty_dst + 8 * ab);
      else mbar_arrive(acc_empty0 + 8 * ab);
    };
    for (int w = walk.first; w < q.nwork && ok; w += walk.step) {
      const int mt = walk.tile(q, w), nt = w % q.ntn;        // (a position tile beyond the last: nothing to store)
      const uint32_t vq = (uint32_t)mt * TILE_M + (uint32_t)(lq * 32 + lane);
      const int co0 = nt * q.bn;
      const int limit = q.Co - co0 < q.bn ? q.Co - co0 : q.bn;            // channels of this tile that exist
      uint32_t n = 0;
      int ho = 0, i0 = 0;
      bool valid = false;
      if (vq < q.VQ) {
        split_q(q, vq, n, ho, i0);
        valid = i0 < q.Wo;                                   // trailing columns of a strip are no output
      }
      float* yrow = q.y + ((int64_t)n * q.Co + co0) * q.HoWo + (int64_t)ho * q.Wo + i0;
      const int ab = ac & (NACC - 1);
      ok = mbar_wait(acc_full0 + 8 * ab, (ac >> ACC_LOG) & 1, &abort_flag, q.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      ++ac;
      tc_fence_after();
      const uint32_t d = tmem_acc + ((uint32_t)(lq * 32) << 16) + ab * BNMAX;
      if constexpr (SPLIT) {
        // the parts of the cluster's tile added up: each CTA finishes its share of the channels
        const ClusterSums sums(a_ring, q.split, share, limit);
        const int position = lq * 32 + lane;
        met = true;
        __syncwarp();
        cluster_sync_all();                                  // (every MMA of every CTA has completed)
#pragma unroll 1
        for (int c0 = h * (BNMAX / 2); c0 < (h + 1) * (BNMAX / 2) && c0 < limit; c0 += 32) {
          uint32_t v[32];
          float f[32];
          tmem_ld32(d + c0, v);
#pragma unroll
          for (int e = 0; e < 32; ++e) f[e] = __uint_as_float(v[e]);
          sums.store(f, c0, limit, position);
        }
        __syncwarp();
        cluster_sync_all();
        if (valid) {
          const int first = share * sums.per, end = first + sums.per < limit ? first + sums.per : limit;
          float zero = 0.f;
          for (int c = first + h; c < end; c += 2) {
            const float sum = sums.sum(c - first, position);
            zero = fmaf(sum, 0.f, zero);
            yrow[(int64_t)c * q.HoWo] = sum;
          }
          if (q.foreign && zero != 0.f) {                    // (a NaN: one of them is not finite)
            const unsigned char* x = q.win + (int64_t)n * q.img_bytes + ((int64_t)ho * q.Wp + (int64_t)i0 * q.s) * q.Kh * ES;
            const int column = q.bn * 128;
            const unsigned char* f = q.fp + (int64_t)nt * q.num_kb * q.G * column;
            for (int c = first & ~15; c < end; c += 16) {
              int which = 0;
              for (int i = 0; i < 16; ++i)
                if (c + i >= first && c + i < end && ((c + i - first) & 1) == h) which |= 1 << i;
              exact_outputs<true>(x, f + c * 128, yrow + (int64_t)c * q.HoWo, q.HoWo, q.chan_bytes, q.C, q.Kh, q.Kw, q.s, q.E, column,
                            q.G * column, q.quad, which);
            }
          }
        }
        break;
      }
#pragma unroll 1
      for (int c0 = h * (BNMAX / 2); c0 < (h + 1) * (BNMAX / 2) && c0 < limit; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(d + c0, v);
        if (c0 + 32 >= (h + 1) * (BNMAX / 2) || c0 + 32 >= limit) {      // the last read of this accumulator
          tc_fence_before();
          __syncwarp();
          if (lane == 0) arrive_empty(ab);
        }
        if (valid) {
          store_strided32(yrow + (int64_t)c0 * q.HoWo, q.HoWo, v, limit - c0);
          float zero = 0.f;
          if (q.foreign) {
#pragma unroll
            for (int j = 0; j < 32; ++j) zero = fmaf(__uint_as_float(c0 + j < limit ? v[j] : 0u), 0.f, zero);
          }
          if (zero != 0.f) {                               // (a NaN: one of them is not finite)
            const unsigned char* x = q.win + (int64_t)n * q.img_bytes + ((int64_t)ho * q.Wp + (int64_t)i0 * q.s) * q.Kh * ES;
            const int column = q.bn * 128;                 // bytes of a filter column's image
            const unsigned char* f = q.fp + (int64_t)nt * q.num_kb * q.G * column;
            for (int c = c0; c < c0 + 32 && c < limit; c += 16)
              exact_outputs<false>(x, f + c * 128, yrow + (int64_t)c * q.HoWo, q.HoWo, q.chan_bytes, q.C, q.Kh, q.Kw, q.s, q.E,
                            column, q.G * column, q.quad, limit - c < 16 ? limit - c : 16);
          }
        }
      }
      if (h * (BNMAX / 2) >= limit) {                      // (no channels for this warp)
        __syncwarp();
        if (lane == 0) arrive_empty(ab);
      }
    }
  }

  if constexpr (SPLIT) {                                     // (the epilogue warps have met theirs, unless a wait gave up)
    if (warp < STAGING_WARPS + 4 || !met) {
      __syncwarp();
      cluster_sync_all();
      cluster_sync_all();
    }
  }

  // ---------------- teardown -----------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (abort_flag) {
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (PAIR) cluster_sync_all();                             // no CTA leaves while its peer may still signal or read it
  if (warp == STAGING_WARPS) {
    __syncwarp();
    tc_fence_after();
    if (PAIR) tmem_dealloc_pair(tmem_acc, 512);
    else tmem_dealloc(tmem_acc, 512);
  }
}

// Filter -> the images the copy warp loads: for every (channel tile nt, k2-block kb, virtual kernel column g) the
// [bn channels][64 k2] in the 128-byte-swizzled order of shared memory.  One block: `rows` channels of one k2-block; per channel its source is one contiguous run of the OIHW
// filter (whole input channels).  Channels beyond Co, k2 beyond C*E and kernel columns beyond Kw are zeros.
__global__ void __launch_bounds__(256) pack_f16_runs_kernel(const uint16_t* __restrict__ f, unsigned char* __restrict__ fp,
                                                        uint32_t* __restrict__ status, int C, int Kh, int Kw, int s, int E, int G,
                                                        int Co, int bn, int num_kb, int rows, int pitch, int quad) {
  extern __shared__ uint16_t pack_h[];
  let_next_kernel_start();                                 // (the convolution sets itself up meanwhile)
  wait_for_previous_kernel();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kStatusBytes / 4) status[threadIdx.x] = 0u;
  const int kb = blockIdx.y, row0 = blockIdx.x * rows;     // (channel blocks along x: any number of channels)
  const int c0 = quad ? 0 : kb * 8 / E * 8;
  int c1 = quad ? C - 1 : (kb * 8 + 7) / E * 8 + 7;
  if (c1 > C - 1) c1 = C - 1;
  const int T2 = Kh * Kw, run = (c1 - c0 + 1) * T2;
  for (int r = 0; r < rows; ++r) {
    const int co = row0 + r;
    if (co >= Co) break;
    const uint16_t* src = f + ((int64_t)co * C + c0) * T2;
    for (int i = threadIdx.x; i < run; i += blockDim.x) pack_h[r * pitch + i] = __ldg(src + i);
  }
  __syncthreads();
  const int items = rows * G * 8;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int ch = it & 7, rg = it >> 3;
    const int r = rg % rows, g = rg / rows;
    const int row = row0 + r, nt = row / bn, rr = row - nt * bn;
    uint32_t p[4] = {};
    const int j = kb * 8 + ch;                               // unit: eight channels at one e, or four channels at two
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int o = j / E, e = quad ? 2 * j + (x >> 2) : j - o * E, c = quad ? (x & 3) : o * 8 + x;
      const int t = e / Kh, u = e - t * Kh, v = g * s + t;
      uint32_t a = 0;
      if (row < Co && c < C && e < E && v < Kw) a = pack_h[r * pitch + (c - c0) * T2 + u * Kw + v];
      p[x >> 1] |= a << (16 * (x & 1));
    }
    *reinterpret_cast<uint4*>(fp + ((((int64_t)nt * num_kb + kb) * G + g) * bn + rr) * 128 + ((ch ^ (rr & 7)) << 4)) =
        make_uint4(p[0], p[1], p[2], p[3]);
  }
}

template <int BNMAX, bool PAIR, int MODE, bool SPLIT>
cudaError_t launch_mode(const RunsParams& q, int smem, cudaStream_t stream) {
  constexpr auto kernel = conv_f16_runs_kernel<BNMAX, PAIR, MODE, SPLIT>;
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRunsSmem);
    if (e == cudaSuccess && SPLIT) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  if constexpr (SPLIT) {
    static KnownClusters known;
    RunsParams shared = q;
    shared.split = ctas_that_fit(kernel, q.split, THREADS, kRunsSmem, known);
    if (shared.split == 1) return launch_mode<BNMAX, PAIR, MODE, false>(shared, smem, stream);
    return launch_after_previous(kernel, shared.nwork * shared.split, shared.split, THREADS, smem, stream, shared);
  }
  const int most = PAIR ? 74 : 148, grid = (q.nwork < most ? q.nwork : most) * (PAIR ? 2 : 1);
  return launch_after_previous(kernel, grid, PAIR ? 2 : 1, THREADS, smem, stream, q);
}

template <int BNMAX, bool PAIR, bool SPLIT>
cudaError_t launch_form(int mode, const RunsParams& q, int smem, cudaStream_t stream) {
  if (mode == HALVES) return launch_mode<BNMAX, PAIR, HALVES, SPLIT>(q, smem, stream);
  if (mode == WORDS) return launch_mode<BNMAX, PAIR, WORDS, SPLIT>(q, smem, stream);
  if (mode == ROW_PAIRS) return launch_mode<BNMAX, PAIR, ROW_PAIRS, SPLIT>(q, smem, stream);
  return launch_mode<BNMAX, PAIR, UNITS, SPLIT>(q, smem, stream);
}

template <int BNMAX>
cudaError_t launch_single(int mode, const RunsParams& q, int smem, cudaStream_t stream) {
  return q.split > 1 ? launch_form<BNMAX, false, true>(mode, q, smem, stream) : launch_form<BNMAX, false, false>(mode, q, smem, stream);
}

}  // namespace

// The window tensor in rows of p.planes channel planes, 8-byte elements (a box may be 256 of them wide).
static bool encode_window_rows(CUtensorMap* map, const uint16_t* window, const Geometry& g, const RunsPlan& p) {
  typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                    const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeTiledFn encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess)
      return false;
    encode = reinterpret_cast<EncodeTiledFn>(fn);
  }
  const cuuint64_t row = (cuuint64_t)p.planes * g.chan_stride * ES;
  const cuuint64_t dims[2] = {row / 8, (cuuint64_t)g.N * g.C / p.planes}, strides[1] = {row};
  const cuuint32_t box[2] = {(cuuint32_t)(p.region / 8), (cuuint32_t)(8 / p.planes)}, ones[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<uint16_t*>(window), dims, strides, box, ones,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Channels of the octets that a k2-block (8 units) can touch: what a block of the pack kernel stages.
static int64_t pack_channels(int64_t E, int C) {
  const int64_t n = ((8 + E - 2) / E + 1) * 8;
  return n < C ? n : C;
}

// CTAs of a cluster that share the k2-blocks of a tile, where there are so few tiles that an SM each is left for them: a k2-block
// takes 1 us, meeting and adding up 1 us and 0.02 for each channel of a tile (fitted to 33 such layers with 1 to 16 CTAs; the choice is
// within 0.7 % of the best on average, 9 % at the most).  Alone / split, us: 3x3 stride 2 on 512 -> 128 channels at 15x15, batch 27, 57 /
// 20; 5x5 stride 2 on 128 channels at 39x39 29 / 12; 3x3 on 64 -> 104 channels at 50x50 (5 k2-blocks) 9.2 either way.
// The tiles are those of the batch these images belong to: they decide the order of the sums.
static int choose_split(const Geometry& g, const RunsPlan& p) {
  // testing aid: CTAs per tile (1 where the kernel is forced and this is not)
  if (const char* v = debug_getenv("IM2WIN_F16_SPLIT")) return atoi(v) < p.num_kb ? atoi(v) : p.num_kb;
  if (debug_getenv("IM2WIN_F16_KERNEL")) return 1;
  const int64_t tiles = ((int64_t)g.plan_N * g.Ho * p.Wq + TILE_M - 1) / TILE_M * p.ntn;
  if (tiles > 74 || g.K > kMostSplitTerms) return 1;
  int split = 1;
  double best = p.num_kb;
  for (int z = 2; z <= kMaxCtas && z <= p.num_kb; ++z) {
    if (tiles * z > 148 || tiles > resident_clusters(z)) continue;
    const double cost = 1.0 + 0.02 * p.bn + (p.num_kb + z - 1) / z + 0.05 * z;
    if (cost < best) { best = cost; split = z; }
  }
  return split;
}

RunsPlan plan_f16_runs(const Geometry& g) {
  RunsPlan p{};
  p.eligible = false;
  const int nsub = g.s < g.Kw ? g.s : g.Kw;
  const int64_t E = (int64_t)nsub * g.Kh;
  if (E > 256 || (int64_t)g.C * E > (1 << 20) || g.chan_stride >= ((int64_t)1 << 30)) return p;
  if (pack_channels(E, g.C) * g.T * ES > 48 * 1024) return p;          // staging of the filter pack
  p.E = (int32_t)E;
  p.G = (g.Kw + g.s - 1) / g.s;
  p.quad = g.C <= 4;
  p.octs = (int32_t)(E >= 3 ? 1 : (E == 2 ? 2 : 4));
  const bool words = E % 2 == 0 && g.s * g.Kh % 2 == 0 && (int64_t)g.Wp * g.Kh % 2 == 0 && (p.G - 1) * group_of(WORDS) <= 32;
  const bool pairs = E == 3 && g.s == 1 && (int64_t)g.Ho * g.Wp % 2 == 0;
  p.mode = words ? WORDS : (pairs ? ROW_PAIRS : HALVES);
  p.units = (int32_t)(p.quad ? (E + 1) / 2 : (g.C + 7) / 8 * E);
  p.num_kb = (p.units + 7) / 8;
  p.nks_last = (p.units - 8 * (p.num_kb - 1) + 1) / 2;
  p.halo = p.G - 1;
  if (p.halo > 31) return p;                                // (one lane per row below the tile)
  p.Wq = (g.Wp + g.s - 1) / g.s;
  p.VQ = (int64_t)g.N * g.Ho * p.Wq;
  if (p.VQ + 2 * TILE_M >= ((int64_t)1 << 31)) return p;
  p.rows = TILE_M + (p.halo + 7) / 8 * 8;
  p.a_stage = p.rows * 128;
  const int64_t per_img = (int64_t)g.Ho * p.Wq;
  const int64_t segs = (TILE_M + p.halo - 2) / per_img + 2;
  if (segs > MAX_SEG) return p;
  // bytes a tile's columns of one channel take in a raw slot, whatever the tile
  const int64_t region = (int64_t)(TILE_M + p.halo) * g.s * g.Kh * ES + segs * 32;
  p.region = (int32_t)((region + 15) / 16 * 16);
  p.ntn = (g.Co + 255) / 256;
  p.bn = ((g.Co + p.ntn - 1) / p.ntn + 15) / 16 * 16;
  p.ntn = (g.Co + p.bn - 1) / p.bn;
  const int64_t ntm = (p.VQ + TILE_M - 1) / TILE_M;
  if (ntm * p.ntn >= ((int64_t)1 << 30)) return p;
  // CTA pairs above 128 channels: each CTA stages its own position tile and half of the filter.  The shared-memory pipe bounds
  // those tiles (an instruction of N = 256 reads 12 KB of operands in 128 cycles, one of a pair 8 KB an SM), and the
  // filter's copies, twice the bytes of all else, halve.
  // (Not for the shortest reductions, which setting up and meeting makes longer: 1.05 to 1.16 times with up to 128 k2 on 15 layers,
  // 0.92 to 1.15 with up to 256 on 13.  N of a pair's instruction: a multiple of 32.  Wider tiles for the others would want more scratch)
  p.pair = p.bn > 128 && p.bn % 32 == 0 && ntm > 1 && p.num_kb * p.G >= 8;
  if (const char* v = debug_getenv("IM2WIN_F16_PAIR")) p.pair = p.pair && v[0] != '0';     // testing aid
  p.split = choose_split(g, p);
  p.pair = p.pair && p.split == 1;
  p.ntm = (int32_t)ntm;
  p.nwork = (int32_t)((p.pair ? (ntm + 1) / 2 : ntm) * p.ntn);
  const int budget = kRunsSmem - 1024;
  // A raw slot holds whole octets, at least three units; rings of two S stages, four slots (else two) and the filter:
  // resident where one channel tile's fits, else two slots of all (up to three) kernel columns of a k2-block, so that the MMA
  // warp waits and commits once a k2-block, else at least three of one column.
  int64_t raw = ((p.quad ? 4 : 8 * p.octs) * (int64_t)p.region + 127) / 128 * 128;
  // Layers whose whole filter columns and bulk copies would not fit stay out, also where a pair's halves would: their scratch is
  // not sized for this kernel's filter.
  const int columns = p.num_kb * p.G, fewest = p.ntn == 1 && columns < 3 ? columns : 3;
  if (2 * (int64_t)p.a_stage + (int64_t)fewest * p.bn * 128 + 2 * raw > budget) return p;
  // Raw copies.  A bulk copy takes the copy engine 100 to 130 cycles whatever its size (3x3 on 64 channels at 56x56: 86 of 109 us
  // with all else left out), a tiled one that brings 8 / planes channels at once hardly more; `planes` channel planes are a
  // multiple of 16 bytes.  A box is as wide as a whole tile's columns, for every image of the tile: two images at most.
  p.planes = 1;
  while (p.planes < 8 && (p.planes * g.chan_stride * ES) % 16 != 0) p.planes *= 2;
  // (every box starts on 128 bytes of shared memory: its 8 / planes rows are a multiple of that)
  const int64_t wide = (int64_t)(TILE_M + p.halo) * g.s * g.Kh * ES + 15;
  const int64_t box = (wide + 16 * p.planes - 1) / (16 * p.planes) * (16 * p.planes);
  if (p.planes == 8 || p.quad || g.C % p.planes != 0 || box > 2048 || segs > 2 || segs * p.octs * p.planes > 32 ||
      (int64_t)g.N * g.C >= ((int64_t)1 << 31))
    p.planes = 0;
  if (const char* v = debug_getenv("IM2WIN_F16_RUNS_TILED")) if (v[0] == '0') p.planes = 0;           // testing aid
  const int64_t tiled_raw = segs * p.octs * 8 * box;
  if (2 * (int64_t)p.a_stage + 3 * (int64_t)(p.pair ? p.bn / 2 : p.bn) * 128 + 4 * ((tiled_raw + 127) / 128 * 128) > budget) p.planes = 0;
  if (p.planes) {
    p.region = (int32_t)box;
    p.seg_bytes = (int32_t)(p.octs * 8 * box);
    raw = (tiled_raw + 127) / 128 * 128;
  }
  for (int pass = 0; pass < 6 && !p.eligible; ++pass) {
    const int kind = pass % 3;                               // resident, whole k2-blocks, columns
    p.cols = kind < 2 && p.G <= 3 ? p.G : 1;
    p.slot_bytes = p.cols * (p.pair ? p.bn / 2 : p.bn) * 128;
    const int units = p.num_kb * p.G / p.cols;
    const bool resident = kind == 0 && p.ntn == 1 && units <= MAX_B;
    if (kind == 0 && !resident) continue;
    if (kind == 1 && p.cols == 1) continue;
    const int least_raw = pass < 3 ? 4 : 2, least_b = resident ? units : (kind == 1 ? 2 : 3);
    if (2 * (int64_t)p.a_stage + (int64_t)least_b * p.slot_bytes + least_raw * raw > budget) continue;
    p.raw_slot = (int32_t)raw;
    p.resident = resident;
    p.sa = 2; p.sr = least_raw; p.sb = least_b;
    auto fits = [&](int a, int r, int b) { return (int64_t)a * p.a_stage + (int64_t)r * raw + (int64_t)b * p.slot_bytes <= budget; };
    if (!resident && p.sb < 3 && fits(p.sa, p.sr, 3)) p.sb = 3;
    if (fits(3, p.sr, p.sb)) p.sa = 3;                       // (before a fourth filter slot: 120 -> 107 us on a pair's tiles)
    if (!resident) while (p.sb < 4 && fits(p.sa, p.sr, p.sb + 1)) ++p.sb;
    p.teams = p.mode == ROW_PAIRS && p.sr == 4 ? 4 : 2;
    // (even: the two copy warps alternate; a multiple of the teams, see stage_tiles.  Four teams on four slots against three on
    // six: 3x3 on 256 channels at 28x28, batch 64, 61 and 68 us, 64 -> 128 channels at 112x112 220 and 246)
    while (p.sr + p.teams <= MAX_RAW && fits(p.sa, p.sr + p.teams, p.sb)) p.sr += p.teams;
    if (!resident) while (p.sb < MAX_B && fits(p.sa, p.sr, p.sb + 1)) ++p.sb;
    p.eligible = true;
  }
  // Teams or unit by unit, measured both ways on 750 layers (time of the teams / unit by unit): rows in pairs 0.70 to 1.05, words of
  // two 0.75 to 1.07; by single elements 0.97 for columns of 3, 6 and 9, 1.02 to 1.16 for one element and the numbers that three
  // does not divide, 0.85 to 1.13 above nine.  1.05 to 1.1 with up to two slots in a tile, 1.1 to 1.4 with rings of one for each team.
  const int slots = ((g.C + 7) / 8 + p.octs - 1) / p.octs;
  bool by_units = slots <= 2 || p.sr == 2 || E <= 2 || (p.mode == HALVES && (E % 3 != 0 || E > 9));
  if (const char* v = debug_getenv("IM2WIN_F16_RUNS_UNITS")) by_units = v[0] != '0';       // testing aid
  if (by_units || p.quad || p.halo * group_of(p.mode) > 32) { p.mode = UNITS; p.teams = 1; }
  p.filter_bytes = (size_t)p.ntn * p.bn * p.num_kb * KB * p.G * 2;
  return p;
}

cudaError_t launch_pack_f16_runs(const uint16_t* filter, void* scratch, const Geometry& g, cudaStream_t stream) {
  const RunsPlan p = plan_f16_runs(g);
  if (!p.eligible) return cudaErrorInvalidValue;
  unsigned char* base = static_cast<unsigned char*>(scratch);
  const int64_t pitch = pack_channels(p.E, g.C) * g.T;
  // Channels per block: staging within 40 KB, and two blocks an SM where the filter has them (a block's channels are loaded one
  // after another, a round trip each: 3x3 on 64 -> 64 channels in 24 blocks took as long as ten times the filter)
  int rows = 8;
  while (rows > 1 && (rows * pitch * ES > 40 * 1024 || (int64_t)p.ntn * p.bn / rows * p.num_kb < 2 * 148)) rows /= 2;
  const size_t smem = (size_t)(rows * pitch * ES);
  dim3 grid((unsigned)(p.ntn * p.bn / rows), (unsigned)p.num_kb);   // (num_kb <= 2^14: C * E <= 2^20)
  return launch_pack<pack_f16_runs_kernel>(grid, 256, smem, stream, filter, base + kStatusBytes, reinterpret_cast<uint32_t*>(base), g.C, g.Kh, g.Kw,
                                                    g.s, p.E, p.G, g.Co, p.bn, p.num_kb, rows, (int)pitch, p.quad);
}

cudaError_t launch_conv_f16_runs(const uint16_t* window, float* y, void* scratch, const Geometry& g, cudaStream_t stream) {
  const RunsPlan p = plan_f16_runs(g);
  if (!p.eligible) return cudaErrorInvalidValue;
  unsigned char* base = static_cast<unsigned char*>(scratch);
  RunsParams q;
  q.win = reinterpret_cast<const unsigned char*>(window);
  q.fp = base + kStatusBytes;
  q.y = y;
  q.status = reinterpret_cast<uint32_t*>(base);
  q.img_bytes = g.img_stride * ES; q.chan_bytes = g.chan_stride * ES; q.win_bytes = g.window_elems * ES;
  q.VQ = (uint32_t)p.VQ;
  q.div_wq = fast_div((uint32_t)p.Wq);
  q.div_ho = fast_div((uint32_t)g.Ho);
  q.C = g.C; q.Wp = g.Wp; q.Wq = p.Wq; q.Ho = g.Ho; q.Wo = g.Wo; q.HoWo = g.Ho * g.Wo;
  q.Co = g.Co; q.Kh = g.Kh; q.Kw = g.Kw; q.s = g.s;
  // kernel columns beyond Kw, channels beyond C in the last octet, the element beyond an odd E
  q.foreign = (g.Kw > g.s && g.Kw % g.s != 0) || (p.quad ? p.E % 2 != 0 : g.C % 8 != 0);
  q.teams = p.teams;
  q.E = p.E; q.G = p.G; q.units = p.units; q.quad = p.quad ? 1 : 0; q.num_kb = p.num_kb; q.nks_last = p.nks_last;
  q.halo = p.halo; q.region = p.region; q.octs = p.octs; q.raw_slot = p.raw_slot; q.a_stage = p.a_stage;
  q.bn = p.bn; q.ntn = p.ntn; q.nwork = p.nwork; q.sa = p.sa; q.sr = p.sr; q.sb = p.sb;
  q.planes = p.planes; q.seg_bytes = p.seg_bytes;
  if (p.planes) {
    if (!encode_window_rows(&q.map, window, g, p)) return cudaErrorInvalidValue;
  }
  q.slot_bytes = p.slot_bytes; q.cols = p.cols; q.ntm = p.ntm; q.resident = p.resident ? 1 : 0;
  q.split = p.split;
  int smem = 1024 + p.sa * p.a_stage + p.sb * p.slot_bytes + p.sr * p.raw_slot;
  if (p.split > 1 && smem < 1024 + cluster_sums_bytes(p.bn)) smem = 1024 + cluster_sums_bytes(p.bn);
  if (p.bn <= 64) return launch_single<64>(p.mode, q, smem, stream);
  if (p.bn <= 128) return launch_single<128>(p.mode, q, smem, stream);
  return p.pair ? launch_form<256, true, false>(p.mode, q, smem, stream) : launch_single<256>(p.mode, q, smem, stream);
}

}  // namespace im2win
