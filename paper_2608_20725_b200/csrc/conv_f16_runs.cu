// fp16-input / fp32-accumulate im2win convolution with the window tensor brought in as contiguous runs.  It needs no
// alignment of planes, strips or images and takes every stride: the layers whose plane pitch is no multiple of 16
// bytes, which conv_f16_mat.cu and conv_f16_raw.cu cannot bring in with tiled copies.
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
// Staging.  The columns a tile needs of one channel are one contiguous run per image it touches: an untiled bulk
// copy from the 16-byte boundary below to the one above brings it into a ring of raw slots (`octs` octets of
// channels each).  Two warpgroups take the units in turn, read the elements of their rows back (thread = row) and
// write the units of S.  Gathering with 2-byte global loads instead (conv_f16_shift.cu) makes every load instruction
// touch 32 rows s*Kh elements apart: three or more L1 wavefronts each, and a round trip to memory per batch.
//
// What bounds it: the staging warps' read-back (without it 89 us where the whole takes 107) and the shared-memory pipe,
// which carries the MMA's operand reads (32 + N/4 cycles per instruction of M = 128, K = 16), the copies, the read-back
// and the S stores.  Measured against the gathering kernel: 3x3 stride 2 on 256 -> 512 channels at 28x28, batch 128,
// 140 -> 115 us (515 TFLOP/s); 5x5 stride 2 on 37 -> 75 channels at 45x61, batch 13, 27 -> 17 us.  Eight staging warps and
// not sixteen (128 us): more of them take issue slots from the MMA warp.
#include <cuda_fp16.h>
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

struct RunsParams {
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
};

__device__ __forceinline__ uint32_t ld_shared_u16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
  return v;
}
constexpr int ES = 2;                         // bytes of an element
constexpr int REGS_STAGING = 80, REGS_MISC = 64, REGS_EPILOGUE = 128;   // 2*80 + 64 + 2*128 = 5*96

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

// The outputs y[i * ystride], i < count <= 16, that came out infinite or NaN although a zero filter element may have met an
// infinity or NaN from outside their window (RunsParams::foreign): in fp32 FMAs, k ascending, from the window at x and
// rows i of the filter image at f.  Sixteen sums at a time keep the loads of the filter (the same address in every lane) in
// flight; they end early once all are NaN.  (A function of its own: expanded beside the epilogue it costs spills.)
__device__ __noinline__ void exact_outputs(const unsigned char* __restrict__ x, const unsigned char* __restrict__ f, float* y,
                                           int64_t ystride, int64_t chan_bytes, int C, int Kh, int Kw, int s, int E, int g_step,
                                           int j_step, int quad, int count) {
  auto not_finite = [](float v) { return !(fabsf(v) <= 3.4028234663852886e38f); };
  bool any = false;
  for (int i = 0; i < count; ++i) any |= not_finite(y[i * ystride]);
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
    if (i < count && not_finite(*p)) *p = acc[i];
  }
}

// The MMAs of one kernel column, straight-line: a lone lane pays for every branch and address computation between them.
template <int NKS>
__device__ __forceinline__ void issue_column(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t more) {
#pragma unroll
  for (int j = 0; j < NKS; ++j) umma_f16_lohi(d, a + 2 * j, b + 2 * j, idesc, j == 0 ? more : 1u);
}

template <int BNMAX>
__global__ void __launch_bounds__(THREADS, 1) conv_f16_runs_kernel(RunsParams q) {
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

  if (threadIdx.x == 0) {
    abort_flag = 0u;
    for (int i = 0; i < MAX_A; ++i) { mbar_init(a_full0 + 8 * i, STAGING_WARPS); mbar_init(a_empty0 + 8 * i, 1); }
    for (int i = 0; i < MAX_RAW; ++i) { mbar_init(raw_full0 + 8 * i, 1); mbar_init(raw_empty0 + 8 * i, STAGING_WARPS); }
    for (int i = 0; i < MAX_B; ++i) { mbar_init(b_full0 + 8 * i, 1); mbar_init(b_empty0 + 8 * i, 1); }
    for (int i = 0; i < MAX_ACC; ++i) { mbar_init(acc_full0 + 8 * i, 1); mbar_init(acc_empty0 + 8 * i, 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == STAGING_WARPS) tmem_alloc(smem_u32(&tmem_base_slot), 512);
  // The raw ring starts as zeros: places no copy fills (channels beyond C in the last octet) meet zero filter
  // elements, but they have to be numbers.
  for (int i = threadIdx.x * 16; i < q.sr * q.raw_slot; i += THREADS * 16) st_shared16(raw_ring + i, 0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_acc = tmem_base_slot;
  wait_for_previous_kernel();

  if (warp < STAGING_WARPS) {
    // ---------------- staging: raw runs -> S ------------------------------------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_STAGING));
    // Warpgroup wg takes every second unit.  Every warp passes every stage and every slot in order, so
    // no wait by phase parity can run ahead.
    const int wg = warp >> 2, row = threadIdx.x & 127;
    const int plane = (q.Ho * q.Wp + q.Wq * q.s - q.Wp) * q.Kh;   // (up to the end of the last virtual column)
    const int per_slot = q.quad ? q.units : q.octs * q.E;
    const uint32_t oct_step = 8u * q.region - (uint32_t)(q.E - 1) * ES, unit_step = q.quad ? 2u * ES : ES;
    bool ok = true;
    int sa = 0, sr = 0;
    uint32_t pa = 0, pr = 0;
    for (int w = blockIdx.x; w < q.nwork && ok; w += gridDim.x) {
      const uint32_t q0 = (uint32_t)(w / q.ntn) * TILE_M;
      const TileRuns tr = tile_runs(q, q0);
      // Place of row r's first element in channel x of a slot's octet: byte inside the raw slot.
      auto locate = [&](int r, uint32_t (&rb)[8]) {
        uint32_t off = 0, phase = 0;
        const uint32_t vq = q0 + r;
        if (vq < q.VQ) {                                     // dead rows read whatever lies at the start: they are dropped
          uint32_t n;
          int ho, i;
          split_q(q, vq, n, ho, i);
          const int g = (int)(n - tr.n0), start = g == 0 ? tr.start0 : 0;
          if (g > 0) off = run_size(plane - tr.start0) + (g - 1) * run_size(plane);
          off += ((ho * q.Wp + i * q.s) * q.Kh - start) * ES;
          phase = (uint32_t)((int64_t)n * q.img_bytes + (int64_t)start * ES);
        }
#pragma unroll
        for (int x = 0; x < 8; ++x) rb[x] = off + x * q.region + ((phase + (uint32_t)x * (uint32_t)q.chan_bytes) & 15u);
        if (q.quad) {
#pragma unroll
          for (int x = 0; x < 4; ++x) rb[4 + x] = rb[x] + ES;
        }
      };
      uint32_t rb[8], hb[8];
      locate(row, rb);
      if (lane < q.halo) locate(TILE_M + lane, hb);
      uint32_t src = 0;                                      // of the current unit; inside the slot: its number, and its e
      int in_slot = 0, e = 0;
      for (int kb = 0; kb < q.num_kb && ok; ++kb) {
        ok = mbar_wait(a_empty0 + 8 * sa, pa ^ 1u, &abort_flag, q.status);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const uint32_t stage = a_ring + sa * q.a_stage;
        const int n_units = q.units - 8 * kb < 8 ? q.units - 8 * kb : 8;
        for (int ch = 0; ch < n_units; ++ch) {
          if (in_slot == 0) {
            ok = mbar_wait(raw_full0 + 8 * sr, pr, &abort_flag, q.status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            src = raw_ring + sr * q.raw_slot;
            e = 0;
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
          if (++in_slot == per_slot || 8 * kb + ch == q.units - 1) {
            __syncwarp();
            if (lane == 0) mbar_arrive(raw_empty0 + 8 * sr);
            if (++sr == q.sr) { sr = 0; pr ^= 1u; }
            in_slot = 0;
          }
          ++e;
          src += e == q.E ? oct_step : unit_step;
          if (e == q.E) e = 0;
        }
        if (!ok) break;
        if ((n_units & 1) != 0 && wg == 1) {                 // zeros up to the end of the MMA's last step
          st_shared16(stage + row * 128 + ((n_units ^ (row & 7)) << 4), 0u, 0u, 0u, 0u);
          if (lane < q.halo) st_shared16(stage + (TILE_M + lane) * 128 + ((n_units ^ (lane & 7)) << 4), 0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(a_full0 + 8 * sa);
        if (++sa == q.sa) { sa = 0; pa ^= 1u; }
      }
    }
  } else if (warp < STAGING_WARPS + 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_MISC));
    if (warp == STAGING_WARPS) {
      // ---------------- MMA issuer -----------------------------------------------------------------------
      const bool leader = elect_one();
      const uint32_t a_lo0 = smem_desc_lo(a_ring), b_lo0 = smem_desc_lo(b_ring);
      const uint32_t idesc = instr_desc_f16(TILE_M, q.bn);
      bool ok = true;
      int sa = 0, slot = 0;
      uint32_t pa = 0, pb = 0, ac = 0;                       // ... tiles so far
      // A wait for a barrier that is already complete costs 200 cycles and more while the shared-memory pipe is busy, and
      // the tensor pipe runs dry meanwhile: every barrier is looked at ahead of the instructions issued before it is
      // needed, and waited for only where that look came too early.
      uint32_t a_seen = 0, b_seen = 0, acc_seen = 0;
      // (testing aid: the commit of the first tile left out; looked up while its first stage is on its way)
      uint32_t drop = blockIdx.x == 0 ? *reinterpret_cast<volatile uint32_t*>(q.status + 2) : 0u;
      auto need = [&](uint32_t bar, uint32_t parity, uint32_t seen) {
        return mbar_wait_unless_seen(bar, parity, seen, &abort_flag, q.status);
      };
      for (int w = blockIdx.x; w < q.nwork && ok; w += gridDim.x, ++ac) {
        const int ab = ac & (NACC - 1);
        ok = need(acc_empty0 + 8 * ab, ((ac >> ACC_LOG) & 1) ^ 1, acc_seen);
        if (!ok) break;
        const uint32_t d = tmem_acc + ab * BNMAX;
        uint32_t more = 0u;                                  // the tile's first instruction clears the accumulator
        const bool fetch_b = !q.resident || w == (int)blockIdx.x;          // (a resident filter is complete after the first tile)
        if (q.resident) slot = 0;
        for (int kb = 0; kb < q.num_kb && ok; ++kb) {
          const int nks = kb == q.num_kb - 1 ? q.nks_last : KB / 16;
          ok = need(a_full0 + 8 * sa, pa, a_seen);
          if (!ok) break;
          tc_fence_after();
          uint32_t a_view = a_lo0 + (uint32_t)(sa * (q.a_stage >> 4));
          int nsa = sa + 1;
          uint32_t npa = pa;
          if (nsa == q.sa) { nsa = 0; npa ^= 1u; }
          for (int g = 0; g < q.G; ++g, a_view += 8u) {      // next view: one row (128 bytes) further down
            const bool last_unit = g + 1 == q.G, last = kb + 1 == q.num_kb && last_unit;
            int nslot = slot + 1;
            uint32_t npb = pb;
            if (nslot == q.sb) { nslot = 0; if (!q.resident) npb ^= 1u; }
            if (fetch_b) {
              ok = need(b_full0 + 8 * slot, pb, b_seen);
              if (!ok) break;
              b_seen = mbar_test_wait(b_full0 + 8 * nslot, npb);
            }
            if (last) acc_seen = mbar_test_wait(acc_empty0 + 8 * ((ac + 1) & (NACC - 1)), (((ac + 1) >> ACC_LOG) & 1) ^ 1);
            if (last_unit) a_seen = mbar_test_wait(a_full0 + 8 * nsa, npa);
            const uint32_t b_lo = b_lo0 + (uint32_t)(slot * (q.slot_bytes >> 4));
            if (leader) {
              if (nks == KB / 16) issue_column<KB / 16>(d, a_view, b_lo, idesc, more);
              else if (nks == 3) issue_column<3>(d, a_view, b_lo, idesc, more);
              else if (nks == 2) issue_column<2>(d, a_view, b_lo, idesc, more);
              else issue_column<1>(d, a_view, b_lo, idesc, more);
              if (!q.resident) umma_commit(b_empty0 + 8 * slot);
              if (last && drop != kDebugDropArrive) umma_commit(acc_full0 + 8 * ab);
              if (last_unit) umma_commit(a_empty0 + 8 * sa);
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
    } else if (warp == STAGING_WARPS + 1) {
      // ---------------- filter copies ----------------------------------------------------------------------
      const bool leader = elect_one();
      bool ok = true;
      int slot = 0;
      uint32_t pb = 0;
      for (int w = blockIdx.x; w < q.nwork && ok; w += gridDim.x) {
        const unsigned char* src = q.fp + (int64_t)(w % q.ntn) * q.num_kb * q.G * q.slot_bytes;
        for (int u = 0; u < q.num_kb * q.G; ++u, src += q.slot_bytes) {
          ok = mbar_wait(b_empty0 + 8 * slot, pb ^ 1u, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (leader) {
            mbar_arrive_expect_tx(b_full0 + 8 * slot, (uint32_t)q.slot_bytes);
            bulk_load(b_ring + slot * q.slot_bytes, src, (uint32_t)q.slot_bytes, b_full0 + 8 * slot);
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
      const int per_slot = q.quad ? 4 : 8 * q.octs, nslots = q.quad ? 1 : (q.C + per_slot - 1) / per_slot;
      for (int w = blockIdx.x; w < q.nwork && ok; w += gridDim.x) {
        const TileRuns tr = tile_runs(q, (uint32_t)(w / q.ntn) * TILE_M);
        const int nseg = (int)(tr.n1 - tr.n0) + 1;
        for (int sl = 0; sl < nslots; ++sl, ++sc) {
          if (sc & 1) {
            if (++sr == q.sr) { sr = 0; pr ^= 1u; }
            continue;
          }
          ok = mbar_wait(raw_empty0 + 8 * sr, pr ^ 1u, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
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
    for (int w = blockIdx.x; w < q.nwork && ok; w += gridDim.x) {
      const int mt = w / q.ntn, nt = w - mt * q.ntn;
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
#pragma unroll 1
      for (int c0 = h * (BNMAX / 2); c0 < (h + 1) * (BNMAX / 2) && c0 < limit; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(d + c0, v);
        if (c0 + 32 >= (h + 1) * (BNMAX / 2) || c0 + 32 >= limit) {      // the last read of this accumulator
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty0 + 8 * ab);
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
            const unsigned char* f = q.fp + (int64_t)nt * q.num_kb * q.G * q.slot_bytes;
            for (int c = c0; c < c0 + 32 && c < limit; c += 16)
              exact_outputs(x, f + c * 128, yrow + (int64_t)c * q.HoWo, q.HoWo, q.chan_bytes, q.C, q.Kh, q.Kw, q.s, q.E,
                            q.slot_bytes, q.G * q.slot_bytes, q.quad, limit - c < 16 ? limit - c : 16);
          }
        }
      }
      if (h * (BNMAX / 2) >= limit) {                      // (no channels for this warp)
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty0 + 8 * ab);
      }
    }
  }

  // ---------------- teardown -----------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (abort_flag) {
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == STAGING_WARPS) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_acc, 512);
  }
}

// Filter -> the images the copy warp loads: for every (channel tile nt, k2-block kb, virtual kernel column g) the
// [bn channels][64 k2] in the 128-byte-swizzled order of shared memory.  One block: `rows` channels of one k2-block; per channel its source is one contiguous run of the OIHW
// filter (whole input channels).  Channels beyond Co, k2 beyond C*E and kernel columns beyond Kw are zeros.
__global__ void __launch_bounds__(256) pack_f16_runs_kernel(const uint16_t* __restrict__ f, unsigned char* __restrict__ fp,
                                                        uint32_t* __restrict__ status, int C, int Kh, int Kw, int s, int E, int G,
                                                        int Co, int bn, int num_kb, int rows, int pitch, int quad) {
  extern __shared__ uint16_t pack_h[];
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

template <int BNMAX>
cudaError_t launch_form(const RunsParams& q, int smem, cudaStream_t stream) {
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(conv_f16_runs_kernel<BNMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRunsSmem);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  return launch_after_previous(conv_f16_runs_kernel<BNMAX>, q.nwork < 148 ? q.nwork : 148, 1, THREADS, smem, stream, q);
}

}  // namespace

// Channels of the octets that a k2-block (8 units) can touch: what a block of the pack kernel stages.
static int64_t pack_channels(int64_t E, int C) {
  const int64_t n = ((8 + E - 2) / E + 1) * 8;
  return n < C ? n : C;
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
  p.slot_bytes = p.bn * 128;
  const int64_t ntm = (p.VQ + TILE_M - 1) / TILE_M;
  if (ntm * p.ntn >= ((int64_t)1 << 30)) return p;
  p.nwork = (int32_t)(ntm * p.ntn);
  const int units = p.num_kb * p.G;
  const int budget = kRunsSmem - 1024;
  // A raw slot holds whole octets, at least three units; rings of two S stages, four slots (else two)
  // and the filter (resident where one channel tile's fits, else at least three units).
  p.octs = (int32_t)(E >= 3 ? 1 : (E == 2 ? 2 : 4));
  const int64_t raw = ((p.quad ? 4 : 8 * p.octs) * (int64_t)p.region + 127) / 128 * 128;
  for (int pass = 0; pass < 4 && !p.eligible; ++pass) {
    const bool resident = (pass & 1) == 0 && p.ntn == 1 && units <= MAX_B;
    if ((pass & 1) == 0 && !resident) continue;
    const int least_raw = pass < 2 ? 4 : 2, least_b = resident ? units : 3;
    if (2 * p.a_stage + least_b * p.slot_bytes + least_raw * raw > budget) continue;
    p.raw_slot = (int32_t)raw;
    p.resident = resident;
    p.sa = 2; p.sr = least_raw; p.sb = least_b;
    auto fits = [&](int a, int r, int b) { return (int64_t)a * p.a_stage + (int64_t)r * raw + (int64_t)b * p.slot_bytes <= budget; };
    if (!resident) while (p.sb < 4 && fits(p.sa, p.sr, p.sb + 1)) ++p.sb;
    if (fits(3, p.sr, p.sb)) p.sa = 3;
    while (p.sr < MAX_RAW && fits(p.sa, p.sr + 2, p.sb)) p.sr += 2;   // (even: the two copy warps alternate)
    if (!resident) while (p.sb < MAX_B && fits(p.sa, p.sr, p.sb + 1)) ++p.sb;
    p.eligible = true;
  }
  p.filter_bytes = (size_t)p.ntn * p.bn * p.num_kb * KB * p.G * 2;
  return p;
}

cudaError_t launch_pack_f16_runs(const uint16_t* filter, void* scratch, const Geometry& g, cudaStream_t stream) {
  const RunsPlan p = plan_f16_runs(g);
  if (!p.eligible) return cudaErrorInvalidValue;
  unsigned char* base = static_cast<unsigned char*>(scratch);
  const int64_t pitch = pack_channels(p.E, g.C) * g.T;
  int rows = 8;                                             // channels per block: staging within 40 KB
  while (rows > 1 && rows * pitch * ES > 40 * 1024) rows /= 2;
  const size_t smem = (size_t)(rows * pitch * ES);
  dim3 grid((unsigned)(p.ntn * p.bn / rows), (unsigned)p.num_kb);   // (num_kb <= 2^14: C * E <= 2^20)
  pack_f16_runs_kernel<<<grid, 256, smem, stream>>>(filter, base + kStatusBytes, reinterpret_cast<uint32_t*>(base), g.C, g.Kh, g.Kw,
                                                    g.s, p.E, p.G, g.Co, p.bn, p.num_kb, rows, (int)pitch, p.quad);
  return cudaGetLastError();
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
  q.E = p.E; q.G = p.G; q.units = p.units; q.quad = p.quad ? 1 : 0; q.num_kb = p.num_kb; q.nks_last = p.nks_last;
  q.halo = p.halo; q.region = p.region; q.octs = p.octs; q.raw_slot = p.raw_slot; q.a_stage = p.a_stage;
  q.bn = p.bn; q.ntn = p.ntn; q.nwork = p.nwork; q.sa = p.sa; q.sr = p.sr; q.sb = p.sb;
  q.slot_bytes = p.slot_bytes; q.resident = p.resident ? 1 : 0;
  const int smem = 1024 + p.sa * p.a_stage + p.sb * p.slot_bytes + p.sr * p.raw_slot;
  if (p.bn <= 64) return launch_form<64>(q, smem, stream);
  if (p.bn <= 128) return launch_form<128>(q, smem, stream);
  return launch_form<256>(q, smem, stream);
}

}  // namespace im2win
