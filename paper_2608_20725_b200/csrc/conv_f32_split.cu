// fp32 im2win convolution on the tensor cores: every fp32 operand is the exact sum of three bf16
// pieces, and six bf16 products per term reproduce the fp32 product.
//
//     2^23 x = x1 + x2 + x3,  x1 = bf16(2^23 x), x2 = bf16(2^23 x - x1), x3 = 2^23 x - x1 - x2   (24 = 8 + 8 + 8 bits)
//     2^46 x w ~ x1 w1 + (x1 w2 + x2 w1) + (x1 w3 + x2 w2 + x3 w1)
//
// The three products left out are below 2^-26 |x w|.  What decides the accuracy is the accumulator: the
// tensor core aligns the addends of an instruction to the largest one, cuts them two bits below fp32's
// last and truncates the sum (measured), so a long chain in one accumulator drifts towards zero.  A chain
// here is therefore short: the products of 64 k2 of one kernel column (a "unit") go into a fresh
// accumulator, the small products first, and the epilogue warps add it to fp32 registers with rounded adds.
// Error against 64 bits, relative 2-norm (round-to-nearest FFMA chain -> this kernel), inputs of both signs and of one:
// K = 147 2.2e-7 -> 0.9e-7, K = 576 4.4e-7 -> 1.8e-7 with the long chains of the narrow tiles (below) and 1.0e-7 without,
// K = 4608 1.1e-6 -> 1.7e-7 and 1.1e-7.
// The last bit of the smallest fp32 values, 2^-149, becomes bf16's smallest normal value, 2^-126, by the scaling: no piece
// of any operand gets lost, or is a subnormal (by whose exponent the tensor core would align its addends: scaled by
// 2^16, weights of 2^-145 gave six times the error).  Elements of 2^104 and sums of 2^82 and more give a non-finite
// accumulator; such outputs (and non-zero ones below 2^-90, whose products the FFMA kernel rounds to fp32's subnormals)
// are computed again with fp32 FMAs in the order of the FFMA kernel, from the window and a copy of the filter
// (exact_outputs).
//
// The GEMM is the shifted-view one of conv_f16_shift.cu: the window tensor's columns are staged once,
//     S[piece][row = virtual column q][k2 = c*Kh + u]     (64 k2 = 128 bytes per row, 128-byte swizzle),
// and kernel column v multiplies the view that starts (v div s) rows further down; with stride s a stage
// holds one column class t = v mod s.  Rows are the virtual positions q = (n*Ho + ho)*Wq + i, Wq = ceil(Wp/s).
//
// What bounds it: the tensor pipe on wide tiles, and next to it the shared-memory pipe the MMA reads its operands
// through: an instruction of M = 128, K = 16 takes max(N/2, 32 + N/4) cycles.  Up to 64 channels the filter
// pieces therefore lie side by side as one operand, [w1 | w2 | w3], and four instructions replace six: x1 against all
// of it into three accumulators (x1w1 | x1w2 | x1w3), and x2w1, x2w2 and x3w1 into a fourth, so that no accumulator holds
// the large products beside the small ones and a chain may take several units: `chain` steps of 16 k (12, or 8 on
// reductions below 288).  Instructions are promised to run in the order of their issue only where accumulator and shape
// are the same, so no accumulator is written under two shapes or from two starts.  (Without that, x2 against [w1 | w2]
// one accumulator further and x3 against w1 two further take 208 cycles a step at 64 channels; this 240, six 288.)
//
// Roles (one persistent CTA per SM): one or two warpgroups of producers (thread = row; 32 loads in flight,
// split, 16-byte stores), an MMA warp, a filter-copy warp (one untiled bulk copy per piece: the pack kernel
// writes shared-memory images), eight epilogue warps that keep the tile's fp32 sums in registers.
// Measured against the FFMA kernel (us, filter packed beforehand): 3x3 on 64 channels at 56x56, batch 128, 543 -> 195 (152
// TFLOP/s; no pipe above half of its rate: hand-offs over two stages); 3x3 on 512 channels at 7x7 627 -> 158; 11x11 on 256
// channels at 28x28, batch 64, 14824 -> 4143 in a long row, where the power limit decides (192 TFLOP/s; 1.5 PFLOP/s of bf16 products with
// the strip ends); 7x7 stride 2 on 3 channels at 224x224 642 -> 385.
// A layer with few tiles is run by clusters of 2 to 16 CTAs that share the stages of a tile and add their
// registers through distributed shared memory, in rank order: 3x3 on 512 channels, one 7x7 image, 225 -> 16 us.  Any number of CTAs
// whose clusters are all resident at once, sums pushed to the CTA that finishes them: against powers of two up to 8 and sums read from the
// other CTAs, 40 layers of 1 to 90 tiles 1.13 times as fast on average (0.91 at the least): 3x5 stride 2 on 427 channels at 66x12, batch 2,
// 35.8 -> 16.3 us, 7x7 on 256 -> 78 channels at 35x35, batch 2 (16 clusters of 8 in two rounds) 87 -> 47.
#include <cuda_bf16.h>
#include <stdlib.h>
#include <string.h>

#define IM2WIN_INLINE_SLOW_WAIT      // (a call cannot be compiled beside the 128 live sums of the epilogue warps)
#include "common.cuh"
#include "launch.cuh"
#include "ptx_sm100.cuh"

namespace im2win {
namespace {

using namespace ptx;

constexpr int TILE_M = 128;
constexpr int KB = 64;
constexpr int A_STAGES = 2;
constexpr int MAX_B = 16;
constexpr int MAX_ACC = 4;
constexpr int CONCAT_BN = 64;                 // channel tiles up to here: the filter pieces side by side in one operand
constexpr int kSplitSmem = 226 * 1024;        // dynamic shared memory a CTA may use

struct SplitParams {
  const float* __restrict__ win;
  const unsigned char* __restrict__ fp;       // packed filter: shared-memory images, see pack_f32_split_kernel
  const float* __restrict__ f;                // the filter as given, for exact_outputs
  float* __restrict__ y;
  uint32_t* status;
  int64_t img_stride, strip, chan_stride;
  uint32_t VQ;
  int32_t K2, C, Wq, Wp, Ho, Wo, HoWo, Co, Kh, Kw, s, nsub, num_kb, nks_last;
  int32_t rows, halo;                         // rows of a sub-tile (128 + halo rounded up to 8), halo
  int32_t bn, ntn, nwork, nstages, split, sb, slot_bytes, chain;
  int32_t n_main, parts;                      // tiles from n_main on are handed out in `parts` parts of their channels
};


// Work item w -> tile, first channel within it, channels.  The last round's tiles may go out in parts of their channels: no
// sum changes.  (Pieces that lie side by side have no parts: PARTS is false.)
struct Item {
  int tile, first, bn;
};
template <bool PARTS>
__device__ __forceinline__ Item work_item(const SplitParams& q, int w) {
  if (!PARTS || w < q.n_main) return {w, 0, q.bn};
  const int t = w - q.n_main, i = t / q.parts, bn = q.bn / q.parts;
  return {q.n_main + i, (t - i * q.parts) * bn, bn};
}

// (volatile: the loads of a batch stay together, ahead of the wait for the stage they are for; left to
// itself the compiler may move them to their uses, one round trip per eight loads)
__device__ __forceinline__ float ld_if(const float* p, bool ok) {
  float v = 0.f;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p ld.global.nc.f32 %0, [%1];\n\t}"
      : "+f"(v)
      : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// Two values -> the three pieces of 2^23 times them, packed (first value in the low half).
constexpr float kScale = 8388608.f, kUnscale = 1.f / (kScale * kScale);
__device__ __forceinline__ uint64_t pair(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
// a - (the two bf16 of p), exact here.
__device__ __forceinline__ uint64_t sub_pieces(uint64_t a, uint32_t p) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r)
      : "l"(pair(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u))), "l"(pair(-1.f, -1.f)), "l"(a));
  return r;
}
__device__ __forceinline__ uint32_t cvt_pair(uint64_t v) {
  return cvt_bf16x2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}
__device__ __forceinline__ void split2(float a, float b, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
  uint64_t v;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(pair(a, b)), "l"(pair(kScale, kScale)));
  p1 = cvt_pair(v);
  v = sub_pieces(v, p1);
  p2 = cvt_pair(v);
  p3 = cvt_pair(sub_pieces(v, p2));
}
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// The wait for loads into r[]: naming the registers keeps every use of them after it.
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
// bf16 operands, fp32 accumulator, both k-major.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// An output that has to be computed again: not finite, or so small that fp32 rounds its products.
__device__ __forceinline__ bool suspicious(float v) {
  const uint32_t u = __float_as_uint(v) << 1, lo = (uint32_t)(127 - 90) << 24;
  return u != 0u && u - lo >= 0xff000000u - lo;
}

// v[e] / 2^46 -> base[e * stride] for e < count, over two address chains.
__device__ __forceinline__ void store16(float* base, int stride, const float (&v)[16], int count, bool& again) {
  float *p0 = base, *p1 = base + stride;
  const int64_t step = 2 * (int64_t)stride;
#pragma unroll
  for (int e = 0; e < 16; e += 2) {
    const float a = v[e] * kUnscale, b = v[e + 1] * kUnscale;
    if (e < count) { *p0 = a; again |= suspicious(a); }
    if (e + 1 < count) { *p1 = b; again |= suspicious(b); }
    p0 += step; p1 += step;
  }
}

// PWG: producer warpgroups.  Two where a tile has several stages (3x3 on 64 channels at 56x56: 351 against 385 thousand
// cycles with one), one with a single stage per tile (7x7 stems: 412 against 472 us) and beside 128 sums a thread.
template <int BNMAX, int PWG_> struct Form {
  static constexpr int PWG = PWG_;
  static constexpr bool CONCAT = BNMAX == CONCAT_BN;
  static constexpr int ACC_COLS = CONCAT ? 4 * CONCAT_BN : BNMAX;   // tensor memory: a ring of accumulators (CONCAT: fours)
  static constexpr int NACC = 512 / ACC_COLS;
  static constexpr int ACC_LOG = BNMAX == 128 ? 2 : 1;
  static constexpr int CH = BNMAX / 32;                   // 16-channel chunks per epilogue warp
  static constexpr int THREADS = 128 * (PWG + 3);
  static constexpr int REGS_PRODUCER = 96;
  static constexpr int REGS_MISC = 64;
  static constexpr int REGS_EPILOGUE = PWG == 1 ? 176 : 112;
  // (the launch holds 128 or 96 registers a thread: 96 + 64 + 2*176 = 4*128, 2*96 + 64 + 2*112 = 5*96)
};

// The suspicious ones among the outputs y[i * ystride], i < count <= 16, of the window at x and the filters f + i * fstep:
// computed again in fp32 FMAs, k ascending.  Sixteen sums at a time share the loads of the window and keep the loads of
// the filter (the same address in every lane) in flight; they end early once all are NaN, as in a tensor full of them.
__device__ __noinline__ void exact_outputs(const float* __restrict__ x, const float* __restrict__ f, float* y, int64_t chan_stride,
                                           int64_t fstep, int64_t ystride, int C, int Kh, int Kw, int count) {
  bool any = false;
  for (int i = 0; i < count; ++i) any |= suspicious(y[i * ystride]);
  if (!any) return;
  float acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.f;
  bool open = true;
#pragma unroll 1
  for (int c = 0; c < C && open; ++c, x += chan_stride, f += Kh * Kw) {
#pragma unroll 1
    for (int v = 0; v < Kw; ++v)
#pragma unroll 1
      for (int u = 0; u < Kh; ++u) {
        const float xv = x[v * Kh + u];
        const float* fk = f + u * Kw + v;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          acc[i] = fmaf(xv, *fk, acc[i]);
          if (i + 1 < count) fk += fstep;
        }
      }
    open = false;
#pragma unroll
    for (int i = 0; i < 16; ++i) open |= acc[i] == acc[i];
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float* p = y + i * ystride;
    if (i < count && suspicious(*p)) *p = acc[i];
  }
}

// The instructions of one filter operand of a unit, straight-line: a lone lane pays for every branch and address
// computation between them.  CONCAT: the operand is [w1 | w2 | w3]; else it is piece 3 - p of the filter.
template <bool CONCAT, int NKS>
__device__ __forceinline__ void issue_steps(uint32_t d, uint32_t bn, uint32_t a, uint32_t sub_lo, uint32_t b, uint32_t id1,
                                            uint32_t id3, uint32_t more, int p) {
  if constexpr (CONCAT) {
    const uint32_t low = d + 3 * bn, b2 = b + 8 * bn;      // (w2: bn rows of 128 bytes further down)
#pragma unroll
    for (int j = 0; j < NKS; ++j) umma_f16_lohi(d, a + 2 * j, b + 2 * j, id3, j == 0 ? more : 1u);
#pragma unroll
    for (int j = 0; j < NKS; ++j) umma_f16_lohi(low, a + 2 * sub_lo + 2 * j, b + 2 * j, id1, j == 0 ? more : 1u);
#pragma unroll
    for (int j = 0; j < NKS; ++j) umma_f16_lohi(low, a + sub_lo + 2 * j, b2 + 2 * j, id1, 1u);
#pragma unroll
    for (int j = 0; j < NKS; ++j) umma_f16_lohi(low, a + sub_lo + 2 * j, b + 2 * j, id1, 1u);
  } else {
#pragma unroll
    for (int i = 2; i >= 0; --i) {
      if (i > p) continue;                                 // (p is a constant of the unrolled caller)
#pragma unroll
      for (int j = 0; j < NKS; ++j) umma_f16_lohi(d, a + i * sub_lo + 2 * j, b + 2 * j, id1, (uint32_t)(p | j));
    }
  }
}

template <int BNMAX, int PWG, bool SHARED>
__global__ void __launch_bounds__(Form<BNMAX, PWG>::THREADS, 1) conv_f32_split_kernel(SplitParams q) {
  using F = Form<BNMAX, PWG>;
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bars[2 * A_STAGES + 2 * MAX_B + 2 * MAX_ACC];
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile uint32_t abort_flag;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int wg = warp >> 2;
  const int sub_bytes = q.rows * 128, a_stage_bytes = 3 * sub_bytes;
  const uint32_t a_ring = smem_u32(smem);
  const uint32_t b_ring = a_ring + A_STAGES * a_stage_bytes;
  const uint32_t a_full0 = smem_u32(&bars[0]), a_empty0 = a_full0 + 8 * A_STAGES;
  const uint32_t b_full0 = a_empty0 + 8 * A_STAGES, b_empty0 = b_full0 + 8 * MAX_B;
  const uint32_t acc_full0 = b_empty0 + 8 * MAX_B, acc_empty0 = acc_full0 + 8 * MAX_ACC;
  int32_t* koff_s = reinterpret_cast<int32_t*>(smem + A_STAGES * a_stage_bytes + q.sb * q.slot_bytes);

  if (threadIdx.x == 0) {
    abort_flag = 0u;
    for (int i = 0; i < A_STAGES; ++i) { mbar_init(a_full0 + 8 * i, 4); mbar_init(a_empty0 + 8 * i, 1); }
    for (int i = 0; i < MAX_B; ++i) { mbar_init(b_full0 + 8 * i, 1); mbar_init(b_empty0 + 8 * i, 1); }
    for (int i = 0; i < MAX_ACC; ++i) { mbar_init(acc_full0 + 8 * i, 1); mbar_init(acc_empty0 + 8 * i, 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == F::PWG * 4 + 2) tmem_alloc(smem_u32(&tmem_base_slot), 512);
  // k2 -> element offset inside the image (channel plane and row of the kernel), -1 for padded k2
  for (int i = threadIdx.x; i < q.num_kb * KB; i += F::THREADS) {
    const int c = i / q.Kh;
    koff_s[i] = i < q.K2 ? (int32_t)(c * q.chan_stride + (i - c * q.Kh)) : -1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_acc = tmem_base_slot;
  wait_for_previous_kernel();

  // Work: tile w = position tile * channel tiles + channel tile.  Not SHARED: the CTA walks tiles w, w + grid, ...;
  // otherwise the cluster has one tile and its CTA r the stages [S r / split, S (r + 1) / split).
  const int rank = SHARED ? (int)cluster_ctarank() : 0;
  const int w_first = SHARED ? (int)blockIdx.x / q.split : (int)blockIdx.x;
  const int w_step = SHARED ? q.nwork : (int)gridDim.x;
  const int st0 = SHARED ? (int)((int64_t)q.nstages * rank / q.split) : 0;
  const int st1 = SHARED ? (int)((int64_t)q.nstages * (rank + 1) / q.split) : q.nstages;
  const int kb0 = st0 / q.nsub, t0 = st0 - kb0 * q.nsub;

  if (wg < F::PWG) {
    // ---------------- producers: thread = row ------------------------------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F::REGS_PRODUCER));
    const int tid = threadIdx.x & 127;
    bool ok = true;
    uint32_t sc = 0;                                       // stages so far, of all producers
    for (int w = w_first; w < q.nwork && ok; w += w_step) {
      const uint32_t q0 = (uint32_t)(work_item<!F::CONCAT>(q, w).tile / q.ntn) * TILE_M;
      // Row -> window column (class 0) and the number of classes that exist there (0 beyond the tensor).
      auto locate = [&](uint32_t vq, const float*& base, int& lim) {
        base = q.win;
        lim = 0;
        if (vq < q.VQ) {
          const uint32_t sg = vq / (uint32_t)q.Wq;
          const int i = (int)(vq - sg * (uint32_t)q.Wq);
          const uint32_t n = sg / (uint32_t)q.Ho;
          const int ho = (int)(sg - n * (uint32_t)q.Ho);
          base += (int64_t)n * q.img_stride + (int64_t)ho * q.strip + (int64_t)i * q.s * q.Kh;
          lim = q.Wp - i * q.s;
        }
      };
      const float *base, *hbase = q.win;
      int lim, hlim = 0;
      locate(q0 + tid, base, lim);
      const int hrow = TILE_M + (tid >> 3), hch = tid & 7;  // halo item: a row below the tile, one chunk of it
      const bool has_halo = tid < q.halo * 8;
      if (has_halo) locate(q0 + hrow, hbase, hlim);
      int kb = kb0, t = t0;
      for (int st = st0; st < st1; ++st, ++sc) {
        if (F::PWG == 1 || (int)(sc & 1) == wg) {
          const int buf = sc & 1;
          const uint32_t stage = a_ring + buf * a_stage_bytes;
          const int nch = kb == q.num_kb - 1 ? 2 * q.nks_last : 8;      // the MMAs stop at the last step with real k2
          const int4* kt = reinterpret_cast<const int4*>(koff_s + kb * KB);
          auto load8 = [&](const float* src, bool row_ok, int ch, float (&v)[8]) {
            const int4 o0 = kt[2 * ch], o1 = kt[2 * ch + 1];
            const int32_t off[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = ld_if(src + off[e], row_ok && off[e] >= 0);
          };
          auto store8 = [&](int row, int ch, const float (&v)[8]) {
            uint32_t p[3][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) split2(v[2 * e], v[2 * e + 1], p[0][e], p[1][e], p[2][e]);
            const uint32_t dst = stage + row * 128 + ((ch ^ (row & 7)) << 4);
#pragma unroll
            for (int i = 0; i < 3; ++i) st_shared16(dst + i * sub_bytes, p[i][0], p[i][1], p[i][2], p[i][3]);
          };
          const bool row_ok = t < lim;
          const float* src = base + t * q.Kh;
          float v[4][8], hv[8];
#pragma unroll
          for (int c = 0; c < 4; ++c) load8(src, row_ok && c < nch, c, v[c]);
          const bool halo_now = has_halo && hch < nch;
          if (halo_now) load8(hbase + t * q.Kh, t < hlim, hch, hv);
          ok = mbar_wait(a_empty0 + 8 * buf, ((sc >> 1) & 1) ^ 1, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
#pragma unroll
          for (int c = 0; c < 4; ++c) if (c < nch) store8(tid, c, v[c]);
          if (halo_now) store8(hrow, hch, hv);
          if (nch > 4) {
#pragma unroll
            for (int c = 0; c < 4; ++c) load8(src, row_ok && 4 + c < nch, 4 + c, v[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) if (4 + c < nch) store8(tid, 4 + c, v[c]);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(a_full0 + 8 * buf);
        }
        if (++t == q.nsub) { t = 0; ++kb; }
      }
    }
  } else if (wg == F::PWG) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F::REGS_MISC));
    if ((warp & 3) == 0) {
      // ---------------- MMA issuer -----------------------------------------------------------------
      const bool leader = elect_one();
      const uint32_t a_lo0 = smem_desc_lo(a_ring), b_lo0 = smem_desc_lo(b_ring);
      const uint32_t sub_lo = (uint32_t)sub_bytes >> 4;
      const uint32_t id3 = instr_desc_bf16(TILE_M, 3 * q.bn);
      bool ok = true;
      uint32_t sc = 0, ac = 0;                             // stages and chains so far
      int slot = 0;
      uint32_t bph = 0;
      // A wait for a barrier that is already complete costs 200 cycles and more while the shared-memory pipe is busy, and
      // the tensor pipe runs dry meanwhile (3x3 at 56x56 254 us without the looks ahead, 228 with them; 64 -> 128 channels at
      // 112x112 413 and 340): every barrier is looked at ahead of the instructions issued before it is needed, and waited
      // for only where that look came too early.
      uint32_t a_seen = 0, b_seen = 0, acc_seen = 0;
      // (testing aid: the first commit of an accumulator left out; looked up while the first stage is on its way)
      uint32_t drop = blockIdx.x == 0 ? *reinterpret_cast<volatile uint32_t*>(q.status + 2) : 0u;
      auto need = [&](uint32_t bar, uint32_t parity, uint32_t seen) {
        return mbar_wait_unless_seen<false>(bar, parity, seen, &abort_flag, q.status);
      };
      auto next_slot = [&](int& sl, uint32_t& ph) { if (++sl == q.sb) { sl = 0; ph ^= 1u; } };
      for (int w = w_first; w < q.nwork && ok; w += w_step) {
        const uint32_t id1 = instr_desc_bf16(TILE_M, work_item<!F::CONCAT>(q, w).bn);
        int kb = kb0, t = t0;
        for (int st = st0; st < st1 && ok; ++st, ++sc) {
          const int buf = sc & 1;
          const int nks = kb == q.num_kb - 1 ? q.nks_last : KB / 16;
          ok = need(a_full0 + 8 * buf, (sc >> 1) & 1, a_seen);
          if (!ok) break;
          tc_fence_after();
          uint32_t a_view = a_lo0 + (uint32_t)(buf * (a_stage_bytes >> 4));
          int links = 0;                                   // steps in the open chain; 0: none is open
          for (int v = t; v < q.Kw; v += q.s, a_view += 8u) {           // next view: one row (128 bytes) further down
            const int ab = ac & (F::NACC - 1);
            if (links == 0) {
              ok = need(acc_empty0 + 8 * ab, ((ac >> F::ACC_LOG) & 1) ^ 1, acc_seen);
              if (!ok) break;
              tc_fence_after();
            }
            const uint32_t d = tmem_acc + ab * F::ACC_COLS, more = links > 0;
            links += nks;
            const bool last_unit = v + q.s >= q.Kw;
            const bool last_link = !F::CONCAT || links + nks > q.chain || last_unit;
            // filter pieces: one operand (CONCAT), or one by one, smallest first: w3 meets x1, w2 meets x2 and x1, w1
            // meets x3, x2 and x1
#pragma unroll
            for (int p = 0; p < (F::CONCAT ? 1 : 3); ++p) {
              ok = need(b_full0 + 8 * slot, bph, b_seen);
              if (!ok) break;
              int nslot = slot;
              uint32_t nbph = bph;
              next_slot(nslot, nbph);
              b_seen = mbar_test_wait(b_full0 + 8 * nslot, nbph);
              if (F::CONCAT || p == 2) {
                if (last_link) acc_seen = mbar_test_wait(acc_empty0 + 8 * ((ac + 1) & (F::NACC - 1)), (((ac + 1) >> F::ACC_LOG) & 1) ^ 1);
                if (last_unit) a_seen = mbar_test_wait(a_full0 + 8 * (buf ^ 1), ((sc + 1) >> 1) & 1);
              }
              const uint32_t b_lo = b_lo0 + (uint32_t)(slot * (q.slot_bytes >> 4));
              if (leader) {
                if (nks == KB / 16) issue_steps<F::CONCAT, KB / 16>(d, q.bn, a_view, sub_lo, b_lo, id1, id3, more, p);
                else if (nks == 3) issue_steps<F::CONCAT, 3>(d, q.bn, a_view, sub_lo, b_lo, id1, id3, more, p);
                else if (nks == 2) issue_steps<F::CONCAT, 2>(d, q.bn, a_view, sub_lo, b_lo, id1, id3, more, p);
                else issue_steps<F::CONCAT, 1>(d, q.bn, a_view, sub_lo, b_lo, id1, id3, more, p);
                umma_commit(b_empty0 + 8 * slot);
                if (F::CONCAT || p == 2) {
                  if (last_link && drop != kDebugDropArrive) umma_commit(acc_full0 + 8 * ab);
                  if (last_unit) umma_commit(a_empty0 + 8 * buf);
                }
              }
              __syncwarp();
              slot = nslot;
              bph = nbph;
            }
            if (!ok) break;
            if (last_link) { ++ac; links = 0; drop = 0u; }
          }
          if (++t == q.nsub) { t = 0; ++kb; }
        }
      }
    } else if ((warp & 3) == 1) {
      // ---------------- filter copies ----------------------------------------------------------------
      const bool leader = elect_one();
      bool ok = true;
      int slot = 0;
      uint32_t bph = 0;
      const int per_unit = F::CONCAT ? 1 : 3;
      for (int w = w_first; w < q.nwork && ok; w += w_step) {
        const Item it = work_item<!F::CONCAT>(q, w);
        const int nt = it.tile % q.ntn;
        const unsigned char* tile = q.fp + (int64_t)nt * q.num_kb * q.Kw * 3 * q.bn * 128 + (int64_t)it.first * 128;
        const uint32_t bytes = F::CONCAT ? (uint32_t)q.slot_bytes : (uint32_t)it.bn * 128u;
        int kb = kb0, t = t0;
        for (int st = st0; st < st1 && ok; ++st) {
          for (int v = t; v < q.Kw && ok; v += q.s) {
            const unsigned char* src = tile + ((int64_t)kb * q.Kw + v) * 3 * q.bn * 128;
            for (int p = 0; p < per_unit; ++p) {
              ok = mbar_wait(b_empty0 + 8 * slot, bph ^ 1u, &abort_flag, q.status);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              if (leader) {
                mbar_arrive_expect_tx(b_full0 + 8 * slot, bytes);
                bulk_load(b_ring + slot * q.slot_bytes, src + (int64_t)p * q.slot_bytes, bytes, b_full0 + 8 * slot);
              }
              __syncwarp();
              if (++slot == q.sb) { slot = 0; bph ^= 1u; }
            }
          }
          if (++t == q.nsub) { t = 0; ++kb; }
        }
      }
      // copies in flight must land before the CTA gives its shared memory back (only after a wait that gave up)
      if (!ok) for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    __syncwarp();
    if (SHARED) { cluster_sync_all(); cluster_sync_all(); }
  } else {
    // ---------------- epilogue: fp32 sums of the tile in registers -------------------------------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(F::REGS_EPILOGUE));
    const int lq = warp & 3, h = (wg - F::PWG - 1);         // tensor-memory quadrant; which chunks of 16 channels
    bool ok = true;
    uint32_t ac = 0;
    float acc[F::CH][16];
    uint32_t n = 0;
    int ho = 0, i0 = 0, nt = 0;
    bool valid = false;
    for (int w = w_first; w < q.nwork && ok; w += w_step) {
      const Item it = work_item<!F::CONCAT>(q, w);
      const int mt = it.tile / q.ntn;
      nt = it.tile - mt * q.ntn;
      const uint32_t vq = (uint32_t)mt * TILE_M + (uint32_t)(lq * 32 + lane);
      valid = false;
      if (vq < q.VQ) {
        const uint32_t sg = vq / (uint32_t)q.Wq;
        i0 = (int)(vq - sg * (uint32_t)q.Wq);
        n = sg / (uint32_t)q.Ho;
        ho = (int)(sg - n * (uint32_t)q.Ho);
        valid = i0 < q.Wo;                                  // trailing columns of a strip are no output
      }
#pragma unroll
      for (int j = 0; j < F::CH; ++j)
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[j][e] = 0.f;
      int kb = kb0, t = t0;
      for (int st = st0; st < st1 && ok; ++st) {
        const int nks = kb == q.num_kb - 1 ? q.nks_last : KB / 16;
        const int units = F::CONCAT ? (q.chain / nks) : 1;  // units of a chain
        for (int v = t; v < q.Kw; v += q.s * units, ++ac) {
          const int ab = ac & (F::NACC - 1);
          ok = mbar_wait(acc_full0 + 8 * ab, (ac >> F::ACC_LOG) & 1, &abort_flag, q.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d = tmem_acc + ((uint32_t)(lq * 32) << 16) + ab * F::ACC_COLS + h * 16;
          if constexpr (F::CONCAT) {
#pragma unroll
            for (int j = 0; j < F::CH; ++j) {
              if ((h + 2 * j) * 16 >= q.bn) break;
              uint32_t r0[16], r1[16], r2[16], r3[16];
              tmem_ld16_issue(d + 32 * j, r0);
              tmem_ld16_issue(d + 32 * j + q.bn, r1);
              tmem_ld16_issue(d + 32 * j + 2 * q.bn, r2);
              tmem_ld16_issue(d + 32 * j + 3 * q.bn, r3);
              tmem_wait16(r0);
              tmem_wait16(r1);
              tmem_wait16(r2);
              tmem_wait16(r3);
#pragma unroll
              for (int e = 0; e < 16; ++e)
                acc[j][e] += __uint_as_float(r0[e]) + (__uint_as_float(r1[e]) + (__uint_as_float(r2[e]) + __uint_as_float(r3[e])));
            }
          } else {
            constexpr int STEP = BNMAX == 256 ? 1 : 2;      // chunks in flight (128 sums leave registers for one)
#pragma unroll
            for (int j = 0; j < F::CH; j += STEP) {         // (columns beyond bn hold nothing and are not stored)
              if ((h + 2 * j) * 16 >= it.bn) break;
              uint32_t r0[16], r1[16];
              tmem_ld16_issue(d + 32 * j, r0);
              if (STEP == 2) tmem_ld16_issue(d + 32 * j + 32, r1);
              tmem_wait16(r0);
              if (STEP == 2) tmem_wait16(r1);
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                acc[j][e] += __uint_as_float(r0[e]);
                if (STEP == 2) acc[j + STEP - 1][e] += __uint_as_float(r1[e]);
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty0 + 8 * ab);
        }
        if (++t == q.nsub) { t = 0; ++kb; }
      }
      if (!ok) break;
      if constexpr (SHARED) {
        // (here and not behind the loop, where the sums would have to be live over everything below)
        const int channels = q.Co - nt * q.bn < q.bn ? q.Co - nt * q.bn : q.bn;
        const ClusterSums sums(a_ring, q.split, rank, channels);
        __syncwarp();
        cluster_sync_all();                                 // (every MMA of every CTA has completed)
#pragma unroll
        for (int j = 0; j < F::CH; ++j) sums.store(acc[j], (h + 2 * j) * 16, channels, lq * 32 + lane);
        __syncwarp();
        cluster_sync_all();
        break;
      }
      if (valid) {
        const int co0 = nt * q.bn + it.first;
        float* yrow = q.y + ((int64_t)n * q.Co + co0) * q.HoWo + (int64_t)ho * q.Wo + i0;
        const int limit = q.Co - co0 < it.bn ? q.Co - co0 : it.bn;      // channels of this item that exist
        bool again = false;
#pragma unroll
        for (int j = 0; j < F::CH; ++j) {
          const int c0 = (h + 2 * j) * 16;
          store16(yrow + (int64_t)c0 * q.HoWo, q.HoWo, acc[j], limit - c0, again);
        }
        if (again) {
          const float* x = q.win + (int64_t)n * q.img_stride + (int64_t)ho * q.strip + (int64_t)i0 * q.s * q.Kh;
          const int64_t K = (int64_t)q.K2 * q.Kw;
          for (int c = h * 16; c < limit; c += 32)
            exact_outputs(x, q.f + (co0 + c) * K, yrow + (int64_t)c * q.HoWo, q.chan_stride, K, q.HoWo, q.C, q.Kh, q.Kw,
                          limit - c < 16 ? limit - c : 16);
        }
      }
    }
    if constexpr (SHARED) {
      if (!ok) { __syncwarp(); cluster_sync_all(); cluster_sync_all(); }      // (a wait gave up: the others wait for this CTA all the same)
      if (ok && valid) {
        const int co0 = nt * q.bn;
        const int channels = q.Co - co0 < q.bn ? q.Co - co0 : q.bn;
        const ClusterSums sums(a_ring, q.split, rank, channels);
        const int first = rank * sums.per, mine = channels - first < sums.per ? channels - first : sums.per;
        float* yrow = q.y + ((int64_t)n * q.Co + co0 + first) * q.HoWo + (int64_t)ho * q.Wo + i0;
        bool again = false;
        for (int c = h; c < mine; c += 2) {
          const float sum = sums.sum(c, lq * 32 + lane) * kUnscale;
          again |= suspicious(sum);
          yrow[(int64_t)c * q.HoWo] = sum;
        }
        if (again) {
          const float* x = q.win + (int64_t)n * q.img_stride + (int64_t)ho * q.strip + (int64_t)i0 * q.s * q.Kh;
          const int64_t K = (int64_t)q.K2 * q.Kw;
          for (int c = h; c < mine; c += 32) {
            const int left = (mine - c + 1) / 2;
            exact_outputs(x, q.f + (co0 + first + c) * K, yrow + (int64_t)c * q.HoWo, q.chan_stride, 2 * K, 2 * (int64_t)q.HoWo, q.C,
                          q.Kh, q.Kw, left < 16 ? left : 16);
          }
        }
      }
    }
  }
  if (wg < F::PWG && SHARED) {
    __syncwarp();
    cluster_sync_all();
    cluster_sync_all();
  }

  // ---------------- teardown -----------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (abort_flag) {
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == F::PWG * 4 + 2) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_acc, 512);
  }
}

// Filter -> the images the copy warp loads: for every (channel tile nt, k2-block kb, kernel column v) the three
// pieces [bn channels][64 k2] in the 128-byte-swizzled order of shared memory, smallest first, or largest first
// where they form one operand (bn <= CONCAT_BN); and a copy of the filter as given.  One block: `rows` channels of one
// k2-block; its source is one contiguous run of the OIHW filter per channel.  Channels beyond Co and k2 beyond C*Kh are
// zeros.
__global__ void __launch_bounds__(256) pack_f32_split_kernel(const float* __restrict__ f, unsigned char* __restrict__ fp,
                                                             float* __restrict__ copy, uint32_t* __restrict__ status, int K2, int Kw, int Co, int bn,
                                                             int num_kb, int rows, int concat) {
  extern __shared__ float pack_f[];
  let_next_kernel_start();                                 // (the convolution sets itself up meanwhile)
  wait_for_previous_kernel();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kStatusBytes / 4) status[threadIdx.x] = 0u;
  const int kb = blockIdx.y, row0 = blockIdx.x * rows;     // (channel blocks along x: any number of channels)
  const int nreal = K2 - kb * KB < KB ? K2 - kb * KB : KB;
  const int run = nreal * Kw, pitch = KB * Kw;
  for (int r = 0; r < rows; ++r) {
    const int co = row0 + r;
    const int64_t first = ((int64_t)co * K2 + (int64_t)kb * KB) * Kw;
    for (int i = threadIdx.x; i < pitch; i += blockDim.x) {
      float v = 0.f;
      if (co < Co && i < run) {
        v = __ldg(f + first + i);
        copy[first + i] = v;
      }
      pack_f[r * pitch + i] = v;
    }
  }
  __syncthreads();
  const int items = rows * Kw * 8;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int ch = it & 7, rv = it >> 3;
    const int r = rv % rows, v = rv / rows;
    const int row = row0 + r, nt = row / bn, rr = row - nt * bn;
    const float* src = pack_f + r * pitch + ch * 8 * Kw + v;
    uint32_t p[3][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) split2(src[(2 * e) * Kw], src[(2 * e + 1) * Kw], p[0][e], p[1][e], p[2][e]);
    const int64_t piece = (int64_t)bn * 128;
    unsigned char* dst = fp + (((int64_t)nt * num_kb + kb) * Kw + v) * 3 * piece + rr * 128 + ((ch ^ (rr & 7)) << 4);
#pragma unroll
    for (int i = 0; i < 3; ++i)
      *reinterpret_cast<uint4*>(dst + (concat ? i : 2 - i) * piece) = make_uint4(p[i][0], p[i][1], p[i][2], p[i][3]);
  }
}

int form_of(int bn) { return bn <= CONCAT_BN ? CONCAT_BN : (bn <= 128 ? 128 : 256); }
int slot_bytes_of(int bn) { return (bn <= CONCAT_BN ? 3 : 1) * bn * 128; }

// Filter slots that fit beside the two S stages and the offset table.
int slots_for(int bn, int rows, int num_kb) {
  const int left = kSplitSmem - 1024 - A_STAGES * 3 * rows * 128 - num_kb * KB * 4;
  const int n = left / slot_bytes_of(bn);
  return n > MAX_B ? MAX_B : n;
}

// Cycles of an instruction of N = n, and of the six products of a 128 x bn tile over 16 k (see the head of this file).
double mma_cycles(int n) { const double pipe = n / 2.0, smem = 32 + n / 4.0; return pipe > smem ? pipe : smem; }
double step_cycles(int bn) { return bn <= CONCAT_BN ? mma_cycles(3 * bn) + 3 * mma_cycles(bn) : 6 * mma_cycles(bn); }

// Parts of its channels that a tile of the last round goes out in, where that round leaves half of the SMs or more idle: an
// instruction of N = 64 takes 3/8 of the time of N = 256, so quarters save 5/8 of a round.  (5x5 on 256 channels at 28x28,
// batch 64, 3.03 rounds of tiles: 966 -> 766 us; 7x7, 3.2 rounds: 1909 -> 1493.)
int channel_parts(int64_t tiles, int bn) {
  const int64_t last = tiles % 148;
  if (last == 0 || bn <= CONCAT_BN) return 1;
  for (int parts = 4; parts > 1; parts /= 2)
    if (last * parts <= 148 && bn % (16 * parts) == 0) return parts;
  return 1;
}

// SHARED: tiles shared by the CTAs of a cluster.  A kernel of its own: decided at run time, meeting and adding up sixteen parts cost the layers
// that share nothing up to 9 % (5x5 on 4 -> 13 channels at 148x148, batch 128, 436 -> 461 us, 3x3 on 8 -> 50 at 195x195, batch 64, 363 -> 396).
template <int BNMAX, int PWG, bool SHARED>
cudaError_t launch_kernel(SplitParams q, int smem, cudaStream_t stream) {
  constexpr auto kernel = conv_f32_split_kernel<BNMAX, PWG, SHARED>;
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem);
    if (e == cudaSuccess && SHARED) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  if constexpr (SHARED) {
    static KnownClusters known;
    q.split = ctas_that_fit(kernel, q.split, Form<BNMAX, PWG>::THREADS, kSplitSmem, known);
    if (q.split == 1) return launch_kernel<BNMAX, PWG, false>(q, smem, stream);
    return launch_after_previous(kernel, q.nwork * q.split, q.split, Form<BNMAX, PWG>::THREADS, smem, stream, q);
  }
  return launch_after_previous(kernel, q.nwork < 148 ? q.nwork : 148, 1, Form<BNMAX, PWG>::THREADS, smem, stream, q);
}

template <int BNMAX, int PWG>
cudaError_t launch_form(const SplitParams& q, int smem, cudaStream_t stream) {
  return q.split > 1 ? launch_kernel<BNMAX, PWG, true>(q, smem, stream) : launch_kernel<BNMAX, PWG, false>(q, smem, stream);
}

}  // namespace

F32SplitPlan plan_f32_split(const Geometry& g) {
  F32SplitPlan p{};
  p.eligible = false;
  const int64_t K2 = (int64_t)g.C * g.Kh;
  p.num_kb = (int32_t)((K2 + KB - 1) / KB);
  p.halo = (g.Kw - 1) / g.s;
  if (p.halo > 16 || g.Kw > 64 || K2 > 6144) return p;      // halo items, filter staging, offset table
  p.rows = TILE_M + (p.halo + 7) / 8 * 8;
  p.nsub = g.s < g.Kw ? g.s : g.Kw;
  p.Wq = (g.Wp + g.s - 1) / g.s;
  p.VQ = (int64_t)g.N * g.Ho * p.Wq;
  // Channel tile and split decide the order of the sums: they are chosen for the batch these images belong to.
  const int64_t plan_VQ = (int64_t)g.plan_N * g.Ho * p.Wq;
  if (plan_VQ + 2 * TILE_M >= ((int64_t)1 << 31)) return p;
  p.nks_last = (int32_t)((K2 - (int64_t)(p.num_kb - 1) * KB + 15) / 16);
  p.nstages = p.num_kb * p.nsub;
  const int64_t ntm = (plan_VQ + TILE_M - 1) / TILE_M;
  const double steps = ((p.num_kb - 1) * 4.0 + p.nks_last) * g.Kw;   // 16-wide steps of a tile
  const char* force_bn = debug_getenv("IM2WIN_F32_SPLIT_BN");        // testing aids: channel tile, CTAs per tile
  const char* force_z = debug_getenv("IM2WIN_F32_SPLIT_CTAS");
  p.cost = 0;
  p.packed_rows = 0;
  const int most = (g.Co + 15) / 16;
  for (int nt = (g.Co + 255) / 256; nt <= most && nt <= (g.Co + 255) / 256 + 32; ++nt) {
    const int bn = ((g.Co + nt - 1) / nt + 15) / 16 * 16;
    if (nt > 1 && (int64_t)(nt - 1) * bn >= g.Co) continue;          // fewer tiles of this width do
    const int sb = slots_for(bn, p.rows, p.num_kb);
    if (sb < (bn <= CONCAT_BN ? 2 : 3)) continue;
    if (nt * bn > p.packed_rows) p.packed_rows = nt * bn;
    if (force_bn && bn != atoi(force_bn)) continue;
    if (ntm * nt >= ((int64_t)1 << 30)) continue;
    for (int z = 1; z <= kMaxCtas && z <= p.nstages; ++z) {
      const int64_t tiles = ntm * nt;
      if (z > 1 && tiles > resident_clusters(z)) continue;           // clusters: one tile each, all resident
      if (force_z && z != atoi(force_z)) continue;
      // The estimate: the tensor pipe, or the shared-memory pipe with operands, copies and staging.  For clusters and reductions of one
      // k2-block the latter is nine tenths of the former, and what is staged.  Else the operands are counted (11x11 on 256
      // channels, a unit of four steps: 3126 cycles in tiles of 256 channels, 2185 in tiles of 128), for layers of one round up to
      // nine tenths; in more rounds the last may go out in parts.  Against nine tenths for all 1.17 times as fast on average on 223
      // layers that choose other tiles for it, 0.97 at the least.  Counted for all, with parts for all: too wide tiles, 0.72 at the
      // least (3x3 stride 2 on 64 -> 256 channels at 14x14, batch 95: 42 tiles of 256 channels in pairs of CTAs 31.6 us, 126 of 96
      // 23.4; 3x3 on 16 -> 256 channels at 16x140: halves of 62 tiles of 256 15.2, 124 of 128 13.4; 5x5 on 8 -> 372 channels at
      // 47x47 26.5 and 22.9).
      const bool counted = z == 1 && p.num_kb > 1 && bn > CONCAT_BN, rounds = z == 1 && p.num_kb > 1 && tiles > 148;
      auto tile_cycles = [&](int cols) {
        const double fill = 3.0 * cols * steps / 4 + 1200.0 * p.nstages;
        const double pipe = steps * (bn <= CONCAT_BN ? step_cycles(bn) : 6 * mma_cycles(cols));
        double wave = pipe * 0.9;
        if (counted) {
          const double operands = steps * 6 * (32 + cols / 4.0);
          wave = rounds || operands < wave ? operands : wave;
        }
        wave += fill;
        // (meeting and adding up: fitted to 40 layers with 1 to 16 CTAs, the choice is within 1 % of the best on average)
        return (pipe > wave ? pipe : wave) * ((p.nstages + z - 1) / z) / p.nstages + (z > 1 ? 5000 + 300 * z + 20 * cols : 1500);
      };
      const int parts = rounds ? channel_parts(tiles, bn) : 1;
      const double last = tiles % 148 == 0 ? 0.0 : tile_cycles(bn / parts);
      const double cost = 6000 + (z > 1 ? tile_cycles(bn) : (double)(tiles / 148) * tile_cycles(bn) + last);
      if (!p.eligible || cost < p.cost) {
        p.eligible = true;
        p.cost = cost;
        p.bn = bn; p.ntn = nt; p.split = z; p.sb = sb;
        const int64_t mine = (p.VQ + TILE_M - 1) / TILE_M * nt;      // tiles of these N images
        p.parts = z > 1 ? 1 : channel_parts(mine, bn);
        p.n_main = (int32_t)(p.parts > 1 ? mine - mine % 148 : mine);
        p.nwork = (int32_t)(p.n_main + (mine - p.n_main) * p.parts);
      }
    }
  }
  if (!p.eligible) return p;
  p.copy_off = ((size_t)p.packed_rows * p.num_kb * KB * g.Kw * 6 + 255) / 256 * 256;
  p.filter_bytes = p.copy_off + (size_t)g.Co * g.K * 4;
  return p;
}

cudaError_t launch_pack_f32_split(const float* filter, void* scratch, const Geometry& g, cudaStream_t stream) {
  const F32SplitPlan p = plan_f32_split(g);
  if (!p.eligible) return cudaErrorInvalidValue;
  unsigned char* base = static_cast<unsigned char*>(scratch);
  // Channels per block: staging within 40 KB, and two blocks an SM where the filter has them (a block's channels are loaded one
  // after another, a round trip each)
  int rows = 8;
  while (rows > 1 && ((size_t)rows * KB * g.Kw * 4 > 40 * 1024 || (int64_t)p.ntn * p.bn / rows * p.num_kb < 2 * 148)) rows /= 2;
  const size_t smem = (size_t)rows * KB * g.Kw * 4;
  dim3 grid((unsigned)(p.ntn * p.bn / rows), (unsigned)p.num_kb);
  return launch_pack<pack_f32_split_kernel>(grid, 256, smem, stream, filter, base + kStatusBytes,
                      reinterpret_cast<float*>(base + kStatusBytes + p.copy_off), reinterpret_cast<uint32_t*>(base), g.C * g.Kh, g.Kw, g.Co,
                      p.bn, p.num_kb, rows, p.bn <= CONCAT_BN ? 1 : 0);
}

cudaError_t launch_conv_f32_split(const float* window, float* y, void* scratch, const Geometry& g, cudaStream_t stream) {
  const F32SplitPlan p = plan_f32_split(g);
  if (!p.eligible) return cudaErrorInvalidValue;
  unsigned char* base = static_cast<unsigned char*>(scratch);
  SplitParams q;
  q.win = window;
  q.fp = base + kStatusBytes;
  q.f = reinterpret_cast<const float*>(base + kStatusBytes + p.copy_off);
  q.y = y;
  q.status = reinterpret_cast<uint32_t*>(base);
  q.img_stride = g.img_stride; q.strip = g.strip; q.chan_stride = g.chan_stride;
  q.VQ = (uint32_t)p.VQ;
  q.K2 = g.C * g.Kh; q.C = g.C; q.Wq = p.Wq; q.Wp = g.Wp; q.Ho = g.Ho; q.Wo = g.Wo; q.HoWo = g.Ho * g.Wo; q.Co = g.Co;
  q.Kh = g.Kh; q.Kw = g.Kw; q.s = g.s; q.nsub = p.nsub; q.num_kb = p.num_kb; q.nks_last = p.nks_last;
  q.rows = p.rows; q.halo = p.halo; q.n_main = p.n_main; q.parts = p.parts;
  q.bn = p.bn; q.ntn = p.ntn; q.nwork = p.nwork; q.nstages = p.nstages; q.split = p.split;
  q.sb = p.sb; q.slot_bytes = slot_bytes_of(p.bn);
  q.chain = g.K >= 288 ? 12 : 8;
  const int rings = A_STAGES * 3 * p.rows * 128 + p.sb * q.slot_bytes + p.num_kb * KB * 4;
  const int smem = 1024 + rings;
  if (p.split > 1 && rings < cluster_sums_bytes(p.bn)) return cudaErrorInvalidValue;
  switch (form_of(p.bn)) {
    case CONCAT_BN: return p.num_kb == 1 ? launch_form<CONCAT_BN, 1>(q, smem, stream) : launch_form<CONCAT_BN, 2>(q, smem, stream);
    case 128: return launch_form<128, 2>(q, smem, stream);
    default: return launch_form<256, 1>(q, smem, stream);
  }
}

}  // namespace im2win
