// Shared host-side definitions of the im2win library: derived geometry,
// scratch layout and launch prototypes.  Device code lives in the .cu files.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/im2win.h"

namespace im2win {

// Quantities derived from an im2win_shape (notation of the paper's Section
// "Notation" and Eq. 2/3): Wp = W + 2p, strip = Kh*Wp elements per (n,c,ho),
// T = Kh*Kw window elements per channel, K = C*T reduction length,
// P = N*Ho*Wo output positions.
struct Geometry {
  int32_t N, C, H, W, Co, Kh, Kw, s, p;
  int32_t Ho, Wo, Wp, T;
  int64_t strip;         // Kh*Wp
  int64_t chan_stride;   // Ho*strip: distance between channels of one image in the window tensor
  int64_t img_stride;    // C*chan_stride
  int64_t K;             // C*T
  int64_t P;             // N*Ho*Wo
  int64_t window_elems;  // N*img_stride
  int64_t out_elems;     // N*Co*Ho*Wo
  int32_t plan_N;        // batch the kernel and the order of its sums are chosen for: N, or what these N images are a part of
};

// Clusters of z CTAs, each CTA an SM to itself, that a B200 holds at once: they lie within a GPC, so that wide ones leave SMs over.
// (What cudaOccupancyMaxActiveClusters says of 226 KB of shared memory a CTA, but for threes and fives, of which it says 45 and 26: started while
// the kernel ahead still leaves its SMs, they take those that are free, not those that fit best, and 42 and 25 are the most that never leave one for
// a second round.  3x3 on 512 -> 64 channels, 128 positions a tile, shared by three: a pass of 42 tiles 27.2 us, of 44 32.8, of 45 37.8; by
// five: 25 tiles 21.3, 26 27.5.  All other sizes up to their full number take the same.  16 clusters of 8 CTAs run in two rounds: 7x7 on
// 256 -> 78 channels at 35x35, batch 2, 87 us in clusters of 8, 47 in clusters of 4.)
// The plans go by this table, so that they do not depend on the machine; the launchers ask the device (ctas_that_fit).
constexpr int kMaxCtas = 16;       // of a cluster (above 8: the non-portable sizes)
// Longest reduction of an fp16 layer whose tiles are shared.  An accumulator truncates every addend, 1e-9 of the sum a term,
// so a shared reduction is the more exact one; beyond this the two would differ by more than fp32 sums in another order do.
constexpr int64_t kMostSplitTerms = 16384;
inline int resident_clusters(int z) {
  constexpr int kResident[kMaxCtas + 1] = {0, 148, 74, 42, 33, 25, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7};
  return z >= 1 && z <= kMaxCtas ? kResident[z] : 0;
}

// The most CTAs up to `want` whose cluster fits (a function of their number), 1 where none of two or more does.
template <typename Fits>
int widest_cluster(int want, const Fits& fits) {
  for (int z = want; z > 1; --z)
    if (fits(z)) return z;
  return 1;
}

// Shared memory with which an SM takes no more of `blocks` blocks than its share.  Blocks that are launched early go to the SMs that the kernel
// ahead leaves first, as many to an SM as it holds, and crowd there while others idle.  (226 KB of an SM, 1 KB a block is the system's.)
constexpr int kMostSpread = 200 * 1024;
inline size_t spread_smem(int64_t blocks, int threads, size_t smem) {
  const int64_t share = (blocks + 147) / 148;
  if (share >= 2048 / threads) return smem;
  int64_t spread = (226 * 1024 / share - 1024) / 128 * 128;
  if (spread > kMostSpread) spread = kMostSpread;
  return (int64_t)smem < spread ? (size_t)spread : smem;
}

// Scratch layout shared by both precisions (offsets in bytes from `scratch`):
//   [0, 256)            status block (uint32 words; word 0 = timeout flag)
//   [256, 256 + 4*Kp)   k -> element offset table (int32), -1 for padded k
//   [filter_off, ...)   repacked filter
struct ScratchLayout {
  int64_t Kp;            // reduction length rounded up to the k-block of the kernel
  int64_t Co_pad;        // Co rounded up to the filter tile of the kernel
  size_t koff_off, filter_off, total;
  size_t ffma_total;     // fp32 only: what the FFMA kernel alone needs
  bool f32_split;        // fp32 only: the tensor-core kernel is used (filter images right after the status block)
  bool f16_runs;         // fp16 only: the run-staged kernel is used (filter images right after the status block)
  bool f16_shift;        // fp16 only: a shifted-view kernel (and its filter layout) is used
  bool f16_raw;          // fp16 only: the bulk-copy variant of the shifted-view kernel is used
  bool f16_mat;          // fp16 only: the matrix-transpose variant is used (own scratch layout)
  bool f16_stem;         // fp16 only: the one-k-block kernel for C*Kh <= 64 is used (filter layout of f16_shift)
};

// Tile geometry of the fp16 shifted-view kernel for one layer (see conv_f16_shift.cu).
struct ShiftPlan {
  bool eligible;
  int32_t Wq;            // virtual positions per strip = ceil(Wp / s)
  int32_t rows;          // rows of one shared-memory sub-tile: 128 + halo, multiple of 8
  int32_t total_rows;    // s * rows
  int32_t items;         // 16-byte chunks each producer thread fills per stage
  int32_t chunks;        // 16-byte chunks staged per row (8, fewer when one short k-block is all)
  int32_t nks_last;      // 16-wide MMA steps of the last k-block
  int64_t K2, K2p;       // C*Kh and its round-up to 64
  int64_t VQ;            // N*Ho*Wq virtual positions
  int32_t bn, split;     // channel tile, CTAs of a cluster that share the k-blocks of a tile
};
ShiftPlan plan_f16_shift(const Geometry& g);

// Tile geometry of the bulk-copy shifted-view kernel (see conv_f16_raw.cu).
struct RawPlan {
  bool eligible;
  int32_t Wq, rows;
  int32_t nslot, pitch, raw_stage_bytes, a_stage_bytes;
  int64_t K2, K2p, VQ;
};
RawPlan plan_f16_raw(const Geometry& g);

// Tile geometry of the matrix-transpose shifted-view kernel (see conv_f16_mat.cu).
struct MatPlan {
  bool eligible;
  int32_t Wq, rows, R, Cp8, nch_last, nplanes, box_bytes, raw_stage_bytes, a_stage_bytes, num_kb;
  int64_t K2p, VQ;
  size_t scratch_bytes;  // status block + packed filter
};
MatPlan plan_f16_mat(const Geometry& g);

// Tile geometry of the one-k-block kernel for layers with C*Kh <= 64 (see conv_f16_stem.cu).
struct StemPlan {
  bool eligible;
  int32_t Wq, ragged, rows, R, nks, chan_region, raw_stage_bytes, a_stage_bytes, b_stage_bytes, bn;
  int32_t sa, rs, sb, resident, smem_bytes, epi_bufs;
  int64_t VQ;
};
StemPlan plan_f16_stem(const Geometry& g);

// Tile geometry of the channel-innermost (NHWC) path (see nhwc.cu).
struct NhwcPlan {
  bool eligible;
  bool pair;               // CTA pairs (cta_group::2)
  int32_t Cp;              // stored channels: C rounded up to 8
  int32_t num_kb;          // 64-wide k-blocks of K
  int32_t tw, bw, G;       // tw tiles of bw output columns along a strip; G strips per tile
  int32_t bn, ntn;         // channel tile and their number
  int32_t ksplit, kb_per_split;
  int64_t K;               // Kw*Kh*Cp
  int64_t strip;           // Wp*Kh*Cp halves per (n, ho)
  int64_t window_elems;    // N*Ho*strip
  int64_t ntm;             // position tiles
  size_t flags_off;        // byte offset of the tail-tile flag words inside the scratch
  size_t partial_off;      // byte offset and size of the partial-sum area (0 bytes: layer of many rounds of tiles)
  size_t partial_bytes;
  size_t scratch_bytes;    // status block + packed filter + flag words + partial sums
};
NhwcPlan plan_nhwc(const Geometry& g);

// What the convolution does with a finished accumulator (last step of the paper's Algorithm 1).
struct EpilogueArgs {
  const float* bias;       // device, Co floats, or nullptr
  int32_t relu;            // 1: max(y, 0) after the bias
  int32_t out16;           // 1: store binary16 (round to nearest even), 0: binary32
  int32_t y_nhwc;          // 1: y is [N][Ho][Wo][Co], 0: [N][Co][Ho][Wo]
};

// Tile shape of the fp32 kernel for a layer (see conv_f32.cu); the packed filter's K is padded to bk.
struct F32Plan {
  int32_t bm, bn, bk;
  bool klanes;             // the window operand is gathered with k along the lanes of a warp
  bool tall;               // 16 positions x 8 channels per thread (position pairs packed)
};
F32Plan plan_f32(const Geometry& g);

// Tile shape of the fp32 kernel that runs on the tensor cores (see conv_f32_split.cu).
struct F32SplitPlan {
  bool eligible;
  int32_t Wq, rows, halo, nsub, num_kb, nks_last, nstages;
  int32_t bn, ntn, split, sb, nwork;   // channel tile and their number, CTAs per tile, filter slots, work items
  int32_t n_main, parts;               // tiles from n_main on go out in parts of their channels
  int32_t packed_rows;                 // most rows (ntn * bn) of any tile width: the filter area does not depend on N
  int64_t VQ;
  size_t copy_off, filter_bytes;       // images, then a copy of the filter as given
  double cost;                         // cycles, estimated
};
F32SplitPlan plan_f32_split(const Geometry& g);

// Tile and ring geometry of the run-staged kernel (see conv_f16_runs.cu).
struct RunsPlan {
  bool eligible, resident, quad, pair; // quad: up to four channels, see the order of k2 there; pair: CTA pairs
  int32_t units, octs, E, G, Wq, rows, halo, num_kb, nks_last;
  int32_t region, raw_slot, a_stage, slot_bytes, cols, planes, seg_bytes;
  int32_t bn, ntn, ntm, nwork, sa, sr, sb;
  int32_t mode, teams;                 // how the staging warps read the raw slots, and how many teams they form
  int32_t split;                       // CTAs of a cluster that share the reduction of a tile
  int64_t VQ;
  size_t filter_bytes;
};
RunsPlan plan_f16_runs(const Geometry& g);

// Environment switches are testing aids: they are looked at only when IM2WIN_DEBUG is set in the
// environment (checked once per process), so the default call path reads no environment.
const char* debug_getenv(const char* name);

constexpr int kStatusBytes = 256;
constexpr int kF32KBlock = 16;     // smallest k-block of the fp32 kernel (see plan_f32)
constexpr int kF16KBlock = 64;     // k-block of the fp16 kernel (64 halves = one 128-byte swizzle row)

im2win_status derive_geometry(const im2win_shape* s, Geometry* g);
im2win_status scratch_layout(const Geometry& g, im2win_dtype dtype, ScratchLayout* l);

// Kernel launchers (each queues work on `stream` and returns the launch status).
cudaError_t launch_transform(const void* x, void* window, const Geometry& g, int elem_bytes,
                             cudaStream_t stream);
cudaError_t launch_pack_f32(const float* filter, void* scratch, const Geometry& g,
                            const ScratchLayout& l, cudaStream_t stream);
cudaError_t launch_pack_f16(const uint16_t* filter, void* scratch, const Geometry& g,
                            const ScratchLayout& l, cudaStream_t stream);
cudaError_t launch_conv_f32(const float* window, float* y, const void* scratch, const Geometry& g,
                            const ScratchLayout& l, cudaStream_t stream);
cudaError_t launch_pack_f16_runs(const uint16_t* filter, void* scratch, const Geometry& g, cudaStream_t stream);
cudaError_t launch_conv_f16_runs(const uint16_t* window, float* y, void* scratch, const Geometry& g, cudaStream_t stream);
// (both plan for g.plan_N images and run on g.N)
cudaError_t launch_pack_f32_split(const float* filter, void* scratch, const Geometry& g, cudaStream_t stream);
cudaError_t launch_conv_f32_split(const float* window, float* y, void* scratch, const Geometry& g, cudaStream_t stream);
cudaError_t launch_pack_f16_shift(const uint16_t* filter, void* scratch, const Geometry& g,
                                  const ScratchLayout& l, cudaStream_t stream);
cudaError_t launch_pack_f16_raw(const uint16_t* filter, void* scratch, const Geometry& g,
                                const ScratchLayout& l, const RawPlan& plan, cudaStream_t stream);
cudaError_t launch_conv_f16_raw(const uint16_t* window, float* y, void* scratch, const Geometry& g,
                                const ScratchLayout& l, cudaStream_t stream);
// Matrix-transpose kernel: filter pack into `scratch` (own layout) and the convolution on it.
cudaError_t launch_pack_f16_mat(const uint16_t* filter, void* scratch, const Geometry& g, cudaStream_t stream);
cudaError_t launch_conv_f16_mat(const uint16_t* window, float* y, void* scratch, const Geometry& g,
                                cudaStream_t stream);
cudaError_t launch_conv_f16_stem(const uint16_t* window, float* y, void* scratch, const Geometry& g,
                                 const ScratchLayout& l, cudaStream_t stream);
cudaError_t launch_conv_f16_gather(const uint16_t* window, float* y, void* scratch, const Geometry& g,
                                   const ScratchLayout& l, cudaStream_t stream);
cudaError_t launch_conv_f16_shift(const uint16_t* window, float* y, void* scratch, const Geometry& g,
                                  const ScratchLayout& l, cudaStream_t stream);

cudaError_t launch_transform_nhwc(const uint16_t* x, int x_is_nhwc, uint16_t* window, const Geometry& g,
                                  cudaStream_t stream);
const char* nhwc_kernel_name(const Geometry& g, const EpilogueArgs& epi);
cudaError_t launch_pack_f16_nhwc(const uint16_t* filter, void* scratch, const Geometry& g, cudaStream_t stream);
cudaError_t launch_conv_f16_nhwc(const uint16_t* window, void* y, void* scratch, const Geometry& g,
                                 const EpilogueArgs& epi, cudaStream_t stream);

}  // namespace im2win
