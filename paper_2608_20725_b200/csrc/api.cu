// C ABI of the im2win library: argument validation, buffer-size queries and
// dispatch to the kernels.  Declarations and the contract of every entry
// point are in include/im2win.h.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace im2win {

static inline int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

const char* debug_getenv(const char* name) {
  static const bool enabled = getenv("IM2WIN_DEBUG") != nullptr;   // looked up once per process
  return enabled ? getenv(name) : nullptr;
}

im2win_status derive_geometry(const im2win_shape* s, Geometry* g) {
  if (!s) return IM2WIN_ERR_NULL_POINTER;
  if (s->N < 1 || s->C < 1 || s->H < 1 || s->W < 1 || s->Co < 1 || s->Kh < 1 || s->Kw < 1 ||
      s->stride < 1 || s->pad < 0)
    return IM2WIN_ERR_INVALID_ARG;
  const int64_t hspan = (int64_t)s->H + 2 * (int64_t)s->pad - s->Kh;
  const int64_t wspan = (int64_t)s->W + 2 * (int64_t)s->pad - s->Kw;
  if (hspan < 0 || wspan < 0) return IM2WIN_ERR_INVALID_ARG;
  g->N = s->N; g->C = s->C; g->H = s->H; g->W = s->W; g->Co = s->Co;
  g->Kh = s->Kh; g->Kw = s->Kw; g->s = s->stride; g->p = s->pad;
  g->Ho = (int32_t)(hspan / s->stride) + 1;
  g->Wo = (int32_t)(wspan / s->stride) + 1;
  const int64_t Wp = (int64_t)s->W + 2 * (int64_t)s->pad;
  const int64_t T = (int64_t)s->Kh * s->Kw;
  // Index ranges of the kernels: 32-bit per-image offsets and counts, 64-bit bases.
  const int64_t lim = (int64_t)1 << 31;
  if (Wp >= lim || T >= lim) return IM2WIN_ERR_UNSUPPORTED;
  g->Wp = (int32_t)Wp;
  g->T = (int32_t)T;
  g->strip = (int64_t)s->Kh * Wp;
  if (g->strip >= lim) return IM2WIN_ERR_UNSUPPORTED;
  g->chan_stride = (int64_t)g->Ho * g->strip;
  if (g->chan_stride >= lim) return IM2WIN_ERR_UNSUPPORTED;
  g->img_stride = (int64_t)s->C * g->chan_stride;
  if (g->img_stride >= lim) return IM2WIN_ERR_UNSUPPORTED;    // k -> offset table is int32
  g->K = (int64_t)s->C * T;
  if (g->K >= lim - 64) return IM2WIN_ERR_UNSUPPORTED;
  if ((int64_t)g->Ho * g->Wo >= lim) return IM2WIN_ERR_UNSUPPORTED;
  g->P = (int64_t)s->N * g->Ho * g->Wo;
  if (g->P >= lim * 64) return IM2WIN_ERR_UNSUPPORTED;        // grid.x of 128-row tiles
  if ((int64_t)s->N * s->C * g->Ho * Wp >= lim * 4) return IM2WIN_ERR_UNSUPPORTED;      // transform grid
  if ((int64_t)s->H * s->W >= lim) return IM2WIN_ERR_UNSUPPORTED;
  if ((int64_t)s->Kh * 8 * 4 > 200 * 1024) return IM2WIN_ERR_UNSUPPORTED;  // transform staging
  if ((int64_t)s->Co * g->K >= lim * 16) return IM2WIN_ERR_UNSUPPORTED;
  g->window_elems = (int64_t)s->N * g->img_stride;
  g->out_elems = (int64_t)s->N * s->Co * g->Ho * g->Wo;
  g->plan_N = s->N;
  return IM2WIN_OK;
}

// Which fp32 kernel: the tensor cores from 64 terms on, but up to 80 only where one stage holds them (not two k2-blocks or
// column classes, the second nearly empty) and up to 256 channels, and below 160 only where 0.6 of the multiplied terms are
// real (a kernel column's C * Kh terms are rounded up to 16).  Measured on 754 layers, FFMA time / time here: of the 345
// with 64 terms and more that the rule takes 2.07 on average, 13 below 0.97, 0.85 at the least, up to 22; of the 169 it leaves
// to the FFMA kernel 1.0 on average (0.62 to 1.47); 0.56 to 1.2 below 64 terms.  Forcing one of the FFMA kernel's forms, or
// IM2WIN_F32_KERNEL=ffma|split, decides it (testing aids).
static bool want_f32_split(const Geometry& g, const F32SplitPlan& p) {
  if (const char* v = debug_getenv("IM2WIN_F32_KERNEL")) return strcmp(v, "split") == 0;
  for (const char* name : {"IM2WIN_F32_BM", "IM2WIN_F32_TALL", "IM2WIN_F32_KLANES", "IM2WIN_F32_BK"})
    if (debug_getenv(name)) return false;
  const int64_t multiplied = ((p.num_kb - 1) * 4 + p.nks_last) * (int64_t)16 * g.Kw;
  if (g.K < 64 || (g.K < 160 && 10 * g.K < 6 * multiplied)) return false;
  return g.K > 80 || (p.nstages == 1 && g.Co <= 256);
}

// Images that a tile of the run-staged kernel touches, on average.
static double images_of_a_tile(const Geometry& g, const RunsPlan& p) { return 1.0 + (128.0 + p.halo) / (double)((int64_t)g.Ho * p.Wq); }

// Of the layers that neither the one-k-block kernel nor a tiled-copy kernel takes, and the shifted-view kernel could: which
// ones the run-staged kernel gets.  Its copies are at most one per channel and image of a tile, so their number for each staged
// element is (images of a tile) / E, with E elements per virtual column; the shifted-view kernel stages all s columns even
// where the kernel has fewer (Kw < s).  Measured over 400 layers (images of 7 to 160, square kernels of 1 to 7, strides 1 and 2, 5
// to 512 channels, batches 1 to 128), shifted-view time / run-staged time:
//   3x3 stride 1, images / E up to 0.7: 65 to 128 channels 1.22 to 1.66, more channels 0.92 to 1.1 with up to 148 tiles and
//   1.1 to 1.6 with more; up to 64 channels 1.43 (1.14 at the least) where rows are staged in pairs, 1.1 (0.94) where not
//   5x5 stride 1: 1.09 to 1.47 with more than 296 tiles, 0.7 to 1.2 with fewer; 7x7 0.84
//   stride 2, up to 0.9: 3x3 1.62; 5x5 and 7x7 1.03 to 2.2 up to 128 channels, 0.9 to 1.1 on more with few tiles
// and over 220 layers that are not square or have larger strides (images of 4 to 100, with the forms the kernel has now):
//   five wide, stride 1, more than 296 tiles: one to four high 1.06 to 1.8 at every images / E; six and seven high 1.1 to 1.7 up to
//   128 channels, 0.93 to 1.5 on more
//   strides 3 and 4, images / E of 0.7 to 0.9 1.4 to 2.1; four virtual columns (11 wide at stride 3) 1.45 to 2.3 up to 128
//   channels, 1.02 to 1.5 on more from three tiles on, 0.92 and 0.99 with fewer
// (256 -> 512 channels, 3x3 stride 2 at 28x28, batch 128: 140 -> 88 us; not taken: 3x3 on 512 channels at 7x7, batch 128, 44 us
// against 55.)
static bool prefer_runs(const Geometry& g, const RunsPlan& p) {
  const double images = images_of_a_tile(g, p);
  const int64_t tiles = (int64_t)p.ntm * p.ntn;
  if (g.s == 1) {
    if (p.G == 5) return tiles > 296 && (g.Kh <= 5 || g.Co <= 128);
    if (p.G > 3 || images > 0.7 * p.E) return false;
    if (g.Co > 64) return g.Co <= 128 || tiles > 148;
    return p.E == 3 && (int64_t)g.Ho * g.Wp % 2 == 0;
  }
  if (p.G > 4 || (p.G > 2 && g.s == 2 && g.Co > 128 && (p.G > 3 || tiles <= 74))) return false;
  if (p.G == 4 && g.Co > 128 && tiles < 3) return false;
  return images <= (g.Kw < g.s ? 2.1 : 0.9) * p.E;
}

// 3x3 layers of stride 1 that the tiled-copy kernels could take: the run-staged kernel below 128 channels (1.29 times as fast on
// 23 such layers, 1.02 at the least: 3x3 on 32 channels at 112x112, batch 64, 134 -> 127 us), and from two and a half rounds
// of tiles on also above (1.05 to 1.13 on ten layers; 0.83 to 1.07 on 19 of fewer tiles.  256 channels at 28x28, batch 64,
// 61 -> 58 us; 64 -> 128 channels at 112x112 223 -> 194).  Not the smallest images: 1.03 to 1.9 on 97 layers of 3 to 12 rows with
// up to 1.25 images / E, 0.84 to 1.2 on 13 above (4x6 images, padded).
static bool runs_before_tiled(const Geometry& g, const RunsPlan& p) {
  return g.s == 1 && g.Kh == 3 && g.Kw == 3 && images_of_a_tile(g, p) <= 1.25 * p.E && (g.Co < 128 || (int64_t)p.ntm * p.ntn > 370);
}

// The same layer with another batch.
static Geometry with_batch(Geometry g, int32_t N) {
  g.N = N;
  g.P = (int64_t)N * g.Ho * g.Wo;
  g.window_elems = (int64_t)N * g.img_stride;
  g.out_elems = (int64_t)N * g.Co * g.Ho * g.Wo;
  g.plan_N = N;
  return g;
}

// What a kernel wants in scratch does not depend on the batch; whether it takes the layer does, and a kernel that takes a
// batch takes every smaller one.  So the plan for one image sizes the scratch, which then serves each part of a batch
// whichever kernel that part goes to.  `plan` is the plan for the whole batch (half the plans walk over many tiles).
template <typename Plan>
static Plan plan_for_any_batch(const Plan& plan, Plan (*make)(const Geometry&), const Geometry& g) {
  return plan.eligible || g.N == 1 ? plan : make(with_batch(g, 1));
}

// (The FFMA kernel's k-block is that of the images it runs on: its sums have one order in every form.)
im2win_status scratch_layout(const Geometry& part, im2win_dtype dtype, ScratchLayout* l) {
  const Geometry g = part.plan_N == part.N ? part : with_batch(part, part.plan_N);
  if (dtype == IM2WIN_F32) {
    l->Kp = round_up(g.K, plan_f32(part).bk);
    l->Co_pad = round_up(g.Co, plan_f32(part).bn);
  } else if (dtype == IM2WIN_F16) {
    l->Kp = round_up(g.K, kF16KBlock);
    l->Co_pad = g.Co;
  } else {
    return IM2WIN_ERR_INVALID_ARG;
  }
  l->f32_split = false;
  l->f16_runs = false;
  l->f16_shift = false;
  l->f16_raw = false;
  l->f16_mat = false;
  l->f16_stem = false;
  l->koff_off = kStatusBytes;
  l->filter_off = (size_t)round_up((int64_t)l->koff_off + 4 * l->Kp, 256);
  int64_t fbytes = l->Kp * l->Co_pad * (dtype == IM2WIN_F32 ? 4 : 2);
  l->total = (size_t)round_up((int64_t)l->filter_off + fbytes, 256);
  int64_t most = (int64_t)l->total;                        // of all layouts, whichever kernel is picked or forced
  if (dtype == IM2WIN_F32) {
    const F32SplitPlan split = plan_f32_split(g);
    l->f32_split = split.eligible && want_f32_split(g, split);
    l->ffma_total = l->total;
    const int64_t Kp = round_up(g.K, 32);                  // (the widest k-block of the FFMA kernel)
    most = round_up((int64_t)kStatusBytes + 4 * Kp, 256) + Kp * l->Co_pad * 4;
    const F32SplitPlan any = plan_for_any_batch(split, plan_f32_split, g);
    if (any.eligible) most = std::max(most, kStatusBytes + (int64_t)any.filter_bytes);
  }
  if (dtype == IM2WIN_F16) {
    // The shifted-view kernel is used whenever the layer is eligible; IM2WIN_F16_KERNEL=gather
    // forces the general gather kernel (a testing aid).
    const ShiftPlan plan = plan_f16_shift(g);
    const StemPlan stem = plan_f16_stem(g);
    const bool stem_ok = stem.eligible;                   // shares the filter layout of the shifted-view kernel
    const int64_t K2p = round_up((int64_t)g.C * g.Kh, kF16KBlock);
    const size_t shift_filter_off = (size_t)round_up((int64_t)kStatusBytes + 4 * K2p, 256);
    if (plan_for_any_batch(plan, plan_f16_shift, g).eligible || plan_for_any_batch(stem, plan_f16_stem, g).eligible)
      most = std::max(most, (int64_t)shift_filter_off + K2p * g.Co * g.Kw * 2);
    if (plan.eligible || stem_ok) {
      const char* force = debug_getenv("IM2WIN_F16_KERNEL");
      const bool use_shift = !(force && strcmp(force, "gather") == 0);
      if (use_shift) {
        l->f16_shift = plan.eligible;
        l->Kp = K2p;
        l->filter_off = shift_filter_off;
        // layers with one k-block: their own kernel unless another one is forced
        l->f16_stem = stem_ok && (!force || strcmp(force, "stem") == 0);
      }
    }
    const MatPlan mat = plan_f16_mat(g);                   // (takes its own scratch layout)
    const char* force = debug_getenv("IM2WIN_F16_KERNEL");
    // measured: the matrix-transpose kernel wins for strided layers (the others stage such layers
    // with 2-byte gathers) and for kernels up to 5 wide with 128 output channels or more (CTA pairs
    // above 128); IM2WIN_F16_KERNEL=mat forces it wherever it can run (a testing aid)
    const bool want = force ? strcmp(force, "mat") == 0 : (g.s > 1 || (g.Co >= 128 && g.Kw <= 5));
    l->f16_mat = mat.eligible && want && !l->f16_stem;
    const RunsPlan runs = plan_f16_runs(g);
    // (planes that are a multiple of 16 bytes: what the tiled-copy kernels need)
    if (!force && runs.eligible && !l->f16_stem && (g.chan_stride * 2) % 16 == 0 && runs_before_tiled(g, runs)) {
      l->f16_runs = true;
      l->f16_mat = false;
    }
    // the bulk-copy variant shares the filter layout of the shifted-view kernel; IM2WIN_F16_KERNEL=shift keeps the gathering one
    // (its plan walks over the tiles of an image: last)
    if (l->f16_shift && !l->f16_stem && !l->f16_mat && !l->f16_runs && !(force && strcmp(force, "shift") == 0))
      l->f16_raw = plan_f16_raw(g).eligible;
    const MatPlan any_mat = plan_for_any_batch(mat, plan_f16_mat, g);
    if (any_mat.eligible) most = std::max(most, (int64_t)any_mat.scratch_bytes);
    if (runs.eligible && !l->f16_runs) {
      const bool rest = !l->f16_stem && !l->f16_mat && !l->f16_raw;
      l->f16_runs = force ? strcmp(force, "runs") == 0 : rest && (!l->f16_shift || prefer_runs(g, runs));
    }
    const RunsPlan any_runs = plan_for_any_batch(runs, plan_f16_runs, g);
    if (any_runs.eligible) most = std::max(most, kStatusBytes + (int64_t)any_runs.filter_bytes);
  }
  l->total = (size_t)round_up(most, 256);
  return IM2WIN_OK;
}

static inline bool misaligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

// mode bit 0: pack the filter into scratch; bit 1: run the convolution on the packed filter.  plan_N: the batch that the
// shape's images are a part of (0: they are all of it).
enum { kDoPack = 1, kDoConv = 2 };
static im2win_status conv_common(const void* window, const void* filter, float* y, void* scratch,
                                 size_t scratch_bytes, const im2win_shape* shape, im2win_dtype dtype,
                                 void* cuda_stream, int mode = kDoPack | kDoConv, int32_t plan_N = 0) {
  if (!scratch || !shape) return IM2WIN_ERR_NULL_POINTER;
  if ((mode & kDoPack) && !filter) return IM2WIN_ERR_NULL_POINTER;
  if ((mode & kDoConv) && (!window || !y)) return IM2WIN_ERR_NULL_POINTER;
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  if (plan_N) g.plan_N = plan_N;
  ScratchLayout l;
  st = scratch_layout(g, dtype, &l);
  if (st != IM2WIN_OK) return st;
  if (misaligned(scratch) || ((mode & kDoPack) && misaligned(filter)) ||
      ((mode & kDoConv) && (misaligned(window) || misaligned(y))))
    return IM2WIN_ERR_MISALIGNED;
  if (scratch_bytes < l.total) return IM2WIN_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaSuccess;
  if (mode & kDoPack) {
    if (l.f32_split) e = launch_pack_f32_split(static_cast<const float*>(filter), scratch, g, stream);
    else if (dtype == IM2WIN_F32) e = launch_pack_f32(static_cast<const float*>(filter), scratch, g, l, stream);
    else if (l.f16_runs) e = launch_pack_f16_runs(static_cast<const uint16_t*>(filter), scratch, g, stream);
    else if (l.f16_stem) e = launch_pack_f16_shift(static_cast<const uint16_t*>(filter), scratch, g, l, stream);
    else if (l.f16_mat) e = launch_pack_f16_mat(static_cast<const uint16_t*>(filter), scratch, g, stream);
    else if (l.f16_raw)
      e = launch_pack_f16_raw(static_cast<const uint16_t*>(filter), scratch, g, l, plan_f16_raw(g), stream);
    else if (l.f16_shift) e = launch_pack_f16_shift(static_cast<const uint16_t*>(filter), scratch, g, l, stream);
    else e = launch_pack_f16(static_cast<const uint16_t*>(filter), scratch, g, l, stream);
    if (e != cudaSuccess) return IM2WIN_ERR_CUDA;
  }
  if (mode & kDoConv) {
    if (l.f32_split) e = launch_conv_f32_split(static_cast<const float*>(window), y, scratch, g, stream);
    else if (dtype == IM2WIN_F32) e = launch_conv_f32(static_cast<const float*>(window), y, scratch, g, l, stream);
    else if (l.f16_runs) e = launch_conv_f16_runs(static_cast<const uint16_t*>(window), y, scratch, g, stream);
    else if (l.f16_stem) e = launch_conv_f16_stem(static_cast<const uint16_t*>(window), y, scratch, g, l, stream);
    else if (l.f16_mat) e = launch_conv_f16_mat(static_cast<const uint16_t*>(window), y, scratch, g, stream);
    else if (l.f16_raw) e = launch_conv_f16_raw(static_cast<const uint16_t*>(window), y, scratch, g, l, stream);
    else if (l.f16_shift) e = launch_conv_f16_shift(static_cast<const uint16_t*>(window), y, scratch, g, l, stream);
    else e = launch_conv_f16_gather(static_cast<const uint16_t*>(window), y, scratch, g, l, stream);
  }
  return e == cudaSuccess ? IM2WIN_OK : IM2WIN_ERR_CUDA;
}

}  // namespace im2win

using namespace im2win;

extern "C" {

const char* im2win_status_string(im2win_status status) {
  switch (status) {
    case IM2WIN_OK: return "ok";
    case IM2WIN_ERR_INVALID_ARG: return "invalid argument";
    case IM2WIN_ERR_NULL_POINTER: return "null pointer";
    case IM2WIN_ERR_MISALIGNED: return "device pointer not 16-byte aligned";
    case IM2WIN_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
    case IM2WIN_ERR_UNSUPPORTED: return "shape beyond the kernels' index ranges";
    case IM2WIN_ERR_CUDA: return "CUDA error";
    case IM2WIN_ERR_TIMEOUT: return "bounded device wait gave up";
  }
  return "unknown status";
}

const char* im2win_conv_kernel_name(const im2win_shape* shape, im2win_dtype dtype) {
  Geometry g;
  ScratchLayout l;
  if (derive_geometry(shape, &g) != IM2WIN_OK || scratch_layout(g, dtype, &l) != IM2WIN_OK) return "none";
  if (dtype == IM2WIN_F32) return l.f32_split ? "f32-split" : "f32-ffma";
  if (l.f16_runs) return "f16-runs";
  if (l.f16_stem) return "f16-stem";
  if (l.f16_mat) return "f16-mat";
  if (l.f16_raw) return "f16-raw";
  if (l.f16_shift) return "f16-shift";
  return "f16-gather";
}

// A testing aid, not part of the interface: how the run-staged kernel would run a layer.  Returns whether it can.
int32_t im2win_f16_runs_form(const im2win_shape* shape, int32_t form[12]) {
  Geometry g;
  if (derive_geometry(shape, &g) != IM2WIN_OK) return 0;
  const RunsPlan p = plan_f16_runs(g);
  const int32_t v[12] = {p.mode, p.pair, p.planes, p.resident, p.teams, p.sr, p.octs, p.E, p.halo, p.bn, p.ntn, p.ntm};
  for (int i = 0; i < 12; ++i) form[i] = v[i];
  return p.eligible;
}

// The same: CTAs that share the reduction of a tile in the kernel that an fp16 layer takes.
int32_t im2win_f16_tile_ctas(const im2win_shape* shape) {
  Geometry g;
  ScratchLayout l;
  if (derive_geometry(shape, &g) != IM2WIN_OK || scratch_layout(g, IM2WIN_F16, &l) != IM2WIN_OK) return 0;
  if (l.f16_runs) return plan_f16_runs(g).split;
  return l.f16_shift && !l.f16_stem && !l.f16_mat && !l.f16_raw ? plan_f16_shift(g).split : 1;
}

// The same: CTAs of a cluster that a launcher takes for `want`, on a device that holds resident[z] clusters of z CTAs.
int32_t im2win_widest_cluster(int32_t want, const int32_t resident[17]) {
  return widest_cluster(want, [&](int z) { return resident[z] > 0; });
}

// The same: shared memory of a block of `threads` that an early launch of `blocks` asks for, which needs `smem`.
int64_t im2win_spread_smem(int64_t blocks, int32_t threads, int64_t smem) { return (int64_t)spread_smem(blocks, threads, (size_t)smem); }

// The same for the fp32 tensor-core kernel: channel tile, CTAs of a tile, parts of the last round's tiles.
int32_t im2win_f32_split_form(const im2win_shape* shape, int32_t form[3]) {
  Geometry g;
  if (derive_geometry(shape, &g) != IM2WIN_OK) return 0;
  const F32SplitPlan p = plan_f32_split(g);
  form[0] = p.bn; form[1] = p.split; form[2] = p.parts;
  return p.eligible;
}

im2win_status im2win_workspace_size(const im2win_shape* shape, im2win_dtype dtype, size_t* window_bytes,
                                    size_t* scratch_bytes, int32_t* Ho, int32_t* Wo) {
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  ScratchLayout l;
  st = scratch_layout(g, dtype, &l);
  if (st != IM2WIN_OK) return st;
  if (window_bytes) *window_bytes = (size_t)g.window_elems * (dtype == IM2WIN_F32 ? 4 : 2);
  if (scratch_bytes) *scratch_bytes = l.total;
  if (Ho) *Ho = g.Ho;
  if (Wo) *Wo = g.Wo;
  return IM2WIN_OK;
}

im2win_status im2win_transform(const void* x_nchw, void* window, const im2win_shape* shape,
                               im2win_dtype dtype, void* cuda_stream) {
  if (!x_nchw || !window || !shape) return IM2WIN_ERR_NULL_POINTER;
  if (dtype != IM2WIN_F32 && dtype != IM2WIN_F16) return IM2WIN_ERR_INVALID_ARG;
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  if (misaligned(x_nchw) || misaligned(window)) return IM2WIN_ERR_MISALIGNED;
  cudaError_t e = launch_transform(x_nchw, window, g, dtype == IM2WIN_F32 ? 4 : 2,
                                   static_cast<cudaStream_t>(cuda_stream));
  return e == cudaSuccess ? IM2WIN_OK : IM2WIN_ERR_CUDA;
}

im2win_status im2win_conv_f32(const float* window, const float* filter_oihw, float* y_nchw, void* scratch,
                              size_t scratch_bytes, const im2win_shape* shape, void* cuda_stream) {
  return conv_common(window, filter_oihw, y_nchw, scratch, scratch_bytes, shape, IM2WIN_F32, cuda_stream);
}

im2win_status im2win_conv_f16(const uint16_t* window, const uint16_t* filter_oihw, float* y_nchw,
                              void* scratch, size_t scratch_bytes, const im2win_shape* shape,
                              void* cuda_stream) {
  return conv_common(window, filter_oihw, y_nchw, scratch, scratch_bytes, shape, IM2WIN_F16, cuda_stream);
}

im2win_status im2win_pack_filter(const void* filter_oihw, void* scratch, size_t scratch_bytes,
                                 const im2win_shape* shape, im2win_dtype dtype, void* cuda_stream) {
  return conv_common(nullptr, filter_oihw, nullptr, scratch, scratch_bytes, shape, dtype, cuda_stream, kDoPack);
}

im2win_status im2win_conv_packed(const void* window, float* y_nchw, void* scratch, size_t scratch_bytes,
                                 const im2win_shape* shape, im2win_dtype dtype, void* cuda_stream) {
  return conv_common(window, nullptr, y_nchw, scratch, scratch_bytes, shape, dtype, cuda_stream, kDoConv);
}

// ---- channel-innermost (NHWC) form ------------------------------------------------------------
static im2win_status epilogue_args(const im2win_epilogue* e, bool nhwc_allowed, EpilogueArgs* out) {
  out->bias = nullptr; out->relu = 0; out->out16 = 0; out->y_nhwc = 0;
  if (!e) return IM2WIN_OK;
  if ((e->relu != 0 && e->relu != 1) || (e->out_dtype != IM2WIN_F32 && e->out_dtype != IM2WIN_F16) ||
      (e->out_layout != IM2WIN_LAYOUT_NCHW && e->out_layout != IM2WIN_LAYOUT_NHWC))
    return IM2WIN_ERR_INVALID_ARG;
  if (e->out_layout == IM2WIN_LAYOUT_NHWC && !nhwc_allowed) return IM2WIN_ERR_UNSUPPORTED;
  if (e->bias && (reinterpret_cast<uintptr_t>(e->bias) & 15u)) return IM2WIN_ERR_MISALIGNED;
  out->bias = e->bias; out->relu = e->relu; out->out16 = e->out_dtype == IM2WIN_F16;
  out->y_nhwc = e->out_layout == IM2WIN_LAYOUT_NHWC;
  return IM2WIN_OK;
}

static im2win_status nhwc_common(const uint16_t* window, const uint16_t* filter, void* y, const im2win_epilogue* epilogue,
                                 void* scratch, size_t scratch_bytes, const im2win_shape* shape, void* cuda_stream,
                                 int mode) {
  if (!scratch || !shape) return IM2WIN_ERR_NULL_POINTER;
  if ((mode & kDoPack) && !filter) return IM2WIN_ERR_NULL_POINTER;
  if ((mode & kDoConv) && (!window || !y)) return IM2WIN_ERR_NULL_POINTER;
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  const NhwcPlan plan = plan_nhwc(g);
  if (!plan.eligible) return IM2WIN_ERR_UNSUPPORTED;
  EpilogueArgs epi;
  st = epilogue_args(epilogue, true, &epi);
  if (st != IM2WIN_OK) return st;
  if (misaligned(scratch) || ((mode & kDoPack) && misaligned(filter)) ||
      ((mode & kDoConv) && (misaligned(window) || misaligned(y))))
    return IM2WIN_ERR_MISALIGNED;
  if (scratch_bytes < plan.scratch_bytes) return IM2WIN_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  if ((mode & kDoPack) && launch_pack_f16_nhwc(filter, scratch, g, stream) != cudaSuccess) return IM2WIN_ERR_CUDA;
  if ((mode & kDoConv) && launch_conv_f16_nhwc(window, y, scratch, g, epi, stream) != cudaSuccess) return IM2WIN_ERR_CUDA;
  return IM2WIN_OK;
}

const char* im2win_nhwc_kernel_name(const im2win_shape* shape, const im2win_epilogue* epilogue) {
  Geometry g;
  EpilogueArgs epi;
  if (!shape || derive_geometry(shape, &g) != IM2WIN_OK || epilogue_args(epilogue, true, &epi) != IM2WIN_OK) return "none";
  return nhwc_kernel_name(g, epi);
}

im2win_status im2win_nhwc_workspace_size(const im2win_shape* shape, size_t* window_bytes, size_t* scratch_bytes,
                                         int32_t* Ho, int32_t* Wo, int32_t* Cp) {
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  const NhwcPlan plan = plan_nhwc(g);
  if (!plan.eligible) return IM2WIN_ERR_UNSUPPORTED;
  if (window_bytes) *window_bytes = (size_t)plan.window_elems * 2;
  if (scratch_bytes) *scratch_bytes = plan.scratch_bytes;
  if (Ho) *Ho = g.Ho;
  if (Wo) *Wo = g.Wo;
  if (Cp) *Cp = plan.Cp;
  return IM2WIN_OK;
}

im2win_status im2win_transform_nhwc(const uint16_t* x, im2win_layout x_layout, uint16_t* window,
                                    const im2win_shape* shape, void* cuda_stream) {
  if (!x || !window || !shape) return IM2WIN_ERR_NULL_POINTER;
  if (x_layout != IM2WIN_LAYOUT_NCHW && x_layout != IM2WIN_LAYOUT_NHWC) return IM2WIN_ERR_INVALID_ARG;
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  if (!plan_nhwc(g).eligible) return IM2WIN_ERR_UNSUPPORTED;
  if (misaligned(x) || misaligned(window)) return IM2WIN_ERR_MISALIGNED;
  cudaError_t e = launch_transform_nhwc(x, x_layout == IM2WIN_LAYOUT_NHWC, window, g, static_cast<cudaStream_t>(cuda_stream));
  return e == cudaSuccess ? IM2WIN_OK : IM2WIN_ERR_CUDA;
}

im2win_status im2win_conv_f16_nhwc(const uint16_t* window, const uint16_t* filter_oihw, void* y,
                                   const im2win_epilogue* epilogue, void* scratch, size_t scratch_bytes,
                                   const im2win_shape* shape, void* cuda_stream) {
  return nhwc_common(window, filter_oihw, y, epilogue, scratch, scratch_bytes, shape, cuda_stream, kDoPack | kDoConv);
}

im2win_status im2win_pack_filter_nhwc(const uint16_t* filter_oihw, void* scratch, size_t scratch_bytes,
                                      const im2win_shape* shape, void* cuda_stream) {
  return nhwc_common(nullptr, filter_oihw, nullptr, nullptr, scratch, scratch_bytes, shape, cuda_stream, kDoPack);
}

im2win_status im2win_conv_packed_nhwc(const uint16_t* window, void* y, const im2win_epilogue* epilogue,
                                      void* scratch, size_t scratch_bytes, const im2win_shape* shape,
                                      void* cuda_stream) {
  return nhwc_common(window, nullptr, y, epilogue, scratch, scratch_bytes, shape, cuda_stream, kDoConv);
}

im2win_status im2win_check_status(const void* scratch, void* cuda_stream) {
  if (!scratch) return IM2WIN_ERR_NULL_POINTER;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  uint32_t word = 0;
  if (cudaMemcpyAsync(&word, scratch, sizeof(word), cudaMemcpyDeviceToHost, stream) != cudaSuccess)
    return IM2WIN_ERR_CUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess) return IM2WIN_ERR_CUDA;
  return word ? IM2WIN_ERR_TIMEOUT : IM2WIN_OK;
}

namespace {
// Two auxiliary streams per device for the chunked host-to-host path (created on first use and kept
// for the life of the process; the only state the library keeps besides the static scratch array).
struct AuxStreams {
  cudaStream_t in, out;
};
bool get_aux_streams(AuxStreams* a) {
  static std::mutex mu;
  static AuxStreams cache[64];
  static bool have[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (!have[dev]) {
    if (cudaStreamCreateWithFlags(&cache[dev].in, cudaStreamNonBlocking) != cudaSuccess) return false;
    if (cudaStreamCreateWithFlags(&cache[dev].out, cudaStreamNonBlocking) != cudaSuccess) {
      cudaStreamDestroy(cache[dev].in);
      return false;
    }
    have[dev] = true;
  }
  *a = cache[dev];
  return true;
}

struct LayerLayout {
  size_t x_off, f_off, win_off, scratch_off, y_off, total;
  size_t x_bytes, f_bytes, win_bytes, scratch_bytes, y_bytes;
};
im2win_status layer_layout(const Geometry& g, im2win_dtype dtype, LayerLayout* L) {
  ScratchLayout l;
  im2win_status st = scratch_layout(g, dtype, &l);
  if (st != IM2WIN_OK) return st;
  const size_t es = dtype == IM2WIN_F32 ? 4 : 2;
  L->x_bytes = (size_t)g.N * g.C * g.H * g.W * es;
  L->f_bytes = (size_t)g.Co * g.K * es;
  L->win_bytes = (size_t)g.window_elems * es;
  L->scratch_bytes = l.total;
  L->y_bytes = (size_t)g.out_elems * 4;
  auto up = [](size_t v) { return (v + 255) / 256 * 256; };
  L->x_off = 0;
  L->f_off = L->x_off + up(L->x_bytes);
  L->win_off = L->f_off + up(L->f_bytes);
  L->scratch_off = L->win_off + up(L->win_bytes);
  L->y_off = L->scratch_off + up(L->scratch_bytes);
  L->total = L->y_off + up(L->y_bytes);
  return IM2WIN_OK;
}
}  // namespace

im2win_status im2win_layer_workspace_size(const im2win_shape* shape, im2win_dtype dtype, size_t* device_bytes) {
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  LayerLayout L;
  st = layer_layout(g, dtype, &L);
  if (st != IM2WIN_OK) return st;
  if (device_bytes) *device_bytes = L.total;
  return IM2WIN_OK;
}

im2win_status im2win_layer_forward_host(const void* x_host, const void* filter_host, float* y_host,
                                        void* device_workspace, size_t device_workspace_bytes,
                                        const im2win_shape* shape, im2win_dtype dtype, void* cuda_stream) {
  if (!x_host || !filter_host || !y_host || !device_workspace || !shape) return IM2WIN_ERR_NULL_POINTER;
  Geometry g;
  im2win_status st = derive_geometry(shape, &g);
  if (st != IM2WIN_OK) return st;
  LayerLayout L;
  st = layer_layout(g, dtype, &L);
  if (st != IM2WIN_OK) return st;
  if ((reinterpret_cast<uintptr_t>(device_workspace) & 255u) != 0) return IM2WIN_ERR_MISALIGNED;
  if (device_workspace_bytes < L.total) return IM2WIN_ERR_WORKSPACE_TOO_SMALL;
  unsigned char* ws = static_cast<unsigned char*>(device_workspace);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const size_t es = dtype == IM2WIN_F32 ? 4 : 2;

  // Large layers are cut into batch chunks so that the upload of chunk i+1, the kernels of chunk
  // i and the download of chunk i-1 overlap (the two copy directions run concurrently on the
  // link).  Chunks start at images whose slices of x, window and y are 16-byte aligned.
  const size_t x_img = (size_t)g.C * g.H * g.W * es, w_img = (size_t)g.img_stride * es,
               y_img = (size_t)g.Co * g.Ho * g.Wo * 4;
  int unit = 1;                                   // images per alignment unit
  while (unit <= 8 && ((unit * x_img) % 16 || (unit * w_img) % 16 || (unit * y_img) % 16)) unit *= 2;
  int nchunk = 1;
  AuxStreams aux{};
  if (unit <= 8 && g.N >= 4 * unit && L.x_bytes + L.y_bytes >= ((size_t)8 << 20) && get_aux_streams(&aux)) nchunk = 4;
  if (nchunk == 1) {
    if (cudaMemcpyAsync(ws + L.x_off, x_host, L.x_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess)
      return IM2WIN_ERR_CUDA;
    if (cudaMemcpyAsync(ws + L.f_off, filter_host, L.f_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess)
      return IM2WIN_ERR_CUDA;
    st = im2win_transform(ws + L.x_off, ws + L.win_off, shape, dtype, cuda_stream);
    if (st != IM2WIN_OK) return st;
    st = conv_common(ws + L.win_off, ws + L.f_off, reinterpret_cast<float*>(ws + L.y_off), ws + L.scratch_off,
                     L.scratch_bytes, shape, dtype, cuda_stream);
    if (st != IM2WIN_OK) return st;
    if (cudaMemcpyAsync(y_host, ws + L.y_off, L.y_bytes, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
      return IM2WIN_ERR_CUDA;
    return IM2WIN_OK;
  }

  // Everything the auxiliary streams do is ordered after the work already queued on `stream`, and
  // `stream` ends up waiting for the last download, so the caller still only synchronises `stream`.
  cudaEvent_t ev;
  auto fence = [&](cudaStream_t from, cudaStream_t to) -> bool {      // `to` waits for what `from` has queued
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return false;
    const bool ok = cudaEventRecord(ev, from) == cudaSuccess && cudaStreamWaitEvent(to, ev, 0) == cudaSuccess;
    cudaEventDestroy(ev);                                              // released once it has completed
    return ok;
  };
  const int per = ((g.N + nchunk - 1) / nchunk + unit - 1) / unit * unit;
  // Chunks run the kernel that the whole batch would, with its order of the sums, so that the result is that of the whole.
  // Every distinct chunk size is validated before anything is queued: its geometry must derive and
  // the scratch its kernels want must fit the scratch that was sized for the whole batch.
  for (int n0 = 0; n0 < g.N; n0 += per) {
    im2win_shape part = *shape;
    part.N = n0 + per < g.N ? per : g.N - n0;
    Geometry gp;
    ScratchLayout lp;
    st = derive_geometry(&part, &gp);
    gp.plan_N = g.N;
    if (st == IM2WIN_OK) st = scratch_layout(gp, dtype, &lp);
    if (st != IM2WIN_OK) return st;
    if (lp.total > L.scratch_bytes) return IM2WIN_ERR_WORKSPACE_TOO_SMALL;
  }
  if (!fence(stream, aux.in) || !fence(stream, aux.out)) return IM2WIN_ERR_CUDA;
  // From here on work is queued on the auxiliary streams: on any failure `stream` is still made to
  // wait for both of them, so that synchronising `stream` completes whatever was queued.
  im2win_status result = IM2WIN_OK;
  if (cudaMemcpyAsync(ws + L.f_off, filter_host, L.f_bytes, cudaMemcpyHostToDevice, aux.in) != cudaSuccess)
    result = IM2WIN_ERR_CUDA;
  for (int n0 = 0; n0 < g.N && result == IM2WIN_OK; n0 += per) {
    const int n1 = n0 + per < g.N ? n0 + per : g.N;
    im2win_shape part = *shape;
    part.N = n1 - n0;
    unsigned char* xd = ws + L.x_off + (size_t)n0 * x_img;
    unsigned char* wd = ws + L.win_off + (size_t)n0 * w_img;
    unsigned char* yd = ws + L.y_off + (size_t)n0 * y_img;
    if (cudaMemcpyAsync(xd, static_cast<const unsigned char*>(x_host) + (size_t)n0 * x_img, (size_t)part.N * x_img,
                        cudaMemcpyHostToDevice, aux.in) != cudaSuccess || !fence(aux.in, stream)) {
      result = IM2WIN_ERR_CUDA;
      break;
    }
    result = im2win_transform(xd, wd, &part, dtype, cuda_stream);
    if (result != IM2WIN_OK) break;
    result = conv_common(wd, ws + L.f_off, reinterpret_cast<float*>(yd), ws + L.scratch_off, L.scratch_bytes, &part,
                         dtype, cuda_stream, kDoPack | kDoConv, g.N);
    if (result != IM2WIN_OK) break;
    if (!fence(stream, aux.out) ||
        cudaMemcpyAsync(reinterpret_cast<unsigned char*>(y_host) + (size_t)n0 * y_img, yd, (size_t)part.N * y_img,
                        cudaMemcpyDeviceToHost, aux.out) != cudaSuccess)
      result = IM2WIN_ERR_CUDA;
  }
  const bool joined = fence(aux.out, stream) & fence(aux.in, stream);
  if (result == IM2WIN_OK && !joined) result = IM2WIN_ERR_CUDA;
  return result;
}

}  // extern "C"
