// The plan of a launch of the tensor-core kernel (snn_tcg.cu): what a problem is to the kernel, the tile of each problem,
// the ring geometry all of them share, and which CTAs take which tiles.  Host code only, without CUDA calls: the kernel's
// source includes it, and so can a program without a GPU.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

#include "snn_internal.h"

namespace snn {
namespace {

// Division of a numerator below 2^31 by a run-time constant d below 2^31: q / d = (2q * m) >> (32 + s) with 2^s >= d and
// m = floor(2^(31 + s) / d) + 1.  m exceeds 2^(31 + s) / d by at most 1, so the quotient by at most q * 2^-(31 + s) < 2^-s <= 1 / d: exact.
struct FastDiv {
  uint32_t m, s;
};
FastDiv make_fastdiv(uint32_t d) {
  FastDiv f;
  f.s = 0;
  while ((1ull << f.s) < d) ++f.s;
  f.m = (uint32_t)((1ull << (31 + f.s)) / d + 1);
  return f;
}
inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Operand modes of the kernel.  Binary activations run on 4-bit e2m1 operands (+1 / -1 / 0 are exact, the
// block scales are all 1, and the fp32 accumulators hold the exact integer sums: |S| <= 9 * c_in < 2^24);
// an MMA then covers 64 input channels in the time an 8-bit MMA covers 32.  fp16 activations run on fp16
// operands.  Both accumulate in fp32.
enum { M_F16 = 1, M_FP4 = 2 };
constexpr int G_EW = 8;                       // epilogue warps = expander warps

// Warps 13 and 17 do not expand: a warp's scheduler is warp % 4, and the MMA-issuing warp (1) then shares its
// scheduler with two epilogue warps and the table warp (13, which has little to do) instead of two expander warps.
constexpr int G_THREADS = 64 + 64 * G_EW + 64;
constexpr int G_EXP_THREADS = 32 * G_EW;
constexpr int G_XTEAMS = 2;                    // teams of expander warps (4-bit operands)
constexpr int G_EXP_ITEMS = 4;                 // loads one expander thread has in flight together
constexpr int G_ROWS = 128;                    // rows of the weight operand: lanes of an accumulator
constexpr int G_MAX_CHUNKS = 8;                // 32-column slices of an accumulator (at most 256 columns)
// What the epilogue needs to know of a tile, written by the table warp (see there), four tiles deep.
struct GTile {
  int l, mg, co, n_slices;             // problem (-1: no more tiles), position tile, first channel, 32-column slices
  int K, kp_log, lg, out_kind;         // channels; GLayer::kp_log, lg (fp16: whether the rows hold pairs, GLayer::pair); GParams::out_type,
                                       // + 4: the epilogue advances the tile's counter itself, + 8: the CTA's last tile
  uint32_t offset[G_MAX_CHUNKS * 32];  // per column: first output pixel, times K for word outputs
  uint32_t mask[G_MAX_CHUNKS * 8];     // [pixel of the group][slice]: which columns' pixel exists
  float alpha[G_ROWS], minus_threshold[G_ROWS];
};
constexpr int G_TILES = 4;
constexpr int G_EPI_BYTES = G_TILES * (int)sizeof(GTile);
constexpr int G_NS_MAX = 8;
constexpr uint32_t G_TMEM_FP4 = 480;          // 4-bit mode: columns 480..511 hold the (unit) block scales
constexpr uint32_t G_TMEM_F16 = 512;
constexpr uint32_t G_SCALE_COL = 480;
constexpr size_t kGTail = 512;
constexpr size_t kGSmemBudget = 226 * 1024;
constexpr uint32_t kGASlotMax = 44 * 1024;         // largest activation unit a problem may stage
constexpr uint32_t kGASlotMaxTma = 60 * 1024;      // ... when it is fetched by TMA (fp16; whole rows of positions)
constexpr int kGRowsMax = 1600;                    // ... and its most rows (the pixel tables hold one word per row)
constexpr uint32_t kGBSlot = 32 * 1024, kGBSlotF16 = 16 * 1024;   // bytes of a weight-stage slot
constexpr int kGTapsMax = 52;                      // 3 kernel rows x at most 17 columns of a group of 8 pixels

// One problem of a launch, as the kernel reads it from shared memory.
struct GLayer {
  const uint8_t* wt;      // [channel tile][channel block][step][chunk][128][16 B], owned by the group
  const float* alpha;
  const float* threshold; // packed-sign output: per channel, the sum its bit changes at (g_sign_threshold)
  int N, H, W, C, K, Cw, pad, Ho, Wo;
  int rs, cm, cs;         // input pixel of position (i, j) in plane (pr, pc): row rs*i + pr - pad, column cm*j + cs*pc - pad
  int G, lg;              // output pixels per position and its logarithm
  int Hq, Wg;             // rows per image / positions per row of the flattened position space
  FastDiv dWg, dHq, dCt, dRr;
  int n_planes, cpl;      // planes of a unit, logarithm of the number of column planes
  int Np, Rr;             // positions per tile; staged rows per plane = Np + largest tap shift
  int cb_chunks, n_cb, kpt;
  int tma;                // fp16: units are fetched by TMA, rows of 64 channels in the 128-byte swizzle
  int n_pu, pu_end[4];    // units per channel block (fetched by TMA, each plane is a unit of its own) and the last step of each
  int steps;              // taps of a tile, or pairs of taps (one activation word per pixel: a K = 64 step covers two taps)
  int st_steps;           // steps per weight stage (the last stage of a channel block holds steps % st_steps, if not 0)
  int kp_log;             // logarithm of the rows of the weight operand that hold the channels once: of each pixel of a group, or
                          // - with single pixels - of each copy of the channels
  uint32_t step_bytes;    // weights of one step of one channel block = kpt * 2 * 128 * 16
  int n_ct, total_tiles;  // channel tiles of 128
  int first;              // this CTA's first tile, filled in by the kernel (GParams::ranks)
  uint32_t Qtot;
  int pair;               // fp16, 33 to 64 output channels: the rows of the weight operand hold two columns of the kernel (see g_pairs); a tile's last
                          // position is not its own then
  // A chain (every member reads the packed signs its predecessor writes, all in one launch): a tile may be
  // staged once the predecessor's tiles that hold its input pixels are complete, and says so itself when done.
  const uint2* deps;          // [position tiles] first and last position tile of the predecessor this one reads (x > y: none)
  const uint32_t* prev_done;  // the predecessor's completion counters, and the count that means "complete"
  uint32_t prev_target;
  int next;                   // the next problem in which this CTA has a tile, filled in as `first` is
  uint32_t* done;             // [position tiles] epilogue warps that have written their part, over all its channel tiles
  uint32_t tap[kGTapsMax];    // per step: start of its rows in the unit (16-byte units) | distance of its two chunks << 16
};

// The launches of a chain of words with tags, counted in one number in device memory: every CTA adds its share when it ends, the
// shares of a launch make 2^32, and the upper half is what all CTAs of the next launch take their tag from.  (A count per CTA
// would never come together again once launches that must not overlap did; this one is whole whenever all have ended.)
struct GLaunches {
  unsigned long long* count;
  unsigned long long share;   // each CTA's; CTA 0 adds what they leave of 2^32 on top
};
inline GLaunches g_launches(unsigned long long* count, uint32_t ctas) { return {count, (1ull << 32) / ctas}; }
__host__ __device__ inline unsigned long long g_launch_share(const GLaunches& l, uint32_t cta, uint32_t ctas) {
  return cta ? l.share : (1ull << 32) - l.share * (ctas - 1);
}

struct GParams {
  const GLayer* layers;
  const uint32_t* ranks;  // [n_layers][grid] CTA b takes a problem's tiles r, r + grid, ... (r: lower half of ranks[b]); upper half:
                          // the next problem in which it has a tile (n_layers: none)
  int n_layers;
  const void* act[SNN_GROUP_MAX];
  void* out[SNN_GROUP_MAX];
  int* status;
  GLaunches launches;     // chain of words with tags
  uint8_t out_type[SNN_GROUP_MAX];   // per member: 0 fp32 alpha*S, 1 int32 S, 2 packed signs of alpha*S + shift, 3 those with tags
  uint32_t acc_cols;      // tensor-memory columns of one accumulator buffer
  int n_acc;              // accumulator buffers (tile seq of a CTA uses buffer seq % n_acc)
  int NA, NS;
  uint32_t a_slot_bytes, b_slot_bytes;
  uint32_t off_b, off_epi, off_pix, off_lay, off_tail;
  int after_weights;      // the launch before this one in the stream writes the weights (2: and the scales): wait for it before they are read
  GLayer one;             // n_layers == 1: the problem itself (layers and ranks are not read: its tiles go to the CTAs in order)
};

// input pixel of row q (a position, possibly past a tile's own) in plane pl, or -1: padding or past the batch
__host__ __device__ __forceinline__ int g_pixel_of(const GLayer& L, uint32_t n, int i, int j, int pl) {
  const int r = L.rs * i + (pl >> L.cpl) - L.pad, c = L.cm * j + L.cs * (pl & ((1 << L.cpl) - 1)) - L.pad;
  if (r < 0 || r >= L.H || c < 0 || c >= L.W) return -1;
  return ((int)n * L.H + r) * L.W + c;
}

// What the sign epilogue adds to a sum: minus the threshold it is compared with.  A threshold of 0 gives +0, so that a sum of 0 is at it whichever sign
// the tensor core gives a zero.
__host__ __device__ inline float g_minus_threshold(float threshold) { return 0.f - threshold; }

// Words of a row that are loaded together: activations are 16-byte aligned, so a row can be read four (two) words
// at a time where the words per pixel and per channel block are multiples of four (two).
__host__ __device__ __forceinline__ int g_word_step(int Cw, int cb_chunks) {
  return (Cw & 3) == 0 && (cb_chunks & 3) == 0 ? 4 : (Cw & 1) == 0 && (cb_chunks & 1) == 0 ? 2 : 1;
}

// Which tap each step of a layer applies, for the weight operand: per chunk of a step the kernel row and the column
// s of the group's window (kernel column s - stride*g for pixel g), 255: none.  Steps of single taps name one tap twice.
struct GTaps {
  uint8_t row[kGTapsMax][2], col[kGTapsMax][2];
};

inline int g_mode_for(int act_type) { return act_type == SNN_ACT_F16 ? M_F16 : M_FP4; }

// A planned layer and the planner's estimate of one tile, in SM cycles.
struct GPlan {
  GLayer L;
  GTaps taps;
  int paired = 0;
  size_t w_bytes = 0, unit_bytes = 0;
  double mma = 0, weights = 0, expand = 0, drain = 0;
  double through() const {   // a tile among others: the slowest role
    double t = mma;
    if (weights > t) t = weights;
    if (expand > t) t = expand;
    if (drain > t) t = drain;
    return t + 300.0;
  }
  double alone() const { return expand + (mma > weights ? mma : weights) + drain + 1500.0; }   // a tile by itself
  // The end of a launch of this layer alone: staging and stores have the time they take with idle neighbours (below).
  double mma_one = 0, stage_one = 0, drain_one = 0;
  int loads = 0;   // loads an expander thread does in a row for one unit
  double end(int sms) const {
    const int waves = (L.total_tiles + sms - 1) / sms;
    const double work = std::max(mma_one, weights);
    return stage_one + work + 0.7 * drain_one + 1500.0 + (waves - 1) * (std::max(work, std::max(stage_one, drain_one)) + 300.0);
  }
};

// Two columns of a 3x3 kernel in the rows of the weight operand (fp16 units fetched by TMA, 33 to 64 output channels, stride 1).  With single pixels
// half of the 128 rows would be idle, and groups of pixels need zeros where a column is outside a pixel's window, which times an infinity
// are no zeros.  Rows 32*q + 0..15 are channels 16*q.. with one column of the kernel, rows 32*q + 16..31 the same channels with the next one:
// both are multiplied with the same positions, so the upper rows' sum of a position stands one column of the accumulator on, and the
// epilogue puts the two together.  Of a kernel row's two steps the first has columns 0 and 1, the second columns 1 and 2: the middle
// column is there twice, with weights of one half (products and sums of halves are as exact as those of ones), so that no row needs a
// zero, an infinity reaches the outputs whose windows hold it and no others, and all instructions that add into an accumulator
// have one shape - those of two shapes would not be ordered among one another.  6 steps instead of 9; all eight epilogue
// warps have channels, too.  us without pairs and with: fp16 ResNet-18 group at batch 64 248 and 232, 8 38.1 and 36.2; 64 channels of 56x56,
// 8 images 6.7 and 6.1; 32 to 64 channels of 28x28 4.5 and 4.2; 16 to 64 4.3 and 4.2, 24 to 64 of 56x56 14.4 and 14.3.  Error against 64
// bits: 64 channels 5.9e-8 and 5.2e-8, 512 5.1e-7 and 3.5e-7, 32 3.4e-8 and 3.2e-8, 16 1.85e-8 and 1.96e-8: not below 32 channels, where there is next to
// nothing to gain.  (At stride 2 the middle column is in a plane of its own, where the next position's window does not reach.)
inline bool g_pairs(const Geom& g, bool tma) { return tma && g.ksize == 3 && g.stride == 1 && g.C >= 32 && g.K > 32 && g.K <= 64; }
// Row r of the weight operand in a step whose lower rows hold kernel column `col` (0 or 1).
struct GPairRow {
  int channel, column, halves;   // (weight: so many halves)
};
__host__ __device__ inline GPairRow g_pair_row(int r, int col) {
  const int column = col + (r >> 4 & 1);
  return {(r >> 5) * 16 + (r & 15), column, column == 1 ? 1 : 2};
}

// The plan of one layer with tiles of Np positions of 2^lg pixels and blocks of at most max_chunks 16-byte chunks of channels; false
// where that does not fit.
bool g_plan_layer(const Geom& g, int mode, int kind, int lg, int Np, bool tma, GPlan* P, int max_chunks = 8) {
  GLayer& o = P->L;
  o.wt = nullptr; o.alpha = o.threshold = nullptr; o.deps = nullptr; o.prev_done = nullptr; o.prev_target = 0; o.done = nullptr;
  o.first = 0;
  o.next = 1;   // (as it is in a launch of one problem)
  const int cpc = mode == M_F16 ? 8 : 32;
  const int S = g.stride, G = 1 << lg;
  const bool one = g.ksize == 1;
  o.N = g.N; o.H = g.H; o.W = g.W; o.C = g.C; o.K = g.K; o.Cw = g.Cw;
  o.pad = g.pad; o.Ho = g.Ho; o.Wo = g.Wo; o.G = G; o.lg = lg; o.Np = Np;
  if (lg && (mode != M_FP4 || g.K > G_ROWS >> lg)) return false;
  o.rs = S;
  o.cs = one ? S : 1;
  o.cm = S * G;
  int row_planes = 1, col_planes = G;
  if (one) {
    // 1x1 layer: the positions are (groups of) the output pixels themselves, no halo
    o.Hq = g.Ho;
    o.Wg = (g.Wo + G - 1) / G;
  } else {
    // one zero column per image row and one zero row per image are shared by neighbours; stride 2 splits the input
    // into its row and column parity planes, in each of which the taps are plain shifts
    row_planes = S;
    col_planes = S * G;
    o.Hq = S == 1 ? g.H + g.pad : g.Ho + 1;
    o.Wg = ((S == 1 ? g.W + g.pad : g.Wo + 1) + G - 1) / G;
  }
  o.n_planes = row_planes * col_planes;
  o.cpl = 0;
  while ((1 << o.cpl) < col_planes) ++o.cpl;
  const long long Q = (long long)g.N * o.Hq * o.Wg;
  const int span = one ? S * (G - 1) + 1 : S * (G - 1) + 3;   // columns of a group's window, in input pixels
  const int halo = one ? 0 : (2 / S) * o.Wg + (span - 1) / col_planes;
  if (Q + 1024 + halo >= (1ll << 31)) return false;
  o.Qtot = (uint32_t)Q;
  o.Rr = Np + halo;
  // fp16 units are fetched by TMA where the rows of the tensor are multiples of 16 bytes and a row of positions fits a box
  o.tma = tma && mode == M_F16 && (g.C & 7) == 0 && o.Wg * S <= 256;
  o.pair = g_pairs(g, o.tma != 0) ? 1 : 0;
  const int tma_rows = (2 * o.Wg + o.Rr - 2) / o.Wg;   // rows of positions a tile can touch
  if (mode == M_F16 && !o.tma) o.Rr |= 1;   // odd: the chunks of a row are copied together, into different banks
  if (!o.tma && (long long)o.n_planes * o.Rr > kGRowsMax) return false;
  P->paired = mode == M_FP4 && g.Cw == 1;
  int d = 0;
  if (o.tma) {
    // 64 channels (fewer where there are no more); every plane is a unit of its own
    P->unit_bytes = (size_t)tma_rows * o.Wg * 128;
    if (P->unit_bytes > kGASlotMaxTma) return false;
    o.n_cb = (g.C + 63) / 64;
    d = o.n_cb > 1 ? 8 : round_up(g.C, 16) / 8;
    o.cb_chunks = d;
    o.kpt = d / 2;
    o.n_pu = o.n_planes;
  } else {
    // channel block: the largest of 8/6/4/2 chunks that divides the channels and whose unit fits a slot; one chunk where
    // there is one activation word per pixel: a K = 64 step then covers two taps, one per chunk
    const int raw = P->paired ? 1 : round_up(g.C, 2 * cpc) / cpc;  // 16-byte chunks along the channels, even
    for (int c = P->paired ? 1 : max_chunks; c >= 1; c -= 2) {
      if (raw % c) continue;
      if ((size_t)o.n_planes * c * o.Rr * 16 <= kGASlotMax) { d = c; break; }
    }
    if (!d) return false;
    o.cb_chunks = d;
    o.n_cb = raw / d;
    o.kpt = P->paired ? 1 : d / 2;
    o.n_pu = 1;
    P->unit_bytes = (size_t)o.n_planes * d * o.Rr * 16;
  }
  const int taps = one ? G : o.pair ? 6 : 3 * span;
  o.steps = P->paired ? (taps + 1) / 2 : taps;
  if (o.steps >= kGTapsMax) return false;
  const uint32_t reach = o.tma ? 8u * (uint32_t)halo : (uint32_t)(o.n_planes * o.Rr);   // largest start of a tap, and chunk distance
  if (reach > 0xffffu || (!o.tma && reach >= (1u << 14))) return false;                 // (the leading-offset field has 14 bits)
  o.n_ct = lg ? 1 : (g.K + G_ROWS - 1) / G_ROWS;
  const int own = Np - o.pair;   // positions a tile gives the sums of
  const long long tiles = (Q + own - 1) / own * o.n_ct;
  if (tiles > 0x7fffffffLL || (Q + own - 1) / own * o.Rr >= (1ll << 31)) return false;
  o.total_tiles = (int)tiles;
  // weight stage: as many whole steps of a channel block as fit a slot
  o.step_bytes = (uint32_t)(o.kpt * 2 * G_ROWS * 16);
  o.st_steps = (int)((mode == M_F16 ? kGBSlotF16 : kGBSlot) / o.step_bytes);
  if (o.st_steps > o.steps) o.st_steps = o.steps;
  P->w_bytes = (size_t)o.n_ct * o.n_cb * o.steps * o.step_bytes;
  // One MMA reads 32 + Np/4 shared-memory lines and takes at least Np/2 cycles (measured).  The other figures are set by
  // hand after traces of single roles, for launches that keep every SM busy: bulk copies of weights 64 bytes a cycle, a
  // 16-byte chunk of activations 0.6 cycles (3 where fp16 is copied by the threads) and 500 a block of channels, units
  // fetched by TMA 40 bytes a cycle and 1000 for the first, stores 16 bytes a cycle, signs 5 cycles a position.
  const double mmas = (double)o.n_cb * o.steps * o.kpt;
  const double lines = mmas * (32 + Np / 4) + (double)o.n_cb * (o.steps * o.step_bytes + (double)o.n_pu * P->unit_bytes) / 128.0;
  P->mma = std::max(mmas * (Np / 2), 1.1 * lines);
  P->weights = (double)o.n_cb * o.steps * o.step_bytes / 64.0;
  // Single pixels of at most 64 channels: a warp reads its own quarter's lanes only, and two or four of the eight would write
  // the whole tile, at 24 cycles a column.  Where that takes longer than the tile's MMAs, the other rows hold copies of the
  // channels and warps of all lane quarters share the columns (fp16, 16 channels of 32x32 maps at batch 128: 13.8 us, with
  // copies 9.7).  Elsewhere they stay zeros, which take less power (64 channels of 56x56: 3 % of the launch).
  const int slices = (Np + 31) / 32;
  const bool copies = lg == 0 && g.K <= 64 && P->mma < 24.0 * std::min(Np, 32 * ((slices + 1) / 2));
  o.kp_log = lg ? 7 - lg : !copies ? 7 : g.K <= 32 ? 5 : 6;
  P->expand = o.tma ? o.n_cb * o.n_pu * (P->unit_bytes / 40.0) + 1000.0 : o.n_cb * ((double)o.n_planes * o.Rr * d * (mode == M_F16 ? 3.0 : 0.6) + 500.0);
  const int k_tile = g.K < G_ROWS ? g.K : G_ROWS;
  P->drain = kind == TCG_WORDS ? (double)Np * G * k_tile * 4 / 16.0 : Np * 5.0;
  // In a launch of this layer alone little else waits for memory: what counts is how many loads one thread does in a row
  // (200 cycles each; 0.2 a chunk where they are many), and the stores go to L2 at 32 bytes a cycle, 24 cycles a column and
  // 250 a slice of signs for the warp that has the most of them.  Fitted to 7,500 plans: all widths and group sizes of 384
  // layers of 16 to 512 channels, maps of 6 to 57, 1 to 128 images.
  const int team = G_EXP_THREADS / G_XTEAMS, word_step = g_word_step(g.Cw, d);
  P->loads = (o.Rr + team - 1) / team * o.n_planes * ((d + word_step - 1) / word_step);
  const int sharing = lg ? 2 : 2 * (G_ROWS >> o.kp_log), most = (slices + sharing - 1) / sharing;
  P->mma_one = mmas * std::max(Np / 2.0, 1.1 * (32 + Np / 4.0));
  P->stage_one = mode == M_F16 ? P->expand : o.n_cb * std::max(0.2 * o.n_planes * o.Rr * d, 200.0 * P->loads);
  P->drain_one = kind == TCG_WORDS ? std::max((double)Np * G * k_tile * 4 / 32.0, 24.0 * std::min(32 * most, Np)) : 250.0 * most;
  return true;
}

// The rest of a chosen plan: division constants, and where each step's rows start in the unit.
void g_finish_plan(const Geom& g, GPlan* P) {
  GLayer& o = P->L;
  o.dWg = make_fastdiv((uint32_t)o.Wg);
  o.dHq = make_fastdiv((uint32_t)o.Hq);
  o.dCt = make_fastdiv((uint32_t)o.n_ct);
  o.dRr = make_fastdiv((uint32_t)o.Rr);
  const int S = g.stride, col_planes = 1 << o.cpl, span = S * (o.G - 1) + 3;
  // taps in ascending order of where their rows start in the unit
  struct Tap { int plane; uint32_t at; uint8_t row, col; } taps[64];
  int n = 0;
  if (o.pair) {   // of a kernel row, columns 0 and 1, then 1 and 2
    for (int ky = 0; ky < 3; ++ky)
      for (int s = 0; s < 2; ++s) taps[n++] = {0, (uint32_t)(ky * o.Wg + s), (uint8_t)ky, (uint8_t)s};
  } else if (g.ksize == 1) {
    for (int q = 0; q < o.G; ++q) taps[n++] = {q, 0, 0, (uint8_t)(S * q)};
  } else {
    for (int ky = 0; ky < 3; ++ky)
      for (int s = 0; s < span; ++s)
        taps[n++] = {(ky % S) * col_planes + s % col_planes, (uint32_t)((ky / S) * o.Wg + s / col_planes), (uint8_t)ky, (uint8_t)s};
  }
  for (int t = 0; t < n; ++t) taps[t].at = o.tma ? taps[t].at * 8 : taps[t].at + (uint32_t)(taps[t].plane * o.Rr);
  std::sort(taps, taps + n, [](const Tap& a, const Tap& b) { return a.plane != b.plane ? a.plane < b.plane : a.at < b.at; });
  for (int t = 0; t < o.steps; ++t) {
    const Tap& a = taps[P->paired ? 2 * t : t];
    const bool second = P->paired && 2 * t + 1 < n;
    const Tap& b = second ? taps[2 * t + 1] : a;
    const uint32_t dist = P->paired ? b.at - a.at : o.tma ? 1u : (uint32_t)(o.n_planes * o.Rr);
    o.tap[t] = a.at | (dist << 16);
    P->taps.row[t][0] = a.row; P->taps.col[t][0] = a.col;
    P->taps.row[t][1] = P->paired && !second ? 255 : b.row;
    P->taps.col[t][1] = b.col;
  }
  for (int u = 0; u < 4; ++u) o.pu_end[u] = o.steps;
  if (o.n_pu > 1)
    for (int u = 0, t = 0; u < o.n_pu; ++u) {
      while (t < n && taps[t].plane == u) ++t;
      o.pu_end[u] = t;
    }
}

// Does the tensor-core path take this layer?  The bound is that of a unit of 128 positions with its halo (row pitch of
// the padded map) in a 40.5 KB slot, two of which fit beside the weight ring; shapes beyond it go to the other paths.
// The tiles themselves are planned by g_plan_layer, which needs less.
// (So it refuses some shapes that could be planned, 3x3 layers of 64 channels on maps wider than 600 among them.)
bool g_path_takes(const Geom& g, int mode) {
  constexpr size_t slot_max = 40 * 1024 + 512, b_slot = 32 * 1024, epi = 40 * 1024, budget = 226 * 1024;
  if (g.N < 1 || g.C > (1 << 20)) return false;            // 9 * c_in stays far below 2^24: exact fp32 sums
  if ((long long)g.N * g.H * g.W >= (1ll << 31) || (long long)g.N * g.Ho * g.Wo >= (1ll << 31)) return false;
  if ((long long)g.N * g.Ho * g.Wo * g.K >= 0xffffffffLL) return false;   // output element offsets are 32-bit
  const int cpc = mode == M_F16 ? 8 : 32, raw = round_up(g.C, 2 * cpc) / cpc;
  const bool one = g.ksize == 1;
  const int Hq = one ? g.Ho : g.stride == 1 ? g.H + g.pad : g.Ho + 1;
  const int Wq = one ? g.Wo : g.stride == 1 ? g.W + g.pad : g.Wo + 1;
  const int planes = one || g.stride == 1 ? 1 : 4;
  const int halo = one ? 0 : g.stride == 1 ? 2 * Wq + 2 : Wq + 1;
  const long long Q = (long long)g.N * Hq * Wq;
  if (Q + 1024 + halo >= (1ll << 31)) return false;
  int d = 0;
  for (int c = 8; c >= 2 && !d; c -= 2)
    if (raw % c == 0 && (size_t)planes * c * (128 + halo) * 16 <= slot_max) d = c;
  if (!d) return false;
  for (int n_acc = 2; n_acc <= (mode == M_FP4 ? 3 : 2); ++n_acc) {
    const int cols = mode == M_F16 ? 256 : n_acc == 3 ? 160 : 240;
    const int nt = mode == M_FP4 ? (g.K <= cols ? round_up(g.K, 16) : 128)
                                 : (g.K <= 256 ? round_up(g.K, 16) : (round_up(g.K, 256) - g.K < 64 ? 256 : 128));
    const long long mtiles = (Q + 127) / 128;
    int mt = 1;
    for (int m = 4; m >= 2 && mt == 1; --m)
      if ((size_t)planes * d * (128 * m + halo) * 16 <= slot_max && m * nt <= cols) mt = m;
    while (mt > 1 && mtiles < mt) --mt;
    const int rows = 128 * mt + halo;
    const long long groups = (mtiles + mt - 1) / mt;
    if ((uint32_t)rows * 16 >= (1u << 18)) return false;
    if (groups * ((g.K + nt - 1) / nt) > 0x7fffffffLL || groups * rows >= (1ll << 31)) return false;
    const size_t unit = (((size_t)planes * d * rows * 16) + 127) & ~(size_t)127;
    const size_t pix = (((size_t)planes * rows * 4) + 127) & ~(size_t)127;
    if (2 * unit + epi + 2 * pix + 256 + kGTail + 3 * b_slot > budget) return false;
  }
  return true;
}

// Epilogue warps that have something to write of a position tile (of all its channel tiles): of each 32 rows that hold a
// channel those two that have a slice.
int g_writing_warps(const GLayer& L) {
  int warps = 0;
  for (int at = 0; at < L.n_ct * G_ROWS; at += 32) {
    const int r = at % G_ROWS, first = L.lg ? 0 : 2 * (r >> L.kp_log);
    if (at - r + (r & ((1 << L.kp_log) - 1)) >= L.K) continue;
    for (int half = 0; half < 2; ++half) warps += first + half < (L.Np + 31) / 32 ? 1 : 0;
  }
  return warps;
}

// Tile sizes the planner chooses from (positions; multiples of 16).
constexpr int kNpTable[] = {256, 240, 208, 192, 160, 144, 128, 112, 96, 80, 64, 48, 32, 16};

// A tile size under consideration: what has to be planned, and the estimates the choice is made by.
struct GChoice {
  int lg = 0, Np = 0, tiles = 0;
  bool tma = false;
  double through = 0, alone = 0;
};

// Best choice for one layer and tiles of at most `cap` positions: the group size 2^lg with the least time over all its tiles.
bool g_best_group(const Geom& g, int mode, int kind, int cap, bool tma, GChoice* out) {
  bool found = false;
  double best = 0;
  GPlan P;
  for (int lg = 0; lg <= 3; ++lg) {
    if (lg && (mode != M_FP4 || g.K > G_ROWS >> lg)) break;
    for (int Np : kNpTable) {
      if (Np > cap) continue;
      if (!g_plan_layer(g, mode, kind, lg, Np, tma, &P) && !(tma && g_plan_layer(g, mode, kind, lg, Np, false, &P))) continue;
      const double t = P.L.total_tiles * P.through();
      if (!found || t < best) {
        best = t;
        *out = {lg, Np, P.L.total_tiles, P.L.tma != 0, P.through(), P.alone()};
        found = true;
      }
      break;   // the largest that fits
    }
  }
  return found;
}

// The plan of one layer by itself whose last tile ends first (binary activations).
bool g_plan_by_end(const Geom& g, int mode, int kind, int sms, GPlan* plan) {
  double best = -1;
  int best_lg = 0, best_np = 0;
  for (int Np : kNpTable) {
    if (Np > (int)G_TMEM_FP4 / 2) continue;
    for (int lg = 0; lg <= 3; ++lg) {
      if (!g_plan_layer(g, mode, kind, lg, Np, false, plan)) continue;
      const int waves = (plan->L.total_tiles + sms - 1) / sms;
      const double t = plan->alone() + (waves - 1) * plan->through();
      if (best < 0 || t < best) { best = t; best_lg = lg; best_np = Np; }
    }
  }
  return best >= 0 && g_plan_layer(g, mode, kind, best_lg, best_np, false, plan);
}

// Do the packed signs between the members of a chain carry tags?  words: the most between two members.  A layer's signs then reach
// the next layer's expanders 1.2 us sooner, but each word is twice as long and the expanders load two of them at a time
// instead of four, which shows once a CTA has many tiles.  Measured on one B200, counters and tags, us: ResNet-20 stack at batch 96
// (98 k words) 94.6 and 79.9, 128 (131 k) 111.7 and 102.4; ResNet-18 16 (100 k) 87.8 and 87.1, 24 (150 k) 93.2 and 97.7, 32 (200 k) 99.6 and 108.0;
// ResNet-34 16 162.9 and 164.6, 24 171.9 and 184.2; on one image ResNet-18 72.3 and 51.3, ResNet-34 139.0 and 96.4, ResNet-20 57.4 and 37.6.
// (One rule for all: 150 k words are too many for the networks of two to sixteen words a pixel, and 131 k still gain where every
// pixel is one.  A stack of one layer has no word between members, and with tags no counters to clear.)
inline bool g_tagged(size_t words) { return words <= (size_t)1 << 17; }

// The ring geometry of a launch of these problems and where its parts lie in shared memory; false where it does not fit.
bool g_ring(const GPlan* plan, int count, int mode, GParams* p, size_t* smem) {
  const uint32_t tmem = mode == M_FP4 ? G_TMEM_FP4 : G_TMEM_F16;
  size_t a_slot = 0, pix_bytes = 0;
  int widest = 16;
  for (int i = 0; i < count; ++i) {
    const GLayer& o = plan[i].L;
    a_slot = std::max(a_slot, plan[i].unit_bytes);
    if (mode == M_F16 && !o.tma) pix_bytes = std::max(pix_bytes, (size_t)o.n_planes * o.Rr * 4);
    widest = std::max(widest, o.Np);
  }
  // accumulator buffers: as many as fit, up to four
  int n_acc = (int)tmem / widest;
  if (n_acc > 4) n_acc = 4;
  a_slot = (a_slot + 1023) & ~(size_t)1023;   // (the swizzle of the TMA units repeats every 1024 bytes)
  const uint32_t b_slot = mode == M_F16 ? kGBSlotF16 : kGBSlot;
  pix_bytes = (pix_bytes + 127) & ~(size_t)127;
  const size_t lay_bytes = ((size_t)count * sizeof(GLayer) + 127) & ~(size_t)127;
  const size_t fixed = (size_t)G_EPI_BYTES + pix_bytes + lay_bytes + kGTail;
  // Ring depths: four activation slots if they fit beside four weight slots, else two (with the 4-bit expanders a
  // multiple of the number of teams) or three; the weights take what is left.
  static_assert(G_XTEAMS == 1 || G_XTEAMS == 2, "the ring depths below are multiples of the team count");
  int na = 4, ns = 0;
  for (; na >= 2; --na) {
    if (mode == M_FP4 && na % G_XTEAMS) continue;
    const int ns_min = mode == M_F16 ? 4 : na > 2 ? 4 : 3;
    if ((size_t)na * a_slot + fixed + ns_min * (size_t)b_slot > kGSmemBudget) continue;
    ns = (int)((kGSmemBudget - fixed - (size_t)na * a_slot) / b_slot);
    break;
  }
  if (na < 2 || ns < 3) return false;
  if (ns > G_NS_MAX) ns = G_NS_MAX;
  p->n_layers = count;
  p->NA = na;
  p->NS = ns;
  p->acc_cols = (tmem / (uint32_t)n_acc) & ~15u;
  p->n_acc = n_acc;
  p->a_slot_bytes = (uint32_t)a_slot;
  p->b_slot_bytes = b_slot;
  p->off_b = (uint32_t)((size_t)na * a_slot);
  p->off_epi = p->off_b + (uint32_t)ns * b_slot;
  p->off_pix = p->off_epi + G_EPI_BYTES;
  p->off_lay = p->off_pix + (uint32_t)pix_bytes;
  p->off_tail = p->off_lay + (uint32_t)lay_bytes;
  *smem = (size_t)p->off_tail + kGTail;
  return *smem <= (size_t)kMaxDynSmem && *smem < (1u << 18);
}

// Another plan for a launch of one layer of few channels, with single pixels or pairs, where its tiles would end at least 15 %
// earlier: the group size of the most throughput leaves most SMs idle when a small layer's work is packed into few heavy
// tiles.  96 to 20 channels, 16 images of 14x14 at stride 2: 16 tiles 20.7 us, 64 tiles 8.2; 6.3 % over those 384 layers.
// The 15 % are what the estimate errs by: without them one layer in thirty got slower, by up to a third.  Of the widths
// only the narrowest that leaves no SM a second tile and the two above are looked at: all of them take another microsecond, which the
// no-allocation entry point pays at the first call of each shape.
void g_plan_alone(const Geom& g, int mode, int kind, int sms, GPlan* plan) {
  constexpr int widths = sizeof(kNpTable) / sizeof(kNpTable[0]);
  double best = 0.85 * plan->end(sms);
  int best_lg = -1, best_np = 0;
  GPlan P;
  for (int lg = 0; lg <= std::min(plan->L.lg, 1); ++lg) {
    // positions of the whole layer, as g_plan_layer counts them
    const int rows = g.ksize == 1 ? g.Ho : g.stride == 1 ? g.H + g.pad : g.Ho + 1, cols = g.ksize == 1 ? g.Wo : g.stride == 1 ? g.W + g.pad : g.Wo + 1;
    const long long Q = (long long)g.N * rows * ((cols + (1 << lg) - 1) >> lg);
    int at = widths - 1;
    while (at > 0 && Q > (long long)kNpTable[at] * sms) --at;
    for (int w = std::max(at - 2, 0); w <= at; ++w) {
      const int Np = kNpTable[w];
      if (Np > (int)G_TMEM_FP4 / 2 || !g_plan_layer(g, mode, kind, lg, Np, false, &P)) continue;
      const double t = P.end(sms);
      if (t < best) { best = t; best_lg = lg; best_np = Np; }
    }
  }
  if (best_lg >= 0) g_plan_layer(g, mode, kind, best_lg, best_np, false, plan);
}

// Both teams of expanders on one tile.  In a launch of one layer with at most one tile per CTA, a tile that is one unit leaves
// one team idle while the other does its loads in a row.  With words that are loaded one at a time (an odd number per
// pixel) and at least 16 loads, blocks of half the channels (a third of six chunks) are 6 to 37 % faster over 182 plans of
// such layers; below 16 the second block's cost shows, and with loads of two or four words half a block has as many.
void g_split_block(const Geom& g, int mode, int kind, int sms, GPlan* plan) {
  const GLayer& o = plan->L;
  if (mode != M_FP4 || o.n_cb != 1 || o.cb_chunks < 4 || o.total_tiles > sms || g_word_step(o.Cw, o.cb_chunks) != 1 || plan->loads < 16) return;
  g_plan_layer(g, mode, kind, o.lg, o.Np, false, plan, o.cb_chunks == 8 ? 4 : 2);
}

// Tiles of independent problems: one size limit for all of them, by the estimated time of the launch.
bool g_plan_independent(const Geom* gs, int count, int mode, int kind, bool tma, int sms, GPlan* plan) {
  GChoice trial[SNN_GROUP_MAX], chosen[SNN_GROUP_MAX];
  double best = -1;
  for (int cap : kNpTable) {
    if (cap > (int)(mode == M_FP4 ? G_TMEM_FP4 : G_TMEM_F16) / 2) continue;
    bool ok = true;
    for (int i = 0; i < count && ok; ++i) ok = g_best_group(gs[i], mode, kind, cap, tma, &trial[i]);
    if (!ok) continue;
    // the machine's share of all tiles (whole tiles where there is one problem), and the last tile's way through the roles
    double sum = 0, last = 0, slowest = 0;
    for (int i = 0; i < count; ++i) {
      const GChoice& c = trial[i];
      sum += count == 1 ? (double)((c.tiles + sms - 1) / sms) * sms * c.through : c.tiles * c.through;
      last = std::max(last, c.alone - c.through);
      slowest = std::max(slowest, c.through);
    }
    const double t = std::max(sum / sms, slowest) + last + (count > 1 ? slowest / 2 : 0);
    if (best < 0 || t < best) {
      best = t;
      std::copy(trial, trial + count, chosen);
    }
  }
  if (best < 0) return false;
  for (int i = 0; i < count; ++i) g_plan_layer(gs[i], mode, kind, chosen[i].lg, chosen[i].Np, chosen[i].tma, &plan[i]);
  if (count == 1) {
    if (mode == M_FP4 && gs[0].K <= G_ROWS / 2) g_plan_alone(gs[0], mode, kind, sms, plan);
    g_split_block(gs[0], mode, kind, sms, plan);
  }
  return true;
}

// The order in which the CTAs walk through independent problems.
//
// HEAVY_FIRST: those with the most MMAs a tile first, so that the tiles that even out the CTAs' ends are small ones, and the heaviest are not all that is
// left when the others are done.  Tiles of less than 1200 cycles take as long as their other roles and stay in the order given (by the MMAs alone the
// ResNet-20 group at batch 4 to 24 is 1 to 3 % slower).  us, in the order given and so: ResNet-18 group on one image 10.5 and 9.2, at batch 3 13.6
// and 11.7, 8 20.2 and 17.2, 16 29.2 and 28.3; ResNet-34 at 4 22.0 and 19.8; with fp16 activations ResNet-18 at 2 32.6 and 23.8, 16 70.6 and 63.2,
// ResNet-20 at 16 12.7 and 11.5; signs of the 1x1 layers at 16 56.0 and 54.0; signs of ResNet-20 at 64 17.4 and 17.8.
//
// GIVEN: where the outputs are more than 256 MB, twice what the L2 holds: networks begin with the layers that write the most, and end with
// outputs that stay in the L2 (ResNet-18 group at batch 64 into a flushed L2, heavy first 94.9 us and so 88.5, later 96.2 and 90.1; back to back the same).
//
// IN_TURN: where the MMAs of all problems take less than a fifth of the time of their stores (1x1 layers: 0.10 to 0.15, one image 0.22; 3x3 networks from
// 0.35 on), the one bound most by its stores, then the one bound least, and so on, so that the memory is neither idle nor asked for more
// than it takes for long.  1x1 layers, us back to back in the order given, heavy first and in turn (from batch 9 on with stores that leave the L2 first, below):
// batch 2 20.3, 20.5 and 19.3; 4 29.3, 29.0, 27.7; 8 50.9, 52.8, 50.4; 12 75.7, 71.9, 68.4; 24 130.4, 131.7, 132.7; 40 220, 220, 217; 64 385, 380, 367.
// One image 15.1, 14.9, 15.4; ResNet-18 at 16 29.2, 28.3, 31.2, 64 92.3, 91.7, 93.3; ResNet-20 at 128 33.3, 33.1, 33.4.
enum GOrder { ORDER_GIVEN, ORDER_HEAVY_FIRST, ORDER_IN_TURN };
struct GStores {
  bool large, bound;   // word outputs of more than twice the L2; MMAs of less than a fifth of the stores' time
};
inline GStores g_stores(const GPlan* plan, int count) {
  double bytes = 0, mma = 0, drain = 0;
  for (int i = 0; i < count; ++i) {
    const GLayer& o = plan[i].L;
    bytes += (double)o.N * o.Ho * o.Wo * o.K * 4.0;
    mma += o.total_tiles * plan[i].mma;
    drain += o.total_tiles * plan[i].drain;
  }
  return {bytes > 256e6, mma < 0.2 * drain};
}
inline GOrder g_order_kind(const GPlan* plan, int count, int kind) {
  if (kind == TCG_SIGNS) return ORDER_HEAVY_FIRST;
  const GStores stores = g_stores(plan, count);
  return stores.bound ? ORDER_IN_TURN : stores.large ? ORDER_GIVEN : ORDER_HEAVY_FIRST;
}
// Do the words that a launch writes leave the L2 before what else is there?  Where they are more than it holds and most of the launch's time: the sooner
// they go to memory, the better the memory takes them (64 to 256 channels of 56x56, 64 images: 37.5 and 35.9 us), and the inputs stay.  1x1 layers,
// us: batch 10 (297 MB) 62.9 and 58.7, 12 73.3 and 67.9, 24 141.9 and 132.5, 32 192.4 and 181.2, 44 269.6 and 259.3, 64 376.5 and 363.6.  Below the line there
// is nothing in it (batch 8 51.7 and 51.0, 6 39.7 and 40.0, 3 26.5 and 26.3) and a kernel that reads the outputs finds them in the L2; nor is
// there where the MMAs take a share of the time (ResNet-18 at 64 95.6 and 95.3, into a flushed L2 the same).
inline bool g_streams(const GPlan* plan, int count, int kind) {
  const GStores stores = g_stores(plan, count);
  return kind == TCG_WORDS && stores.bound && stores.large;
}
inline void g_order(const GPlan* plan, int count, GOrder by, int* order) {
  for (int i = 0; i < count; ++i) order[i] = i;
  if (by == ORDER_HEAVY_FIRST) {
    std::stable_sort(order, order + count, [&](int a, int b) { return std::max(plan[a].mma, 1200.0) > std::max(plan[b].mma, 1200.0); });
  } else if (by == ORDER_IN_TURN) {
    std::vector<int> bound(order, order + count);
    std::vector<double> by_stores(count);
    for (int i = 0; i < count; ++i) by_stores[i] = plan[i].drain / plan[i].mma;
    std::stable_sort(bound.begin(), bound.end(), [&](int a, int b) { return by_stores[a] > by_stores[b]; });
    for (int i = 0; i < count; ++i) order[i] = i & 1 ? bound[count - 1 - i / 2] : bound[i / 2];
  }
}

// Which CTAs take a problem's odd tiles.  Every CTA gets floor(tiles / grid) tiles of a problem
// and the first (tiles % grid) CTAs in the problem's rank order get one more; the rank order is
// by the time the CTAs have been given so far, least first, so that the CTAs end close
// together although a tile of one problem may take six times as long as a tile of another.
void g_assign(const std::vector<GPlan>& P, int grid, std::vector<uint32_t>* ranks) {
  std::vector<double> busy(grid, 0.0);
  std::vector<int> order(grid);
  for (size_t i = 0; i < P.size(); ++i) {
    const double cost = P[i].through();
    for (int b = 0; b < grid; ++b) order[b] = b;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return busy[a] < busy[b]; });
    const int base = P[i].L.total_tiles / grid, rem = P[i].L.total_tiles % grid;
    for (int r = 0; r < grid; ++r) {
      (*ranks)[i * grid + order[r]] = (uint32_t)r;
      busy[order[r]] += cost * (base + (r < rem ? 1 : 0));
    }
  }
  for (int b = 0; b < grid; ++b) {
    uint32_t next = (uint32_t)P.size();
    for (size_t i = P.size(); i-- > 0;) {
      uint32_t& at = (*ranks)[i * grid + b];
      const bool has = at < (uint32_t)P[i].L.total_tiles;
      at |= next << 16;
      if (has) next = (uint32_t)i;
    }
  }
}

}  // namespace
}  // namespace snn
