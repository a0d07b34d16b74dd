// The tensor-core kernel: one or several sub-bit convolutions in ONE persistent launch.
//
// Each problem of a launch is the forward pass of Sec. 3 / Algorithm 1 for one layer (3x3, or the 1x1
// extension of the appendix) on its own input: decoded +1/-1 weights as 4-bit e2m1 operands (binary
// activations) or fp16 operands (fp16 activations), implicit GEMM over a padded, flattened position space
// in which the taps are the same staged activations read from shifted start addresses.  One CTA per
// SM walks through all problems without any grid-wide step in between: while the MMAs of one problem's
// last tile run, the expander warps already stage the next problem's first activations, the weight
// producer streams its first stages, and the epilogue warps still drain the tile before.  A single layer is a
// launch of one problem.
//
// Orientation.  The weights are the M operand (128 rows of output channels), the positions the N operand (up to
// 240, or 256 with fp16), so an accumulator has channels along its lanes and positions along its columns:
//   * an MMA reads 32 + N/4 shared-memory lines of 128 bytes and takes max(N/2, 32 + N/4) cycles (measured for
//     N = 16..256, any operand type, any start shift): at N = 240 it leaves a quarter of the shared-memory
//     bandwidth to the other roles, at N = 128 none;
//   * a stage of weights serves 240 positions;
//   * the 32 lanes of an epilogue warp are 32 consecutive channels of one pixel, so that a store instruction
//     writes one whole 128-byte line straight from registers, with no transposition through shared memory, and any
//     channel count and row alignment takes the same path.
// With positions along M and at most 128 to 160 channels along N the shared memory was the bound: operands at N = 128 take
// all of its 128 bytes per cycle, the epilogue's transposition another 8 lines per output row, and weights are streamed
// once per 128 positions.  Both layouts on one GPU, that one first: ResNet-18 group at batch 64 122 and 106 us, with fp16
// activations 312 and 259, ResNet-34 stack at batch 128 504 and 392, ResNet-20 group at batch 128 58 and 42, the 1x1
// layers 441 and 390.
//
// Few output channels (binary activations only).  With at most 64, 32 or 16 channels a lane set holds G = 2, 4 or 8
// neighbouring output pixels of a row: rows g*(128/G)..  of the weight operand are the channels of pixel G*j + g,
// and position j of the operand stands for that group of pixels.  The taps of a group are the kernel rows times the
// columns the group's windows span (stride*(G-1) + 3 instead of G times 3); a row of weights holds zeros where a
// column is outside its pixel's window.  0 * (+1 / -1 / 0) is exactly 0; with fp16 activations 0 * infinity would
// not be, so those keep G = 1.  With G = 1 the idle rows may hold copies of the channels, which share the columns (see
// g_plan_layer).
//
// Independent problems (a group) need nothing else.  A chain (a stack: problem i + 1 reads the packed signs
// problem i writes) runs in the same launch.  Where few words lie between its members (g_tagged) every word carries the tag of
// the launch that wrote it, and the expanders look at the words themselves until all they need are there: no fence, counter
// or memset between a sign and its reader.  The tag is a count of launches kept in device memory (GLaunches), so that a
// replayed graph counts too.  Other chains run on per-tile completion counters: the epilogue bumps the counter
// of a position tile when its part is written, and the expanders of the successor wait (bounded) until the
// tiles under a tile's input window are complete.  The launch is cooperative then, so that all CTAs are
// resident while some of them wait.
//
// What makes one launch possible is a ring geometry that is the same for every problem:
//   activation units  NA slots of a_slot_bytes   (a problem's unit uses a prefix)
//   weight stages     NS slots of b_slot_bytes   (a stage = whole taps of one channel block)
//   accumulators      n_acc buffers of acc_cols tensor-memory columns
// so slots, barriers and phases simply carry on from one problem to the next.
// Tiles of a problem are dealt to the CTAs round-robin; which CTAs get a problem's odd
// tiles is decided on the host from the time the CTAs have been given so far, so that the
// CTAs end close together.
//
//      warp 0        one thread streams weight stages (cp.async.bulk onto mbarriers)
//      warp 1        issues tcgen05.mma and commits barriers (warp-uniform, one elected lane)
//      warps 2-9     epilogue: TMEM -> registers -> alpha -> 128-byte stores; or TMEM -> registers ->
//                    threshold -> 32 x 32 bit transposition in the warp -> packed sign words
//      warps 10-19   expanders (but 13 and 17): packed bits -> e2m1 nibbles (or fp16 copied)
//                    into the activation ring
//      warp 13       writes the epilogue's tables (where the columns of a tile go) ahead of it, and in a chain on counters says
//                    which tiles have been written
//      warp 17       in a chain on counters: waits for the tiles that the CTA's next tile reads
// The kernel is compiled per operand mode and per output kind (words, words that leave the L2 first, packed signs, chains on counters, chains of words
// with tags), so that no variant carries another one's code in its loops; the plan (tile shapes, accumulator buffers) is made
// per output kind, the same for both kinds of chains.
// The loops around the waits, tiles and problems that all variants have are not unrolled (the compiler unrolls them four times,
// innermost and all around): a variant is 62 KB of code then instead of 112, and five kinds of roles share an SM's instruction caches.  On one GPU,
// as a graph, unrolled and not: 1x1 layers at batch 16 108.8 and 94.6 us (signs 79.8 and 71.0), ResNet-18 group at
// batch 16 36.7 and 32.3, ResNet-34 stack at batch 128 390 and 362, one layer of 256 channels 9.8 and 9.3, 39 layers 4 %.
// Every wait is bounded; one that runs out raises a status word the host reads, and
// the CTA still frees its tensor memory and returns.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cuda.h>   // tensor maps (types only; the encoder is looked up at run time)

#include "snn_tc_common.cuh"
#include "snn_tc_plan.h"

namespace snn {

namespace {

// Profiling aid (build with -DSNN_TRACE): every role's reporting lane adds up the cycles it spends in its
// waits; the host prints the averages over the CTAs after each launch.  No effect on an ordinary build.
#ifdef SNN_TRACE
__device__ long long g_trace[256 * 16];
#define TR_WAIT(var, expr) ([&]() { const long long _t = clock64(); const bool _r = (expr); var += clock64() - _t; return _r; }())
#define TR_REPORT(role, total, w0, w1, w2)                         \
  do {                                                             \
    long long* _o = g_trace + (size_t)blockIdx.x * 16 + (role)*4;  \
    _o[0] = (total); _o[1] = (w0); _o[2] = (w1); _o[3] = (w2);     \
  } while (0)
#else
#define TR_WAIT(var, expr) (expr)
#define TR_REPORT(role, total, w0, w1, w2) do { } while (0)
#endif

// A value that is the same in all lanes, in a form that the compiler knows to be: tensor-core instructions take their operands from the
// registers of a warp, and what it cannot know to be uniform is moved there one operand at a time before each of them.  The MMA issuer's loops
// were bound by that (98 cycles an MMA whatever its width; the tensor core takes 40 to 64): with its values, and the warp's
// number that the roles branch on, known to be uniform, and MMAs under a predicate instead of a branch, one layer of 256 channels
// 8.95 and 8.31 us, 512 channels of 7x7 at batch 8 7.33 and 6.74, ResNet-18 stack on one image 64.1 and 60.5 (the predicates alone 8.32,
// 6.74, 61.2; taps and the answers of waits made uniform, too: nothing, or less).
__device__ __forceinline__ int uni(int x) { return __shfl_sync(0xffffffffu, x, 0); }
__device__ __forceinline__ uint32_t fdiv(uint32_t q, const FastDiv& f) {
  return __umulhi(2u * q, f.m) >> f.s;
}
__device__ __forceinline__ int g_position_to_pixel(const GLayer& L, uint32_t q, int pl) {
  if (q >= L.Qtot) return -1;
  const uint32_t rg = fdiv(q, L.dWg);
  const int j = (int)(q - rg * (uint32_t)L.Wg);
  const uint32_t n = fdiv(rg, L.dHq);
  return g_pixel_of(L, n, (int)(rg - n * (uint32_t)L.Hq), j, pl);
}

// Waits (bounded) until the completion counters first..last, advanced by other CTAs, have reached `target`.  Whole-warp
// call: a lane looks at one counter, 32 at a time - one after the other, each look is a round trip to L2, and a tile's
// window spans up to six tiles of the predecessor.  False when the limit ran out or the CTA is giving up.  What was
// written before the counters were advanced is visible to the warp afterwards.
__device__ __forceinline__ bool g_wait_counters(const uint32_t* ctr, uint32_t first, uint32_t last, uint32_t target, int lane,
                                                volatile int* abort_flag) {
  for (uint32_t it = 0; first <= last; ++it) {
    uint32_t v = target;
    if (first + (uint32_t)lane <= last)
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr + first + (uint32_t)lane) : "memory");
    if (__all_sync(0xffffffffu, v >= target)) {
      first += 32u;
    } else {
      if (it >= (1u << 21) || __any_sync(0xffffffffu, *abort_flag != 0)) return false;
      __nanosleep(20);
    }
  }
  __syncwarp();
  return true;
}
// Loads of the scales and of the activations.  LATE: the launch may be a programmatic dependent, resident while the kernel before still writes them;
// the read-only path is for memory that nothing writes while a kernel lives.  (Independent problems take the same time either way.  A chain, which
// starts when the kernel before has ended, 0.6 % longer with plain loads.)
template <bool LATE, class T>
__device__ __forceinline__ T g_ld(const T* p) { return LATE ? *p : __ldg(p); }
// Activation words; fresh: another CTA of this launch wrote them, they are read from L2.
template <bool LATE, class T>
__device__ __forceinline__ T g_ld_act(const uint32_t* p, bool fresh) {
  const T* const q = reinterpret_cast<const T*>(p);
  return fresh ? __ldcg(q) : g_ld<LATE>(q);
}
// Words with tags, between the members of a chain: the word in the low half, the tag of the launch that wrote it in the high half,
// stored and loaded 64 bits at once.  A word whose tag is this launch's is this launch's word, so that neither side
// needs a fence or a counter.
__device__ __forceinline__ void g_st_tagged(void* p, size_t i, uint32_t word, uint32_t tag) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(reinterpret_cast<uint64_t*>(p) + i), "l"((uint64_t)word | (uint64_t)tag << 32) : "memory");
}
// A word and its tag, or two of each: loads under a predicate into the registers that hold them, with no branch and nothing to move behind it
// (ResNet-18 stack on one image 67.0 and 64.4 us, ResNet-34 126.5 and 122.6, ResNet-20 at batch 96 94.3 and 90.8; plain words so gained nothing).
__device__ __forceinline__ void g_ld_tagged(uint4& v, const uint64_t* p, int words) {
  uint64_t a = (uint64_t)v.y << 32 | v.x, b = (uint64_t)v.w << 32 | v.z;
  asm volatile("{\n\t.reg .pred a, b;\n\tsetp.gt.s32 a, %3, 0;\n\tsetp.gt.s32 b, %3, 1;\n\t@a ld.relaxed.gpu.global.b64 %0, [%2];\n\t@b ld.relaxed.gpu.global.b64 %1, [%2+8];\n\t}"
               : "+l"(a), "+l"(b) : "l"(p), "r"(words) : "memory");
  v = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}
// Tensor maps of the fp16 activations, a kernel parameter of its own (the other variants have one unused entry).
template <int MODE>
struct GMaps {
  CUtensorMap m[MODE == M_F16 ? SNN_GROUP_MAX : 1];
};

// The MMAs of one activation unit of one tile: steps t..t_last x KPT.  The body of a step is straight-line code.
// Weight stages are waited for and released as the step counter crosses their boundaries.
template <int MODE, int KPT>
__device__ __forceinline__ bool g_issue_block(const GLayer& L, int st_steps, int t, int t_last, uint64_t a_fixed, uint32_t k_step, uint32_t a_unit, uint32_t w_base, uint32_t b_slot_units,
                                              uint32_t d0, uint32_t idesc, uint32_t& acc, int NS, uint32_t bar_bfull,
                                              uint32_t bar_bempty, int& b_slot, uint32_t& b_phase, bool leader, uint32_t sf,
                                              long long& tr_b) {
  constexpr uint64_t fixed = ((uint64_t)1 << 46) | ((uint64_t)8 << 32);   // descriptor version; 8-row groups 128 bytes apart
  constexpr uint64_t w_fixed = fixed | ((uint64_t)128 << 16);             // the weights' chunks are 128 rows apart
  uint32_t tap = MODE == M_FP4 && KPT == 1 ? 0u : L.tap[t];
#pragma unroll 1
  while (t < t_last) {
    // a weight stage holds whole steps: one wait, then nothing but MMAs until its last step
    if (!TR_WAIT(tr_b, mbar_wait(bar_bfull + 8 * b_slot, b_phase))) return false;
    tc_fence_after();
    uint32_t wa = w_base + (uint32_t)b_slot * b_slot_units;
    if constexpr (MODE == M_FP4 && KPT == 1) {
      // One MMA a step: those of a stage are straight-line code behind one branch, their taps read together.  In the loop
      // below the read, the branch and the address arithmetic of a step run between two MMAs (one warp by itself, 9 MMAs of
      // 64 positions: 1870 cycles, so 1080; 70 channels 45x37 at stride 2: 8.0 and 7.4 us).  With two or more MMAs a step, and
      // with fp16 operands, the longer code costs the other roles more than this gains (fp16 group at batch 1 12 %).
      constexpr int ST = (int)(kGBSlot / (KPT * 2 * G_ROWS * 16));   // most steps of a stage (g_plan_layer)
      const int n = t_last - t < st_steps ? t_last - t : st_steps;
      {
        uint32_t rows[ST];
#pragma unroll
        for (int i = 0; i < ST; ++i) rows[i] = i < n ? L.tap[t + i] + a_unit : 0u;   // (start and chunk distance of the low word)
#pragma unroll
        for (int i = 0; i < ST; ++i) {
          if (i < n) mma_ss_fp4(d0, w_fixed | (uint64_t)(wa + (uint32_t)(i * 256)), a_fixed | (uint64_t)rows[i], idesc, i == 0 ? acc : 1u, sf, sf + 16, leader);
        }
        if (leader) tc_commit(bar_bempty + 8 * b_slot);
      }
      t += n;
      acc = 1;
      if (++b_slot == NS) { b_slot = 0; b_phase ^= 1u; }
      continue;
    }
    const int t_end = t + st_steps < t_last ? t + st_steps : t_last;
    if constexpr (MODE == M_FP4 && KPT == 2) {
      // Two MMAs a step: two steps at a time, for the same reason (87->40 channels of 8x24 5.0 and 4.7 us, 100->311 of 8x28 5.1 and
      // 4.9; a whole stage at a time made the 1x1 layers, whose stages are one step, 3 % slower).
#pragma unroll 1
      for (; t + 1 < t_end; t += 2) {
        const uint32_t one = L.tap[t] + a_unit, two = L.tap[t + 1] + a_unit;
        {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_ss_fp4(d0, w_fixed | (uint64_t)(wa + (uint32_t)(k * 256)), a_fixed | (uint64_t)((k < 2 ? one : two) + (uint32_t)(k & 1) * k_step), idesc, k == 0 ? acc : 1u, sf, sf + 16, leader);
        }
        acc = 1;
        wa += 4 * 256;
      }
      tap = L.tap[t];
    }
#pragma unroll 1
    for (; t < t_end; ++t) {
      const uint32_t cur = tap;
      if (t + 1 < t_last) tap = L.tap[t + 1];
      const uint64_t bd = a_fixed | ((uint64_t)(cur >> 16) << 16) | (uint64_t)(a_unit + (cur & 0xffffu));
      const uint64_t wd = w_fixed | (uint64_t)wa;
      {
#pragma unroll
        for (int k = 0; k < KPT; ++k) {
          const uint32_t accum = k == 0 ? acc : 1u;
          if (MODE == M_FP4) mma_ss_fp4(d0, wd + (uint64_t)(k * 256), bd + (uint64_t)((uint32_t)k * k_step), idesc, accum, sf, sf + 16, leader);
          else mma_ss_f16(d0, wd + (uint64_t)(k * 256), bd + (uint64_t)((uint32_t)k * k_step), idesc, accum, leader);
        }
      }
      acc = 1;
      wa += KPT * 256;
    }
    if (leader) tc_commit(bar_bempty + 8 * b_slot);  // the slot is free once these MMAs have read it
    if (++b_slot == NS) { b_slot = 0; b_phase ^= 1u; }
  }
  return true;
}

// Two 32 x 32 bit matrices side by side (lane r holds row r of both): rows to columns (lane c holds column c, bit r = row r).  A
// stage is a shuffle and two instructions (the two widest one): bytes by a lane's own permutation, bits by its own rotation and mask.
__device__ __forceinline__ void g_transpose32(uint32_t& x, uint32_t& z, int lane) {
  uint32_t* const m[2] = {&x, &z};
#pragma unroll
  for (int s = 16; s >= 8; s >>= 1) {
    const uint32_t order = s == 16 ? ((lane & 16) ? 0x3276u : 0x5410u) : (lane & 8) ? 0x3715u : 0x6240u;
#pragma unroll
    for (int i = 0; i < 2; ++i) *m[i] = __byte_perm(*m[i], __shfl_xor_sync(0xffffffffu, *m[i], s), order);
  }
#pragma unroll
  for (int s = 4; s >= 1; s >>= 1) {
    const uint32_t low = s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u, own = (lane & s) ? ~low : low;
    const uint32_t turn = (lane & s) ? 32 - s : s;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t y = __shfl_xor_sync(0xffffffffu, *m[i], s);
      *m[i] = (*m[i] & own) | (__funnelshift_l(y, y, turn) & ~own);
    }
  }
}

}  // namespace

// OUTK: what the epilogue is compiled for.  0: fp32 or int32 words for every member; 1: packed signs for every
// member; 2: a chain - packed signs between the members, any type for the last, and the dependency waits and
// completion counters; 3: a chain whose words carry tags instead; 4: words that leave the L2 first (g_streams).  Keeping the variants apart keeps each one's
// registers and code to what it needs (a cache policy in a register for both kinds of words took all others 0.2 to 1 %).
enum { OUT_WORDS = 0, OUT_SIGNS = 1, OUT_CHAIN = 2, OUT_TAGGED = 3, OUT_STREAM = 4 };

template <int MODE, int OUTK>
__global__ void __launch_bounds__(G_THREADS, 1) tcg_conv_kernel(const __grid_constant__ GParams p, const __grid_constant__ GMaps<MODE> maps) {
  constexpr bool F16 = MODE == M_F16;   // fp16 activations (copied, not expanded)
  constexpr bool FP4 = MODE == M_FP4;   // binary activations as e2m1 nibbles
  constexpr bool TAGGED = OUTK == OUT_TAGGED;   // a chain without waits for whole tiles: every word is looked at until it is there
  constexpr bool CHAIN = OUTK == OUT_CHAIN;
  constexpr bool STREAM = OUTK == OUT_STREAM;
  constexpr bool WORDS = OUTK == OUT_WORDS || STREAM;
  constexpr bool LATE = !CHAIN && !TAGGED;      // see g_ld
  extern __shared__ __align__(1024) uint8_t smem[];
  // carve-up: [NA activation slots][NS weight slots][epilogue tables][pixel tables][problem table][barriers, flags]
  uint8_t* a_smem = smem;
  uint8_t* b_smem = smem + p.off_b;
  uint8_t* epi_smem = smem + p.off_epi;
  int* pix_tab = reinterpret_cast<int*>(smem + p.off_pix);
  // The problems' descriptions are read from shared memory where they are needed instead of
  // being held in registers: the roles are at different problems at the same time.
  GLayer* lay = reinterpret_cast<GLayer*>(smem + p.off_lay);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_tail);
  // barriers: b_full[8] b_empty[8] a_full[4] a_empty[4] acc_full[4] acc_empty[4] tab_full[4] tab_empty[4]
  // acc_full and the epilogue's tables are indexed by the tile's sequence number in the CTA (seq % 4), acc_empty by
  // the accumulator buffer.
  const uint32_t bar_bfull = smem_u32(bars), bar_bempty = smem_u32(bars + 8);
  const uint32_t bar_afull = smem_u32(bars + 16), bar_aempty = smem_u32(bars + 20);
  const uint32_t bar_accfull = smem_u32(bars + 24), bar_accempty = smem_u32(bars + 28);
  const uint32_t bar_tabfull = smem_u32(bars + 32), bar_tabempty = smem_u32(bars + 36);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 40);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* ready_tiles = tmem_slot + 2;   // chain: tiles of this CTA whose input has been written

  const int tid = threadIdx.x, warp = uni(tid >> 5), lane = tid & 31;
  const int NS = p.NS, NA = p.NA;
  const int G = (int)gridDim.x;

  // Whole-warp wait: a phase that is over already costs one look and a vote.  Every lane sees the phase's end for itself (what one lane has seen and
  // shuffled would not order the other lanes' accesses), and no lane takes a path of its own, which cost more than the looks: with lane 0 waiting and
  // shuffling its answer the smallest layer took 4.0 us, now 3.4, ragged layer 6.7 and 6.1, ResNet-20 group 34.9 and 33.2, ResNet-18 stack on one image
  // 59.7 and 51.3, ResNet-34 at batch 128 320 and 297; 1x1 layers at batch 64 369 and 372.  False: the wait ran out, or the CTA is giving up.
  auto wait_phase = [&](uint32_t bar, uint32_t parity, uint32_t ns, int code) -> bool {
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
    const bool over = __all_sync(0xffffffffu, !*abort_flag && mbar_wait_backoff(bar, parity, ns));
    if (!over && lane == 0 && !*abort_flag) {
      *abort_flag = 1;
      raise_status(p.status, code);
    }
    return over;
  };

  // Set-up.  Warp 2 allocates tensor memory while the others write the barriers and the problems' descriptions; only the MMA
  // issuer and the epilogue warps wait for it (barrier 1).  The producer, the expanders and the table warp start as
  // soon as the descriptions are there (barrier 2): 39 single layers 1.4 % faster, as a graph, than with both behind two barriers
  // of all threads.
  constexpr int SETUP_THREADS = G_THREADS - 32;
  uint32_t tmem_base = 0;
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else {
    const int rank = warp > 2 ? tid - 32 : tid;
    if (rank < 40) {
      uint32_t count = 1;
      if ((rank >= 28 && rank < 32) || rank >= 36) count = G_EW;               // acc_empty, tab_empty: one arrival per epilogue warp of the tile
      if (rank >= 16 && rank < 20) count = FP4 ? G_EW / G_XTEAMS : G_EW;    // a_full: one arrival per expander warp of the unit
      mbar_init(smem_u32(bars + rank), count);
    }
    if (rank == 64) {
      *abort_flag = 0;
      *ready_tiles = 0;
    }
    constexpr int at_first = (int)offsetof(GLayer, first) / 4;   // (this CTA's first tile is put in here)
    uint32_t* dst = reinterpret_cast<uint32_t*>(smem + p.off_lay);
    if (p.n_layers == 1) {
      // a launch of one problem is short: its description comes with the launch, not from memory
      const uint32_t* src = reinterpret_cast<const uint32_t*>(&p.one);
#pragma unroll 1
      for (int i = rank; i < (int)(sizeof(GLayer) / 4); i += SETUP_THREADS) dst[i] = i == at_first ? blockIdx.x : src[i];
    } else {
      const uint32_t* src = reinterpret_cast<const uint32_t*>(p.layers);
      const int words = p.n_layers * (int)(sizeof(GLayer) / 4);
      for (int i = rank; i < words; i += SETUP_THREADS) dst[i] = __ldg(src + i);
      // (loaded here for all problems: a global load at the start of a problem would queue behind the epilogue's stores)
      uint32_t own = 0;
      if (rank < p.n_layers) own = __ldg(p.ranks + (size_t)rank * G + blockIdx.x);
      bar_sync_some<2, SETUP_THREADS>();
      if (rank < p.n_layers) {
        lay[rank].first = (int)(own & 0xffffu);
        lay[rank].next = (int)(own >> 16);
      }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bar_sync_some<2, SETUP_THREADS>();
  }
  grid_dep_launch();
  const uint32_t tag = TAGGED ? (uint32_t)(__ldcg(p.launches.count) >> 32) + 1u : 0u;   // (complete only when all CTAs have ended)
  if (warp >= 1 && warp < 2 + G_EW) {
    tc_fence_before();
    bar_sync_some<1, 32 * (1 + G_EW)>();
    tc_fence_after();
    tmem_base = *tmem_slot;
    if (FP4) {
      // unit block scales: every byte of the scale columns is the ue8m0 code of 1.0, in all 128 lanes
      // (warps 2..5 cover the four lane quarters), whatever part of them an MMA reads
      if (warp >= 2 && warp < 6) tmem_fill32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + G_SCALE_COL, 0x7f7f7f7fu);
      tc_fence_before();
      bar_sync_some<1, 32 * (1 + G_EW)>();
      tc_fence_after();
    }
  }

  if (warp == 0) {
    // ------------------------------------------------ weight producer (one lane)
    if (lane == 0) {
      if (p.after_weights) grid_dep_wait();
      int b_slot = 0;
      long long b_issued = 0;
      uint32_t b_phase = 1;  // parity of the previous use of a slot (valid from the second lap)
      bool ok = true;
      long long tr_w0 = 0, tr_t0 = clock64();
      (void)tr_w0; (void)tr_t0;
#pragma unroll 1
      for (int l = 0; l < p.n_layers && ok; ++l) {
        const GLayer& L = lay[l];
        const int n_cb = L.n_cb, n_ct = L.n_ct, total = L.total_tiles, steps = L.steps, st_steps = L.st_steps, n_pu = L.n_pu;
        const uint32_t step_bytes = L.step_bytes;
        const uint8_t* wt = L.wt;
        const size_t ct_bytes = (size_t)n_cb * (size_t)steps * step_bytes;   // one channel tile
        const FastDiv dCt = L.dCt;
#pragma unroll 1
        for (int tile = L.first; tile < total && ok; tile += G) {
          if (*abort_flag) { ok = false; break; }
          const uint8_t* src = wt + (size_t)(tile - (int)fdiv((uint32_t)tile, dCt) * n_ct) * ct_bytes;
#pragma unroll 1
          for (int u = 0, t = 0; u < n_cb * n_pu && ok; ++u) {
            const int t_last = L.pu_end[u & (n_pu - 1)];
#pragma unroll 1
            for (t = t >= steps ? 0 : t; t < t_last; t += st_steps) {
              const uint32_t stage_bytes = (uint32_t)(t_last - t < st_steps ? t_last - t : st_steps) * step_bytes;
              if (b_issued >= NS && !TR_WAIT(tr_w0, mbar_wait_backoff(bar_bempty + 8 * b_slot, b_phase, 32))) { ok = false; break; }
              mbar_expect_tx(bar_bfull + 8 * b_slot, stage_bytes);
              bulk_g2s(smem_u32(b_smem) + (uint32_t)b_slot * p.b_slot_bytes, src, stage_bytes, bar_bfull + 8 * b_slot);
              src += stage_bytes;
              ++b_issued;
              if (++b_slot == NS) { b_slot = 0; b_phase ^= 1u; }
            }
            t = t_last;
          }
        }
      }
      if (!ok && !*abort_flag) {
        *abort_flag = 1;
        raise_status(p.status, 2);
      }
      TR_REPORT(0, clock64() - tr_t0, tr_w0, 0, 0);
      // never leave with copies in flight: wait (bounded) for the last load of every slot
#pragma unroll 1
      for (int s = 0; s < NS; ++s) {
        long long last = -1;
        if (b_issued > s) last = s + (b_issued - 1 - s) / NS * NS;
        if (last >= 0) mbar_wait_backoff(bar_bfull + 8 * s, (uint32_t)((last / NS) & 1), 64);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    // The whole warp walks the loops and waits together, so that every address and descriptor
    // is a warp-uniform value; the MMAs and the commits are predicated on one elected lane.  Where a wait runs out in one
    // lane it leaves the problem, and all lanes stop where they come together behind it (no shuffle stands inside).
    {
      const bool leader = elect_one();
      bool ok = true;
      int a_slot = 0, b_slot = 0, acc_slot = 0, full_slot = 0;
      uint32_t a_phase = 0, b_phase = 0, acc_phase = 1;
      const int n_acc = p.n_acc;
      long long tiles_done = 0;
      long long tr_w0 = 0, tr_w1 = 0, tr_w2 = 0, tr_t0 = clock64();
      (void)tr_w0; (void)tr_w1; (void)tr_w2; (void)tr_t0;
      const uint32_t a_slot_units = p.a_slot_bytes >> 4, b_slot_units = p.b_slot_bytes >> 4;
      const uint32_t a_base = smem_u32(a_smem) >> 4, w_base = smem_u32(b_smem) >> 4, sf = tmem_base + G_SCALE_COL;
#pragma unroll 1
      for (int l = 0; l < p.n_layers && ok; ++l) {
        const GLayer& L = lay[l];
        const int n_pu = uni(L.n_pu), n_units = uni(L.n_cb) * n_pu, kpt = uni(L.kpt), total = uni(L.total_tiles), tile0 = uni(L.first), st_steps = uni(L.st_steps);
        const int end[4] = {uni(L.pu_end[0]), FP4 ? 0 : uni(L.pu_end[1]), FP4 ? 0 : uni(L.pu_end[2]), FP4 ? 0 : uni(L.pu_end[3])};
        // activation operand: rows of 16 bytes, 8-row groups 128 bytes apart, a K step two chunks on; or rows of 128 bytes
        // in the 128-byte swizzle, 8-row groups 1024 bytes apart, a K step 32 bytes on.  (The swizzle permutes address
        // bits, so a tap's start may be any row.)
        const bool swz = F16 && uni(L.tma);
        const uint64_t a_fixed = ((uint64_t)1 << 46) | (swz ? ((uint64_t)2 << 61) | ((uint64_t)64 << 32) : (uint64_t)8 << 32);
        const uint32_t k_step = swz ? 2u : 2u * (uint32_t)uni(L.n_planes * L.Rr);
        const uint32_t Np = (uint32_t)uni(L.Np);
        // instruction descriptor: D format, A/B formats, K-major both, N>>3, M>>4
        // (4-bit mode: A/B format e2m1, scale format ue8m0, scale ids 0)
        const uint32_t idesc =
            F16 ? ((1u << 4) | ((Np >> 3) << 17) | ((128u >> 4) << 24))
                : ((1u << 7) | (1u << 10) | ((Np >> 3) << 17) | (1u << 23) | ((128u >> 4) << 24));
#pragma unroll 1
        for (int tile = tile0; tile < total && ok; tile += G, ++tiles_done) {
          if (tiles_done >= n_acc) {
            if (!TR_WAIT(tr_w0, mbar_wait(bar_accempty + 8 * acc_slot, acc_phase))) { ok = false; break; }
            tc_fence_after();
          }
          const uint32_t d0 = tmem_base + (uint32_t)acc_slot * p.acc_cols;
          uint32_t acc = 0;  // 0 only for the first MMA of the tile
          uint32_t row0 = 0;   // a unit fetched by TMA starts at the beginning of a row of positions
          if (swz) {
            const uint32_t Q0 = fdiv((uint32_t)tile, L.dCt) * (uint32_t)(L.Np - L.pair);
            row0 = 8u * (Q0 - fdiv(Q0, L.dWg) * (uint32_t)L.Wg);
          }
#pragma unroll 1
          for (int u = 0, t = 0; u < n_units && ok; ++u) {
            if (!TR_WAIT(tr_w1, mbar_wait(bar_afull + 8 * a_slot, a_phase))) { ok = false; break; }
            tc_fence_after();
            const uint32_t a_unit = a_base + (uint32_t)a_slot * a_slot_units + row0;
            const int pu = u & (n_pu - 1), t_last = FP4 || pu == 0 ? end[0] : pu == 1 ? end[1] : pu == 2 ? end[2] : end[3];
            if (pu == 0) t = 0;
#define G_ISSUE(KP)                                                                                                  \
  ok = g_issue_block<MODE, KP>(L, st_steps, t, t_last, a_fixed, k_step, a_unit, w_base, b_slot_units, d0, idesc, acc, NS, bar_bfull, bar_bempty, b_slot, \
                               b_phase, leader, sf, tr_w2)
            if (kpt == 4) G_ISSUE(4);
            else if (kpt == 2) G_ISSUE(2);
            else if (kpt == 3) G_ISSUE(3);
            else G_ISSUE(1);
#undef G_ISSUE
            t = t_last;
            if (!ok) break;
            if (leader) tc_commit(bar_aempty + 8 * a_slot);  // the activation unit may be overwritten
            if (++a_slot == NA) { a_slot = 0; a_phase ^= 1u; }
          }
          if (!ok) break;
          if (leader) tc_commit(bar_accfull + 8 * full_slot);  // fires when this tile's MMAs are complete
          full_slot = (full_slot + 1) & 3;
          if (++acc_slot == n_acc) { acc_slot = 0; acc_phase ^= 1u; }
        }
        ok = __all_sync(0xffffffffu, ok);
      }
      if (!ok && leader && !*abort_flag) {
        *abort_flag = 1;
        raise_status(p.status, 3);
      }
      if (leader) TR_REPORT(1, clock64() - tr_t0, tr_w0, tr_w1, tr_w2);
    }
    __syncwarp();
  } else if (warp < 2 + G_EW) {
    // ------------------------------------------------ epilogue warps
    grid_dep_wait();  // an earlier kernel in the stream may still read the output buffers
    // Warp w reads TMEM lanes 32*(w%4)..: 32 rows of the weight operand = 32 channels (or, with 8 pixels per
    // position, 16 channels of two pixels).  32 columns = 32 positions are read at a time.
    const int ew = warp - 2;
    const int rq = warp & 3, half = ew >> 2;
    const int row = rq * 32 + lane;
    const int n_acc = p.n_acc;
    uint32_t seq = 0;   // tile of this CTA, over all problems
    int acc_slot = 0;   // its buffer: seq % n_acc
    long long tr_w0 = 0, tr_t0 = clock64();
    (void)tr_w0; (void)tr_t0;
    for (;;) {
      const GTile* const T = reinterpret_cast<const GTile*>(epi_smem) + (seq & 3u);
      const uint32_t tile_phase = (seq >> 2) & 1u;   // (acc_full and the tables are indexed and flip alike)
      if (!wait_phase(bar_tabfull + 8u * (seq & 3u), tile_phase, 100, 6)) break;
      const int4 h0 = *reinterpret_cast<const int4*>(&T->l), h1 = *reinterpret_cast<const int4*>(&T->K);
      const int l = h0.x, n_slices = h0.w, K = h1.x, kp_log = h1.y, lg = F16 ? 0 : h1.z;
      const bool pair = F16 && h1.z;   // (see g_pairs)
      if (l < 0) break;   // no more tiles
      const int out_kind = WORDS ? (int)p.out_type[0] : OUTK == OUT_SIGNS ? 2 : h1.w & 3;
      uint32_t* const out32 = reinterpret_cast<uint32_t*>(p.out[l]);  // int32 and fp32 outputs share the layout
      // this lane's row of the weight operand: channel c of pixel g of a position's group, or of a copy of the channels
      const int c_lane = pair ? 16 * rq + (lane & 15) : row & ((1 << kp_log) - 1), c_warp = pair ? 16 * rq : (rq * 32) & ((1 << kp_log) - 1);   // (_warp: of lane 0)
      const int g_lane = lg ? row >> kp_log : 0, g_warp = lg ? (rq * 32) >> kp_log : 0;
      // the warps of a lane quarter, and the copies, take the 32-column slices in turn
      const int s_first = half + (lg || pair ? 0 : 2 * ((rq * 32) >> kp_log)), s_step = lg || pair ? 2 : 2 << (7 - kp_log);
      const int co = h0.z + c_lane, co_warp = h0.z + c_warp;
      const bool active = co_warp < K;   // does any of the warp's rows hold a channel?
      const float al = T->alpha[c_lane], minus_threshold = WORDS ? 0.f : T->minus_threshold[c_lane];
      const uint32_t flip = al < 0.f ? 0u : 0xffffffffu;   // (the bit is set below the threshold, or - where the sign bit of the difference is clear - from there on)
      {
        if (!TR_WAIT(tr_w0, wait_phase(bar_accfull + 8u * (seq & 3u), tile_phase, 100, 4))) break;
        tc_fence_after();
        const uint32_t d0 = tmem_base + (uint32_t)acc_slot * p.acc_cols + ((uint32_t)(rq * 32) << 16);
        // this warp has read its part of the accumulator buffer: hand it back to the MMA issuer
        auto release = [&]() {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_accempty + 8 * acc_slot);
        };
        if (!active || s_first >= n_slices) {
          release();
        } else {
          uint32_t* const obase = out32 + (size_t)((uint32_t)(g_lane * K + co));
          uint32_t first = 0;   // signs: the bits of the slice before, where that waits for this one
          bool held = false;
          // this lane's column of slice s: word w of the warp's channels (the table's offsets are those of a pixel's words)
          auto store_signs = [&](int s, uint32_t w) {
            const uint32_t here = 1u << lane, Kw = (uint32_t)(K + 31) >> 5;
            const uint32_t at = T->offset[32 * s + lane] + (uint32_t)g_warp * Kw + (uint32_t)(co_warp >> 5);
            if (kp_log >= 5) {
              if (T->mask[g_warp * G_MAX_CHUNKS + s] & here) {
                if (TAGGED && out_kind == 3) g_st_tagged(out32, at, w, tag);
                else out32[at] = w;
              }
            } else {   // 16 rows per pixel: one word each for two pixels
              const bool one = T->mask[g_warp * G_MAX_CHUNKS + s] & here, two = T->mask[(g_warp + 1) * G_MAX_CHUNKS + s] & here;
              if (TAGGED && out_kind == 3) {
                if (one) g_st_tagged(out32, at, w & 0xffffu, tag);
                if (two) g_st_tagged(out32, at + 1, w >> 16, tag);
              } else {
                if (one) out32[at] = w & 0xffffu;
                if (two) out32[at + 1] = w >> 16;
              }
            }
          };
          // (a last slice of 16 columns is read as 32: the others belong to the next buffer or the scales and go nowhere)
#pragma unroll 1
          for (int s = s_first; s < n_slices; s += s_step) {
            uint32_t v[32];
            __syncwarp();   // the load is a warp-wide instruction
            tmem_ld32(d0 + (uint32_t)(32 * s), v);
            if (F16 && pair) {
              // Lanes 0..15 hold a channel's sums over one and a half columns of the kernel, lanes 16..31 those over the others, which belong to
              // the position before: the lower lanes put even positions together and the upper ones odd positions, a shuffle for
              // both.  A store writes 16 channels of two positions.
              uint32_t next = 0;
              const int after = 32 * s + 32;   // the upper lanes need the first column of the next slice
              if (after < lay[l].Np) next = tmem_ld1(d0 + (uint32_t)after);
              if (s + s_step >= n_slices) release();
              const bool upper = lane >= 16;
              const uint32_t mask = co < K ? T->mask[s] >> (lane >> 4) : 0u;
              const uint32_t* const at = &T->offset[32 * s + (lane >> 4)];
#pragma unroll
              for (int e = 0; e < 32; e += 2) {
                const float other = __uint_as_float(__shfl_xor_sync(0xffffffffu, v[e + 1], 16));
                const float mine = __uint_as_float(upper ? (e + 2 < 32 ? v[e + 2] : next) : v[e]);
                const uint32_t y = __float_as_uint(__fmul_rn(__fadd_rn(mine, other), al));
                asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p st.global.b32 [%0], %1;\n\t}" ::"l"(obase + at[e]), "r"(y),
                             "r"(mask & (1u << e))
                             : "memory");
              }
              continue;
            }
            if (s + s_step >= n_slices) release();
            if (WORDS || out_kind < 2) {
              const uint32_t mask = co < K ? T->mask[g_lane * G_MAX_CHUNKS + s] : 0u;
              // Scaled (or converted) first, stored by one loop for both: a store loop for each kind doubles the code, and the
              // roles share the instruction caches (with two loops the ResNet-18 group took 7 % longer, the 1x1 layers 4 %).
              // (Pairs are multiplied together, each half rounded as by itself: ResNet-20 group at batch 128 36.6 and 35.9 us, ResNet-18 94.0 and 92.6.)
              if (out_kind == 0) {
#pragma unroll
                for (int e = 0; e < 32; e += 2)
                  asm("{\n\t.reg .b64 x, a;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 a, {%2, %2};\n\tmul.rn.f32x2 x, x, a;\n\tmov.b64 {%0, %1}, x;\n\t}" : "+r"(v[e]), "+r"(v[e + 1]) : "f"(al));
              } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = (uint32_t)__float2int_rn(__uint_as_float(v[e]));   // integer sums: exact
              }
              // One column = one pixel of 32 channels per step: a predicated store of a whole 128-byte line.
#pragma unroll
              for (int e = 0; e < 32; e += 4) {
                const uint4 o4 = *reinterpret_cast<const uint4*>(&T->offset[32 * s + e]);
                const uint32_t o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  if (STREAM)
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p st.global.cs.b32 [%0], %1;\n\t}" ::"l"(obase + o[j]),
                                 "r"(v[e + j]), "r"(mask & (1u << (e + j)))
                                 : "memory");
                  else
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p st.global.b32 [%0], %1;\n\t}" ::"l"(obase + o[j]),
                                 "r"(v[e + j]), "r"(mask & (1u << (e + j)))
                                 : "memory");
                }
              }
            } else {
              // Packed signs of the scaled output (Algorithm 1: the next layer consumes sign(a)): a sum is compared with the
              // channel's threshold (g_sign_threshold; the difference of two integers is exact), a lane gathers the bits of its
              // channel over the 32 columns, and a 32 x 32 bit transposition in the warp gives lane j the word of column j.
              // Bound by latency: 204 cycles of a slice's 970 went into scaled and shifted bits, 303 into the transposition, 290 into
              // the table and the store.  The transposition and the stores behind it are a chain, so two slices go through them
              // together.  Group of the 1x1 layers at batch 16 68.9 and 64.8 us, ResNet-18 68.8 and 65.2, ResNet-34 stack at batch 128
              // 360 and 349; one slice a warp (64 channels of 56x56, 4 images) 5.21 and 5.24.  (The vote on a comparison is a column's word
              // without any transposition, but 32 votes and selections take longer: those groups 79 and 75 us.)
              unsigned long long t2;
              asm("mov.b64 %0, {%1, %1};" : "=l"(t2) : "f"(minus_threshold));
              uint32_t part[4] = {0, 0, 0, 0};   // four chains of eight bits: one of 32 waits for itself
#pragma unroll
              for (int e = 6; e >= 0; e -= 2) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  unsigned long long x;
                  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(v[8 * c + e]), "r"(v[8 * c + e + 1]));
                  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(x) : "l"(t2));
                  uint32_t y0, y1;
                  asm("mov.b64 {%0, %1}, %2;" : "=r"(y0), "=r"(y1) : "l"(x));
                  part[c] = __funnelshift_l(y1, part[c], 1);
                  part[c] = __funnelshift_l(y0, part[c], 1);
                }
              }
              uint32_t w = (part[0] | (part[1] << 8) | (part[2] << 16) | (part[3] << 24)) ^ flip;
              if (!held && s + s_step < n_slices) {
                first = w;
                held = true;
                continue;
              }
              g_transpose32(w, first, lane);
              store_signs(s, w);
              if (held) store_signs(s - s_step, first);
              held = false;
            }
          }
        }
        if (CHAIN && (h1.w & 4) && active && s_first < n_slices) {
          // one of the CTA's last tiles in this member of a chain: this warp's part is written, the successor may read it
          __syncwarp();
          if (lane == 0) {
            __threadfence();   // (cumulative: it covers what the other lanes wrote before the barrier)
            asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(lay[l].done + h0.y) : "memory");
          }
        }
      }
      __syncwarp();   // the table has been read
      if (lane == 0) mbar_arrive(bar_tabempty + 8u * (seq & 3u));
      // The CTA's last tile: no look at the table for an end mark (independent problems: smallest layer 4.14 and 4.04 us, fp16 layer of 64
      // channels 6.19 and 6.08; in chains the larger code costs more than that gains).
      if (!CHAIN && !TAGGED && (h1.w & 8)) break;
      ++seq;
      if (++acc_slot == n_acc) acc_slot = 0;
    }
    if (warp == 2 && lane == 0) TR_REPORT(2, clock64() - tr_t0, tr_w0, 0, 0);
  } else if (warp == 13) {
    // ------------------------------------------------ table warp
    // Writes down what the epilogue needs of every tile, up to four tiles ahead: where its columns' pixels go, which
    // of them exist, the scales and thresholds.  Done by the epilogue warps themselves, each for itself, this took a
    // fifth of their time (the geometry is a chain of divisions, and a global load behind a warp's own stores waits
    // until those have drained).
    if (p.after_weights > 1) grid_dep_wait();
    bool ok = true;
    uint32_t seq = 0;
    // Chains on counters: the oldest tile whose counter has not been advanced.  The fence between a tile's signs and its counter waits
    // for the stores to arrive, 1200 cycles: done by every epilogue warp for its part it was a fifth of their time in the shallow layers
    // of large batches.  Here it is done once a tile, beside them (their arrivals and the fence are cumulative: it covers what they
    // wrote).  That is some 300 cycles later, so the last two of a CTA's tiles in a member, and members with fewer than three tiles a
    // CTA, whose successors wait for just those, are left to the epilogue warps.  ResNet-34 stack at batch 128 344 and 330 us, ResNet-18 at 96
    // 156.4 and 151.8; without the line at three tiles ResNet-34 at 64 250 and 255, with it at four ResNet-34 at 128 338.
    uint32_t unsaid = 0;
    auto say_written = [&]() {
      const GTile* const T = reinterpret_cast<const GTile*>(epi_smem) + (unsaid & 3u);
      if (T->l + 1 < p.n_layers && !(T->out_kind & 4)) {
        // the epilogue warps that had something to write (see there): lane w stands for warp 2 + w
        const int first_row = ((lane + 2) & 3) * 32, first_slice = (lane >> 2) + (T->lg ? 0 : 2 * (first_row >> T->kp_log));
        const uint32_t wrote = __ballot_sync(0xffffffffu, lane < G_EW && T->co + (first_row & ((1 << T->kp_log) - 1)) < T->K && first_slice < T->n_slices);
        if (lane == 0) {
          __threadfence();
          asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(lay[T->l].done + T->mg), "r"((uint32_t)__popc(wrote)) : "memory");
        }
        __syncwarp();
      }
      ++unsaid;
    };
    auto take_slot = [&]() -> bool {
      if (CHAIN) {   // what has been written meanwhile is said first
        while (unsaid < seq && seq - unsaid < G_TILES && __all_sync(0xffffffffu, mbar_test(bar_tabempty + 8u * (unsaid & 3u), (unsaid >> 2) & 1u)))
          say_written();
        if (seq - unsaid < G_TILES) return true;
      }
      if (seq < G_TILES) return true;
      if (!wait_phase(bar_tabempty + 8u * (seq & 3u), ((seq >> 2) & 1u) ^ 1u, 100, 7)) return false;
      if (CHAIN) say_written();
      return true;
    };
#pragma unroll 1
    for (int l = 0; l < p.n_layers && ok; ++l) {
      const GLayer& L = lay[l];
      const FastDiv dWg = L.dWg, dHq = L.dHq, dCt = L.dCt;
      const int Np = L.Np, K = L.K, Wg = L.Wg, Hq = L.Hq, Ho = L.Ho, Wo = L.Wo, lg = L.lg, n_ct = L.n_ct, total = L.total_tiles;
      const uint32_t Qtot = L.Qtot;
      const int own = Np - (F16 ? L.pair : 0);   // positions of a tile
      const int n_slices = (Np + 31) >> 5;
      const int out_kind = WORDS ? (int)p.out_type[0] : OUTK == OUT_SIGNS ? 2 : (int)p.out_type[l];
      const uint32_t scale = out_kind >= 2 ? (uint32_t)(K + 31) >> 5 : (uint32_t)K;   // words of a pixel
      const bool few = total < 3 * G;
#pragma unroll 1
      for (int tile = L.first; tile < total; tile += G, ++seq) {
        if (!take_slot()) { ok = false; break; }
        GTile* const T = reinterpret_cast<GTile*>(epi_smem) + (seq & 3u);
        const int mg = (int)fdiv((uint32_t)tile, dCt), co = (tile - mg * n_ct) * G_ROWS;
        float al[4], th[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = co + 32 * i + lane;
          al[i] = c < K ? g_ld<LATE>(L.alpha + c) : 0.f;
          th[i] = !WORDS && c < K ? __ldg(L.threshold + c) : __int_as_float(0x7f800000);   // (no sum reaches infinity: bits of channels that do not exist are 0)
        }
        if (lane == 0) {
          *reinterpret_cast<int4*>(&T->l) = make_int4(l, mg, co, n_slices);
          *reinterpret_cast<int4*>(&T->K) = make_int4(K, L.kp_log, F16 ? L.pair : lg, out_kind | (CHAIN && (few || tile + 2 * G >= total) ? 4 : 0) |
                                                                 (!CHAIN && !TAGGED && tile + G >= total && L.next >= p.n_layers ? 8 : 0));
        }
#pragma unroll 1
        for (int s = 0; s < n_slices; ++s) {
          const int c = 32 * s + lane;
          const uint32_t q = (uint32_t)mg * (uint32_t)own + (uint32_t)c;
          const uint32_t rg = fdiv(q, dWg), n = fdiv(rg, dHq);
          const int x = (int)(q - rg * (uint32_t)Wg) << lg, y = (int)(rg - n * (uint32_t)Hq);
          T->offset[c] = ((n * (uint32_t)Ho + (uint32_t)y) * (uint32_t)Wo + (uint32_t)x) * scale;
          const int rem = c < own && q < Qtot && y < Ho ? Wo - x : 0;   // pixels from x to the end of the row
#pragma unroll 1
          for (int g = 0; g < (1 << lg); ++g) {
            const uint32_t m = __ballot_sync(0xffffffffu, g < rem);
            if (lane == 0) T->mask[g * G_MAX_CHUNKS + s] = m;
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          T->alpha[32 * i + lane] = al[i];
          if (!WORDS) T->minus_threshold[32 * i + lane] = g_minus_threshold(th[i]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tabfull + 8u * (seq & 3u));
      }
    }
    if (ok && take_slot()) {   // the end mark
      if (lane == 0) {
        (reinterpret_cast<GTile*>(epi_smem) + (seq & 3u))->l = -1;
        mbar_arrive(bar_tabfull + 8u * (seq & 3u));
      }
      __syncwarp();
      if (CHAIN) {   // the last tiles
        for (const uint32_t tiles = seq; ok && unsaid < tiles;) {
          seq = unsaid + G_TILES;
          ok = take_slot();
        }
      }
    }
  } else if (CHAIN && warp == 17) {
    // ------------------------------------------------ dependency warp (chains)
    // Waits, tile by tile, until the predecessor has written every input pixel of the tile, and counts the tiles whose
    // input may be read.  One warp per CTA looks at the counters: when every expander warp did, the looks of all CTAs at
    // the same few lines of L2 held up the counters themselves.
    uint32_t done = 0;
    for (int l = 0; l < p.n_layers; ++l) {
      const GLayer& L = lay[l];
      const uint2* const deps = L.deps;
      const uint32_t* const ctr = L.prev_done;
      const uint32_t target = L.prev_target;
      const FastDiv dCt = L.dCt;
      const int total = L.total_tiles;
      bool ok = true;
      for (int tile = L.first; tile < total && ok; tile += G) {
        if (deps) {
          const uint2 d = __ldg(deps + fdiv((uint32_t)tile, dCt));
          ok = g_wait_counters(ctr, d.x, d.y, target, lane, abort_flag);
        }
        ++done;
        if (ok && lane == 0) asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(ready_tiles)), "r"(done) : "memory");
      }
      if (!ok) {
        if (lane == 0 && !*abort_flag) {
          *abort_flag = 1;
          raise_status(p.status, 5);
        }
        break;
      }
    }
  } else if (warp != 17) {
    // ------------------------------------------------ expanders (warps 10-12, 14-16, 18, 19)
    // Fill activation unit (problem, tile, channel block) of the ring: for every plane, row and
    // 32-channel word, bits -> one 16-byte chunk of nibbles (fp16: 8-channel chunks are copied).
    const int et = (warp - 10 - (warp > 13) - (warp > 17)) * 32 + lane;  // rank among the expander threads
    int a_slot = 0;
    long long a_done = 0;
    uint32_t a_phase = 1;  // parity of the previous use of a slot (valid from the second lap)
    bool stop = false;
    long long tr_w0 = 0, tr_t0 = clock64();
    (void)tr_w0; (void)tr_t0; (void)a_done;
    // until the MMAs have read what slot a_slot held
    auto wait_slot = [&]() -> bool { return TR_WAIT(tr_w0, wait_phase(bar_aempty + 8 * a_slot, a_phase, 64, 1)); };
    // this warp's part of a unit is written: make it visible to the tensor core and say so
    auto unit_done = [&](int slot) {
      fence_proxy_async();  // generic-proxy writes -> visible to the tensor core's reads
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_afull + 8 * slot);
    };
    if constexpr (FP4) {
      // A two-stage software pipeline per thread: a "group" is up to four items of one unit - an item is the words of
      // one position in one plane that one load brings - and the loads of group g + 1 are issued (into registers)
      // before group g is expanded into shared memory, so that a unit does not cost a full round trip to memory.
      // A thread keeps the geometry of its position while it walks through the planes and words: these eight warps
      // are bound by how many instructions a unit takes one warp, not by the issue slots of the SM.
      constexpr int XI = CHAIN || TAGGED ? G_EXP_ITEMS / 2 : G_EXP_ITEMS;   // (a chain's tiles are small: less code is worth 2 %)
      struct XGroup {
        uint4 t[XI];       // the items' words (one, two or four of them)
        uint32_t da[XI];   // where an item's first chunk goes
        uint32_t cstride;  // bytes from one chunk to the next
        uint32_t flags;    // bit j: item j exists; bit 4 + j: its words exist (the pixel is inside the image); bits
                           // 12..14: words per item; 9: first group of its unit; 10: last group of its unit; 11: words with tags
        const uint64_t* src[TAGGED ? XI : 1];   // words with tags: where they are, to be looked at again
      };
      // The expander warps form XG teams that take the units in turn (the ring has a multiple of XG slots, so a
      // slot always belongs to the same team): with few rows per unit a unit is a chain of latencies, and two
      // chains in flight are what doubles the rate.
      constexpr int XG = G_XTEAMS, XT = G_EXP_THREADS / XG;
      // (from the warp's number, which is known to be uniform: single layers 1 % faster; chains with tags are as much slower)
      const int gx = TAGGED ? et / XT : (warp - 10 - (warp > 13) - (warp > 17)) / (XT / 32), etg = et % XT;
      // issue side: the unit (il, itile, icb) with sequence number iu, and the next item to load in it
      int il = 0, itile = 0, itotal = 0, icb = 0, i_slot = 0, iu = 0;
      int pos0 = 0, ipl = 0, ik0 = 0;                 // first position of the thread's row of positions, plane, word
      int Rr = 0, n_cb = 0, cbc = 0, Cw = 0, planes = 1, kstep = 2, cpl = 0, H = 0, W = 0, cs = 0;
      uint32_t Q0 = 0;
      int row = 0, col = 0, img_row = 0;              // of this thread's position: input row and column in plane 0, n*H
      bool inside = false;                            // it lies in the batch
      const uint32_t* act = nullptr;
      bool ivalid = false, ready = false;             // is there a unit; may its input be read (chain)
      uint32_t tile_seq = ~0u;                        // tile of the CTA, over all problems
      auto enter_tile = [&]() {
        const GLayer& L = lay[il];
        const uint32_t mg = fdiv((uint32_t)itile, L.dCt);
        Q0 = mg * (uint32_t)L.Np;
        ready = !CHAIN;
        ++tile_seq;
      };
      // The CTA's first tile in layer il (n_layers: there is none).  Which layers it has tiles in comes from the host: a search
      // for the next one in here was compiled wrongly for the variant with tags (nvcc 12.9.86: found in layer 1, it went on with the
      // first tile of layer 2; not with the compiler's optimiser at -O1, whatever ptxas did, nor with a note taken in the loop).
      auto enter_layer = [&]() {
        ivalid = il < p.n_layers;
        if (!ivalid) return;
        const GLayer& L = lay[il];
        itile = L.first; itotal = L.total_tiles;
        Rr = L.Rr; n_cb = L.n_cb; cbc = L.cb_chunks; Cw = L.Cw; planes = L.n_planes; cpl = L.cpl; H = L.H; W = L.W; cs = L.cs;
        act = reinterpret_cast<const uint32_t*>(p.act[il]);
        kstep = g_word_step(Cw, cbc);
        if (TAGGED && il > 0 && kstep > 2) kstep = 2;
        icb = 0;
        enter_tile();
      };
      auto next_unit = [&]() {     // the unit after (il, itile, icb) in the CTA's sequence
        ++iu;
        i_slot = i_slot + 1 == NA ? 0 : i_slot + 1;
        if (++icb >= n_cb) {
          icb = 0;
          itile += G;
          if (itile >= itotal) {
            il = lay[il].next;
            enter_layer();
          } else {
            enter_tile();
          }
        }
      };
      auto seek_own = [&]() {      // on to this team's next unit
        while (ivalid && (iu % XG) != gx) next_unit();
      };
      // chain: may the tile's input be read?  (blocking: waits, bounded.)
      auto check_ready = [&](bool blocking) -> bool {
        for (uint32_t it = 0; CHAIN && !ready; ++it) {
          uint32_t v;
          asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(ready_tiles)) : "memory");
          ready = __all_sync(0xffffffffu, v > tile_seq);
          if (ready || !blocking || it >= (1u << 23) || __any_sync(0xffffffffu, *abort_flag != 0)) break;
          __nanosleep(20);
        }
        return ready;
      };
      // where position pos of the unit (il, itile) reads
      auto locate = [&](int pos) {
        const GLayer& L = lay[il];
        const uint32_t q = Q0 + (uint32_t)pos;
        const uint32_t rg = fdiv(q, L.dWg), n = fdiv(rg, L.dHq);
        row = L.rs * (int)(rg - n * (uint32_t)L.Hq) - L.pad;
        col = L.cm * (int)(q - rg * (uint32_t)L.Wg) - L.pad;
        img_row = (int)n * H;
        inside = q < L.Qtot;
      };
      auto issue = [&](XGroup& g) {   // loads of the group at the issue position; moves the position on
        const GLayer& L = lay[il];
        const bool fresh = CHAIN && L.deps != nullptr;   // written by other CTAs of this launch: read from L2
        const uint32_t cstride = (uint32_t)(planes * Rr) * 16u;
        const bool tagged = TAGGED && il > 0;   // (the first member's input is the caller's)
        uint32_t flags = ((uint32_t)kstep << 12) | ((pos0 | ipl | ik0) == 0 ? 0x200u : 0u) | (tagged ? 0x800u : 0u);
        // the items of a position are dealt to 2^tpl neighbouring threads, so that a small tile's are all looked at together
        // instead of one look after another
        const int items = cbc >> (kstep >> 1), tpl = !TAGGED ? 0 : items == 4 ? 2 : items == 2 ? 1 : 0;
        const int own = TAGGED ? (etg & ((1 << tpl) - 1)) * kstep : 0;   // this thread's words of a position start there
        const uint32_t unit = smem_u32(a_smem) + (uint32_t)i_slot * p.a_slot_bytes;
        bool ended = false;
#pragma unroll
        for (int j = 0; j < XI; ++j) {
          if (ended) break;
          const int pos = pos0 + (TAGGED ? etg >> tpl : etg), ik = ik0 + own;
          if (TAGGED && (ipl | ik0) == 0) locate(pos);
          const int r = row + (ipl >> cpl), c = col + cs * (ipl & ((1 << cpl) - 1)), word = icb * cbc + ik;
          const bool on = inside && pos < Rr && (uint32_t)r < (uint32_t)H && (uint32_t)c < (uint32_t)W && word < Cw;
          g.da[j] = unit + (uint32_t)ik * cstride + (uint32_t)(ipl * Rr + pos) * 16u;
          g.t[j] = make_uint4(0, 0, 0, 0);
          if (pos < Rr) flags |= 1u << j;
          if (on) {
            flags |= 0x10u << j;
            const size_t at = wide_mul((uint32_t)((img_row + r) * W + c), (uint32_t)Cw) + (size_t)word;
            const uint32_t* src = act + at;
            if (TAGGED && tagged) {
              g.src[TAGGED ? j : 0] = reinterpret_cast<const uint64_t*>(act) + at;
              g_ld_tagged(g.t[j], g.src[TAGGED ? j : 0], kstep);
            } else if (kstep == 4) {
              g.t[j] = g_ld_act<LATE, uint4>(src, fresh);
            } else if (kstep == 2) {
              const uint2 v = g_ld_act<LATE, uint2>(src, fresh);
              g.t[j].x = v.x;
              g.t[j].y = v.y;
            } else {
              g.t[j].x = g_ld_act<LATE, uint32_t>(src, fresh);
            }
          }
          ik0 += TAGGED ? kstep << tpl : kstep;
          if (ik0 >= cbc) {
            ik0 = 0;
            if (++ipl == planes) {
              ipl = 0;
              pos0 += TAGGED ? XT >> tpl : XT;
              ended = pos0 >= Rr;
              if (!TAGGED && !ended) locate(pos0 + etg);
            }
          }
        }
        if (ended) {   // the unit ends with this group
          pos0 = 0;
          flags |= 0x400u;
          next_unit();
          seek_own();
          if (!TAGGED && ivalid) locate(etg);
        }
        g.cstride = cstride;
        g.flags = flags;
      };
      if (lay[0].first >= lay[0].total_tiles) il = lay[0].next;
      enter_layer();
      seek_own();
      if (!TAGGED && ivalid) locate(etg);
      // The activations may come from the previous kernel in the stream.  (What does not read them stands before the wait, and a unit's first
      // position is located when the unit before it has been issued: smallest layer 4.24 and 4.04 us, 256 channels 8.28 and 8.05, ragged layer 6.89 and
      // 6.67.  In chains of words with tags the latter costs 1 to 3 % on one image.)
      grid_dep_wait();
      if (!CHAIN && !TAGGED && (p.n_layers > 1 || lay[0].total_tiles > G)) {
        // Independent problems: all inputs exist when the launch starts and are small beside the L2 (1/29 of the
        // outputs; fp16 inputs are not: half of the outputs).  The CTAs pull them into L2 together, once, so that the
        // staging loads below see L2 latency instead of DRAM latency.  (Not where every CTA has one tile: its loads go out now anyway,
        // 0.3 us earlier without this; 14 single layers 1 %.)
#pragma unroll 1
        for (int l = 0; l < p.n_layers; ++l) {
          const GLayer& L = lay[l];
          const size_t bytes = (size_t)L.N * L.H * L.W * ((size_t)L.Cw * 4);
          const char* base = reinterpret_cast<const char*>(p.act[l]);
#pragma unroll 1
          for (size_t off = ((size_t)blockIdx.x * G_EXP_THREADS + et) * 128; off < bytes; off += (size_t)G * G_EXP_THREADS * 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(base + off));
        }
      }
      // completion side: this team's slots gx, gx + XG, ... of the ring
      a_slot = gx;
      XGroup cur, nxt = {};   // (a unit's last group leaves items unwritten, and all of them are copied)
      auto not_ready = [&]() {     // the wait for a chain's input ran out
        if (lane == 0 && !*abort_flag) {
          *abort_flag = 1;
          raise_status(p.status, 5);
        }
        stop = true;
      };
      auto expand = [&]() {        // the group in hand into shared memory
        if ((cur.flags & 0x200u) && a_done >= NA / XG && !wait_slot()) {
          stop = true;
          return;
        }
#pragma unroll
        for (int j = 0; j < XI; ++j) {
          if (cur.flags & (1u << j)) {
            const bool on = (cur.flags & (0x10u << j)) != 0;
            const uint32_t sign = on ? 0x88888888u : 0u, one = on ? 0x22222222u : 0u;
            const uint32_t d = cur.da[j], cst = cur.cstride;
            sts16(d, expand_word_fp4(cur.t[j].x, sign, one));
            if (cur.flags & 0x6000u) {
              sts16(d + cst, expand_word_fp4(cur.t[j].y, sign, one));
              if (cur.flags & 0x4000u) {
                sts16(d + 2 * cst, expand_word_fp4(cur.t[j].z, sign, one));
                sts16(d + 3 * cst, expand_word_fp4(cur.t[j].w, sign, one));
              }
            }
          }
        }
        if (cur.flags & 0x400u) {
          unit_done(a_slot);
          ++a_done;
          a_slot += XG;
          if (a_slot >= NA) { a_slot -= NA; a_phase ^= 1u; }
        }
      };
      // words with tags: looks (bounded) until all of the group's are this launch's, without a pause between the looks (with 20 ns from the
      // third on, ResNet-20 stacks 2 to 3.5 % slower, the others 1 to 1.5 %)
      auto settle = [&]() -> bool {
        const bool two = (cur.flags & 0x6000u) != 0;
#pragma unroll 1
        for (uint32_t it = 0;; ++it) {
          bool all = true;
#pragma unroll
          for (int j = 0; j < XI; ++j) {
            if ((cur.flags & (0x10u << j)) && (cur.t[j].y != tag || (two && cur.t[j].w != tag))) {
              all = false;
              g_ld_tagged(cur.t[j], cur.src[TAGGED ? j : 0], two ? 2 : 1);
            }
          }
          if (__all_sync(0xffffffffu, all)) break;
          if (it >= (1u << 21) || __any_sync(0xffffffffu, *abort_flag != 0)) return false;
        }
#pragma unroll
        for (int j = 0; j < XI; ++j) cur.t[j].y = cur.t[j].z;
        return true;
      };
      if constexpr (CHAIN) {
        bool nvalid = false;
        while (ivalid || nvalid) {
          if (!nvalid) {
            if (!check_ready(true)) {
              not_ready();
              break;
            }
            issue(nxt);
          }
          cur = nxt;
          // (the next input may depend on the unit in hand: it is only looked at, never waited for, here)
          nvalid = ivalid && check_ready(false);
          if (nvalid) issue(nxt);
          expand();
          if (stop) break;
        }
      } else {
        // One copy of the load issue instead of two: 10 KB of code.  (In chains on counters, whose tiles are small, two are 1 to 3 %
        // faster; chains of words with tags have not been timed with two.)
        bool in_hand = false;   // is there a group to expand?
#pragma unroll 1
        for (;;) {
          const bool more = ivalid;
          if (more) issue(nxt);
          if (TAGGED && in_hand && (cur.flags & 0x800u) && !settle()) {
            not_ready();
            break;
          }
          if (in_hand) expand();
          if (!more || stop) break;
          cur = nxt;
          in_hand = true;
        }
      }
    } else {
      int pending = 0, oldest = 0;   // units whose copies are still in flight, the slot of the oldest
      // For the kernel before, from which the activations may come: right before the first copies (fp16 ResNet-18 group at batch 8 37.8 and
      // 36.6 us, one layer of 64 channels 6.07 and 5.94, rows copied by the threads 6.99 and 6.80).
      bool waited = false;
      auto complete = [&](int left) {   // say that all of them but the `left` newest are written
#pragma unroll 1
        while (pending > left) {
          if (pending == 3) asm volatile("cp.async.wait_group 2;" ::: "memory");
          else if (pending == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
          else asm volatile("cp.async.wait_group 0;" ::: "memory");
          unit_done(oldest);
          oldest = oldest + 1 == NA ? 0 : oldest + 1;
          --pending;
        }
      };
#pragma unroll 1
      for (int l = 0; l < p.n_layers && !stop; ++l) {
        const GLayer& L = lay[l];
        const int Rr = L.Rr, n_cb = L.n_cb, cb_chunks = L.cb_chunks, all_rows = L.n_planes * Rr;
        const int C = L.C, total = L.total_tiles;
        const FastDiv dCt = L.dCt, dRr = L.dRr;
        const void* act = p.act[l];
        const bool vec = (C & 7) == 0;                   // rows start at multiples of 16 bytes
        if (L.tma) {
          // The rows of positions a tile touches are fetched with one copy of 64 channels per row and plane, dealt to the
          // warps (issuing them all from one thread took longer than the MMAs of a small map): padding columns, rows
          // above and below the image and channels past the last are out of the tensor's bounds and read as zeros.
          const uint32_t row_bytes = (uint32_t)L.Wg * 128u, ew = (uint32_t)(et >> 5), Hq = (uint32_t)L.Hq;
          const FastDiv dHq = L.dHq, dWg = L.dWg;
          const int n_pu = L.n_pu, rs = L.rs, pad = L.pad, cpl = L.cpl, own = L.Np - L.pair;
#pragma unroll 1
          for (int tile = L.first; tile < total && !stop; tile += G) {
            const uint32_t Q0 = fdiv((uint32_t)tile, dCt) * (uint32_t)own;
            const uint32_t r_first = fdiv(Q0, dWg), r_last = fdiv(Q0 + (uint32_t)Rr - 1u, dWg);
#pragma unroll 1
            for (int u = 0; u < n_cb * n_pu; ++u) {
              if (pending) complete(0);
              if (a_done >= NA && !wait_slot()) {
                stop = true;
                break;
              }
              if (!waited) {   // (what does not read them stands before)
                grid_dep_wait();
                waited = true;
              }
              if (lane == 0) {
                const uint32_t bar = bar_afull + 8u * (uint32_t)a_slot, unit = smem_u32(a_smem) + (uint32_t)a_slot * p.a_slot_bytes;
                const int pl = u & (n_pu - 1), cb = n_pu == 1 ? u : u >> 2;
                const int x = (pl & (rs - 1)) - pad, y0 = (pl >> cpl) - pad;
                const uint32_t mine = r_last >= r_first + ew ? ((r_last - r_first - ew) >> 3) + 1u : 0u;   // this warp's rows
                if (mine) mbar_expect_tx(bar, mine * row_bytes);
                else mbar_arrive(bar);
                for (uint32_t r = r_first + ew; r <= r_last; r += G_EW) {
                  const uint32_t n = fdiv(r, dHq);
                  tma_load_4d(unit + (r - r_first) * row_bytes, &maps.m[l], cb * 64, x, rs * (int)(r - n * Hq) + y0, (int)n, bar);
                }
              }
              __syncwarp();
              ++a_done;
              if (++a_slot == NA) { a_slot = 0; a_phase ^= 1u; }
            }
          }
          continue;
        }
        oldest = pending ? oldest : a_slot;
#pragma unroll 1
        for (int tile = L.first; tile < total && !stop; tile += G) {
          const uint32_t Q0 = fdiv((uint32_t)tile, dCt) * (uint32_t)L.Np;
          // Input pixel of every staged row, once per tile; a thread reads back only entries it wrote itself.
          // (plane, row) pairs form one index space f = plane*Rr + row, dealt to the threads at a stride of
          // the expander count.
#pragma unroll 1
          for (int f = et; f < all_rows; f += G_EXP_THREADS) {
            const int pl = (int)fdiv((uint32_t)f, dRr);
            pix_tab[f] = g_position_to_pixel(L, Q0 + (uint32_t)(f - pl * Rr), pl);
          }
#pragma unroll 1
          for (int cb = 0; cb < n_cb; ++cb) {
            // the next slot is not free yet: finish the units in flight first, the MMAs may be waiting for them
            if (pending && a_done >= NA &&
                !__shfl_sync(0xffffffffu, lane == 0 ? (int)mbar_test(bar_aempty + 8 * a_slot, a_phase) : 0, 0))
              complete(0);
            if (a_done >= NA && !wait_slot()) {
              stop = true;
              break;
            }
            if (!waited) {
              grid_dep_wait();
              waited = true;
            }
            const uint32_t unit = smem_u32(a_smem) + (uint32_t)a_slot * p.a_slot_bytes;
            const uint32_t cstride = (uint32_t)all_rows * 16u;   // bytes from one chunk to the next
            if (vec) {
              // Asynchronous 16-byte copies straight into the unit (zero-filled where the row is padding or the channels
              // end), all in flight together.  A warp takes 32 rows at a time, its lanes run along a row's chunks
              // first: an instruction reads whole lines.
              const int per = 32 / cb_chunks, sub = lane / cb_chunks, chunk = lane - sub * cb_chunks;
              const int ch = (cb * cb_chunks + chunk) * 8;  // first channel of this lane's chunk
              for (int rb = et; rb - lane < all_rows; rb += G_EXP_THREADS) {
                const int mine = rb < all_rows ? pix_tab[rb] : -2;
                const uint32_t dst = unit + (uint32_t)(rb - lane) * 16u + (uint32_t)chunk * cstride;
                for (int r0 = 0; r0 < 32; r0 += per) {
                  const int px = __shfl_sync(0xffffffffu, mine, r0 + sub);
                  if (sub >= per || r0 + sub >= 32 || px == -2) continue;
                  const bool on = px >= 0 && ch < C;
                  const __half* src = (const __half*)act + (on ? wide_mul((uint32_t)px, (uint32_t)C) + ch : 0);
                  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)(r0 + sub) * 16u), "l"(src),
                               "r"(on ? 16 : 0)
                               : "memory");
                }
              }
            } else {
#pragma unroll 1
              for (int f = et; f < all_rows; f += G_EXP_THREADS) {
                const int px = pix_tab[f];
#pragma unroll 1
                for (int c0 = 0; c0 < cb_chunks; ++c0) {
                  const int ch = (cb * cb_chunks + c0) * 8;
                  uint32_t w[4] = {0, 0, 0, 0};
                  if (px >= 0) {
                    const __half* src = (const __half*)act + wide_mul((uint32_t)px, (uint32_t)C) + ch;
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                      if (ch + e < C) w[e >> 1] |= (uint32_t)__half_as_ushort(src[e]) << (16 * (e & 1));
                  }
                  sts16(unit + (uint32_t)f * 16u + (uint32_t)c0 * cstride, make_uint4(w[0], w[1], w[2], w[3]));
                }
              }
            }
            // the unit's copies stay in flight while the next two units' are issued
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (++pending == 3) complete(2);
            ++a_done;
            if (++a_slot == NA) { a_slot = 0; a_phase ^= 1u; }
          }
        }
      }
      if (!stop) complete(0);
      asm volatile("cp.async.wait_all;" ::: "memory");
      if (stop && et == 0) {   // giving up: never leave with copies in flight (bounded)
        for (int i = 0; i < NA && i < a_done; ++i) {
          const long long last = a_done - 1 - i;
          mbar_wait_backoff(bar_afull + 8u * (uint32_t)(last % NA), (uint32_t)((last / NA) & 1), 64);
        }
      }
    }
    if (et == 0) TR_REPORT(3, clock64() - tr_t0, tr_w0, 0, 0);
  }

  // ---------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (TAGGED && tid == 0)
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p.launches.count), "l"(g_launch_share(p.launches, blockIdx.x, gridDim.x))
                 : "memory");
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// ------------------------------------------------------------------ host side
struct GroupDev {
  int count = 0, act_type = 0, mode = M_FP4;
  int order[SNN_GROUP_MAX] = {};  // which of the caller's problems each one is
  int kind = TCG_WORDS;           // what the tiles were planned for (word outputs, packed signs, chain)
  bool stream = false;            // word outputs leave the L2 first (g_streams)
  int chain = 0;                  // 1: member i + 1 reads the packed signs member i writes (one launch, on counters or with tags)
  uint8_t* mem = nullptr;         // all device memory of the group; the pointers below lie in it
  uint8_t* chain_buf = nullptr;   // the packed signs between the members, one buffer per boundary
  size_t chain_off[SNN_GROUP_MAX] = {};
  int tagged = 0;                 // a chain of words with tags (and without counters)
  uint32_t* done = nullptr;       // a chain on counters: those of all members' position tiles
  size_t done_words = 0;
  GLayer* layers_dev = nullptr;   // [count]
  uint32_t* ranks = nullptr;      // [count][grid] tile assignment, see GParams
  GParams p{};                    // everything but the per-call pointers
  size_t smem = 0;
  int grid = 0;
  struct Map { bool tma; int C, W, H, N, stride, box; } map[SNN_GROUP_MAX] = {};   // fp16 activations fetched by TMA
};

namespace {

// The driver's tensor-map encoder, looked up once (the library does not link the driver).
using MapEncoder = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
MapEncoder g_map_encoder() {
  static const MapEncoder f = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<MapEncoder>(p);
  }();
  return f;
}

// The packed-sign bit of a channel is fl(fl(alpha*S) + shift) >= 0 for an integer sum S of -most..most: two roundings of a function that
// never falls (alpha >= 0) or never rises (alpha < 0) along S, so the bit changes once, and comparing S with where it does is
// the same decision.  Returns the least S whose bit is set (alpha < 0: clear), most + 1 where there is none.
__device__ float g_sign_threshold(float alpha, float shift, int most) {
  int lo = -most, hi = most + 1;
  while (lo < hi) {
    const int mid = lo + (hi - lo) / 2;   // (rounds towards lo: lo + hi may be negative)
    const bool bit = __fadd_rn(__fmul_rn(alpha, (float)mid), __fadd_rn(shift, 0.f)) >= 0.f;   // (a shift of -0 is +0: no sum is -0)
    if (bit == (alpha < 0.f)) lo = mid + 1;
    else hi = mid;
  }
  return (float)lo;
}

// Operand of the weights: wt[channel tile][channel block][step][chunk][128][16 B]; a chunk is 16 bytes along the
// input channels (8 fp16 or 32 e2m1 values), cb_chunks chunks per block.  With p = 2^kp_log, row r of a tile is channel
// r % p of pixel r / p or, with single pixels, of copy r / p.  Channels that do not exist, and columns outside a pixel's window, are zeros, so whatever the
// activation operand holds there adds 0.
template <int MODE>
__global__ void g_expand_weights_kernel(const uint32_t* __restrict__ wplanes, uint8_t* __restrict__ wt, int C, int K,
                                        int Cw, long long total, int cb_chunks, int n_cb, int steps, int paired, int lg,
                                        int kp_log, int win_step, int ksize, const GTaps taps, const float* __restrict__ alpha,
                                        const float* __restrict__ shift, float* __restrict__ threshold, int pair) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= total) return;
  if (threshold && i < K) threshold[i] = g_sign_threshold(alpha[i], shift[i], ksize * ksize * C);   // (there are more chunks than channels)
  const int row = (int)(i & (G_ROWS - 1));
  long long r = i / G_ROWS;
  const int chunks = paired ? 2 : cb_chunks;
  const int c = (int)(r % chunks);
  r /= chunks;
  const int t = (int)(r % steps);
  r /= steps;
  const int cb = (int)(r % n_cb), tile = (int)(r / n_cb);
  const int g = lg ? row >> kp_log : 0;
  int co = tile * G_ROWS + (row & ((1 << kp_log) - 1));
  const int which = paired ? c : 0;
  const int ky = taps.row[t][which];
  int kx = (int)taps.col[t][which] - win_step * g;
  uint32_t value = 0x3c00u;   // fp16 1.0
  if (MODE == M_F16 && pair) {   // (see g_pairs)
    const GPairRow at = g_pair_row(row, kx);
    co = at.channel;
    kx = at.column;
    if (at.halves == 1) value = 0x3800u;   // 0.5
  }
  constexpr int cpc = MODE == M_F16 ? 8 : 32;
  uint4 v = make_uint4(0, 0, 0, 0);
  if (co < K && ky < ksize && kx >= 0 && kx < ksize) {
    const int ch0 = paired ? 0 : (cb * cb_chunks + c) * cpc;
    const int wd = ch0 >> 5, sh = ch0 & 31;
    const uint32_t bits = wd < Cw ? wplanes[((size_t)(ky * ksize + kx) * Cw + wd) * K + co] >> sh : 0u;
    uint32_t w[4] = {0, 0, 0, 0};
    if (MODE == M_F16) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (ch0 + e < C) w[e >> 1] |= (((bits >> e) & 1u) ? value : value | 0x8000u) << (16 * (e & 1));  // + / -
    } else {
#pragma unroll
      for (int e = 0; e < 32; ++e)
        if (ch0 + e < C) w[e & 3] |= (((bits >> e) & 1u) ? 0x2u : 0xau) << (4 * (e >> 2));         // e2m1 +1.0 / -1.0
    }
    v = make_uint4(w[0], w[1], w[2], w[3]);
  }
  reinterpret_cast<uint4*>(wt)[i] = v;
}

}  // namespace

cudaError_t tcg_create(const LayerDev* const* layers, const Geom* geoms, int count, int act_type, int kind, cudaStream_t s,
                       GroupDev** out, int* launched) {
  *out = nullptr;
  if (count < 1 || count > SNN_GROUP_MAX) return cudaErrorInvalidConfiguration;
  const LayerDev* Ls[SNN_GROUP_MAX];   // in the order in which the CTAs walk through them
  Geom gs[SNN_GROUP_MAX];
  int order[SNN_GROUP_MAX];
  for (int i = 0; i < count; ++i) { Ls[i] = layers[i]; gs[i] = geoms[i]; order[i] = i; }
  if (kind != TCG_WORDS && act_type != SNN_ACT_BIN) return cudaErrorInvalidConfiguration;
  const int chain = kind == TCG_CHAIN;
  const int mode = g_mode_for(act_type);
  for (int i = 0; i < count; ++i)
    if (!g_path_takes(gs[i], mode)) return cudaErrorInvalidConfiguration;
  const int sms = sm_count();
  const bool tma = mode == M_F16 && g_map_encoder() != nullptr;
  // Tile sizes.  A chain's members run one after the other as far as their inputs go, so each takes the size that makes
  // its own tiles end first; the members of a group share the machine, and one size limit for all of them is chosen by
  // the time of the busiest CTA.
  std::vector<GPlan> plan(count);
  for (int i = 0; i < count && chain; ++i)
    if (!g_plan_by_end(gs[i], mode, kind, sms, &plan[i])) return cudaErrorInvalidConfiguration;
  if (!chain && !g_plan_independent(gs, count, mode, kind, tma, sms, plan.data())) return cudaErrorInvalidConfiguration;
  if (!chain) {
    g_order(plan.data(), count, g_order_kind(plan.data(), count, kind), order);
    const std::vector<GPlan> given(plan);
    for (int i = 0; i < count; ++i) { plan[i] = given[order[i]]; Ls[i] = layers[order[i]]; gs[i] = geoms[order[i]]; }
  }
  for (int i = 0; i < count; ++i) g_finish_plan(gs[i], &plan[i]);
  GParams ring{};
  size_t smem = 0;
  if (!g_ring(plan.data(), count, mode, &ring, &smem)) return cudaErrorInvalidConfiguration;
  size_t w_off[SNN_GROUP_MAX], w_total = 0;
  size_t threshold_off[SNN_GROUP_MAX], threshold_words = 0;
  long long tiles = 0, most = 0;
  for (int i = 0; i < count; ++i) {
    threshold_off[i] = threshold_words;
    if (kind != TCG_WORDS) threshold_words += (size_t)gs[i].K;
    w_off[i] = w_total;
    w_total += (plan[i].w_bytes + 255) & ~(size_t)255;
    tiles += plan[i].L.total_tiles;
    most = std::max(most, (long long)plan[i].L.total_tiles);
  }
  int grid = tiles < sms ? (int)tiles : sms;
  // A chain's CTAs wait for one another, so all of them must be resident together (a cooperative launch
  // checks that); members with fewer tiles than CTAs simply leave some CTAs without work in that member.
  if (chain && grid > most) grid = (int)most;
  std::vector<uint2> deps;
  std::vector<size_t> deps_off(count, 0), done_off(count, 0);
  size_t done_words = 0, chain_bytes = 0;
  size_t chain_off[SNN_GROUP_MAX] = {};
  size_t words = 0;   // most words between two members
  for (int i = 0; i + 1 < count && chain; ++i) words = std::max(words, (size_t)gs[i].N * gs[i].Ho * gs[i].Wo * ((gs[i].K + 31) / 32));
  const bool tagged = chain && g_tagged(words);
  if (chain) {
    for (int i = 0; i < count; ++i) {
      if (i > 0 && (gs[i].C != gs[i - 1].K || gs[i].H != gs[i - 1].Ho || gs[i].W != gs[i - 1].Wo || gs[i].N != gs[0].N))
        return cudaErrorInvalidConfiguration;
      const GLayer& L = plan[i].L;
      const int mgroups = L.total_tiles / L.n_ct;
      done_off[i] = done_words;
      if (!tagged) done_words += (size_t)mgroups;
      if (i + 1 < count) {
        chain_off[i] = chain_bytes;
        chain_bytes += ((size_t)gs[i].N * gs[i].Ho * gs[i].Wo * ((gs[i].K + 31) / 32) * (tagged ? 8 : 4) + 255) & ~(size_t)255;
      }
      if (i == 0 || tagged) continue;
      // which position tiles of the predecessor hold the input pixels of each of this member's position tiles
      const GLayer& P = plan[i - 1].L;
      deps_off[i] = deps.size();
      for (int mg = 0; mg < mgroups; ++mg) {
        const long long Q0 = (long long)mg * L.Np;
        long long lo = -1, hi = -1;
        for (int r = 0; r < L.Rr; ++r) {
          const long long q = Q0 + r;
          if (q >= (long long)L.Qtot) break;
          const long long rg = q / L.Wg, n = rg / L.Hq;
          for (int pl = 0; pl < L.n_planes; ++pl) {
            const int px = g_pixel_of(L, (uint32_t)n, (int)(rg - n * L.Hq), (int)(q - rg * L.Wg), pl);
            if (px < 0) continue;
            if (lo < 0 || px < lo) lo = px;
            if (px > hi) hi = px;
          }
        }
        uint2 d = make_uint2(1u, 0u);
        if (lo >= 0) {
          // output pixel of the predecessor -> its position -> its position tile
          auto group_of = [&](long long px) {
            const long long n = px / ((long long)P.Ho * P.Wo);
            const long long rem = px - n * (long long)P.Ho * P.Wo;
            const long long y = rem / P.Wo, x = rem - y * P.Wo;
            return (uint32_t)(((n * P.Hq + y) * P.Wg + (x >> P.lg)) / P.Np);
          };
          d = make_uint2(group_of(lo), group_of(hi));
        }
        deps.push_back(d);
      }
    }
  }
  std::vector<uint32_t> ranks((size_t)count * grid);
  g_assign(plan, grid, &ranks);
  GroupDev* Gd = new GroupDev();
  Gd->count = count;
  Gd->act_type = act_type;
  Gd->mode = mode;
  Gd->grid = grid;
  Gd->chain = chain;
  std::copy(order, order + count, Gd->order);
  Gd->kind = kind;
  Gd->stream = mode == M_FP4 && g_streams(plan.data(), count, kind);
  // One allocation and one copy for everything the group owns: [weight operands][descriptions][ranks][dependencies]
  // [counters][count of launches][thresholds of the signs][packed signs between the members]; the three from the descriptions on come from the host.
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const size_t rank_at = up(sizeof(GLayer) * (size_t)count), deps_at = rank_at + up(ranks.size() * sizeof(uint32_t));
  const size_t blob_bytes = deps_at + up(deps.size() * sizeof(uint2)), blob_at = up(w_total), done_at = blob_at + blob_bytes;
  const size_t launches_at = done_at + up(done_words * sizeof(uint32_t));
  const size_t threshold_at = launches_at + (tagged ? up(sizeof(unsigned long long)) : 0);
  const size_t chain_at = threshold_at + up(threshold_words * sizeof(float));
  cudaError_t e = cudaMalloc(&Gd->mem, chain_at + chain_bytes);
  if (e == cudaSuccess) {
    Gd->layers_dev = reinterpret_cast<GLayer*>(Gd->mem + blob_at);
    Gd->ranks = reinterpret_cast<uint32_t*>(Gd->mem + blob_at + rank_at);
    Gd->done = reinterpret_cast<uint32_t*>(Gd->mem + done_at);
    Gd->chain_buf = Gd->mem + chain_at;
  }
  Gd->done_words = done_words;
  Gd->tagged = tagged;
  // no launch has written a word yet: tags start at 1
  if (tagged && e == cudaSuccess) e = cudaMemsetAsync(Gd->mem + launches_at, 0, chain_at + chain_bytes - launches_at, s);   // (thresholds are written later)
  for (int i = 0; i < count; ++i) Gd->chain_off[i] = chain_off[i];
  const uint2* const deps_dev = reinterpret_cast<const uint2*>(Gd->mem + blob_at + deps_at);
  std::vector<uint8_t> blob(blob_bytes);
  for (int i = 0; i < count && e == cudaSuccess; ++i) {
    GLayer& L = plan[i].L;
    L.wt = Gd->mem + w_off[i];
    Gd->map[i] = {L.tma != 0, L.C, L.W, L.H, L.N, L.rs, L.Wg};
    L.alpha = Ls[i]->alpha;
    float* const thresholds = kind == TCG_WORDS ? nullptr : reinterpret_cast<float*>(Gd->mem + threshold_at) + threshold_off[i];
    L.threshold = thresholds;
    if (chain && !tagged) {
      L.done = Gd->done + done_off[i];
      if (i > 0) {
        L.deps = deps_dev + deps_off[i];
        L.prev_done = Gd->done + done_off[i - 1];
        L.prev_target = (uint32_t)g_writing_warps(plan[i - 1].L);
      }
    }
    const long long total = (long long)plan[i].w_bytes / 16;
    const unsigned blocks = (unsigned)((total + 255) / 256);
    const int win_step = gs[i].stride, ks = gs[i].ksize;
    if (mode == M_F16)
      g_expand_weights_kernel<M_F16><<<blocks, 256, 0, s>>>(Ls[i]->wplanes, Gd->mem + w_off[i], gs[i].C, gs[i].K, gs[i].Cw,
                                                            total, L.cb_chunks, L.n_cb, L.steps, plan[i].paired, L.lg, L.kp_log,
                                                            win_step, ks, plan[i].taps, Ls[i]->alpha, Ls[i]->shift, thresholds, L.pair);
    else
      g_expand_weights_kernel<M_FP4><<<blocks, 256, 0, s>>>(Ls[i]->wplanes, Gd->mem + w_off[i], gs[i].C, gs[i].K, gs[i].Cw,
                                                            total, L.cb_chunks, L.n_cb, L.steps, plan[i].paired, L.lg, L.kp_log,
                                                            win_step, ks, plan[i].taps, Ls[i]->alpha, Ls[i]->shift, thresholds, L.pair);
    e = cudaGetLastError();
    if (e == cudaSuccess) *launched += 1;
  }
  for (int i = 0; i < count; ++i) memcpy(blob.data() + sizeof(GLayer) * (size_t)i, &plan[i].L, sizeof(GLayer));
  memcpy(blob.data() + rank_at, ranks.data(), ranks.size() * sizeof(uint32_t));
  if (!deps.empty()) memcpy(blob.data() + deps_at, deps.data(), deps.size() * sizeof(uint2));
  if (e == cudaSuccess) e = cudaMemcpyAsync(Gd->mem + blob_at, blob.data(), blob_bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host arrays live on this stack
  if (e != cudaSuccess) {
    tcg_destroy(Gd);
    return e;
  }
  Gd->p = ring;
  Gd->p.layers = Gd->layers_dev;
  Gd->p.ranks = Gd->ranks;
  if (tagged) Gd->p.launches = g_launches(reinterpret_cast<unsigned long long*>(Gd->mem + launches_at), (uint32_t)grid);
  Gd->p.one = plan[0].L;
  Gd->smem = smem;
  *out = Gd;
  return cudaSuccess;
}

// ------------------------------------------------------------------ launches from the stored form of a layer
namespace {

struct StaticState {
  GPlan plan;
  GParams ring;
  size_t smem;
  int grid;
};
static_assert(sizeof(StaticState) <= sizeof(TcgStatic::opaque), "TcgStatic holds the plan of a launch");

// Which step and chunk of the weight operand holds kernel row ky and window column s: step * 2 + chunk, 255: none.
struct GStepOf {
  uint8_t at[3][17];
};

// The weight operand straight from the stored form (Sec. 4.4: index stream, codebook).  A warp takes 8 rows of the operand, one
// after the other but with all their loads out together; a lane is an input channel of a 32-channel word.  The indices of a
// row's word are consecutive bits of the stream, nine votes of the codes' bits are its nine taps, and lane t writes tap t.
// Bound by latency: two loads, a look-up, nine votes and the launch around them.
// With one thread per row and word, 64 byte loads and 33 KB of straight-line code a thread, 14 calls took 4 % longer waited for
// (193->168 channels of 9x26: 36.8 us, now 33.8).  The stored form comes as a parameter where it fits one, read through its generic
// address: 8 images of a 128-channel 28x28 layer 9.8 us a call back to back, copied to the device before the launch 14.4, by four
// decode kernels and the popcount kernel 46.
constexpr int G_SW_ROWS = 8, G_SW_WARPS = 4;
template <int BYTES>
struct alignas(16) GStored {
  uint8_t b[BYTES];   // [codebook][scales][index stream]
};
template <int BYTES>   // of the stored form that come as a parameter; 16: it is in memory
__global__ void __launch_bounds__(32 * G_SW_WARPS) g_static_weights_kernel(const uint8_t* stream, int n_bytes, const uint16_t* codebook, uint8_t* __restrict__ wt,
                                                                           const __grid_constant__ GLayer L, int tau, int paired,
                                                                           const __grid_constant__ GStepOf step_of, float* alpha,
                                                                           const __grid_constant__ GStored<BYTES> stored) {
  grid_dep_launch();   // the layer's launch may set itself up beside this one; its weight producer waits for this one to end
  if (BYTES > 16) {
    // (read through its generic address: as a parameter, addresses that differ by lane are served one after the other, 62 us a call)
    const uint8_t* p;
    asm volatile("mov.b64 %0, %1;" : "=l"(p) : "l"(stored.b));
    codebook = reinterpret_cast<const uint16_t*>(p);
    stream = p + 1024 + (size_t)L.K * 4;
    if ((blockIdx.x | blockIdx.y | blockIdx.z) == 0) {
      grid_dep_wait();   // the call before may still read them
      for (int i = threadIdx.x; i < L.K; i += 32 * G_SW_WARPS) alpha[i] = reinterpret_cast<const float*>(p + 1024)[i];
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wd = blockIdx.x, ct = blockIdx.y;                       // 32-channel word, channel tile
  const int row0 = (blockIdx.z * G_SW_WARPS + warp) * G_SW_ROWS;    // (all of the warp's rows are of one pixel of a group)
  const int g = L.lg ? row0 >> L.kp_log : 0, co0 = ct * G_ROWS + (row0 & ((1 << L.kp_log) - 1));
  __shared__ uint16_t codes[512];
  // all loads first: one round trip to memory instead of one per row
  const int n_ch = L.C - 32 * wd < 32 ? L.C - 32 * wd : 32;   // channels of this word
  uint32_t index[G_SW_ROWS];
#pragma unroll
  for (int i = 0; i < G_SW_ROWS; ++i) {
    index[i] = 0;
    if (co0 + i < L.K && lane < n_ch) {
      const int bit = ((co0 + i) * L.C + 32 * wd + lane) * tau;   // (at most 512 x 512 indices)
      const int at = bit >> 3;   // an index spans at most two bytes (9 bits from any bit of a byte: 16 bits)
      uint32_t v = stream[at];
      if (at + 1 < n_bytes) v |= (uint32_t)stream[at + 1] << 8;
      index[i] = (v >> (bit & 7)) & ((1u << tau) - 1u);
    }
  }
  for (int i = threadIdx.x; i < (1 << tau); i += 32 * G_SW_WARPS) codes[i] = codebook[i];
  __syncthreads();
  const int chunks = paired ? 2 : L.cb_chunks, cb = paired ? 0 : wd / L.cb_chunks, c0 = paired ? 0 : wd - cb * L.cb_chunks;
  uint4* const base = reinterpret_cast<uint4*>(wt) + (size_t)(ct * L.n_cb + cb) * L.steps * chunks * G_ROWS + row0;
  grid_dep_wait();   // the call before may still read its operand
  if (L.G > 1 || paired) {   // columns outside the pixel's window, and a last step's missing tap
    const int kinds = paired ? 2 : 1;
#pragma unroll 1
    for (int i = lane; i < L.steps * kinds * G_SW_ROWS; i += 32) {
      const int place = i / G_SW_ROWS, t = paired ? place >> 1 : place, c = paired ? place & 1 : 0;
      base[(size_t)(t * chunks + c0 + c) * G_ROWS + (i & (G_SW_ROWS - 1))] = make_uint4(0, 0, 0, 0);
    }
    __syncwarp();   // before the taps are written over some of them
  }
  const int tap = lane < 9 ? lane : 0, at = step_of.at[tap / 3][tap % 3 + L.rs * g];
  uint4* const dst = base + (size_t)((at >> 1) * chunks + c0 + (at & 1)) * G_ROWS;
  const uint32_t channels = n_ch > 0 ? 0xffffffffu >> (32 - n_ch) : 0u;   // (a block's last words may hold none)
#pragma unroll 2
  for (int i = 0; i < G_SW_ROWS; ++i) {
    uint32_t mine = index[0];
#pragma unroll
    for (int j = 1; j < G_SW_ROWS; ++j) mine = i == j ? index[j] : mine;
    const uint32_t code = codes[mine];
    uint32_t plane = 0;   // bit b: this lane's tap of channel 32*wd + b is +1
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const uint32_t v = __ballot_sync(0xffffffffu, (code >> (8 - t)) & 1u);
      plane = lane == t ? v : plane;
    }
    // nibbles in the expanders' order: channel 4n + k of the word in nibble n of word k; channels that do not exist are 0
    const uint32_t exists = co0 + i < L.K ? channels : 0u;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = ((~(plane << (3 - k)) & 0x88888888u) | 0x22222222u) & (((exists >> k) & 0x11111111u) * 15u);
    if (lane < 9) dst[i] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

}  // namespace

bool tcg_static_plan(const Geom& g, TcgStatic* out) {
  if (g.ksize != 3 || !g_path_takes(g, M_FP4)) return false;
  StaticState st;
  const int sms = sm_count();
  if (!g_plan_independent(&g, 1, M_FP4, TCG_WORDS, false, sms, &st.plan)) return false;
  g_finish_plan(g, &st.plan);
  st.ring = GParams{};
  if (!g_ring(&st.plan, 1, M_FP4, &st.ring, &st.smem)) return false;
  st.grid = st.plan.L.total_tiles < sms ? st.plan.L.total_tiles : sms;
  out->bytes = st.plan.w_bytes;
  memcpy(out->opaque, &st, sizeof(st));
  return true;
}

cudaError_t tcg_static_forward(const TcgStatic& plan, const Geom& g, const uint8_t* stream_dev, const uint16_t* codebook_dev,
                               const float* alpha_dev, uint8_t* mem, const Launch& l, int* status_dev, int* launched) {
  StaticState st;
  memcpy(&st, plan.opaque, sizeof(st));
  GLayer& L = st.plan.L;
  L.wt = mem;
  L.alpha = alpha_dev;
  GStepOf step_of;
  memset(&step_of, 255, sizeof(step_of));
  for (int t = 0; t < L.steps; ++t)
    for (int c = 0; c < (st.plan.paired ? 2 : 1); ++c)
      if (st.plan.taps.row[t][c] < 3) step_of.at[st.plan.taps.row[t][c]][st.plan.taps.col[t][c]] = (uint8_t)(2 * t + c);
  const int n_bytes = (int)(((long long)g.K * g.C * g.tau + 7) / 8);
  const dim3 blocks((unsigned)(st.plan.paired ? 1 : L.n_cb * L.cb_chunks), (unsigned)L.n_ct, G_ROWS / (G_SW_ROWS * G_SW_WARPS));
  cudaError_t e;
  if (!plan.stored.codebook) {
    g_static_weights_kernel<16><<<blocks, 32 * G_SW_WARPS, 0, l.stream>>>(stream_dev, n_bytes, codebook_dev, mem, L, g.tau, st.plan.paired, step_of, nullptr,
                                                                          GStored<16>{});
    e = cudaGetLastError();
  } else {
    // Parameters are copied whole: three sizes.  A programmatic dependent of the call before: it reads the stored form beside that one's
    // last tiles, and waits for its end before it writes.
    const size_t bytes = tcg_stored_bytes(g);
    GStored<(int)kTcgStoredMax> stored;
    memcpy(stored.b, plan.stored.codebook, sizeof(uint16_t) << g.tau);
    memcpy(stored.b + 1024, plan.stored.alpha, (size_t)g.K * 4);
    memcpy(stored.b + 1024 + (size_t)g.K * 4, plan.stored.stream, (size_t)n_bytes);
    float* alpha = const_cast<float*>(alpha_dev);
    int n = n_bytes, tau = g.tau, paired = st.plan.paired;
    const uint8_t* none = nullptr;
    const uint16_t* no_codes = nullptr;
    void* args[] = {&none, &n, &no_codes, &mem, &L, &tau, &paired, &step_of, &alpha, &stored};
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t wcfg{};
    wcfg.stream = l.stream;
    wcfg.attrs = pdl;
    wcfg.numAttrs = 1;
    wcfg.gridDim = blocks;
    wcfg.blockDim = dim3(32 * G_SW_WARPS);
    const void* const kernel = bytes <= 3072 ? (const void*)g_static_weights_kernel<3072> : bytes <= 12288 ? (const void*)g_static_weights_kernel<12288>
                                                                                                         : (const void*)g_static_weights_kernel<(int)kTcgStoredMax>;
    e = cudaLaunchKernelExC(&wcfg, kernel, args);
  }
  if (e != cudaSuccess) return e;
  *launched += 1;
  GParams p = st.ring;
  p.one = L;
  p.act[0] = l.act;
  p.out[0] = l.out;
  p.out_type[0] = (uint8_t)l.out_i32;
  p.status = status_dev;
  // A programmatic dependent of the kernel above: the weight producer waits for that one, and the expanders and the epilogue do
  // as after any other.
  p.after_weights = plan.stored.codebook ? 2 : 1;
  static unsigned long long done = 0;
  e = allow_max_smem(tcg_conv_kernel<M_FP4, OUT_WORDS>, &done);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.stream = l.stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)st.grid);
  cfg.blockDim = dim3(G_THREADS);
  cfg.dynamicSmemBytes = st.smem;
  e = cudaLaunchKernelEx(&cfg, tcg_conv_kernel<M_FP4, OUT_WORDS>, p, GMaps<M_FP4>{});
  if (e == cudaSuccess) *launched += 1;
  return e;
}

void tcg_destroy(GroupDev* G) {
  if (!G) return;
  cudaFree(G->mem);
  delete G;
}

bool tcg_supported(const Geom& g, int act_type) { return g_path_takes(g, g_mode_for(act_type)); }

cudaError_t tcg_forward(GroupDev* G, const void* const* act, void* const* out, int out_type, cudaStream_t s,
                        int* status_dev, int* launched) {
  GParams p = G->p;
  cudaLaunchAttribute attr[1];
  if (G->chain) {
    // act[0] is the first member's input and out[0] the last member's output; the packed signs in between
    // stay in the group's own buffers
    for (int i = 0; i < G->count; ++i) {
      p.act[i] = i == 0 ? act[0] : (const void*)(G->chain_buf + G->chain_off[i - 1]);
      p.out[i] = i + 1 == G->count ? out[0] : (void*)(G->chain_buf + G->chain_off[i]);
      p.out_type[i] = (uint8_t)(i + 1 == G->count ? out_type : G->tagged ? 3 : 2);
    }
    cudaError_t e0 = G->tagged ? cudaSuccess : cudaMemsetAsync(G->done, 0, G->done_words * sizeof(uint32_t), s);
    if (e0 != cudaSuccess) return e0;
    attr[0].id = cudaLaunchAttributeCooperative;   // the CTAs wait for one another: all must be resident
    attr[0].val.cooperative = 1;
  } else {
    for (int i = 0; i < G->count; ++i) {
      p.act[i] = act[G->order[i]];
      p.out[i] = out[G->order[i]];
      p.out_type[i] = (uint8_t)out_type;
    }
    // Launched as a programmatic dependent of its predecessor in the stream: set-up overlaps that
    // kernel's tail; the warps that read activations or write outputs wait on the device for it.
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
  }
  p.status = status_dev;
  cudaLaunchConfig_t cfg{};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)G->grid);
  cfg.blockDim = dim3(G_THREADS);
  cfg.dynamicSmemBytes = G->smem;
  cudaError_t e;
  GMaps<M_FP4> none{};
  const int outk = G->tagged ? OUT_TAGGED : G->chain ? OUT_CHAIN : (out_type == 2 ? OUT_SIGNS : G->stream ? OUT_STREAM : OUT_WORDS);
  if (!G->chain && (outk == OUT_SIGNS) != (G->kind == TCG_SIGNS)) return cudaErrorInvalidValue;  // planned for the other kind
#define G_LAUNCH(M, O, MAPS)                                                    \
  do {                                                                          \
    static unsigned long long done = 0;                                         \
    e = allow_max_smem(tcg_conv_kernel<M, O>, &done);                           \
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, tcg_conv_kernel<M, O>, p, MAPS); \
  } while (0)
  if (G->mode == M_F16) {
    GMaps<M_F16> maps;
    for (int i = 0; i < G->count; ++i) {
      const GroupDev::Map& m = G->map[i];
      if (!m.tma) continue;
      // [N][H][W][C] halves; a box is 64 channels of one row of positions
      const cuuint64_t dim[4] = {(cuuint64_t)m.C, (cuuint64_t)m.W, (cuuint64_t)m.H, (cuuint64_t)m.N};
      const cuuint64_t pitch[3] = {(cuuint64_t)m.C * 2, (cuuint64_t)m.W * m.C * 2, (cuuint64_t)m.H * m.W * m.C * 2};
      const cuuint32_t box[4] = {64, (cuuint32_t)((m.box - 1) * m.stride + 1), 1, 1}, step[4] = {1, (cuuint32_t)m.stride, 1, 1};
      if (g_map_encoder()(&maps.m[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(act[G->order[i]]), dim, pitch, box, step,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    }
    if (outk == OUT_WORDS) G_LAUNCH(M_F16, OUT_WORDS, maps);
    else return cudaErrorInvalidValue;   // packed signs and chains need binary activations
  } else if (outk == OUT_WORDS) G_LAUNCH(M_FP4, OUT_WORDS, none);
  else if (outk == OUT_STREAM) G_LAUNCH(M_FP4, OUT_STREAM, none);
  else if (outk == OUT_SIGNS) G_LAUNCH(M_FP4, OUT_SIGNS, none);
  else if (outk == OUT_CHAIN) G_LAUNCH(M_FP4, OUT_CHAIN, none);
  else G_LAUNCH(M_FP4, OUT_TAGGED, none);
#undef G_LAUNCH
  if (e != cudaSuccess) return e;
  *launched += 1;
#ifdef SNN_TRACE
  {
    static long long h[256 * 16];
    cudaDeviceSynchronize();
    cudaMemcpyFromSymbol(h, g_trace, sizeof(h));
    static const char* role[4] = {"producer", "mma", "epilogue", "expander"};
    for (int r = 0; r < 4; ++r) {
      double a[4] = {0, 0, 0, 0}, mx = 0;
      for (int b = 0; b < G->grid; ++b) {
        for (int k = 0; k < 4; ++k) a[k] += (double)h[b * 16 + r * 4 + k] / G->grid;
        if ((double)h[b * 16 + r * 4] > mx) mx = (double)h[b * 16 + r * 4];
      }
      fprintf(stderr, "[trace] %-9s total %8.0f (max %8.0f)  waits %8.0f %8.0f %8.0f cycles\n", role[r], a[0], mx, a[1], a[2],
              a[3]);
    }
  }
#endif
  return cudaGetLastError();
}

}  // namespace snn
