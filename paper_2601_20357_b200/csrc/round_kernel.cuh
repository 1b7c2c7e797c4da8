// Persistent kernel for one whole drafting round (Algorithm 1 steps 4-8): gamma batched
// shared-weight decoder steps, each followed by softmax + weighted-average ensemble + draw, in ONE
// cooperative launch with one CTA per SM.
//
// Why one kernel: with m <= 4 drafting inputs a decoder step moves ~125-630 MB of weights through
// dozens of strictly dependent phases; as separate launches every phase pays a launch plus a cold
// DRAM round trip.  Here
//   * the weights never stop streaming: every CTA owns a fixed share of the weight tiles of every
//     phase (its unit list is made at set-up), and a ring of shared-memory slots is
//     kept full by bulk asynchronous copies (cp.async.bulk + mbarrier) several phases ahead of the
//     arithmetic, so HBM stays busy across the phase boundaries;
//   * the weights are read from a private copy laid out for this kernel at set-up: every unit (16 or 8
//     output rows x kchunk input columns, rows padded to a bank-conflict-free shared-memory pitch)
//     is one contiguous block, hence ONE bulk copy;
//   * there is NO grid barrier.  Every activation that crosses CTAs travels as an 8-byte word
//     {value, epoch} written with one 64-bit store; the epoch names the launch, the step and the
//     phase that produced it, so a consumer polls the data itself and starts as soon as ITS inputs
//     have arrived.  5 phases per layer (QKV, attention, O, gate/up, down);
//   * what bounds a phase is the chain from the arrival of its words to the departure of its results, so what can be moved off
//     it is: the PRODUCER of an activation does the work on it (rotation and rounding of q, k, v; the attention's division; the
//     gated product), and its words hold two bf16 values in the order in which a consumer's mma fragment needs them.  The
//     summed index of a tile is dealt to all warps of a group, so a warp polls exactly the words that ARE its B fragments: no
//     staging in shared memory, no block barrier between a word's arrival and the product.  (The residual travels as fp32
//     and is normalised and rounded by its consumers, whose warps meet once to add their sums of squares.)  The partial tiles
//     of the warps meet in shared memory behind one barrier;
//   * a tile always takes its whole input dimension on ONE CTA (long rows as sub-units whose products
//     accumulate in registers), so no projection leaves split-K partial sums behind; every sum has a fixed order: deterministic;
//   * products: mma.sync m16n8k16, bf16 x bf16 -> fp32, 16 weight rows x up to 8 slots.  The contraction is HBM-bound
//     (<= 8 flop per weight byte); the tensor pipe only keeps the ALUs off the critical path;
//   * all cross-CTA data is read with relaxed gpu-scope loads (L2): L1 is not coherent across SMs;
//   * loops are deliberately not unrolled except the few hot ones: every phase runs its code once,
//     so unrolling buys nothing and only inflates the instruction footprint.
//
// Rows: up to 4 rows feed both pending tokens of a fully accepted block in the first step's weight pass
// (2 R <= 8 slots); with 5 - 8 rows the first of the two gets a pass of its own before step 0 (all layers,
// no LM head, only the rows that have two pending tokens are active), so a pass never has more than 8 slots.
//
// Waits are bounded: a flagged word or a copy that does not arrive within the spin limit sets an
// error bit, the CTA drains its copies in flight and returns.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "decide_kernels.cuh"
#include "exact_math.cuh"
#include "forward_kernels.cuh"

namespace tabed {

constexpr int kPT = 384;                 // threads per CTA
constexpr int kPW = kPT / 32;            // warps per CTA
constexpr int kGW = kPW / 2;             // warps of a group
constexpr int kGT = kPT / 2;
constexpr int kPSlots = 8;               // slots (row, position) per step: one mma n-tile
constexpr int kPRing = 16;               // upper bound of ring slots
constexpr int kPRound = 4;               // most units between two barriers of a group
constexpr int kPPos = kGW * 16;          // cache positions per attention chunk: 16 a warp of group 1
constexpr int kPMaxD = 2048;             // d_model bound
constexpr int kTraceRec = 8;             // words per record of the phase timeline
constexpr int kPMaxL = 64;               // layers (the pointers of their gains live in shared memory)
constexpr int kPMaxHeads = 64;           // query heads
constexpr int kMaxUnits = 1024;          // units of one CTA in one decoder step
constexpr int kMaxPhase = 4 * kPMaxL + 1;
constexpr int kPMaxChunks = 1280;        // attention chunks of one CTA
constexpr int kPMaxStages = 3;           // chunks of K and V on their way to a warp
constexpr int kProbeWords = 128;         // words that nobody writes, for the test of the bounded waits (64 masses of two words)
// Partial tiles of a round in shared memory: [unit][slot pair][warp][2][16 rows], 40 floats a warp and 8 idle ones a pair, which
// make the fragments' stores and the sums' loads free of bank conflicts.  Up to 4 slots take two pairs and rounds of 4 units,
// up to 8 slots four pairs and rounds of 2 units; two buffers a group, so that a round needs one barrier; group 1 has one tile
// a round.
constexpr int kPPair = kGW * 40 + 8;
constexpr int kPBuf = 8 * kPPair;
constexpr int kPPartFloats = 3 * kPBuf;

enum { KIND_QKV = 0, KIND_O = 1, KIND_GU = 2, KIND_DN = 3, KIND_LM = 4 };
enum { PERR_BARRIER = 8, PERR_COPY = 16, PERR_KV = 4 };

struct LayerW { const __nv_bfloat16 *wq, *wk, *wv, *wo, *wg, *wu, *wd, *n1, *n2; };

// A phase's weight matrix is cut into tiles of 16 output rows (O and down: 8, their few tiles would leave most CTAs without one);
// a tile is nsub units of kchunk input columns each.  unit u -> tile = u / nsub, sub = u % nsub.
struct PhaseGeom { int rows, n_tiles, nsub, kchunk, n_units; };

struct RoundArgs {
  // drafter
  const LayerW* layers;
  const __nv_bfloat16 *embed, *final_norm;
  const float *rope_cos, *rope_sin;
  int L, d, F, H, Hkv, hd, V, cap, qkv_w;
  float eps, attn_scale;
  PhaseGeom geom[5];
  const unsigned char* packed;          // weights re-laid out unit by unit (k_pack_units)
  unsigned long long pack_off[5];       // byte offset of a kind's units inside a layer block (LM: absolute)
  unsigned long long pack_layer_stride;
  int slot_bytes, n_ring, round_units, kv_stages;     // (a round's units are in the ring together)
  const uint16_t* pstart;               // [CTAs][4 L + 2] first entry of every phase in a CTA's unit list
  const uint32_t* ulist;                // [CTAs][max_units]
  int max_units;
  // round
  int R, B, m, G, greedy;
  const int* kv_len;                    // [R] committed lengths (constant during the round)
  const int* pending;                   // [B][3]
  __nv_bfloat16 *kc, *vc;               // [R][L][Hkv][cap][hd]
  // activations exchanged through L2 as {value, epoch} pairs (one 8-byte store, polled by the consumer)
  uint2 *xa, *x1;                       // [d/16][8][16] residual entering a layer / after its attention block
  uint2* qkv;                           // [8][qkv_w/2] q, k (rotated) and v, two bf16 values a word
  uint2 *att, *mid;                     // [d/16][8][8], [F/16][8][8] attention outputs, gated products: two bf16 values a word
  uint2* part;                          // attention: partial results [8][H][n_part][hd] of four words: output, maximum, sum, -
  int n_part;
  unsigned epoch0;                      // the launch's first epoch; phase p of pass i stamps epoch0 + i * (5 L + 8) + p + 1
  int prepass;                          // more than kPSlots / 2 rows: a fully accepted block's first pending token is fed in a
                                        // pass of its own (all layers, no LM head) before step 0, instead of as R more slots
  // ensemble
  float* logits_own;                    // [G][R][V]
  const float* logits_override;         // or null
  const float* w;                       // [B][m]
  const float* u;                       // [B][G]
  float *qk, *q;                        // [B][G][m][V], [B][G][V]
  uint2* rowmax;                        // [8][CTAs, to an even number] every CTA's maxima of the logit rows
  uint2* rowsum;                        // [8][CTAs][2] every CTA's integer exp sums, low and high word
  uint2 *slice_mass, *mass;             // [B][CTAs][2] mass of a CTA's slice of q, low and high word (greedy: best value, its index); [B][V][2] of every token
  int *tokens, *out_tokens;             // [B][G]
  // diagnostics
  int* err;
  unsigned long long* trace;            // optional [G][trace_stride][kTraceRec] phase timeline
  int trace_stride, trace_cta;          // the CTA that records
};

// ------------------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// global -> shared bulk copy; dst/src 16-byte aligned, bytes a multiple of 16.  No multicast.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
// transposes an 8 x 8 matrix of 16-bit elements held one row per quad (lane (g, t): row g, columns 2t, 2t+1)
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// Flagged words: an aligned 8-byte {value, epoch} pair is written by ONE store and read by one load, so a
// reader sees either the old pair or the new one; a 16-byte load returns two such pairs.
__device__ __forceinline__ void ll_store(uint2* p, uint32_t value, uint32_t epoch) {
  asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(value), "r"(epoch) : "memory");
}
// two neighbouring words (p 16-byte aligned) by one store; each half stays a flagged word of its own
__device__ __forceinline__ void ll_store2(uint2* p, uint32_t v0, uint32_t v1, uint32_t epoch) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %2};" ::"l"(p), "r"(v0), "r"(epoch), "r"(v1) : "memory");
}
__device__ __forceinline__ uint2 ll_load1(const uint2* p) {
  uint2 v;
  asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ll_load2(const uint2* p) {           // p 16-byte aligned: pairs p[0], p[1]
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
// ... from p + OFF bytes if j < n; else v stays as it is
template <int OFF>
__device__ __forceinline__ void ll_load2_if(uint4& v, const uint2* p, int j, int n) {
  asm volatile("{\n .reg .pred p;\n setp.lt.s32 p, %5, %6;\n @p ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4 + %7];\n}\n"
               : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(p), "r"(j), "r"(n), "n"(OFF) : "memory");
}
__device__ __forceinline__ unsigned long long global_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ float4 bf16x4_to_float4(uint2 v) {
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u),
                     __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
}
// ------------------------------------------------------------------------------------------------
// per-CTA state
// ------------------------------------------------------------------------------------------------
struct PSlot { int row, pos, active, tok; };

struct PShared {
  uint64_t full[kPRing];
  const __nv_bfloat16* gain[kPMaxL][2];
  uint2 gains[kPMaxD / 4];              // of the norm at hand
  uint32_t ulist[kMaxUnits];            // this CTA's units of one decoder step, in consumption order
  uint16_t pstart[kMaxPhase + 1];       // first entry of every phase in ulist
  alignas(16) float red[2][kPSlots][8]; // sums of squares of the slots by warp (the last two are zero)
  float am[kGW][kMaxGroup], al[kGW][kMaxGroup];   // attention: maximum and sum by warp and head
  uint32_t lmmax[kPSlots], rmax[kPSlots];
  float mix_w[kPSlots];
  PSlot slot[kPSlots];
  int kv_len[kPSlots], pending[kPSlots][3];
  int lm_src[kPSlots];
  int nkb[5], nsub[5], col[2][kPSlots], any;
  uint32_t chunks[kPMaxChunks];         // attention: this CTA's chunks of the step: slot (3 bits), KV head (6), split (9), splits (9)
  int n_chunk, n_tot;                   // their number, and that of all CTAs
  int pair_base[kPSlots], pair_ns[kPSlots];   // per slot: chunks before its first pair, chunks per pair (0: inactive)
  unsigned char nseg[kPSlots][kPMaxHeads];    // per (slot, head): partial attention results of the step
  int tok[kPSlots];
  unsigned long long row_part[kPSlots], row_sum[kPSlots], req_mass[kPSlots];   // exp sums of all CTAs, of this one; its mass (best) of q
  int pre_units, per_step, total_units; // the stream of units
  int issued[kPRing];                   // copies asked for by ring slot
};

// a unit of the list: kind (3 bits), layer (7), sub-unit of its tile (6), tile (16) - no division where it is used
constexpr int kUnitTiles = 1 << 16;
__host__ __device__ __forceinline__ uint32_t unit_pack(int kind, int layer, int tile, int sub) {
  return (uint32_t)kind | ((uint32_t)layer << 3) | ((uint32_t)sub << 10) | ((uint32_t)tile << 16);
}
__device__ __forceinline__ int unit_sub(uint32_t e) { return (int)((e >> 10) & 63u); }
__device__ __forceinline__ int unit_tile(uint32_t e) { return (int)(e >> 16); }

// A value that is the same in all lanes, told to the compiler: branches on it are uniform (each shuffle or vote behind one that
// might not be gets a second, slow version), and what follows from it lives in uniform registers.
__device__ __forceinline__ int uni(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// The thread's number, anew: what a part of the kernel derives from it (lanes' offsets into everything) is then not kept in
// registers through the other parts, which need them all (spilled registers go to L2: the L1 is all shared memory).
__device__ __forceinline__ int own_tid() {
  int t = threadIdx.x;
  asm volatile("" : "+r"(t));
  return t;
}

// Operand words of 16 columns: [block][slot][8 pairs].  A lane (slot g, t) of a B fragment takes columns 4t .. 4t+3 of the
// block, its words 2t and 2t + 1; the weights' columns are packed in the matching order (k_pack_units).
__device__ __forceinline__ size_t op_word(int block, int slot) { return ((size_t)block * kPSlots + slot) * 8; }

// Issue the bulk copy of unit k of the stream into its ring slot (one thread).
__device__ __forceinline__ void issue_unit(const RoundArgs& A, PShared& S, unsigned char* ring, int k, int slot) {
  if (k >= S.total_units) return;
  const uint32_t e = S.ulist[k < S.pre_units ? k : (k - S.pre_units) % S.per_step];
  const int kind = e & 7, layer = (e >> 3) & 127, u = unit_tile(e) * S.nsub[kind] + unit_sub(e);
  const unsigned bytes = (kind == KIND_O || kind == KIND_DN ? 8u : 16u) * ((unsigned)S.nkb[kind] * 32u + 16u);
  const unsigned char* src = A.packed + A.pack_off[kind] + (size_t)u * bytes +
                             (kind == KIND_LM ? 0ull : (unsigned long long)layer * A.pack_layer_stride);
  mbar_expect_tx(&S.full[slot], bytes);
  bulk_g2s(ring + (size_t)slot * A.slot_bytes, src, bytes, &S.full[slot]);
  *(volatile int*)&S.issued[slot] = S.issued[slot] + 1;
}

template <int ID> __device__ __forceinline__ void bar_sync(int n) { asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(n) : "memory"); }
template <int ID> __device__ __forceinline__ int bar_sync_or(int n, int pred) {
  int r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.or.pred q, %2, %3, p;\n selp.s32 %0, 1, 0, q;\n}\n"
               : "=r"(r) : "r"(pred), "n"(ID), "r"(n) : "memory");
  return r;
}

// Re-lay one weight matrix (or the QKV / gate-up group) of one layer into units.  grid (n_units), block 256.
// Rows: QKV rows are the concatenation wq | wk | wv, a tile of wq or wk holding 8 dims of a head's first half, then their
// partners of the rotation, half a head further; gate/up units hold 8 gate rows then the 8 matching up rows; LM-head rows
// beyond V are zero.  Columns of a block of 16: 0,1,4,5,8,9,12,13 | 2,3,6,7,10,11,14,15 (op_word).
struct PackArgs {
  const __nv_bfloat16 *w0, *w1, *w2;    // source matrices [rows_i][K]
  int rows0, rows1, rows2, K, kind, hd;
  PhaseGeom g;
  unsigned char* dst;                   // first unit of this (layer, kind)
};
__global__ void k_pack_units(const PackArgs P) {
  const int u = blockIdx.x;
  const int tile = u / P.g.nsub, sub = u - tile * P.g.nsub;
  const int pitch = P.g.kchunk * 2 + 16;
  unsigned char* unit = P.dst + (size_t)u * P.g.rows * pitch;
  const int vec_per_row = pitch / 16;                      // 16-byte vectors per padded row
  for (int idx = threadIdx.x; idx < P.g.rows * vec_per_row; idx += blockDim.x) {
    const int r = idx / vec_per_row, c16 = idx - r * vec_per_row;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (c16 * 8 < P.g.kchunk) {
      const __nv_bfloat16* base = nullptr;
      int row;
      if (P.kind == KIND_GU) { row = tile * 8 + (r & 7); base = (r < 8) ? P.w0 : P.w1; if (row >= P.rows0) base = nullptr; }
      else {
        row = tile * P.g.rows + r;
        if (P.kind == KIND_QKV && tile * 16 < P.rows0 + P.rows1) {
          const int in_head = (tile * 16) % P.hd;
          row = tile * 16 - in_head + (in_head >> 1) + (r & 7) + (r < 8 ? 0 : P.hd >> 1);
        }
        if (row < P.rows0) base = P.w0;
        else if (row < P.rows0 + P.rows1) { base = P.w1; row -= P.rows0; }
        else if (row < P.rows0 + P.rows1 + P.rows2) { base = P.w2; row -= P.rows0 + P.rows1; }
      }
      if (base) {
        const uint4* p = reinterpret_cast<const uint4*>(base + (size_t)row * P.K + (size_t)sub * P.g.kchunk + (c16 >> 1) * 16);
        const uint4 a = p[0], b = p[1];
        v = (c16 & 1) ? make_uint4(a.y, a.w, b.y, b.w) : make_uint4(a.x, a.z, b.x, b.z);
      }
    }
    *reinterpret_cast<uint4*>(unit + (size_t)r * pitch + (size_t)c16 * 16) = v;
  }
}

constexpr unsigned kSpinLimit = 1u << 21;

// Bounded wait for filling number `fill` of a ring slot; on a timeout the error bit is set and `dead` raised.  (The copy may
// not have been asked for yet: its slot may still hold a unit of the other group.  Only then does the parity name one filling.)
__device__ __forceinline__ void wait_full(PShared& S, int slot, int fill, int& dead, int* err) {
  unsigned spins = 0;
#pragma unroll 1
  while (*(volatile int*)&S.issued[slot] <= fill || !mbar_try_wait(&S.full[slot], (unsigned)fill & 1u)) {
    if (dead || ++spins > kSpinLimit) { if (!dead) atomicOr(err, PERR_COPY); dead = 1; break; }
    if (spins > 4096) __nanosleep(64);
  }
}

// Bounded polls of flagged words.  On a timeout the error bit is set and `dead` raised: the thread waits no more, and the CTA
// leaves at the end of the step.
__device__ __forceinline__ int ll_timeout(int* err) {      // (inlined: a call would have every wait save its registers)
  atomicOr(err, PERR_BARRIER);
  return 1;
}
__device__ __forceinline__ uint32_t ll_wait1(const uint2* p, uint32_t epoch, int& dead, int* err) {
  uint2 v = ll_load1(p);
  unsigned spins = 0;
#pragma unroll 1
  while (v.y != epoch) {
    if (dead) break;
    if (++spins > kSpinLimit) { dead = ll_timeout(err); break; }
    if (spins > 256) __nanosleep(spins > 4096 ? 64 : 20);
    v = ll_load1(p);
  }
  return v.x;
}
// n groups of PER neighbouring 16-byte pieces (two flagged words each), group j at p + j * STRIDE words, all in flight
// together.  Where something is missing, the lanes ask for their last piece alone until it is there (57 000 threads asking
// for everything would flood L2), then for all of them again.  All 32 lanes call together, with the same n (v[] beyond it
// is zero).  The offsets are immediates: as addresses in registers they were what the kernel spilled for.  The code is short
// on purpose: every phase runs it once, out of the instruction caches.
template <int J, int N, int PER, int STRIDE>
__device__ __forceinline__ void ll_load_all(uint4 (&v)[N], const uint2* p, int n) {
  if constexpr (J < N) {
    ll_load2_if<((J / PER) * STRIDE + 2 * (J % PER)) * 8>(v[J], p, J / PER, n);
    ll_load_all<J + 1, N, PER, STRIDE>(v, p, n);
  }
}
template <int N, int PER, int STRIDE>
__device__ __forceinline__ void ll_poll(const uint2* p, int n, uint32_t epoch, uint4 (&v)[N], int& dead, int* err) {
#pragma unroll
  for (int j = 0; j < N; ++j) { v[j].y = v[j].w = epoch; v[j].x = v[j].z = 0u; }
  unsigned spins = 0;
#pragma unroll 1
  while (true) {
    ll_load_all<0, N, PER, STRIDE>(v, p, n);
    uint32_t miss = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) miss |= (v[j].y ^ epoch) | (v[j].w ^ epoch);
    if (!__any_sync(0xffffffffu, miss != 0 && !dead)) break;
    // (a lane may come in with a wait of its own that ran out: the warp stays together, or the votes below would miss it)
    if (__any_sync(0xffffffffu, dead)) { dead = 1; break; }
    uint4 x;
#pragma unroll 1
    do {
      x = ll_load2(p + (n - 1) * STRIDE);
      if (++spins > kSpinLimit) { dead = ll_timeout(err); break; }
    } while (__any_sync(0xffffffffu, x.y != epoch));
    if (dead) break;
  }
}
// two neighbouring words
__device__ __forceinline__ uint4 ll_wait2(const uint2* p, uint32_t epoch, int& dead, int* err) {
  uint4 v = ll_load2(p);
  unsigned spins = 0;
#pragma unroll 1
  while ((v.y != epoch || v.w != epoch) && !dead) {
    if (++spins > kSpinLimit) { dead = ll_timeout(err); break; }
    if (spins > 4) __nanosleep(spins > 4096 ? 200 : 40);
    v = ll_load2(p);
  }
  return v;
}

// A lane's pieces of K and V of chunk c (of n) in a layer, into its places of a stage: one group of copies, empty where there is
// no such chunk or no cached position for the warp.  (16 bytes each, which go past the L1: it does not see the rows that other
// SMs append.)  A lane without a position of its own asks for the last one (a weight of 0
// does not cancel what an unwritten row may hold).
template <int HD> __host__ __device__ constexpr int kv_pieces() { return HD == 32 ? 6 : HD / 8; }      // of K and V, per lane
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
template <int HD>
__device__ __forceinline__ void kv_request(const RoundArgs& A, PShared& S, unsigned char* stage, int c, int n, int layer, int gw, int lane) {
  constexpr int KP = HD / 32, VP = HD <= 64 ? 1 : HD / 64, kPiece = kGT * 16;
  if (c < n) {
    const uint32_t e = uni(S.chunks[c]);
    const int s = e & 7, gk = (e >> 3) & 63, split = (e >> 9) & 511, gq = lane >> 2, t4 = lane & 3;
    const int lim = min(kPPos, uni(S.slot[s].pos) - (s >= A.R ? 1 : 0) - split * kPPos) - gw * 16;
    const unsigned row = ((unsigned)(uni(S.slot[s].row) * A.L + layer) * A.Hkv + gk) * A.cap + split * kPPos + gw * 16;      // (of all caches' rows: below 2^31)
    if (lim > 0) {
      uint32_t dst = smem_u32(stage) + (gw * 32 + lane) * 16;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const __nv_bfloat16* src = A.kc + (size_t)(row + min(i * 8 + gq, lim - 1)) * HD + t4 * 8;
#pragma unroll
        for (int j = 0; j < KP; ++j, dst += kPiece) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + j * 32) : "memory");
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const __nv_bfloat16* src = A.vc + (size_t)(row + min((i >> 1) * 8 + 2 * t4 + (i & 1), lim - 1)) * HD;
#pragma unroll
        for (int j = 0; j < VP; ++j, dst += kPiece)            // pieces g, g + 8 (head size 32: g & 3, of which the lane uses half)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + ((HD == 32 ? gq & 3 : gq) + 8 * j) * 8) : "memory");
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// the attention's output of one (slot, column), from neighbouring lanes, as an operand word of the O projection
__device__ __forceinline__ void store_att(const RoundArgs& A, int slot, int column, float x, unsigned epoch) {
  const float right = __shfl_down_sync(0xffffffffu, x, 1);
  if ((column & 1) == 0) ll_store(A.att + op_word(column >> 4, slot) + ((column & 15) >> 1), pack_bf16(x, right), epoch);
}

// ---- pieces of the ensemble ------------------------------------------------------------------------
// largest value of the warp, lowest index on ties
__device__ __forceinline__ void best_of_warp(float& bv, int& bi) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
}
// One warp: the first of n flagged masses (two words each) whose running sum exceeds the threshold, which is drawn from their
// total by u (draw) or given; and what is left of it there.  at -1: there is none.  A lane takes a contiguous range.
// (A function of its own, used twice a step: inlined, its registers would cost the phases theirs.)
struct Found { unsigned long long thr; int at, dead; };
__device__ __noinline__ Found find_mass(const uint2* w, int n, bool draw, float u, unsigned epoch, unsigned long long thr, int dead, int* err) {
  const int lane = threadIdx.x & 31, per = (n + 31) >> 5, cnt = max(0, min(per, n - lane * per));
  w += (size_t)lane * per * 2;
  uint4 v[8];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int j = 0; j < 8; ++j) { v[j].x = v[j].z = 0u; v[j].y = v[j].w = epoch; }
    unsigned spins = 0;
#pragma unroll 1
    while (true) {
      uint32_t miss = 0;
      ll_load_all<0, 8, 1, 2>(v, w + 2 * j0, cnt - j0);
#pragma unroll
      for (int j = 0; j < 8; ++j) miss |= (v[j].y ^ epoch) | (v[j].w ^ epoch);
      if (!__any_sync(0xffffffffu, miss != 0 && !dead)) break;
      if (++spins > kSpinLimit) { dead = ll_timeout(err); break; }
    }
  };
  auto mass = [&](int j) { return (unsigned long long)v[j].x | ((unsigned long long)v[j].z << 32); };
  unsigned long long sum = 0;
#pragma unroll 1
  for (int j0 = 0; j0 < per; j0 += 8) {
    fetch(j0);
#pragma unroll
    for (int j = 0; j < 8; ++j) sum += mass(j);
  }
  unsigned long long incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (draw) {
    const unsigned long long total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0ull) return Found{0ull, -1, dead};
    thr = draw_threshold(u, total);
  }
  const unsigned over = __ballot_sync(0xffffffffu, incl > thr);
  if (!over) return Found{0ull, -1, dead};
  const int owner = __ffs(over) - 1;
  unsigned long long run = incl - sum, before = 0;
  int at = -1;
#pragma unroll 1
  for (int j0 = 0; j0 < per; j0 += 8) {
    if (per > 8) fetch(j0);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const unsigned long long next = run + mass(j);
      if (at < 0 && next > thr) { at = lane * per + j0 + j; before = run; }
      run = next;
    }
  }
  return Found{thr - __shfl_sync(0xffffffffu, before, owner), __shfl_sync(0xffffffffu, at, owner), dead};
}

// ------------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------------
// HD: head size.  NF: blocks of 16 input columns that a warp holds of a row (a group's warps share the row's blocks); the code
// is that long in every phase that normalises, so a row takes the shortest that holds it (NF 6 against 8, us per pass of three
// rounds, 1 / 3 / 6 rows: 256 columns 723 / 781 / 900 against 748 / 796 / 918, 576 columns 819 / 897 / 1139 against 839 / 910 / 1160).
//
// What bounds a phase is the chain from the arrival of its words to the departure of its results, and on that chain the number
// of instructions that the CTA's warps issue (16 warps that all run 500 instructions take 2000 cycles of the four
// schedulers, twice that out of the instruction cache's next level).  Hence two groups of six warps that take turns: group 0
// has the phases that normalise (QKV, gate/up, LM head), group 1 the others (attention, O, down).  While a group works, the
// other one has already set up its next phase and polls for its words.  Twelve warps have 168 registers a thread.
// With those nothing is spilled at head size 64 up to NF 8 and at 32 up to NF 12; elsewhere bytes of spill stores a thread: head
// size 64 28 / 412 at NF 12 / 24, 32 292 at NF 24, 128 128 - 164 up to NF 12 and 540 at 24 (with TRACE more, up to 1284: a
// timeline's phases are that much longer than an untraced round's).
template <int HD, int NF, bool TRACE>
__global__ void __launch_bounds__(kPT, 1) k_draft_round(const RoundArgs A) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  __shared__ PShared S;
  constexpr unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = uni(tid >> 5);
  const int group = warp / kGW, gw = warp - group * kGW;   // group, warp within it
  const int cta = blockIdx.x, NC = gridDim.x;
  unsigned char* ring = dyn_smem;
  float* part = reinterpret_cast<float*>(dyn_smem + (size_t)A.n_ring * A.slot_bytes);   // partial tiles of a round
  float* s_o = part + kPPartFloats;                      // attention: [kGW][grp * HD]
  const int kvd = A.Hkv * HD, grp = A.H / A.Hkv;
  // K and V on their way: kv_stages times [piece][warp of group 1][lane][16 bytes]
  constexpr int kv_piece = kGT * 16, kv_stage_bytes = kv_pieces<HD>() * kv_piece;
  unsigned char* kv_area = reinterpret_cast<unsigned char*>(s_o + kGW * grp * HD);
  constexpr int half = HD >> 1;
  const int R = A.R, B = A.B, m = A.m, G = A.G, V = A.V, d = A.d;
  const int n_phase = 4 * A.L + 1;
  int dead = 0;                                          // a wait of this thread (or one it has met at a barrier) has run out

  // ---- set-up -----------------------------------------------------------------------------------
  if (tid == 0) {
#pragma unroll 1
    for (int s = 0; s < A.n_ring; ++s) { mbar_init(&S.full[s], 1); S.issued[s] = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < R) { S.mix_w[tid] = A.w[tid]; S.kv_len[tid] = A.kv_len[tid]; }
  if (tid < 3 * B) S.pending[tid / 3][tid % 3] = A.pending[tid];
  if (tid < 2 * kPSlots) S.red[tid >> 3][tid & 7][6] = S.red[tid >> 3][tid & 7][7] = 0.0f;
  if (tid < 5) { S.nkb[tid] = A.geom[tid].kchunk >> 4; S.nsub[tid] = A.geom[tid].nsub; }
#pragma unroll 1
  for (int i = tid; i < A.L; i += kPT) { S.gain[i][0] = A.layers[i].n1; S.gain[i][1] = A.layers[i].n2; }
  // this CTA's units of one decoder step (made at set-up)
#pragma unroll 1
  for (int i = tid; i <= n_phase; i += kPT) S.pstart[i] = A.pstart[(size_t)cta * (n_phase + 1) + i];
#pragma unroll 1
  for (int i = tid; i < A.max_units; i += kPT) S.ulist[i] = A.ulist[(size_t)cta * A.max_units + i];
  // Some request has two pending tokens (the same answer in every CTA): with few rows the first step takes both, else an extra
  // pass the first of them.
  const int two = __syncthreads_or(tid < B && A.pending[3 * tid] == 2);
  const int pre = two && A.prepass ? 1 : 0;
  // the stream of units is [the list without its LM-head units, if the round has the extra pass] then the whole list per step
  if (tid == 0) {
    S.pre_units = pre ? S.pstart[n_phase - 1] : 0;
    S.per_step = S.pstart[n_phase];
    S.total_units = S.pre_units + S.per_step * G;
#pragma unroll 1
    for (int k = 0; k < A.n_ring; ++k) issue_unit(A, S, ring, k, k);
  }
  const unsigned EPS = 5u * (unsigned)A.L + 8u;          // epochs per decoder step

  // phase timeline (one CTA, thread 0): per phase one record of kTraceRec words: [0] nanosecond timer at the end of the phase (O,
  // down: when their results have arrived), [1..5] clock cycles of that thread spent in waiting for words, products and weight
  // tiles, the barrier behind them, epilogue, everything else
  const bool tr_on = TRACE && A.trace != nullptr && cta == (A.trace_cta < NC ? A.trace_cta : 0) && tid == 0;
  long long t_sec[6] = {0, 0, 0, 0, 0, 0};
  long long t_mark = 0;
  unsigned long long t_last = 0;
#define TSEC(k)                                       \
  do {                                                \
    if (TRACE && tr_on) {                             \
      const long long t_now = clock64();              \
      t_sec[k] += t_now - t_mark;                     \
      t_mark = t_now;                                 \
    }                                                 \
  } while (0)
  // a record of its own for every phase, also where the CTA had nothing to do: the timer ticks every 32 ns
#define TRACE_REC()                                                        \
  do {                                                                     \
    TSEC(4);                                                               \
    if (TRACE && tr_on && step >= 0 && trace_n < A.trace_stride) {         \
      unsigned long long* rec = A.trace + ((size_t)step * A.trace_stride + trace_n++) * kTraceRec; \
      unsigned long long now = global_timer();                             \
      for (int spin = 0; now <= t_last && spin < 1024; ++spin) now = global_timer(); \
      rec[0] = t_last = now;                                               \
      for (int k = 0; k < 6; ++k) { rec[1 + k] = (unsigned long long)t_sec[k]; t_sec[k] = 0; }     \
      t_mark = clock64();                                                  \
    }                                                                      \
  } while (0)
  // (A CTA that has seen a wait run out leaves before or after the ensemble.  Elsewhere nobody leaves: a thread whose wait ran
  // out waits no more, and the step runs through on what there is.)
  if (tr_on) t_mark = clock64();

#pragma unroll 1
  for (int it = 0; it < G + pre; ++it) {
    const int step = it - pre;                          // -1: the extra pass
    const unsigned ep_base = A.epoch0 + (unsigned)it * EPS;
    int trace_n = 0;
    // ---- slot table of the step ------------------------------------------------------------------
    const int ns = step == 0 && two && !A.prepass ? 2 * R : R;
    if (tid < kPSlots) {
      PSlot sl{0, 0, 0, 0};
      if (tid < ns) {
        const int row = tid % R, b = row / m, second = tid >= R;
        const int* pend = S.pending[b];
        sl.row = row;
        if (step < 0) {                                 // the first of two pending tokens, for the rows that have two
          sl.pos = S.kv_len[row];
          sl.tok = pend[1];
          sl.active = pend[0] == 2;
        } else if (step == 0 && A.prepass) {            // the last pending token
          sl.pos = S.kv_len[row] + pend[0] - 1;
          sl.tok = pend[pend[0]];
          sl.active = 1;
        } else if (step == 0) {
          sl.pos = S.kv_len[row] + second;
          sl.tok = pend[1 + second];
          sl.active = second ? (pend[0] == 2) : 1;
        } else {
          sl.pos = S.kv_len[row] + pend[0] + step - 1;
          sl.tok = S.tok[b];
          sl.active = 1;
        }
        if (sl.active && sl.pos >= A.cap) { sl.active = 0; atomicOr(A.err, PERR_KV); }
      }
      S.slot[tid] = sl;
      S.lmmax[tid] = S.rmax[tid] = 0u;
      S.row_part[tid] = S.row_sum[tid] = S.req_mass[tid] = 0ull;
      if (tid < R) {
        const int b = tid / m;
        S.lm_src[tid] = (step == 0 && !A.prepass && S.pending[b][0] == 2) ? R + tid : tid;
      }
      // Whose words feed column tid of the products (LM head: of the row's last token).  A column without an active slot takes
      // another one's: the columns of a product do not mix, and its own is not read.
      __syncwarp((1u << kPSlots) - 1u);
      const unsigned act = __ballot_sync((1u << kPSlots) - 1u, sl.active);
      const int any = act ? __ffs(act) - 1 : 0;
      S.col[0][tid] = sl.active ? tid : any;
      S.col[1][tid] = tid < R ? S.lm_src[tid] : S.lm_src[0];
      if (tid == 0) S.any = act != 0u;
    }
    __syncthreads();
    const int k_base = uni(step < 0 ? 0 : S.pre_units + step * S.per_step);     // first unit of this pass in the stream
    if (group == 1) {
      // Chunks of kPPos positions of all (slot, KV head) caches in (slot, head, position) order; this CTA's contiguous range of
      // them (the same for every layer of the step), and the partial results every (slot, head) pair will have.
      int T = 0;
#pragma unroll 1
      for (int s = 0; s < kPSlots; ++s) {
        const int nsp = (s < ns && S.slot[s].active) ? (S.slot[s].pos + kPPos) / kPPos : 0;
        if (tid == kGT) { S.pair_base[s] = T; S.pair_ns[s] = nsp; }
        T += A.Hkv * nsp;
      }
      // (T <= 8 slots x 64 heads x 342 chunks, so c * T stays far below 2^31)
      const int lo = cta * T / NC, hi = (cta + 1) * T / NC;
      if (tid == kGT) { S.n_tot = T; S.n_chunk = hi - lo; }
      bar_sync<2>(kGT);
#pragma unroll 1
      for (int i = lo + tid - kGT; i < hi; i += kGT) {
        int s = 0;
#pragma unroll 1
        while (i >= S.pair_base[s] + A.Hkv * S.pair_ns[s]) ++s;
        const int rem = i - S.pair_base[s], nsp = S.pair_ns[s], gk = rem / nsp;
        S.chunks[i - lo] = (uint32_t)s | ((uint32_t)gk << 3) | ((uint32_t)(rem - gk * nsp) << 9) | ((uint32_t)nsp << 18);
      }
#pragma unroll 1
      for (int i = tid - kGT; i < kPSlots * A.Hkv; i += kGT) {
        const int s = i / A.Hkv, gk = i - s * A.Hkv, nsp = S.pair_ns[s], g0 = S.pair_base[s] + gk * nsp;
        const int cnt = nsp == 0 ? 0 : ((T >= NC) ? ((g0 + nsp) * NC - 1) / T - ((g0 + 1) * NC - 1) / T + 1 : nsp);
#pragma unroll 1
        for (int t = 0; t < grp; ++t) S.nseg[s][gk * grp + t] = (unsigned char)cnt;
      }
      bar_sync<2>(kGT);
#pragma unroll 1
      for (int i = 0; i < A.kv_stages; ++i) kv_request<HD>(A, S, kv_area + i * kv_stage_bytes, i, uni(S.n_chunk), 0, gw, lane);
    }
    const int any = uni(S.any);
    const int n_half = step < 0 ? 2 * A.L : 2 * A.L + 1;
#pragma unroll 1
    for (int ph = 0; ph < n_half; ++ph) {                      // half layers: QKV, attention, O | gate/up, down; at last the LM head
      const int layer = ph >> 1;
      // epochs of the words that are read and written here
      const unsigned ep_prev_dn = ep_base + 5u * (unsigned)layer;                    // down projection of the layer before
      const unsigned ep_qkv = ep_prev_dn + 1u, ep_att = ep_qkv + 1u, ep_o = ep_qkv + 2u, ep_gu = ep_qkv + 3u, ep_dn = ep_qkv + 4u;
      if (group == 0) {
        const int kind = ph == 2 * A.L ? KIND_LM : ((ph & 1) ? KIND_GU : KIND_QKV);
        const int phase = 4 * layer + (kind == KIND_GU ? 2 : 0), ia = uni(S.pstart[phase]), ib = uni(S.pstart[phase + 1]);     // this CTA's units in the list
        if (ia < ib) {
          const int tid = own_tid(), lane = tid & 31, gw = uni(tid >> 5), gq = lane >> 2, t4 = lane & 3;
          const int n_in = kind == KIND_LM ? R : ns, n_pair = n_in > 4 ? 4 : 2, nkb = uni(S.nkb[kind]);
          const int col = S.col[kind == KIND_LM ? 1 : 0][gq];  // the slot whose words feed the lane's column of the products
          const int n = (nkb - gw + kGW - 1) / kGW;            // the warp's blocks of 16 columns: every sixth
          int r_fill = (k_base + ia) / A.n_ring, r_cur = k_base + ia - r_fill * A.n_ring;      // the next unit's filling and ring slot
          // ---- the warp's blocks of the residual as they arrive -> RMSNorm * gain, rounded: its B fragments ----------
          uint32_t bf[NF][2];
          {
            // the gains of the warp's columns wait in shared memory
            if (lane < 4) {
              const uint2* gp = reinterpret_cast<const uint2*>(kind == KIND_LM ? A.final_norm : S.gain[layer][ph & 1]) + gw * 4 + lane;
#pragma unroll 1
              for (int j = 0; j < n; ++j)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(&S.gains[(gw + j * kGW) * 4 + lane])), "l"(gp + j * kGW * 4) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            float4 xv[NF];
            if (ph == 0) {
              const uint2* er2 = reinterpret_cast<const uint2*>(A.embed + (size_t)S.slot[col].tok * d) + gw * 4 + t4;
#pragma unroll
              for (int j = 0; j < NF; ++j) {
                xv[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (j < n) xv[j] = bf16x4_to_float4(__ldg(er2 + j * kGW * 4));
              }
            } else {
              constexpr int NB = NF > 12 ? NF / 2 : NF;        // blocks in flight
#pragma unroll
              for (int h0 = 0; h0 < NF; h0 += NB) {
                uint4 raw[2 * NB];
                ll_poll<2 * NB, 2, kGW * kPSlots * 16>(((ph & 1) ? A.x1 : A.xa) + ((size_t)(gw + h0 * kGW) * kPSlots + col) * 16 + 4 * t4, any ? min(n - h0, NB) : 0,
                                                       (ph & 1) ? ep_o : ep_prev_dn, raw, dead, A.err);
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                  xv[h0 + j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                  if (h0 + j < n) xv[h0 + j] = make_float4(__uint_as_float(raw[2 * j].x), __uint_as_float(raw[2 * j].z), __uint_as_float(raw[2 * j + 1].x), __uint_as_float(raw[2 * j + 1].z));
                }
              }
              TSEC(0);
              TRACE_REC();
            }
            float sq = 0.0f;
#pragma unroll
            for (int j = 0; j < NF; ++j) sq += fmaf(xv[j].x, xv[j].x, fmaf(xv[j].y, xv[j].y, fmaf(xv[j].z, xv[j].z, xv[j].w * xv[j].w)));
            sq += __shfl_xor_sync(FULL, sq, 1);
            sq += __shfl_xor_sync(FULL, sq, 2);
            if (t4 == 0) S.red[ph & 1][gq][gw] = sq;
            cp_async_wait<0>();
            bar_sync<1>(kGT);
            const float4* rr = reinterpret_cast<const float4*>(S.red[ph & 1][gq]);      // the warps in their order
            const float4 ra = rr[0], rb = rr[1];             // (the last two are zero)
            const float sc = __frsqrt_rn((((ra.x + ra.y) + (ra.z + ra.w)) + ((rb.x + rb.y) + (rb.z + rb.w))) / (float)d + A.eps);
#pragma unroll
            for (int j = 0; j < NF; ++j) {
              const float4 g4 = bf16x4_to_float4(S.gains[(gw + max(0, min(j, n - 1)) * kGW) * 4 + t4]);
              bf[j][0] = pack_bf16(xv[j].x * sc * g4.x, xv[j].y * sc * g4.y);
              bf[j][1] = pack_bf16(xv[j].z * sc * g4.z, xv[j].w * sc * g4.w);
            }
          }
          // the epilogue's identity of the warp: slots 2 pr, 2 pr + 1 of the units q0, q0 + wpp ... of a round; of the lane: row er, slot en
          const int np = (n_in + 1) >> 1, wpp = np == 1 ? kGW : (np == 2 ? kGW / 2 : (np == 3 ? kGW / 3 : kGW / 4)), q0 = gw / np, pr = gw - q0 * np;
          const int er = lane & 15, en = 2 * pr + (lane >> 4);
          const bool e_warp = q0 < wpp, e_on = en < n_in && (kind == KIND_LM || S.slot[en].active);
          const uint32_t a_lane = smem_u32(ring) + (uint32_t)((lane & 7) + ((lane >> 3) & 1) * 8) * ((uint32_t)nkb * 32u + 16u) + (uint32_t)(lane >> 4) * 16u + (uint32_t)gw * 32u;
          // rounds of tiles; the LM head's ring is refilled twice as often with rounds of two
          const int per_round = n_in > 4 || kind == KIND_LM ? kPRound / 2 : A.round_units;
          float lm_max = -INFINITY;
          int pbuf = 0;                                        // (between phases the barrier of the sums of squares keeps the buffers apart)
#pragma unroll 1
          for (int i0 = ia; i0 < ib;) {
            const int nu = min(per_round, ib - i0), r0 = r_cur;
            float* p_warp = part + pbuf * kPBuf + t4 * kPPair + gw * 40 + gq;
#pragma unroll 1
            for (int q = 0; q < nu; ++q) {
              wait_full(S, r_cur, r_fill, dead, A.err);
              const uint32_t a_base = a_lane + (uint32_t)r_cur * (uint32_t)A.slot_bytes;
              float c[4] = {0.0f, 0.0f, 0.0f, 0.0f}, c2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
              for (int j = 0; j < NF; j += 2) {
                // (two sums and two fragments at a time)
                if (j >= n) break;
                uint32_t a[4], a2[4];
                ldsm_x4(a, a_base + (uint32_t)j * (kGW * 32u));
                const bool pair = j + 1 < n;
                if (pair) ldsm_x4(a2, a_base + (uint32_t)(j + 1) * (kGW * 32u));
                mma_bf16(c, a, bf[j]);
                if (pair) mma_bf16(c2, a2, bf[j + 1]);
              }
#pragma unroll
              for (int e = 0; e < 4; ++e) c[e] += c2[e];
              if (2 * t4 < n_in) { p_warp[0] = c[0]; p_warp[16] = c[1]; p_warp[8] = c[2]; p_warp[24] = c[3]; }
              p_warp += n_pair * kPPair;
              if (++r_cur == A.n_ring) { r_cur = 0; ++r_fill; }
            }
            TSEC(1);
            dead |= bar_sync_or<1>(kGT, dead);           // units fully read, partial tiles complete
            TSEC(2);
            if (tid == kGT - 32 && !dead) {
              int r = r0;
#pragma unroll 1
              for (int q = 0; q < nu; ++q) { issue_unit(A, S, ring, k_base + i0 + q + A.n_ring, r); if (++r == A.n_ring) r = 0; }
            }
            if (e_warp) {
#pragma unroll 1
              for (int q = q0; q < nu; q += wpp) {
                const float* pp = part + pbuf * kPBuf + (q * n_pair + pr) * kPPair + lane;
                const int tile = unit_tile(uni(S.ulist[i0 + q]));
                float v = 0.0f;
#pragma unroll
                for (int w2 = 0; w2 < kGW; ++w2) v += pp[w2 * 40];
                if (kind == KIND_GU) {
                  const float up = __shfl_down_sync(FULL, v, 8);
                  const float gated = v / (1.0f + expf(-v)) * up;
                  const float right = __shfl_down_sync(FULL, gated, 1);
                  if (e_on && (er & 9) == 0)
                    ll_store(A.mid + op_word(tile >> 1, en) + (tile & 1) * 4 + (er >> 1), pack_bf16(gated, right), ep_gu);
                } else if (kind == KIND_LM) {
                  const int o = tile * 16 + er;
                  if (e_on && o < V) {
                    A.logits_own[((size_t)step * R + en) * V + o] = v;
                    lm_max = fmaxf(lm_max, v);
                  }
                } else {
                  // q and k: rows r and r + 8 are a pair of the rotation (dims half a head apart)
                  int cq = tile * 16 + er;
                  if (tile * 16 < d + kvd) {
                    const int in_head = (tile * 16) & (HD - 1);
                    const size_t at = (size_t)S.slot[en].pos * half + (in_head >> 1) + (er & 7);
                    const float cs = e_on ? __ldg(A.rope_cos + at) : 0.0f, sn = e_on ? __ldg(A.rope_sin + at) : 0.0f;
                    const float other = __shfl_xor_sync(FULL, v, 8);
                    v = er < 8 ? v * cs - other * sn : v * cs + other * sn;
                    cq = tile * 16 - (in_head >> 1) + (er & 7) + (er < 8 ? 0 : half);
                  }
                  const float right = __shfl_down_sync(FULL, v, 1);
                  if (e_on && (er & 1) == 0) ll_store(A.qkv + (((size_t)en * A.qkv_w + cq) >> 1), pack_bf16(v, right), ep_qkv);
                }
              }
            }
            i0 += nu;
            pbuf ^= 1;
            TSEC(3);
          }
          if (kind == KIND_LM) {
            // running maxima of the logits: 16 lanes of a slot, then the CTA
#pragma unroll
            for (int o2 = 8; o2 > 0; o2 >>= 1) lm_max = fmaxf(lm_max, __shfl_xor_sync(FULL, lm_max, o2));
            if (e_warp && er == 0 && en < R && lm_max > -INFINITY) atomicMax(&S.lmmax[en], ord_encode(lm_max));
          }
        } else if (ph) {
          TRACE_REC();
        }
        if (kind != KIND_LM) TRACE_REC();
      }
      // ---- attention over the rows' caches (after the QKV phase; group 1) ---------------------------
      // The caches of all (slot, KV head) pairs are cut into chunks of kPPos positions; the chunks, in (slot, head,
      // position) order, are dealt to the CTAs in contiguous ranges, so a CTA walks along one cache for several chunks.
      // A warp owns 16 positions of a chunk: K and V as mma A fragments (positions, resp. dims, as rows; the heads of the group
      // are the 8 columns of B): scores^T = K q^T, out^T = V^T P^T with P as a sum of bf16 terms.
      // The order of the summed index of a product is free, so the dims of q.k are dealt to the k-steps such that lane (g, t)
      // needs whole 16-byte pieces t, t + 4 ... of rows g and g + 8; in V^T P^T rows g and g + 8 of an m-tile stand for two
      // neighbouring dims of the pieces that the lane holds of the four positions 2t, 2t+1, 8+2t, 9+2t (pairs of
      // positions are interleaved with byte permutes).  So a lane copies its own pieces into its own places of a stage in shared
      // memory (cp.async; nobody else reads them: no barrier), kv_stages chunks ahead: the cached positions do not depend on
      // this step, and a layer's first chunks are on their way before the down projection of the layer before.
      // A warp carries its (max, sum, un-normalised output) in registers through a segment (= the part of one pair's cache
      // this CTA owns).  At the end of a segment the warps are merged into one partial result per head.  The CTA with a pair's last segment puts
      // the pair's partial results together (when it is through with its own chunks) and hands the O projection its operand.
      const int n_chunk = group == 0 || (ph & 1) || ph == 2 * A.L ? 0 : uni(S.n_chunk);
      if (n_chunk) {
        const int tid = own_tid() - kGT, lane = tid & 31, gw = uni(tid >> 5), gq = lane >> 2, t4 = lane & 3;
        constexpr int KP = HD / 32, MT = HD / 16;              // 16-byte pieces of a K row per lane; m-tiles of V^T P^T
        uint32_t qa[HD / 16][2];
        float oc[MT][4], m_run[2], l_run[2];                   // heads 2t, 2t + 1
        int fin = -1;                                          // slot * 256 + KV head of a pair whose partial results are still to be added
        const float scale2 = A.attn_scale * 1.4426950408889634f;      // scores in base-2 units
        int stage = 0;
        bool appended = false;
#pragma unroll
        for (int j = 0; j < HD / 16; ++j) qa[j][0] = qa[j][1] = 0u;
#pragma unroll 1
        for (int gc = 0; gc < n_chunk; ++gc) {
          const uint32_t ce = uni(S.chunks[gc]);
          const int s = ce & 7, gk = (ce >> 3) & 63, split = (ce >> 9) & 511, nsplit = ce >> 18;
          const int pos = uni(S.slot[s].pos), n_fresh = s >= R ? 2 : 1;      // the positions pos (and pos - 1) are this phase's own
          if (gc == 0 || split == 0) {
            // ---- a segment begins ----
            if (gc) dead |= bar_sync_or<2>(kGT, dead);         // the segment before has been merged
            const uint2* qw = A.qkv + ((unsigned)(s * A.qkv_w + gk * grp * HD) >> 1);
            {
              uint4 raw[HD / 16];
              ll_poll<HD / 16, 2, 16>(qw + (gq < grp ? gq : 0) * half + 4 * t4, HD / 32, ep_qkv, raw, dead, A.err);
#pragma unroll
              for (int j = 0; j < HD / 16; ++j) { qa[j][0] = raw[j].x; qa[j][1] = raw[j].z; }
            }
            m_run[0] = m_run[1] = -INFINITY; l_run[0] = l_run[1] = 0.0f;
#pragma unroll
            for (int j = 0; j < MT; ++j) oc[j][0] = oc[j][1] = oc[j][2] = oc[j][3] = 0.0f;
          }
          // ---- the warp's 16 positions ----
          const int p0 = split * kPPos + gw * 16, lim = pos + 1 - p0, cached = lim - n_fresh;      // its positions (if fewer), those from the cache
          if (A.kv_stages == 1) cp_async_wait<0>(); else if (A.kv_stages == 2) cp_async_wait<1>(); else cp_async_wait<2>();
          unsigned char* st = kv_area + stage * kv_stage_bytes + (gw * 32 + lane) * 16;
          if (lim > 0 && cached < 16) {
            // the positions produced in this very phase come as words: they take their places in the stage, the last one in the cache too
            if (cached <= 0) {                                 // (nothing was asked for: the places of the others must not hold what is not finite)
#pragma unroll
              for (int i = 0; i < kv_pieces<HD>(); ++i) *reinterpret_cast<uint4*>(st + i * kv_piece) = make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll 1
            for (int j = 0; j < n_fresh; ++j) {
              const int r = pos - j - p0;
              if (r < 0 || r > 15) continue;
              const uint2* kw = A.qkv + ((unsigned)((s - j * R) * A.qkv_w + d + gk * HD) >> 1) + t4 * 4;
              const uint2* vv = A.qkv + ((unsigned)((s - j * R) * A.qkv_w + d + kvd + gk * HD) >> 1) + (HD == 32 ? (gq & 3) * 4 + (gq >> 2) * 2 : gq * 4);
              constexpr int VP = HD == 32 ? 1 : HD / 32;       // 16-byte loads (two words) of V
              uint4 x[2 * KP + VP];
              unsigned spins = 0;
              uint32_t miss;
#pragma unroll 1
              do {
                miss = 0;
#pragma unroll
                for (int i = 0; i < 2 * KP; ++i) x[i] = ll_load2(kw + (i >> 1) * 16 + 2 * (i & 1));
#pragma unroll
                for (int i = 0; i < VP; ++i) x[2 * KP + i] = ll_load2(vv + (i >> 1) * 32 + 2 * (i & 1));
#pragma unroll
                for (int i = 0; i < 2 * KP + VP; ++i) miss |= (x[i].y ^ ep_qkv) | (x[i].w ^ ep_qkv);
                if (++spins > kSpinLimit) dead = ll_timeout(A.err);
              } while (miss && !dead);
              const size_t row = (size_t)((unsigned)((S.slot[s].row * A.L + layer) * A.Hkv + gk) * A.cap + pos) * HD;
              appended = true;
              if (gq == (r & 7)) {
#pragma unroll
                for (int i = 0; i < KP; ++i) {
                  const uint4 k8 = make_uint4(x[2 * i].x, x[2 * i].z, x[2 * i + 1].x, x[2 * i + 1].z);
                  *reinterpret_cast<uint4*>(st + ((r >> 3) * KP + i) * kv_piece) = k8;
                  if (j == 0) *reinterpret_cast<uint4*>(A.kc + row + (t4 + 4 * i) * 8) = k8;
                }
              }
              if (t4 == ((r & 7) >> 1)) {
                const int i = (r >> 3) * 2 + (r & 1);
                if constexpr (HD == 32) {
                  const uint2 v4 = make_uint2(x[2 * KP].x, x[2 * KP].z);
                  *reinterpret_cast<uint2*>(st + (2 * KP + i) * kv_piece + (gq >> 2) * 8) = v4;
                  if (j == 0) *reinterpret_cast<uint2*>(A.vc + row + (gq & 3) * 8 + (gq >> 2) * 4) = v4;
                } else {
#pragma unroll
                  for (int q = 0; q < VP / 2; ++q) {
                    const uint4 v8 = make_uint4(x[2 * KP + 2 * q].x, x[2 * KP + 2 * q].z, x[2 * KP + 2 * q + 1].x, x[2 * KP + 2 * q + 1].z);
                    *reinterpret_cast<uint4*>(st + (2 * KP + i * (VP / 2) + q) * kv_piece) = v8;
                    if (j == 0) *reinterpret_cast<uint4*>(A.vc + row + (gq + 8 * q) * 8) = v8;
                  }
                }
              }
            }
          }
          uint32_t vw[4][MT];
          float sc[2][4];
          if (lim > 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if constexpr (HD == 32) {
                const uint2 x = *reinterpret_cast<const uint2*>(st + (2 * KP + i) * kv_piece + (gq >> 2) * 8);     // dims 8 (g & 3) + 4 (g >> 2) ..
                vw[i][0] = x.x; vw[i][1] = x.y;
              } else {
#pragma unroll
                for (int j = 0; j < MT / 4; ++j) {
                  const uint4 x = *reinterpret_cast<const uint4*>(st + (2 * KP + i * (MT / 4) + j) * kv_piece);
                  vw[i][4 * j] = x.x; vw[i][4 * j + 1] = x.y; vw[i][4 * j + 2] = x.z; vw[i][4 * j + 3] = x.w;
                }
              }
            }
            // scores: entries 0, 1: position g, heads 2t, 2t+1; entries 2, 3: position g + 8
#pragma unroll
            for (int e = 0; e < 4; ++e) sc[0][e] = sc[1][e] = 0.0f;
#pragma unroll
            for (int j = 0; j < KP; ++j) {
              const uint4 k0 = *reinterpret_cast<const uint4*>(st + j * kv_piece), k1 = *reinterpret_cast<const uint4*>(st + (KP + j) * kv_piece);
              const uint32_t a0[4] = {k0.x, k1.x, k0.y, k1.y}, a1[4] = {k0.z, k1.z, k0.w, k1.w};
              mma_bf16(sc[0], a0, qa[2 * j]); mma_bf16(sc[1], a1, qa[2 * j + 1]);
            }
          }
          // (the scores have read all of the stage's pieces of K, and those of V were asked for before them)
          kv_request<HD>(A, S, kv_area + stage * kv_stage_bytes, gc + A.kv_stages, n_chunk, layer, gw, lane);
          if (++stage == A.kv_stages) stage = 0;
          if (lim > 0) {
            // ---- softmax and P V for all heads of the group at once ----
            float pw[4], f[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              // (the maximum is of the rounded products, any reference will do; the weight's exponent is rounded once, behind the
              // subtraction: a score's own rounding would cost a weight 2^-24 times the score)
              const float x0 = gq < lim ? sc[0][e] + sc[1][e] : -INFINITY, x1 = gq + 8 < lim ? sc[0][e + 2] + sc[1][e + 2] : -INFINITY;
              float mx = fmaxf(x0 * scale2, x1 * scale2);
#pragma unroll
              for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
              const float Mn = fmaxf(m_run[e], mx), N = Mn > -INFINITY ? Mn : 0.0f;
              f[e] = ex2_approx(m_run[e] - N);
              m_run[e] = Mn;
              pw[e] = ex2_approx(fmaf(x0, scale2, -N)); pw[e + 2] = ex2_approx(fmaf(x1, scale2, -N));
              l_run[e] = fmaf(l_run[e], f[e], pw[e] + pw[e + 2]);
            }
            // The weights as bf16 terms of 8 bits (fp32 sums), moved from accumulator layout (positions as rows) to B-operand
            // layout (positions as the summed index): three terms, all of an fp32 weight - two for the cached positions of head size 64.
            // (With two for all of them a sum of 300 positions that cancel is eleven times as far off, at head sizes 32 and 128; the
            // third term costs at most 1 % of a round: 3 rows of 6000 positions at 32 / 128 919 / 1010 -> 907 / 1018 us with
            // all that is here, of 8192 at 64, where the new positions have it, 4057 -> 4095.)
            uint32_t t0, t1, w0[2], w1[2], w2[2];
            auto term = [&](uint32_t (&w)[2]) {
              t0 = pack_bf16(pw[0], pw[1]); t1 = pack_bf16(pw[2], pw[3]);
              w[0] = movmatrix_trans(t0); w[1] = movmatrix_trans(t1);
            };
            auto remainder = [&]() {
              pw[0] -= __uint_as_float(t0 << 16); pw[1] -= __uint_as_float(t0 & 0xFFFF0000u);
              pw[2] -= __uint_as_float(t1 << 16); pw[3] -= __uint_as_float(t1 & 0xFFFF0000u);
            };
            auto values = [&](int j, uint32_t (&af)[4]) {
              af[0] = __byte_perm(vw[0][j], vw[1][j], 0x5410u); af[1] = __byte_perm(vw[0][j], vw[1][j], 0x7632u);
              af[2] = __byte_perm(vw[2][j], vw[3][j], 0x5410u); af[3] = __byte_perm(vw[2][j], vw[3][j], 0x7632u);
            };
            term(w0); remainder(); term(w1);
            if constexpr (HD != 64) { remainder(); term(w2); }
#pragma unroll
            for (int j = 0; j < MT; ++j) {
              uint32_t af[4];
              values(j, af);
              // (the tensor core's sums are cut off, not rounded: the smallest terms first, and only these 16 positions'.  Sums
              // carried through it were 9 % further off at head size 32; 8192 positions 4098 -> 4139 us)
              float t[4] = {0.0f, 0.0f, 0.0f, 0.0f};
              if constexpr (HD != 64) mma_bf16(t, af, w2);
              mma_bf16(t, af, w1);
              mma_bf16(t, af, w0);
#pragma unroll
              for (int e = 0; e < 4; ++e) oc[j][e] = fmaf(oc[j][e], f[e & 1], t[e]);
            }
            if (HD == 64 && cached < 16) {
              remainder(); term(w2);
#pragma unroll
              for (int j = 0; j < MT; ++j) {
                uint32_t af[4];
                values(j, af);
                mma_bf16(oc[j], af, w2);
              }
            }
          }
          if (split == nsplit - 1 || gc == n_chunk - 1) {
            // ---- a segment ends: the warps' states, in warp order -> its partial result ----
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int head = 2 * t4 + e;
              float l = l_run[e];
#pragma unroll
              for (int o = 4; o < 32; o <<= 1) l += __shfl_xor_sync(FULL, l, o);
              if (head < grp) {
                // (rows g and g + 8 of m-tile j: two neighbouring dims)
                float* so = s_o + (gw * grp + head) * HD + (HD == 32 ? 8 * (gq & 3) + 4 * (gq >> 2) : 8 * gq);
#pragma unroll
                for (int j = 0; j < MT; ++j) *reinterpret_cast<float2*>(so + (HD == 32 ? 2 * j : 64 * (j >> 2) + 2 * (j & 3))) = make_float2(oc[j][e], oc[j][e + 2]);
                if (gq == 0) { S.am[gw][head] = m_run[e]; S.al[gw][head] = l; }
              }
            }
            dead |= bar_sync_or<2>(kGT, dead);
            const int n_seg = uni(S.nseg[s][gk * grp]);
            if (n_seg > 1 && split == nsplit - 1) fin = s * 256 + gk;
#pragma unroll 1
            for (int i = gw; i < grp * (HD / 32); i += kGW) {
              // 32 dims of a head; a lane: dim dd of head t of the group
              const int t = i / (HD / 32), dd = (i % (HD / 32)) * 32 + lane, head = gk * grp + t;
              // lane w: warp w's state
              float mw = -INFINITY, lw = 0.0f;
              if (lane < kGW) { mw = S.am[lane][t]; lw = S.al[lane][t]; }
              const float M = warp_max_f32(mw), f = mw > -INFINITY ? ex2_approx(mw - M) : 0.0f;
              const float l = warp_sum_f32(f * lw);
              float v = 0.0f;
              const float* so = s_o + t * HD + dd;
#pragma unroll
              for (int w2 = 0; w2 < kGW; ++w2, so += grp * HD) v = fmaf(__shfl_sync(FULL, f, w2), *so, v);
              if (n_seg == 1) {
                store_att(A, s, head * HD + dd, v / l, ep_att);
              } else {
                // Its place among the pair's partial results: with at least as many chunks as CTAs every CTA owns
                // chunks, so the segments of a pair sit on consecutive CTAs; with fewer, a segment is one chunk.
                const int T = S.n_tot, g0 = S.pair_base[s] + gk * nsplit, ord = (T >= NC) ? cta - ((g0 + 1) * NC - 1) / T : split;
                uint2* p = A.part + ((size_t)((s * A.H + head) * A.n_part + ord) * HD + dd) * 4;
                ll_store2(p, __float_as_uint(v), __float_as_uint(M), ep_att);
                ll_store2(p + 2, __float_as_uint(l), 0u, ep_att);
              }
            }
          }
        }
        if (fin >= 0)
#pragma unroll 1
        for (int i = gw; i < grp * (HD / 32); i += kGW) {
          // the partial results of the pair's segments, in their order, six of them in flight
          const int ps = fin >> 8, head = (fin & 255) * grp + i / (HD / 32), dd = (i % (HD / 32)) * 32 + lane, n_seg = uni(S.nseg[ps][head]);
          const uint2* p = A.part + ((size_t)((ps * A.H + head) * A.n_part) * HD + dd) * 4;
          float M = -INFINITY, l = 0.0f, v = 0.0f;
#pragma unroll 1
          for (int j0 = 0; j0 < n_seg; j0 += 6, p += 6 * HD * 4) {
            uint4 raw[12];
            const int n = min(6, n_seg - j0);
            ll_poll<12, 2, HD * 4>(p, n, ep_att, raw, dead, A.err);
            float Mn = M;
#pragma unroll
            for (int j = 0; j < 6; ++j) if (j < n) Mn = fmaxf(Mn, __uint_as_float(raw[2 * j].z));
            const float N = Mn > -INFINITY ? Mn : 0.0f, fo = ex2_approx(M - N);
            v *= fo; l *= fo;
#pragma unroll
            for (int j = 0; j < 6; ++j) {
              if (j >= n) break;
              const float f = ex2_approx(__uint_as_float(raw[2 * j].z) - N);
              v = fmaf(f, __uint_as_float(raw[2 * j].x), v); l = fmaf(f, __uint_as_float(raw[2 * j + 1].x), l);
            }
            M = Mn;
          }
          store_att(A, ps, head * HD + dd, v / l, ep_att);
        }
        // (the new rows are read from the cache one step later, by CTAs that have heard of this one since)
        if (appended) __threadfence();
      }
      if (group == 0) {
        if (!(ph & 1) && ph < 2 * A.L) TRACE_REC();
      } else if (ph < 2 * A.L) {
        if ((ph & 1) && layer + 1 < A.L)                       // the next layer's first chunks of K and V
#pragma unroll 1
          for (int i = 0; i < A.kv_stages; ++i) kv_request<HD>(A, S, kv_area + i * kv_stage_bytes, i, uni(S.n_chunk), layer + 1, gw, lane);
        const int kind = (ph & 1) ? KIND_DN : KIND_O, phase = 4 * layer + kind, ia = uni(S.pstart[phase]), ib = uni(S.pstart[phase + 1]);
        if (ia < ib) {
          const int tid = own_tid(), lane = tid & 31, gw = uni(tid >> 5) - kGW, gq = lane >> 2, t4 = lane & 3;
          const int nkb = uni(S.nkb[kind]), nsub = uni(S.nsub[kind]), col = S.col[0][gq];
          const int er = lane & 7, en = 4 * gw + (lane >> 3);  // the epilogue: a warp has four slots, a lane a row of one
          const bool e_warp = 4 * gw < ns, e_on = en < ns && S.slot[en & 7].active;
          const uint32_t a_lane = smem_u32(ring) + (uint32_t)(lane & 7) * ((uint32_t)nkb * 32u + 16u) + (uint32_t)((lane >> 3) & 1) * 16u;
          int r_fill = (k_base + ia) / A.n_ring, r_cur = k_base + ia - r_fill * A.n_ring;      // the next unit's filling and ring slot
          float c[4] = {0.0f, 0.0f, 0.0f, 0.0f}, c2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
          int kb = gw, pbuf = ph & 1;                          // the warp's next block of its tile; buffer of the next partial tile
#pragma unroll 1
          for (int i0 = ia; i0 < ib;) {
            // a round: sub-units of one tile, as many as the ring takes
            const uint32_t u0 = uni(S.ulist[i0]);
            const int sub0 = unit_sub(u0), nu = min(A.round_units, nsub - sub0), tile = unit_tile(u0), r0 = r_cur;
            const bool last = sub0 + nu == nsub;
            // the residual that the epilogue adds to arrived phases ago: requested now
            const unsigned x_word = ((unsigned)(tile >> 1) * kPSlots + (en & 7)) * 16 + (tile & 1) * 8 + er;
            const uint2* base_p = ((ph & 1) ? A.x1 : A.xa) + x_word;
            uint2 base_w = make_uint2(0u, 0u);
            if (last && e_warp && e_on) {
              if (ph == 0) base_w.x = __float_as_uint(__bfloat162float(A.embed[(size_t)S.slot[en].tok * d + tile * 8 + er]));
              else base_w = ll_load1(base_p);
            }
#pragma unroll 1
            for (int q = 0; q < nu; ++q) {
              wait_full(S, r_cur, r_fill, dead, A.err);
              if (++r_cur == A.n_ring) { r_cur = 0; ++r_fill; }
            }
            if (sub0 == 0) { c[0] = c[1] = c[2] = c[3] = c2[0] = c2[1] = c2[2] = c2[3] = 0.0f; kb = gw; }
            const int end = (sub0 + nu) * nkb;
            int lk = kb - sub0 * nkb, rs = r0;                 // block within its unit, the unit's slot
#pragma unroll 1
            while (kb < end) {
              // the warp's words ARE its B fragments: sixteen blocks in flight
              uint4 raw[16];
              const int n = min(16, (end - kb + kGW - 1) / kGW);
              ll_poll<16, 1, kGW * kPSlots * 8>(((ph & 1) ? A.mid : A.att) + op_word(kb, col) + 2 * t4, any ? n : 0, (ph & 1) ? ep_gu : ep_att, raw, dead, A.err);
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                if (j >= n) break;
#pragma unroll 1
                while (lk >= nkb) { lk -= nkb; if (++rs == A.n_ring) rs = 0; }
                uint32_t a2[2];
                ldsm_x2(a2, a_lane + (uint32_t)rs * (uint32_t)A.slot_bytes + (uint32_t)lk * 32u);
                const uint32_t a[4] = {a2[0], 0u, a2[1], 0u}, b[2] = {raw[j].x, raw[j].z};      // (rows 8 - 15 of the product are idle)
                if (j & 1) mma_bf16(c2, a, b); else mma_bf16(c, a, b);
                lk += kGW;
              }
              kb += n * kGW;
            }
            if (last && 2 * t4 < ns) {
              float* p_warp = part + 2 * kPBuf + pbuf * (kPBuf / 2) + t4 * kPPair + gw * 40 + gq;
              p_warp[0] = c[0] + c2[0]; p_warp[16] = c[1] + c2[1];
            }
            dead |= bar_sync_or<2>(kGT, dead);           // units fully read, partial tiles complete
            if (last && e_warp) {
              const float* pp = part + 2 * kPBuf + pbuf * (kPBuf / 2) + (en >> 1) * kPPair + (en & 1) * 16 + er;
              float v = 0.0f;
              if (e_on) {
#pragma unroll
                for (int w2 = 0; w2 < kGW; ++w2) v += pp[w2 * 40];
                const unsigned ep_b = (ph & 1) ? ep_o : ep_prev_dn;
                v += __uint_as_float(ph == 0 || base_w.y == ep_b ? base_w.x : ll_wait1(base_p, ep_b, dead, A.err));
                ll_store(((ph & 1) ? A.xa : A.x1) + x_word, __float_as_uint(v), (ph & 1) ? ep_dn : ep_o);
              }
            }
            if (tid == kPT - 32 && !dead) {
              int r = r0;
#pragma unroll 1
              for (int q = 0; q < nu; ++q) { issue_unit(A, S, ring, k_base + i0 + q + A.n_ring, r); if (++r == A.n_ring) r = 0; }
            }
            i0 += nu;
            if (last) pbuf ^= 1;
            if (last && i0 < ib) bar_sync<2>(kGT);             // (several tiles: the next phase starts with either buffer)
          }
        }
      }
    }  // half layers

    if (step < 0) {
      // The extra pass ends with its last layer.  Its cache rows are read in step 0 by CTAs that may not have waited for
      // anything behind this CTA's part of it: every CTA tells every other one that it is through (in the table of the sums,
      // which step 0 writes only after every CTA has been heard of again).
      __syncthreads();
      if (tid == 0) { __threadfence(); ll_store(A.rowsum + (size_t)cta * 2, 1u, ep_base + 5u * (unsigned)A.L + 1u); }
#pragma unroll 1
      for (int c2 = tid; c2 < NC; c2 += kPT) ll_wait1(A.rowsum + (size_t)c2 * 2, ep_base + 5u * (unsigned)A.L + 1u, dead, A.err);
      if (__syncthreads_or(dead)) goto drain;
      continue;
    }
    if (__syncthreads_or(dead)) goto drain;
    TRACE_REC();

    // ---- ensemble: exact softmax of the m rows, weighted average, draw (Algorithm 1 steps 6-7) -----
    // A CTA has the vocabulary slice of its own LM-head tiles: it reads back logits that it wrote itself.  Three exchanges, each
    // a table of flagged words that every CTA polls whole: every CTA's maxima of the rows, its integer exp sums, the masses of its
    // slice of q.  Then every CTA finds the drawn slice and, in that slice's own masses (words too), the token.
    {
      const int tid = own_tid(), lane = tid & 31, warp = uni(tid >> 5);
      const float* lg = (A.logits_override ? A.logits_override : A.logits_own) + (size_t)step * R * V;
      const int nt = A.geom[KIND_LM].n_tiles, v_lo = (int)((long long)cta * nt / NC) * 16, nv = max(0, min((int)((long long)(cta + 1) * nt / NC) * 16, V) - v_lo);
      const int n_cp = (NC + 1) & ~1;                 // maxima: [row][n_cp] words
      const unsigned ep_lm = ep_base + 5u * (unsigned)A.L + 1u, ep_sum = ep_lm + 2u, ep_mix = ep_lm + 3u;
      const int wpr = kPW / R, row = warp / wpr, ti = (warp - row * wpr) * 32 + lane, tn = wpr * 32;      // warps of a row
      const bool row_on = row < R;
      const float* lrow = lg + (size_t)(row_on ? row : 0) * V + v_lo;
      if (A.logits_override) {                        // the maxima gathered by the LM head belong to other logits
        if (tid < kPSlots) S.lmmax[tid] = 0u;
        __syncthreads();
        float mx = -INFINITY;
        if (row_on) {
#pragma unroll 1
          for (int i = ti; i < nv; i += tn) mx = fmaxf(mx, __ldcg(lrow + i));
        }
        mx = warp_max_f32(mx);
        if (row_on && lane == 0 && mx > -INFINITY) atomicMax(&S.lmmax[row], ord_encode(mx));
        __syncthreads();
      }
      const unsigned ep_max = A.logits_override ? ep_lm + 1u : ep_lm;
      if (tid < R) {
        ll_store(A.rowmax + (size_t)tid * n_cp + cta, S.lmmax[tid], ep_max);
        if (cta == NC - 1 && (NC & 1)) ll_store(A.rowmax + (size_t)tid * n_cp + NC, 0u, ep_max);
      }
      if (A.logits_override) TRACE_REC();
      float x0 = ti < nv ? __ldcg(lrow + ti) : 0.0f, x1 = ti + tn < nv ? __ldcg(lrow + ti + tn) : 0.0f;      // (stored before the barrier)
      if (row_on) {
        uint32_t mx = 0;
#pragma unroll 1
        for (int i = ti; i < n_cp / 2; i += tn) {
          const uint4 w = ll_wait2(A.rowmax + (size_t)row * n_cp + 2 * i, ep_max, dead, A.err);
          mx = max(mx, max(w.x, w.z));
        }
        mx = __reduce_max_sync(FULL, mx);
        if (lane == 0) atomicMax(&S.rmax[row], mx);
      }
      __syncthreads();
      float* s_e = part;                              // the exponentials of the slice, where they fit
      const bool keep = R * nv <= kPPartFloats;
      {
        const float mx = ord_decode(S.rmax[row_on ? row : 0]);
        unsigned long long sm = 0;
        if (row_on) {
#pragma unroll 1
          for (int i = ti; i < nv; i += tn) {
            const float e = xexp(__fsub_rn(x0, mx));
            x0 = x1;
            if (i + 2 * tn < nv) x1 = __ldcg(lrow + i + 2 * tn);
            if (keep) s_e[row * nv + i] = e;
            sm += mass_of(e);
          }
        }
        sm = warp_sum_u64(sm);
        if (row_on && lane == 0) atomicAdd(&S.row_sum[row], sm);
      }
      __syncthreads();
      if (tid < R) {
        const unsigned long long t = S.row_sum[tid];
        ll_store2(A.rowsum + ((size_t)tid * NC + cta) * 2, (uint32_t)t, (uint32_t)(t >> 32), ep_sum);
      }
      TRACE_REC();
      // every CTA's sums -> the rows' normalisers (integer sums: order-free)
      if (row_on) {
        unsigned long long t = 0;
#pragma unroll 1
        for (int i = ti; i < NC; i += 2 * tn) {                // two in flight
          const uint2 *w0 = A.rowsum + ((size_t)row * NC + i) * 2, *w1 = i + tn < NC ? w0 + 2 * tn : w0;
          uint4 a = ll_load2(w0), b = ll_load2(w1);
          if (a.y != ep_sum || a.w != ep_sum) a = ll_wait2(w0, ep_sum, dead, A.err);
          if (b.y != ep_sum || b.w != ep_sum) b = ll_wait2(w1, ep_sum, dead, A.err);
          t += (unsigned long long)a.x | ((unsigned long long)a.z << 32);
          if (w1 != w0) t += (unsigned long long)b.x | ((unsigned long long)b.z << 32);
        }
        t = warp_sum_u64(t);
        if (lane == 0) atomicAdd(&S.row_part[row], t);
      }
      __syncthreads();
      // mix: a request's warps share the slice
      const int wpb = kPW / B, b = warp / wpb;
      if (b < B) {
        const int tj = (warp - b * wpb) * 32 + lane;
        unsigned long long sm = 0;
        float bv = -1.0f; int bi = 0x7fffffff;
#pragma unroll 1
        for (int i = tj; i < nv; i += wpb * 32) {
          float acc = 0.0f;
#pragma unroll 1
          for (int k = 0; k < m; ++k) {
            const int r2 = b * m + k;
            const float e = keep ? s_e[r2 * nv + i] : xexp(__fsub_rn(__ldcg(lg + (size_t)r2 * V + v_lo + i), ord_decode(S.rmax[r2])));
            const float a = __fdiv_rn(e, norm_of(S.row_part[r2])), t = __fmul_rn(S.mix_w[r2], a);
            acc = (k == 0) ? t : __fadd_rn(acc, t);
            A.qk[(((size_t)b * G + step) * m + k) * V + v_lo + i] = a;
          }
          A.q[((size_t)b * G + step) * V + v_lo + i] = acc;
          if (A.greedy) {
            if (acc > bv) { bv = acc; bi = v_lo + i; }
          } else {
            const unsigned long long ms = mass_of(acc);
            ll_store2(A.mass + ((size_t)b * V + v_lo + i) * 2, (uint32_t)ms, (uint32_t)(ms >> 32), ep_mix);
            sm += ms;
          }
        }
        if (A.greedy) {
          best_of_warp(bv, bi);
          // (values are not negative: their bits are in their order; the lowest index wins)
          if (lane == 0 && bv >= 0.0f) atomicMax(&S.req_mass[b], ((unsigned long long)__float_as_uint(bv) << 32) | (uint32_t)~bi);
        } else {
          sm = warp_sum_u64(sm);
          if (lane == 0) atomicAdd(&S.req_mass[b], sm);
        }
      }
      __syncthreads();
      if (tid < B) {
        const unsigned long long t = S.req_mass[tid];
        uint2* dst = A.slice_mass + ((size_t)tid * NC + cta) * 2;
        if (!A.greedy) ll_store2(dst, (uint32_t)t, (uint32_t)(t >> 32), ep_mix);
        else ll_store2(dst, t ? (uint32_t)(t >> 32) : __float_as_uint(-1.0f), t ? ~(uint32_t)t : 0x7fffffffu, ep_mix);
      }
      TRACE_REC();
      // a warp a request: every CTA locates the drawn token itself (the next step's embedding gather needs it)
      if (warp < B) {
        const uint2* sl = A.slice_mass + (size_t)warp * NC * 2;
        int y = 0;
        if (A.greedy) {
          float bv = -1.0f; int bi = 0x7fffffff;
#pragma unroll 1
          for (int i = lane; i < NC; i += 32) {
            const uint4 w = ll_wait2(sl + 2 * i, ep_mix, dead, A.err);
            const float cv = __uint_as_float(w.x);
            if (cv > bv || (cv == bv && (int)w.z < bi)) { bv = cv; bi = (int)w.z; }
          }
          best_of_warp(bv, bi);
          y = bi;
          if ((unsigned)y >= (unsigned)V) { if (lane == 0) atomicOr(A.err, 1); y = 0; }      // (no value compares: not finite)
        } else {
          Found f = find_mass(sl, NC, true, A.u[warp * G + step], ep_mix, 0ull, dead, A.err);
          if (f.at < 0) {
            if (lane == 0) atomicOr(A.err, 1);
          } else {
            const int lo = (int)((long long)f.at * nt / NC) * 16, n = min((int)((long long)(f.at + 1) * nt / NC) * 16, V) - lo;
            f = find_mass(A.mass + ((size_t)warp * V + lo) * 2, n, false, 0.0f, ep_mix, f.thr, f.dead, A.err);
            if (f.at < 0 && lane == 0) atomicOr(A.err, 2);
            y = f.at < 0 ? 0 : lo + f.at;
          }
          dead |= f.dead;
        }
        if (lane == 0) {
          S.tok[warp] = y;
          if (cta == 0) {
            A.tokens[warp * G + step] = y;
            if (A.out_tokens) A.out_tokens[warp * G + step] = y;
          }
        }
      }
      if (__syncthreads_or(dead)) goto drain;
    }
  }  // steps
#undef TRACE_REC
#undef TSEC
  return;

drain:
  // a wait ran out: let the copies already issued land before the shared memory is released
  __syncthreads();
  if (tid < A.n_ring && S.issued[tid]) {
    unsigned spins = 0;
#pragma unroll 1
    while (!mbar_try_wait(&S.full[tid], (unsigned)(S.issued[tid] - 1) & 1u) && ++spins < kSpinLimit) __nanosleep(64);
  }
  __syncthreads();
}

}  // namespace tabed
