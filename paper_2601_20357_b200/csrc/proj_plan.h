// How the tensor-core projections cut their work.  Plain C++ on the host side (no CUDA header), so that a CPU test can ask
// for the plan of any shape and check what the kernels rely on.
#pragma once
#include <stddef.h>

#include <algorithm>

#ifdef __CUDACC__
#define TABED_HD __host__ __device__
#else
#define TABED_HD
#endif

namespace tabed {

constexpr int kTcM = 128;          // weight rows per tile (MMA M)
constexpr int kTcKC = 128;         // input columns per pipeline stage
constexpr int kTcMaxN = 256;       // slots per launch (MMA N is their count rounded up to 16)

// Canonical K-major no-swizzle operand block of `rows` rows x kTcKC columns (bf16):
// element (r, k) at ((k/8) * (rows/8) + r/8) * 128 + (r%8) * 16 + (k%8) * 2 bytes.
TABED_HD inline size_t tc_block_bytes(int rows) { return (size_t)rows * kTcKC * 2; }

// MMAs of 16 columns in a stage of `kc` columns that starts at column k0 of K.  The products stop there: in the activations'
// blocks nobody writes the columns beyond K (to the next 16), and since the buffer is shared by layouts with different
// n_pad, another slot's value may lie in them - one that is not finite would turn its zero weight into a NaN of this slot.
TABED_HD inline int tc_k_steps(int K, int k0, int kc) {
  const int left = (K - k0 + 15) / 16;
  return left < kc / 16 ? left : kc / 16;
}

// Columns of tensor memory that the accumulator of n_pad slots takes (powers of two from 32 on).
TABED_HD inline int tc_tmem_cols(int n_pad) { return n_pad <= 32 ? 32 : (n_pad <= 64 ? 64 : (n_pad <= 128 ? 128 : 256)); }
// An allocation of tensor memory waits until the SM has the columns, without a limit, and a CTA of a cluster that waits there
// keeps its partners waiting on theirs.  So no SM may ever hold CTAs that want more than its 512 columns together, whichever
// launches they belong to: every CTA takes at least the same share of the SM's 228 KB of shared memory (CTAs of 544
// columns, the next sum, would need 238 KB).  (k_gemm_tc's stages are more than that for every n_pad.)
TABED_HD inline size_t tc_least_smem(int n_pad) { return (size_t)tc_tmem_cols(n_pad) * 448u; }

constexpr int kProjMaxSplit = 8;      // CTAs of a cluster (portable size)
constexpr int kProjMaxStages = 8;
constexpr size_t kProjHalfSmem = 112u * 1024u;     // dynamic shared memory of a CTA that leaves room for a second one on its SM
constexpr size_t kProjMaxSmem = 220u * 1024u;      // ... of one that has the SM to itself

// Bytes of one 128-column block of the operand that the RMSNorm prologue builds: its 8-column groups are 16 bytes further
// apart than in a packed block, so that a warp's stores of one slot (16 groups) fall into different banks.
TABED_HD inline unsigned proj_norm_block_bytes(int n_pad) { return 16u * ((unsigned)n_pad * 16u + 16u); }
// Slots that one CTA of the cluster finishes: they are dealt round-robin.
TABED_HD inline int proj_owned(int n_pad, int ks) { return (n_pad + ks - 1) / ks; }

// A layer projection's cut into slot tiles and K splits: a cluster of ks CTAs per (128 output rows, n_pad slots), cps chunks of
// the input dimension each.
struct ProjPlan {
  int n_pad, n_tiles, ks, cps, n_stages;
  bool norm;               // the RMSNorm is taken in the kernel's prologue
  unsigned recv_off;       // offset of the receive buffer (slabs are pushed), or 0 (one split, or slabs are pulled)
  size_t smem;
  float us;                // what the plan is expected to cost
};

// The plan for n_slots slots; fit_of[ks]: clusters of ks CTAs that the device keeps resident at once, one CTA per SM.  What a
// choice costs, in us, as measured on the kernel's own time line (18 - 1024 slots, 768 - 4864 columns): 2 us whatever it does;
// its operands, which a CTA draws from L2 at 75 KB/us alone (60 with a ring of two stages, which does not cover the trip) and
// all of them together at 6.5 MB/us; 0.25 for every 8 slots of the epilogue; the exchange between the CTAs of a cluster 1 us,
// and 0.02 per slot more where the slabs are pulled for lack of a receive buffer; a normalising prologue 1.2 us and 0.02 per
// slot and 128 columns, against 3 us for a launch that packs the operand; a wave that is not full costs a wave; 0.5 us less
// where half of the shared memory is left for the next kernel's start.  All plans of 12 drafters of 256 - 1024 columns were timed
// at 3 - 96 rows: nine launches in ten are within 1 us of their best; the worst are down projections of 768 - 1024 columns with
// two stages in half of the memory (1.5 - 2.7 us slower than three in all of it) and gate/up at 832 columns (2.3 us).
inline ProjPlan plan_proj(int m_tiles, int k_chunks, int n_slots, bool can_norm, const int* fit_of) {
  ProjPlan best{};
  best.us = 1e30f;
  int last_pad = 0;
  for (int tiles = (n_slots + kTcMaxN - 1) / kTcMaxN; tiles <= std::max(1, n_slots / 32); ++tiles) {
    const int n_pad = ((n_slots + tiles - 1) / tiles + 15) / 16 * 16;
    if (n_pad == last_pad) continue;
    last_pad = n_pad;
    const int n_tiles = (n_slots + n_pad - 1) / n_pad, units = m_tiles * n_tiles;
    const size_t a = tc_block_bytes(kTcM), b = tc_block_bytes(n_pad), bn = proj_norm_block_bytes(n_pad), slab = (size_t)n_pad * kTcM * sizeof(float);
    for (int want = 1; want <= std::min(kProjMaxSplit, k_chunks); ++want) {
      const int cps = (k_chunks + want - 1) / want, ks = (k_chunks + cps - 1) / cps;
      if (ks != want) continue;
      const size_t recv = ks > 1 ? (size_t)ks * proj_owned(n_pad, ks) * kTcM * sizeof(float) : 0;
      const int deep = std::min(cps, kProjMaxStages), least = std::min(2, deep);
      for (int norm = 0; norm <= (can_norm ? 1 : 0); ++norm) {
        const size_t fixed = norm ? (size_t)cps * bn : 0, per_stage = norm ? a : a + b;
        for (int half = 0; half < 2; ++half) {
          const size_t budget = half ? kProjHalfSmem : kProjMaxSmem;
          // slabs are pushed where the receive buffer fits beside the operands, else pulled
          const size_t extra = recv && fixed + recv + least * per_stage <= budget ? recv : 0;
          if (std::max(fixed + extra + least * per_stage, extra ? 0 : slab) > budget) continue;
          ProjPlan p{};
          p.n_pad = n_pad; p.n_tiles = n_tiles; p.ks = ks; p.cps = cps; p.norm = norm != 0;
          p.n_stages = (int)std::min<size_t>(deep, (budget - fixed - extra) / per_stage);
          const size_t operands = fixed + p.n_stages * per_stage;
          p.recv_off = extra ? (unsigned)operands : 0u;
          p.smem = std::max(std::max(operands + extra, extra ? 0 : slab), tc_least_smem(n_pad));
          const int fit = std::max(1, fit_of[ks] * (p.smem <= kProjHalfSmem ? 2 : 1)) * ks, ctas = units * ks;
          const float waves = (float)((ctas + fit - 1) / fit);
          const float rate = std::min(p.n_stages >= std::min(deep, 3) ? 75.0f : 60.0f, 6500.0f / (float)std::min(ctas, fit));       // KB per us and CTA
          p.us = waves * ((float)(cps * (a + b)) / 1024.0f / rate + 2.0f + 0.25f * (float)((proj_owned(n_pad, ks) + 7) / 8) + (ks > 1 ? 1.0f : 0.0f) +
                          (ks > 1 && !extra ? 0.02f * (float)n_pad : 0.0f) + (norm ? 1.2f + 0.02f * (float)(std::min(n_pad, n_slots) * cps) : 0.0f)) +
                 (can_norm && !norm ? 3.0f : 0.0f) - (p.smem <= kProjHalfSmem ? 0.5f : 0.0f);      // (room for the next kernel's start)
          if (p.us < best.us) best = p;
        }
      }
    }
  }
  return best;                                                 // (256 slots in one CTA: two stages are 192 KB - always found)
}

}  // namespace tabed
