// The plain tensor-core projection: out[slot][o] = sum_k W[o][k] act[slot][k] on the 5th-generation tensor cores, for the LM
// head of the tensor-core path (the layers' projections, with everything around the product, are k_proj_tc) and for
// tabed_debug_gemm_tc.
//
//   D[128 weight rows][N slots] += A[128][16] * B[N][16]^T     (kind::f16, bf16 inputs, fp32 accumulate)
//
// * A work unit is (tile of 128 weight rows, range of input columns).  Units write fp32 partial sums
//   [k-split][slot][row] (the LM head has one split: its logits are stored directly).
// * Operands reach shared memory by bulk asynchronous copies (cp.async.bulk + mbarrier), three stages of
//   128 input columns.  Both operands are stored in global memory already in the tensor core's canonical
//   K-major, no-swizzle layout (8 rows x 16 bytes core matrices), so a stage is two contiguous copies and
//   needs no tensor map: the weights are re-laid once at set-up (k_pack_tc), the activations by the kernel
//   that normalises and rounds them (k_prep_row).
// * One thread issues the copies and the MMAs; tcgen05.commit releases a stage / signals the epilogue;
//   eight warps read the accumulator with tcgen05.ld (warps w and w + 4 own TMEM lanes 32w..32w+31, half of the columns each) and store
//   coalesced rows.  Every wait is bounded; on a timeout the CTA sets an error bit, drains and frees TMEM.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "proj_plan.h"
#include "round_kernel.cuh"   // PTX wrappers: mbarrier, bulk copy

namespace tabed {

constexpr int kTcStages = 3;        // pipeline stages (2 when more than 128 slots share the shared memory)
constexpr int kTcMaxStages = 8;
constexpr int kTcThreads = 256;      // eight warps: warps w and w + 4 read the same 32 accumulator lanes, half of the columns each
constexpr int kPrefillChunk = 1024;       // positions of one row prefilled as slots of one weight pass
__host__ __device__ inline int tc_stages(int n_pad) { return n_pad > 128 ? 2 : kTcStages; }
// The most dynamic shared memory that any launch takes (three stages of 128 slots, or two of 256).  The limit belongs to the
// function, not to a launch: whoever sets it sets this value.
constexpr size_t kTcMaxSmem = 3u * (kTcM + 128u) * kTcKC * 2u + 1024u;

struct TcGemmArgs {
  const unsigned char* a_packed;   // [m_tiles][k_chunks] blocks of 128 rows
  const unsigned char* b_packed;   // [k_chunks] blocks of n_pad rows
  float* partial;                  // [ks] slabs of `slab` floats; slab layout [slot][rows_total], first slot of this launch at +0
  size_t slab;                     // floats between k-split slabs
  int rows_total;                  // output rows of the projection (multiple of 128 after padding in a_packed)
  int rows_valid;                  // rows actually stored
  int n_pad, n_slots;              // MMA N (multiple of 16) / slots stored
  int K, k_chunks;                 // the input dimension, and its chunks of 128 columns
  int ks;                          // k-splits; unit (m_tile, split) covers chunks [split*cps, min((split+1)*cps, k_chunks))
  int cps;                         // chunks per split
  int kc;                          // input columns per pipeline stage: 128 (a whole block) or 64 (half a block: a block's
                                   // 16-byte column groups are its outer index, so half of it is contiguous too)
  int n_stages;                    // pipeline stages, <= kTcMaxStages
  int* err;
};

__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  // shared-memory matrix descriptor: start address, leading (K) and stride (row group) byte offsets in
  // 16-byte units, descriptor version 1 (bits 46-47), no swizzle (bits 61-63 = 0)
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

__device__ __forceinline__ bool tc_wait(uint64_t* bar, unsigned parity, int* err) {
  unsigned spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if (++spins > (1u << 20)) { atomicOr(err, PERR_COPY); return false; }
    if (spins > 2048) __nanosleep(64);
  }
  return true;
}

// grid (m_tiles * ks), block kTcThreads, dynamic shared memory n_stages * (A + B of a stage) + 1 KB
__global__ void __launch_bounds__(kTcThreads, 1) k_gemm_tc(const TcGemmArgs G) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ uint64_t s_full[kTcMaxStages], s_empty[kTcMaxStages], s_done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m_tile = blockIdx.x / G.ks, split = blockIdx.x - m_tile * G.ks;
  // the CTA's range of the input dimension in units of one stage (kc columns); a_bytes, b_bytes = one stage of each operand
  const int per_chunk = kTcKC / G.kc;
  const int c_lo = split * G.cps, c_hi = min(c_lo + G.cps, G.k_chunks), n_ch = (c_hi - c_lo) * per_chunk;
  const size_t a_bytes = tc_block_bytes(kTcM) / per_chunk, b_bytes = tc_block_bytes(G.n_pad) / per_chunk;
  const int n_stages = G.n_stages;
  const uint32_t tmem_cols = (uint32_t)tc_tmem_cols(G.n_pad);

  if (tid == 0) {
    for (int s = 0; s < n_stages; ++s) { mbar_init(&s_full[s], 1); mbar_init(&s_empty[s], 1); }
    mbar_init(&s_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_bad = 0;
  }
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // the next kernel may be scheduled once every CTA of this one holds its tensor memory: a successor that took the
  // columns first would wait for this grid while this grid waits for the columns
  pdl_trigger();
  const uint32_t tmem = s_tmem;
  const unsigned char* a_src = G.a_packed + ((size_t)m_tile * G.k_chunks + c_lo) * tc_block_bytes(kTcM);
  const unsigned char* b_src = G.b_packed + (size_t)c_lo * tc_block_bytes(G.n_pad);
  const int pre = n_ch < n_stages ? n_ch : n_stages;
  // The weights do not depend on the kernels before this one: their first stages are requested before
  // the wait on those kernels (transaction bytes announced without an arrival, so a stage's barrier
  // cannot complete before its activations have been requested too).
  if (tid == 0) {
    for (int c = 0; c < pre; ++c) {
      asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_full[c])), "r"((unsigned)a_bytes) : "memory");
      bulk_g2s(tc_smem + (size_t)c * (a_bytes + b_bytes), a_src + (size_t)c * a_bytes, (unsigned)a_bytes, &s_full[c]);
    }
  }
  pdl_wait();
  if (tid == 0 && n_ch > 0) {
    // instruction descriptor: fp32 accumulator, bf16 x bf16, both operands K-major, N and M
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(G.n_pad >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
    bool ok = true;
    for (int c = 0; c < pre; ++c) {
      mbar_expect_tx(&s_full[c], (unsigned)b_bytes);
      bulk_g2s(tc_smem + (size_t)c * (a_bytes + b_bytes) + a_bytes, b_src + (size_t)c * b_bytes, (unsigned)b_bytes, &s_full[c]);
    }
    int issued = pre;
    for (int c = 0; c < n_ch && ok; ++c) {
      const int s = c % n_stages;
      ok = tc_wait(&s_full[s], (unsigned)(c / n_stages) & 1u, G.err);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a_s = smem_u32(tc_smem + (size_t)s * (a_bytes + b_bytes));
      const uint32_t b_s = a_s + (uint32_t)a_bytes;
      const uint32_t a_lbo = (kTcM / 8) * 128, b_lbo = (uint32_t)(G.n_pad / 8) * 128;
      const int steps = tc_k_steps(G.K, c_lo * kTcKC + c * G.kc, G.kc);
#pragma unroll 1
      for (int j = 0; j < steps; ++j) {
        const uint64_t da = tc_smem_desc(a_s + (uint32_t)j * 2u * a_lbo, a_lbo, 128u);
        const uint64_t db = tc_smem_desc(b_s + (uint32_t)j * 2u * b_lbo, b_lbo, 128u);
        const uint32_t acc = (c > 0 || j > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
            ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
      }
      // the stage may be refilled once these MMAs have read it
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&s_empty[s])) : "memory");
      if (issued < n_ch) {
        ok = tc_wait(&s_empty[s], (unsigned)(c / n_stages) & 1u, G.err);
        if (!ok) break;
        unsigned char* st = tc_smem + (size_t)s * (a_bytes + b_bytes);
        mbar_expect_tx(&s_full[s], (unsigned)(a_bytes + b_bytes));
        bulk_g2s(st, a_src + (size_t)issued * a_bytes, (unsigned)a_bytes, &s_full[s]);
        bulk_g2s(st + a_bytes, b_src + (size_t)issued * b_bytes, (unsigned)b_bytes, &s_full[s]);
        ++issued;
      }
    }
    if (ok) asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&s_done)) : "memory");
    else {
      s_bad = 1;
      // let the copies in flight land before the shared memory is released
      for (int s = 0; s < n_stages; ++s) {
        unsigned spins = 0;
        while (!mbar_try_wait(&s_full[s], 0) && !mbar_try_wait(&s_full[s], 1) && ++spins < (1u << 16)) __nanosleep(64);
      }
    }
  }
  __syncwarp();
  bool done_ok = true;
  if (n_ch > 0) {
    // everybody waits for the accumulator (or for the issuing thread to give up)
    unsigned spins = 0;
    while (!mbar_try_wait(&s_done, 0)) {
      if (*(volatile int*)&s_bad) { done_ok = false; break; }
      if (++spins > (1u << 21)) { atomicOr(G.err, PERR_COPY); done_ok = false; break; }
      if (spins > 2048) __nanosleep(64);
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (done_ok) {
    const int lq = warp & 3;                                        // the warp's quarter of the 128 accumulator lanes
    const int row = m_tile * kTcM + lq * 32 + lane;
    float* out = G.partial + (size_t)split * G.slab + row;
    // the warp's columns: the first or the second half of the groups of 16
    const int n16 = G.n_pad >> 4, c_begin = (warp >> 2) ? ((n16 + 1) >> 1) << 4 : 0, c_end = (warp >> 2) ? G.n_pad : ((n16 + 1) >> 1) << 4;
    // two loads of 16 columns in flight: the next one is requested before the current one is stored
    auto ld16 = [&](uint32_t (&v)[16], int c0) {
      const uint32_t taddr = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)c0;
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                   : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                     "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                   : "r"(taddr));
    };
    auto st16 = [&](const uint32_t (&v)[16], int c0) {
      if (row < G.rows_valid) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c0 + j < G.n_slots) out[(size_t)(c0 + j) * G.rows_total] = __uint_as_float(v[j]);
      }
    };
    if (n_ch > 0 && c_begin < c_end) {
      uint32_t va[16], vb[16];
      ld16(va, c_begin);
#pragma unroll 1
      for (int c0 = c_begin; c0 < c_end; c0 += 32) {
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const bool more = c0 + 16 < c_end;
        if (more) ld16(vb, c0 + 16);
        st16(va, c0);
        if (more) {
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (c0 + 32 < c_end) ld16(va, c0 + 32);
          st16(vb, c0 + 16);
        }
      }
    } else if (n_ch == 0) {
      if (row < G.rows_valid)
        for (int c = c_begin; c < min(c_end, G.n_slots); ++c) out[(size_t)c * G.rows_total] = 0.0f;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
}

// ---- operand packing ------------------------------------------------------------------------------
// Weights [rows][K] (one or two matrices concatenated: rows0 of w0 then rows1 of w1) -> blocks
// [m_tile][k_chunk] in the canonical layout; rows beyond rows0+rows1 and columns beyond K are zero.
// paired: a tile holds 64 rows of w0, then the same 64 rows of w1 (gate and up, for the gated product's epilogue).
// grid (k_chunks, m_tiles), block 256.
__global__ void k_pack_tc(const __nv_bfloat16* __restrict__ w0, int rows0, const __nv_bfloat16* __restrict__ w1, int rows1,
                          const __nv_bfloat16* __restrict__ w2, int rows2, int K, int k_chunks, unsigned char* __restrict__ dst,
                          int paired = 0) {
  const int kc = blockIdx.x, mt = blockIdx.y;
  unsigned char* blk = dst + ((size_t)mt * k_chunks + kc) * tc_block_bytes(kTcM);
  for (int idx = threadIdx.x; idx < kTcM * (kTcKC / 8); idx += blockDim.x) {
    const int r = idx % kTcM, k8 = idx / kTcM;
    int row = mt * kTcM + r;
    const int k = kc * kTcKC + k8 * 8;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    const __nv_bfloat16* base = nullptr;
    if (paired) {
      row = mt * (kTcM / 2) + (r & (kTcM / 2 - 1));
      if (row < rows0) base = r < kTcM / 2 ? w0 : w1;
    } else if (row < rows0) base = w0;
    else if (row < rows0 + rows1) { base = w1; row -= rows0; }
    else if (row < rows0 + rows1 + rows2) { base = w2; row -= rows0 + rows1; }
    if (base && k < K) v = *reinterpret_cast<const uint4*>(base + (size_t)row * K + k);
    *reinterpret_cast<uint4*>(blk + ((size_t)k8 * (kTcM / 8) + (r >> 3)) * 128 + (r & 7) * 16) = v;
  }
}

// Activations fp32 [n][K] (row stride `stride`) -> bf16 blocks [k_chunk] of n_pad rows in the canonical
// layout.  Rows >= n and columns >= K are zero.  grid (k_chunks), block 256.
__global__ void k_prep_act(const float* __restrict__ x, int stride, int n, int n_pad, int K, unsigned char* __restrict__ dst) {
  const int kc = blockIdx.x;
  unsigned char* blk = dst + (size_t)kc * tc_block_bytes(n_pad);
  for (int idx = threadIdx.x; idx < n_pad * (kTcKC / 8); idx += blockDim.x) {
    const int r = idx % n_pad, k8 = idx / n_pad;
    const int k = kc * kTcKC + k8 * 8;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r < n && k < K) {
      const float4 a = *reinterpret_cast<const float4*>(x + (size_t)r * stride + k);
      const float4 b = *reinterpret_cast<const float4*>(x + (size_t)r * stride + k + 4);
      v.x = pack_bf16(a.x, a.y); v.y = pack_bf16(a.z, a.w); v.z = pack_bf16(b.x, b.y); v.w = pack_bf16(b.z, b.w);
    }
    *reinterpret_cast<uint4*>(blk + ((size_t)k8 * (n_pad / 8) + (r >> 3)) * 128 + (r & 7) * 16) = v;
  }
}

}  // namespace tabed
