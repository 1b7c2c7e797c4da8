// The layer projections of the tensor-core path, each ONE launch with everything around the product in it:
//
//   QKV     : RMSNorm of the residual rows -> product -> RoPE, q stored, k and v appended to the caches
//   O, down : product -> residual add, and the row's partial sums of squares for the next RMSNorm
//   gate/up : RMSNorm -> product -> SiLU(gate) * up, rounded, in the operand layout of the down projection
//
// out[slot][o] = sum_k W[o][k] act[slot][k] with D[128 weight rows][N slots] in tensor memory (tcgen05.mma kind::f16,
// bf16 inputs, fp32 accumulate), as in k_gemm_tc.  With 16 - 256 slots a launch reads a few MB and takes a few
// microseconds whatever it does: the layer is bound by its CHAIN of launches and by the trips to L2 between them.
// Hence:
//   * split-K over the CTAs of a CLUSTER: the slabs meet in distributed shared memory and are added there in
//     split order (deterministic), so no slab goes through L2 and no further kernel has to sum them;
//   * after the exchange a warp holds 128 output rows of one slot (4 per lane), which is the layout that the rotation
//     (partner rows are hd/8 lanes away), the gated product (tiles of 64 gate + 64 up rows: partner 16 lanes away), the
//     residual add and the sum of squares need: they are the epilogue instead of launches of their own;
//   * RMSNorm is the prologue: the producer leaves one partial sum of squares per (128-row tile, slot), the consumer adds
//     the few of them, scales, rounds and writes its own columns of the operand straight into shared memory;
//   * the weights of the first stages are requested before the wait on the kernel before (they depend on nothing).
// 9 launches a layer became 5 (one of them the attention): a layer of 768 columns and 18 rows 49.6 -> 40.9 us, 96 rows 78.6 ->
// 69.2, of 256 columns and 39 rows 32.2 -> 30.5.  What a launch's parts cost stands at plan_proj.
// Every wait is bounded; on a timeout the CTA sets an error bit, lets its copies land, frees TMEM and leaves.
#pragma once
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_tc.cuh"

namespace tabed {

enum ProjEpi { PROJ_QKV = 0, PROJ_RESID = 1, PROJ_SWIGLU = 2, PROJ_ANY = 3 };

struct ProjArgs {
  int epi;                            // ProjEpi
  const unsigned char* a_packed;      // weights [m_tiles][k_chunks] blocks of 128 rows
  int K, k_chunks, ks, cps;           // input columns; cluster of ks CTAs; CTA r covers chunks [r * cps, min((r + 1) * cps, k_chunks))
  int n_stages;                       // stages of the weight ring
  unsigned recv_off;                  // > 0: offset of the receive buffer for the other CTAs' slabs (they push); 0: slabs are pulled
  const SlotDesc* slots;
  int n_slots, n_pad;                 // tiles of n_pad slots
  // act operand: packed blocks, or (x != null) the residual rows with their RMSNorm still to be taken
  const unsigned char* b_packed;
  const float* x; int d;
  const float* ss_in; int n_ss;       // partial sums of squares [slot][n_ss], n_ss a multiple of 4 (unused ones are zero)
  const __nv_bfloat16* gain; float eps;
  // epilogues
  int rows;                           // output rows (QKV: (H + 2 Hkv) hd; RESID: d)
  float* x_out; float* ss_out;        // RESID: residual [slot][rows], partial sums of squares [slot][n_ss] (entry m_tile)
  float* qkv;                         // QKV: [slot][rows], the q part is written
  const float *rope_cos, *rope_sin;
  __nv_bfloat16 *kc, *vc;
  int H, Hkv, hd, layer, L, cap;
  unsigned char* act_out; int act_npad, act_chunks;       // SWIGLU: operand blocks of the down projection (its tiles, its k_chunks)
  int* err;
};

__device__ __forceinline__ float proj_rms_scale(const float* __restrict__ ss_row, int n_ss, int d, float eps) {
  float ss = 0.0f;
#pragma unroll 1
  for (int j = 0; j < n_ss; j += 8) {                          // two loads in flight, fixed order of addition
    const float4 a = *reinterpret_cast<const float4*>(ss_row + j);
    const float4 b = j + 4 < n_ss ? *reinterpret_cast<const float4*>(ss_row + j + 4) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    ss += ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w));
  }
  return 1.0f / sqrtf(ss / (float)d + eps);
}

// grid (m_tiles * ks, slot tiles) in clusters of ks, block 256.  Dynamic shared memory: the weight ring, the act blocks
// (packed: one per stage; RMSNorm: all cps of them) and the receive buffer [ks][owned slots][128] fp32; without room for
// that (recv_off = 0) a CTA leaves its slab [n_pad][128] over the operands and the others read it from there.
// The code runs once per launch, so what it costs is trips to L2 and instruction fetch: loads that do not depend on one
// another are issued together, loops stay loops, and the three epilogues are branches of ONE kernel (PROJ_ANY): its code is
// still in the instruction caches from the launch before, which three instantiations pushed out for one another (a layer of
// 256 columns and 39 rows 35.2 -> 30.5 us, of 768 columns and 18 rows 45.8 -> 40.9).  Long prompts run the code often enough
// to gain from instantiations without the branches (step_plan).
template <int EPI>
__global__ void __launch_bounds__(kTcThreads, 2) k_proj_tc(const ProjArgs P) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(128) unsigned char pj_smem[];
  __shared__ uint64_t s_full[kProjMaxStages], s_empty[kProjMaxStages], s_done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_bad;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int epi = EPI == PROJ_ANY ? P.epi : EPI, split = (int)cluster.block_rank(), m_tile = blockIdx.x / P.ks;
  const int slot0 = blockIdx.y * P.n_pad, n_here = min(P.n_pad, P.n_slots - slot0);
  const int c_lo = split * P.cps, c_hi = min(c_lo + P.cps, P.k_chunks), n_ch = c_hi - c_lo;   // (the host leaves no split empty)
  const int n_stages = P.n_stages, last_steps = tc_k_steps(P.K, (c_hi - 1) * kTcKC, kTcKC);
  const unsigned a_bytes = (unsigned)tc_block_bytes(kTcM), b_bytes = P.x ? proj_norm_block_bytes(P.n_pad) : (unsigned)tc_block_bytes(P.n_pad);
  const uint32_t tmem_cols = (uint32_t)tc_tmem_cols(P.n_pad);
  unsigned char* a_ring = pj_smem;
  unsigned char* b_area = pj_smem + (size_t)n_stages * a_bytes;
  const bool push = P.recv_off != 0;
  if (tid == 0) {
    for (int s = 0; s < n_stages; ++s) { mbar_init(&s_full[s], 1); mbar_init(&s_empty[s], 1); }
    mbar_init(&s_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_bad = 0;
  }
  if (warp == 0) {
    __syncwarp();
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
  const unsigned char* a_src = P.a_packed + ((size_t)m_tile * P.k_chunks + c_lo) * a_bytes;
  const unsigned char* b_src = P.x ? nullptr : P.b_packed + ((size_t)blockIdx.y * P.k_chunks + c_lo) * b_bytes;
  const int pre = n_ch < n_stages ? n_ch : n_stages;
  // weights first: announced without an arrival, so that a stage cannot complete before the arrival that follows below
  if (tid == 0) {
    for (int c = 0; c < pre; ++c) {
      asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_full[c])), "r"(a_bytes) : "memory");
      bulk_g2s(a_ring + (size_t)c * a_bytes, a_src + (size_t)c * a_bytes, a_bytes, &s_full[c]);
    }
  }
  __syncwarp();
  if (push) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // (waited for before the slabs are pushed)
  pdl_wait();
  if (gridDim.y > 1) {
    // several slot tiles (the second half of a round's first step may be idle): a tile that nobody needs lets its copies
    // land, gives the tensor memory back and leaves - the same decision in every CTA of the cluster
    int any = 0;
    for (int s = tid; s < n_here; s += kTcThreads) any |= P.slots[slot0 + s].active;
    if (!__syncthreads_or(any)) {
      if (tid == 0) {
        for (int c = 0; c < pre; ++c) {
          mbar_expect_tx(&s_full[c], 0u);
          unsigned spins = 0;
          while (!mbar_try_wait(&s_full[c], 0) && ++spins < (1u << 20)) __nanosleep(32);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
      if (push) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
      return;
    }
  }
  if (epi != PROJ_RESID && P.x) {
    // RMSNorm prologue.  Warp w takes slots w, w + 8, ...; a unit is one slot's 128 columns of a chunk = one warp-wide
    // 512-byte load (4 columns per lane), eight units and the slots' sums of squares in flight together.
    float scale = 0.0f;                                        // lane i: slot warp + 8 i
    const int n_i = (n_here - warp + 7) >> 3, units = n_i * n_ch;
    const float* xw = P.x + (size_t)(slot0 + warp) * P.d + lane * 4;
    unsigned char* dw = b_area + (size_t)(lane >> 1) * ((unsigned)P.n_pad * 16u + 16u) + warp * 16 + (lane & 1) * 8;
    int i = 0, ch = 0;                                         // the unit: slot warp + 8 i, chunk ch
#pragma unroll 1
    for (int u0 = 0; u0 < units; u0 += 8) {
      float4 xv[8];
      uint2 gw[8];
      int at[8];                                               // i | ch << 8
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k0 = (c_lo + ch) * kTcKC;
        const bool in = u0 + j < units && k0 + lane * 4 < P.d;             // columns beyond d are zero
        at[j] = i | (ch << 8);
        xv[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f); gw[j] = make_uint2(0u, 0u);
        if (in) {
          xv[j] = *reinterpret_cast<const float4*>(xw + (size_t)(8 * i) * P.d + k0);
          gw[j] = __ldg(reinterpret_cast<const uint2*>(P.gain + k0 + lane * 4));
        }
        if (++i == n_i) { i = 0; ++ch; }
      }
      if (u0 == 0 && lane < n_i) scale = proj_rms_scale(P.ss_in + (size_t)(slot0 + warp + 8 * lane) * P.n_ss, P.n_ss, P.d, P.eps);
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int ij = at[j] & 255;
        const float sc = __shfl_sync(0xffffffffu, scale, ij);
        const float4 g = bf16x4_to_float4(gw[j]);
        if (u0 + j < units)
          *reinterpret_cast<uint2*>(dw + (size_t)(at[j] >> 8) * b_bytes + ij * 128) =
              make_uint2(pack_bf16(xv[j].x * sc * g.x, xv[j].y * sc * g.y), pack_bf16(xv[j].z * sc * g.z, xv[j].w * sc * g.w));
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // written by threads, read by the tensor core
    __syncthreads();
  }
  if (tid == 0) {
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.n_pad >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
    bool ok = true;
    for (int c = 0; c < pre; ++c) {
      mbar_expect_tx(&s_full[c], P.x ? 0u : b_bytes);
      if (!P.x) bulk_g2s(b_area + (size_t)c * b_bytes, b_src + (size_t)c * b_bytes, b_bytes, &s_full[c]);
    }
    int issued = pre;
#pragma unroll 1
    for (int c = 0; c < n_ch; ++c) {
      const int s = c % n_stages;
      ok = tc_wait(&s_full[s], (unsigned)(c / n_stages) & 1u, P.err);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a_lbo = (kTcM / 8) * 128, b_lbo = (uint32_t)P.n_pad * 16u + (P.x ? 16u : 0u);
      uint64_t da = tc_smem_desc(smem_u32(a_ring + (size_t)s * a_bytes), a_lbo, 128u);
      uint64_t db = tc_smem_desc(smem_u32(b_area + (size_t)(P.x ? c : s) * b_bytes), b_lbo, 128u);
      const int steps = c == n_ch - 1 ? last_steps : kTcKC / 16;
#pragma unroll 1
      for (int j = 0; j < steps; ++j) {
        const uint32_t acc = (c > 0 || j > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
            ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
        da += (2u * a_lbo) >> 4; db += (2u * b_lbo) >> 4;      // (the start address field stays below 2^14)
      }
      if (issued < n_ch) {
        // the stage may be refilled once these MMAs have read it
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&s_empty[s])) : "memory");
        ok = tc_wait(&s_empty[s], (unsigned)(c / n_stages) & 1u, P.err);
        if (!ok) break;
        mbar_expect_tx(&s_full[s], a_bytes + (P.x ? 0u : b_bytes));
        bulk_g2s(a_ring + (size_t)s * a_bytes, a_src + (size_t)issued * a_bytes, a_bytes, &s_full[s]);
        if (!P.x) bulk_g2s(b_area + (size_t)s * b_bytes, b_src + (size_t)issued * b_bytes, b_bytes, &s_full[s]);
        ++issued;
      }
    }
    if (ok) asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&s_done)) : "memory");
    else {
      *(volatile int*)&s_bad = 1;
      // let the copies in flight land before the shared memory is reused
      for (int s = 0; s < n_stages; ++s) {
        unsigned spins = 0;
        while (!mbar_try_wait(&s_full[s], 0) && !mbar_try_wait(&s_full[s], 1) && ++spins < (1u << 16)) __nanosleep(64);
      }
    }
  }
  __syncwarp();
  // What the epilogue of the warp's first slots reads besides the product is requested before the wait for the product.
  const int o = m_tile * kTcM + lane * 4;
  const int half = P.hd >> 1, head = epi == PROJ_QKV ? o / P.hd : 0, hi = epi == PROJ_QKV ? o - head * P.hd : 0;
  const bool in_rows = epi == PROJ_SWIGLU || o < P.rows;
  // The warp's j-th slot of the tile: slot_of(j) = (8 j + warp) ks + split (slots are dealt to the cluster's CTAs, a CTA's to
  // its warps).  Lane j holds the slot's table entry, so that no further trip to L2 is needed for it.
  auto slot_of = [&](int j) { return (j * 8 + warp) * P.ks + split; };
  int4 sd = make_int4(0, 0, 0, 0);                              // row, pos, active
  if (slot_of(lane) < n_here) sd = *reinterpret_cast<const int4*>(P.slots + slot0 + slot_of(lane));
  constexpr int kBatch = 2;                                     // slots finished together
  float4 e0[kBatch], e1[kBatch];
  auto epi_load = [&](int j0) {
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      e0[q] = e1[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (epi == PROJ_SWIGLU) continue;
      const int sl = slot_of(j0 + q), pos = __shfl_sync(0xffffffffu, sd.y, j0 + q);
      if (sl >= n_here || !in_rows) continue;
      if (epi == PROJ_RESID) e0[q] = *reinterpret_cast<const float4*>(P.x_out + (size_t)(slot0 + sl) * P.rows + o);
      if (epi == PROJ_QKV && head < P.H + P.Hkv && pos < P.cap) {      // (a slot past the capacity is inactive)
        const size_t at = (size_t)pos * half + (hi < half ? hi : hi - half);
        e0[q] = __ldg(reinterpret_cast<const float4*>(P.rope_cos + at));
        e1[q] = __ldg(reinterpret_cast<const float4*>(P.rope_sin + at));
      }
    }
  };
  epi_load(0);
  bool done_ok = true;
  {
    unsigned spins = 0;
    while (!mbar_try_wait(&s_done, 0)) {
      if (*(volatile int*)&s_bad) { done_ok = false; break; }
      if (++spins > (1u << 21)) { atomicOr(P.err, PERR_COPY); done_ok = false; break; }
      if (spins > 2048) __nanosleep(64);
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (push) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");      // every CTA of the cluster has started
  // accumulator -> [slot][128 rows]: into the receive buffer of the CTA that finishes the slot, or over the own operands
  // (every product has been taken: s_done)
  const int owned = proj_owned(P.n_pad, P.ks);
  float* red = reinterpret_cast<float*>(pj_smem + P.recv_off);
  if (done_ok) {
    const int lq = warp & 3;                                        // the warp's quarter of the 128 accumulator lanes
    const int row = lq * 32 + lane;
    const uint32_t t_row = tmem + ((uint32_t)(lq * 32) << 16);
    // warps w and w + 4 share the lanes: odd and even groups of 16 slots
#pragma unroll 1
    for (int c0 = (warp >> 2) * 16; c0 < n_here; c0 += 32) {
      uint32_t v[16];
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                   : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                     "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                   : "r"(t_row + (uint32_t)c0));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (push) {
        int own = c0 % P.ks, li = c0 / P.ks;
        float* mine = red + (size_t)split * owned * kTcM + row;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (c0 + j < n_here) cluster.map_shared_rank(mine, own)[(size_t)li * kTcM] = __uint_as_float(v[j]);
          if (++own == P.ks) { own = 0; ++li; }
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) red[(size_t)(c0 + j) * kTcM + row] = __uint_as_float(v[j]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (P.ks > 1) cluster.sync(); else __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");

  // epilogue: warp = slot, lane = 4 consecutive output rows; kBatch slots at a time without branches between them (a slot is
  // a chain of dependent instructions, and two warps per scheduler do not hide one)
  // SWIGLU: this lane's column pair in the operand blocks of the next projection, whose slot tiles may be cut elsewhere
  unsigned char* act_dst = nullptr;
  size_t act_tile = 0;
  int act_r = 0;
  const float act_inv = epi == PROJ_SWIGLU ? 1.0f / (float)P.act_npad : 0.0f;
  if (epi == PROJ_SWIGLU) {
    const int f = m_tile * (kTcM / 2) + (lane & 15) * 4 + (lane >> 4) * 2, t0 = slot0 / P.act_npad;
    act_tile = (size_t)P.act_chunks * tc_block_bytes(P.act_npad);
    act_r = slot0 - t0 * P.act_npad;
    act_dst = P.act_out + (size_t)t0 * act_tile + (size_t)(f / kTcKC) * tc_block_bytes(P.act_npad) + (size_t)((f % kTcKC) >> 3) * (P.act_npad >> 3) * 128 + (f & 7) * 2;
  }
#pragma unroll 1
  for (int j0 = 0; slot_of(j0) < n_here; j0 += kBatch) {
    if (j0) epi_load(j0);
    float v[kBatch][4];
    bool on[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      on[q] = __shfl_sync(0xffffffffu, sd.z, (j0 + q) & 31) != 0 && slot_of(j0 + q) < n_here;
      v[q][0] = v[q][1] = v[q][2] = v[q][3] = 0.0f;
    }
#pragma unroll
    for (int r = 0; r < kProjMaxSplit; ++r) {
      if (r >= P.ks) break;                                     // (split order)
      const float* pr = (push || P.ks == 1 ? red + (size_t)r * owned * kTcM : cluster.map_shared_rank(red, r)) + lane * 4;
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int at = push ? (j0 + q) * 8 + warp : slot_of(j0 + q);
        if (on[q]) {
          const float4 t = *reinterpret_cast<const float4*>(pr + (size_t)at * kTcM);
          v[q][0] += t.x; v[q][1] += t.y; v[q][2] += t.z; v[q][3] += t.w;
        }
      }
    }
    if (epi == PROJ_RESID) {
      float ss[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        v[q][0] += e0[q].x; v[q][1] += e0[q].y; v[q][2] += e0[q].z; v[q][3] += e0[q].w;
        if (on[q] && in_rows) *reinterpret_cast<float4*>(P.x_out + (size_t)(slot0 + slot_of(j0 + q)) * P.rows + o) = make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
        ss[q] = in_rows ? fmaf(v[q][0], v[q][0], fmaf(v[q][1], v[q][1], fmaf(v[q][2], v[q][2], v[q][3] * v[q][3]))) : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) ss[q] = warp_sum_f32(ss[q]);
#pragma unroll
      for (int q = 0; q < kBatch; ++q)
        if (lane == 0 && on[q]) P.ss_out[(size_t)(slot0 + slot_of(j0 + q)) * P.n_ss + m_tile] = ss[q];
    } else if (epi == PROJ_QKV) {
      // rotation pairs are half a head apart; heads do not straddle tiles (hd divides 128)
      const bool rot = head < P.H + P.Hkv;
      const float sgn = hi < half ? -1.0f : 1.0f;
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        float w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = __shfl_xor_sync(0xffffffffu, v[q][j], P.hd >> 3);
        const int row = __shfl_sync(0xffffffffu, sd.x, (j0 + q) & 31), pos = __shfl_sync(0xffffffffu, sd.y, (j0 + q) & 31);
        if (rot) {
          v[q][0] = v[q][0] * e0[q].x + sgn * w[0] * e1[q].x; v[q][1] = v[q][1] * e0[q].y + sgn * w[1] * e1[q].y;
          v[q][2] = v[q][2] * e0[q].z + sgn * w[2] * e1[q].z; v[q][3] = v[q][3] * e0[q].w + sgn * w[3] * e1[q].w;
        }
        if (!on[q] || !in_rows) continue;
        if (head < P.H) {
          *reinterpret_cast<float4*>(P.qkv + (size_t)(slot0 + slot_of(j0 + q)) * P.rows + o) =
              make_float4(round_bf16(v[q][0]), round_bf16(v[q][1]), round_bf16(v[q][2]), round_bf16(v[q][3]));
        } else {
          const int g = head - P.H - (rot ? 0 : P.Hkv);
          __nv_bfloat16* dst = (rot ? P.kc : P.vc) + ((((size_t)row * P.L + P.layer) * P.Hkv + g) * P.cap + pos) * P.hd + hi;
          *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(v[q][0], v[q][1]), pack_bf16(v[q][2], v[q][3]));
        }
      }
    } else {
      // lanes 0 - 15 hold the gate of 4 columns, lanes 16 - 31 the up of the same columns (columns beyond d_ffn are zero:
      // zero weights); an exchange of two values each leaves every lane with gate and up of 2 columns
      const bool low = lane < 16;
      float m[kBatch][2];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const float a = __shfl_xor_sync(0xffffffffu, low ? v[q][2] : v[q][0], 16), b = __shfl_xor_sync(0xffffffffu, low ? v[q][3] : v[q][1], 16);
        const float g0 = low ? v[q][0] : a, g1 = low ? v[q][1] : b, u0 = low ? a : v[q][2], u1 = low ? b : v[q][3];
        m[q][0] = g0 / (1.0f + expf(-g0)) * u0; m[q][1] = g1 / (1.0f + expf(-g1)) * u1;
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int r = act_r + slot_of(j0 + q), t = (int)(((float)r + 0.5f) * act_inv), at = r - t * P.act_npad;      // (r < 1024: exact)
        if (on[q]) *reinterpret_cast<uint32_t*>(act_dst + (size_t)t * act_tile + (at >> 3) * 128 + (at & 7) * 16) = pack_bf16(m[q][0], m[q][1]);
      }
    }
  }
  if (P.ks > 1 && !push) cluster.sync();                        // a CTA's slab stays until every CTA has read it
}

// RMSNorm of the residual rows into operand blocks (tc_act_offset): for the LM head, and for a projection whose operand is
// packed once instead of normalised by every CTA (plan_proj).  grid (n), block 128.
// src_slot (optional) maps row r to the slot whose residual it reads (LM head: the last slot of a row).
struct PrepRowArgs {
  const float* x; int d;                 // residual stream [slot][d]
  const float* ss; int n_ss;             // partial sums of squares of the slots [slot][n_ss]
  const int* src_slot;                   // or null
  const SlotDesc* slots;                 // activity of the slots (null: all active)
  const __nv_bfloat16* gain; float eps;
  int n_pad, k_chunks;
  unsigned char* dst;
};
__global__ void __launch_bounds__(128) k_prep_row(const PrepRowArgs P) {
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.x;
  const int s = P.src_slot ? P.src_slot[r] : r;
  if (P.slots && !P.slots[s].active) return;
  const float sc = proj_rms_scale(P.ss + (size_t)s * P.n_ss, P.n_ss, P.d, P.eps);
  const float* xr = P.x + (size_t)s * P.d;
  for (int k = threadIdx.x * 8; k < P.d; k += 128 * 8) {
    const float4 a = *reinterpret_cast<const float4*>(xr + k), b = *reinterpret_cast<const float4*>(xr + k + 4);
    float g[8];
    Elem<__nv_bfloat16>::unpack(__ldg(reinterpret_cast<const uint4*>(P.gain + k)), g);
    uint4 v;
    v.x = pack_bf16(a.x * sc * g[0], a.y * sc * g[1]); v.y = pack_bf16(a.z * sc * g[2], a.w * sc * g[3]);
    v.z = pack_bf16(b.x * sc * g[4], b.y * sc * g[5]); v.w = pack_bf16(b.z * sc * g[6], b.w * sc * g[7]);
    *reinterpret_cast<uint4*>(P.dst + tc_act_offset(r, k, P.n_pad, P.k_chunks)) = v;
  }
}

}  // namespace tabed
