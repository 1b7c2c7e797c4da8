// Causal attention of a prompt's positions (all of one cache row) over that row's bf16 cache, K and V of the positions
// themselves already appended: the chunk of positions that one pass of the tensor-core projections feeds.
//
// A CTA takes 16 QW positions of one query head and walks the cache in tiles of T positions (cp.async, two buffers, 16-byte
// pieces XOR-swizzled so that every ldmatrix is conflict-free); a warp owns 16 positions.  The tiles are dealt to NG groups of
// QW warps (a tile's chain of products and softmax is 1.8 us for a lone group); their states meet in shared memory at the
// end.  scores = Q K^T and out += P V on mma.sync m16n8k16 (bf16 x bf16 -> fp32): q is a bf16 value already, the softmax
// weights are split into a bf16 head and a bf16 remainder (two products), so products are exact to ~2^-17 and sums are fp32,
// as in the decode kernels.  A prompt of 576 positions and 12 heads is 2 GFLOP against 0.9 MB of cache per head: neither
// roofline is near, what counts is that the K, V tiles are shared by the CTA's positions (the decode kernel reads the cache
// once per position).  A launch for 128 positions of a 768-wide layer takes 12.8 us by itself.  The longest CTAs (last positions)
// start first.  Short prompts would leave most SMs idle with 64 positions a CTA (128 positions x 12 heads: 24 CTAs, whose
// products then wait for one another on the tensor pipe): where these CTAs fill at most half of the SMs, 32 positions and
// tiles of 32 in eight groups are taken.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "attn_tc.cuh"

namespace tabed {

// groups of a CTA: 16 warps in all, 8 for 128-wide heads
template <int HD, int QW> __host__ __device__ constexpr int prompt_attn_groups() { return (HD <= 64 ? 16 : 8) / QW; }
// two buffers of K and V per group
template <int HD, int QW, int T> __host__ __device__ constexpr size_t prompt_attn_smem() { return (size_t)prompt_attn_groups<HD, QW>() * 4 * T * HD * 2; }

struct PromptAttnArgs {
  const float* qkv; int qkv_w;                 // [n][qkv_w] rotated q
  const SlotDesc* slots; int n;                // slot i: position slots[0].pos + i of row slots[0].row
  const __nv_bfloat16 *kc, *vc;
  int H, Hkv, layer, L, cap;
  float scale;
  unsigned char* act_out; int act_npad, act_chunks;      // the output as the next projection's operand blocks
};

// 16 bytes, of which the first n (0 or 16) come from src and the rest are zero
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t n) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// grid (tiles of 16 QW positions, H)
template <int HD, int QW, int T>
__global__ void __launch_bounds__(QW * 32 * prompt_attn_groups<HD, QW>(), 1) k_prompt_attn(const PromptAttnArgs A) {
  extern __shared__ __align__(128) unsigned char pa_smem[];
  constexpr int NG = prompt_attn_groups<HD, QW>(), kPaQ = 16 * QW, kPaT = T, kPaGroup = 32 * QW;
  __shared__ float s_ml[NG][QW][2][16];         // (max, sum) of every position by group
  constexpr int PIECES = HD / 8;               // 16-byte pieces of a cache row
  constexpr int KK = HD / 16, NT = HD / 8;
  constexpr unsigned FULL = 0xffffffffu;
  const int grp = threadIdx.x / kPaGroup, tid = threadIdx.x % kPaGroup, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3, r8 = lane & 7, ti = lane >> 3;
  pdl_trigger();
  pdl_wait();
  const SlotDesc first = A.slots[0];
  const int q0 = (gridDim.x - 1 - blockIdx.x) * kPaQ, head = blockIdx.y, hk = head / (A.H / A.Hkv);
  const int last = min(first.pos + min(q0 + kPaQ, A.n) - 1, A.cap - 1), n_tiles = last / kPaT + 1;      // last cache position needed
  const size_t base = ((((size_t)first.row * A.L + A.layer) * A.Hkv + hk) * A.cap) * HD;
  const __nv_bfloat16 *kb = A.kc + base, *vb = A.vc + base;
  constexpr uint32_t TILE = kPaT * HD * 2;
  const uint32_t s0 = smem_u32(pa_smem) + grp * 4 * TILE;
  // piece c of row r sits at r * HD * 2 + ((c ^ (r & 7)) * 16), for 32-wide heads (4 pieces) with the row pair's bits
  auto piece = [](int r, int c) { return (uint32_t)(r * HD * 2 + ((HD >= 64 ? (c ^ (r & 7)) : (c ^ ((r >> 1) & 3))) << 4)); };
  auto fetch = [&](int t, int buf) {
    const uint32_t kd = s0 + buf * 2 * TILE, vd = kd + TILE;
#pragma unroll 4
    for (int i = tid; i < kPaT * PIECES; i += kPaGroup) {
      const int r = i / PIECES, c = i - r * PIECES;
      // rows past the last position are masked, but a weight of 0 does not cancel what an earlier, longer prompt of the row
      // may have left there if that is not finite: they read as zeros
      const int p = min(t * kPaT + r, last);
      const uint32_t n = t * kPaT + r <= last ? 16u : 0u;
      cp_async16(kd + piece(r, c), kb + (size_t)p * HD + c * 8, n);
      cp_async16(vd + piece(r, c), vb + (size_t)p * HD + c * 8, n);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (grp < n_tiles) fetch(grp, 0);
  // q fragments of the warp's 16 positions (rows past the last one repeat it)
  uint32_t qa[KK][4];
  const int qi0 = min(q0 + warp * 16 + g, A.n - 1), qi1 = min(q0 + warp * 16 + g + 8, A.n - 1);
  {
    const float* r0 = A.qkv + (size_t)qi0 * A.qkv_w + head * HD + 2 * t4;
    const float* r1 = A.qkv + (size_t)qi1 * A.qkv_w + head * HD + 2 * t4;
#pragma unroll
    for (int k = 0; k < KK; ++k) {
      const float2 a = *reinterpret_cast<const float2*>(r0 + k * 16), b = *reinterpret_cast<const float2*>(r1 + k * 16);
      const float2 c = *reinterpret_cast<const float2*>(r0 + k * 16 + 8), d = *reinterpret_cast<const float2*>(r1 + k * 16 + 8);
      qa[k][0] = pack_bf16(a.x, a.y); qa[k][1] = pack_bf16(b.x, b.y); qa[k][2] = pack_bf16(c.x, c.y); qa[k][3] = pack_bf16(d.x, d.y);
    }
  }
  float o[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.0f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.0f, 0.0f};       // positions g, g + 8; base-2 units
  const float scale2 = A.scale * 1.4426950408889634f;
  const int p0 = first.pos + q0 + warp * 16 + g, p1 = p0 + 8;             // the last cache position that each row sees
  int buf = 0;
#pragma unroll 1
  for (int t = grp; t < n_tiles; t += NG, buf ^= 1) {
    if (t + NG < n_tiles) {
      fetch(t + NG, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kPaGroup) : "memory");
    const uint32_t ks = s0 + buf * 2 * TILE, vs = ks + TILE;
    float sc[kPaT / 8][4];
#pragma unroll
    for (int j = 0; j < kPaT / 8; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.0f;
#pragma unroll
    for (int k = 0; k < KK; ++k)
#pragma unroll
      for (int j = 0; j < kPaT / 16; ++j) {
        uint32_t b[4];
        ldsm_x4(b, ks + piece(j * 16 + (ti >> 1) * 8 + r8, 2 * k + (ti & 1)));
        const uint32_t b0[2] = {b[0], b[1]}, b1[2] = {b[2], b[3]};
        mma_bf16(sc[2 * j], qa[k], b0);
        mma_bf16(sc[2 * j + 1], qa[k], b1);
      }
    const bool edge = t * kPaT + kPaT - 1 > first.pos + q0 + warp * 16;      // some row of the warp does not see the whole tile
    float mx0 = -INFINITY, mx1 = -INFINITY;
    const float m_old[2] = {m_run[0], m_run[1]};
#pragma unroll
    for (int j = 0; j < kPaT / 8; ++j) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        sc[j][e] *= scale2;
        if (edge && t * kPaT + j * 8 + 2 * t4 + (e & 1) > ((e >> 1) ? p1 : p0)) sc[j][e] = -INFINITY;
      }
      mx0 = fmaxf(mx0, fmaxf(sc[j][0], sc[j][1])); mx1 = fmaxf(mx1, fmaxf(sc[j][2], sc[j][3]));
    }
#pragma unroll
    for (int s = 1; s < 4; s <<= 1) {
      mx0 = fmaxf(mx0, __shfl_xor_sync(FULL, mx0, s));
      mx1 = fmaxf(mx1, __shfl_xor_sync(FULL, mx1, s));
    }
    m_run[0] = fmaxf(m_run[0], mx0); m_run[1] = fmaxf(m_run[1], mx1);
    // (a row that has seen no position of this group's tiles yet: every weight is 0)
    const float n0 = m_run[0] > -INFINITY ? m_run[0] : 0.0f, n1 = m_run[1] > -INFINITY ? m_run[1] : 0.0f;
    const float f0 = ex2_approx(m_old[0] - n0), f1 = ex2_approx(m_old[1] - n1);
    l_run[0] *= f0; l_run[1] *= f1;
#pragma unroll
    for (int j = 0; j < NT; ++j) { o[j][0] *= f0; o[j][1] *= f0; o[j][2] *= f1; o[j][3] *= f1; }
#pragma unroll
    for (int j = 0; j < kPaT / 8; ++j) {
      sc[j][0] = ex2_approx(sc[j][0] - n0); sc[j][1] = ex2_approx(sc[j][1] - n0);
      sc[j][2] = ex2_approx(sc[j][2] - n1); sc[j][3] = ex2_approx(sc[j][3] - n1);
      l_run[0] += sc[j][0] + sc[j][1]; l_run[1] += sc[j][2] + sc[j][3];
    }
#pragma unroll
    for (int k = 0; k < kPaT / 16; ++k) {
      uint32_t ph[4], pl[4];
      split_bf16x2(sc[2 * k][0], sc[2 * k][1], ph[0], pl[0]);
      split_bf16x2(sc[2 * k][2], sc[2 * k][3], ph[1], pl[1]);
      split_bf16x2(sc[2 * k + 1][0], sc[2 * k + 1][1], ph[2], pl[2]);
      split_bf16x2(sc[2 * k + 1][2], sc[2 * k + 1][3], ph[3], pl[3]);
#pragma unroll
      for (int j = 0; j < NT / 2; ++j) {
        uint32_t b[4];
        ldsm_x4_trans(b, vs + piece(k * 16 + (ti & 1) * 8 + r8, 2 * j + (ti >> 1)));
        const uint32_t b0[2] = {b[0], b[1]}, b1[2] = {b[2], b[3]};
        mma_bf16(o[2 * j], ph, b0); mma_bf16(o[2 * j], pl, b0);
        mma_bf16(o[2 * j + 1], ph, b1); mma_bf16(o[2 * j + 1], pl, b1);
      }
    }
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kPaGroup) : "memory");      // the tile's buffer may be refilled
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    l_run[e] += __shfl_xor_sync(FULL, l_run[e], 1);
    l_run[e] += __shfl_xor_sync(FULL, l_run[e], 2);
  }
  // the groups' states meet in the tile buffers: [group][warp][n-tile][lane] accumulators; every group finishes its share
  // of the n-tiles, adding the states in group order
  __syncthreads();
  float4* st = reinterpret_cast<float4*>(pa_smem);
#pragma unroll
  for (int j = 0; j < NT; ++j) st[((grp * QW + warp) * NT + j) * 32 + lane] = make_float4(o[j][0], o[j][1], o[j][2], o[j][3]);
  if (t4 == 0) {
    s_ml[grp][warp][0][g] = m_run[0]; s_ml[grp][warp][0][g + 8] = m_run[1];
    s_ml[grp][warp][1][g] = l_run[0]; s_ml[grp][warp][1][g + 8] = l_run[1];
  }
  __syncthreads();
  float f[2][NG];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float M = -INFINITY, l = 0.0f;
#pragma unroll
    for (int i = 0; i < NG; ++i) M = fmaxf(M, s_ml[i][warp][0][g + 8 * e]);
#pragma unroll
    for (int i = 0; i < NG; ++i) { f[e][i] = ex2_approx(s_ml[i][warp][0][g + 8 * e] - M); l = fmaf(f[e][i], s_ml[i][warp][1][g + 8 * e], l); }
#pragma unroll
    for (int i = 0; i < NG; ++i) f[e][i] /= l;
  }
  const int r0 = q0 + warp * 16 + g, r1 = r0 + 8;
#pragma unroll
  for (int j = grp; j < NT; j += NG) {
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const float4 x = st[((i * QW + warp) * NT + j) * 32 + lane];
      v.x = fmaf(f[0][i], x.x, v.x); v.y = fmaf(f[0][i], x.y, v.y); v.z = fmaf(f[1][i], x.z, v.z); v.w = fmaf(f[1][i], x.w, v.w);
    }
    const int k = head * HD + j * 8 + 2 * t4;
    if (r0 < A.n) *reinterpret_cast<uint32_t*>(A.act_out + tc_act_offset(r0, k, A.act_npad, A.act_chunks) + (k & 7) * 2) = pack_bf16(v.x, v.y);
    if (r1 < A.n) *reinterpret_cast<uint32_t*>(A.act_out + tc_act_offset(r1, k, A.act_npad, A.act_chunks) + (k & 7) * 2) = pack_bf16(v.z, v.w);
  }
}

}  // namespace tabed
