// Causal attention of passes of 17 tokens and more over a bf16 KV cache (with heads of 64 those that fill blocks of 128
// queries go to attn_mma.cuh, see attn_mma_pays).  The keys and values of the pass are in the cache: the QKV
// contraction put them there and rotated and scaled the queries (rotated = 1, see PairRope), or kv_append_kernel
// did (rotated = 0: the queries are rotated here).
//
// A CTA takes up to 64 consecutive queries of one (series, head), 16 per warp (the M side of mma.sync
// m16n8k16), and streams the keys they may see in tiles of 64 through two shared-memory stages that all its
// warps read.  (Every warp streaming its own keys, as attn_flash_kernel does for single query tiles, brings
// each key in four times and leaves room for eight warps on an SM: 166 us for 64 series x 20 heads x 255
// tokens, 65 us for 16 x 8 x 256 tokens behind 768 to 1000 keys, 44 us for 200 x 16 x 30 tokens; now 122, 52
// and 27 us.)
//   * running softmax per query row in registers, 32 keys at a time, as in attn_flash_body: queries split
//     into bf16 high and low parts, scores in base-2 units, probabilities rounded to bf16 for P V;
//   * warps skip the half tiles behind their last query; only the rows of a half tile that holds a visible
//     key are fetched;
//   * the query blocks with the most keys start first;
//   * a value that a query must not see does not reach it, although an infinity or NaN times its probability of 0 is NaN: a
//     block that ends with such outputs beside finite sums of probabilities goes over its keys again, with these values as
//     0 in the tiles that only some of its queries see, and NaN for the queries that do see them (the look at the outputs:
//     nothing to be seen from 33 tokens on, 0.3 to 0.6 us a launch of 8 to 17 at 18 to 30).
// Bound: latency of a block's first loads and of the mma.sync chains with 16 warps per SM (64 x 20 x 255: tensor pipe
// 31 % busy, issue slots 34 %).
// grid = (heads, B, ceil(q_len / (16 warps))), block = 32 x warps, warps = 2 where q_len <= 32, else 4.
#pragma once
#include "attn_flash.cuh"

namespace tsfm {

template <int DH> struct TilesGeom {
  static constexpr int KEYS = 64, HALF_KEYS = 32, ROW_BYTES = DH * 2;
  static constexpr int TILE_BYTES = KEYS * ROW_BYTES, STAGE_BYTES = 2 * TILE_BYTES, SMEM_BYTES = 2 * STAGE_BYTES;
};

template <int DH>
__global__ void __launch_bounds__(128, DH <= 64 ? 4 : 2)
attn_tiles_kernel(const float *qkv, const bf16 *Kc, const bf16 *Vc, const float2 *__restrict__ rope, PassGeom g, int n_heads,
                  int rotated, bf16 *__restrict__ out) {
  using G = TilesGeom<DH>;
  constexpr int HALF = DH / 2, KS = DH / 16, CPR = DH / 8;
  extern __shared__ __align__(256) unsigned char tiles_smem[];
  __shared__ int bad_row;                                      // first value row of a tile with an infinity or NaN
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(tiles_smem);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const int gr = lane >> 2, q4 = lane & 3, d = n_heads * DH;
  const int h = blockIdx.x, slot = blockIdx.y, qb = (gridDim.z - 1 - blockIdx.z) * n_warps * 16;
  const SlotPos sp = slot_lookup(g, slot);                     // before the dependency wait: see SlotPos
  pdl_sync();                                                  // (the rows of the pass come from the preceding kernel)
  if (sp.dead) return;
  const int p0 = sp.p0;
  const size_t row0 = (size_t)slot * g.q_len;
  const bf16 *Kb = Kc + ((size_t)sp.b * n_heads + h) * g.cap * DH, *Vb = Vc + ((size_t)sp.b * n_heads + h) * g.cap * DH;
  const int jq = qb + w * 16, nq = min(16, g.q_len - jq);      // this warp's queries (nq <= 0: none)
  const int n_keys = p0 + min(qb + n_warps * 16, g.q_len);     // keys the block's last query sees
  const int n_tiles = (n_keys + G::KEYS - 1) / G::KEYS;

  auto issue = [&](int tile) {
    if (tile < n_tiles) {
      const int t0 = tile * G::KEYS, rows = min(G::KEYS, (n_keys - t0 + G::HALF_KEYS - 1) & ~(G::HALF_KEYS - 1));
      const uint32_t kst = ring + (uint32_t)((tile & 1) * G::STAGE_BYTES), vst = kst + G::TILE_BYTES;
      for (int idx = threadIdx.x; idx < rows * CPR; idx += blockDim.x) {
        const int r = idx / CPR, ch = idx % CPR;
        const size_t src = (size_t)min(t0 + r, n_keys - 1) * DH + ch * 8;   // rows past the range repeat its last key (masked below)
        const uint32_t off = (uint32_t)(r * G::ROW_BYTES + flash_swz<DH>(r, ch) * 16);
        flash_cp16(kst + off, Kb + src);
        flash_cp16(vst + off, Vb + src);
      }
    }
    flash_commit();
  };
  issue(0);

  // rotated, scaled queries as A fragments (rows gr and gr + 8), high and low bf16 parts
  uint32_t qhi[KS][4], qlo[KS][4];
  {
    const float sc = rsqrtf((float)DH) * 1.4426950408889634f;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int i = gr + rr * 8;
      const bool live = i < nq;
      const int j = live ? jq + i : 0;
      const float *src = qkv + (row0 + j) * 3 * d + h * DH;
      const float2 *rp = rope + (size_t)(p0 + j) * HALF;
#pragma unroll
      for (int ks = 0; ks < KS / 2; ++ks)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int c = ks * 16 + hh * 8 + q4 * 2;             // first-half dims c, c + 1; partners c + HALF
          const float2 q1 = __ldcg(reinterpret_cast<const float2 *>(src + c));
          const float2 q2 = __ldcg(reinterpret_cast<const float2 *>(src + c + HALF));
          float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);                     // cos0 sin0 cos1 sin1
          if (!rotated) cs = *reinterpret_cast<const float4 *>(rp + c);
          float a0 = (q1.x * cs.x - q2.x * cs.y) * sc, a1 = (q1.y * cs.z - q2.y * cs.w) * sc;
          float b0 = (q2.x * cs.x + q1.x * cs.y) * sc, b1 = (q2.y * cs.z + q1.y * cs.w) * sc;
          if (rotated) { a0 = q1.x; a1 = q1.y; b0 = q2.x; b1 = q2.y; }
          if (!live) a0 = a1 = b0 = b1 = 0.f;
          split_bf16x2(a0, a1, qhi[ks][hh * 2 + rr], qlo[ks][hh * 2 + rr]);
          split_bf16x2(b0, b1, qhi[ks + KS / 2][hh * 2 + rr], qlo[ks + KS / 2][hh * 2 + rr]);
        }
    }
  }
  const int qpos0 = p0 + jq + gr;                              // position of row gr; row gr + 8 is 8 further
  const FlashLane<DH> fl(lane);
  float o[DH / 8][4], m_run[2], l_run[2];
  bool nan_seen[2] = {false, false};
  for (bool again = false;; again = true) {
#pragma unroll
    for (int n = 0; n < DH / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    m_run[0] = m_run[1] = -INFINITY;
    l_run[0] = l_run[1] = 0.f;
    if (again) issue(0);
    for (int tile = 0; tile < n_tiles; ++tile) {
      issue(tile + 1);
      flash_wait<1>();
      __syncthreads();
      if (again && (tile + 1) * G::KEYS > p0 + qb + 1) {       // (the same for the whole block)
        if (threadIdx.x == 0) bad_row = G::KEYS;
        __syncthreads();
        for (int idx = threadIdx.x; idx < G::KEYS * CPR; idx += blockDim.x) {
          uint4 *v = reinterpret_cast<uint4 *>(tiles_smem + (tile & 1) * G::STAGE_BYTES + G::TILE_BYTES + idx * 16);
          const uint4 u = *v;                                  // (an exponent of all ones carries into its sign)
          if ((((u.x & 0x7f807f80u) + 0x00800080u) | ((u.y & 0x7f807f80u) + 0x00800080u) | ((u.z & 0x7f807f80u) + 0x00800080u) |
               ((u.w & 0x7f807f80u) + 0x00800080u)) & 0x80008000u) {
            *v = make_uint4(0u, 0u, 0u, 0u);
            atomicMin(&bad_row, idx / CPR);
          }
        }
        __syncthreads();
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) nan_seen[rr] |= qpos0 + rr * 8 >= tile * G::KEYS + bad_row;
      }
      const uint32_t stage = ring + (uint32_t)((tile & 1) * G::STAGE_BYTES);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        const int t0 = tile * G::KEYS + half * G::HALF_KEYS;
        if (nq <= 0 || t0 > p0 + jq + nq - 1) break;           // no key of this half is visible to this warp
        const uint32_t kst = stage + (uint32_t)(half * G::HALF_KEYS * G::ROW_BYTES), vst = kst + G::TILE_BYTES;
        flash_step<DH>(kst, vst, fl, qhi, qlo, o, m_run, l_run, [&](float (&s)[4][4]) {
          if (t0 + G::HALF_KEYS - 1 > p0 + jq) {               // (only halves that reach past the first query)
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (t0 + n * 8 + q4 * 2 + (e & 1) > qpos0 + (e >> 1) * 8) s[n][e] = -INFINITY;
          }
        });
      }
      if (tile + 1 < n_tiles) __syncthreads();                 // the stage is free for the tile after next
    }
    // outputs; they leave before the vote (behind it: 3 % of a launch of 33 to 240 tokens)
    bool bad = false;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      l_run[rr] += __shfl_xor_sync(0xffffffffu, l_run[rr], 1);
      l_run[rr] += __shfl_xor_sync(0xffffffffu, l_run[rr], 2);
      float c[2] = {0.f, 0.f};                                 // 0, or NaN where an output is infinite or NaN
#pragma unroll
      for (int n = 0; n < DH / 8; ++n) {
        c[0] = fmaf(o[n][rr * 2], 0.f, c[0]);
        c[1] = fmaf(o[n][rr * 2 + 1], 0.f, c[1]);
      }
      const int i = gr + rr * 8;
      if (i >= nq) continue;
      bad |= c[0] + c[1] != 0.f && l_run[rr] == l_run[rr];
      const float inv = nan_seen[rr] ? __int_as_float(0x7fffffff) : 1.f / l_run[rr];
      uint32_t *dst = reinterpret_cast<uint32_t *>(out + (row0 + jq + i) * d + h * DH);
#pragma unroll
      for (int n = 0; n < DH / 8; ++n) dst[n * 4 + q4] = pack_bf16x2(o[n][rr * 2] * inv, o[n][rr * 2 + 1] * inv);
    }
    if (again || !__syncthreads_or(bad)) break;
  }
}

// The same for passes of 17 to 32 tokens whose queries see at most 32 keys (windows of up to 32 patches: prefill and scoring):
// one tile, so nothing is carried from tile to tile.  The queries' values are used up by the scores before the outputs begin,
// and outputs leave eight dims at a time: 80 instead of 127 registers and 8 instead of 16 KB, 24 warps on an SM.
// Bound: round trips (keys, values and queries together, then the outputs) with 24 warps in flight; 900 instructions a warp.
// us a launch, attn_tiles_kernel -> here: 200 series x 16 heads x 30 tokens 18.0 -> 14.8, 256 x 16 x 29 26.2 -> 20.7, 93 x 16 x 26
// 9.0 -> 8.1, 32 x 8 x 29 4.0 -> 3.5; heads of 32, 200 x 16 x 30 11.4 -> 9.5.
// grid = (heads, B), block = 64 (16 queries a warp), dynamic shared memory: 64 rows of DH.
template <int DH>
__global__ void __launch_bounds__(64, 12)
attn_short_kernel(const float *qkv, const bf16 *Kc, const bf16 *Vc, const float2 *__restrict__ rope, PassGeom g, int n_heads, int rotated,
                  bf16 *__restrict__ out) {
  constexpr int HALF = DH / 2, KS = DH / 16, CPR = DH / 8, RB = DH * 2, KEYS = 32;
  extern __shared__ __align__(256) unsigned char tiles_smem[];
  __shared__ int bad_row;                                      // first value row with an infinity or NaN
  const uint32_t kst = (uint32_t)__cvta_generic_to_shared(tiles_smem), vst = kst + KEYS * RB;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, gr = lane >> 2, q4 = lane & 3, d = n_heads * DH;
  const int h = blockIdx.x, slot = blockIdx.y;
  const SlotPos sp = slot_lookup(g, slot);                     // before the dependency wait: see SlotPos
  pdl_sync();
  if (sp.dead) return;
  const int p0 = sp.p0, n_keys = p0 + g.q_len;
  const size_t row0 = (size_t)slot * g.q_len;
  const bf16 *Kb = Kc + ((size_t)sp.b * n_heads + h) * g.cap * DH, *Vb = Vc + ((size_t)sp.b * n_heads + h) * g.cap * DH;
#pragma unroll
  for (int i = 0; i < KEYS * CPR / 64; ++i) {
    const int idx = i * 64 + threadIdx.x, r = idx / CPR, ch = idx % CPR;
    const size_t src = (size_t)min(r, n_keys - 1) * DH + ch * 8;          // rows past the range repeat its last key (masked below)
    const uint32_t off = (uint32_t)(r * RB + flash_swz<DH>(r, ch) * 16);
    flash_cp16(kst + off, Kb + src);
    flash_cp16(vst + off, Vb + src);
  }
  flash_commit();
  const int jq = w * 16, nq = min(16, g.q_len - jq);           // this warp's queries
  float2 qa[2][KS / 2][2], qb[2][KS / 2][2];                   // rows gr, gr + 8: first-half dims and their partners
#pragma unroll
  for (int rr = 0; rr < 2; ++rr) {
    const int j = min(jq + gr + rr * 8, g.q_len - 1);
    const float *src = qkv + (row0 + j) * 3 * d + h * DH + q4 * 2;
#pragma unroll
    for (int ks = 0; ks < KS / 2; ++ks)
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        qa[rr][ks][hh] = __ldcg(reinterpret_cast<const float2 *>(src + ks * 16 + hh * 8));
        qb[rr][ks][hh] = __ldcg(reinterpret_cast<const float2 *>(src + ks * 16 + hh * 8 + HALF));
      }
  }
  const FlashLane<DH> fl(lane);
  float s[4][4];
#pragma unroll
  for (int n = 0; n < 4; ++n) s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
  flash_wait<0>();
  __syncthreads();
  const float sc = rsqrtf((float)DH) * 1.4426950408889634f;
#pragma unroll
  for (int ks = 0; ks < KS / 2; ++ks) {
    uint32_t hi[2][4], lo[2][4];                               // of k-steps ks and ks + KS / 2
#pragma unroll
    for (int rr = 0; rr < 2; ++rr)
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        float2 a = qa[rr][ks][hh], b = qb[rr][ks][hh];
        if (!rotated) {
          const int j = min(jq + gr + rr * 8, g.q_len - 1);
          const float4 cs = *reinterpret_cast<const float4 *>(rope + (size_t)(p0 + j) * HALF + ks * 16 + hh * 8 + q4 * 2);   // cos0 sin0 cos1 sin1
          const float2 x = a, y = b;
          a = make_float2((x.x * cs.x - y.x * cs.y) * sc, (x.y * cs.z - y.y * cs.w) * sc);
          b = make_float2((y.x * cs.x + x.x * cs.y) * sc, (y.y * cs.z + x.y * cs.w) * sc);
        }
        split_bf16x2(a.x, a.y, hi[0][hh * 2 + rr], lo[0][hh * 2 + rr]);
        split_bf16x2(b.x, b.y, hi[1][hh * 2 + rr], lo[1][hh * 2 + rr]);
      }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t ka = (kst + fl.ka) ^ (uint32_t)((ks + u * (KS / 2)) * 32);
      uint32_t b0[4], b1[4];
      flash_ldsm4(ka, b0);
      flash_ldsm4(ka + 16 * RB, b1);
      mma_bf16_16816(s[0], hi[u], b0[0], b0[1]);
      mma_bf16_16816(s[1], hi[u], b0[2], b0[3]);
      mma_bf16_16816(s[2], hi[u], b1[0], b1[1]);
      mma_bf16_16816(s[3], hi[u], b1[2], b1[3]);
      mma_bf16_16816(s[0], lo[u], b0[0], b0[1]);
      mma_bf16_16816(s[1], lo[u], b0[2], b0[3]);
      mma_bf16_16816(s[2], lo[u], b1[0], b1[1]);
      mma_bf16_16816(s[3], lo[u], b1[2], b1[3]);
    }
  }
  const int qpos0 = p0 + jq + gr;                              // position of row gr; row gr + 8 is 8 further
  uint32_t pa[2][4];
  float inv[2];
#pragma unroll
  for (int rr = 0; rr < 2; ++rr) {
    float mx = -INFINITY;
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float &v = s[n][rr * 2 + e];
        if (n * 8 + q4 * 2 + e > qpos0 + rr * 8) v = -INFINITY;
        mx = fmaxf(mx, v);
      }
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float m_use = mx == -INFINITY ? 0.f : mx;
    float sum = 0.f;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const float a = flash_ex2(s[n][rr * 2] - m_use), b = flash_ex2(s[n][rr * 2 + 1] - m_use);
      sum += a + b;
      pa[n >> 1][(n & 1) * 2 + rr] = pack_bf16x2(a, b);
    }
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    inv[rr] = 1.f / sum;
  }
  for (bool again = false;; again = true) {                    // (again: see attn_tiles_kernel)
    if (again) {
      if (threadIdx.x == 0) bad_row = KEYS;
      __syncthreads();
      for (int idx = threadIdx.x; idx < KEYS * CPR; idx += 64) {
        uint4 *v = reinterpret_cast<uint4 *>(tiles_smem + KEYS * RB + idx * 16);
        const uint4 u = *v;                                    // (an exponent of all ones carries into its sign)
        if ((((u.x & 0x7f807f80u) + 0x00800080u) | ((u.y & 0x7f807f80u) + 0x00800080u) | ((u.z & 0x7f807f80u) + 0x00800080u) |
             ((u.w & 0x7f807f80u) + 0x00800080u)) & 0x80008000u) {
          *v = make_uint4(0u, 0u, 0u, 0u);
          atomicMin(&bad_row, idx / CPR);
        }
      }
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < 2; ++rr)
        if (qpos0 + rr * 8 >= bad_row) inv[rr] = __int_as_float(0x7fffffff);
    }
    float c[2] = {0.f, 0.f};                                   // 0, or NaN where an output is infinite or NaN
#pragma unroll
    for (int t = 0; t < KS; ++t) {                             // 16 dims
      float o[2][4];
#pragma unroll
      for (int n = 0; n < 2; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        uint32_t b[4];
        flash_ldsm4_trans(((vst + fl.va) ^ (uint32_t)(t * 32)) + (uint32_t)(k * 16 * RB), b);
        mma_bf16_16816(o[0], pa[k], b[0], b[1]);
        mma_bf16_16816(o[1], pa[k], b[2], b[3]);
      }
#pragma unroll
      for (int rr = 0; rr < 2; ++rr) {
        uint32_t *dst = reinterpret_cast<uint32_t *>(out + (row0 + jq + gr + rr * 8) * d + h * DH + t * 16);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          c[rr] = fmaf(o[n][rr * 2], 0.f, fmaf(o[n][rr * 2 + 1], 0.f, c[rr]));
          if (gr + rr * 8 < nq) dst[n * 4 + q4] = pack_bf16x2(o[n][rr * 2] * inv[rr], o[n][rr * 2 + 1] * inv[rr]);
        }
      }
    }
    bool bad = false;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) bad |= gr + rr * 8 < nq && c[rr] != 0.f && inv[rr] == inv[rr];
    if (again || !__syncthreads_or(bad)) break;
  }
}

}  // namespace tsfm
