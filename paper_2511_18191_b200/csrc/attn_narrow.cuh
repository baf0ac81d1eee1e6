// Causal attention of passes of at most 8 tokens (draft and decode steps, short verifications) over a bf16 KV
// cache: attn_flash_kernel's work split with the operands the other way round.
//
// A 16-row query tile that holds one to eight queries spends half its registers and tensor instructions on
// rows that do not exist.  Here the keys are the M side of mma.sync m16n8k16 and the queries its N side:
// S^T = K Q^T (K through ldmatrix as the A operand), P^T becomes the B operand of O^T = V^T P^T by one 8 x 8
// transpose (movmatrix) per eight keys.  Half the MMAs, 40 instead of 80 registers of fragments, keys in steps
// of 16 or 32: registers for 24 instead of 16 of these latency-bound warps per SM.  (Shared memory, head size 64: 24
// warps with rows of up to 32 keys in one stage, 16 with 48, 12 with 64; three CTAs, 12 warps, with the ring.)
//   * SINGLE: the whole row of a (series, head), cached keys and keys of the pass, sits in one shared-memory
//     stage of `rows` rows (a multiple of 16, at most 64); otherwise a ring of ST stages of 32 keys.
//   * mode FLASH_WARP: one warp per (series, head); grid = ceil(pairs / 4).  mode FLASH_SPLIT: four warps share
//     the keys of one pair and merge through shared memory; grid = (heads, B).
// Precision as there: queries split into bf16 high and low parts, base-2 scores, probabilities rounded to bf16
// for P V, sums in fp32.
// Bound: L2 / HBM reads of the cache with many pairs, the chain of a warp's round trips with few.
#pragma once
#include "attn_flash.cuh"

namespace tsfm {

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

template <int DH> struct NarrowState {
  uint32_t qh[DH / 16][2], ql[DH / 16][2];                     // query lane / 4: B fragments, high and low parts
  float o[DH / 16][4];                                         // dims 16 t + lane / 4 (+ 8) x queries 2 (lane % 4), + 1
  float m[2], l[2];                                            // of queries 2 (lane % 4), + 1; l of this lane's keys only
};

// One step of the running softmax over 16 KT keys at shared-memory rows kst.. (values vst..), positions t0..;
// keys at or past t_lim and keys behind a query's own position p0 + i are masked.
template <int DH, int KT>
__device__ __forceinline__ void narrow_step(NarrowState<DH> &st, uint32_t kst, uint32_t vst, uint32_t ka, uint32_t va, int t0, int t_lim,
                                            int p0, int gr, int q4) {
  constexpr int KS = DH / 16, RB = DH * 2;
  float s[KT][4], s2[KT][4];
#pragma unroll
  for (int k = 0; k < KT; ++k)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[k][e] = s2[k][e] = 0.f;
#pragma unroll
  for (int ks = 0; ks < KS; ++ks)
#pragma unroll
    for (int k = 0; k < KT; ++k) {
      uint32_t a[4];
      flash_ldsm4(((kst + ka) ^ (uint32_t)(ks * 32)) + (uint32_t)(k * 16 * RB), a);
      mma_bf16_16816(s[k], a, st.qh[ks][0], st.qh[ks][1]);
      mma_bf16_16816(s2[k], a, st.ql[ks][0], st.ql[ks][1]);
    }
  const bool edge = t0 + 16 * KT > t_lim || t0 + 16 * KT - 1 > p0;
#pragma unroll
  for (int k = 0; k < KT; ++k)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      s[k][e] += s2[k][e];
      if (edge) {
        const int t = t0 + k * 16 + gr + (e >> 1) * 8;
        if (t >= t_lim || t > p0 + q4 * 2 + (e & 1)) s[k][e] = -INFINITY;
      }
    }
  float alpha[2], use[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float mx = fmaxf(s[0][c], s[0][c + 2]);
#pragma unroll
    for (int k = 1; k < KT; ++k) mx = fmaxf(mx, fmaxf(s[k][c], s[k][c + 2]));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    const float m_new = fmaxf(st.m[c], mx);
    use[c] = m_new == -INFINITY ? 0.f : m_new;                 // nothing visible yet: every p below is 0
    alpha[c] = flash_ex2(st.m[c] - use[c]);
    st.m[c] = m_new;
    st.l[c] *= alpha[c];
  }
#pragma unroll
  for (int t = 0; t < KS; ++t) {
    st.o[t][0] *= alpha[0]; st.o[t][1] *= alpha[1];
    st.o[t][2] *= alpha[0]; st.o[t][3] *= alpha[1];
  }
#pragma unroll
  for (int k = 0; k < KT; ++k) {
    const float p00 = flash_ex2(s[k][0] - use[0]), p01 = flash_ex2(s[k][1] - use[1]);
    const float p10 = flash_ex2(s[k][2] - use[0]), p11 = flash_ex2(s[k][3] - use[1]);
    st.l[0] += p00 + p10;
    st.l[1] += p01 + p11;
    const uint32_t b0 = movmatrix_trans(pack_bf16x2(p00, p01)), b1 = movmatrix_trans(pack_bf16x2(p10, p11));
#pragma unroll
    for (int t = 0; t < KS; ++t) {
      uint32_t a[4];
      flash_ldsm4_trans(((vst + va) ^ (uint32_t)(t * 32)) + (uint32_t)(k * 16 * RB), a);
      mma_bf16_16816(st.o[t], a, b0, b1);
    }
  }
}

template <int DH, bool SINGLE, int ST>
__device__ __forceinline__ void
attn_narrow_body(const float *qkv, bf16 *Kc, bf16 *Vc, const float2 *__restrict__ rope, const PassGeom &g, int n_heads, int n_pairs,
                 int mode, int rows, bf16 *__restrict__ out) {
  using G = FlashGeom<DH, ST>;
  constexpr int HALF = DH / 2, KS = DH / 16, CPR = DH / 8, RB = G::ROW_BYTES;
  extern __shared__ __align__(256) unsigned char flash_smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int gr = lane >> 2, q4 = lane & 3, d = n_heads * DH;
  int h = blockIdx.x, slot = blockIdx.y;
  if (mode == FLASH_WARP) {
    const int pair = blockIdx.x * 4 + w;
    if (pair >= n_pairs) return;                               // no block-wide barrier in this mode
    slot = pair / n_heads;
    h = pair % n_heads;
  }
  const int v_off = SINGLE ? rows * RB : G::TILE_BYTES;        // values behind the keys of a stage
  const int warp_bytes = SINGLE ? 2 * rows * RB : G::WARP_BYTES;
  unsigned char *ring = flash_smem + (size_t)w * warp_bytes;
  const uint32_t ring32 = (uint32_t)__cvta_generic_to_shared(ring);
  const SlotPos sp = slot_lookup(g, slot);                     // before the dependency wait: see SlotPos
  if (sp.dead) return;                                         // per warp (FLASH_WARP) or per CTA: no barrier is pending
  const int p0 = sp.p0, nq = g.q_len;
  const size_t row0 = (size_t)slot * nq;
  bf16 *Kb = Kc + ((size_t)sp.b * n_heads + h) * g.cap * DH;
  bf16 *Vb = Vc + ((size_t)sp.b * n_heads + h) * g.cap * DH;

  // this warp's cached keys [t_beg, t_end), and whether it takes the keys of the pass itself
  int t_beg = 0, t_end = p0;
  bool own_pass_keys = true;
  if (mode == FLASH_SPLIT) {
    // whole chunks, the keys of the pass counted as one more chunk at the end
    const int R = (((p0 + G::CHUNK - 1) / G::CHUNK + 1 + 3) / 4) * G::CHUNK;
    t_beg = min(w * R, p0);
    t_end = min(t_beg + R, p0);
    own_pass_keys = w == 3;
  }
  const int n_c = t_end - t_beg, nch = SINGLE ? 0 : (n_c + G::CHUNK - 1) / G::CHUNK;
  auto issue = [&](int c) {
    if (c < nch) {
      const int t0 = t_beg + c * G::CHUNK;
      const uint32_t kst = ring32 + (uint32_t)((c % ST) * G::STAGE_BYTES), vst = kst + G::TILE_BYTES;
#pragma unroll
      for (int i = 0; i < CPR; ++i) {
        const int idx = i * 32 + lane, r = idx / CPR, ch = idx % CPR;
        const int t = min(t0 + r, t_end - 1);                  // rows past the range repeat its last key (masked below)
        const uint32_t off = (uint32_t)(r * RB + flash_swz<DH>(r, ch) * 16);
        flash_cp16(kst + off, Kb + (size_t)t * DH + ch * 8);
        flash_cp16(vst + off, Vb + (size_t)t * DH + ch * 8);
      }
    }
    flash_commit();
  };
  // Cached keys before the dependency wait: rows below pos0 of this layer's cache were written by this layer's
  // attention in an earlier pass, a whole layer of kernels ago at least.
  if (SINGLE) {
    for (int idx = lane; idx < n_c * CPR; idx += 32) {
      const int r = idx / CPR, ch = idx % CPR;
      const uint32_t off = (uint32_t)(r * RB + flash_swz<DH>(r, ch) * 16);
      flash_cp16(ring32 + off, Kb + (size_t)r * DH + ch * 8);
      flash_cp16(ring32 + v_off + off, Vb + (size_t)r * DH + ch * 8);
    }
    flash_commit();
  } else {
#pragma unroll
    for (int c = 0; c < ST - 1; ++c) issue(c);
  }
  // rotation of this lane's query (constants)
  const bool live = gr < nq;
  float4 cs[KS];
  {
    const float2 *rp = rope + (size_t)(p0 + (live ? gr : 0)) * HALF;
#pragma unroll
    for (int i = 0; i < KS; ++i) cs[i] = *reinterpret_cast<const float4 *>(rp + i * 8 + q4 * 2);   // cos0 sin0 cos1 sin1
  }
  pdl_sync();
  // q, k, v of the pass come from the preceding kernel: ld.global.cg behind the wait (see attn_flash_body).  All
  // first loads are in flight before any is used.
  NarrowState<DH> st;
  float2 qa[KS], qb[KS];
  {
    const float *src = qkv + (row0 + (live ? gr : 0)) * 3 * d + h * DH;
#pragma unroll
    for (int i = 0; i < KS; ++i) {
      qa[i] = __ldcg(reinterpret_cast<const float2 *>(src + i * 8 + q4 * 2));
      qb[i] = __ldcg(reinterpret_cast<const float2 *>(src + i * 8 + q4 * 2 + HALF));
    }
  }
  // keys and values of the pass: one lane handles the element pairs (c, c + 1) and (c + HALF, c + HALF + 1) of a token
  const int n_own = own_pass_keys ? nq * (HALF / 2) : 0;
  float2 oka, okb, ova, ovb;
  float4 ocs;
  auto own_load = [&](int i) {
    const int j = i / (HALF / 2), c = (i % (HALF / 2)) * 2;
    const float *src = qkv + (row0 + j) * 3 * d + h * DH + c;
    oka = __ldcg(reinterpret_cast<const float2 *>(src + d));
    okb = __ldcg(reinterpret_cast<const float2 *>(src + d + HALF));
    ova = __ldcg(reinterpret_cast<const float2 *>(src + 2 * d));
    ovb = __ldcg(reinterpret_cast<const float2 *>(src + 2 * d + HALF));
    ocs = *reinterpret_cast<const float4 *>(rope + (size_t)(p0 + j) * HALF + c);                   // cos0 sin0 cos1 sin1
  };
  if (lane < n_own) own_load(lane);
  {
    const float sc = rsqrtf((float)DH) * 1.4426950408889634f;
#pragma unroll
    for (int i = 0; i < KS; ++i) {
      float a0 = (qa[i].x * cs[i].x - qb[i].x * cs[i].y) * sc, a1 = (qa[i].y * cs[i].z - qb[i].y * cs[i].w) * sc;
      float b0 = (qb[i].x * cs[i].x + qa[i].x * cs[i].y) * sc, b1 = (qb[i].y * cs[i].z + qa[i].y * cs[i].w) * sc;
      if (!live) a0 = a1 = b0 = b1 = 0.f;
      // dims 8 i + 2 q4, + 1 and HALF further: k-step i / 2, half i % 2 of the fragment
      split_bf16x2(a0, a1, st.qh[i / 2][i % 2], st.ql[i / 2][i % 2]);
      split_bf16x2(b0, b1, st.qh[(i + KS) / 2][i % 2], st.ql[(i + KS) / 2][i % 2]);
    }
  }
#pragma unroll
  for (int t = 0; t < KS; ++t) st.o[t][0] = st.o[t][1] = st.o[t][2] = st.o[t][3] = 0.f;
  st.m[0] = st.m[1] = -INFINITY;
  st.l[0] = st.l[1] = 0.f;
  // ldmatrix rows of this lane: keys as A (rows lane % 16, chunk lane / 16), values transposed
  const int krow = lane & 15, vrow = (lane & 7) + ((lane >> 4) & 1) * 8;
  const uint32_t ka = (uint32_t)(krow * RB + flash_swz<DH>(krow, lane >> 4) * 16);
  const uint32_t va = (uint32_t)(vrow * RB + flash_swz<DH>(vrow, (lane >> 3) & 1) * 16);

  // The pass's own keys: rotated, rounded to bf16, appended to the cache and put into the ring's last stage (not
  // used before its first refill) or behind the cached rows of the single stage.  Value rows past the last key of
  // a 16-row block are zeroed: their probabilities are 0, but 0 x NaN would not be.
  {
    unsigned char *own = ring + (SINGLE ? 0 : (ST - 1) * G::STAGE_BYTES);
    uint32_t *ks = reinterpret_cast<uint32_t *>(own), *vs = reinterpret_cast<uint32_t *>(own + v_off);
    const int in_base = SINGLE ? n_c : 0;
    for (int i = lane; i < n_own; i += 32) {
      const int j = i / (HALF / 2), c = (i % (HALF / 2)) * 2, jr = in_base + j;
      const uint32_t k1 = pack_bf16x2(oka.x * ocs.x - okb.x * ocs.y, oka.y * ocs.z - okb.y * ocs.w);
      const uint32_t k2 = pack_bf16x2(okb.x * ocs.x + oka.x * ocs.y, okb.y * ocs.z + oka.y * ocs.w);
      const uint32_t v1 = pack_bf16x2(ova.x, ova.y), v2 = pack_bf16x2(ovb.x, ovb.y);
      if (i + 32 < n_own) own_load(i + 32);
      const int w1 = c / 2, w2 = (c + HALF) / 2;               // 32-bit words of the row
      const int a1 = jr * (DH / 2) + flash_swz<DH>(jr, w1 >> 2) * 4 + (w1 & 3);
      const int a2 = jr * (DH / 2) + flash_swz<DH>(jr, w2 >> 2) * 4 + (w2 & 3);
      ks[a1] = k1; ks[a2] = k2;
      vs[a1] = v1; vs[a2] = v2;
      uint32_t *kg = reinterpret_cast<uint32_t *>(Kb + (size_t)(p0 + j) * DH);
      uint32_t *vg = reinterpret_cast<uint32_t *>(Vb + (size_t)(p0 + j) * DH);
      kg[w1] = k1; kg[w2] = k2;
      vg[w1] = v1; vg[w2] = v2;
    }
    if (SINGLE || own_pass_keys) {
      const int filled = in_base + (own_pass_keys ? nq : 0);   // stage rows that hold keys
      for (int i = filled * (DH / 2) + lane; i < ((filled + 15) & ~15) * (DH / 2); i += 32) vs[i] = 0u;
      if (SINGLE) {
        flash_wait<0>();
        __syncwarp();
        const int t_lim = p0 + nq;
        for (int r = 0; r < filled; r += 32) {
          const uint32_t kst = ring32 + (uint32_t)(r * RB), vst = kst + (uint32_t)v_off;
          if (filled - r > 16) narrow_step<DH, 2>(st, kst, vst, ka, va, r, t_lim, p0, gr, q4);
          else narrow_step<DH, 1>(st, kst, vst, ka, va, r, t_lim, p0, gr, q4);
        }
      } else {
        __syncwarp();
        const uint32_t s32 = ring32 + (uint32_t)((ST - 1) * G::STAGE_BYTES);
        narrow_step<DH, 1>(st, s32, s32 + G::TILE_BYTES, ka, va, p0, p0 + nq, p0, gr, q4);
        // the first refill of this stage follows the warp barrier at the top of the loop below
      }
    }
  }
  if (!SINGLE) {
    for (int c = 0; c < nch; ++c) {
      flash_wait<ST - 2>();
      __syncwarp();
      issue(c + ST - 1);                                       // refills the stage consumed in the previous turn
      const uint32_t kst = ring32 + (uint32_t)((c % ST) * G::STAGE_BYTES);
      narrow_step<DH, 2>(st, kst, kst + G::TILE_BYTES, ka, va, t_beg + c * G::CHUNK, t_end, p0, gr, q4);
    }
    flash_wait<0>();
    __syncwarp();
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    st.l[c] += __shfl_xor_sync(0xffffffffu, st.l[c], 4);
    st.l[c] += __shfl_xor_sync(0xffffffffu, st.l[c], 8);
    st.l[c] += __shfl_xor_sync(0xffffffffu, st.l[c], 16);
  }
  if (mode != FLASH_SPLIT) {
    const float i0 = 1.f / st.l[0], i1 = 1.f / st.l[1];
    uint32_t *dst = reinterpret_cast<uint32_t *>(out + (row0 + (live ? gr : 0)) * d + h * DH);
#pragma unroll
    for (int t = 0; t < KS; ++t) {
      // transposed: query lane / 4, dims 16 t + 2 (lane % 4), + 1 and 8 further
      const uint32_t lo = movmatrix_trans(pack_bf16x2(st.o[t][0] * i0, st.o[t][1] * i1));
      const uint32_t hi = movmatrix_trans(pack_bf16x2(st.o[t][2] * i0, st.o[t][3] * i1));
      if (live) {
        dst[t * 8 + q4] = lo;
        dst[t * 8 + 4 + q4] = hi;
      }
    }
    return;
  }
  // ---- merge the four key ranges: this warp's (o, m, l) into its ring, then every thread combines
  float *ob = reinterpret_cast<float *>(ring);                 // [8][DH]
  float *mb = ob + 8 * DH, *lb = mb + 8;                       // [8], [8]
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int i = q4 * 2 + c;
#pragma unroll
    for (int t = 0; t < KS; ++t) {
      ob[i * DH + t * 16 + gr] = st.o[t][c];
      ob[i * DH + t * 16 + 8 + gr] = st.o[t][c + 2];
    }
    if (gr == 0) { mb[i] = st.m[c]; lb[i] = st.l[c]; }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nq * (DH / 2); idx += blockDim.x) {
    const int i = idx / (DH / 2), c = (idx % (DH / 2)) * 2;
    float m = -INFINITY;
#pragma unroll
    for (int ww = 0; ww < 4; ++ww) m = fmaxf(m, reinterpret_cast<const float *>(flash_smem + (size_t)ww * warp_bytes)[8 * DH + i]);
    float l = 0.f, ox = 0.f, oy = 0.f;
#pragma unroll
    for (int ww = 0; ww < 4; ++ww) {
      const float *wb = reinterpret_cast<const float *>(flash_smem + (size_t)ww * warp_bytes);
      const float mw = wb[8 * DH + i];
      if (mw == -INFINITY) continue;                           // that range held no visible key
      const float sc = exp2f(mw - m);
      const float2 ov = *reinterpret_cast<const float2 *>(wb + i * DH + c);
      l = fmaf(wb[8 * DH + 8 + i], sc, l);
      ox = fmaf(ov.x, sc, ox);
      oy = fmaf(ov.y, sc, oy);
    }
    const float inv = 1.f / l;
    *reinterpret_cast<uint32_t *>(out + (row0 + i) * d + h * DH + c) = pack_bf16x2(ox * inv, oy * inv);
  }
}

template <int DH, int ST>
__global__ void __launch_bounds__(128)
attn_narrow_ring_kernel(const float *qkv, bf16 *Kc, bf16 *Vc, const float2 *__restrict__ rope, PassGeom g, int n_heads, int n_pairs,
                        int mode, bf16 *__restrict__ out) {
  attn_narrow_body<DH, false, ST>(qkv, Kc, Vc, rope, g, n_heads, n_pairs, mode, 0, out);
}
template <int DH>
__global__ void __launch_bounds__(128, DH <= 64 ? 6 : 4)
attn_narrow_single_kernel(const float *qkv, bf16 *Kc, bf16 *Vc, const float2 *__restrict__ rope, PassGeom g, int n_heads, int n_pairs,
                          int rows, bf16 *__restrict__ out) {
  attn_narrow_body<DH, true, 2>(qkv, Kc, Vc, rope, g, n_heads, n_pairs, FLASH_WARP, rows, out);
}

}  // namespace tsfm
