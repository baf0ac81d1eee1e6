// Fused acceptance step of one speculative round (Sec. 3.2 Eq. 5, Sec. 3.3, Algorithm 1):
// per series, the K tempered Gaussian log-ratios, the K Philox uniforms, the first rejection
// by warp ballot, the correction / bonus patch, the new committed count (= the ragged KV
// rollback length) and the round's counters, and with the last series the end of the round: one launch per round.
#pragma once
#include <type_traits>
#include "common.cuh"

namespace tsfm {

// Philox4x32-10 (Salmon et al., SC'11): 128-bit counter, 64-bit key, ten rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// u in (0, 1) on a 23-bit grid, exact in fp32: ((w >> 9) + 0.5) * 2^-23.
__device__ __forceinline__ float uniform_from_word(uint32_t w) {
  return ((float)(w >> 9) + 0.5f) * 1.1920928955078125e-07f;
}

// Standard normal draw for element e of a patch, for the sampled variants of Sec. 3.3: Box-Muller
// on the Philox words of counter (series, round, position, stream | e / 2); the even element takes
// the cosine branch, the odd one the sine branch.
constexpr uint32_t NOISE_PROPOSAL = 0x10000000u, NOISE_FALLBACK = 0x20000000u;
__device__ __forceinline__ float standard_normal(uint2 key, uint32_t series, uint32_t round, uint32_t pos,
                                                 uint32_t stream, int e) {
  const uint4 w = philox4x32_10(make_uint4(series, round, pos, stream | (uint32_t)(e >> 1)), key);
  const float rad = sqrtf(-2.f * logf(uniform_from_word(w.x)));
  float sn, cs;
  sincospif(2.f * uniform_from_word(w.y), &sn, &cs);
  return rad * ((e & 1) ? sn : cs);
}

__device__ float head_normal(const DevState *st, int series, int k_pos, int e) {
  return standard_normal(make_uint2(st->key0, st->key1), (uint32_t)series, (uint32_t)st->round, (uint32_t)k_pos, NOISE_PROPOSAL, e);
}

struct AcceptCounters {            // device mirror of the integer part of tsfm_stats
  unsigned long long drafted, tested, accepted, committed, near_margin;
  unsigned long long tested_by_pos[32], accepted_by_pos[32], L_hist[34];
};

struct AcceptArgs {
  // proposals x_i (= draft means in the deployed scheme) and draft means mu_q^(i):
  // element (b, i, :) at x + b * x_stride_b + i * P   (i = 0..K-1)
  const float *x, *mu_q;
  long long x_stride_b;
  // where the draft means live when they are not the proposals themselves (sampled proposals):
  // element (b, i, :) at mu_q_alt + (b * K + i) * P; NULL = use mu_q as above
  const float *mu_q_alt;
  const float *mu_p;               // [B, K+1, P] boundary predictions
  // where committed patches go: patch c of this round (c = 0..n) at
  // commit + b * commit_stride_b + c * P.  When commit_accepted == 0 the accepted
  // proposals already sit there and only the correction / bonus patch is written.
  float *commit;
  long long commit_stride_b;
  int commit_accepted;
  // commit_follows_done: the base above additionally advances by done[b] * P (history buffer)
  int commit_follows_done;
  int *done;                       // [B] in/out
  int B, K, P, T;
  float sigma_p, sigma_q, margin;
  uint2 key;
  int round_idx, series0;
  const float *forced_u;           // [B, K] or NULL
  int *n_accept;                   // [B] (or NULL)
  float *ell, *log_u;              // [B, K] (or NULL)
  AcceptCounters *ctr;             // or NULL
  // When st is non-NULL the scales (tau), the Philox key and the round index come from it, n_accept / ell / log_u are
  // per-round arrays indexed by that round, and the CTA that finishes last closes the round:
  DevState *st;
  int *ticket;                     // CTAs that are done (0 before and after)
  int *unfinished;                 // [T] series still short of T after each round
  int *live, *n_live;              // the unfinished series in ascending order, for the next round's compacted passes
  cudaGraphConditionalHandle handle;   // inside a captured graph (use_handle): its WHILE node
  int use_handle;
  const int *body_launches;        // kernel launches of a round, added to launch_ctr
  unsigned long long *launch_ctr;
};

// The state of a call that its statistics are made of, in one piece.
struct CallState {
  DevState st;
  AcceptCounters ctr;
  int status, ticket;
};

// Closes a round (all threads of the last CTA): lists the series that still have patches to commit, accumulates the phase
// clocks, advances the round counter, adds the round's launches to the device-side launch counter and, inside a captured
// graph, tells the WHILE node whether another round is needed.
__device__ __forceinline__ void close_round(const AcceptArgs &a) {
  constexpr int U = 4;                                         // series a lane has in flight (8: 60 registers, a CTA less on an SM at K = 4)
  __shared__ int warp_count[2][8];                             // (in turn: one barrier a step)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int base = 0, turn = 0;
  // ordered compaction: a warp takes n x 32 neighbouring series, the block nw times that at a time
  auto step = [&](int b0, auto series) {
    constexpr int n = decltype(series)::value;
    const int first = b0 + w * n * 32 + lane;
    int done[n], count = 0;
    unsigned m[n];
#pragma unroll
    for (int u = 0; u < n; ++u) done[u] = first + 32 * u < a.B ? __ldcg(a.done + first + 32 * u) : a.T;
#pragma unroll
    for (int u = 0; u < n; ++u) count += __popc(m[u] = __ballot_sync(0xffffffffu, done[u] < a.T));
    if (lane == 0) warp_count[turn][w] = count;
    __syncthreads();
    int off = base;
    for (int i = 0; i < nw; ++i) {
      if (i < w) off += warp_count[turn][i];
      base += warp_count[turn][i];
    }
    turn ^= 1;
#pragma unroll
    for (int u = 0; u < n; ++u) {
      if (done[u] < a.T) a.live[off + __popc(m[u] & ((1u << lane) - 1u))] = first + 32 * u;
      off += __popc(m[u]);
    }
  };
  if (a.B <= blockDim.x) step(0, std::integral_constant<int, 1>{});
  else for (int b0 = 0; b0 < a.B; b0 += U * blockDim.x) step(b0, std::integral_constant<int, U>{});
  if (threadIdx.x != 0) return;
  DevState *st = a.st;
  const int r = st->round;
  const unsigned long long now = globaltimer_ns();
  *a.n_live = a.unfinished[r] = base;
  *a.ticket = 0;
  if (r == 0) st->ns_prefill = st->t_phase[0] - st->t_call;
  st->ns_draft += st->t_phase[1] - st->t_phase[0];
  const unsigned long long t_accept = *reinterpret_cast<const volatile unsigned long long *>(&st->t_phase[2]);   // (another CTA's)
  st->ns_verify += t_accept - st->t_phase[1];
  st->ns_accept += now - t_accept;
  st->round = r + 1;
  if (a.body_launches && a.launch_ctr) *a.launch_ctr += (unsigned long long)*a.body_launches;
  // every round commits at least one patch per unfinished series, so T rounds always suffice:
  // the second condition bounds the loop whatever the counters say
  if (a.use_handle) cudaGraphSetConditional(a.handle, (base > 0 && r + 1 < a.T) ? 1u : 0u);
}

// A few warps per series, one per position in turn (the last position has the bonus patch, which is only kept).  Everything but the
// verification pass's means was written several kernels ago and is fetched before the dependency wait: the call's state, the
// committed count, the proposals.  The rows of mu_p stay in shared memory for the commit where they fit.  Bound: the chain
// of round trips.  With one warp per series, that went through its positions one after the other behind the wait, and the end of
// the round as a launch of its own, a round's two links took 10 us at K = 3 and 4, 9 of them for a single series.
// nw_log < 0: a series a CTA; otherwise eight warps, 2^nw_log of them a series (see launch_accept).  Dynamic shared memory: stage_rows rows
// of P floats a series ((K + 1), or 0: not kept).
constexpr int ACCEPT_WARPS = 8, ACCEPT_E = 4;                  // elements of a row that a lane has in flight
constexpr int ACCEPT_STAGE_BYTES = 40 * 1024;
__global__ void __launch_bounds__(32 * ACCEPT_WARPS) accept_kernel(AcceptArgs a, int nw_log, int stage_rows) {
  extern __shared__ float accept_rows[];
  __shared__ float all_ep[ACCEPT_WARPS * 32], all_eq[ACCEPT_WARPS * 32];   // energies of every position of the CTA's series
  __shared__ int last;
  const bool alone = nw_log < 0;                               // one series: all of the CTA's warps
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = alone ? blockDim.x >> 5 : 1 << nw_log;
  const int s = alone ? 0 : warp >> nw_log, w = alone ? warp : warp & (nw - 1);
  const int b = alone ? blockIdx.x : (blockIdx.x * (blockDim.x >> 5) + warp) >> nw_log;
  float *const pos_ep = all_ep + s * 32, *const pos_eq = all_eq + s * 32;
  const int K = a.K, P = a.P;
  int flags = 0;
  float fallback_r = 0.f;
  if (a.st) {
    const volatile DevState *st = a.st;
    const int r = st->round;
    a.sigma_p = st->tau;
    a.sigma_q = st->sigma_q;
    a.key = make_uint2(st->key0, st->key1);
    a.round_idx = r;
    flags = st->flags;
    fallback_r = st->fallback_r;
    if (a.n_accept) a.n_accept += (size_t)r * a.B;
    if (a.ell) a.ell += (size_t)r * a.B * a.K;
    if (a.log_u) a.log_u += (size_t)r * a.B * a.K;
  }
  const int m = b < a.B ? *reinterpret_cast<const volatile int *>(a.done + b) : a.T;
  const bool finished = m >= a.T;                              // earlier (or no series): nothing to decide
  const long long hist_adv = a.commit_follows_done && !finished ? (long long)m * P : 0;
  const float *xb = a.x + b * a.x_stride_b + hist_adv;
  const bool apart = a.mu_q_alt && (flags & VAR_SAMPLE_PROPOSALS);
  const float *qb = apart ? a.mu_q_alt + (size_t)b * a.K * a.P : a.mu_q + b * a.x_stride_b + hist_adv;
  const bool same = qb == xb;                                  // proposals that are the draft's means
  const float *pb = a.mu_p + (size_t)b * (K + 1) * P;
  float *const rows = accept_rows + s * stage_rows * P;
  float x0[ACCEPT_E], q0[ACCEPT_E];                            // the start of this warp's first row
#pragma unroll
  for (int e = 0; e < ACCEPT_E; ++e) {
    const int c = lane + 32 * e;
    const bool in = !finished && w < K && c < P;
    x0[e] = in ? __ldcg(xb + (size_t)w * P + c) : 0.f;
    q0[e] = same ? x0[e] : in ? __ldcg(qb + (size_t)w * P + c) : 0.f;
  }
  // log u of position `lane`
  float lu = 0.f;
  if (w == 0 && lane < K && !finished)
    lu = logf(a.forced_u ? a.forced_u[(size_t)b * K + lane]
                         : uniform_from_word(philox4x32_10(make_uint4((uint32_t)(a.series0 + b), (uint32_t)a.round_idx, (uint32_t)lane, 0u), a.key).x));
  pdl_sync();
  if (a.st && b == 0 && threadIdx.x == 0) a.st->t_phase[2] = globaltimer_ns();
  if (!finished) {
    // energies ||x - mu_p||_d^2 and ||x - mu_q||_d^2 of every position
    for (int i = w; i <= K; i += nw) {
      float ep = 0.f, eq = 0.f;
      for (int c0 = 0; c0 < P; c0 += 32 * ACCEPT_E) {
        float xv[ACCEPT_E], qv[ACCEPT_E], pv[ACCEPT_E];
#pragma unroll
        for (int e = 0; e < ACCEPT_E; ++e) {
          const int c = c0 + lane + 32 * e;
          const bool in = c < P, first = i == w && c0 == 0;
          pv[e] = in ? __ldcg(pb + (size_t)i * P + c) : 0.f;
          xv[e] = first ? x0[e] : in && i < K ? __ldcg(xb + (size_t)i * P + c) : 0.f;
          qv[e] = same ? xv[e] : first ? q0[e] : in && i < K ? __ldcg(qb + (size_t)i * P + c) : 0.f;
        }
#pragma unroll
        for (int e = 0; e < ACCEPT_E; ++e) {
          const int c = c0 + lane + 32 * e;
          const float dp = xv[e] - pv[e], dq = xv[e] - qv[e];
          ep = fmaf(dp, dp, ep);
          eq = fmaf(dq, dq, eq);
          if (i < stage_rows && c < P) rows[i * P + c] = pv[e];
        }
      }
      ep = warp_sum(ep) / (float)P;
      eq = warp_sum(eq) / (float)P;
      if (lane == 0 && i < K) pos_ep[i] = ep, pos_eq[i] = eq;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(1 + s), "r"(32 * nw) : "memory");
    if (w == 0) {
      // Eq. 5 and the log-domain test  log u <= min(l, 0)
      bool ok = true;
      float l = 0.f;
      if (lane < K) {
        l = -pos_ep[lane] / (2.f * a.sigma_p * a.sigma_p) + pos_eq[lane] / (2.f * a.sigma_q * a.sigma_q)
            + 0.5f * logf((a.sigma_q * a.sigma_q) / (a.sigma_p * a.sigma_p));
        if (flags & VAR_NO_TEMPERING) l *= (float)P;     // l is (1/d) log p/q: undo the 1/d (component ablation)
        ok = (lu <= l) && (lu <= 0.f);                   // log u <= min(l, 0); a NaN statistic compares false: rejected
        if (a.ell) a.ell[(size_t)b * K + lane] = l;
        if (a.log_u) a.log_u[(size_t)b * K + lane] = lu;
      }
      const unsigned rejected = __ballot_sync(0xffffffffu, !ok);     // lanes >= K vote "accepted"
      const int n = rejected ? min(__ffs(rejected) - 1, K) : K;      // leading accepts
      const int L = n + 1;
      const int keep = min(L, a.T - m);

      // commit: accepted proposals (if they are not in place already) then mu_p^(n+1)
      float *cb = a.commit + b * a.commit_stride_b + hist_adv;
      if (a.commit_accepted)
        for (int c = lane; c < n * P; c += 32) cb[c] = xb[c];
      for (int c = lane; c < P; c += 32) {
        float t = n < stage_rows ? rows[n * P + c] : __ldcg(pb + (size_t)n * P + c);
        if (fallback_r != 0.f)                          // t = mu_p + r eps (Algorithm 1, correction and bonus)
          t += fallback_r * standard_normal(a.key, (uint32_t)(a.series0 + b), (uint32_t)a.round_idx, (uint32_t)n, NOISE_FALLBACK, c);
        cb[(size_t)n * P + c] = t;
      }

      const bool tested = lane < min(n + 1, K);
      const bool near = tested && fabsf(l - lu) < a.margin;
      const unsigned near_mask = __ballot_sync(0xffffffffu, near);
      if (a.ctr) {
        if (tested) {
          atomicAdd(&a.ctr->tested_by_pos[lane], 1ull);
          if (lane < n) atomicAdd(&a.ctr->accepted_by_pos[lane], 1ull);
        }
        if (lane == 0) {
          atomicAdd(&a.ctr->drafted, (unsigned long long)K);
          atomicAdd(&a.ctr->tested, (unsigned long long)min(n + 1, K));
          atomicAdd(&a.ctr->accepted, (unsigned long long)n);
          atomicAdd(&a.ctr->committed, (unsigned long long)keep);
          atomicAdd(&a.ctr->near_margin, (unsigned long long)__popc(near_mask));
          atomicAdd(&a.ctr->L_hist[L], 1ull);
        }
      }
      if (lane == 0) {
        a.done[b] = m + keep;
        if (a.n_accept) a.n_accept[b] = n;
      }
    }
  } else if (w == 0 && lane == 0 && b < a.B && a.n_accept) {
    a.n_accept[b] = -1;
  }
  if (!a.st) return;
  if (!alone) __syncthreads();                                 // the other series' counts
  if (threadIdx.x == 0) {
    __threadfence();                                           // done[b], the time stamp: before the ticket
    last = atomicAdd(a.ticket, 1) == (int)gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (last) close_round(a);
}

}  // namespace tsfm
