// Hint-bank candidate step: the next verification tree from the request's
// hint bank (Section 4, "Suffix matching" and "Candidate boundary").
//
// The committed prefix y is matched against the bank (tokenised views joined
// by EOS): for n = 7 down to 1 the length-n suffix of y is searched, and the
// tokens after each occurrence become candidate lanes, ahead of the native
// lanes, under a lane budget; the lanes are packed into a prefix tree rooted
// at y's last token.  An occurrence counts only when a non-EOS token follows
// it; the longest n with any counted occurrence is used; lanes are taken in
// bank order, cut at the lane depth or before an EOS; a lane counts towards
// the budget only when it creates a node.
//
// k_hint_match: for every 256-position chunk of the bank the longest n whose suffix
// ends in it (0 when none does before a token that is not EOS) and the set of the
// positions where it ends; a warp per chunk.  What it cannot do without is reading the
// bank once, so it compares every token with y's last one and goes on only where
// that matches.  y's last token may be a common one, in every chunk: the sets are formed
// by warp votes from the tokens in registers, and only the set of the chunk's own
// maximum is written (32 bytes; the call's maximum is all that packing asks for).  A
// bank of 64 M tokens of which 0 / 1 / 5 / 50 % are y's last one takes 56 / 99 / 108 / 126
// us; with a loop per matching position and a byte per position it took 55 / 111 / 150 /
// 261.
// k_hint_pack: one block finds the chunks that hold an occurrence, in bank
// order -- from the chunk maxima themselves in a bank of up to kHintFlat chunks,
// through maxima of 256-chunk spans in a larger one -- gathers the occurrences of
// eight chunks at a time and loads eight lanes at a time, one per warp; warp 0
// inserts them into the tree held in shared memory.
#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace oos {

constexpr int kHintMaxN = 7;        // longest suffix tried
constexpr int kHintThreads = 256;   // threads of both kernels, positions of a chunk, chunks of a span
constexpr int kHintWarps = kHintThreads / 32;
// Chunks whose maxima the packing block reads in one load of 16 bytes a thread.
// Up to there (1 Mi tokens) the span maxima, the atomics that build them and the
// copy that zeroes them are left out: three launches become two.
constexpr int kHintFlat = kHintThreads * 16;
constexpr int kHintUnroll = 4;      // chunks a warp has in flight

// Sets of positions of a chunk: bit l of word [h][k] is position 128 h + 4 l + k, the
// k-th token of lane l's h-th load.
struct HintSet {
  uint32_t w[2][4];
  OOS_DEV bool any() const {
    return ((w[0][0] | w[0][1] | w[0][2] | w[0][3]) | (w[1][0] | w[1][1] | w[1][2] | w[1][3])) != 0u;
  }
};
// where the tokens equal t
OOS_DEV HintSet hint_eq(const int4 (&v)[2], int t) {
  HintSet s;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    s.w[h][0] = __ballot_sync(0xffffffffu, v[h].x == t);
    s.w[h][1] = __ballot_sync(0xffffffffu, v[h].y == t);
    s.w[h][2] = __ballot_sync(0xffffffffu, v[h].z == t);
    s.w[h][3] = __ballot_sync(0xffffffffu, v[h].w == t);
  }
  return s;
}
// m without the positions whose J-th token before them is not t.  o: for the 8 tokens
// ahead of the chunk, in bits 30 and 31 of word k, whether they are t.
template <int J>
OOS_DEV HintSet hint_step(const HintSet& m, const int4 (&v)[2], const uint32_t (&o)[4], int t) {
  const HintSet e = hint_eq(v, t);
  HintSet r;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      constexpr int L = 8;   // k - J + L > 0
      const int at = (k - J + L) & 3, lanes = (L - (k - J + L) + 3) / 4;   // token of the lane that many below
      const uint32_t x = lanes == 0 ? e.w[h][at] : __funnelshift_l(h ? e.w[0][at] : o[at], e.w[h][at], lanes);
      r.w[h][k] = m.w[h][k] & x;
    }
  return r;
}
// The longest suffix from J tokens on: m holds the positions where J match, at least
// one.  before: the 8 tokens ahead of the chunk in lanes 30 and 31 (`is`: where there are).
template <int J>
OOS_DEV int hint_longer(HintSet& m, const int4 (&v)[2], int4 before, bool is, const int* suf, int nmax) {
  if constexpr (J < kHintMaxN) {
    if (J < nmax) {
      const int t = suf[J];
      const uint32_t o[4] = {__ballot_sync(0xffffffffu, is && before.x == t), __ballot_sync(0xffffffffu, is && before.y == t),
                             __ballot_sync(0xffffffffu, is && before.z == t), __ballot_sync(0xffffffffu, is && before.w == t)};
      const HintSet r = hint_step<J>(m, v, o, t);
      if (r.any()) {
        m = r;
        return hint_longer<J + 1>(m, v, before, is, suf, nmax);
      }
    }
  }
  return J;
}
// From one token on; the tokens ahead of the chunk (`ahead`, nullptr where the bank
// starts) are loaded only where two would match if they did.
OOS_DEV int hint_longest(HintSet& m, const int4 (&v)[2], const int32_t* ahead, const int* suf, int nmax) {
  if (nmax < 2) return 1;
  const uint32_t all[4] = {~0u, ~0u, ~0u, ~0u};
  if (!hint_step<1>(m, v, all, suf[1]).any()) return 1;
  const int lane = threadIdx.x & 31;
  const bool is = ahead && lane >= 30;
  int4 before = make_int4(0, 0, 0, 0);
  if (is) {
    const int32_t* p = ahead + (lane - 30) * 4;
    before = make_int4(p[0], p[1], p[2], p[3]);
  }
  return hint_longer<1>(m, v, before, is, suf, nmax);
}

// prefix_len_dev: the prefix length in device memory (the decode loop's
// committed length), or nullptr to use prefix_len.  Lane l of a chunk's warp holds
// positions 4l .. 4l+3 of both 128-position halves, so that a 16-byte load of the
// warp is one contiguous run.  vec: the bank address is 16-byte aligned.
// smax, best: nullptr in a bank of up to kHintFlat chunks.
__global__ void __launch_bounds__(kHintThreads, 3) k_hint_match(const int32_t* __restrict__ bank, int N, int eos,
                                                             const int32_t* __restrict__ prefix, int prefix_len,
                                                             const int32_t* __restrict__ prefix_len_dev, int vec,
                                                             uint32_t* __restrict__ sets, uint8_t* __restrict__ cmax,
                                                             int* __restrict__ smax, int* __restrict__ best) {
  __shared__ int suf[kHintMaxN];
  pdl_wait();   // the committed tokens and their count may come from the previous kernel
  pdl_trigger();
  if (prefix_len_dev) prefix_len = *prefix_len_dev;
  const int nmax = prefix_len < kHintMaxN ? prefix_len : kHintMaxN;
  // suf[j] is the token j places before y's last token
  if (threadIdx.x < nmax) suf[threadIdx.x] = prefix[prefix_len - 1 - threadIdx.x];
  __syncthreads();
  const int last = suf[0];
  const int lane = threadIdx.x & 31;
  const long long n_chunks = ((long long)N + kHintThreads - 1) / kHintThreads;
  const long long n_warps = (long long)gridDim.x * kHintWarps;
  int wbest = 0;
  for (long long c0 = (long long)blockIdx.x * kHintWarps + (threadIdx.x >> 5); c0 < n_chunks;
       c0 += n_warps * kHintUnroll) {
    int4 v[kHintUnroll][2];
#pragma unroll
    for (int u = 0; u < kHintUnroll; ++u) {
      const long long c = c0 + u * n_warps;
      if (vec && (c + 1) * kHintThreads <= N) {
        const int4* src = reinterpret_cast<const int4*>(bank + c * kHintThreads) + lane;
        v[u][0] = __ldcs(src);
        v[u][1] = __ldcs(src + 32);
      }
    }
    uint32_t some = 0u;       // chunks that hold y's last token
#pragma unroll
    for (int u = 0; u < kHintUnroll; ++u) {
      const long long c = c0 + u * n_warps, p0 = c * kHintThreads;
      if (!vec || p0 + kHintThreads > N) {
        int t[8];   // past the bank: EOS, as if that followed its last token
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const long long p = p0 + (i >> 2) * 128 + lane * 4 + (i & 3);
          t[i] = p < N ? bank[p] : eos;
        }
        v[u][0] = make_int4(t[0], t[1], t[2], t[3]);
        v[u][1] = make_int4(t[4], t[5], t[6], t[7]);
      }
      bool hit = false;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        hit = hit || v[u][h].x == last || v[u][h].y == last || v[u][h].z == last || v[u][h].w == last;
      if (c < n_chunks && __any_sync(0xffffffffu, hit)) some |= 1u << u;
    }
#pragma unroll
    for (int u = 0; u < kHintUnroll; ++u) {
      const long long c = c0 + u * n_warps;
      if (c >= n_chunks) break;
      int lmax = 0;
      if (some >> u & 1u) {
        HintSet m = hint_eq(v[u], last);
        // a match counts unless EOS, or nothing, follows: the set of the next tokens' EOS
        const HintSet f = hint_eq(v[u], eos);
        bool after = false;   // after the chunk's last position, asked for only where that one matches
        if (m.w[1][3] >> 31) after = (c + 1) * kHintThreads >= N || bank[(c + 1) * kHintThreads] == eos;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int k = 0; k < 3; ++k) m.w[h][k] &= ~f.w[h][k + 1];
          m.w[h][3] &= ~__funnelshift_r(f.w[h][0], h ? (after ? 1u : 0u) : f.w[1][0], 1);
        }
        // a token past the bank is not one of it
        const long long left = N - c * kHintThreads;
        if (left < kHintThreads) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int n = ((int)left - 128 * h - k + 3) / 4;   // lanes whose k-th token is
              m.w[h][k] &= n <= 0 ? 0u : n >= 32 ? ~0u : (1u << n) - 1u;
            }
        }
        if (m.any()) {
          lmax = hint_longest(m, v[u], c > 0 ? bank + c * kHintThreads - 8 : nullptr, suf, nmax);
          uint32_t mine = m.w[0][0];
#pragma unroll
          for (int i = 1; i < 8; ++i) mine = lane == i ? m.w[i >> 2][i & 3] : mine;
          if (lane < 8) sets[c * 8 + lane] = mine;
        }
      }
      if (lane == 0) {
        cmax[c] = (uint8_t)lmax;
        if (smax && lmax > 0) atomicMax(&smax[c / kHintThreads], lmax);
      }
      wbest = max(wbest, lmax);
    }
  }
  if (best && lane == 0 && wbest > 0) atomicMax(best, wbest);
}

// Whole block: the values of the threads whose `has` is set, in thread order,
// into out[0..count); returns count (the same in every thread).  Two block
// barriers; every thread of the block must call it.
OOS_DEV int ordered_select(bool has, int32_t value, int32_t* out, int* s_wcnt, int* s_cnt) {
  const int warp = threadIdx.x >> 5, lane_id = threadIdx.x & 31;
  const unsigned bal = __ballot_sync(0xffffffffu, has);
  if (lane_id == 0) s_wcnt[warp] = __popc(bal);
  __syncthreads();
  if (has) {
    int off = __popc(bal & ((1u << lane_id) - 1u));
    for (int w = 0; w < warp; ++w) off += s_wcnt[w];
    out[off] = value;
  }
  if (threadIdx.x == 0) {
    int k = 0;
    for (int w = 0; w < kHintThreads / 32; ++w) k += s_wcnt[w];
    *s_cnt = k;
  }
  __syncthreads();
  return *s_cnt;
}

// The tree being built: per node its token, parent, depth and path (the 128-bit set
// of the nodes from the root down to it, itself included).
struct HintTree {
  int32_t tok[kMaxT], par[kMaxT], dep[kMaxT];
  uint32_t path[4][kMaxT];
};

// Insert one lane into the tree (warp 0, all lanes of the warp together).  The
// nodes whose token is the lane's at their depth are found for all nodes at once;
// the lane's longest prefix in the tree ends at the deepest node whose whole path
// is among them (nodes are distinct per (parent, token), so there is one at most
// per depth).  The rest of the lane is appended under it, as far as the node
// budget goes.  Returns whether a node was created.
OOS_DEV bool hint_insert(HintTree& tr, int& T, int max_nodes, const int32_t* lane, int len) {
  const int lane_id = threadIdx.x & 31;
  uint32_t ok[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int i = 32 * b + lane_id;
    const int d = i < T ? tr.dep[i] : 0;
    ok[b] = __ballot_sync(0xffffffffu, i == 0 || (i < T && d <= len && tr.tok[i] == lane[d - 1]));
  }
  uint32_t best = 0u;   // depth * 128 + node of the deepest one
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int i = 32 * b + lane_id;
    if (i < T) {
      bool all = true;
#pragma unroll
      for (int w = 0; w < 4; ++w) all = all && (tr.path[w][i] & ~ok[w]) == 0u;
      if (all) best = max(best, (uint32_t)(tr.dep[i] * kMaxT + i));
    }
  }
  best = __reduce_max_sync(0xffffffffu, best);
  const int cur = (int)(best % kMaxT), j = (int)(best / kMaxT);
  const int add = min(len - j, max_nodes - T);
  if (add <= 0) return false;
  for (int k = lane_id; k < add; k += 32) {
    const int i = T + k;
    tr.tok[i] = lane[j + k];
    tr.par[i] = k == 0 ? cur : i - 1;
    tr.dep[i] = j + k + 1;
#pragma unroll
    for (int w = 0; w < 4; ++w) {   // cur's path and the new nodes T .. i
      const int lo = max(T - 32 * w, 0), hi = min(i - 32 * w, 31);
      const uint32_t run = hi < lo ? 0u : (0xffffffffu >> (31 - hi)) & (0xffffffffu << lo);
      tr.path[w][i] = tr.path[w][cur] | run;
    }
  }
  __syncwarp();
  T += add;
  return true;
}

__global__ void __launch_bounds__(kHintThreads) k_hint_pack(const int32_t* __restrict__ bank, int N, int eos,
                                                            const int32_t* __restrict__ prefix, int prefix_len,
                                                            const uint32_t* __restrict__ sets,
                                                            const uint8_t* __restrict__ cmax,
                                                            const int* __restrict__ smax,
                                                            const int* __restrict__ best,
                                                            const int32_t* __restrict__ native,
                                                            const int32_t* __restrict__ native_len, int n_native,
                                                            int native_stride, int max_lanes, int depth,
                                                            int max_nodes, const int32_t* __restrict__ prefix_len_dev,
                                                            int pad_to, int32_t* out_tok, int32_t* out_par,
                                                            int32_t* out_T, int32_t* out_info) {
  __shared__ HintTree tr;
  __shared__ int32_t s_pos[kHintWarps * kHintThreads];   // occurrences in the chunks being visited, in bank order
  __shared__ int32_t s_chunk[kHintFlat];                 // chunks holding an occurrence, in order
  __shared__ int32_t s_span[kHintThreads];               // this round's spans holding an occurrence, in order
  __shared__ int32_t s_lane[kHintWarps][kMaxT];          // the lanes being inserted
  __shared__ int32_t s_native[kHintWarps][kMaxT];        // the first native lanes
  __shared__ int s_nlen[kHintWarps];
  __shared__ int s_len[kHintWarps];
  __shared__ int s_wcnt[kHintWarps];
  __shared__ int s_nc, s_ns, s_done;
  const int warp = threadIdx.x >> 5, lane_id = threadIdx.x & 31;
  // The caller's inputs were written before the match kernel started (it waits for
  // the kernel before it and lets this one launch only then): what the call needs
  // of them is loaded while the match kernel runs.
  auto native_load = [&](int i, int32_t* dst) {   // one native lane, by a warp; returns its length
    int len = native_len[i];
    len = len < depth ? len : depth;
    len = len < native_stride ? len : native_stride;
    len = len < 0 ? 0 : len;
    for (int j = lane_id; j < len; j += 32) dst[j] = native[(size_t)i * native_stride + j];
    return len;
  };
  if (warp < n_native) {
    const int len = native_load(warp, s_native[warp]);
    if (lane_id == 0) s_nlen[warp] = len;
  }
  if (prefix_len_dev) prefix_len = *prefix_len_dev;
  const int root = prefix[prefix_len - 1];
  pdl_wait();   // the match kernel's results
  pdl_trigger();
  int T = 1, lanes = 0, hint_lanes = 0;       // warp 0's copies are the authoritative ones
  if (threadIdx.x == 0) {
    tr.tok[0] = root;
    tr.par[0] = -1;
    tr.dep[0] = 0;
    tr.path[0][0] = 1u;
    tr.path[1][0] = tr.path[2][0] = tr.path[3][0] = 0u;
    s_done = (max_lanes <= 0 || max_nodes <= 1) ? 1 : 0;
  }
  const int n_chunks = (int)(((long long)N + kHintThreads - 1) / kHintThreads);

  // the lanes of the occurrences in the nc chunks of s_chunk
  auto visit = [&](int nc) {
    for (int ci = 0; ci < nc && !s_done; ci += kHintWarps) {
      // one chunk per warp, 8 positions per lane
      const int c = ci + warp < nc ? s_chunk[ci + warp] : -1;
      uint4 m = make_uint4(0u, 0u, 0u, 0u);
      if (c >= 0) m = reinterpret_cast<const uint4*>(sets + (size_t)c * 8)[lane_id >> 4];
      uint32_t hit = 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t w = (i & 3) == 0 ? m.x : (i & 3) == 1 ? m.y : (i & 3) == 2 ? m.z : m.w;
        hit |= (w >> (2 * (lane_id & 15) + (i >> 2)) & 1u) << i;
      }
      const int mine = c >= 0 ? __popc(hit) : 0;
      int upto = mine;   // hits of lanes 0 .. lane_id
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane_id >= o) upto += y;
      }
      if (lane_id == 31) s_wcnt[warp] = upto;
      __syncthreads();
      int off = upto - mine, total = 0;
      for (int w = 0; w < kHintWarps; ++w) {
        if (w < warp) off += s_wcnt[w];
        total += s_wcnt[w];
      }
      for (int i = 0; mine && i < 8; ++i)
        if ((hit >> i) & 1u) s_pos[off++] = c * kHintThreads + lane_id * 8 + i;
      __syncthreads();
      for (int k = 0; k < total && !s_done; k += kHintWarps) {
        // one lane per warp: up to depth tokens after the occurrence, stopping before an EOS
        if (k + warp < total) {
          const long long q0 = (long long)s_pos[k + warp] + 1;
          int len = depth;
          for (int j0 = 0; j0 < depth; j0 += 32) {
            const int j = j0 + lane_id;
            const int t = j < depth && q0 + j < N ? bank[q0 + j] : eos;
            if (j < depth) s_lane[warp][j] = t;
            const unsigned end = __ballot_sync(0xffffffffu, t == eos);
            if (end) {
              len = min(depth, j0 + __ffs(end) - 1);
              break;
            }
          }
          if (lane_id == 0) s_len[warp] = len;
        }
        __syncthreads();
        if (warp == 0) {
          for (int u = 0; u < kHintWarps && k + u < total; ++u) {
            if (lanes >= max_lanes || T >= max_nodes) break;
            if (hint_insert(tr, T, max_nodes, s_lane[u], s_len[u])) {
              ++lanes;
              ++hint_lanes;
            }
          }
          if (lane_id == 0 && (lanes >= max_lanes || T >= max_nodes)) s_done = 1;
        }
        __syncthreads();
      }
    }
  };

  int n = 0;   // the longest suffix with a counted occurrence
  if (!smax) {
    // every chunk maximum: 16 a thread
    const int b0 = threadIdx.x * 16;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    if (b0 < n_chunks) w = reinterpret_cast<const uint4*>(cmax)[threadIdx.x];
    const uint32_t wd[4] = {w.x, w.y, w.z, w.w};
    int mx[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      mx[i] = b0 + i < n_chunks ? (int)((wd[i >> 2] >> (8 * (i & 3))) & 255u) : 0;
      n = max(n, mx[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n = max(n, __shfl_xor_sync(0xffffffffu, n, o));
    if (lane_id == 0) s_wcnt[warp] = n;
    __syncthreads();
    for (int k = 0; k < kHintWarps; ++k) n = max(n, s_wcnt[k]);
    __syncthreads();
    if (n > 0) {
      int mine = 0;
#pragma unroll
      for (int i = 0; i < 16; ++i) mine += mx[i] >= n ? 1 : 0;
      int upto = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane_id >= o) upto += y;
      }
      if (lane_id == 31) s_wcnt[warp] = upto;
      __syncthreads();
      int off = upto - mine, nc = 0;
      for (int k = 0; k < kHintWarps; ++k) {
        if (k < warp) off += s_wcnt[k];
        nc += s_wcnt[k];
      }
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (mx[i] >= n) s_chunk[off++] = b0 + i;
      __syncthreads();
      visit(nc);
    }
  } else {
    n = *best;
    __syncthreads();
    const int n_spans = (n_chunks + kHintThreads - 1) / kHintThreads;
    for (int sb = 0; n > 0 && sb < n_spans && !s_done; sb += kHintThreads) {
      const int sp = sb + threadIdx.x;
      const int ns = ordered_select(sp < n_spans && smax[sp] >= n, sp, s_span, s_wcnt, &s_ns);
      for (int si = 0; si < ns && !s_done; ++si) {
        const int c = s_span[si] * kHintThreads + threadIdx.x;
        const int nc = ordered_select(c < n_chunks && cmax[c] >= n, c, s_chunk, s_wcnt, &s_nc);
        visit(nc);
      }
    }
  }
  __syncthreads();
  // native lanes fill what the budgets leave
  if (warp == 0) {
    for (int i = 0; i < n_native; ++i) {
      if (lanes >= max_lanes || T >= max_nodes) break;
      const int32_t* nl = i < kHintWarps ? s_native[i] : s_lane[0];
      const int len = i < kHintWarps ? s_nlen[i] : native_load(i, s_lane[0]);
      __syncwarp();
      if (hint_insert(tr, T, max_nodes, nl, len)) ++lanes;
      __syncwarp();
    }
    for (int i = lane_id; i < T; i += 32) {
      out_tok[i] = tr.tok[i];
      out_par[i] = tr.par[i];
    }
    // padding up to a fixed node count (the decode loop verifies a fixed T):
    // leaves under the root carrying the root's token; the verifier is told
    // the real node count and never accepts them
    for (int i = T + lane_id; i < pad_to; i += 32) {
      out_tok[i] = root;
      out_par[i] = 0;
    }
    if (lane_id == 0) {
      *out_T = T;
      out_info[0] = n;
      out_info[1] = hint_lanes;
      out_info[2] = lanes;
    }
  }
}

// Workspace: the call's n (best) and the span maxima first, so that one
// zeroing copy covers both; then the chunks' sets (32 bytes each; a byte per position is
// reserved) and the chunk maxima.
static size_t hint_head_bytes(size_t spans) { return (4 + spans * 4 + 255) / 256 * 256; }

size_t hint_workspace_bytes(long long bank_len) {
  const size_t chunks = (size_t)((bank_len + kHintThreads - 1) / kHintThreads);
  const size_t spans = (chunks + kHintThreads - 1) / kHintThreads;
  return hint_head_bytes(spans) + chunks * kHintThreads + spans * kHintThreads;
}

cudaError_t launch_hint_tree(const int32_t* bank, int N, int eos, const int32_t* prefix, int prefix_len,
                             const int32_t* prefix_len_dev, const int32_t* native, const int32_t* native_len,
                             int n_native, int native_stride, int max_lanes, int depth, int max_nodes, int pad_to,
                             void* ws, int32_t* out_tok, int32_t* out_par, int32_t* out_T, int32_t* out_info,
                             cudaStream_t st) {
  const long long n_chunks = ((long long)N + kHintThreads - 1) / kHintThreads;
  const long long n_spans = (n_chunks + kHintThreads - 1) / kHintThreads;
  int* best = (int*)ws;
  int* smax = best + 1;
  uint32_t* sets = (uint32_t*)((uint8_t*)ws + hint_head_bytes((size_t)n_spans));
  uint8_t* cmax = (uint8_t*)sets + n_chunks * kHintThreads;
  cudaError_t e = cudaSuccess;
  if (n_chunks <= kHintFlat) {
    best = smax = nullptr;
  } else {
    e = cudaMemsetAsync(best, 0, (size_t)(1 + n_spans) * sizeof(int), st);
    if (e != cudaSuccess) return e;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // one warp per 256-position chunk, as many blocks as the SMs hold at once
  const long long want = (n_chunks + kHintThreads / 32 - 1) / (kHintThreads / 32);
  const int grid = (int)(want < (long long)sms * 3 ? want : (long long)sms * 3);
  const int vec = ((uintptr_t)bank & 15) == 0 ? 1 : 0;
  // the packing block launches while the match kernel runs (programmatic
  // dependent launch) and waits for it before reading its results
  e = launch(true, k_hint_match, dim3(grid), dim3(kHintThreads), 0, st, bank, N, eos, prefix, prefix_len,
             prefix_len_dev, vec, sets, cmax, smax, best);
  if (e != cudaSuccess) return e;
  return launch(true, k_hint_pack, dim3(1), dim3(kHintThreads), 0, st, bank, N, eos, prefix, prefix_len,
                (const uint32_t*)sets, (const uint8_t*)cmax, (const int*)smax, (const int*)best, native, native_len,
                n_native, native_stride, max_lanes, depth, max_nodes, prefix_len_dev, pad_to, out_tok, out_par, out_T,
                out_info);
}

}  // namespace oos

using namespace oos;

extern "C" {

size_t oos_hint_workspace_bytes(int32_t bank_len) { return bank_len < 1 ? 0 : hint_workspace_bytes(bank_len); }

int oos_hint_tree(const int32_t* bank, int32_t bank_len, int32_t eos, const int32_t* prefix, int32_t prefix_len,
                  const int32_t* native, const int32_t* native_len, int32_t n_native, int32_t native_stride,
                  int32_t max_lanes, int32_t depth, int32_t max_nodes, void* workspace, size_t ws_bytes,
                  int32_t* out_tokens, int32_t* out_parent, int32_t* out_T, int32_t* out_info, void* stream) {
  if (!bank || bank_len < 1 || !prefix || prefix_len < 1 || n_native < 0 || max_lanes < 0) return OOS_EINVAL;
  if (n_native > 0 && (!native || !native_len || native_stride < 1)) return OOS_EINVAL;
  if (depth < 1 || depth > kMaxT || max_nodes < 1 || max_nodes > kMaxT) return OOS_EINVAL;
  if (!out_tokens || !out_parent || !out_T || !out_info) return OOS_EINVAL;
  if (!workspace || ((uintptr_t)workspace & 255) || ws_bytes < hint_workspace_bytes(bank_len)) return OOS_EWORKSPACE;
  return launch_hint_tree(bank, bank_len, eos, prefix, prefix_len, nullptr, native, native_len, n_native,
                          native_stride, max_lanes, depth, max_nodes, 0, workspace, out_tokens, out_parent, out_T,
                          out_info, (cudaStream_t)stream) == cudaSuccess
             ? OOS_OK
             : OOS_ECUDA;
}

}  // extern "C"
