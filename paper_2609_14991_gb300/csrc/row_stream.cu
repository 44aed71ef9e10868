// Row pass of the fused decode step in its streaming form (greedy decoding,
// at most one n-gram LM, decoder option fusion_path 0): one CTA per
// hypothesis row.  The joint kernel before it wrote, for every label v of
// the row, logit[v] + D[v] with the call's shared defaults
// D[v] = lambda*log p(v) + beta*bonus*[the trie root has a child v] (0 for
// blank), and per-tile softmax partials of the raw logits; this pass finishes
// Eq. 1 for the row, takes the greedy decision and advances the state.
//
// Eq. 1 for label v < V at the row's state is
//   fused[v] = logit[v] - lse + lambda*log p_LM(v | h) + beta*bonus*(g(v) - depth)
// where the LM state is kept as its whole suffix chain (one state per order):
// log p_LM(v | h) is the arc v of the deepest chain state s_l that has one
// plus the backoff weights of the deeper states, or log p(v) plus all of
// them; g(v) is the depth of v's goto node from the deepest trie chain node
// with a child v (the trie chain holds every trie node that is a suffix of
// the current match), else [the root has a child v].  So
//   fused[v] + lse = (logit[v] + D[v]) + c_r + delta[v],
//   c_r = lambda*(summed backoff of the state) - beta*bonus*depth,
//   delta[v] = lambda*(log p(v | s_l) - summed backoff of s_l - log p(v))
//            + beta*bonus*(g(v) - [the root has a child v]),
// delta[v] = 0 for a label no chain element continues with.  For row r at
// label step s the pass
//   1. (before waiting for the joint kernel) loads the row's state and chains
//      (after the chunk's first step from the row's own copy, indexed by
//      row) and builds delta[v] in shared memory.  Level 0 (the previous
//      label's continuations, up to every label) is streamed once and writes
//      every label's level-0 delta (for a state with many continuations from
//      its dense row: per label log p(v | u) - log p(v) - cum_0, 0 for no
//      arc); meanwhile every arc of the levels above 0 (few: they continue
//      longer contexts) sets its level's bit in its label's level mask.  The
//      model is suffix-closed (a deeper level's labels are a subset of a
//      shallower one's), so a label's deepest level is its mask's highest bit,
//      and after a barrier that level's arc (held in registers) overwrites the
//      label's delta.  The trie chain nodes are scattered shallowest first
//      (the deepest overwrites);
//   2. (after the wait) the argmax of logit + D + c_r + delta over the labels
//      (blank: its logit alone; ties to the lowest label), i.e. the greedy
//      decision, and (for an emitted label) the log-sum-exp from the tile
//      partials for its fused score;
//   3. blank (or the per-frame label limit) advances the frame; a label y is
//      emitted and advances the chains, assembled from independent searches
//      of y in every chain element, each hit carrying the next state's table
//      record (first arc, arcs, summed backoff) in the same 16-byte load;
//   4. writes the joint input of step s, bf16(ReLU(enc_t + E[last])): it needs
//      the decision alone, so its loads go out before the searches'.
//
// Bound by dependent round trips to L2, not by bytes: after the joint kernel's
// logits are there, one trip for them, then the embedding row beside the
// searches (their first loads were made before the wait; a hit costs one or
// two more).  256 rows, V 1024, H 1024, order 6: 3.3 us from the logits to the
// last joint input, 4.9 with the joint input after the chains' assembly, 128
// threads a row and no early loads; a step 8.2 against 10.4 us.
#include <algorithm>

#include "row_common.cuh"

namespace tsd {

namespace {

using row::best_merge;
using row::checked;
using row::kNegInf;
using row::first_load;
using row::level_groups;
using row::lse_merge;
using row::touch;
using row::warp_find_wide;

constexpr int kStream = 4;  // level-0 arc groups of four per thread whose loads are issued together

// mode: 0 = label step, 1 = final step (apply the last decision only),
// 2 = replay (redo the step's work without committing any state or output;
// used only to time the kernel in isolation).
// VAR bit 0: the stateful form (LSTM input rows instead of the joint input);
// bit 2: few rows (two or three per SM): eight warps, so that every chain
// element's search is one warp's and its first load precedes the wait.
// Otherwise four warps: seven CTAs per SM at 72 registers.  72 also let two
// rows of eight warps start beside a joint CTA (80 registers and 192 threads:
// 629 us a chunk of 256 rows, 64 registers, which spill: 675, this: 616).
template <int VAR>
constexpr int kThreadsOf = (VAR & 4) ? 256 : 128;

template <int VAR>
__global__ void __maxnreg__(72) k_row_fz(DecView d, int step, int mode) {
  constexpr bool PRED = (VAR & 1) != 0, FEW = (VAR & 4) != 0;
  constexpr int kFzThreads = kThreadsOf<VAR>, kFzWarps = kFzThreads / 32;
  constexpr int kDense = FEW ? 2 : 8;  // dense level-0 quads per thread whose loads are issued together
  constexpr int QB = FEW ? 2 : 8;      // label quads per thread whose loads are issued together
  constexpr int kHeld = 1;  // arc groups of four of the levels above 0 a thread keeps in registers
  const Params* __restrict__ P = d.params;
  const int r = blockIdx.x;
  const int V = d.V;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool commit = (mode != 2);
  const bool counting = (mode == 2 || d.count);
  extern __shared__ __align__(16) unsigned char smem[];
  // per label: its LM delta (0: none); the LM chain levels above 0 with an
  // arc for it (bit l); its trie goto depth (0: none)
  float* dlm = reinterpret_cast<float*>(smem);              // [V4]
  uint16_t* lev = reinterpret_cast<uint16_t*>(dlm + d.V4);  // [V4]
  uint8_t* dep = reinterpret_cast<uint8_t*>(lev + d.V4);    // [V4]

  __shared__ int s_t, s_sym, s_cnt, s_last, s_slot, s_T, s_n;
  __shared__ int s_nl, s_nt;
  __shared__ int32_t* s_out_tok;
  __shared__ int32_t* s_out_frame;
  __shared__ float* s_out_score;
  __shared__ int32_t* s_out_count;
  __shared__ const uint16_t* s_enc;
  __shared__ float s_lam, s_beta, s_lse;
  __shared__ int s_lm[kLmChain], s_tr[kTrChain];
  __shared__ int4 s_lmr[kLmChain];    // LM chain records: (first arc, arcs, summed backoff bits, -)
  __shared__ int4 s_trr[kTrChain];    // trie chain records: (first child, children, depth of the children, -)
  __shared__ int4 s_lm_hit[kLmChain]; // target record of y's arc at each old level (x = -2: none)
  __shared__ int4 s_tr_hit[kTrChain]; // child record of y at each old trie node (x = -1: none)
  __shared__ float s_bv[kFzWarps];
  __shared__ int s_bi[kFzWarps];
  __shared__ unsigned long long s_bytes;  // algorithmic bytes of the row-step (when counting)
  __shared__ int s_bad;                   // TSD_CHECKS: a range check failed; the row stops

  // 1. Row state.  It was written by the previous row pass; under
  // programmatic launch this grid may start before its own wait, so these
  // loads go through L2 only (ld.global.cg), never a possibly stale L1 line.
  // After the chunk's first step the row's own copy of its state is read,
  // indexed by row, together with the slot (the chains are read whole: their
  // arrays have room for the longest).
  if (tid == 0) {
    const int slot = __ldcg(P->slots + r);
    s_slot = slot;
    s_T = __ldcg(&P->T);
    s_out_tok = P->out_tok;
    s_out_frame = P->out_frame;
    s_out_score = P->out_score;
    s_out_count = P->out_count;
    s_enc = P->enc;
    s_lam = P->lambda;
    s_beta = P->beta;
    s_n = P->n;
    s_bytes = 0;
    s_bad = !checked(slot >= 0 && slot < d.lm_stride, d.err, 1);
    if (step > 0) {
      s_t = __ldcg(d.r_t + r); s_sym = __ldcg(d.r_sym + r); s_cnt = __ldcg(d.r_cnt + r);
      s_nl = __ldcg(d.m_lm_len + r);
      s_nt = __ldcg(d.m_tr_len + r);
      s_last = __ldcg(d.m_last + r);
    }
  } else if (step > 0 && tid >= 32 && tid < 32 + kLmChain) {
    const int l = tid - 32;
    s_lm[l] = __ldcg(d.m_lm + (size_t)r * kLmChain + l);
    s_lmr[l] = __ldcg(d.m_lmr + (size_t)r * kLmChain + l);
  } else if (step > 0 && tid >= 64 && tid < 64 + kTrChain) {
    const int k = tid - 64;
    s_tr[k] = __ldcg(d.m_tr + (size_t)r * kTrChain + k);
    s_trr[k] = __ldcg(d.m_trr + (size_t)r * kTrChain + k);
  }
  {  // per-label scratch reset (the deltas are reset once the state is known)
    uint2* v4 = reinterpret_cast<uint2*>(lev);
    uint32_t* e4 = reinterpret_cast<uint32_t*>(dep);
    for (int q = tid; q < d.V4 / 4; q += blockDim.x) {
      v4[q] = make_uint2(0u, 0u);
      e4[q] = 0u;
    }
  }
  row::block_sync();
  if (s_bad) return;
  const int slot = s_slot, T = s_T;
  if (step == 0) {
    // the chunk's first step: the stream's state by slot, and the row's copy
    if (tid == 0) {
      s_t = 0; s_sym = 0; s_cnt = 0;
      s_nl = d.has_lm ? __ldcg(d.s_lm_len + slot) : 0;
      s_nt = d.has_tr ? __ldcg(d.s_tr_len + slot) : 0;
      s_last = __ldcg(d.s_last + slot);
      if (commit) {
        d.m_lm_len[r] = s_nl;
        d.m_tr_len[r] = s_nt;
        d.m_last[r] = s_last;
      }
    } else if (tid >= 32 && tid < 32 + kLmChain) {
      const int l = tid - 32;
      if (d.has_lm) {
        s_lm[l] = __ldcg(d.s_lm_chain + (size_t)slot * kLmChain + l);
        s_lmr[l] = __ldcg(d.s_lm_rec + (size_t)slot * kLmChain + l);
        if (commit) {
          d.m_lm[(size_t)r * kLmChain + l] = s_lm[l];
          d.m_lmr[(size_t)r * kLmChain + l] = s_lmr[l];
        }
      }
    } else if (tid >= 64 && tid < 64 + kTrChain) {
      const int k = tid - 64;
      if (d.has_tr) {
        s_tr[k] = __ldcg(d.s_tr_chain + slot * kTrChain + k);
        s_trr[k] = __ldcg(d.s_tr_rec + (size_t)slot * kTrChain + k);
        if (commit) {
          d.m_tr[(size_t)r * kTrChain + k] = s_tr[k];
          d.m_trr[(size_t)r * kTrChain + k] = s_trr[k];
        }
      }
    }
    row::block_sync();
  }
#ifdef TSD_CHECKS
  if (tid == 0) {  // every index the row will follow is inside its table
    bool ok = checked(s_nl >= 0 && s_nl <= kLmChain && s_nt >= 0 && s_nt <= kTrChain, d.err, 2) &&
              checked(s_last >= 0 && s_last <= V, d.err, 3);
    for (int l = 0; ok && l < s_nl; ++l) {
      const int4 c = s_lmr[l];
      ok = checked(s_lm[l] >= 0 && s_lm[l] < d.lm.n_states, d.err, 4) &&
           checked(c.x >= 0 && c.y >= 0 && (int64_t)c.x + c.y <= d.lm.n_arcs, d.err, 5) &&
           checked(l > 0 || (c.w >= -1 && c.w < d.lm.n_dense), d.err, 6);
    }
    for (int k = 0; ok && k < s_nt; ++k) {
      const int4 c = s_trr[k];
      ok = checked(s_tr[k] > 0 && s_tr[k] < d.tr.n_nodes, d.err, 7) &&
           checked(c.x >= 0 && c.y >= 0 && c.x + c.y <= d.tr.n_children && c.z >= 1 && c.z <= 63, d.err, 8);
    }
    s_bad = !ok;
  }
  row::block_sync();
  if (s_bad) return;
#endif
  // the encoder frames this step can use (t, or t+1 after a frame advance)
  // go to L1: no kernel of the chunk writes them
  if (!PRED && s_t < T) {
    const size_t fb = (size_t)d.H * 2;
    const uint16_t* f0 = s_enc + ((size_t)r * T + s_t) * d.H;
    row::prefetch_span(f0, s_t + 1 < T ? 2 * fb : fb, 0);
  }
  // In replay mode every row redoes a full step even if it had finished.
  const bool evaluated = (step > 0) && (s_t < T || !commit);
  const int nl_old = s_nl, nt_old = s_nt;
  const float lam = s_lam;
  const float bscale = s_beta * (d.has_tr ? d.tr.bonus : 0.f);

  // warp w searches chain elements w, w + warps, ...: the first one's first load
  int4 pre = make_int4(0, 0, 0, 0);
  if (FEW && evaluated && warp < nl_old + nt_old) {
    const bool is_lm = warp < nl_old;
    const int4 c = is_lm ? s_lmr[warp] : s_trr[warp - nl_old];
    pre = first_load((is_lm ? d.lm.arc_tok : d.tr.ch_tok) + c.x, c.y, lane);
  }
  if (evaluated) {
    const int4* t4 = reinterpret_cast<const int4*>(d.lm.arc_tok);
    const float4* p4 = reinterpret_cast<const float4*>(d.lm.arc_logp);
    // the aligned arc groups of the levels above 0, in level order: group g's
    // level and first arc (g below their count G)
    int G = 0;
    for (int l = 1; l < nl_old; ++l) G += level_groups(s_lmr[l].x, s_lmr[l].y);
    auto locate = [&](int g, int& l) {
      for (l = 1;; ++l) {
        const int n = level_groups(s_lmr[l].x, s_lmr[l].y);
        if (g < n) break;
        g -= n;
      }
      return (s_lmr[l].x & ~3) + 4 * g;
    };
    auto delta_of = [&](int l, float lp, int v) {
      return __fmul_rn(lam, (lp - __int_as_float(s_lmr[l].z)) - __ldg(d.lm.uni_logp + v));
    };
    // 1a. the levels above 0 (few arcs: they continue longer contexts): each
    //     thread loads its first arc groups, labels and log-probabilities,
    //     and keeps them in registers
    int4 ht[kHeld];
    float4 hp[kHeld];
    int hl[kHeld], hi[kHeld];
#pragma unroll
    for (int u = 0; u < kHeld; ++u) {
      const int g = tid + u * kFzThreads;
      hl[u] = -1;
      hi[u] = 0;
      if (g < G) {
        int l;
        hi[u] = locate(g, l);
        ht[u] = __ldg(t4 + (hi[u] >> 2));
        hp[u] = __ldg(p4 + (hi[u] >> 2));
        hl[u] = l;
      }
    }
    //     and warp w the first 128 children of trie chain node w
    int4 ct = make_int4(0, 0, 0, 0);
    if (warp < nt_old && lane < level_groups(s_trr[warp].x, s_trr[warp].y))
      ct = __ldg(reinterpret_cast<const int4*>(d.tr.ch_tok) + (s_trr[warp].x >> 2) + lane);
    // trie chain node k's children get their depth (shallower nodes first)
    auto trie_node = [&](int k) {
      const int b = s_trr[k].x, e = b + s_trr[k].y, a0 = b & ~3;
      const uint8_t dd = (uint8_t)s_trr[k].z;
      auto put = [&](int i0, int4 t) {
        if (i0 >= b && i0 < e) dep[t.x] = dd;
        if (i0 + 1 >= b && i0 + 1 < e) dep[t.y] = dd;
        if (i0 + 2 >= b && i0 + 2 < e) dep[t.z] = dd;
        if (i0 + 3 >= b && i0 + 3 < e) dep[t.w] = dd;
      };
      const bool held = k < kFzWarps;
      if (held && warp == k) put(a0 + 4 * lane, ct);
      for (int g = (held ? 32 : 0) + tid; a0 + 4 * g < e; g += kFzThreads)
        put(a0 + 4 * g, __ldg(reinterpret_cast<const int4*>(d.tr.ch_tok + a0) + g));
    };
    // 1b. level 0 (the previous label's continuations, up to all V labels),
    //     streamed once: every label's level-0 delta (0 for no arc), which
    //     the deepest level above overwrites below
    if (nl_old > 0 && s_lmr[0].w >= 0 && (PRED || s_lmr[0].y >= max(32, V / 8))) {
      // many continuations (the stateful form: any, as in the one-launch form, whose bits it gives)
      // the state's dense row: per label log p(v | u) - log p(v) - cum_0, 0
      // for no arc (whose delta is 0 as well), contiguous
      const float4* R = reinterpret_cast<const float4*>(d.lm.dense0 + (size_t)s_lmr[0].w * d.lm.V4);
      float4* k4 = reinterpret_cast<float4*>(dlm);
      const int nq4 = d.lm.V4 / 4;
      for (int q0 = tid; q0 < nq4; q0 += kDense * kFzThreads) {
        float4 rq[kDense];
#pragma unroll
        for (int u = 0; u < kDense; ++u) {
          const int q = q0 + u * kFzThreads;
          if (q < nq4) rq[u] = __ldg(R + q);
        }
#pragma unroll
        for (int u = 0; u < kDense; ++u) {
          const int q = q0 + u * kFzThreads;
          if (q < nq4)
            k4[q] = make_float4(__fmul_rn(lam, rq[u].x), __fmul_rn(lam, rq[u].y), __fmul_rn(lam, rq[u].z), __fmul_rn(lam, rq[u].w));
        }
      }
    } else {
      // every label's delta starts at 0 (a dense row above writes them all)
      float4* k4 = reinterpret_cast<float4*>(dlm);
      for (int q = tid; q < d.V4 / 4; q += blockDim.x) k4[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      row::block_sync();
    }
    if (nl_old > 0 && !(s_lmr[0].w >= 0 && (PRED || s_lmr[0].y >= max(32, V / 8)))) {
      const int b0 = s_lmr[0].x, c0 = s_lmr[0].y;
      const int a0 = b0 & ~3, G0 = level_groups(b0, c0);
      for (int gb = 0; gb < G0; gb += kStream * kFzThreads) {
        int4 tk[kStream];
        float4 lp[kStream];
#pragma unroll
        for (int u = 0; u < kStream; ++u) {
          const int g = gb + u * kFzThreads + tid;
          if (g < G0) {
            tk[u] = __ldg(t4 + (a0 >> 2) + g);
            lp[u] = __ldg(p4 + (a0 >> 2) + g);
          }
        }
#pragma unroll
        for (int u = 0; u < kStream; ++u) {
          const int g = gb + u * kFzThreads + tid;
          if (g < G0) {
            const int i0 = a0 + 4 * g;
            const int tv[4] = {tk[u].x, tk[u].y, tk[u].z, tk[u].w};
            const float pv[4] = {lp[u].x, lp[u].y, lp[u].z, lp[u].w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (i0 + j >= b0 && i0 + j < b0 + c0 && checked(tv[j] >= 0 && tv[j] < V, d.err, 9))
                dlm[tv[j]] = delta_of(0, pv[j], tv[j]);
          }
        }
      }
    }
    // 1c. every arc of the levels above 0 sets its level's bit in its
    //     label's word (two labels per 32-bit word), so a label's deepest
    //     level with an arc is its highest bit
    uint32_t* lev2 = reinterpret_cast<uint32_t*>(lev);
    auto offer = [&](int l, int i0, int4 tk) {
      const int b = s_lmr[l].x, c = s_lmr[l].y;
      const int tv[4] = {tk.x, tk.y, tk.z, tk.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i0 + j >= b && i0 + j < b + c && checked(tv[j] >= 0 && tv[j] < V, d.err, 9))
          atomicOr(lev2 + (tv[j] >> 1), 1u << (l + 16 * (tv[j] & 1)));
    };
#pragma unroll
    for (int u = 0; u < kHeld; ++u)
      if (hl[u] >= 0) offer(hl[u], hi[u], ht[u]);
    for (int g = tid + kHeld * kFzThreads; g < G; g += kFzThreads) {  // past what registers hold
      int l;
      const int i0 = locate(g, l);
      offer(l, i0, __ldg(t4 + (i0 >> 2)));
    }
    if (nt_old > 0) trie_node(nt_old - 1);  // the trie chain nodes, shallowest first (the deepest overwrites)
    float hu[kHeld][4];  // the held arcs' unigram terms, on their way over the barrier
#pragma unroll
    for (int u = 0; u < kHeld; ++u) {
      if (hl[u] >= 0) {
        const int b = s_lmr[hl[u]].x, e = b + s_lmr[hl[u]].y;
        const int tv[4] = {ht[u].x, ht[u].y, ht[u].z, ht[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          hu[u][j] = hi[u] + j >= b && hi[u] + j < e && checked(tv[j] >= 0 && tv[j] < V, d.err, 9)
                         ? __ldg(d.lm.uni_logp + tv[j])
                         : 0.f;
      }
    }
    row::block_sync();
    // 1d. the arc of each label at its deepest level writes the label's delta
    //     (one writer per label: a level's arcs have distinct labels)
    auto deepest = [&](int v) { return 31 - __clz((int)lev[v]); };
#pragma unroll
    for (int u = 0; u < kHeld; ++u) {
      if (hl[u] >= 0) {
        const int l = hl[u], b = s_lmr[l].x, c = s_lmr[l].y;
        const int tv[4] = {ht[u].x, ht[u].y, ht[u].z, ht[u].w};
        const float pv[4] = {hp[u].x, hp[u].y, hp[u].z, hp[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int i = hi[u] + j;
          if (i >= b && i < b + c && checked(tv[j] >= 0 && tv[j] < V, d.err, 9) && deepest(tv[j]) == l)
            dlm[tv[j]] = __fmul_rn(lam, (pv[j] - __int_as_float(s_lmr[l].z)) - hu[u][j]);
        }
      }
    }
    for (int g = tid + kHeld * kFzThreads; g < G; g += kFzThreads) {  // past what registers hold
      int l;
      const int i0 = locate(g, l);
      const int4 tk = __ldg(t4 + (i0 >> 2));
      const float4 lq = __ldg(p4 + (i0 >> 2));
      const int b = s_lmr[l].x, c = s_lmr[l].y;
      const int tv[4] = {tk.x, tk.y, tk.z, tk.w};
      const float pv[4] = {lq.x, lq.y, lq.z, lq.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i0 + j >= b && i0 + j < b + c && checked(tv[j] >= 0 && tv[j] < V, d.err, 9) && deepest(tv[j]) == l)
          dlm[tv[j]] = delta_of(l, pv[j], tv[j]);
    }
    if (nt_old > 1) trie_node(nt_old - 2);
    for (int k = nt_old - 3; k >= 0; --k) {
      row::block_sync();
      trie_node(k);
    }
    row::block_sync();
  }
  // the parameters used after the wait go through the constant cache once now
  touch(d.logits); touch(d.part); touch(d.droot); touch(d.E); touch(d.A); touch(d.tr.root_rec); touch(d.lm.uni_rec);
  touch(d.lm.arc_tok); touch(d.lm.arc_rec); touch(d.tr.ch_tok); touch(d.tr.ch_rec); touch(d.s_lm_chain);
  touch(d.s_lm_rec); touch(d.m_lm); touch(d.m_lmr); touch(d.s_lm_len); touch(d.m_lm_len); touch(d.s_tr_chain);
  touch(d.s_tr_rec); touch(d.m_tr); touch(d.m_trr); touch(d.s_tr_len); touch(d.m_tr_len); touch(d.s_last);
  touch(d.m_last); touch(d.r_t); touch(d.r_sym); touch(d.r_cnt); touch(d.cap_rows);
  // Programmatic dependent launch: everything above reads only state the
  // previous row pass wrote (complete before the joint kernel in between let
  // this grid launch) and constant tables; the logits need the wait.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  int y = V;
  float best = 0.f;
  if (evaluated) {
    // 2. the argmax of logit + D + c_r + delta over the labels (blank takes
    //    its logit alone); the log-sum-exp of the raw logits (from the tile
    //    partials) is needed only for an emitted label's score
    const float* lg = d.logits + (size_t)r * d.N_pad;
    if (counting && tid == 0) {
      // Algorithmic bytes: the row's logits and partials read, the row state
      // read and written, every arc of every LM chain level (label +
      // log-probability) and every child of every trie chain node (label)
      // with its record; searches and the joint input are added where they
      // happen; the call's shared rows once per launch by the host.
      unsigned long long ab = 0;
      for (int l = 0; l < nl_old; ++l) ab += 16 + 8ull * s_lmr[l].y;
      for (int k = 0; k < nt_old; ++k) ab += 16 + 4ull * s_trr[k].y;
      s_bytes = ab + 4ull * (V + 1) + 16ull * d.n_ptiles + 2ull * (24 + 4 * (nl_old + nt_old));
    }
    float bv = kNegInf;
    int bi = INT_MAX;
    {
      // c_r = lambda*(summed backoff of the state) - beta*bonus*depth
      const float cum_top = nl_old ? __int_as_float(s_lmr[nl_old - 1].z) : 0.f;
      const int depth_cur = nt_old ? s_trr[0].z - 1 : 0;
      const float cr = row::row_constant(lam, cum_top, bscale, depth_cur);
      const int nq = (V + 3) >> 2;  // quads holding labels < V
      const float4* l4 = reinterpret_cast<const float4*>(lg);
      const float4* k4 = reinterpret_cast<const float4*>(dlm);
      const uint32_t* e4 = reinterpret_cast<const uint32_t*>(dep);
      for (int q0 = tid; q0 < nq; q0 += QB * kFzThreads) {
        float4 lq[QB];
#pragma unroll
        for (int u = 0; u < QB; ++u) {
          const int q = q0 + u * kFzThreads;
          if (q < nq) lq[u] = __ldcg(l4 + q);
        }
#pragma unroll
        for (int u = 0; u < QB; ++u) {
          const int q = q0 + u * kFzThreads;
          if (q < nq) {
            const float4 kq = k4[q];
            const uint32_t eq = e4[q];
            const float lv[4] = {lq[u].x, lq[u].y, lq[u].z, lq[u].w};
            float dl[4] = {kq.x, kq.y, kq.z, kq.w};
            if (eq) {  // a label of this quad has a trie goto node
              const uint32_t rb = __ldg(d.droot + (q >> 3)) >> ((4 * q) & 31);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const uint32_t e = (eq >> (8 * j)) & 0xffu;
                if (e) dl[j] = row::trie_delta(dl[j], e, (rb >> j) & 1u, bscale);
              }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float fv = lv[j] + __fadd_rn(cr, dl[j]);
              if (4 * q + j < V && fv > bv) { bv = fv; bi = 4 * q + j; }
            }
          }
        }
      }
      if (tid == 0) {
        const float fb = __ldcg(lg + V);  // blank: D[V] = 0, no fusion terms
        if (fb > bv) { bv = fb; bi = V; }
      }
    }
    row::reconverge();
    for (int o = 16; o > 0; o >>= 1) {
      const float v2 = __shfl_xor_sync(0xffffffffu, bv, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
      best_merge(bv, bi, v2, i2);
    }
    if (lane == 0) {
      s_bv[warp] = bv;
      s_bi[warp] = bi;
    }
    row::block_sync();
    // every thread merges the warps' bests (no second barrier)
    float b = s_bv[0];
    int bix = s_bi[0];
#pragma unroll
    for (int w = 1; w < kFzWarps; ++w) best_merge(b, bix, s_bv[w], s_bi[w]);
    y = (bix >= 0 && bix <= V) ? bix : V;
    best = b;  // the fused score less the log-sum-exp
  }
  // the frame, the labels in it and the last label after the decision
  const bool label = evaluated && y != V;
  int t1 = s_t, sym1 = s_sym;
  if (label) {
    if (++sym1 >= d.max_sym) { ++t1; sym1 = 0; }
  } else if (evaluated) {
    ++t1;
    sym1 = 0;
  }
  const int last1 = label ? y : s_last;
  const int t = commit ? t1 : min(t1, T - 1);
  const bool next = mode != 1 && t < T;  // another label step follows
  // 4. the joint input of this step needs y alone: its loads go out before the
  //    searches', and it is written while they are in flight
  const bool joint = !PRED && next;
  const uint4* enc_row = reinterpret_cast<const uint4*>(s_enc + ((size_t)r * T + t) * d.H);
  const uint4* emb_row = reinterpret_cast<const uint4*>(d.E + (size_t)last1 * d.H);
  uint4 jx, jz;
  if (joint && tid < d.H / 8) {
    jx = row::load_now(enc_row + tid);
    jz = row::load_now(emb_row + tid);
  }
  uint4 px;
  bool stepped = false;
  const uint4* pred_src[2] = {nullptr, nullptr};
  if (PRED) {
    // Stateful form: the prediction network reads the label just emitted
    // (or, at a stream's first step, the start of sequence) and the row's h
    // from before this step; the LSTM kernel after this one runs the cell.
    const bool fresh = step == 0 && __ldcg(d.pred_fresh + slot) != 0;
    stepped = fresh || label;
    if (tid == 0) {
      d.pflag[r] = stepped ? 1 : 0;
      if (fresh && commit) d.pred_fresh[slot] = 0;
    }
    pred_src[0] = reinterpret_cast<const uint4*>(d.pred_emb + (size_t)(fresh ? V : y) * d.pred_D);
    pred_src[1] = reinterpret_cast<const uint4*>(d.pred_h + (size_t)slot * d.pred_D) - d.pred_D / 8;
    if (stepped && tid < d.pred_D / 4) px = tid < d.pred_D / 8 ? __ldg(pred_src[0] + tid) : __ldcg(pred_src[1] + tid);
  }
  const int4 rhit = warp == 1 && label && d.has_tr ? __ldg(d.tr.root_rec + y) : make_int4(0, 0, 0, 0);
  const int4 uhit = warp == 0 && label && d.has_lm && d.lm.order >= 2 ? __ldg(d.lm.uni_rec + y) : make_int4(-1, 0, 0, 0);
  if (label) {
    // 3a. independent searches of y in every chain element; each hit's
    //     record is the next chain element's
    // the last warp's first tile partials load while it searches
    const float4* pr = d.part + (size_t)r * d.n_ptiles;
    float4 p0 = make_float4(kNegInf, 0.f, 0.f, 0.f);
    if (warp == kFzWarps - 1 && lane < d.n_ptiles) p0 = __ldcg(pr + lane);  // written by the joint kernel
    for (int task = warp; task < nl_old + nt_old; task += kFzWarps) {
      const bool is_lm = task < nl_old;
      const int k = is_lm ? task : task - nl_old;
      const int4 rec = is_lm ? s_lmr[k] : s_trr[k];
      const int32_t* arr = (is_lm ? d.lm.arc_tok : d.tr.ch_tok) + rec.x;
      const int i = FEW && task == warp ? warp_find_wide<true>(arr, rec.y, y, lane, pre)
                                        : warp_find_wide<false>(arr, rec.y, y, lane, pre);
      if (lane == 0) {
        if (is_lm) s_lm_hit[k] = (i >= 0) ? __ldg(d.lm.arc_rec + rec.x + i) : make_int4(-2, 0, 0, 0);
        else s_tr_hit[k] = (i >= 0) ? __ldg(d.tr.ch_rec + rec.x + i) : make_int4(-1, 0, 0, 0);
        if (counting) atomicAdd(&s_bytes, 4ull * (32 - __clz(rec.y + 1)) + 16);
      }
    }
    if (warp == kFzWarps - 1) {  // the log-sum-exp of the raw logits
      float pm = kNegInf, ps = 0.f;
      lse_merge(pm, ps, p0.x, p0.y);
      for (int j = lane + 32; j < d.n_ptiles; j += 32) {
        const float4 p = __ldcg(pr + j);
        lse_merge(pm, ps, p.x, p.y);
      }
      const float lse = row::warp_lse(pm, ps);
      if (lane == 0) s_lse = lse;
    }
  }
  if (joint) {
    uint4* a = reinterpret_cast<uint4*>(d.A + (size_t)r * d.H);
    if (tid < d.H / 8) a[tid] = row::joint_input(jx, jz);
    for (int i = tid + kFzThreads; i < d.H / 8; i += kFzThreads) a[i] = row::joint_input(__ldg(enc_row + i), __ldg(emb_row + i));
  }
  if (PRED && stepped) {
    uint4* dst = reinterpret_cast<uint4*>(d.pred_x + (size_t)r * 2 * d.pred_D);
    if (tid < d.pred_D / 4) dst[tid] = px;
    for (int i = tid + kFzThreads; i < d.pred_D / 4; i += kFzThreads)
      dst[i] = i < d.pred_D / 8 ? __ldg(pred_src[0] + i) : __ldcg(pred_src[1] + i);
  }
  if (label) {
    row::block_sync();
    // 3b. assemble the new chains in place (shared memory) and commit them
    //     (by slot, and by row for the next step): warp 0 the LM chain
    //     (y's unigram state, then the targets of y's arcs at the old levels
    //     up to the first level without one), warp 1 the trie chain (y's
    //     children of the old chain nodes, deepest first, then the root's;
    //     completing a phrase resets it), warp 2 the outputs
    if (warp == 0) {
      int ln = 0;
      if (d.has_lm && d.lm.order >= 2) {
        const int4 h = lane < nl_old ? s_lm_hit[lane] : make_int4(-2, 0, 0, 0);
        const bool cont =
            h.x >= 0 && checked(h.x < d.lm.n_states && h.y >= 0 && h.z >= 0 && (int64_t)h.y + h.z <= d.lm.n_arcs,
                                d.err, 10);
        const unsigned miss = __ballot_sync(0xffffffffu, !cont);
        ln = 1 + min(miss ? __ffs((int)miss) - 1 : 32, kLmChain - 1);
        const int4 u = uhit;  // u.x is y's dense row
        // lane l >= 1 takes the hit of old level l - 1
        const int px = __shfl_up_sync(0xffffffffu, h.x, 1), py = __shfl_up_sync(0xffffffffu, h.y, 1);
        const int pz = __shfl_up_sync(0xffffffffu, h.z, 1), pw = __shfl_up_sync(0xffffffffu, h.w, 1);
        const int nst = lane == 0 ? 1 + y : px;
        const int4 nrec = lane == 0 ? make_int4(u.y, u.z, u.w, u.x) : make_int4(py, pz, pw, 0);
        __syncwarp();
        if (lane < ln) {
          s_lm[lane] = nst;
          s_lmr[lane] = nrec;
          if (commit) {
            d.s_lm_chain[(size_t)slot * kLmChain + lane] = nst;
            d.s_lm_rec[(size_t)slot * kLmChain + lane] = nrec;
            d.m_lm[(size_t)r * kLmChain + lane] = nst;
            d.m_lmr[(size_t)r * kLmChain + lane] = nrec;
          }
        }
      }
      if (lane == 0) {
        s_nl = ln;
        if (commit) {
          if (d.has_lm) d.s_lm_len[slot] = ln;
          d.m_lm_len[r] = ln;
        }
      }
    } else if (warp == 1) {
      const int4 h = lane < nt_old ? s_tr_hit[lane] : make_int4(-1, 0, 0, 0);
      const int dd = lane < nt_old ? s_trr[lane].z + 1 : 0;  // the child's children sit one deeper
      const bool ok = h.x >= 0 && checked(h.x > 0 && h.x < d.tr.n_nodes && h.w >= 0 && h.z + h.w <= d.tr.n_children,
                                          d.err, 11);
      const unsigned vm = __ballot_sync(0xffffffffu, ok);
      const int nv = __popc(vm);
      const int4 rh = rhit;
      const bool root = rh.x != 0;
      // the first element of the new chain ends a phrase: the chain resets
      const int f = __ffs((int)vm) - 1;
      const int fy = __shfl_sync(0xffffffffu, h.y, f < 0 ? 0 : f);
      const bool reset = nv > 0 ? fy == 0 : (root && rh.y == 0);
      const int tn = reset ? 0 : min(nv + (root ? 1 : 0), kTrChain);
      __syncwarp();
      const int pos = __popc(vm & ((1u << lane) - 1u));
      if (ok && pos < tn) {
        s_tr[pos] = h.x;
        s_trr[pos] = make_int4(h.z, h.w, dd, 0);
      }
      if (lane == 0 && root && nv < tn) {
        s_tr[nv] = rh.x;
        s_trr[nv] = make_int4(rh.z, rh.w, 2, 0);
      }
      __syncwarp();
      if (commit && lane < tn) {
        d.s_tr_chain[slot * kTrChain + lane] = s_tr[lane];
        d.s_tr_rec[(size_t)slot * kTrChain + lane] = s_trr[lane];
        d.m_tr[(size_t)r * kTrChain + lane] = s_tr[lane];
        d.m_trr[(size_t)r * kTrChain + lane] = s_trr[lane];
      }
      if (lane == 0) {
        s_nt = tn;
        if (commit) {
          if (d.has_tr) d.s_tr_len[slot] = tn;
          d.m_tr_len[r] = tn;
        }
      }
    }
  }
  if (counting && tid == 0 && evaluated) atomicAdd(d.ctr, s_bytes);
  if (tid == 64) {  // the outputs and the row's place in the chunk
    const int cnt = s_cnt;
    if (label && commit) {
      const int o = r * T * d.max_sym + cnt;
      s_out_tok[o] = y;
      s_out_frame[o] = s_t;
      s_out_score[o] = best - s_lse;
      d.s_last[slot] = y;
      d.m_last[r] = y;
    }
    const int cnt1 = cnt + (label ? 1 : 0);
    if (mode == 1) {
      s_out_count[r] = cnt1;
    } else if (commit) {
      d.r_t[r] = t1;
      d.r_sym[r] = sym1;
      d.r_cnt[r] = cnt1;
    }
  }
  if (counting && tid == 0 && joint) atomicAdd(d.ctr, 6ull * d.H);  // encoder frame, embedding row, A row
  if (d.cap_rows && step < d.cap_steps && mode == 0) {
    row::block_sync();
    if (tid == 0) {
      int* c = d.cap_rows + ((size_t)step * s_n + r) * 4;
      c[0] = next ? t : -1;
      c[1] = next ? last1 : -1;
      c[2] = next ? (s_nl ? s_lm[s_nl - 1] : 0) : -1;
      c[3] = next ? (s_nt ? s_tr[0] : 0) : -1;
    }
  }
}

}  // namespace

size_t row_stream_smem_bytes(int V4) { return (size_t)V4 * (sizeof(float) + sizeof(uint16_t) + sizeof(uint8_t)); }

cudaError_t prepare_stream_kernels(size_t smem) {
  const void* f[] = {(const void*)k_row_fz<0>, (const void*)k_row_fz<1>, (const void*)k_row_fz<4>, (const void*)k_row_fz<5>};
  // the joint kernel's shared-memory split: the next row pass starts on an SM
  // whose joint CTA still runs only if neither kernel asks for another
  for (const void* k : f) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_row_stream(const DecView& d, int M, int step, int mode, size_t smem, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(M);
  // Eight warps a row up to two rows per SM: 304 rows, V 1024: 732 us a chunk of
  // 13 frames against 733 with four, 208 rows: 588 / 711.  A third row leaves no
  // room for a joint CTA beside the rows (400 rows: 804 / 769; V 512, 450 rows:
  // 712 / 628), which costs nothing where the joint kernel's tiles fill the SMs
  // by themselves (not its 64-row tiles): 400 rows, V 2048: 803 / 974, V 4096:
  // 895 / 1054.
  const bool tiles64 = d.n_ptiles * 64 >= d.N && (M + 63) / 64 * d.n_ptiles <= d.sms;
  const bool few = M <= (tiles64 || d.pred_D ? 2 : 3) * d.sms;
  cfg.blockDim = dim3(few ? kThreadsOf<4> : kThreadsOf<0>);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  if (d.pred_D) {
    if (few) cudaLaunchKernelEx(&cfg, k_row_fz<5>, d, step, mode);
    else cudaLaunchKernelEx(&cfg, k_row_fz<1>, d, step, mode);
  } else {
    if (few) cudaLaunchKernelEx(&cfg, k_row_fz<4>, d, step, mode);
    else cudaLaunchKernelEx(&cfg, k_row_fz<0>, d, step, mode);
  }
}

}  // namespace tsd
