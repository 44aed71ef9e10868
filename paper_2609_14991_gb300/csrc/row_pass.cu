// Row pass of the fused decode step with several n-gram LMs (Eq. 1, the sum
// over LMs), or one whose unigram states have no dense rows or whose weight is
// not 1: one CTA per hypothesis row.  (Otherwise greedy decoding runs
// row_stream.cu or row_fused.cu.)
//
// The joint kernel before it wrote the row's logits and per-tile softmax
// partials.  For row r at label step s the pass
//   1. loads the row's state and chains, and 2. builds the fusion bias of
//      Eq. 1, sum_i lambda w_i log p_i(v | state i) + beta * boost(v | trie
//      state) for every label v, in shared memory, both before it waits for
//      the joint kernel;
//   3. takes the argmax of logit + bias (blank: its logit alone; ties to the
//      lowest label): blank or the per-frame label limit advances the frame;
//   4. writes the joint input of step s, bf16(ReLU(enc_t + E[last]));
//   5. searches an emitted label in every chain element and 6. assembles the
//      next chains, every hit carrying the next element's table record.
//
// LM state and phrase state are both kept as their whole suffix chain (one
// LM state per order; every trie node that is a suffix of the current one),
// so the next chain after label y is assembled from independent searches of
// y in each chain element -- no dependent pointer chase.
//
// Bound by dependent round trips to L2 and barriers, not by bytes.  With the
// bias built after the decision and added by the joint kernel's epilogue (a
// dependent load and a barrier per level and LM between two joint kernels), a
// chunk of 256 rows (2 LMs, V 1024, H 1024, 13 frames) took 898 us; built
// while the joint kernel runs, with every LM's and node's first loads in one
// round, 570.
#include <algorithm>

#include "row_common.cuh"

namespace tsd {

namespace {

using row::best_merge;
using row::kNegInf;
using row::lse_merge;

// mode: 0 = label step, 1 = final step (apply the last decision only),
// 2 = replay (redo the step's work without committing any state or output;
// used only to time the kernel in isolation).
// L: LMs fused.
template <int L>
__global__ void __launch_bounds__(kRowThreads, 3) k_row(DecView d, int step, int mode) {
  const Params* __restrict__ P = d.params;
  const int r = blockIdx.x;
  const int V = d.V;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kRowThreads / 32;
  const bool commit = (mode != 2);
  const bool counting = (mode == 2 || d.count);
  extern __shared__ __align__(16) unsigned char smem[];
  // per label: the LM value from one LM's chain (NaN: none), the bias (with
  // one LM in the same place), the trie goto depth (0: none)
  float* lmv = reinterpret_cast<float*>(smem);
  float* bias = L > 1 ? lmv + d.V4 : lmv;
  uint8_t* dep = reinterpret_cast<uint8_t*>(bias + d.V4);

  __shared__ int s_t, s_sym, s_cnt, s_last, s_slot, s_T, s_n, s_nt;
  __shared__ int s_nl[L];
  __shared__ int32_t* s_out_tok;
  __shared__ int32_t* s_out_frame;
  __shared__ float* s_out_score;
  __shared__ int32_t* s_out_count;
  __shared__ const uint16_t* s_enc;
  __shared__ float s_lam, s_beta, s_lse;
  __shared__ int s_lm[L][kLmChain], s_tr[kTrChain];
  __shared__ int4 s_lmr[L][kLmChain];     // LM chain records: (first arc, arcs, summed backoff bits, -)
  __shared__ int4 s_trr[kTrChain];        // trie chain records: (first child, children, depth of the children, -)
  __shared__ int4 s_lm_hit[L][kLmChain];  // target record of y's arc at each old level (x = -2: none)
  __shared__ int4 s_tr_hit[kTrChain];     // child record of y at each old trie node (x = -1: none)
  __shared__ float s_bv[kWarps];
  __shared__ int s_bi[kWarps];
  __shared__ unsigned long long s_bytes;

  // 1. Row state, written by the previous row pass: under programmatic launch
  // this grid may start before its own wait, so these loads go through L2
  // only (ld.global.cg), never a possibly stale L1 line.
  if (tid == 0) {
    s_slot = __ldcg(P->slots + r);
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
    s_t = step ? __ldcg(d.r_t + r) : 0;
    s_sym = step ? __ldcg(d.r_sym + r) : 0;
    s_cnt = step ? __ldcg(d.r_cnt + r) : 0;
  }
  row::block_sync();
  const int slot = s_slot, T = s_T;
  if (tid < L * kLmChain) {  // the chains whole: their arrays have room for the longest
    const int i = tid / kLmChain, l = tid % kLmChain;
    const size_t at = ((size_t)i * d.lm_stride + slot) * kLmChain + l;
    s_lm[i][l] = __ldcg(d.s_lm_chain + at);
    s_lmr[i][l] = __ldcg(d.s_lm_rec + at);
  } else if (tid >= 64 && tid < 64 + L) {
    s_nl[tid - 64] = __ldcg(d.s_lm_len + (size_t)(tid - 64) * d.lm_stride + slot);
  } else if (tid == 96) {
    s_nt = d.has_tr ? __ldcg(d.s_tr_len + slot) : 0;
    s_last = __ldcg(d.s_last + slot);
  } else if (tid >= 128 && tid < 128 + kTrChain && d.has_tr) {
    s_tr[tid - 128] = __ldcg(d.s_tr_chain + (size_t)slot * kTrChain + tid - 128);
    s_trr[tid - 128] = __ldcg(d.s_tr_rec + (size_t)slot * kTrChain + tid - 128);
  }
  const int nq = d.V4 / 4;
  const float unset = row::unset_value();
  {
    float4* l4 = reinterpret_cast<float4*>(lmv);
    uint32_t* d4 = reinterpret_cast<uint32_t*>(dep);
    for (int q = tid; q < nq; q += kRowThreads) {
      l4[q] = make_float4(unset, unset, unset, unset);
      d4[q] = 0u;
    }
  }
  row::block_sync();
  // the encoder frames this step can use go to L1
  if (s_t < T) {
    const size_t fb = (size_t)d.H * 2;
    row::prefetch_span(s_enc + ((size_t)r * T + s_t) * d.H, s_t + 1 < T ? 2 * fb : fb, 0);
  }
  // In replay mode every row redoes a full step even if it had finished.
  const bool evaluated = (step > 0) && (s_t < T || !commit);
  const int nt = s_nt;
  int ntask = nt;  // chain elements over all LMs and the trie
#pragma unroll
  for (int i = 0; i < L; ++i) ntask += s_nl[i];
  // chain element `task`: (LM or -1, its level or node), its record and its labels
  auto element = [&](int task, int& i, int& k, int4& rec) -> const int32_t* {
#pragma unroll
    for (i = 0; i < L; ++i) {
      if (task < s_nl[i]) {
        k = task;
        rec = s_lmr[i][k];
        return TSD_LMX(d, i, arc_tok) + rec.x;
      }
      task -= s_nl[i];
    }
    i = -1;
    k = task;
    rec = s_trr[k];
    return d.tr.ch_tok + rec.x;
  };
  const float lam = s_lam;
  int4 pre = make_int4(0, 0, 0, 0);
  if (evaluated) {
    // 2. the bias row.  Every LM's first arc group and unigram quad per
    //    thread, each trie node's first children and the first search's first
    //    load go out together
    int4 ht[L];
    float4 hp[L], hu[L];
    int hl[L], hi[L], G[L];
#pragma unroll
    for (int i = 0; i < L; ++i) {
      G[i] = 0;
      hl[i] = -1;
      hi[i] = 0;
      int g = tid;
      for (int l = 0; l < s_nl[i]; ++l) {  // arc groups in level order
        const int4 c = s_lmr[i][l];
        const int n = row::level_groups(c.x, c.y);
        if (g >= 0 && g < n) {
          hl[i] = l;
          hi[i] = (c.x & ~3) + 4 * g;
        }
        g -= n;
        G[i] += n;
      }
      if (hl[i] >= 0) {
        ht[i] = __ldg(reinterpret_cast<const int4*>(d.lmx[i].arc_tok + hi[i]));
        hp[i] = __ldg(reinterpret_cast<const float4*>(d.lmx[i].arc_logp + hi[i]));
      }
      if (tid < nq) hu[i] = __ldg(reinterpret_cast<const float4*>(d.lmx[i].uni_logp) + tid);  // padded past V
    }
    int4 ct = make_int4(0, 0, 0, 0);
    if (warp < nt && lane < row::level_groups(s_trr[warp].x, s_trr[warp].y))
      ct = __ldg(reinterpret_cast<const int4*>(d.tr.ch_tok) + (s_trr[warp].x >> 2) + lane);
    if (warp < ntask) {
      int i, k;
      int4 rec;
      const int32_t* arr = element(warp, i, k, rec);
      pre = row::first_load(arr, rec.y, lane);
    }
    // the trie nodes shallowest first (the deepest overwrites), one before each barrier
    int tk = nt - 1;
    auto next_trie = [&]() {
      if (tk < 0) return;
      const int k = tk--;
      const int b = s_trr[k].x, e = b + s_trr[k].y, a0 = b & ~3;
      const uint8_t dd = (uint8_t)s_trr[k].z;
      auto put = [&](int i0, int4 t) {
        if (i0 >= b && i0 < e) dep[t.x] = dd;
        if (i0 + 1 >= b && i0 + 1 < e) dep[t.y] = dd;
        if (i0 + 2 >= b && i0 + 2 < e) dep[t.z] = dd;
        if (i0 + 3 >= b && i0 + 3 < e) dep[t.w] = dd;
      };
      if (warp == k) put(a0 + 4 * lane, ct);
      for (int g = (k < kWarps ? 32 : 0) + tid; a0 + 4 * g < e; g += kRowThreads)
        put(a0 + 4 * g, __ldg(reinterpret_cast<const int4*>(d.tr.ch_tok + a0) + g));
    };
    float4* l4 = reinterpret_cast<float4*>(lmv);
    float4* b4 = reinterpret_cast<float4*>(bias);
    const uint32_t* d4 = reinterpret_cast<const uint32_t*>(dep);
    const int depth_cur = nt ? s_trr[0].z - 1 : 0;
    const float bscale = s_beta * (d.has_tr ? d.tr.bonus : 0.f);
    const float tr_base = -bscale * (float)depth_cur;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      const int n = s_nl[i];
      const float cum_top = n ? __int_as_float(s_lmr[i][n - 1].z) : 0.f;
      // the levels deepest first: a label keeps the first value it gets
      int end = G[i];
      for (int l = n - 1; l >= 0; --l) {
        const int4 c = s_lmr[i][l];
        const int b = c.x, e = c.x + c.y, first = end - row::level_groups(c.x, c.y);
        const float off = cum_top - __int_as_float(c.z);
        auto put = [&](int i0, int4 t, float4 v) {
          if (i0 >= b && i0 < e && isnan(lmv[t.x])) lmv[t.x] = off + v.x;
          if (i0 + 1 >= b && i0 + 1 < e && isnan(lmv[t.y])) lmv[t.y] = off + v.y;
          if (i0 + 2 >= b && i0 + 2 < e && isnan(lmv[t.z])) lmv[t.z] = off + v.z;
          if (i0 + 3 >= b && i0 + 3 < e && isnan(lmv[t.w])) lmv[t.w] = off + v.w;
        };
        if (hl[i] == l) put(hi[i], ht[i], hp[i]);
        for (int g = max(first, kRowThreads) + tid; g < end; g += kRowThreads) {  // past what registers hold
          const int i0 = (b & ~3) + 4 * (g - first);
          put(i0, __ldg(reinterpret_cast<const int4*>(d.lmx[i].arc_tok + i0)),
              __ldg(reinterpret_cast<const float4*>(d.lmx[i].arc_logp + i0)));
        }
        end = first;
        next_trie();
        row::block_sync();
      }
      if (i == L - 1) {
        while (tk >= 0) {
          next_trie();
          row::block_sync();
        }
      }
      const float alpha = lam * d.lm_w[i];
      for (int q = tid; q < nq; q += kRowThreads) {
        const float4 l = l4[q];
        const float4 u = q == tid ? hu[i] : __ldg(reinterpret_cast<const float4*>(d.lmx[i].uni_logp) + q);
        float4 a = i == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : b4[q];
        a.x += alpha * (isnan(l.x) ? u.x + cum_top : l.x);
        a.y += alpha * (isnan(l.y) ? u.y + cum_top : l.y);
        a.z += alpha * (isnan(l.z) ? u.z + cum_top : l.z);
        a.w += alpha * (isnan(l.w) ? u.w + cum_top : l.w);
        if (i == L - 1) {
          const uint32_t dd = d4[q];
          const uint32_t rb = __ldg(d.droot + (q >> 3)) >> ((4 * q) & 31);
          auto boost = [&](int j) {
            const int dj = (dd >> (8 * j)) & 0xff;
            return dj ? bscale * (float)(dj - depth_cur) : (((rb >> j) & 1u) ? bscale : 0.f) + tr_base;
          };
          a.x += boost(0);
          a.y += boost(1);
          a.z += boost(2);
          a.w += boost(3);
        } else {
          l4[q] = make_float4(unset, unset, unset, unset);
        }
        b4[q] = a;
      }
      if (i < L - 1) row::block_sync();
    }
  }
  // the parameters used after the wait go through the constant cache once now
  row::touch(d.logits); row::touch(d.part); row::touch(d.E); row::touch(d.A); row::touch(d.tr.root_rec);
  row::touch(d.tr.ch_rec); row::touch(d.r_t); row::touch(d.r_sym); row::touch(d.r_cnt); row::touch(d.cap_rows);
  // Programmatic dependent launch: everything above reads only state the
  // previous row pass wrote (complete before the joint kernel in between let
  // this grid launch) and constant tables; the logits need the wait.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  int y = V;
  float best = 0.f;
  if (evaluated) {
    // 3. the argmax of logit + bias (blank: its logit alone), each thread over
    //    the quads whose bias it wrote
    const float* lg = d.logits + (size_t)r * d.N_pad;
    float bv = kNegInf;
    int bi = INT_MAX;
    const float4* l4 = reinterpret_cast<const float4*>(lg);
    const float4* b4 = reinterpret_cast<const float4*>(bias);
    for (int q0 = tid; q0 < nq; q0 += 2 * kRowThreads) {
      float4 lq[2];
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (q0 + u * kRowThreads < nq) lq[u] = __ldcg(l4 + q0 + u * kRowThreads);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = q0 + u * kRowThreads;
        if (q >= nq) break;
        const float4 b = b4[q];
        const float f[4] = {lq[u].x + b.x, lq[u].y + b.y, lq[u].z + b.z, lq[u].w + b.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (4 * q + j < V && f[j] > bv) { bv = f[j]; bi = 4 * q + j; }
      }
    }
    if (tid == 0) {
      const float fb = __ldcg(lg + V);
      if (fb > bv) { bv = fb; bi = V; }
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
    if (counting && tid == 0) {
      // Algorithmic bytes: the row's logits and partials, the state read and
      // written, every arc of every LM level and every child of every trie
      // node with its record; searches and the joint input below.
      unsigned long long ab = 4ull * (V + 1) + 16ull * d.n_ptiles + 2ull * (24 + 4 * ntask);
#pragma unroll
      for (int i = 0; i < L; ++i)
        for (int l = 0; l < s_nl[i]; ++l) ab += 16 + 8ull * s_lmr[i][l].y;
      for (int k = 0; k < nt; ++k) ab += 16 + 4ull * s_trr[k].y;
      s_bytes = ab;
    }
    row::block_sync();
    best = s_bv[0];
    int bix = s_bi[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) best_merge(best, bix, s_bv[w], s_bi[w]);
    y = (bix >= 0 && bix <= V) ? bix : V;
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
  // 4. the joint input of this step: its loads go out before the searches'
  const uint4* enc_row = reinterpret_cast<const uint4*>(s_enc + ((size_t)r * T + t) * d.H);
  const uint4* emb_row = reinterpret_cast<const uint4*>(d.E + (size_t)last1 * d.H);
  uint4 jx, jz;
  if (next && tid < d.H / 8) {
    jx = row::load_now(enc_row + tid);
    jz = row::load_now(emb_row + tid);
  }
  int4 own = make_int4(-1, 0, 0, 0);  // y's unigram state in LM `warp`, y's child of the root (warp L)
  if (label) {
    // 5. independent searches of y in every chain element; each hit's record
    //    is the next chain element's
    if (warp < L) {
      if (TSD_LMX(d, warp, order) >= 2) own = __ldg(TSD_LMX(d, warp, uni_rec) + y);
    } else if (warp == L) {
      own = d.has_tr ? __ldg(d.tr.root_rec + y) : make_int4(0, 0, 0, 0);
    }
    const float4* pr = d.part + (size_t)r * d.n_ptiles;
    float4 p0 = make_float4(kNegInf, 0.f, 0.f, 0.f);
    if (warp == kWarps - 1 && lane < d.n_ptiles) p0 = __ldcg(pr + lane);  // written by the joint kernel
    for (int task = warp; task < ntask; task += kWarps) {
      int i, k;
      int4 rec;
      const int32_t* arr = element(task, i, k, rec);
      const int at = task == warp ? row::warp_find_wide<true>(arr, rec.y, y, lane, pre)
                                  : row::warp_find_wide<false>(arr, rec.y, y, lane, pre);
      if (lane == 0) {
        if (i >= 0) s_lm_hit[i][k] = at >= 0 ? __ldg(TSD_LMX(d, i, arc_rec) + rec.x + at) : make_int4(-2, 0, 0, 0);
        else s_tr_hit[k] = at >= 0 ? __ldg(d.tr.ch_rec + rec.x + at) : make_int4(-1, 0, 0, 0);
        if (counting) atomicAdd(&s_bytes, 4ull * (32 - __clz(rec.y + 1)) + 16);
      }
    }
    if (warp == kWarps - 1) {  // the log-sum-exp of the raw logits
      float pm = kNegInf, ps = 0.f;
      lse_merge(pm, ps, p0.x, p0.y);
      for (int j = lane + 32; j < d.n_ptiles; j += 32) {
        const float4 p = __ldcg(pr + j);
        lse_merge(pm, ps, p.x, p.y);
      }
      row::reconverge();
      for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, pm, o);
        const float s2 = __shfl_xor_sync(0xffffffffu, ps, o);
        lse_merge(pm, ps, m2, s2);
      }
      if (lane == 0) s_lse = pm + logf(ps);
    }
  }
  if (next) {
    uint4* a = reinterpret_cast<uint4*>(d.A + (size_t)r * d.H);
    if (tid < d.H / 8) a[tid] = row::joint_input(jx, jz);
    for (int i = tid + kRowThreads; i < d.H / 8; i += kRowThreads)
      a[i] = row::joint_input(__ldg(enc_row + i), __ldg(emb_row + i));
  }
  if (label) {
    row::block_sync();
    // 6. the new chains: warp i LM i (y's unigram state, then the targets of
    //    y's arcs at the old levels up to the first level without one), warp
    //    L the trie (y's children of the old nodes, deepest first, then the
    //    root's; completing a phrase resets it)
    if (warp < L) {
      const int i = warp;
      int ln = 0;
      if (TSD_LMX(d, i, order) >= 2) {
        const int4 h = lane < s_nl[i] ? s_lm_hit[i][lane] : make_int4(-2, 0, 0, 0);
        const unsigned miss = __ballot_sync(0xffffffffu, h.x < 0);
        ln = 1 + min(miss ? __ffs((int)miss) - 1 : 32, kLmChain - 1);
        // lane l >= 1 takes the hit of old level l - 1
        const int px = __shfl_up_sync(0xffffffffu, h.x, 1), py = __shfl_up_sync(0xffffffffu, h.y, 1);
        const int pz = __shfl_up_sync(0xffffffffu, h.z, 1), pw = __shfl_up_sync(0xffffffffu, h.w, 1);
        if (lane < ln) {
          const int nst = lane == 0 ? 1 + y : px;
          s_lm[i][lane] = nst;
          if (commit) {
            const size_t at = ((size_t)i * d.lm_stride + slot) * kLmChain + lane;
            d.s_lm_chain[at] = nst;
            d.s_lm_rec[at] = lane == 0 ? make_int4(own.y, own.z, own.w, own.x) : make_int4(py, pz, pw, 0);
          }
        }
      }
      __syncwarp();
      if (lane == 0) {
        s_nl[i] = ln;
        if (commit) d.s_lm_len[(size_t)i * d.lm_stride + slot] = ln;
      }
    } else if (warp == L) {
      const int4 h = lane < nt ? s_tr_hit[lane] : make_int4(-1, 0, 0, 0);
      const int dd = lane < nt ? s_trr[lane].z + 1 : 0;  // the child's children sit one deeper
      const unsigned vm = __ballot_sync(0xffffffffu, h.x >= 0);
      const int nv = __popc(vm);
      const bool root = own.x != 0;
      // the first element of the new chain ends a phrase: the chain resets
      const int f = __ffs((int)vm) - 1;
      const int fy = __shfl_sync(0xffffffffu, h.y, f < 0 ? 0 : f);
      const bool reset = nv > 0 ? fy == 0 : (root && own.y == 0);
      const int tn = reset ? 0 : min(nv + (root ? 1 : 0), kTrChain);
      const int pos = __popc(vm & ((1u << lane) - 1u));
      auto put = [&](int p, int node, int4 rec) {
        if (p == 0) s_tr[0] = node;
        if (commit) {
          d.s_tr_chain[(size_t)slot * kTrChain + p] = node;
          d.s_tr_rec[(size_t)slot * kTrChain + p] = rec;
        }
      };
      if (h.x >= 0 && pos < tn) put(pos, h.x, make_int4(h.z, h.w, dd, 0));
      if (lane == 0 && root && nv < tn) put(nv, own.x, make_int4(own.z, own.w, 2, 0));
      if (lane == 0) {
        s_nt = tn;
        if (commit && d.has_tr) d.s_tr_len[slot] = tn;
      }
    }
  }
  if (counting && tid == 0) {  // encoder frame, embedding row, A row
    if (evaluated || next) atomicAdd(d.ctr, (evaluated ? s_bytes : 0ull) + (next ? 6ull * d.H : 0ull));
  }
  if (tid == kRowThreads - 1) {  // the outputs and the row's place in the chunk
    const int cnt = s_cnt;
    if (label && commit) {
      const int o = r * T * d.max_sym + cnt;
      s_out_tok[o] = y;
      s_out_frame[o] = s_t;
      s_out_score[o] = best - s_lse;
      d.s_last[slot] = y;
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
  if (d.cap_rows && step < d.cap_steps && mode == 0) {
    row::block_sync();
    if (tid == 0) {
      int* c = d.cap_rows + ((size_t)step * s_n + r) * 4;
      c[0] = next ? t : -1;
      c[1] = next ? last1 : -1;
      c[2] = next ? (s_nl[0] ? s_lm[0][s_nl[0] - 1] : 0) : -1;
      c[3] = next ? (s_nt ? s_tr[0] : 0) : -1;
    }
  }
}

// After a chain is written from the host: its elements' table records.
__global__ void k_fix_records(DecView d, int slot) {
  const int l = threadIdx.x;
  for (int i = 0; i < d.n_lm && l < kLmChain; ++i) {
    const size_t h = (size_t)i * d.lm_stride + slot;
    if (l >= d.s_lm_len[h]) continue;
    const int st = d.s_lm_chain[h * kLmChain + l];
    // the fourth field of the first (unigram) level: its dense row, if any
    const int dense = (l == 0 && TSD_LMX(d, i, order) >= 2 && st >= 1 && st <= d.V) ? TSD_LMX(d, i, uni_dense)[st - 1] : -1;
    d.s_lm_rec[h * kLmChain + l] = make_int4(TSD_LMX(d, i, st_begin)[st], TSD_LMX(d, i, st_count)[st],
                                             __float_as_int(TSD_LMX(d, i, st_cum)[st]), dense);
  }
  if (d.has_tr && l < kTrChain && l < d.s_tr_len[slot]) {
    const int q = d.s_tr_chain[(size_t)slot * kTrChain + l];
    d.s_tr_rec[(size_t)slot * kTrChain + l] = make_int4(d.tr.nd_begin[q], d.tr.nd_count[q], d.tr.nd_depth[q] + 1, 0);
  }
}

__global__ void k_open(DecView d, int slot) {
  if (threadIdx.x == 0) {
    d.s_last[slot] = d.V;
    for (int i = 0; i < (d.n_lm > 1 ? d.n_lm : 1); ++i) d.s_lm_len[i * d.lm_stride + slot] = 0;
    d.s_tr_len[slot] = 0;
  }
}

__global__ void k_repack(const uint16_t* __restrict__ W, uint16_t* __restrict__ Wt, int H, int N, int N_pad) {
  __shared__ uint16_t tile[32][33];
  int k0 = blockIdx.y * 32, v0 = blockIdx.x * 32;
  int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int i = ty; i < 32; i += 8) {
    int k = k0 + i, v = v0 + tx;
    tile[i][tx] = (k < H && v < N) ? W[(size_t)k * N + v] : (uint16_t)0;
  }
  row::block_sync();
  for (int i = ty; i < 32; i += 8) {
    int v = v0 + i, k = k0 + tx;
    if (v < N_pad && k < H) Wt[(size_t)v * H + k] = tile[tx][i];
  }
}

}  // namespace

size_t row_smem_bytes(int V4, int n_lm) {
  return (size_t)V4 * ((n_lm > 1 ? 2 : 1) * sizeof(float) + sizeof(uint8_t));
}


namespace {
// Per-call defaults of the fusion bias, which the row pass combines with
// the row's own terms: lambda * log p(v) for every label (0 past V), and a
// bitmask of the labels the trie root has a child for.  One small launch at
// the start of every chunk.
__global__ void k_defaults(DecView d) {
  const Params* P = d.params;
  const float lam = P->lambda;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.V4) d.dflt[i] = (d.has_lm && i < d.V) ? lam * __ldg(d.lm.uni_logp + i) : 0.f;
  if (d.fused && i < d.N_pad) {
    // the defaults the joint kernel adds to its logits (0 from blank on)
    const bool label = i < d.V;
    d.dvec[i] = row::default_term(lam, label && d.has_lm ? __ldg(d.lm.uni_logp + i) : 0.f,
                                  label && d.has_tr && __ldg(d.tr.root_child + i) != 0, P->beta, d.tr.bonus);
  }

  if (i < (d.V4 + 31) / 32) {
    uint32_t m = 0;
    if (d.has_tr)
      for (int b = 0; b < 32; ++b) {
        const int v = i * 32 + b;
        if (v < d.V && __ldg(d.tr.root_child + v) != 0) m |= 1u << b;
      }
    d.droot[i] = m;
  }
}
}  // namespace

void launch_defaults(const DecView& d, cudaStream_t s) {
  k_defaults<<<(std::max(d.V4, d.N_pad) + 255) / 256, 256, 0, s>>>(d);
}

cudaError_t prepare_kernels(size_t row_smem) {
  // dynamic scratch plus the kernel's static shared memory may pass the
  // 48 KB default even when the scratch alone does not; the joint kernel's
  // shared-memory split, so that a row can start beside a joint CTA
  const void* f[] = {(const void*)k_row<1>, (const void*)k_row<2>, (const void*)k_row<3>, (const void*)k_row<4>};
  for (const void* k : f) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_repack(const uint16_t* W, uint16_t* Wt, int H, int N, int N_pad, cudaStream_t s) {
  dim3 grid((N_pad + 31) / 32, (H + 31) / 32), block(32, 8);
  k_repack<<<grid, block, 0, s>>>(W, Wt, H, N, N_pad);
}

void launch_open(const DecView& d, int slot, cudaStream_t s) { k_open<<<1, 32, 0, s>>>(d, slot); }

void launch_fix_records(const DecView& d, int slot, cudaStream_t s) { k_fix_records<<<1, 32, 0, s>>>(d, slot); }

namespace {
// Stateful form, stream open: zero LSTM state, the start-of-sequence step pending.
__global__ void k_open_pred(DecView d, int slot) {
  const int D = d.pred_D;
  for (int u = threadIdx.x; u < D; u += blockDim.x) {
    d.pred_h[(size_t)slot * D + u] = 0;
    d.pred_c[(size_t)slot * D + u] = 0.f;
  }
  if (threadIdx.x == 0) d.pred_fresh[slot] = 1;
}

// Stateful form: the chunk's encoder frames (from the call's parameter
// block) to the fixed buffer the projection GEMM reads by TMA.
__global__ void k_copy_enc(DecView d, int64_t n16) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint4* src = reinterpret_cast<const uint4*>(d.params->enc);
  uint4* dst = reinterpret_cast<uint4*>(d.pred_enc);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = __ldg(src + i);
}
}  // namespace

void launch_open_pred(const DecView& d, int slot, cudaStream_t s) { k_open_pred<<<1, 256, 0, s>>>(d, slot); }

void launch_copy_enc(const DecView& d, int64_t elems, cudaStream_t s, bool pdl) {
  const int64_t n16 = elems / 8;  // H_enc is a multiple of 64
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min<int64_t>((n16 + 255) / 256, 152 * 8));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k_copy_enc, d, n16);
}

void launch_row(const DecView& d, int M, int step, int mode, size_t smem, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(M);
  cfg.blockDim = dim3(kRowThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  if (d.n_lm <= 1) cudaLaunchKernelEx(&cfg, k_row<1>, d, step, mode);
  else if (d.n_lm == 2) cudaLaunchKernelEx(&cfg, k_row<2>, d, step, mode);
  else if (d.n_lm == 3) cudaLaunchKernelEx(&cfg, k_row<3>, d, step, mode);
  else cudaLaunchKernelEx(&cfg, k_row<4>, d, step, mode);
}

}  // namespace tsd
