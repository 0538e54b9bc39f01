// Acceptance of one tree call, shared by the frame kernel and the batched path.
#pragma once
#include "mcd_internal.cuh"
#include "mcd_sampler.cuh"

namespace mcd {

// What the step reads and where its results go.
struct TreeCall {
  const TreeDef* tree;
  const DevState* st;                       // the state the call ran with (a copy: the step rewrites it)
  const int (*cand)[kMaxTreeRank];          // candidates of the call's nodes
  const TopkRec* recs;                      // [row][1 + draft]
  const float* logits;                      // [row][kMaxDraft + 1][V]
  int heads;                                // LM heads to count
  int passes;                               // weight passes of the call
  unsigned stream_id, frame_id;
  int* codes_out;
  mcd_frame_stats* stats;
  uint8_t* trace;
};

// Call row whose draft logits gave the next candidates, and their depths.
struct TreeDrafts {
  int row, n;
};

// Acceptance step of a tree call (one stream, by the 256 consumer threads of one CTA).
// One warp walks the tree from the first row: the children of the current node are tested
// in rank order, test i keeping its candidate x iff U * S' < 2^53 * W_x, S' being the
// node's weight sum without the candidates rejected so far (one-hot draft distributions);
// a kept child continues the walk, otherwise a code is drawn from the remainder (purpose 0)
// and the call ends.  Then: the next call's candidates (the top-m ids by logit of each
// draft distribution of the last visited row), the kept nodes' K / V moved to their
// positions, the state update and the trace.
static __device__ __forceinline__ TreeDrafts accept_tree_call(const FrameParams& p, const TreeCall& in) {
  const DevState& st0 = *in.st;
  const TreeDef& tree = *in.tree;
  const int a = st0.a, pos0 = st0.pos0, n_rows = st0.n_rows, round = st0.round;
  const unsigned sid = in.stream_id, fid = in.frame_id;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const TopkRec* cur = in.recs;
  __shared__ int t_emit[kMaxDraft + 1], t_path[kMaxDraft + 1], t_path_row[kMaxDraft + 1], t_res[4];
  __shared__ int t_next[kMaxDraft][kMaxTreeRank];
  if (warp == 0) {
    int node = -1, row = st0.first_head_row, n_emit = 0, plen = 0, tests = 0;
    while (true) {
      const int s = a + 1 + plen;                     // code position of the node's children
      const TopkRec* pr = cur + (size_t)row * (kMaxDraft + 1);
      unsigned long long S_rem = pr->S;
      int rej[kMaxTreeRank];
      int n_rej = 0, kept = -1, kx = -1;
      if (pos0 > 0) {
        for (int r = 0; r < kMaxTreeRank && kept < 0; ++r) {
          int ch = -1;
          for (int k = 0; k < tree.n; ++k)
            if (tree.parent[k] == node && tree.rank[k] == r) ch = k;
          if (ch < 0 || a + tree.depth[ch] > p.P) continue;
          const int x = in.cand[tree.depth[ch] - 1][r];
          const unsigned long long W = warp_weight(pr, x);
          const uint32_t purpose = n_rej == 0 ? (uint32_t)PURPOSE_ACCEPT : kPurposeSibling + (uint32_t)n_rej;
          const unsigned long long U = uniform_U(p.seed, sid, fid, round, s, purpose);
          ++tests;
          if (W > 0 && lt128(mul64(U, S_rem), shl53(W))) {
            kept = ch;
            kx = x;
          } else {
            rej[n_rej++] = x;
            S_rem -= W;
          }
        }
      }
      if (kept >= 0) {
        // rows are the first nodes in tree order: node i was fed at row i + 1 if it exists
        const int kr = kept + 1 < n_rows ? kept + 1 : -1;
        if (lane == 0) {
          t_emit[n_emit] = kx;
          t_path[plen] = kept;
          t_path_row[plen] = kr;
        }
        ++n_emit;
        ++plen;
        if (s == p.P || kr < 0) break;                // the last position: nothing follows
        node = kept;
        row = kr;
        continue;
      }
      if (s <= p.P) {
        const int x = warp_draw_excluding(pr, rej, n_rej, S_rem, uniform_U(p.seed, sid, fid, round, s, PURPOSE_TARGET));
        if (lane == 0) t_emit[n_emit] = x;
        ++n_emit;
      }
      break;
    }
    if (lane == 0) {
      t_res[0] = n_emit;
      t_res[1] = plen;
      t_res[2] = row;
      t_res[3] = tests;
    }
  }
  consumer_sync();
  const int n_emit = t_res[0], plen = t_res[1], drow = t_res[2];
  const int a_new = a + n_emit, n_next = min(tree.maxd, p.P - a_new);
  // next candidates: warp j - 1 ranks the draft distribution of depth j of row drow (the
  // record's ids with their fp32 logits; largest logit first, ties to the lower id)
  for (int j = 1 + warp; j <= n_next; j += kConsumerWarps) {
    const TopkRec* dr = cur + (size_t)drow * (kMaxDraft + 1) + j;
    const float* lg = in.logits + ((size_t)drow * (kMaxDraft + 1) + j) * p.V;
    unsigned long long key[kDrawPerLane];
#pragma unroll
    for (int e = 0; e < kDrawPerLane; ++e) {
      const int i = lane * kDrawPerLane + e;
      key[e] = 0ull;
      if (i < dr->n) {
        const int id = dr->ids[i];
        key[e] = ((unsigned long long)f32_key(__ldcg(lg + id)) << 32) | (0xFFFFFFFFu - (uint32_t)id);
      }
    }
    for (int r = 0; r < tree.m[j - 1]; ++r) {
      unsigned long long best = 0ull;
#pragma unroll
      for (int e = 0; e < kDrawPerLane; ++e) best = key[e] > best ? key[e] : best;
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, best, off);
        best = o > best ? o : best;
      }
#pragma unroll
      for (int e = 0; e < kDrawPerLane; ++e)
        if (key[e] == best) key[e] = 0ull;
      if (lane == 0) t_next[j - 1][r] = best ? (int)(0xFFFFFFFFu - (uint32_t)(best & 0xFFFFFFFFull)) : -1;
    }
  }
  // the kept nodes' keys and values: slot kMaxPos + row -> position a + 2 + t
  {
    int n_mv = 0;
    for (int t = 0; t < plen; ++t) n_mv += t_path_row[t] >= 0 ? 1 : 0;
    const int D4 = p.D >> 2, per = p.L * p.NKV * n_mv * D4;
    for (int i = threadIdx.x; i < 2 * per; i += kConsumerThreads) {
      const bool isv = i >= per;
      const int k = isv ? i - per : i;
      const int d4 = k % D4, t = (k / D4) % n_mv, lg = k / (D4 * n_mv);   // lg = layer * NKV + kv head
      float* base = (isv ? p.vcache : p.kcache) + (size_t)lg * p.kv_slots * p.D;
      const float4 v = __ldcg(reinterpret_cast<const float4*>(base + (size_t)(kMaxPos + t_path_row[t]) * p.D) + d4);
      reinterpret_cast<float4*>(base + (size_t)(a + 2 + t) * p.D)[d4] = v;
    }
  }
  consumer_sync();
  // state of the next call
  if (threadIdx.x == 0) {
    int nv = 0, md = 0;
    for (int i = 0; i < tree.n; ++i) {
      const int d = tree.depth[i];
      if (d <= n_next && a_new + d < p.P) {
        ++nv;
        md = max(md, d);
      }
    }
    DevState* st = p.st;
    int* codes_out = in.codes_out;
    for (int t = 0; t < n_emit; ++t) {
      st->codes[a + 1 + t] = t_emit[t];
      if (codes_out) codes_out[a + t] = t_emit[t];
      st->emitted_last[t] = t_emit[t];
    }
    const int calls = st0.calls + 1, heads = st0.heads_read + in.heads;
    const int kvr = st0.kv_rows + pos0 + n_rows, rf = st0.rows_fed + n_rows;
    const int drafted = st0.drafted + t_res[3], accepted = st0.accepted + plen;
    st->n_emit_last = n_emit;
    st->n_acc_last = plen;
    st->a = a_new;
    st->n_d = n_next;
    st->pos0 = a_new + 1;
    st->n_rows = 1 + nv;
    st->top_pos = a_new + 1 + md;
    st->round = round + 1;
    st->tpass = 0;
    st->first_head_row = 0;
    st->calls = calls;
    st->heads_read = heads;
    st->kv_rows = kvr;
    st->rows_fed = rf;
    st->drafted = drafted;
    st->accepted = accepted;
    st->call = st0.call + 1;
    st->done = a_new >= p.P ? 1 : 0;
    if (a_new >= p.P && in.stats) {
      mcd_frame_stats* fs = in.stats;
      fs->calls = calls;
      fs->codes = a_new;
      fs->drafted = drafted;
      fs->accepted = accepted;
      fs->status = *(volatile int*)p.err;
      fs->heads_read = heads;
      fs->kv_rows = kvr;
      fs->rows_fed = rf;
    }
  }
  for (int i = threadIdx.x; i < kMaxDraft * kMaxTreeRank; i += kConsumerThreads) {
    const int d = i / kMaxTreeRank, r = i % kMaxTreeRank;
    p.tree_cand[i] = (d < n_next && r < tree.m[d]) ? t_next[d][r] : -1;
  }
  consumer_sync();
  // optional trace: the chain record and the tree record (the caller copies the logits)
  if (in.trace && round < kMaxCalls) {
    uint8_t* tb = in.trace;
    mcd_call_trace* tr = reinterpret_cast<mcd_call_trace*>(tb) + round;
    const size_t chain_bytes = sizeof(mcd_call_trace) * kMaxCalls + (size_t)2 * kMaxCalls * kMaxRows * p.V * 4;
    mcd_tree_trace* tt = reinterpret_cast<mcd_tree_trace*>(tb + chain_bytes) + round;
    if (threadIdx.x == 0) {
      tr->a = a;
      tr->n_rows = n_rows;
      tr->pos0 = pos0;
      tr->n_drafts = t_res[3];
      // code fed at call row n: the first call is one pass of plain rows; a tree call feeds
      // c_a, then node n - 1's candidate
      auto row_id = [&](int n) {
        if (n >= n_rows) return -1;
        if (pos0 == 0) return n == 0 ? -1 : st0.codes[0];
        if (n == 0) return st0.codes[a];
        return in.cand[tree.depth[n - 1] - 1][tree.rank[n - 1]];
      };
      for (int n = 0; n < kMaxRows; ++n) tr->input_ids[n] = row_id(n);
      for (int i = 0; i < kMaxRows; ++i) tr->drafts[i] = -1;
      tr->n_acc = plen;
      tr->n_emit = n_emit;
      for (int t = 0; t < kMaxRows; ++t) tr->emitted[t] = t < n_emit ? t_emit[t] : -1;
      tr->n_next = n_next;
      for (int j = 0; j < kMaxRows; ++j) tr->next_drafts[j] = j < n_next ? t_next[j][0] : -1;
      tr->draft_row = drow;
      tt->n_rows = n_rows;
      for (int n = 0; n < kMaxTreeRows; ++n) {
        tt->row_node[n] = n >= n_rows || pos0 == 0 ? -1 : n - 1;
        tt->row_id[n] = row_id(n);
      }
      tt->n_passes = in.passes;
      tt->path_len = plen;
      for (int t = 0; t < kMaxDraft + 1; ++t) tt->path[t] = t < plen ? t_path[t] : -1;
      tt->draft_row = drow;
      tt->n_next = n_next;
      for (int d = 0; d < kMaxDraft + 1; ++d)
        for (int r = 0; r < kMaxTreeRank; ++r)
          tt->next_cand[d][r] = (d < n_next && d < kMaxDraft && r < tree.m[d]) ? t_next[d][r] : -1;
    }
  }
  consumer_sync();
  return TreeDrafts{drow, n_next};
}

}  // namespace mcd
