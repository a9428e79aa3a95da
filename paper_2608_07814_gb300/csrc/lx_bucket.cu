// Bucketing: per node the ascending list of tokens whose selected experts' root
// paths contain the node (the (token, node) pairs whose products the amortised
// forward computes once, Sec. 5.1), per assignment and path level the row of
// that pair, and per expert its assignments in token order.
//
// Keys are the N nodes followed by the E experts.  Three launches: one CTA per
// block of 256 tokens records which (key, token) pairs occur as bits in shared
// memory (8 words a key) and counts them; a single CTA sums the blocks' counts
// per key, scans them into offsets and builds the tile plans of the grouped
// GEMMs; a warp per token then reads its rows off as offset + earlier blocks +
// set bits before it (so the order inside a bucket is the token order, with no
// order-dependent atomics).  Everything is deterministic.
#include <mutex>

#include "lx_internal.cuh"

namespace lx {

namespace {

constexpr int BK_TOK = 256;            // tokens of a block
constexpr int BK_WORDS = BK_TOK / 32;  // bitmap words of a key in a block

// Block b (CTA b): bits[b][key][w] bit i <-> token 256 b + 32 w + i has the key,
// and their number cnt[b][key].  A byte per (key, token) pair, cleared, marked,
// scanned and read back, took a memset and two more launches (38 us for the
// five at 8192 tokens and 256 keys, 25 for these three); word w belongs to warp
// w alone, so the shared-memory atomics meet only inside a warp.
__global__ void __launch_bounds__(BK_TOK)
k_mark_bits(const int* topk_id, int T, int k, int N, int E,
            const int* __restrict__ paths, uint32_t* __restrict__ bits, int* __restrict__ cnt) {
  extern __shared__ __align__(16) uint32_t sb[];
  const int keys = N + E, tid = threadIdx.x;
  for (int i = tid; i < keys * BK_WORDS; i += BK_TOK) sb[i] = 0u;
  pdl_wait();
  __syncthreads();
  const int t = blockIdx.x * BK_TOK + tid, w = tid >> 5;
  const uint32_t bit = 1u << (tid & 31);
  if (t < T) {
    constexpr int U = 8;  // slots whose ids and paths are in flight at once
    for (int s0 = 0; s0 < k; s0 += U) {
      int e[U];
      int4 p[U];
#pragma unroll
      for (int u = 0; u < U; ++u) e[u] = s0 + u < k ? ld_dep(topk_id + (size_t)t * k + s0 + u) : -1;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (e[u] >= E) e[u] = -1;  // invalid ids are ignored
        p[u] = e[u] >= 0 ? __ldg(reinterpret_cast<const int4*>(paths) + e[u]) : make_int4(-1, -1, -1, -1);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (e[u] < 0) continue;
        atomicOr(&sb[(N + e[u]) * BK_WORDS + w], bit);
        const int q[LX_MAX_DEPTH] = {p[u].x, p[u].y, p[u].z, p[u].w};
#pragma unroll
        for (int l = 0; l < LX_MAX_DEPTH; ++l)
          if (q[l] >= 0) atomicOr(&sb[q[l] * BK_WORDS + w], bit);
      }
    }
  }
  __syncthreads();
  uint4* gb = reinterpret_cast<uint4*>(bits + (size_t)blockIdx.x * keys * BK_WORDS);
  for (int key = tid; key < keys; key += BK_TOK) {
    const uint4 a = reinterpret_cast<const uint4*>(sb)[2 * key];
    const uint4 b = reinterpret_cast<const uint4*>(sb)[2 * key + 1];
    gb[2 * key] = a;
    gb[2 * key + 1] = b;
    cnt[(size_t)blockIdx.x * keys + key] = __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w) +
                                           __popc(b.x) + __popc(b.y) + __popc(b.z) + __popc(b.w);
  }
}
static_assert(BK_WORDS == 8 && LX_MAX_DEPTH == 4, "two 16-byte pieces a key, one a path");

// number of tokens before t that have the key (pre: those of earlier blocks)
__device__ __forceinline__ int rank_before(const uint32_t* bits, const int* pre, int keys, int key, int t) {
  const size_t row = (size_t)(t / BK_TOK) * keys + key;
  const uint4 a = ld_dep(reinterpret_cast<const uint4*>(bits) + 2 * row);
  const uint4 b = ld_dep(reinterpret_cast<const uint4*>(bits) + 2 * row + 1);
  const uint32_t v[BK_WORDS] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  const int w = (t % BK_TOK) >> 5;
  const uint32_t below = (1u << (t & 31)) - 1u;
  int r = ld_dep(pre + row);
#pragma unroll
  for (int j = 0; j < BK_WORDS; ++j) r += __popc(v[j] & (j < w ? 0xffffffffu : j == w ? below : 0u));
  return r;
}

struct PlanArgs {
  int n_items[N_PLANS];
  OpShape shape[N_PLANS];
  int bm[N_PLANS], bn[N_PLANS];  // token rows and output columns per tile
  int n_plans;
  int first;                      // plan p fills tile-plan slot first + p
};

// tiles of one node in one plan
__device__ __forceinline__ int plan_tiles(const PlanArgs& pa, int p, int r, int rows) {
  const OpShape sh = pa.shape[p];
  const int Ng = sh.n_const + sh.n_rank * r;
  const int ncol = (Ng + pa.bn[p] - 1) / pa.bn[p];
  return ((rows + pa.bm[p] - 1) / pa.bm[p]) * sh.groups * ncol;
}



// Work items of the streaming launches: one (node, token block) pair per
// `blk` rows of every active node's bucket, in node-table order, packed as
// node * STREAM_DEP_TB + block.  blk = 0 (batches the streaming kernels do not
// take) publishes an empty list.  One warp; which = 0: the anchors, 1: the
// corrections (their items follow the anchors' area).
__device__ void publish_active(const int* cnt, const int* list, int n, int which, int n_anchor, int blk,
                               int* act, int* act_n) {
  const int lane = threadIdx.x & 31;
  int* out = act + (which == 0 ? 0 : n_anchor * STREAM_DEP_TB);
  int base = 0;
  constexpr int U = 4;  // groups of 32 nodes whose scans overlap
  for (int i0 = 0; i0 < n && blk > 0; i0 += 32 * U) {
    int node[U], nb[U], incl[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + 32 * u + lane;
      node[u] = i < n ? list[i] : -1;
      // blocks of this node's bucket (the host passes blk only for batches of
      // at most STREAM_DEP_TB blocks)
      nb[u] = incl[u] = node[u] >= 0 ? (cnt[node[u]] + blk - 1) / blk : 0;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int x = __shfl_up_sync(0xffffffffu, incl[u], o);
        if (lane >= o) incl[u] += x;
      }
    int total[U];
#pragma unroll
    for (int u = 0; u < U; ++u) total[u] = __shfl_sync(0xffffffffu, incl[u], 31);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      for (int b = 0; b < nb[u]; ++b) out[base + incl[u] - nb[u] + b] = node[u] * STREAM_DEP_TB + b;
      base += total[u];
    }
  }
  if (lane == 0) act_n[which] = base;
}

// One warp: exclusive offsets out[0 .. n] of counts v(i), i < n.  Four groups of
// 32 at a time, so that their scans' shuffles (about 40 cycles each) overlap.
template <typename F>
__device__ __forceinline__ void warp_offsets(int n, F v, int* out) {
  const int lane = threadIdx.x & 31;
  constexpr int U = 4;
  int carry = 0;
  for (int base = 0; base < n; base += 32 * U) {
    int x[U], incl[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + 32 * u + lane;
      x[u] = incl[u] = i < n ? v(i) : 0;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int y = __shfl_up_sync(0xffffffffu, incl[u], o);
        if (lane >= o) incl[u] += y;
      }
    int total[U];
#pragma unroll
    for (int u = 0; u < U; ++u) total[u] = __shfl_sync(0xffffffffu, incl[u], 31);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + 32 * u + lane;
      if (i < n) out[i] = carry + incl[u] - x[u];
      carry += total[u];
    }
  }
  if (lane == 0) out[n] = carry;
}

constexpr int OP_THREADS = 1024;
inline size_t op_smem(int keys, int N) { return sizeof(int) * ((size_t)keys + 2 * (size_t)N); }

// One CTA: every key's count and the blocks' exclusive prefixes pre[b][key],
// then, a warp each, the node offsets, the expert offsets, the streaming work
// items and the tile prefix of every plan.  The layer's tables are staged
// before the wait for the preceding kernel; the plans, one after another over
// the whole CTA, had made this 9.8 us at 8192 tokens (6.6 now).
__global__ void __launch_bounds__(OP_THREADS)
k_offsets_plan(const int* cnt, int nblk, int N, int E, int* __restrict__ pre,
               int* __restrict__ key_off, const int* __restrict__ rank, int* __restrict__ tile_off,
               int max_items, PlanArgs pa, const int* __restrict__ anchors, int n_anchor,
               const int* __restrict__ corrs, int n_corr, int blk, int* __restrict__ act,
               int* __restrict__ act_n, int* __restrict__ sctr, int n_sctr) {
  extern __shared__ int osh[];
  const int keys = N + E, tid = threadIdx.x, warp = tid >> 5;
  int* kc = osh;            // [keys]
  int* srank = kc + keys;   // [N]
  int* slist = srank + N;   // [N]: the anchors, then the corrections
  for (int i = tid; i < N; i += OP_THREADS) {
    srank[i] = rank[i];
    slist[i] = i < n_anchor ? anchors[i] : corrs[i - n_anchor];
  }
  pdl_wait();
  for (int i = tid; i < n_sctr; i += OP_THREADS) sctr[i] = 0;
  for (int key = tid; key < keys; key += OP_THREADS) {
    int run = 0;
    for (int b0 = 0; b0 < nblk; b0 += 16) {
      int v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = b0 + u < nblk ? ld_dep(cnt + (size_t)(b0 + u) * keys + key) : 0;
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (b0 + u < nblk) {
          pre[(size_t)(b0 + u) * keys + key] = run;
          run += v[u];
        }
    }
    kc[key] = run;
  }
  __syncthreads();
  if (warp == 0) {
    warp_offsets(N, [&](int i) { return kc[i]; }, key_off);
  } else if (warp == 1) {
    warp_offsets(E, [&](int i) { return kc[N + i]; }, key_off + N + 1);
  } else if (warp == 2 || warp == 3) {
    if (act)
      publish_active(kc, warp == 2 ? slist : slist + n_anchor, warp == 2 ? n_anchor : n_corr, warp - 2,
                     n_anchor, blk, act, act_n);
  } else if (warp - 4 < pa.n_plans) {
    const int p = warp - 4;
    const int* items = pa.shape[p].on_anchors ? slist : slist + n_anchor;
    warp_offsets(pa.n_items[p], [&](int i) { return plan_tiles(pa, p, srank[items[i]], kc[items[i]]); },
                 tile_off + (pa.first + p) * (max_items + 1));
  }
}
static_assert(4 + N_OPS < OP_THREADS / 32 && 4 + N_OPS < 32, "a warp for every role, here and in k_bucket_small");

// The fused path's per-cluster-row tables (flat layers on the tensor-core
// path; al_g == nullptr: none): see k_assign_rows.
struct CtMeta {
  const float* topk_w;
  float* al_g;
  int* al_row;
  int* rho2al;
  const int* child_col;
  int nch, gstride, rstride, pslot;
};

// Per token its distinct rows, ascending, -1 after the last (trow [T][TOK_ROWS]),
// and the slots whose path holds each (tmask [T][TOK_ROWS]), for the tensor-core
// path's SwiGLU and combine; flat layers (CtMeta given): the anchor rows alone.
struct TokRows {
  int* trow;  // nullptr: none
  uint8_t* tmask;
};

// token rows copied into anchor-row order: x [T][vec], xg [rows][vec] (16-byte pieces)
struct XRows {
  const uint4* x;
  uint4* xg;
  long cap;
  int vec;
};

// The rows of every assignment, one warp per token (lane s = top-k slot s):
// its position in its expert's bucket (perm), the rows of the nodes on its
// path (node_row; the (token, node) pairs shared by several slots write the
// same node_tok values), and, for flat layers on the fused
// tensor-core path, the per-cluster-row tables: for each anchor row a of the
// token, al_g[a] = {dominant's gate, gates of child slots 0, 1, ...} (0 where
// not selected; slots whose experts share a node add up, in slot order) and
// al_row[a] = the child rows (-1 where not selected), written by the first
// slot of that anchor row; rho2al maps every child row to its anchor row.
// gr.xg (tensor-core path): the token's row of x is also copied to its anchor
// rows, where the anchor GEMM reads TMA boxes: once read, it is written to each
// of them.  A launch of its own, a warp per row, read x once per row (27.5 us
// beside this kernel's 14 at 8192 tokens): a forward of 8192 tokens 584 -> 572 us
// without it, of the 256-expert layer's 4096 592 -> 575.  Two tokens a CTA, so
// that a batch of hundreds spreads over the SMs.
__global__ void __launch_bounds__(256)
k_assign_rows(const int* topk_id, int T, int k, int N, int E, int D,
              const int* __restrict__ paths, const int* __restrict__ path_len,
              const int* key_off, const uint32_t* bits, const int* pre, int* __restrict__ node_tok,
              int* __restrict__ perm, int* __restrict__ node_row, const CtMeta cm, const TokRows tr,
              const XRows gr) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= T) return;
  const size_t a = (size_t)t * k + lane;
  int e = lane < k ? ld_dep(topk_id + a) : -1, len = 0;
  if (e < 0 || e >= E) e = -1;
  const unsigned twins = __match_any_sync(0xffffffffu, e);
  if (e >= 0) {
    len = path_len[e];
    if (lane == __ffs(twins) - 1)  // a repeated id counts once, with its first slot
      perm[ld_dep(key_off + N + 1 + e) + rank_before(bits, pre, N + E, N + e, t)] = (int)a;
  }
  int arow = -1;  // the anchor's row: the last level
  int r0 = -1, r1 = -1, n0 = -1, ev = -1;  // ev: entry `lane` = slot lane / D, level lane % D
#pragma unroll
  for (int l = 0; l < LX_MAX_DEPTH; ++l) {
    if (l >= D) break;
    int row = -1;
    if (l < len) {
      const int n = paths[e * LX_MAX_DEPTH + l];
      row = ld_dep(key_off + n) + rank_before(bits, pre, N + E, n, t);
      node_tok[row] = t;
      if (l == 0) n0 = n;
      if (l == len - 1) arow = row;
    }
    if (lane < k) node_row[a * D + l] = row;
    if (l == 0) r0 = row;
    if (l == 1) r1 = row;
    if (tr.tmask) {
      const int q = __shfl_sync(0xffffffffu, row, min(lane / D, 31));
      if (lane % D == l && lane < k * D) ev = q;
    }
  }
  if (tr.tmask) {
    // distinct rows: the first entry of each writes it at its rank
    const unsigned same = __match_any_sync(0xffffffffu, ev);
    const bool first = ev >= 0 && lane == __ffs(same) - 1;
    const unsigned fm = __ballot_sync(0xffffffffu, first);
    int rank = 0;
    for (unsigned b = fm; b; b &= b - 1) rank += __shfl_sync(0xffffffffu, ev, __ffs(b) - 1) < ev;
    unsigned slots = 0;
    for (int sl = 0; sl < k; ++sl)
      if ((same >> (sl * D)) & ((1u << D) - 1u)) slots |= 1u << sl;
    if (first) {
      tr.trow[(size_t)t * TOK_ROWS + rank] = ev;
      tr.tmask[(size_t)t * TOK_ROWS + rank] = (uint8_t)slots;
    }
    if (lane >= __popc(fm)) tr.trow[(size_t)t * TOK_ROWS + lane] = -1;
  }
  if (gr.xg) {
    constexpr int U = 8;  // 16-byte loads in flight a lane
    const unsigned same = __match_any_sync(0xffffffffu, arow);
    const unsigned lead = __ballot_sync(0xffffffffu, arow >= 0 && arow < gr.cap && lane == __ffs(same) - 1);
    const uint4* src = gr.x + (size_t)t * gr.vec;
    for (int c0 = 0; lead && c0 < gr.vec; c0 += 32 * U) {
      const int i0 = c0 + lane;
      uint4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + 32 * u < gr.vec) v[u] = ld_dep(src + i0 + 32 * u);
      for (unsigned b = lead; b; b &= b - 1) {
        uint4* dst = gr.xg + (size_t)__shfl_sync(0xffffffffu, arow, __ffs(b) - 1) * gr.vec;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i0 + 32 * u < gr.vec) dst[i0 + 32 * u] = v[u];
      }
    }
  }
  if (!cm.al_g) return;
  // flat layers: a path is [anchor] (the dominant) or [member, anchor]
  const bool member = len >= 2;
  const int an = lane < k && e >= 0 ? (member ? r1 : r0) : -1;
  const int j = member ? cm.child_col[n0] / cm.pslot : -1;
  const float g = an >= 0 ? cm.topk_w[a] : 0.f;
  if (member) cm.rho2al[r0] = an;
  const unsigned same = __match_any_sync(0xffffffffu, an);
  const bool leader = an >= 0 && lane == __ffs(same) - 1;
  float rg[1 + CT_MAX_CH];
  int rr[CT_MAX_CH];
#pragma unroll
  for (int i = 0; i <= CT_MAX_CH; ++i) rg[i] = 0.f;
#pragma unroll
  for (int i = 0; i < CT_MAX_CH; ++i) rr[i] = -1;
  for (int sl = 0; sl < k; ++sl) {
    const int as = __shfl_sync(0xffffffffu, an, sl), js = __shfl_sync(0xffffffffu, j, sl);
    const int rs = __shfl_sync(0xffffffffu, r0, sl);
    const float gs = __shfl_sync(0xffffffffu, g, sl);
    if (as == an && as >= 0) {
#pragma unroll
      for (int i = 0; i <= CT_MAX_CH; ++i)
        if (i == js + 1) rg[i] += gs;
#pragma unroll
      for (int i = 0; i < CT_MAX_CH; ++i)
        if (i == js) rr[i] = rs;
    }
  }
  {
    const unsigned lm = __ballot_sync(0xffffffffu, leader);
    int rank = 0;
    for (unsigned b = lm; b; b &= b - 1) rank += __shfl_sync(0xffffffffu, an, __ffs(b) - 1) < an;
    if (leader) tr.trow[(size_t)t * TOK_ROWS + rank] = an;
    if (lane >= __popc(lm)) tr.trow[(size_t)t * TOK_ROWS + lane] = -1;
  }
  if (leader) {
#pragma unroll
    for (int i = 0; i <= CT_MAX_CH; ++i)
      if (i <= cm.nch) cm.al_g[(size_t)an * cm.gstride + i] = rg[i];
#pragma unroll
    for (int i = 0; i < CT_MAX_CH; ++i)
      if (i < cm.nch) cm.al_row[(size_t)an * cm.rstride + i] = rr[i];
  }
}

// ---------------------------------------------------------------------------
// Small batches (decode): top-k and the whole bucketing in one CTA, the (key,
// token) pairs as bits in shared memory (at most 8 words a key), so that counts
// and ranks are popcounts: a byte per pair and a pass of ballots over all keys
// for the ranks took 8.5 us at 64 tokens and 256 keys, 7.6 now.  Same outputs,
// same order, as the multi-kernel path above.
// ---------------------------------------------------------------------------
constexpr int SB_THREADS = 1024;
constexpr int SB_MAX_T = 256;
constexpr size_t SB_SMEM_LIMIT = 160 * 1024;

// The batches this form takes: those for which two bytes per (key, token), the ids
// and the tables fit SB_SMEM_LIMIT, about 81000 (key, token) pairs.  The bits need a
// fraction of that; the line is where the byte tables of an earlier form ended.
// Bucketing calls back to back at it and above, one CTA / three launches: 512 keys,
// 200 tokens 8.5 / 9.6 us, 256 tokens 12.5 / 10.0; 1024 keys, 128 tokens 7.7 / 11.1,
// 256 tokens 13.4 / 11.4; 2048 keys, 64 tokens 8.7 / 15.4, 256 tokens 16.9 / 15.7: a line
// by the tokens alone (up to about 200) would be the better one.
__host__ __device__ inline size_t sb_fit(int T, int k, int keys, int E, int N) {
  const size_t Tp = ((size_t)T + 15) / 16 * 16;
  return (size_t)T * k * 4 + 2 * (size_t)keys * Tp + (size_t)keys * 4 + ((size_t)keys + 2) * 4 +
         (size_t)E * (LX_MAX_DEPTH + 1) * 4 + 2 * (size_t)N * 4 + 64;
}

// shared memory: ids, bits, counts, offsets and the layer's tables
__host__ __device__ inline size_t sb_smem(int T, int k, int keys, int E, int N) {
  return 4 * ((size_t)T * k + (size_t)keys * ((T + 31) / 32) + (size_t)keys + (size_t)keys + 2 +
              (size_t)E * (LX_MAX_DEPTH + 1) + 2 * (size_t)N);
}

__global__ void __launch_bounds__(SB_THREADS)
k_bucket_small(const float* logits, const int* ids_in, int T, int k,
               int E, int N, int D, const int* __restrict__ paths,
               const int* __restrict__ path_len, const int* __restrict__ rank,
               int* __restrict__ topk_id, float* __restrict__ topk_w, int* __restrict__ key_off_g,
               int* __restrict__ node_tok, int* __restrict__ node_row,
               int* __restrict__ perm, int* __restrict__ tile_off, int max_items, PlanArgs pa,
               const int* __restrict__ anchors, int n_anchor, const int* __restrict__ corrs,
               int n_corr, int blk, int* __restrict__ act, int* __restrict__ act_n,
               int* __restrict__ sctr, int n_sctr) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int keys = N + E;
  const int W = (T + 31) >> 5;  // words of a key
  int* ids = reinterpret_cast<int*>(sm);
  uint32_t* bits = reinterpret_cast<uint32_t*>(ids + T * k);  // [keys][W]
  int* cnt = reinterpret_cast<int*>(bits + keys * W);
  int* off = cnt + keys;
  int* spaths = off + keys + 2;                 // [E][LX_MAX_DEPTH]
  int* splen = spaths + E * LX_MAX_DEPTH;       // [E]
  int* srank = splen + E;                       // [N]
  int* slist = srank + N;                       // [N]: the anchors, then the corrections
  const int tid = threadIdx.x, nth = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, nw = nth >> 5;
  // Before the wait for the preceding kernel: cleared bits and the layer's
  // tables (constants of the layer) staged in shared memory.
  for (int i = tid; i < keys * W; i += nth) bits[i] = 0u;
  {
    const int n_paths = E * LX_MAX_DEPTH, n_tab = n_paths + E + N;
    for (int i = tid; i < n_tab + N; i += nth) {
      if (i < n_paths) spaths[i] = paths[i];
      else if (i < n_paths + E) splen[i - n_paths] = path_len[i - n_paths];
      else if (i < n_tab) srank[i - n_paths - E] = rank[i - n_paths - E];
      else if (i < n_tab + n_anchor) slist[i - n_tab] = anchors[i - n_tab];
      else slist[i - n_tab] = corrs[i - n_tab - n_anchor];
    }
  }
  pdl_wait();
  if (!logits)  // the given ids (written by the preceding kernel)
    for (int i = tid; i < T * k; i += nth) ids[i] = ld_dep(ids_in + i);
  // 1. routing (or the given ids)
  if (logits) {
    for (int t = warp; t < T; t += nw) {
      int id;
      float w;
      warp_topk(logits + (size_t)t * E, E, k, id, w);
      if (lane < k) {
        ids[t * k + lane] = id;
        topk_id[(size_t)t * k + lane] = id;
        topk_w[(size_t)t * k + lane] = w;
      }
    }
  }
  __syncthreads();
  // 2. the pairs
  for (int a = tid; a < T * k; a += nth) {
    const int t = a / k, e = ids[a], w = t >> 5;
    const uint32_t bit = 1u << (t & 31);
    if (e < 0 || e >= E) continue;
    atomicOr(&bits[(N + e) * W + w], bit);
    const int len = splen[e];
    for (int l = 0; l < len; ++l) atomicOr(&bits[spaths[e * LX_MAX_DEPTH + l] * W + w], bit);
  }
  __syncthreads();
  // 3. counts
  for (int key = tid; key < keys; key += nth) {
    int c = 0;
    for (int w = 0; w < W; ++w) c += __popc(bits[key * W + w]);
    cnt[key] = c;
  }
  // tokens before t that have the key
  auto rank_of = [&](int key, int t) {
    const uint32_t* b = bits + key * W;
    const int w = t >> 5;
    int r = __popc(b[w] & ((1u << (t & 31)) - 1u));
    for (int j = 0; j < w; ++j) r += __popc(b[j]);
    return r;
  };
  __syncthreads();
  // 4. node offsets (warp 0), expert offsets (warp 1) and, from the same counts,
  // the streaming work items (warps 2 and 3) and the tile plans (a warp each); the
  // others clear the counters
  if (warp == 0) {
    warp_offsets(N, [&](int i) { return cnt[i]; }, off);
  } else if (warp == 1) {
    warp_offsets(E, [&](int i) { return cnt[N + i]; }, off + N + 1);
  } else if (warp < 4) {
    publish_active(cnt, warp == 2 ? slist : slist + n_anchor, warp == 2 ? n_anchor : n_corr, warp - 2, n_anchor,
                   blk, act, act_n);
  } else if (warp - 4 < pa.n_plans) {
    const int p = warp - 4;
    warp_offsets(pa.n_items[p], [&](int i) {
      const int n = pa.shape[p].on_anchors ? slist[i] : slist[n_anchor + i];
      return plan_tiles(pa, p, srank[n], cnt[n]);
    }, tile_off + (pa.first + p) * (max_items + 1));
  } else {
    const int first = 32 * (4 + pa.n_plans);
    for (int i = tid - first; i < n_sctr; i += nth - first) sctr[i] = 0;
  }
  __syncthreads();
  for (int i = tid; i < keys + 2; i += nth) key_off_g[i] = off[i];
  // 5. scatter from the assignments: bucket rows, node rows, permutation
  for (int a = tid; a < T * k; a += nth) {
    const int t = a / k, e = ids[a];
    const bool valid = e >= 0 && e < E;
    const int len = valid ? splen[e] : 0;
    if (valid) perm[off[N + 1 + e] + rank_of(N + e, t)] = a;
    for (int l = 0; l < D; ++l) {
      int row = -1;
      if (l < len) {
        const int n = spaths[e * LX_MAX_DEPTH + l];
        row = off[n] + rank_of(n, t);
        node_tok[row] = t;   // (t, n) pairs shared by several slots write the same values
      }
      node_row[(size_t)a * D + l] = row;
    }
  }
}

}  // namespace

int bucket_blocks(int T) { return (T + BK_TOK - 1) / BK_TOK; }
int bucket_words() { return BK_WORDS; }

// Plans for slots [first, first + n_plans): 0 = the generic GEMMs' six ops,
// PLAN_TC = the tensor-core GEMMs' six ops.
static PlanArgs make_plans(const lx_layer* L, int n_plans, int first = 0) {
  PlanArgs pa;
  pa.n_plans = n_plans;
  pa.first = first;
  for (int p = 0; p < n_plans; ++p) {
    const int slot = first + p;
    const int op = slot % N_OPS;
    pa.shape[p] = op_shape(L, op);
    pa.n_items[p] = pa.shape[p].on_anchors ? L->n_anchor : L->n_corr;
    pa.bm[p] = slot < PLAN_TC ? G_BM : tc_tile_rows(L, op);
    pa.bn[p] = slot < PLAN_TC ? G_BN : tc_tile_cols();
    if (L->ct && slot == PLAN_TC + OP_UP_U) {
      // the fused correction + SwiGLU kernel takes this slot: tiles of 128
      // cluster rows x CT_CW d_ff columns over the anchors
      pa.shape[p] = OpShape{L->I, 0, 0, 0, 1, 1};
      pa.n_items[p] = L->n_anchor;
      pa.bm[p] = 128;
      pa.bn[p] = CT_CW;
    }
  }
  return pa;
}

// Token rows per streaming work item, or 0 for batches the streaming kernels
// do not take (more blocks than the dependency counters cover).
static int stream_item_rows(int T) {
  const int blk = stream_tile_tokens();
  return T <= STREAM_DEP_TB * blk ? blk : 0;
}

bool bucket_small_fits(const lx_layer* L, int T, int k) {
  return T <= SB_MAX_T &&
         sb_fit(T, k, L->N + L->E, L->E, L->N) <= SB_SMEM_LIMIT;
}

lx_status launch_bucket_small(lx_layer* L, const float* logits, const int* ids_in, int T, int k,
                              int* topk_id, float* topk_w, cudaStream_t s, bool plans) {
  Workspace& w = L->ws;
  const size_t smem = sb_smem(T, k, L->N + L->E, L->E, L->N);
  const PlanArgs pa = make_plans(L, plans ? N_OPS : 0);
  static bool done[64] = {};
  LX_CUDA(smem_cap_once((const void*)k_bucket_small, (int)SB_SMEM_LIMIT, L->device, done));
  ProfScope ps(L, s, logits ? "topk_bucket_small" : "bucket_small");
  launch_k(L, k_bucket_small, 1, SB_THREADS, smem, s, logits, ids_in, T, k, L->E, L->N, L->max_depth,
                                             L->d_paths, L->d_path_len, L->d_rank, topk_id, topk_w,
                                             w.key_off, w.node_tok, w.node_row, w.perm,
                                             w.tile_off, op_max_items(L), pa, L->d_anchors,
                                             L->n_anchor, L->d_corrs, L->n_corr,
                                             stream_item_rows(T), w.act, w.act_n, w.sctr,
                                             sctr_ints(L));
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

static lx_status mark_bits_cap(const lx_layer* L, size_t* smem) {
  *smem = sizeof(uint32_t) * BK_WORDS * (size_t)(L->N + L->E);  // at most 160 KB (5120 keys)
  static bool done[64] = {};
  LX_CUDA(smem_cap_once((const void*)k_mark_bits, 200 * 1024, L->device, done));
  static bool done_o[64] = {};
  LX_CUDA(smem_cap_once((const void*)k_offsets_plan, 100 * 1024, L->device, done_o));
  return LX_OK;
}

lx_status launch_bucket(lx_layer* L, const int* topk_id, int T, int k, cudaStream_t s,
                        int plan_first, const void* x) {
  Workspace& w = L->ws;
  const int keys = L->N + L->E, nblk = bucket_blocks(T);
  size_t smem = 0;
  LX_TRY(mark_bits_cap(L, &smem));
  {
    ProfScope ps(L, s, "bucket_mark");
    launch_k(L, k_mark_bits, nblk, BK_TOK, smem, s, topk_id, T, k, L->N, L->E, L->d_paths, w.bits,
             w.blk_cnt);
    LX_CUDA(cudaGetLastError());
  }
  {
    const PlanArgs pa = plan_first < 0 ? make_plans(L, 0) : make_plans(L, N_OPS, plan_first);
    ProfScope ps(L, s, "bucket_offsets");
    launch_k(L, k_offsets_plan, 1, OP_THREADS, op_smem(keys, L->N), s, w.blk_cnt, nblk, L->N, L->E,
             w.blk_pre, w.key_off, L->d_rank, w.tile_off, op_max_items(L), pa, L->d_anchors, L->n_anchor,
             L->d_corrs, L->n_corr, stream_item_rows(T), w.act, w.act_n, w.sctr, sctr_ints(L));
    LX_CUDA(cudaGetLastError());
  }
  {
    // the fused tensor-core path of flat layers also takes its per-cluster-row
    // tables from this pass
    CtMeta cm{};
    if (L->ct && plan_first == PLAN_TC) {
      cm.topk_w = w.topk_w;
      cm.al_g = w.al_g;
      cm.al_row = w.al_row;
      cm.rho2al = w.rho2al;
      cm.child_col = L->d_child_col;
      cm.nch = L->ct_nch;
      cm.gstride = ct_gstride(L);
      cm.rstride = ct_rstride(L);
      cm.pslot = 2 * std::max(1, L->max_rank);
    }
    TokRows tr{};
    if (plan_first == PLAN_TC) {
      tr.trow = w.trow;
      if (!L->ct) tr.tmask = w.tmask;
    }
    XRows gr{};
    if (plan_first == PLAN_TC) {
      gr.x = static_cast<const uint4*>(x);
      gr.xg = reinterpret_cast<uint4*>(w.xg);
      gr.cap = w.rows_cap;
      gr.vec = L->H / 8;
    }
    ProfScope ps(L, s, "bucket_rows");
    launch_k(L, k_assign_rows, (unsigned)((T + 1) / 2), 64, 0, s, topk_id, T, k, L->N, L->E,
             L->max_depth, L->d_paths, L->d_path_len, w.key_off, w.bits, w.blk_pre, w.node_tok,
             w.perm, w.node_row, cm, tr, gr);
    LX_CUDA(cudaGetLastError());
  }
  return LX_OK;
}

}  // namespace lx

// ---------------------------------------------------------------------------
// lx_bucket_noalloc: the same kernels, with every temporary buffer carved out
// of one static device array instead of the layer's (cudaMalloc'd) workspace.
// ---------------------------------------------------------------------------
namespace lx {
namespace {

// The scratch itself.  In host code this name is only a handle for
// cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_bucket_scratch[LX_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_addr[kMaxDevices] = {};

// Device address of g_bucket_scratch on `device` (which must be current).
lx_status scratch_address(int device, void** out) {
  if (device < 0 || device >= kMaxDevices) return fail(LX_ERR_UNSUPPORTED, "device id above 63");
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_addr[device]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_bucket_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_bucket_scratch)");
    g_scratch_addr[device] = p;
  }
  *out = g_scratch_addr[device];
  return LX_OK;
}

size_t round256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

}  // namespace lx

extern "C" lx_status lx_bucket_noalloc(lx_layer* L, const int32_t* topk_id, int32_t T, int32_t k,
                                       int32_t* node_off, int32_t* node_tok, int32_t* node_row,
                                       int32_t* expert_off, int32_t* perm, void* stream) {
  using namespace lx;
  if (!L) return fail(LX_ERR_ARG, "layer is NULL");
  if (T < 0) return fail(LX_ERR_ARG, "T < 0");
  if (k < 1 || k > LX_MAX_K || k > L->E) return fail(LX_ERR_ARG, "k must be in 1..min(E, LX_MAX_K)");
  cudaStream_t s = (cudaStream_t)stream;
  if (T == 0) {
    // no assignments: every bucket is empty, so both offset arrays are zero
    if (node_off) LX_CUDA(cudaMemsetAsync(node_off, 0, sizeof(int) * (L->N + 1), s));
    if (expert_off) LX_CUDA(cudaMemsetAsync(expert_off, 0, sizeof(int) * (L->E + 1), s));
    return LX_OK;
  }
  if (!topk_id || !node_off || !node_tok || !node_row || !expert_off || !perm)
    return fail(LX_ERR_ARG, "NULL topk_id or output pointer");
  int dev = -1;
  LX_CUDA(cudaGetDevice(&dev));
  if (dev != L->device) return fail(LX_ERR_ARG, "the layer's device must be current");

  // The admitted batches: those whose marks and ranks (a byte and an int per key
  // and token), counts, offsets and row->node table fit the array, as the header
  // states.  The kernels now need less (bits and block counts), carved below.
  const long Tp = ((long)T + 15) / 16 * 16;
  const long keys = (long)L->N + L->E;
  const long D = L->max_depth;
  const size_t b_marks = round256((size_t)keys * Tp);
  const size_t b_rank = round256(sizeof(int) * (size_t)keys * Tp);
  const size_t b_cnt = round256(sizeof(int) * (size_t)keys);
  const size_t b_off = round256(sizeof(int) * (size_t)(keys + 2));
  const size_t b_rown = round256(sizeof(int) * (size_t)T * k * D);
  const size_t need = b_marks + b_rank + b_cnt + b_off + b_rown;
  if (need > (size_t)LX_NOALLOC_SCRATCH_BYTES)
    return fail(LX_ERR_SHAPE, "lx_bucket_noalloc: T=" + std::to_string(T) + " needs " +
                                  std::to_string(need) + " scratch bytes, the fixed array has " +
                                  std::to_string((size_t)LX_NOALLOC_SCRATCH_BYTES));
  void* base = nullptr;
  LX_TRY(scratch_address(dev, &base));
  const int nblk = bucket_blocks(T);
  char* p = static_cast<char*>(base);
  uint32_t* bits = reinterpret_cast<uint32_t*>(p);
  int* cnt = reinterpret_cast<int*>(p += round256(sizeof(uint32_t) * BK_WORDS * (size_t)keys * nblk));
  int* pre = reinterpret_cast<int*>(p += round256(sizeof(int) * (size_t)keys * nblk));
  int* key_off = reinterpret_cast<int*>(p += round256(sizeof(int) * (size_t)keys * nblk));
  const size_t used = (size_t)(p - static_cast<char*>(base)) + b_off;
  if (used > (size_t)LX_NOALLOC_SCRATCH_BYTES)
    return fail(LX_ERR_SHAPE, "lx_bucket_noalloc: scratch layout exceeds the fixed array");

  size_t smem = 0;
  LX_TRY(mark_bits_cap(L, &smem));
  k_mark_bits<<<nblk, BK_TOK, smem, s>>>(topk_id, T, k, L->N, L->E, L->d_paths, bits, cnt);
  LX_CUDA(cudaGetLastError());
  const PlanArgs pa = make_plans(L, 0);
  k_offsets_plan<<<1, OP_THREADS, op_smem((int)keys, L->N), s>>>(
      cnt, nblk, L->N, L->E, pre, key_off, L->d_rank, nullptr, op_max_items(L), pa, L->d_anchors,
      L->n_anchor, L->d_corrs, L->n_corr, 0, nullptr, nullptr, nullptr, 0);
  LX_CUDA(cudaGetLastError());
  k_assign_rows<<<(unsigned)((T + 7) / 8), 256, 0, s>>>(topk_id, T, k, L->N, L->E, L->max_depth,
                                                        L->d_paths, L->d_path_len, key_off, bits, pre,
                                                        node_tok, perm, node_row, CtMeta{},
                                                        TokRows{}, XRows{});
  LX_CUDA(cudaGetLastError());
  LX_CUDA(cudaMemcpyAsync(node_off, key_off, sizeof(int) * (L->N + 1), cudaMemcpyDeviceToDevice, s));
  LX_CUDA(cudaMemcpyAsync(expert_off, key_off + L->N + 1, sizeof(int) * (L->E + 1),
                          cudaMemcpyDeviceToDevice, s));
  return LX_OK;
}
