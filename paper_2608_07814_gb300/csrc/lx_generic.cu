// Generic expert path (fp32 intermediates and sums, every dtype and shape; bf16
// weights on mma.sync with exact products, fp32 weights on the CUDA cores).
//
// For every node n and every token t in its bucket the shared product is
// evaluated once (Sec. 5.1):
//   anchor:     h[(t,n)] = x_t [Wg;Wu]^T                       (2I values)
//   correction: P[(t,n)] = x_t [Vg|Vu],  h[(t,n)] = [Pg Ug^T | Pu Uu^T]
// then per (t, n) the SwiGLU outputs of the selected experts whose path holds n
// are aggregated with their gates (linearity of the down projection):
//   z[(t,n)] = sum_{s : n in path(e_s)} g_s * silu(sum_l h_g[(t,path_l)]) * (sum_l h_u[...])
// and the down projection is again evaluated once per (t, n):
//   anchor:     ypart[(t,n)] = z Wd^T;   correction: ypart[(t,n)] = (z Vd) Ud^T
// y_t is the sum of ypart over t's rows in ascending node order.
#include <algorithm>
#include <initializer_list>
#include <type_traits>

#include "lx_internal.cuh"

namespace lx {

namespace {

// ---------------------------------------------------------------------------
// Grouped GEMM over tiles of G_BM = 32 bucket rows x G_BN = 64 output columns.
//
// What bounds it: at the batches this path serves, the weight bytes (a bucket
// holds tens of rows, so a weight meets few of them) and, in small layers, the
// latency of a tile's chain of loads.  Hence 16-byte cp.async copies into a
// ring of GG_STAGES chunks (128 bytes of K per row: 64 bf16 or 32 fp32 weights),
// four warps a CTA and three CTAs an SM, and the products that do not depend
// on one another in one launch (up to two ops, their tiles side by side).
//
// bf16 weights: mma.sync m16n8k16, the weights as the 16-row operand and the
// rows as the 8-column one; empty 8-row groups of a ragged tile are skipped.
// An fp32 activation is split into three bf16 parts (eight significant bits
// each, together all 24), so every product is exact, and each 64-deep chunk is
// summed by the tensor core from zero and added to the fp32 sum with an ordinary
// rounded addition: the tensor core's own accumulation spans 64 products only.
// A sum that comes out a NaN is formed again by plain multiply-adds (infinite
// weights; see the epilogue).
// fp32 weights: fused multiply-adds in ascending K (4 x 4 outputs a thread).
// Measured on the Qwen3-30B-A3B-shaped layer with rank 32 at 96 tokens, whole
// forward: 1669 us with a scalar-load, single-buffered form, 195 us with this
// one (212 before the first tile of a launch was looked up, and its weights
// requested, ahead of the wait for the preceding one); the tiny fp32 layer
// (d_model 64, 256 tokens) 74.6 -> 30.6 us.
// ---------------------------------------------------------------------------
constexpr int GG_THREADS = 128;
constexpr int GG_STAGES = 4;
constexpr int GG_CTAS_PER_SM = 3;

struct GemmLaunch {
  GemmArgs op[2];
  int n_ops;
  // 1: the tile lists and buckets were complete before the preceding launch
  // (only the rows of A come from it): the first tile is looked up and its
  // weights are requested before the wait for that launch
  int early;
};

template <typename TA, typename TW>
struct GG {
  static constexpr bool MMA = sizeof(TW) == 2;
  static constexpr int BK = 128 / (int)sizeof(TW);         // K per chunk
  static constexpr int AROW = BK * (int)sizeof(TA);        // bytes of a row's chunk
  static constexpr int ALD = MMA ? AROW : AROW + 16;       // fp32 form: rows 16 bytes apart mod 128
  static constexpr int WLD = MMA ? 128 : 144;
  static constexpr int STAGE = G_BN * WLD + G_BM * ALD;
  static constexpr int SMEM = GG_STAGES * STAGE;
};

__device__ __forceinline__ void gg_cp16(uint32_t dst, const void* src, bool ok) {
  const int n = ok ? 16 : 0;  // 0 source bytes: the 16 bytes are filled with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ uint4 gg_lds(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void gg_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                       uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Position of 16-byte unit u of row m of a staged chunk.  bf16 rows (8 units):
// the 128-byte XOR swizzle.  fp32 rows beside bf16 weights (16 units): lane q
// of a half-unit (c, h) reads unit 4 q + 2 c + h, so units are stored q fastest
// and odd rows take the other 64 bytes: the eight lanes of a shared-memory phase
// (two rows, four q) touch eight distinct bank groups.
template <int UNITS>
__device__ __forceinline__ int gg_pos(int u, int m) {
  if constexpr (UNITS == 8) return u ^ (m & 7);
  else return (((u & 3) << 2) | (u >> 2)) ^ ((m & 1) << 2);
}
// x = hi + mid + lo, each part the leading eight significant bits of what is left
// (by truncation: no part overflows), two values packed as bf16; exact for |x| >=
// 2^-110 (below, what is under 2^-133, the least bf16, is cut); an infinity is hi
// alone (inf - inf would make it a NaN)
__device__ __forceinline__ float gg_rest(float x, float& head) {
  head = __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);
  return fabsf(x) == INFINITY ? 0.f : x - head;
}
__device__ __forceinline__ uint32_t gg_pack(float a, float b) {  // the upper halves
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
__device__ __forceinline__ void gg_split(uint32_t xb, uint32_t yb, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  float hx, hy, mx, my;
  const float rx = gg_rest(__uint_as_float(xb), hx), ry = gg_rest(__uint_as_float(yb), hy);
  const float lx_ = gg_rest(rx, mx), ly = gg_rest(ry, my);
  hi = gg_pack(hx, hy);
  mid = gg_pack(mx, my);
  lo = gg_pack(lx_, ly);
}

// element k of weight row c (stored in rows of K, or tiled 64 x 64)
template <typename TW>
__device__ __forceinline__ const TW* gg_weight(const TW* W, bool tiled, int c, int k, int K) {
  return tiled ? W + (((size_t)(c >> 6) * (K >> 6) + (k >> 6)) * 64 + (c & 63)) * 64 + (k & 63)
               : W + (size_t)c * K + k;
}

// One chunk of a tile's tensor-core product: NT groups of eight rows.
template <typename TA, int NT>
__device__ __forceinline__ void gg_chunk_mma(uint32_t ws, uint32_t as, float (&sum)[G_BM / 8][4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, q = lane & 3;
  float acc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[j][c] = 0.f;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    // lane q takes the eight K values 8 (2 q + c) .. of both operands
    const int u = 2 * q + c;
    const int wr = 16 * warp + g;  // wr & 7 == g
    const uint4 w0 = gg_lds(ws + wr * 128 + 16 * gg_pos<8>(u, g));
    const uint4 w1 = gg_lds(ws + (wr + 8) * 128 + 16 * gg_pos<8>(u, g));
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int m = 8 * j + g;
      if constexpr (sizeof(TA) == 2) {
        const uint4 x = gg_lds(as + m * 128 + 16 * gg_pos<8>(u, m));
        gg_mma(acc[j], w0.x, w1.x, w0.y, w1.y, x.x, x.y);
        gg_mma(acc[j], w0.z, w1.z, w0.w, w1.w, x.z, x.w);
      } else {
        const uint4 xa = gg_lds(as + m * 256 + 16 * gg_pos<16>(2 * u, m));
        const uint4 xb = gg_lds(as + m * 256 + 16 * gg_pos<16>(2 * u + 1, m));
        uint32_t hi[4], mid[4], lo[4];
        gg_split(xa.x, xa.y, hi[0], mid[0], lo[0]);
        gg_split(xa.z, xa.w, hi[1], mid[1], lo[1]);
        gg_split(xb.x, xb.y, hi[2], mid[2], lo[2]);
        gg_split(xb.z, xb.w, hi[3], mid[3], lo[3]);
        // the small parts first
        gg_mma(acc[j], w0.x, w1.x, w0.y, w1.y, lo[0], lo[1]);
        gg_mma(acc[j], w0.z, w1.z, w0.w, w1.w, lo[2], lo[3]);
        gg_mma(acc[j], w0.x, w1.x, w0.y, w1.y, mid[0], mid[1]);
        gg_mma(acc[j], w0.z, w1.z, w0.w, w1.w, mid[2], mid[3]);
        gg_mma(acc[j], w0.x, w1.x, w0.y, w1.y, hi[0], hi[1]);
        gg_mma(acc[j], w0.z, w1.z, w0.w, w1.w, hi[2], hi[3]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) sum[j][c] += acc[j][c];
}

// The sums of this thread's fragments that came out NaN (bit 4 j + c of `nan`), term
// by term in ascending K: a zero part of a split activation times an infinite weight
// is a NaN that the plain product is not.  Out of line and by value, so that the
// kernel's registers do not see it (rank 32, 96 tokens: 198 us a forward with it and
// without; 202 with the sums passed by reference, 210 in line).
__device__ __noinline__ void gg_redo_nan(unsigned nan, const float* const* arow, int rows, int cols,
                                         bool tiled, const __nv_bfloat16* W, int col0, int K, float* out,
                                         long ldo) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (; nan; nan &= nan - 1) {
    const int e = __ffs(nan) - 1, j = e >> 2, c = e & 3;
    const int m = 8 * j + 2 * (lane & 3) + (c & 1), col = 16 * warp + (lane >> 2) + (c >= 2 ? 8 : 0);
    if (m >= rows || col >= cols) continue;
    float v = 0.f;
    for (int k = 0; k < K && v == v; ++k) v = fmaf(arow[m][k], to_f32(*gg_weight(W, tiled, col0 + col, k, K)), v);
    out[(size_t)m * ldo + col] = v;
  }
}

// OPK only names the instantiation (one kernel symbol per product in profiles)
template <typename TA, typename TW, int OPK>
__global__ void __launch_bounds__(GG_THREADS, GG_CTAS_PER_SM)
k_grouped_gemm(const __grid_constant__ GemmLaunch P) {
  using C = GG<TA, TW>;
  constexpr int BK = C::BK, UA = C::AROW / 16;
  constexpr int EW = 16 / (int)sizeof(TW), EA = 16 / (int)sizeof(TA);  // elements of a unit
  if (P.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  else pdl_wait();
  bool waited = !P.early;
  extern __shared__ __align__(128) unsigned char gsm[];
  __shared__ const TA* arow[G_BM];  // the tile's rows of A (null past the bucket)
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(gsm));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tiles0 = P.op[0].tile_off[P.op[0].n_items];
  const int total = tiles0 + (P.n_ops > 1 ? P.op[1].tile_off[P.op[1].n_items] : 0);
  for (int tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const GemmArgs& o = P.op[tile >= tiles0 ? 1 : 0];
    const int t = tile >= tiles0 ? tile - tiles0 : tile;
    // item = last index with tile_off[item] <= t
    int lo = 0, hi = o.n_items;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (o.tile_off[mid] <= t) lo = mid; else hi = mid;
    }
    const int n = o.items[lo];
    const int local = t - o.tile_off[lo];
    const int r = o.rank[n];
    const int Ng = o.shape.n_const + o.shape.n_rank * r;
    const int K = o.shape.k_const + o.shape.k_rank * r;
    const int ncol = (Ng + G_BN - 1) / G_BN;
    const int per_rt = ncol * o.shape.groups;
    const int rt = local / per_rt, rem = local % per_rt;
    const int grp = rem / ncol, ct = rem % ncol;
    const int row0 = o.node_off[n] + rt * G_BM;
    const int rows = min(G_BM, o.node_off[n + 1] - row0);
    const int col0 = ct * G_BN, cols = min(G_BN, Ng - col0);
    const TW* W = reinterpret_cast<const TW*>(o.W[n]) + (size_t)grp * Ng * K;
    __syncthreads();  // the previous tile's reads of arow and of the stages are done
    if (tid < G_BM) {
      const int grow = row0 + tid;
      arow[tid] = tid < rows ? reinterpret_cast<const TA*>(o.A) +
                                   (o.gather ? (long)o.gather[grow] : (long)grow) * o.lda + (long)grp * K
                             : nullptr;
    }
    __syncthreads();
    // whole 16-byte units of K in rows that start on a 16-byte boundary; else
    // (a rank that is no multiple of eight, bf16, or of four, fp32) element loads
    const bool vec = K % EW == 0 && K % EA == 0 && o.lda % EA == 0;
    const int nch = (K + BK - 1) / BK;
    auto w_at = [&](int c, int kx) { return gg_weight(W, o.tiled, col0 + c, kx, K); };
    // what: 1 the weights, 2 the rows of A, 3 both
    auto fetch = [&](int ch, int what) {
      if (ch >= nch) return;
      const int k0 = ch * BK;
      const uint32_t ws = base + (ch % GG_STAGES) * C::STAGE, as = ws + G_BN * C::WLD;
      if (vec) {
        if (what & 1) {
#pragma unroll
          for (int i = 0; i < G_BN * 8 / GG_THREADS; ++i) {
            const int q = tid + i * GG_THREADS, c = q >> 3, u = q & 7;
            const bool ok = c < cols && k0 + u * EW < K;
            gg_cp16(ws + c * C::WLD + 16 * (C::MMA ? gg_pos<8>(u, c) : u), ok ? w_at(c, k0 + u * EW) : W, ok);
          }
        }
        if (what & 2) {
#pragma unroll
          for (int i = 0; i < G_BM * UA / GG_THREADS; ++i) {
            const int q = tid + i * GG_THREADS, m = q / UA, u = q % UA;
            const bool ok = m < rows && k0 + u * EA < K;
            gg_cp16(as + m * C::ALD + 16 * (C::MMA ? gg_pos<UA>(u, m) : u),
                    ok ? (const void*)(arow[m] + k0 + u * EA) : o.A, ok);
          }
        }
      } else {
        unsigned char* wsp = gsm + (ch % GG_STAGES) * C::STAGE;
        unsigned char* asp = wsp + G_BN * C::WLD;
        if (what & 1)
          for (int q = tid; q < G_BN * BK; q += GG_THREADS) {
            const int c = q / BK, k = q % BK, u = k / EW;
            TW v = from_f32<TW>(0.f);
            if (c < cols && k0 + k < K) v = *w_at(c, k0 + k);
            *reinterpret_cast<TW*>(wsp + c * C::WLD + 16 * (C::MMA ? gg_pos<8>(u, c) : u) + (k % EW) * sizeof(TW)) = v;
          }
        if (what & 2)
          for (int q = tid; q < G_BM * BK; q += GG_THREADS) {
            const int m = q / BK, k = q % BK, u = k / EA;
            TA v = from_f32<TA>(0.f);
            if (m < rows && k0 + k < K) v = arow[m][k0 + k];
            *reinterpret_cast<TA*>(asp + m * C::ALD + 16 * (C::MMA ? gg_pos<UA>(u, m) : u) + (k % EA) * sizeof(TA)) = v;
          }
      }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    float sum[G_BM / 8][4];  // mma: [8-row group][fragment]; fp32: [row][column]
#pragma unroll
    for (int j = 0; j < G_BM / 8; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) sum[j][c] = 0.f;
    int left = 3;  // what is left to fetch of the first chunks
    if (!waited) {
      for (int ch = 0; ch < GG_STAGES - 1; ++ch) fetch(ch, 1);
      asm volatile("griddepcontrol.wait;" ::: "memory");
      waited = true;
      left = 2;
    }
    for (int ch = 0; ch < GG_STAGES - 1; ++ch) {
      fetch(ch, left);
      commit();
    }
    const int nt = (rows + 7) / 8;
    const int tx = tid & 15, ty = tid >> 4;
    for (int ch = 0; ch < nch; ++ch) {
      asm volatile("cp.async.wait_group %0;" ::"n"(GG_STAGES - 2) : "memory");
      __syncthreads();  // chunk ch has landed, and chunk ch - 1's stage is free
      fetch(ch + GG_STAGES - 1, 3);
      commit();
      const uint32_t ws = base + (ch % GG_STAGES) * C::STAGE, as = ws + G_BN * C::WLD;
      if constexpr (C::MMA) {
        if (nt == 1) gg_chunk_mma<TA, 1>(ws, as, sum);
        else if (nt == 2) gg_chunk_mma<TA, 2>(ws, as, sum);
        else gg_chunk_mma<TA, 4>(ws, as, sum);
      } else {
        // columns tx + 16 j, rows 4 ty + i
        if (4 * ty < rows) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            float4 w[4], a[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              w[j] = *reinterpret_cast<const float4*>(gsm + (ws - base) + (tx + 16 * j) * C::WLD + 16 * u);
              a[j] = *reinterpret_cast<const float4*>(gsm + (as - base) + (4 * ty + j) * C::ALD + 16 * u);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                sum[i][j] = fmaf(a[i].x, w[j].x, sum[i][j]);
                sum[i][j] = fmaf(a[i].y, w[j].y, sum[i][j]);
                sum[i][j] = fmaf(a[i].z, w[j].z, sum[i][j]);
                sum[i][j] = fmaf(a[i].w, w[j].w, sum[i][j]);
              }
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    float* out = o.out + (size_t)row0 * o.ldo + (size_t)grp * Ng + col0;
    if constexpr (C::MMA) {
      const int g = lane >> 2, q = lane & 3;
#pragma unroll
      for (int j = 0; j < G_BM / 8; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int m = 8 * j + 2 * q + (c & 1), col = 16 * warp + g + (c >= 2 ? 8 : 0);
          if (m < rows && col < cols) out[(size_t)m * o.ldo + col] = sum[j][c];
        }
      if constexpr (sizeof(TA) == 4) {
        unsigned nan = 0;
#pragma unroll
        for (int j = 0; j < G_BM / 8; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) nan |= (sum[j][c] != sum[j][c] ? 1u : 0u) << (4 * j + c);
        if (nan) gg_redo_nan(nan, arow, rows, cols, o.tiled, W, col0, K, out, o.ldo);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (4 * ty + i < rows && tx + 16 * j < cols) out[(size_t)(4 * ty + i) * o.ldo + tx + 16 * j] = sum[i][j];
    }
  }
  // (a CTA without tiles: this grid may not complete before its predecessor)
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ float silu_f(float v) { return v / (1.f + expf(-v)); }
// the bf16 paths' SiLU: CUDA's fast exponential and division intrinsics (their
// error is far below the bf16 rounding of the operands)
__device__ __forceinline__ float silu_fast(float v) { return __fdividef(v, 1.f + __expf(-v)); }

// One CTA per token.  Its k selected experts' gated SwiGLU outputs,
//   a_s = g_s * silu(sum_l h_gate[row(s,l)]) * sum_l h_up[row(s,l)],
// are added, slot by slot in ascending order, into the z row of every node on
// the slot's path: z[(t,n)] = sum_{s : n in path(e_s)} a_s.  Each thread owns
// four columns; its per-row partial sums live in its own shared-memory slice.
constexpr int SW_T = 256;


template <typename TZ>
__device__ __forceinline__ void store4(TZ* p, float4 v);
template <>
__device__ __forceinline__ void store4<float>(float* p, float4 v) {
  *reinterpret_cast<float4*>(p) = v;
}
template <>
__device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&a);
  u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}

template <typename TZ>
__global__ void __launch_bounds__(SW_T)
k_swiglu_aggregate(const float* topk_w, const int* node_row, int T, int k, int D, const float* h, int I,
                   TZ* __restrict__ z) {
  pdl_wait();
  extern __shared__ float4 zacc[];  // [distinct rows][SW_T]
  __shared__ int rows[LX_MAX_K * LX_MAX_DEPTH], lrow[LX_MAX_K * LX_MAX_DEPTH];
  __shared__ int drow[LX_MAX_K * LX_MAX_DEPTH];
  __shared__ float gw[LX_MAX_K];
  __shared__ int nd_s;
  const int kD = k * D;
  for (int t = blockIdx.x; t < T; t += gridDim.x) {
    for (int j = threadIdx.x; j < kD; j += blockDim.x) rows[j] = ld_dep(node_row + (size_t)t * kD + j);
    for (int j = threadIdx.x; j < k; j += blockDim.x) gw[j] = ld_dep(topk_w + (size_t)t * k + j);
    __syncthreads();
    // distinct rows, numbered in order of first appearance (entry j owns the
    // number of first appearances before it)
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      int base = 0;
      for (int j0 = 0; j0 < kD; j0 += 32) {
        const int j = j0 + lane;
        const int r = j < kD ? rows[j] : -1;
        bool first = r >= 0;
        for (int q = 0; q < j && first; ++q) first = rows[q] != r;
        const uint32_t fm = __ballot_sync(0xffffffffu, first);
        if (first) {
          const int d = base + __popc(fm & ((1u << lane) - 1u));
          drow[d] = r;
        }
        base += __popc(fm);
      }
      if (lane == 0) nd_s = base;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kD; j += blockDim.x) {
      const int r = rows[j];
      int d = -1;
      if (r >= 0)
        for (int q = 0; q < nd_s; ++q)
          if (drow[q] == r) d = q;
      lrow[j] = d;
    }
    __syncthreads();
    const int nd = nd_s;
    for (int c0 = 0; c0 < I; c0 += 4 * SW_T) {
      const int i = c0 + 4 * threadIdx.x;
      if (i < I) {
        for (int d = 0; d < nd; ++d) zacc[d * SW_T + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int sl = 0; sl < k; ++sl) {
          float4 pg = make_float4(0.f, 0.f, 0.f, 0.f), pu = pg;
          for (int l = 0; l < D; ++l) {
            const int r = rows[sl * D + l];
            if (r < 0) continue;
            const float4 a = ld_dep(reinterpret_cast<const float4*>(h + (size_t)r * 2 * I + i));
            const float4 b = ld_dep(reinterpret_cast<const float4*>(h + (size_t)r * 2 * I + I + i));
            pg.x += a.x; pg.y += a.y; pg.z += a.z; pg.w += a.w;
            pu.x += b.x; pu.y += b.y; pu.z += b.z; pu.w += b.w;
          }
          const float g = gw[sl];
          const float4 act = make_float4(g * silu_f(pg.x) * pu.x, g * silu_f(pg.y) * pu.y,
                                         g * silu_f(pg.z) * pu.z, g * silu_f(pg.w) * pu.w);
          for (int l = 0; l < D; ++l) {
            const int d = lrow[sl * D + l];
            if (d < 0) continue;
            float4& acc = zacc[d * SW_T + threadIdx.x];
            acc.x += act.x; acc.y += act.y; acc.z += act.z; acc.w += act.w;
          }
        }
        for (int d = 0; d < nd; ++d) store4<TZ>(z + (size_t)drow[d] * I + i, zacc[d * SW_T + threadIdx.x]);
      }
    }
    __syncthreads();
  }
}

// y[t] = sum of ypart over t's distinct rows in ascending row (= node) order;
// each thread owns four columns and issues four rows' loads at a time.
template <typename TY>
__global__ void __launch_bounds__(256)
k_combine(const int* node_row, int k, int D, const float* ypart, int H, TY* __restrict__ y, int T) {
  pdl_wait();
  __shared__ int raw_s[LX_MAX_K * LX_MAX_DEPTH];
  __shared__ int rows_s[LX_MAX_K * LX_MAX_DEPTH];
  __shared__ int nrows_s;
  for (int t = blockIdx.x; t < T; t += gridDim.x) {
    for (int j = threadIdx.x; j < k * D; j += blockDim.x) raw_s[j] = ld_dep(node_row + (long)t * k * D + j);
    __syncthreads();
    // distinct rows in ascending order: each first occurrence takes the rank
    // of its value among the distinct values
    for (int j = threadIdx.x; j < k * D; j += blockDim.x) {
      const int r = raw_s[j];
      bool first = r >= 0;
      for (int q = 0; q < j && first; ++q) first = raw_s[q] != r;
      if (first) {
        int rank = 0;
        for (int q = 0; q < k * D; ++q) {
          const int v = raw_s[q];
          bool fq = v >= 0 && v < r;
          for (int u = 0; u < q && fq; ++u) fq = raw_s[u] != v;
          rank += fq;
        }
        rows_s[rank] = r;
      }
    }
    if (threadIdx.x < 32) {
      int cntd = 0;
      for (int j0 = 0; j0 < k * D; j0 += 32) {
        const int j = j0 + threadIdx.x;
        const int r = j < k * D ? raw_s[j] : -1;
        bool first = r >= 0;
        for (int q = 0; q < j && first; ++q) first = raw_s[q] != r;
        cntd += __popc(__ballot_sync(0xffffffffu, first));
      }
      if (threadIdx.x == 0) nrows_s = cntd;
    }
    __syncthreads();
    const int m = nrows_s;
    for (int c = 4 * threadIdx.x; c < H; c += 4 * blockDim.x) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      int q = 0;
      for (; q + 4 <= m; q += 4) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          v[u] = ld_dep(reinterpret_cast<const float4*>(ypart + (size_t)rows_s[q + u] * H + c));
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w;
        }
      }
      for (; q < m; ++q) {
        const float4 v = ld_dep(reinterpret_cast<const float4*>(ypart + (size_t)rows_s[q] * H + c));
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
      }
      store4<TY>(y + (size_t)t * H + c, acc);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Warp-per-token SwiGLU aggregation and combine (k <= 8, k * D <= 32).
//
// A warp reads the token's k * D path rows (node_row), finds its distinct rows
// with match/ballot/shuffle (no block barrier), and keeps them, in ascending
// order, in a per-warp shared-memory block with, for each distinct row, the
// bit mask of the top-k slots whose path passes through it.
// ---------------------------------------------------------------------------
constexpr int WT_WARPS = 8;
constexpr int WT_SLOTS = 8;

struct WarpRows {
  int rows[32];       // entry j = slot j / D, level j % D (-1: none)
  int lrow[32];       // entry j: index of its row among the distinct rows (-1: none)
  int drow[32];       // distinct rows, ascending
  unsigned dmask[32]; // slots whose path holds distinct row d
  float g[WT_SLOTS];
  int nd;
  unsigned anchor_rows;  // bit d: distinct row d belongs to an anchor
};

// v: entry `lane` of the token's node rows (-1 for lanes >= kD)
__device__ __forceinline__ void warp_token_rows(int v, int kD, int D, WarpRows& wr) {
  const int lane = threadIdx.x & 31;
  const int key = v >= 0 ? v : INT_MAX;
  const unsigned same = __match_any_sync(0xffffffffu, key);
  const bool first = key != INT_MAX && lane == __ffs(same) - 1;
  const unsigned fm = __ballot_sync(0xffffffffu, first);
  // rank of this entry's row among the distinct rows (the loop is warp-uniform)
  int rank = 0;
  for (unsigned b = fm; b; b &= b - 1) {
    const int q = __ffs(b) - 1;
    rank += __shfl_sync(0xffffffffu, key, q) < key;
  }
  if (lane < kD) {
    wr.rows[lane] = v;
    wr.lrow[lane] = key != INT_MAX ? rank : -1;
  }
  if (first) wr.drow[rank] = key;
  // entry j holds its path's anchor if it is the path's last valid level
  // (paths are stored from the expert's own node up to the anchor)
  const int v_next = __shfl_down_sync(0xffffffffu, v, 1);
  const bool anchor_entry = v >= 0 && (lane % D == D - 1 || lane + 1 >= kD || v_next < 0);
  const unsigned am = __ballot_sync(0xffffffffu, anchor_entry);
  unsigned mask = 0, anc = 0;
  for (int j = 0; j < kD; ++j) {
    const int rj = __shfl_sync(0xffffffffu, key != INT_MAX ? rank : -1, j);
    if (rj == lane) mask |= 1u << (j / D);
    if (rj >= 0 && ((am >> j) & 1u)) anc |= 1u << rj;
  }
  wr.dmask[lane] = mask;
  if (lane == 0) {
    wr.nd = __popc(fm);
    wr.anchor_rows = anc;
  }
  __syncwarp();
}

// CPL consecutive columns of one row (CPL = 1: one float per lane, for small
// batches, where every row load of a token can then be in flight at once;
// CPL = 4: one 16-byte load)
template <int CPL>
struct Cols {
  float v[CPL];
};
template <int CPL>
__device__ __forceinline__ Cols<CPL> ld_cols(const float* p) {
  Cols<CPL> r;
  if constexpr (CPL == 8) {
    const float4 f = ld_dep(reinterpret_cast<const float4*>(p));
    const float4 g = ld_dep(reinterpret_cast<const float4*>(p + 4));
    r.v[0] = f.x; r.v[1] = f.y; r.v[2] = f.z; r.v[3] = f.w;
    r.v[4] = g.x; r.v[5] = g.y; r.v[6] = g.z; r.v[7] = g.w;
  } else if constexpr (CPL == 4) {
    const float4 f = ld_dep(reinterpret_cast<const float4*>(p));
    r.v[0] = f.x; r.v[1] = f.y; r.v[2] = f.z; r.v[3] = f.w;
  } else if constexpr (CPL == 2) {
    const float2 f = ld_dep(reinterpret_cast<const float2*>(p));
    r.v[0] = f.x; r.v[1] = f.y;
  } else {
#pragma unroll
    for (int i = 0; i < CPL; ++i) r.v[i] = ld_dep(p + i);
  }
  return r;
}
template <int CPL>
__device__ __forceinline__ Cols<CPL> ld_cols(const __nv_bfloat16* p) {
  Cols<CPL> r;
  if constexpr (CPL == 8) {
    const uint4 u = ld_dep(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      r.v[2 * i] = __uint_as_float(w[i] << 16);
      r.v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  } else if constexpr (CPL == 4) {
    const uint2 u = ld_dep(reinterpret_cast<const uint2*>(p));
    r.v[0] = __uint_as_float(u.x << 16); r.v[1] = __uint_as_float(u.x & 0xFFFF0000u);
    r.v[2] = __uint_as_float(u.y << 16); r.v[3] = __uint_as_float(u.y & 0xFFFF0000u);
  } else if constexpr (CPL == 2) {
    const uint32_t u = ld_dep(reinterpret_cast<const unsigned int*>(p));
    r.v[0] = __uint_as_float(u << 16); r.v[1] = __uint_as_float(u & 0xFFFF0000u);
  } else {
#pragma unroll
    for (int i = 0; i < CPL; ++i) r.v[i] = __bfloat162float(ld_dep(p + i));
  }
  return r;
}
// CPL raw bf16 values (CPL = 4: one 8-byte load) and their widening
template <int CPL>
struct RawB {
  uint32_t w[(CPL + 1) / 2];
};
template <int CPL>
__device__ __forceinline__ RawB<CPL> ld_raw(const __nv_bfloat16* p) {
  RawB<CPL> r;
  if constexpr (CPL == 4) {
    const uint2 u = ld_dep(reinterpret_cast<const uint2*>(p));
    r.w[0] = u.x;
    r.w[1] = u.y;
  } else if constexpr (CPL == 2) {
    r.w[0] = ld_dep(reinterpret_cast<const unsigned int*>(p));
  } else {
    r.w[0] = (uint32_t)ld_dep(reinterpret_cast<const unsigned short*>(p));
  }
  return r;
}
template <int CPL>
__device__ __forceinline__ void add_raw(Cols<CPL>& a, const RawB<CPL>& r, bool valid) {
  if constexpr (CPL == 4) {
    if (valid) {
      a.v[0] += __uint_as_float(r.w[0] << 16); a.v[1] += __uint_as_float(r.w[0] & 0xFFFF0000u);
      a.v[2] += __uint_as_float(r.w[1] << 16); a.v[3] += __uint_as_float(r.w[1] & 0xFFFF0000u);
    }
  } else if constexpr (CPL == 2) {
    if (valid) {
      a.v[0] += __uint_as_float(r.w[0] << 16); a.v[1] += __uint_as_float(r.w[0] & 0xFFFF0000u);
    }
  } else {
    if (valid) a.v[0] += __uint_as_float(r.w[0] << 16);
  }
}
template <typename T, int CPL>
__device__ __forceinline__ void st_cols(T* p, const Cols<CPL>& c) {
  if constexpr (CPL == 8 && std::is_same<T, __nv_bfloat16>::value) {
    uint4 u;
    uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(c.v[2 * i], c.v[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&b);
    }
    *reinterpret_cast<uint4*>(p) = u;
  } else if constexpr (CPL == 8) {
    store4<T>(p, make_float4(c.v[0], c.v[1], c.v[2], c.v[3]));
    store4<T>(p + 4, make_float4(c.v[4], c.v[5], c.v[6], c.v[7]));
  } else if constexpr (CPL == 4) {
    store4<T>(p, make_float4(c.v[0], c.v[1], c.v[2], c.v[3]));
  } else if constexpr (CPL == 2 && std::is_same<T, __nv_bfloat16>::value) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(c.v[0], c.v[1]);
  } else if constexpr (std::is_same<T, float>::value) {
#pragma unroll
    for (int i = 0; i < CPL; ++i) p[i] = c.v[i];
  } else {
#pragma unroll
    for (int i = 0; i < CPL; ++i) p[i] = __float2bfloat16_rn(c.v[i]);
  }
}
template <int CPL>
__device__ __forceinline__ void add_cols(Cols<CPL>& a, const Cols<CPL>& b) {
#pragma unroll
  for (int i = 0; i < CPL; ++i) a.v[i] += b.v[i];
}

template <typename TH, typename TZ, int D, bool SPLIT, int CPL>
__global__ void __launch_bounds__(WT_WARPS * 32, (sizeof(TH) == 2 && CPL >= 4 && D <= 2) ? 3 : 2)
k_swiglu_warp(const float* topk_w, const int* node_row, int T, int k, const TH* h, int I,
              TZ* __restrict__ z, int cols_per_item,
              const SplitParts hs) {
  extern __shared__ float zsm[];  // bf16 path: [warp][k slots][32 lanes * CPL] activations
  __shared__ WarpRows wrs[WT_WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpRows& wr = wrs[warp];
  const int kD = k * D;
  const int per_tok = (I + cols_per_item - 1) / cols_per_item;
  const long items = (long)T * per_tok;
  long it = (long)blockIdx.x * WT_WARPS + warp;
  // The routing tables (node rows, gates) come from the routing and bucketing
  // kernels, and the x-side products between them and this launch trigger only after
  // their wait for the bucketing: the first item's rows are found before the wait
  // for the preceding kernel (a small batch has one item a warp, and the search is
  // a chain of shuffles).
  if (it < items) {
    const int t = (int)(it / per_tok);
    warp_token_rows(lane < kD ? ld_dep(node_row + (size_t)t * kD + lane) : -1, kD, D, wr);
    if (lane < k) wr.g[lane] = ld_dep(topk_w + (size_t)t * k + lane);
    __syncwarp();
  }
  pdl_wait();
  for (bool first = true; it < items; it += (long)gridDim.x * WT_WARPS, first = false) {
    const int t = (int)(it / per_tok);
    const int c_begin = (int)(it % per_tok) * cols_per_item;
    const int c_end = min(I, c_begin + cols_per_item);
    if (!first) {
      warp_token_rows(lane < kD ? ld_dep(node_row + (size_t)t * kD + lane) : -1, kD, D, wr);
      if (lane < k) wr.g[lane] = ld_dep(topk_w + (size_t)t * k + lane);
      __syncwarp();
    }
    const int nd = wr.nd;
    for (int c = c_begin + CPL * lane; c < c_end; c += 32 * CPL) {
      Cols<CPL> act[WT_SLOTS];
      if constexpr (sizeof(TH) == 2) {
        // bf16 rows, in batches of SG slots: every path-row load of a batch
        // first (rows past a path's end are not read), so that they are in
        // flight at once; each slot's act then goes to this lane's slice of
        // the warp's shared block
        float* as = zsm + (size_t)warp * k * 32 * CPL;
        constexpr int NS = SPLIT ? LX_STREAM_MAX_SPLIT : 1;
        constexpr int SG = (CPL >= 4 && D >= 2) ? 4 : WT_SLOTS;  // bounds the live registers
#pragma unroll
        for (int s0 = 0; s0 < WT_SLOTS; s0 += SG) {
          if (s0 >= k) break;
          RawB<CPL> rg[SG][D], ru[SG][D];
          bool val[SG][D], anc[SG][D];
          Cols<CPL> sg[SG][NS], su[SG][NS];  // the anchor row's split-K partials
#pragma unroll
          for (int j = 0; j < SG; ++j) {
            const int sl = s0 + j;
            int ra = 0;
#pragma unroll
            for (int l = 0; l < D; ++l) {
              const int r = sl < k ? wr.rows[sl * D + l] : -1;
              const int rn = (sl < k && l + 1 < D) ? wr.rows[sl * D + l + 1] : -1;
              val[j][l] = r >= 0;
              anc[j][l] = SPLIT && r >= 0 && rn < 0;  // the path's anchor row
              if (anc[j][l]) ra = r;
              if (r >= 0 && !anc[j][l]) {
                const __nv_bfloat16* hp =
                    reinterpret_cast<const __nv_bfloat16*>(h) + (size_t)r * 2 * I + c;
                rg[j][l] = ld_raw<CPL>(hp);
                ru[j][l] = ld_raw<CPL>(hp + I);
              }
            }
            if constexpr (SPLIT) {
#pragma unroll
              for (int sp = 0; sp < NS; ++sp) {
                const float* hp2 = hs.part + (long)(sp < hs.splits ? sp : 0) * hs.stride +
                                   (size_t)ra * 2 * I + c;
                sg[j][sp] = ld_cols<CPL>(hp2);
                su[j][sp] = ld_cols<CPL>(hp2 + I);
              }
            }
          }
#pragma unroll
          for (int j = 0; j < SG; ++j) {
            const int sl = s0 + j;
            Cols<CPL> pg, pu;
#pragma unroll
            for (int i = 0; i < CPL; ++i) pg.v[i] = pu.v[i] = 0.f;
#pragma unroll
            for (int l = 0; l < D; ++l) {  // path order: the expert's node up to its anchor
              if (anc[j][l]) {
                // anchor row: its split-K partials (not h), in split order
#pragma unroll
                for (int sp = 0; sp < NS; ++sp) {
                  if (sp < hs.splits) {
                    add_cols(pg, sg[j][sp]);
                    add_cols(pu, su[j][sp]);
                  }
                }
              } else {
                add_raw(pg, rg[j][l], val[j][l]);
                add_raw(pu, ru[j][l], val[j][l]);
              }
            }
            if (sl < k) {
              const float g = wr.g[sl];
#pragma unroll
              for (int i = 0; i < CPL; ++i)
                as[(sl * 32 + lane) * CPL + i] = g * silu_fast(pg.v[i]) * pu.v[i];
            }
          }
        }
        // z: every distinct row's z is the sum of the acts of the slots whose
        // path holds it (the row's slot mask), slots ascending
        for (int d = 0; d < nd; ++d) {
          Cols<CPL> zc;
#pragma unroll
          for (int i = 0; i < CPL; ++i) zc.v[i] = 0.f;
          for (unsigned m = wr.dmask[d]; m; m &= m - 1) {
            const int sl = __ffs(m) - 1;
#pragma unroll
            for (int i = 0; i < CPL; ++i) zc.v[i] += as[(sl * 32 + lane) * CPL + i];
          }
          st_cols<TZ, CPL>(z + (size_t)wr.drow[d] * I + c, zc);
        }
        continue;
      } else {
#pragma unroll
      for (int sl = 0; sl < WT_SLOTS; ++sl) {
#pragma unroll
        for (int i = 0; i < CPL; ++i) act[sl].v[i] = 0.f;
        if (sl < k) {
          Cols<CPL> pg, pu;
#pragma unroll
          for (int i = 0; i < CPL; ++i) pg.v[i] = pu.v[i] = 0.f;
#pragma unroll
          for (int l = 0; l < D; ++l) {  // path order: the expert's node up to its anchor
            const int r = wr.rows[sl * D + l];
            if (r >= 0) {
              if (SPLIT && (l + 1 == D || wr.rows[sl * D + l + 1] < 0)) {
                // anchor row: its split-K partials, in split order
#pragma unroll
                for (int sp = 0; sp < LX_STREAM_MAX_SPLIT; ++sp) {
                  if (sp < hs.splits) {
                    const float* hp = hs.part + sp * hs.stride + (size_t)r * 2 * I;
                    add_cols(pg, ld_cols<CPL>(hp + c));
                    add_cols(pu, ld_cols<CPL>(hp + I + c));
                  }
                }
              } else {
                add_cols(pg, ld_cols<CPL>(h + (size_t)r * 2 * I + c));
                add_cols(pu, ld_cols<CPL>(h + (size_t)r * 2 * I + I + c));
              }
            }
          }
          const float g = wr.g[sl];
#pragma unroll
          for (int i = 0; i < CPL; ++i) act[sl].v[i] = g * silu_f(pg.v[i]) * pu.v[i];
        }
      }
      }
      for (int d = 0; d < nd; ++d) {
        const unsigned m = wr.dmask[d];
        Cols<CPL> acc;
#pragma unroll
        for (int i = 0; i < CPL; ++i) acc.v[i] = 0.f;
#pragma unroll
        for (int sl = 0; sl < WT_SLOTS; ++sl)  // slots ascending
          if ((m >> sl) & 1u) add_cols(acc, act[sl]);
        st_cols<TZ, CPL>(z + (size_t)wr.drow[d] * I + c, acc);
      }
    }
    __syncwarp();
  }
}

// y[t] = sum of ypart over t's distinct rows in ascending row order (an
// anchor row split into K ranges contributes its partials in split order)
template <typename TP, typename TY, int CPL, bool SPLIT>
__global__ void __launch_bounds__(WT_WARPS * 32, 2)
k_combine_warp(const int* node_row, int k, int D, const TP* ypart, int H, TY* __restrict__ y,
               int T, int cols_per_item, const SplitParts ys) {
  __shared__ WarpRows wrs[WT_WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpRows& wr = wrs[warp];
  const int kD = k * D;
  const int per_tok = (H + cols_per_item - 1) / cols_per_item;
  const long items = (long)T * per_tok;
  long it = (long)blockIdx.x * WT_WARPS + warp;
  // node rows come from the bucketing, and the x-side products in between trigger
  // only after their wait for it: the first item's rows are found before the wait
  // for the preceding kernel
  if (it < items)
    warp_token_rows(lane < kD ? ld_dep(node_row + (size_t)(it / per_tok) * kD + lane) : -1, kD, D, wr);
  pdl_wait();
  for (bool first = true; it < items; it += (long)gridDim.x * WT_WARPS, first = false) {
    const int t = (int)(it / per_tok);
    const int c_begin = (int)(it % per_tok) * cols_per_item;
    const int c_end = min(H, c_begin + cols_per_item);
    if (!first) warp_token_rows(lane < kD ? ld_dep(node_row + (size_t)t * kD + lane) : -1, kD, D, wr);
    const int nd = wr.nd;
    for (int c = c_begin + CPL * lane; c < c_end; c += 32 * CPL) {
      Cols<CPL> acc;
#pragma unroll
      for (int i = 0; i < CPL; ++i) acc.v[i] = 0.f;
      if constexpr (SPLIT) {
        // four distinct rows per batch, every load of the batch first: an
        // anchor row contributes its split partials (fp32, split order), any
        // other row its ypart row
        constexpr int NS = LX_STREAM_MAX_SPLIT;
        for (int q0 = 0; q0 < nd; q0 += 4) {
          Cols<CPL> v[4][NS];
          bool isa[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int d = q0 + u < nd ? q0 + u : q0;
            const size_t ro = (size_t)wr.drow[d] * H + c;
            isa[u] = q0 + u < nd && ((wr.anchor_rows >> d) & 1u);
            if (isa[u]) {
#pragma unroll
              for (int sp = 0; sp < NS; ++sp)
                v[u][sp] = ld_cols<CPL>(ys.part + (long)(sp < ys.splits ? sp : 0) * ys.stride + ro);
            } else {
              v[u][0] = ld_cols<CPL>(ypart + ro);
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (q0 + u >= nd) break;
            if (isa[u]) {
#pragma unroll
              for (int sp = 0; sp < NS; ++sp)
                if (sp < ys.splits) add_cols(acc, v[u][sp]);
            } else {
              add_cols(acc, v[u][0]);
            }
          }
        }
      } else {
        int q = 0;
        for (; q + 8 <= nd; q += 8) {
          Cols<CPL> v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = ld_cols<CPL>(ypart + (size_t)wr.drow[q + u] * H + c);
#pragma unroll
          for (int u = 0; u < 8; ++u) add_cols(acc, v[u]);
        }
        for (; q < nd; ++q) add_cols(acc, ld_cols<CPL>(ypart + (size_t)wr.drow[q] * H + c));
      }
      st_cols<TY, CPL>(y + (size_t)t * H + c, acc);
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// The same two steps for prefill batches, a CTA per token: the bucketing has
// written the token's distinct rows (and the slots that share each), every thread
// owns a few columns and has several rows' loads in flight.  Finding the rows
// in the same kernel, a warp a token, is a chain of dependent shuffles that few
// resident warps hid: combine 38 -> 27.5 us (8192 tokens) and 23.5 ->
// 7.4 (1031 tokens) of the Qwen3-30B-A3B-shaped layer, whose rows take 22
// and 3 us at the HBM rate; SwiGLU of the depth-2 tree, 2048 tokens, 49 ->
// 43 us (17 at that rate).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 bf2(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}
__device__ __forceinline__ uint32_t pack2(float2 v) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&b);
}

// y[t] = sum of ypart over t's listed rows in ascending row order
__global__ void __launch_bounds__(256, 6)
k_combine_tok(const int* trow, int max_rows, const __nv_bfloat16* ypart, int H,
              __nv_bfloat16* __restrict__ y) {
  const int4* rows = reinterpret_cast<const int4*>(trow + (size_t)blockIdx.x * TOK_ROWS);
  // (the list comes from the bucketing, and tc_up_anchor in between triggers only
  // after its wait for it)
  int4 r = ld_dep(rows);
  pdl_wait();
  for (int c = 8 * threadIdx.x; c < H; c += 8 * blockDim.x) {
    float2 acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = make_float2(0.f, 0.f);
    int4 q = r;
    for (int d = 0; d < max_rows && q.x >= 0; d += 4) {
      const int rr[4] = {q.x, q.y, q.z, q.w};
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (rr[u] >= 0) v[u] = ld_dep(reinterpret_cast<const uint4*>(ypart + (size_t)rr[u] * H + c));
      if (d + 4 < max_rows) q = ld_dep(rows + d / 4 + 1);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (rr[u] >= 0) {
          const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i] = add2(acc[i], bf2(w[i]));
        }
    }
    *reinterpret_cast<uint4*>(y + (size_t)blockIdx.x * H + c) =
        make_uint4(pack2(acc[0]), pack2(acc[1]), pack2(acc[2]), pack2(acc[3]));
  }
}

// z(t, n) = sum of g_s silu(sum of h_g over the path) * (sum of h_u) over the
// slots s whose path holds n.  A thread owns four columns: every distinct row's
// gate and up values are loaded once (six rows in flight) and added to the slots
// whose path holds the row, rows ascending; then the acts, then the rows' z.
__global__ void __launch_bounds__(256, 2)
k_swiglu_tok(const float* topk_w, const int* trow, const uint8_t* tmask, int k, const __nv_bfloat16* h,
             int I, __nv_bfloat16* __restrict__ z) {
  __shared__ int srow[TOK_ROWS], smask[TOK_ROWS];
  __shared__ float sg[WT_SLOTS];
  const int t = blockIdx.x, tid = threadIdx.x;
  if (tid < TOK_ROWS) {  // (ahead of the wait: as in k_combine_tok)
    srow[tid] = trow[(size_t)t * TOK_ROWS + tid];
    smask[tid] = tmask[(size_t)t * TOK_ROWS + tid];
    if (tid < WT_SLOTS) sg[tid] = tid < k ? topk_w[(size_t)t * k + tid] : 0.f;
  }
  pdl_wait();
  const int nd = __syncthreads_count(tid < TOK_ROWS && srow[tid < TOK_ROWS ? tid : 0] >= 0);
  for (int c = 4 * tid; c < I; c += 4 * blockDim.x) {
    float2 pg[WT_SLOTS][2], pu[WT_SLOTS][2];
#pragma unroll
    for (int s = 0; s < WT_SLOTS; ++s) pg[s][0] = pg[s][1] = pu[s][0] = pu[s][1] = make_float2(0.f, 0.f);
    constexpr int U = 6;
    for (int d0 = 0; d0 < nd; d0 += U) {
      uint2 g[U], u[U];
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (d0 + q < nd) {
          const __nv_bfloat16* hp = h + (size_t)srow[d0 + q] * 2 * I + c;
          g[q] = ld_dep(reinterpret_cast<const uint2*>(hp));
          u[q] = ld_dep(reinterpret_cast<const uint2*>(hp + I));
        }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (d0 + q >= nd) break;
        const int m = smask[d0 + q];
        const float2 g0 = bf2(g[q].x), g1 = bf2(g[q].y), u0 = bf2(u[q].x), u1 = bf2(u[q].y);
#pragma unroll
        for (int s = 0; s < WT_SLOTS; ++s)
          if ((m >> s) & 1) {  // CTA-uniform
            pg[s][0] = add2(pg[s][0], g0);
            pg[s][1] = add2(pg[s][1], g1);
            pu[s][0] = add2(pu[s][0], u0);
            pu[s][1] = add2(pu[s][1], u1);
          }
      }
    }
#pragma unroll
    for (int s = 0; s < WT_SLOTS; ++s)  // the slot's act, in place of its gate sums
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        pg[s][i].x = sg[s] * silu_fast(pg[s][i].x) * pu[s][i].x;
        pg[s][i].y = sg[s] * silu_fast(pg[s][i].y) * pu[s][i].y;
      }
    for (int d = 0; d < nd; ++d) {
      const int m = smask[d];
      float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
      for (int s = 0; s < WT_SLOTS; ++s)  // slots ascending
        if ((m >> s) & 1) {
          a0 = add2(a0, pg[s][0]);
          a1 = add2(a1, pg[s][1]);
        }
      *reinterpret_cast<uint2*>(z + (size_t)srow[d] * I + c) = make_uint2(pack2(a0), pack2(a1));
    }
  }
}

}  // namespace

bool warp_kernels_fit(const lx_layer* L, int k) {
  return k <= WT_SLOTS && k * L->max_depth <= 32 && L->I % 4 == 0 && L->H % 8 == 0;
}

// Columns per warp work item: whole rows when the batch alone fills the GPU
// (the distinct-row search then runs once per token), else blocks of `unit`
// columns so that a small batch still spreads over the SMs.
static int warp_item_cols(const lx_layer* L, int T, int width, int unit) {
  const long want = (long)L->num_sms * 4 * WT_WARPS;
  const int blocks = (width + unit - 1) / unit;
  int per = blocks;
  while (per > 1 && (long)T * ((blocks + per - 1) / per) < want) per = (per + 1) / 2;
  return per * unit;
}

static int warp_grid(const lx_layer* L, int T, int width, int cols) {
  const long items = (long)T * ((width + cols - 1) / cols);
  return (int)std::min<long>((items + WT_WARPS - 1) / WT_WARPS, (long)L->num_sms * 4);
}

// One float per lane for batches too small to fill the GPU with 128-column items.
static bool narrow_cols(const lx_layer* L, int T, int width) {
  return (long)T * ((width + 127) / 128) < (long)L->num_sms * 4 * WT_WARPS;
}

template <typename TH, typename TZ, int D, int CPL>
static void launch_swiglu_c(lx_layer* L, int T, int k, const TH* h, TZ* z, cudaStream_t s,
                            const SplitParts& hs) {
  Workspace& w = L->ws;
  const int cols = warp_item_cols(L, T, L->I, 32 * CPL);
  const int grid = warp_grid(L, T, L->I, cols);
  const size_t zs = sizeof(TH) == 2 ? (size_t)WT_WARPS * k * 32 * CPL * 4 : 0;
  if (zs > 0) {  // the accumulators plus the static rows may pass the 48 KB default
    static bool done_s[64] = {}, done_n[64] = {};
    if constexpr (CPL == 1) {
      if (hs.splits > 1)
        (void)smem_cap_once((const void*)k_swiglu_warp<TH, TZ, D, true, CPL>, 128 * 1024,
                            L->device, done_s);
    }
    (void)smem_cap_once((const void*)k_swiglu_warp<TH, TZ, D, false, CPL>, 128 * 1024, L->device,
                        done_n);
  }
  if constexpr (CPL == 1) {
    if (hs.splits > 1) {
      launch_k(L, k_swiglu_warp<TH, TZ, D, true, CPL>, grid, WT_WARPS * 32, zs, s, w.topk_w,
               w.node_row, T, k, h, L->I, z, cols, hs);
      return;
    }
  }
  launch_k(L, k_swiglu_warp<TH, TZ, D, false, CPL>, grid, WT_WARPS * 32, zs, s, w.topk_w,
           w.node_row, T, k, h, L->I, z, cols, hs);
}

template <typename TH, typename TZ, int D>
static void launch_swiglu_d(lx_layer* L, int T, int k, const TH* h, TZ* z, cudaStream_t s,
                            const SplitParts& hs) {
  // split partials (small batches only) take the one-column-per-lane form
  // (measured on GB300: four columns per lane beat two for large batches)
  if (narrow_cols(L, T, L->I) || hs.splits > 1)
    launch_swiglu_c<TH, TZ, D, 1>(L, T, k, h, z, s, hs);
  else
    launch_swiglu_c<TH, TZ, D, 4>(L, T, k, h, z, s, hs);
}

template <typename TH, typename TZ>
static void launch_swiglu_warp(lx_layer* L, int T, int k, const TH* h, TZ* z, cudaStream_t s,
                               const SplitParts& hs) {
  switch (L->max_depth) {
    case 1: launch_swiglu_d<TH, TZ, 1>(L, T, k, h, z, s, hs); break;
    case 2: launch_swiglu_d<TH, TZ, 2>(L, T, k, h, z, s, hs); break;
    case 3: launch_swiglu_d<TH, TZ, 3>(L, T, k, h, z, s, hs); break;
    default: launch_swiglu_d<TH, TZ, 4>(L, T, k, h, z, s, hs); break;
  }
}

// (the combine reads few rows per token: 16-byte columns measured faster at
// every batch size)
template <typename TP, typename TY>
static void launch_combine_warp(lx_layer* L, int T, int k, const TP* ypart, TY* y, cudaStream_t s,
                                const SplitParts& ys) {
  Workspace& w = L->ws;
  if (ys.splits > 1) {
    const int cols = warp_item_cols(L, T, L->H, 128);
    const int grid = warp_grid(L, T, L->H, cols);
    launch_k(L, k_combine_warp<TP, TY, 4, true>, grid, WT_WARPS * 32, 0, s, w.node_row, k,
             L->max_depth, ypart, L->H, y, T, cols, ys);
    return;
  }
  // eight columns per lane (16-byte bf16 loads): half the per-element address
  // and loop instructions of four (measured faster at decode and prefill)
  const int cols = warp_item_cols(L, T, L->H, 256);
  const int grid = warp_grid(L, T, L->H, cols);
  launch_k(L, k_combine_warp<TP, TY, 8, false>, grid, WT_WARPS * 32, 0, s, w.node_row, k,
           L->max_depth, ypart, L->H, y, T, cols, ys);
}

// threads of a CTA that gives each thread `per` of `width` columns
static int tok_threads(int width, int per) { return std::min(256, (width / per + 31) / 32 * 32); }

lx_status launch_swiglu_tok(lx_layer* L, int T, int k, cudaStream_t s) {
  Workspace& w = L->ws;
  ProfScope ps(L, s, "swiglu");
  launch_k(L, k_swiglu_tok, T, tok_threads(L->I, 4), 0, s, w.topk_w, w.trow, w.tmask, k, w.hb, L->I, w.zb);
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

lx_status launch_combine_tok(lx_layer* L, int T, int k, void* y, cudaStream_t s) {
  Workspace& w = L->ws;
  ProfScope ps(L, s, "combine");
  launch_k(L, k_combine_tok, T, tok_threads(L->H, 8), 0, s, w.trow, k * (L->ct ? 1 : L->max_depth), w.yb,
           L->H, static_cast<__nv_bfloat16*>(y));
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

lx_status launch_swiglu(lx_layer* L, int T, int k, bool bf16, cudaStream_t s, SplitParts hs) {
  Workspace& w = L->ws;
  ProfScope ps(L, s, bf16 ? "swiglu" : "generic_swiglu");
  if (warp_kernels_fit(L, k)) {
    if (bf16)
      launch_swiglu_warp(L, T, k, w.hb, w.zb, s, hs);
    else
      launch_swiglu_warp(L, T, k, w.h, w.z, s, hs);
    LX_CUDA(cudaGetLastError());
    return LX_OK;
  }
  // large k or deep paths: the block-per-token form (generic path only)
  if (bf16 || hs.splits > 1) return fail(LX_ERR_STATE, "bf16 SwiGLU needs k <= 8, k * depth <= 32");
  const int grid = std::min(T, L->num_sms * 8);
  const size_t smem = sizeof(float4) * SW_T * k * L->max_depth;
  static bool done_f[64] = {};
  LX_CUDA(smem_cap_once((const void*)k_swiglu_aggregate<float>, 200 * 1024, L->device, done_f));
  launch_k(L, k_swiglu_aggregate<float>, grid, SW_T, smem, s, w.topk_w, w.node_row, T,
           k, L->max_depth, w.h, L->I, w.z);
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

lx_status launch_combine(lx_layer* L, int T, int k, void* y, bool bf16, cudaStream_t s,
                         SplitParts ys) {
  Workspace& w = L->ws;
  ProfScope ps(L, s, "combine");
  if (warp_kernels_fit(L, k)) {
    if (bf16)
      launch_combine_warp(L, T, k, L->ws.yb, static_cast<__nv_bfloat16*>(y), s, ys);
    else if (L->dtype == LX_BF16)
      launch_combine_warp(L, T, k, L->ws.ypart, static_cast<__nv_bfloat16*>(y), s, ys);
    else
      launch_combine_warp(L, T, k, L->ws.ypart, static_cast<float*>(y), s, ys);
    LX_CUDA(cudaGetLastError());
    return LX_OK;
  }
  if (bf16 || ys.splits > 1) return fail(LX_ERR_STATE, "bf16 combine needs k <= 8, k * depth <= 32");
  const int grid = std::min(T, L->num_sms * 8);
  if (L->dtype == LX_BF16)
    launch_k(L, k_combine<__nv_bfloat16>, grid, 256, 0, s, w.node_row, k, L->max_depth, w.ypart, L->H,
                                                  (__nv_bfloat16*)y, T);
  else
    launch_k(L, k_combine<float>, grid, 256, 0, s, w.node_row, k, L->max_depth, w.ypart, L->H, (float*)y, T);
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

namespace {

GemmArgs gemm_op(lx_layer* L, int op, const void* A, long lda, const int* gather,
                 const void* const* W, float* out, long ldo) {
  const OpShape sh = op_shape(L, op);
  GemmArgs g;
  g.items = sh.on_anchors ? L->d_anchors : L->d_corrs;
  g.n_items = sh.on_anchors ? L->n_anchor : L->n_corr;
  g.tile_off = L->ws.tile_off + op * (op_max_items(L) + 1);
  g.node_off = L->ws.key_off;
  g.gather = gather;
  g.A = A;
  g.lda = lda;
  g.W = W;
  g.rank = L->d_rank;
  g.shape = sh;
  g.out = out;
  g.ldo = ldo;
  g.tiled = L->tiled ? 1 : 0;
  return g;
}

template <typename TA, typename TW, int OPK>
lx_status run_gemm(lx_layer* L, std::initializer_list<GemmArgs> ops, cudaStream_t s, const char* name) {
  GemmLaunch P;
  P.n_ops = 0;
  P.early = OPK != OP_UP_ANCHOR;  // the x side follows the bucketing directly
  for (const GemmArgs& g : ops)
    if (g.n_items > 0) P.op[P.n_ops++] = g;
  if (P.n_ops == 0) return LX_OK;
  if (P.n_ops == 1) P.op[1] = P.op[0];
  constexpr int smem = GG<TA, TW>::SMEM;
  static bool done[64] = {};
  LX_CUDA(smem_cap_once((const void*)k_grouped_gemm<TA, TW, OPK>, smem, L->device, done));
  ProfScope ps(L, s, name);
  launch_k(L, k_grouped_gemm<TA, TW, OPK>, L->num_sms * GG_CTAS_PER_SM, GG_THREADS, smem, s, P);
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

template <typename TX>
lx_status generic_impl(lx_layer* L, const void* x, int T, int k, void* y, cudaStream_t s) {
  Workspace& w = L->ws;
  const long H = L->H, I = L->I, rmax = std::max(1, L->max_rank);
  auto up = (const void* const*)L->d_w_up, dn = (const void* const*)L->d_w_dn;
  // x-side products
  LX_TRY((run_gemm<TX, TX, OP_UP_ANCHOR>(
      L, {gemm_op(L, OP_UP_ANCHOR, x, H, w.node_tok, up, w.h, 2 * I),
          gemm_op(L, OP_UP_V, x, H, w.node_tok, up, w.P, 2 * rmax)}, s, "generic_up_anchor_V")));
  LX_TRY((run_gemm<float, TX, OP_UP_U>(
      L, {gemm_op(L, OP_UP_U, w.P, 2 * rmax, nullptr, (const void* const*)L->d_w_upU, w.h, 2 * I)}, s,
      "generic_up_U")));
  LX_TRY(launch_swiglu(L, T, k, false, s));
  // z-side products
  LX_TRY((run_gemm<float, TX, OP_DN_ANCHOR>(
      L, {gemm_op(L, OP_DN_ANCHOR, w.z, I, nullptr, dn, w.ypart, H),
          gemm_op(L, OP_DN_V, w.z, I, nullptr, dn, w.Q, rmax)}, s, "generic_dn_anchor_V")));
  LX_TRY((run_gemm<float, TX, OP_DN_U>(
      L, {gemm_op(L, OP_DN_U, w.Q, rmax, nullptr, (const void* const*)L->d_w_dnU, w.ypart, H)}, s,
      "generic_dn_U")));
  LX_TRY(launch_combine(L, T, k, y, false, s));
  return LX_OK;
}

}  // namespace

lx_status launch_generic_experts(lx_layer* L, const void* x, int T, int k, void* y,
                                 cudaStream_t s) {
  if (L->dtype == LX_BF16) return generic_impl<__nv_bfloat16>(L, x, T, k, y, s);
  return generic_impl<float>(L, x, T, k, y, s);
}

}  // namespace lx
