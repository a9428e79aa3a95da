// Compression of one member projection (Sec. 3.2 Stage 3 (ii)): the residual
// R = W_mem - W_dom ([rows][cols], Eq. svd), its rank-r randomized SVD (range
// finder with power iterations, Halko-Martinsson-Tropp, with the Gaussian test
// matrix given by the caller) and the symmetric split of Eq. factors,
// U = U_r S_r^(1/2) [rows][r], V = V_r S_r^(1/2) [cols][r].
//
// Kernels (the products with R of bf16 weights run on the tensor cores, in
// lx_compress_tc.cu):
//   k_cgemm     fp32 GEMM (CUDA-core FMA, 64 x 64 tiles, 32-deep K chunks in
//               shared memory); its A operand is R (rows of W_mem - W_dom,
//               formed on load; fp32 weights), R^T (columns of the same), or an
//               fp32 matrix (the bases times the small factors).
//   k_gram      G = X^T X to float64 accuracy (exact fp32 products, error-free
//               two-sum accumulation on the fp32 pipes), stored in float64.
//   k_chol32    one CTA: Cholesky G + s I = L L^T (fp32 in shared memory,
//               blocked by 16 columns; a small relative shift in the first
//               pass keeps rank-deficient bases factorable).
//   k_trsm      X L^-T by blocked substitution, so that its columns are
//               orthonormal (CholeskyQR).
//   k_trmm      M = L1 L2, the triangular factor of R^T Q = Z2 M^T.
//   k_jacobi_cluster
//               one-sided Jacobi SVD of M, M W = U S, over a thread-block
//               cluster (fp32 rotations, column blocks exchanged through
//               distributed shared memory).
//   k_ritz      sigma_j = |M w_j| / |w_j| in float64 (Rayleigh quotients).
//   k_finish    the r largest sigma and the fp32 matrices that turn the bases
//               into the split factors.
//   k_sign      each factor column's largest-magnitude entry of U made
//               positive (U and V negated together).
// The Gram sums, M and the Rayleigh quotients reach float64 accuracy by
// compensated fp32 arithmetic: this GPU's float64 rate is a small fraction of
// its fp32 rate.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lx_internal.cuh"

namespace lx {
namespace {

constexpr int CG_TILE = 64;
constexpr int CG_KC = 32;
constexpr int CG_LD = CG_TILE + 4;
constexpr int CG_THREADS = 256;

enum { A_RES = 0, A_RES_T = 1, A_F32 = 2 };

__device__ __forceinline__ void cload8(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 q = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 f = __bfloat1622float2(h[e]);
    v[2 * e] = f.x;
    v[2 * e + 1] = f.y;
  }
}
__device__ __forceinline__ void cload8(const float* p, float (&v)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// C [M][N] = A [M][K] * B [K][N] (fp32, row-major).  A element (m, k):
//   A_RES:   Wm[m * ldw + k] - Wd[m * ldw + k]   (R itself; M = rows, K = cols = ldw)
//   A_RES_T: Wm[k * ldw + m] - Wd[k * ldw + m]   (R^T; M = cols = ldw, K = rows)
//   A_F32:   X[m * K + k]
// A_RES / A_RES_T need ldw % 8 == 0 and 16-byte aligned weights (8-element
// vector loads); A_F32 and B take scalar loads (any K, N).
template <typename TW, int MODE>
__global__ void __launch_bounds__(CG_THREADS)
k_cgemm(const TW* __restrict__ Wm, const TW* __restrict__ Wd, const float* __restrict__ X,
        int ldw, const float* __restrict__ B, float* __restrict__ C, int M, int N, int K) {
  __shared__ __align__(16) float As[CG_KC][CG_LD];
  __shared__ __align__(16) float Bs[CG_KC][CG_LD];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * CG_TILE, n0 = blockIdx.x * CG_TILE;
  const int ty = tid >> 4, tx = tid & 15;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += CG_KC) {
    const int kc = min(CG_KC, K - k0);
    if (MODE == A_RES) {
      const int row = tid >> 2, kq = (tid & 3) * 8;
      const bool ok = m0 + row < M && kq < kc;  // kc is a multiple of 8 here
      float a[8], d[8];
      if (ok) {
        cload8(Wm + (size_t)(m0 + row) * ldw + k0 + kq, a);
        cload8(Wd + (size_t)(m0 + row) * ldw + k0 + kq, d);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) As[kq + e][row] = ok ? a[e] - d[e] : 0.f;
    } else if (MODE == A_RES_T) {
      const int kr = tid >> 3, mq = (tid & 7) * 8;
      const bool ok = kr < kc && m0 + mq < M;
      float a[8], d[8];
      if (ok) {
        cload8(Wm + (size_t)(k0 + kr) * ldw + m0 + mq, a);
        cload8(Wd + (size_t)(k0 + kr) * ldw + m0 + mq, d);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) As[kr][mq + e] = ok ? a[e] - d[e] : 0.f;
    } else {
      const int row = tid >> 2, kq = (tid & 3) * 8;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const bool ok = m0 + row < M && kq + e < kc;
        As[kq + e][row] = ok ? X[(size_t)(m0 + row) * K + k0 + kq + e] : 0.f;
      }
    }
    {
      const int kr = tid >> 3, nq = (tid & 7) * 8;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const bool ok = kr < kc && n0 + nq + e < N;
        Bs[kr][nq + e] = ok ? B[(size_t)(k0 + kr) * N + n0 + nq + e] : 0.f;
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < CG_KC; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(av[r], bv[c], acc[r][c]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int m = m0 + ty * 4 + r;
    if (m >= M) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int n = n0 + tx * 4 + c;
      if (n < N) C[(size_t)m * N + n] = acc[r][c];
    }
  }
}

// G [L][L] = X^T X for X [n][L] fp32 row-major, as pairs hi + lo, to float64 accuracy on the
// fp32 pipes (this GPU's float64 rate is a small fraction of its fp32 rate).
// Each product is formed exactly as the pair p + e (p = x y rounded,
// e = fma(x, y, -p)); the sum is carried as an unevaluated pair hi + lo, hi
// taking the products through Knuth's error-free two-sum and lo collecting the
// two-sum and product errors (the compensated dot product "Dot2" of Ogita,
// Rump and Oishi, 2005), so G = hi + lo is as accurate as a dot product in
// twice the fp32 precision: within 2^-24 |G| + (n 2^-24)^2 sum |x y| of the
// exact sum, far below the fp32 rounding the Cholesky applies to it.  Four
// such pairs per thread take the rows of a chunk in turn (independent chains)
// and are added pairwise at the end; each 64-row chunk is staged in shared
// memory while the next one is already loading into registers.  16 x 16
// outputs per CTA; only the tiles on or below the diagonal are computed (the
// Cholesky reads the lower triangle alone).  The triangle's tiles alone (45 at
// L = 136) leave most SMs idle and each runs n serial steps, so the rows are
// cut into up to GR_SPLITS ranges (blockIdx.z) of 256 or more, whose pairs the
// Cholesky adds in order: 26.9 -> 19.1 us a launch at L = 136 (n = 768 and 2048).
// The issue rate bounds it, so the ranges are counted by the rows of the SM with
// the most CTAs (gram_parts): n = 2048 takes 3 (135 CTAs, one an SM, 683 rows
// each) before 4 (180 CTAs, two on some SMs): 28.0 -> 24.4 us.
constexpr int GR_SPLITS = 4;
constexpr int GR_T = 16;
constexpr int GR_KC = 64;
constexpr int GR_CH = 4;
static_assert(GR_KC * GR_T % (GR_T * GR_T) == 0, "whole staged values per thread");

// row ranges of a Gram of n rows and L columns
static int gram_parts(int n, int L, int sms) {
  const int t = (L + GR_T - 1) / GR_T, tiles = t * (t + 1) / 2;
  int best = 1, cost = 0x7fffffff;
  for (int p = 1; p <= std::min(GR_SPLITS, std::max(1, n / 256)); ++p) {
    const int c = (tiles * p + sms - 1) / sms * ((n + p - 1) / p);
    if (c < cost) {
      cost = c;
      best = p;
    }
  }
  return best;
}

struct DF {
  float hi, lo;
};
// hi + lo += p + e, by the two-sum of hi and p (every step rounded on its own:
// the intrinsics are never contracted into fused operations)
__device__ __forceinline__ void df_add(DF& d, float p, float e) {
  const float s = __fadd_rn(d.hi, p);
  const float v = __fsub_rn(s, d.hi);
  const float err = __fadd_rn(__fsub_rn(d.hi, __fsub_rn(s, v)), __fsub_rn(p, v));
  d.hi = s;
  d.lo = __fadd_rn(d.lo, __fadd_rn(err, e));
}

__global__ void __launch_bounds__(GR_T * GR_T)
k_gram(const float* __restrict__ X, int n_all, int L, int span, float2* __restrict__ Gp) {
  constexpr int PER = GR_KC * GR_T / (GR_T * GR_T);  // staged values per thread and side
  __shared__ float Xi[GR_KC][GR_T], Xj[GR_KC][GR_T];
  if (blockIdx.x > blockIdx.y) return;  // strictly above the diagonal
  const int n_lo = blockIdx.z * span, n = min(n_all, n_lo + span);
  float2* G = Gp + (size_t)blockIdx.z * L * L;
  const int ti = threadIdx.x / GR_T, tj = threadIdx.x % GR_T;
  const int i0 = blockIdx.y * GR_T, j0 = blockIdx.x * GR_T;
  DF acc[GR_CH];
#pragma unroll
  for (int c = 0; c < GR_CH; ++c) acc[c] = DF{0.f, 0.f};
  // the next chunk's rows are loaded into registers while this one is summed
  float ri[PER], rj[PER];
  auto fetch = [&](int m0) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int q = threadIdx.x + e * GR_T * GR_T;
      const int mr = q / GR_T, c = q % GR_T;
      const bool okm = m0 + mr < n;
      ri[e] = (okm && i0 + c < L) ? X[(size_t)(m0 + mr) * L + i0 + c] : 0.f;
      rj[e] = (okm && j0 + c < L) ? X[(size_t)(m0 + mr) * L + j0 + c] : 0.f;
    }
  };
  fetch(n_lo);
  for (int m0 = n_lo; m0 < n; m0 += GR_KC) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int q = threadIdx.x + e * GR_T * GR_T;
      Xi[q / GR_T][q % GR_T] = ri[e];
      Xj[q / GR_T][q % GR_T] = rj[e];
    }
    __syncthreads();
    if (m0 + GR_KC < n) fetch(m0 + GR_KC);
#pragma unroll
    for (int mr = 0; mr < GR_KC; mr += GR_CH) {
#pragma unroll
      for (int c = 0; c < GR_CH; ++c) {
        const float x = Xi[mr + c][ti], y = Xj[mr + c][tj];
        const float p = __fmul_rn(x, y);
        df_add(acc[c], p, __fmaf_rn(x, y, -p));
      }
    }
    __syncthreads();
  }
  // (chain 0 + chain 1) + (chain 2 + chain 3), each pair added as hi + lo
  DF s01 = acc[0], s23 = acc[2];
  df_add(s01, acc[1].hi, acc[1].lo);
  df_add(s23, acc[3].hi, acc[3].lo);
  df_add(s01, s23.hi, s23.lo);
  if (i0 + ti < L && j0 + tj < L)
    G[(size_t)(i0 + ti) * L + j0 + tj] = make_float2(s01.hi, s01.lo);
}

// One CTA (L <= 256).  Cholesky of G + s I in fp32 (the row ranges' pairs of G
// added in order and rounded once; s = shift_rel * max diag(G)) in a
// packed lower triangle in shared memory (L (L + 1) / 2 floats, row i from
// i (i + 1) / 2), pivots floored at 1e-30, blocked by 16 columns (right-looking).
// One SM's latency bounds it, so each part keeps its chain in registers: warp 0
// factors the diagonal block with lane i holding row i (shuffles, no shared
// memory), one thread per row below solves its 16 panel entries against it
// (vector loads of a transposed copy), and the trailing triangle takes the
// panel's rank-16 update with a warp on four rows, lanes along the columns.
// The factor goes to Lout [L][L] (zero above the diagonal) and the inverses of
// its 16 x 16 diagonal blocks to Dinv [blocks][16][16], which is all that the
// solve below needs.  A zero Gram gives Lout = Dinv = 0.  Measured at L = 136:
// 152 us with in-place shared-memory steps and the whole inverse formed here,
// 42 us now.
constexpr int CH_THREADS = 512;  // 16 warps: at most 16 diagonal blocks
constexpr int CH_B = 16;  // block width
__device__ __forceinline__ int tri_off(int i) { return i * (i + 1) / 2; }
inline int ch_ldp(int L) { return (L + 127) / 128 * 128; }  // panel copy: whole column chunks

__global__ void __launch_bounds__(CH_THREADS, 1)
k_chol32(const float2* __restrict__ Gp, int parts, int L, int ldp, float shift_rel,
         float* __restrict__ Lout, float* __restrict__ Dinv) {
  extern __shared__ __align__(16) float Ls[];
  float* Pt = Ls + ((tri_off(L) + 3) & ~3);          // [CH_B][ldp] panel, transposed
  __shared__ __align__(16) float sD[2][CH_B][CH_B];  // by block parity: sD[c][i] = l_ic of the diagonal block
  __shared__ float s_md;
  __shared__ float s_rdiag[256];  // reciprocals of the factor's diagonal
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = CH_THREADS / 32;
  const int nb = (L + CH_B - 1) / CH_B;
  // the lower triangle of G rounded to fp32, a batch's loads in flight at once
  // (rows q and L - 1 - q together hold L + 1 entries: entry e of the fold)
  const int nfold = (L + 1) / 2 * (L + 1);
  constexpr int U = 5;
  for (int e0 = tid; e0 < nfold; e0 += U * CH_THREADS) {
    float2 g[U][GR_SPLITS];
    int at[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * CH_THREADS, q = e / (L + 1), pos = e - q * (L + 1);
      const bool low = pos < L - q;  // row L - 1 - q, else row q
      const int i = low ? L - 1 - q : q, c = low ? pos : pos - (L - q);
      const bool ok = e < nfold && (low || 2 * q != L - 1);  // (an odd L's middle row once)
      at[u] = ok ? tri_off(i) + c : -1;
#pragma unroll
      for (int z = 0; z < GR_SPLITS; ++z)
        g[u][z] = ok && z < parts ? Gp[(size_t)z * L * L + i * L + c] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      DF t{g[u][0].x, g[u][0].y};
#pragma unroll
      for (int z = 1; z < GR_SPLITS; ++z) df_add(t, g[u][z].x, g[u][z].y);
      if (at[u] >= 0) Ls[at[u]] = __fadd_rn(t.hi, t.lo);
    }
  }
  __syncthreads();
  if (warp == 0) {
    float md = 0.f;
    for (int i = lane; i < L; i += 32) md = fmaxf(md, Ls[tri_off(i) + i]);
#pragma unroll
    for (int o = 16; o; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
    if (lane == 0) s_md = md;
  }
  __syncthreads();
  const float md = s_md;
  if (!(md > 0.f)) {
    for (int e = tid; e < L * L; e += CH_THREADS) Lout[e] = 0.f;
    for (int e = tid; e < nb * CH_B * CH_B; e += CH_THREADS) Dinv[e] = 0.f;
    return;
  }
  const float shift = (float)((double)shift_rel * (double)md);
  for (int i = tid; i < L; i += CH_THREADS) Ls[tri_off(i) + i] += shift;  // (float) g_ii + shift
  __syncthreads();
  // ---- factorization.  Warp 0 factors the diagonal block; while the other
  // warps finish a step's trailing update it brings the next diagonal block up
  // to date itself and factors it.
  auto factor_diag = [&](int kb, float (&a)[CH_B]) {
    // lane i: row j0 + i of the diagonal block (identity rows past bw)
    const int j0 = kb * CH_B, bw = min(CH_B, L - j0);
    float(*D)[CH_B] = sD[kb & 1];
#pragma unroll
    for (int j = 0; j < CH_B; ++j) {
      // rd = 1 / sqrt(p), d = sqrt(p): the fast reciprocal root and a Newton
      // step each (the IEEE root and division double this chain's latency)
      const float p = fmaxf(__shfl_sync(0xffffffffu, a[j], j), 1e-30f);
      const float r0 = rsqrtf(p), rd = fmaf(r0, fmaf(-0.5f * p * r0, r0, 0.5f), r0);
      const float d0 = p * rd, d = fmaf(fmaf(-d0, d0, p), 0.5f * rd, d0);
      const float l = lane == j ? d : lane > j ? a[j] * rd : 0.f;
      a[j] = l;
      if (lane == 0 && j < bw) s_rdiag[j0 + j] = rd;
#pragma unroll
      for (int c = j + 1; c < CH_B; ++c) {
        const float lc = __shfl_sync(0xffffffffu, l, c);
        a[c] = fmaf(-l, lc, a[c]);
      }
    }
    if (lane < CH_B)
#pragma unroll
      for (int c = 0; c < CH_B; ++c) {
        D[c][lane] = a[c];
        if (lane < bw && c <= lane) Ls[tri_off(j0 + lane) + j0 + c] = a[c];
      }
  };
  // the inverse of block kb's diagonal block (lane m: column m, forward
  // substitution against the transposed copy)
  auto invert_diag = [&](int kb) {
    const int j0 = kb * CH_B, bw = min(CH_B, L - j0);
    const float(*D)[CH_B] = sD[kb & 1];
    float x[CH_B];
#pragma unroll
    for (int i = 0; i < CH_B; ++i) x[i] = i == lane ? 1.f : 0.f;
#pragma unroll
    for (int p = 0; p < CH_B; ++p) {
      x[p] *= p < bw ? s_rdiag[j0 + p] : 1.f;
      float l[CH_B];
#pragma unroll
      for (int v = (p + 1) / 4; v < CH_B / 4; ++v)
        *reinterpret_cast<float4*>(l + 4 * v) = *reinterpret_cast<const float4*>(&D[p][4 * v]);
#pragma unroll
      for (int i = p + 1; i < CH_B; ++i) x[i] = fmaf(-l[i], x[p], x[i]);
    }
    if (lane < CH_B)
#pragma unroll
      for (int i = 0; i < CH_B; ++i)
        Dinv[(kb * CH_B + i) * CH_B + lane] = (i < bw && lane <= i) ? x[i] : 0.f;
  };
  if (warp == 0) {
    float a[CH_B];
    const int bw = min(CH_B, L);
#pragma unroll
    for (int c = 0; c < CH_B; ++c)
      a[c] = (lane < bw && c <= lane) ? Ls[tri_off(min(lane, bw - 1)) + c] : (c == lane ? 1.f : 0.f);
    factor_diag(0, a);
  }
  __syncthreads();
  for (int kb = 0; kb + 1 < nb; ++kb) {
    const int j0 = kb * CH_B, j1 = j0 + CH_B, nt = L - j1;
    // panel: row i solves x L_kk^T = a_i[j0 : j1] (rows below: the block is full)
    for (int i = j1 + tid; i < L; i += CH_THREADS) {
      float x[CH_B];
      float* Ai = Ls + tri_off(i) + j0;
#pragma unroll
      for (int c = 0; c < CH_B; ++c) x[c] = Ai[c];
#pragma unroll
      for (int c = 0; c < CH_B; ++c) {
        x[c] *= s_rdiag[j0 + c];
        float l[CH_B];
#pragma unroll
        for (int v = (c + 1) / 4; v < CH_B / 4; ++v)
          *reinterpret_cast<float4*>(l + 4 * v) = *reinterpret_cast<const float4*>(&sD[kb & 1][c][4 * v]);
#pragma unroll
        for (int c2 = c + 1; c2 < CH_B; ++c2) x[c2] = fmaf(-x[c], l[c2], x[c2]);
      }
#pragma unroll
      for (int c = 0; c < CH_B; ++c) {
        Ai[c] = x[c];
        Pt[c * ldp + (i - j1)] = x[c];
      }
    }
    __syncthreads();
    // trailing triangle: A_ic -= sum_m P_im P_cm
    const int n4 = (nt + 3) / 4, nd = min(n4, CH_B / 4);
    if (warp == 0) {
      // the next diagonal block: lane i its row i, then its factor
      const int bw = min(CH_B, nt), row = min(lane, bw - 1);
      float acc[CH_B];
#pragma unroll
      for (int c = 0; c < CH_B; ++c) acc[c] = 0.f;
#pragma unroll 4
      for (int m = 0; m < CH_B; ++m) {
        const float pi = Pt[m * ldp + row];
#pragma unroll
        for (int v = 0; v < CH_B / 4; ++v) {
          const float4 q = *reinterpret_cast<const float4*>(Pt + m * ldp + 4 * v);
          acc[4 * v] = fmaf(pi, q.x, acc[4 * v]);
          acc[4 * v + 1] = fmaf(pi, q.y, acc[4 * v + 1]);
          acc[4 * v + 2] = fmaf(pi, q.z, acc[4 * v + 2]);
          acc[4 * v + 3] = fmaf(pi, q.w, acc[4 * v + 3]);
        }
      }
#pragma unroll
      for (int c = 0; c < CH_B; ++c)
        acc[c] = (lane < bw && c <= lane) ? Ls[tri_off(j1 + row) + j1 + c] - acc[c] : (c == lane ? 1.f : 0.f);
      factor_diag(kb + 1, acc);
    } else {
      if (warp == nw - 1) invert_diag(kb);
      // the rows below it: four a warp, lanes along the columns
      for (int g0 = warp - 1; g0 < n4 - nd && warp < nw - 1; g0 += nw - 2) {
        const int rg = n4 - 1 - g0;
        for (int cb = 0; cb <= 4 * rg + 3; cb += 128) {
          float acc[4][4] = {};
#pragma unroll 4
          for (int m = 0; m < CH_B; ++m) {
            const float4 a = *reinterpret_cast<const float4*>(Pt + m * ldp + 4 * rg);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              if (cb + 32 * v > 4 * rg + 3) break;  // warp-uniform: right of the diagonal
              const float bv = Pt[m * ldp + cb + lane + 32 * v];
#pragma unroll
              for (int u = 0; u < 4; ++u) acc[u][v] = fmaf(av[u], bv, acc[u][v]);
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = j1 + 4 * rg + u;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const int c = j1 + cb + lane + 32 * v;
              if (i < L && c <= i) Ls[tri_off(i) + c] -= acc[u][v];
            }
          }
        }
      }
    }
    __syncthreads();
  }
  if (warp == 0) {
    invert_diag(nb - 1);
    return;
  }
  for (int i = warp - 1; i < L; i += nw - 1) {
    const float* Ai = Ls + tri_off(i);
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int c = lane + 32 * v;
      if (c < L) Lout[(size_t)i * L + c] = c <= i ? Ai[c] : 0.f;
    }
  }
}

__device__ __forceinline__ uint32_t os_smem(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Y = X L^-T for X [n][l] fp32 (the second half of a CholeskyQR pass): row by
// row, block column k of Y is (X_k - sum_{j < k} Y_j L_kj^T) Dinv_k^T, so the
// factor's inverse is never formed and half of the products of a full GEMM are
// left out.  One CTA takes TS_ROWS rows against the whole factor in shared
// memory (block rows of 16, each as long as it is, four words of padding so
// that eight rows read at once fall on distinct banks); thread (row, c) owns
// column c of a block.  Instruction latency of its few warps bounds it: at
// l = 136 16.8 us with two columns a thread and copies of 4 bytes, 9.7 so (the
// GEMM with the formed inverse took 13, but forming it 80 of the Cholesky's 152).
constexpr int TS_ROWS = 16;
constexpr int TS_THREADS = CH_B * TS_ROWS;
__host__ __device__ inline int ts_off(int kb) { return CH_B * (8 * kb * (kb + 1) + 4 * kb); }
__host__ __device__ inline int ts_ldy(int nb) { return nb * CH_B + 4; }

__global__ void __launch_bounds__(TS_THREADS)
k_trsm(const float* __restrict__ X, const float* __restrict__ Lf, const float* __restrict__ Dinv,
       int n, int L, int vec, float* __restrict__ Y) {
  extern __shared__ __align__(16) float ts[];
  const int nb = (L + CH_B - 1) / CH_B, ldy = ts_ldy(nb);
  float* Lb = ts;                       // block row kb at ts_off(kb), rows of 16 (kb + 1) + 4
  float* Ys = ts + ts_off(nb);          // [TS_ROWS][ldy]
  float* Ss = Ys + TS_ROWS * ldy;       // [TS_ROWS][CH_B + 4]
  float* Ds = Ss + TS_ROWS * (CH_B + 4);  // [nb][CH_B][CH_B + 4]
  const int tid = threadIdx.x, row0 = blockIdx.x * TS_ROWS;
  // every copy in flight at once: 16 bytes each where the rows allow it
  auto cp4 = [](float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(os_smem(dst)), "l"(src) : "memory");
  };
  auto cp16 = [](float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(os_smem(dst)), "l"(src) : "memory");
  };
  if (L % 4 == 0 && vec) {
    for (int r = tid >> 4; r < L; r += TS_THREADS / 16) {
      const int kb = r / CH_B, ld = CH_B * (kb + 1) + 4;
      float* dst = Lb + ts_off(kb) + (r - kb * CH_B) * ld;
      for (int c = 4 * (tid & 15); c < CH_B * kb; c += 64) cp16(dst + c, Lf + (size_t)r * L + c);
    }
    for (int r = tid >> 4; r < TS_ROWS; r += TS_THREADS / 16)
      for (int c = 4 * (tid & 15); c < nb * CH_B; c += 64) {
        if (row0 + r < n && c < L) cp16(Ys + r * ldy + c, X + (size_t)(row0 + r) * L + c);
        else *reinterpret_cast<float4*>(Ys + r * ldy + c) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
  } else {
    for (int r = tid >> 5; r < L; r += TS_THREADS / 32) {
      const int kb = r / CH_B, ld = CH_B * (kb + 1) + 4;
      float* dst = Lb + ts_off(kb) + (r - kb * CH_B) * ld;
      for (int c = tid & 31; c < CH_B * kb; c += 32) cp4(dst + c, Lf + (size_t)r * L + c);
    }
    for (int r = tid >> 5; r < TS_ROWS; r += TS_THREADS / 32)
      for (int c = tid & 31; c < nb * CH_B; c += 32) {
        if (row0 + r < n && c < L) cp4(Ys + r * ldy + c, X + (size_t)(row0 + r) * L + c);
        else Ys[r * ldy + c] = 0.f;
      }
  }
  for (int e = 4 * tid; e < nb * CH_B * CH_B; e += 4 * TS_THREADS)
    cp16(Ds + (e / CH_B) * (CH_B + 4) + e % CH_B, Dinv + e);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int c = tid % CH_B, r = tid / CH_B;
  float* yr = Ys + r * ldy;
  float* sr = Ss + r * (CH_B + 4);
  for (int kb = 0; kb < nb; ++kb) {
    const int j0 = kb * CH_B, ld = CH_B * (kb + 1) + 4;
    const float* l0 = Lb + ts_off(kb) + c * ld;
    float s0[4] = {};
    if (j0 + c < L) {  // a factor row that exists
#pragma unroll 4
      for (int j = 0; j < j0; j += 4) {
        const float4 y = *reinterpret_cast<const float4*>(yr + j);
        const float4 a = *reinterpret_cast<const float4*>(l0 + j);
        s0[0] = fmaf(y.x, a.x, s0[0]);
        s0[1] = fmaf(y.y, a.y, s0[1]);
        s0[2] = fmaf(y.z, a.z, s0[2]);
        s0[3] = fmaf(y.w, a.w, s0[3]);
      }
    }
    sr[c] = yr[j0 + c] - ((s0[0] + s0[1]) + (s0[2] + s0[3]));
    __syncwarp();  // a row's sixteen threads are in one warp
    const float* d0 = Ds + (j0 + c) * (CH_B + 4);
    float t0 = 0.f;
#pragma unroll
    for (int p = 0; p < CH_B; p += 4) {
      const float4 s = *reinterpret_cast<const float4*>(sr + p);
      const float4 a = *reinterpret_cast<const float4*>(d0 + p);
      t0 = fmaf(s.w, a.w, fmaf(s.z, a.z, fmaf(s.y, a.y, fmaf(s.x, a.x, t0))));
    }
    yr[j0 + c] = t0;
    __syncwarp();
  }
  __syncthreads();
  for (int q = tid >> 5; q < TS_ROWS; q += TS_THREADS / 32)
    for (int cc = tid & 31; cc < L; cc += 32)
      if (row0 + q < n) Y[(size_t)(row0 + q) * L + cc] = Ys[q * ldy + cc];
}

// Mt (column-major, Mt[j][i] = M[i][j]) of M = L1 L2 for lower-triangular
// L1, L2 [L][L] (fp32, sums to float64 accuracy).  CTA i, thread j.
__global__ void k_trmm(const float* __restrict__ L1, const float* __restrict__ L2, int L,
                       float* __restrict__ Mt) {
  const int i = blockIdx.x, j = threadIdx.x;
  if (j >= L) return;
  // two compensated sums (as in the Gram): a float64 fma and the widening of its
  // operands run at 1/64 of the fp32 rate.  Thirty-two loads in flight, and a
  // warp's lanes walk the same k from its first column on (zeros before a lane's
  // own), so that a load reads one row piece: 20.1 us at L = 136 with every lane starting at its column, 5.6 so.
  DF acc[2] = {DF{0.f, 0.f}, DF{0.f, 0.f}};
  for (int k = j & ~31; k <= i; k += 32) {
    float a[32], b[32];
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const bool in = k + u >= j && k + u <= i;
      a[u] = in ? L1[(size_t)i * L + k + u] : 0.f;
      b[u] = in ? L2[(size_t)(k + u) * L + j] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const float p = __fmul_rn(a[u], b[u]);
      df_add(acc[u & 1], p, __fmaf_rn(a[u], b[u], -p));
    }
  }
  df_add(acc[0], acc[1].hi, acc[1].lo);
  Mt[(size_t)j * L + i] = __fadd_rn(acc[0].hi, acc[0].lo);
}

// One-sided Jacobi SVD of M (Hestenes): the columns of M are orthogonalised by
// plane rotations applied from the right, M W = U S, W orthogonal.  For a pair:
// alpha = |m_p|^2, beta = |m_q|^2, gamma = m_p . m_q (fp32, each lane a strided
// share, then a butterfly that leaves every lane the same sums), and unless
// |gamma| <= 1e-6 sqrt(alpha beta) columns p, q of M and of W are rotated by the
// angle that makes them orthogonal (zeta = (beta - alpha) / (2 gamma),
// t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)), c = 1 / sqrt(1 + t^2), s = c t).
// Sweeps end when none of a sweep's pairs had |gamma| above 2e-5
// sqrt(alpha beta) (the rotations of that sweep leave products of such angles,
// below the rounding of an fp32 dot product), or after OS_MAX_SWEEPS.
//
// On one SM a round (half the columns against the other half) moves all of M
// and W through shared memory: 1.44 us at L = 136, 1.76 ms in all.  So the
// sweep is spread over a thread-block cluster of OS_P = 8 CTAs: the columns form
// 16 blocks of b, a CTA holds two, and a super-step rotates every pair across its
// two blocks in b rounds of b pairs (a half-warp keeps its column of the first
// block in registers, the second block's go round in shared memory); between
// super-steps the blocks are paired anew by the circle method, each block copied
// (cp.async.bulk between the CTAs' shared memories, 1 mbarrier a buffer) straight
// into the other buffer of the CTA that needs it next.  Pairs inside a block are
// rotated once a sweep, in its first super-step.  A round's latency bounds it (the
// reduction, the angle, a barrier).  Measured at L = 136: 570 us (892 with
// four CTAs, a warp a pair and the blocks fetched by loads).
// Output: Wt [L][L], Wt[j][k] = W[k][j].
constexpr int OS_MAX_SWEEPS = 30;
constexpr int OS_P = 8;           // CTAs of the cluster
constexpr int OS_MAX_WARPS = 8;   // 16 columns a block at L = 256, a half-warp each

__device__ __forceinline__ uint32_t os_map(uint32_t a, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
  return r;
}
__device__ __forceinline__ uint32_t os_ld_remote(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void os_cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void os_cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void os_cluster_sync() {
  os_cluster_arrive();
  os_cluster_wait();
}
// bounded wait for a phase of this CTA's mbarrier (its copies were issued by
// CTAs that are resident beside it, so it ends)
__device__ __forceinline__ bool os_wait(uint32_t bar, uint32_t parity) {
  const unsigned long long t0 = clock64();
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > kDefaultWaitCycles) return false;
  }
}
__device__ __forceinline__ float2 os_mul2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 os_fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float os_sqrt(float v) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// Rotates the columns x and y of this half-warp's pair (`on`: it has one).  A
// column is L rows of M, then L rows of W, 32 values a chunk, two a lane; the
// last chunk of M (v = KV - 1) is cut at L by m0, m1.  The tangent comes as
// 2 gamma / (|d| + sqrt(d^2 + 4 gamma^2)), d = beta - alpha, and may be off by
// its rounding (the next sweep sees what is left); the rotation may not be:
// c = 1 / sqrt(1 + t^2) takes a Newton step to full precision.  True if the
// pair was further than 2e-5 from orthogonal.
template <int KV>
__device__ __forceinline__ bool os_rotate(float2 (&x)[2 * KV], float2 (&y)[2 * KV], bool on, bool m0,
                                          bool m1) {
  float2 a2{0.f, 0.f}, b2{0.f, 0.f}, g2{0.f, 0.f};
#pragma unroll
  for (int v = 0; v < KV; ++v) {
    const float2 p = v + 1 < KV ? x[v] : make_float2(m0 ? x[v].x : 0.f, m1 ? x[v].y : 0.f);
    const float2 q = v + 1 < KV ? y[v] : make_float2(m0 ? y[v].x : 0.f, m1 ? y[v].y : 0.f);
    a2 = os_fma2(p, p, a2);
    b2 = os_fma2(q, q, b2);
    g2 = os_fma2(p, q, g2);
  }
  float a = a2.x + a2.y, b = b2.x + b2.y, g = g2.x + g2.y;
#pragma unroll
  for (int o = 8; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    g += __shfl_xor_sync(0xffffffffu, g, o);
  }
  const float ab = a * b, gg = g * g;
  if (!(on && gg > 1e-12f * ab)) return false;  // the same for the half-warp
  const float d = b - a, den = fabsf(d) + os_sqrt(fmaf(d, d, 4.f * gg));
  const float t = __fdividef(d >= 0.f ? 2.f * g : -2.f * g, fmaxf(den, 1e-37f));
  const float u = fmaf(t, t, 1.f), c0 = rsqrtf(u);
  const float c = fmaf(c0, fmaf(-0.5f * u * c0, c0, 0.5f), c0), sn = t * c;
  const float2 c2{c, c}, s2{sn, sn}, ns2{-sn, -sn};
#pragma unroll
  for (int v = 0; v < 2 * KV; ++v) {
    const float2 p = x[v], q = y[v];
    x[v] = os_fma2(c2, p, os_mul2(ns2, q));
    y[v] = os_fma2(s2, p, os_mul2(c2, q));
  }
  return gg > 4e-10f * ab;
}

// the two blocks of cluster rank c in super-step st of a sweep (n = 2 P blocks)
__device__ __forceinline__ void os_pair(int st, int c, int n, int& p, int& q) {
  p = st + c;
  if (p >= n - 1) p -= n - 1;
  q = st - c;
  if (q < 0) q += n - 1;
  if (c == 0) q = n - 1;
}
// where block k is in super-step st: cluster rank and which of its two
__device__ __forceinline__ void os_where(int k, int st, int n, int& c, int& h) {
  if (k == n - 1) {
    c = 0;
    h = 1;
    return;
  }
  const int d = k >= st ? k - st : k - st + n - 1;
  if (d < n / 2) {
    c = d;
    h = 0;
  } else {
    c = n - 1 - d;
    h = 1;
  }
}

template <int KV>
__global__ void __launch_bounds__(32 * OS_MAX_WARPS)
k_jacobi_cluster(const float* __restrict__ Mt, int L, int b, float* __restrict__ Wt) {
  constexpr int CL = 64 * KV;  // floats of a column: L of M, L of W, zeros
  constexpr int NC = 2 * KV;   // its chunks of 32
  constexpr int NBLK = 2 * OS_P, NST = NBLK - 1;
  extern __shared__ __align__(128) float osm[];  // [2 buffers][2 blocks][b columns][CL]
  __shared__ __align__(8) uint64_t s_full[2];    // by buffer: both blocks have landed
  __shared__ unsigned s_far[2];  // by sweep parity: a pair of this CTA was far from orthogonal
  __shared__ unsigned s_max, s_go;
  const int tid = threadIdx.x, lane = tid & 31, hl = lane & 15;
  const int w = 2 * (tid >> 5) + (lane >> 4);  // this half-warp's pair
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int bb = b + (b & 1);
  const bool m0 = 32 * (KV - 1) + 2 * hl < L, m1 = 32 * (KV - 1) + 2 * hl + 1 < L;
  const bool on = w < b;
  const uint32_t base = os_smem(osm), full0 = os_smem(s_full);
  const uint32_t blk_bytes = (uint32_t)(b * CL) * 4u;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_far[0] = s_far[1] = s_max = 0;
  }
  __syncthreads();
  int pb, qb;
  os_pair(0, (int)rank, NBLK, pb, qb);
  float2 x[NC], y[NC];
  // the first super-step's columns; M scaled by a power of two so that its
  // largest entry is near 1 (the squares below then neither overflow nor, for
  // any column that counts, underflow; W does not see the scale)
  {
    const int cx = pb * b + w, cy = qb * b + w;
    float mx = 0.f;
    auto first = [&](int col, int e) {  // element e of column col before any rotation
      if (!on || col >= L || e >= 2 * L) return 0.f;
      if (e >= L) return e - L == col ? 1.f : 0.f;
      const float v = Mt[(size_t)col * L + e];
      mx = fmaxf(mx, fabsf(v));
      return v;
    };
#pragma unroll
    for (int v = 0; v < NC; ++v) {
      const int e = 32 * v + 2 * hl;
      x[v] = make_float2(first(cx, e), first(cx, e + 1));
      y[v] = make_float2(first(cy, e), first(cy, e + 1));
    }
    atomicMax(&s_max, __float_as_uint(mx));
    __syncthreads();
    os_cluster_sync();  // also: every CTA's mbarriers are initialised
    unsigned m = 0;
    for (int c = 0; c < OS_P; ++c) m = max(m, os_ld_remote(os_map(os_smem(&s_max), (uint32_t)c)));
    const int ex = min(max((int)(m >> 23) - 127, -120), 120);
    const float sc = m ? __uint_as_float((uint32_t)(127 - ex) << 23) : 1.f;
    float* B = osm + 2 * hl;
    if (on)
#pragma unroll
      for (int v = 0; v < NC; ++v) {
        const int e = 32 * v + 2 * hl;
        if (e < L) x[v].x *= sc, y[v].x *= sc;
        if (e + 1 < L) x[v].y *= sc, y[v].y *= sc;
        *reinterpret_cast<float2*>(B + (size_t)w * CL + 32 * v) = x[v];
        *reinterpret_cast<float2*>(B + (size_t)(b + w) * CL + 32 * v) = y[v];
      }
    __syncthreads();
  }
  bool alive = true, far = false;
  int sweep = 0, st = 0;
  for (uint32_t k = 0;; ++k) {
    const uint32_t cur = k & 1;
    os_pair(st, (int)rank, NBLK, pb, qb);
    float* B = osm + (size_t)cur * 2 * b * CL + 2 * hl;
    if (k > 0 && alive) alive = os_wait(full0 + 8 * cur, ((k - 1) >> 1) & 1);
    __syncwarp();
    os_cluster_arrive();  // this CTA holds its blocks of super-step k
    if (st == 0) {
      // the pairs inside each of the two blocks: half-warps 0 .. bb/2 - 1 the
      // first, the next bb/2 the second (circle method on bb columns)
      const int half = bb / 2, g = w < half ? w : w - half;
      for (int rd = 0; rd < bb - 1; ++rd) {
        int i = rd, j = bb - 1;
        if (g > 0) {
          i = rd + g;
          if (i >= bb - 1) i -= bb - 1;
          j = rd - g;
          if (j < 0) j += bb - 1;
        }
        const bool in = w < bb && i < b && j < b;
        float* ci = B + (size_t)((w < half ? 0 : b) + (in ? i : 0)) * CL;
        float* cj = B + (size_t)((w < half ? 0 : b) + (in ? j : 0)) * CL;
#pragma unroll
        for (int v = 0; v < NC; ++v) {
          x[v] = in ? *reinterpret_cast<const float2*>(ci + 32 * v) : make_float2(0.f, 0.f);
          y[v] = in ? *reinterpret_cast<const float2*>(cj + 32 * v) : make_float2(0.f, 0.f);
        }
        far |= os_rotate<KV>(x, y, in, m0, m1);
        if (in)
#pragma unroll
          for (int v = 0; v < NC; ++v) {
            *reinterpret_cast<float2*>(ci + 32 * v) = x[v];
            *reinterpret_cast<float2*>(cj + 32 * v) = y[v];
          }
        __syncthreads();
      }
    }
#pragma unroll
    for (int v = 0; v < NC; ++v)
      x[v] = on ? *reinterpret_cast<const float2*>(B + (size_t)w * CL + 32 * v) : make_float2(0.f, 0.f);
    // every pair across the two blocks
    for (int rd = 0; rd < b; ++rd) {
      int j = w + rd;
      if (j >= b) j -= b;
      float* cj = B + (size_t)(b + (on ? j : 0)) * CL;
#pragma unroll
      for (int v = 0; v < NC; ++v)
        y[v] = on ? *reinterpret_cast<const float2*>(cj + 32 * v) : make_float2(0.f, 0.f);
      far |= os_rotate<KV>(x, y, on, m0, m1);
      if (on)
#pragma unroll
        for (int v = 0; v < NC; ++v) *reinterpret_cast<float2*>(cj + 32 * v) = y[v];
      __syncthreads();
    }
    if (on)
#pragma unroll
      for (int v = 0; v < NC; ++v) *reinterpret_cast<float2*>(B + (size_t)w * CL + 32 * v) = x[v];
    const bool last = st == NST - 1;
    if (last && far && hl == 0) s_far[sweep & 1] = 1;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the copies read the columns
    __syncthreads();
    os_cluster_wait();  // every CTA holds its blocks of super-step k: the other buffers are free
    if (last) {
      // every CTA reads the same flags, so all leave after the same sweep
      os_cluster_sync();
      if (tid == 0) {
        unsigned go = 0;
        for (int c = 0; c < OS_P; ++c) go |= os_ld_remote(os_map(os_smem(&s_far[sweep & 1]), (uint32_t)c));
        s_go = go;
        s_far[(sweep + 1) & 1] = 0;  // last read a sweep ago
      }
      __syncthreads();
      ++sweep;
      if (!s_go || sweep == OS_MAX_SWEEPS) break;
      far = false;
    }
    st = last ? 0 : st + 1;
    if (tid == 0) {
      // each block straight into the other buffer of the CTA that needs it next
      const uint32_t nbuf = cur ^ 1;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full0 + 8 * nbuf),
                   "r"(2 * blk_bytes)
                   : "memory");
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int c, hd;
        os_where(h ? qb : pb, st, NBLK, c, hd);
        const uint32_t src = base + (cur * 2 + h) * blk_bytes;
        const uint32_t dst = os_map(base + (nbuf * 2 + hd) * blk_bytes, (uint32_t)c);
        const uint32_t bar = os_map(full0 + 8 * nbuf, (uint32_t)c);
        asm volatile(
            "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
            "r"(src), "r"(blk_bytes), "r"(bar)
            : "memory");
      }
    }
    __syncwarp();
  }
  // this CTA's columns are in the buffer worked on last
  os_pair(NST - 1, (int)rank, NBLK, pb, qb);
  // (the buffer's parity is that of the super-steps done, NST a sweep)
  const float* B = osm + (size_t)((sweep * NST - 1) & 1) * 2 * b * CL;
  if (on)
    for (int h = 0; h < 2; ++h) {
      const int col = (h ? qb : pb) * b + w;
      if (col >= L) continue;
      for (int i = hl; i < L; i += 16) Wt[(size_t)col * L + i] = B[(size_t)(h * b + w) * CL + L + i];
    }
  __syncwarp();
  os_cluster_sync();  // no CTA leaves while its flags are read
}

// CTA j: v = M w_j to float64 accuracy, sigma_j = |v| / |w_j| (the Rayleigh quotient of
// the converged rotation, second-order accurate in the rotation's error);
// MWn[j] = v / |w_j|, Wn[j] = w_j / |w_j| (fp32, column j stored contiguously).
__global__ void __launch_bounds__(256)
k_ritz(const float* __restrict__ Mt, const float* __restrict__ Wt, int L, float* __restrict__ MWn,
       float* __restrict__ Wn, double* __restrict__ sig64) {
  __shared__ float w[256];
  __shared__ double red[2][8];
  __shared__ double s_inv;
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int k = tid; k < L; k += 256) w[k] = Wt[(size_t)j * L + k];
  __syncthreads();
  double v = 0.0, ww = 0.0;
  if (tid < L) {
    // two compensated sums (as in the Gram), thirty-two loads in flight
    DF p2[2] = {DF{0.f, 0.f}, DF{0.f, 0.f}};
    for (int k = 0; k < L; k += 32) {
      float m[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) m[u] = k + u < L ? Mt[(size_t)(k + u) * L + tid] : 0.f;
#pragma unroll
      for (int u = 0; u < 32; ++u) {
        const float wv = k + u < L ? w[k + u] : 0.f;
        const float p = __fmul_rn(m[u], wv);
        df_add(p2[u & 1], p, __fmaf_rn(m[u], wv, -p));
      }
    }
    df_add(p2[0], p2[1].hi, p2[1].lo);
    v = (double)p2[0].hi + (double)p2[0].lo;
    ww = (double)w[tid] * (double)w[tid];
  }
  double v2 = v * v, w2 = ww;
  for (int o = 16; o; o >>= 1) {
    v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    w2 += __shfl_xor_sync(0xffffffffu, w2, o);
  }
  if (lane == 0) {
    red[0][warp] = v2;
    red[1][warp] = w2;
  }
  __syncthreads();
  if (tid == 0) {
    // the float64 root and division once: they run at a fraction of the fp32 rate
    double tv = 0.0, tw = 0.0;
    for (int q = 0; q < 8; ++q) {
      tv += red[0][q];
      tw += red[1][q];
    }
    const double nw_ = sqrt(tw);
    s_inv = nw_ > 0.0 ? 1.0 / nw_ : 0.0;
    sig64[j] = nw_ > 0.0 ? sqrt(tv) / nw_ : 0.0;
  }
  __syncthreads();
  if (tid < L) {
    const double inv = s_inv;
    MWn[(size_t)j * L + tid] = (float)(v * inv);
    Wn[(size_t)j * L + tid] = (float)((double)w[tid] * inv);
  }
}

// CTA k (of L): the r largest sigma (ties: lower index first) and row k of the
// fp32 matrices Wu [L][r] = MWn[i_c] / sqrt(sigma_c), Wv [L][r] = Wn[i_c]
// sqrt(sigma_c) (zero for sigma_c <= 1e-6 sigma_0), so that Q Wu = U_r S_r^(1/2)
// and Z2 Wv = V_r S_r^(1/2) (Eq. factors); CTA 0 writes sig [r] fp32.  Every CTA
// ranks the sigma for itself (non-negative float64 values compare as their
// bits do), so that no single CTA takes the L r square roots and divisions:
// 87 us with one CTA, 6.7 us now at L = 136, r = 128.
__global__ void __launch_bounds__(256)
k_finish(const double* __restrict__ sig64, const float* __restrict__ MWn,
         const float* __restrict__ Wn, int L, int r, float* __restrict__ Wu,
         float* __restrict__ Wv, float* __restrict__ sig) {
  __shared__ double sv[256];
  __shared__ int order[256];
  const int tid = threadIdx.x, k = blockIdx.x;
  if (tid < L) sv[tid] = sig64[tid];
  __syncthreads();
  if (tid < L) {
    const unsigned long long* sb = reinterpret_cast<const unsigned long long*>(sv);
    const unsigned long long si = sb[tid];
    int rk = 0;
#pragma unroll 4
    for (int j = 0; j < L; ++j) rk += (sb[j] > si || (sb[j] == si && j < tid)) ? 1 : 0;
    order[rk] = tid;
  }
  __syncthreads();
  if (tid < r) {
    const double s0 = sv[order[0]];
    const int i = order[tid];
    const double sg = sv[i];
    const bool keep = sg > 1e-6 * s0 && sg > 0.0;
    const float rs = (float)sqrt(sg);
    Wu[(size_t)k * r + tid] = keep ? MWn[(size_t)i * L + k] / rs : 0.f;
    Wv[(size_t)k * r + tid] = keep ? Wn[(size_t)i * L + k] * rs : 0.f;
    if (k == 0) sig[tid] = (float)sg;
  }
}

// Column c of U [rows][r]: the entry of largest magnitude (lowest row on
// ties) is made positive by negating U[:, c] and V[:, c] together.
__global__ void k_sign(float* __restrict__ U, float* __restrict__ V, int rows, int cols, int r) {
  __shared__ float bv[32];
  __shared__ int bi[32];
  __shared__ float s_sign;
  const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float best = -1.f;
  int bidx = 0x7fffffff;
  for (int m = tid; m < rows; m += blockDim.x) {
    const float a = fabsf(U[(size_t)m * r + c]);
    if (a > best || (a == best && m < bidx)) {
      best = a;
      bidx = m;
    }
  }
  for (int o = 16; o; o >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
    if (ob > best || (ob == best && oi < bidx)) {
      best = ob;
      bidx = oi;
    }
  }
  if (lane == 0) {
    bv[warp] = best;
    bi[warp] = bidx;
  }
  __syncthreads();
  if (tid == 0) {
    float b = -1.f;
    int i = 0x7fffffff;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w)
      if (bv[w] > b || (bv[w] == b && bi[w] < i)) {
        b = bv[w];
        i = bi[w];
      }
    s_sign = (i < rows && U[(size_t)i * r + c] < 0.f) ? -1.f : 1.f;
  }
  __syncthreads();
  if (s_sign < 0.f) {
    for (int m = tid; m < rows; m += blockDim.x) U[(size_t)m * r + c] = -U[(size_t)m * r + c];
    for (int m = tid; m < cols; m += blockDim.x) V[(size_t)m * r + c] = -V[(size_t)m * r + c];
  }
}

bool g_ch_cap[64] = {};
bool g_ts_cap[64] = {};
bool g_jac_cap[8][64] = {};

}  // namespace
}  // namespace lx

namespace lx {
namespace {
constexpr int CP_MAX_L = 256;
constexpr size_t CP_SMEM_CAP = 200 * 1024;

size_t al256(size_t v) { return (v + 255) / 256 * 256; }

struct CompressWs {
  float *y0, *y1, *z0, *z1, *Dinv, *Wu, *Wv, *L1, *L2, *Mt, *Wt, *MWn, *Wn;
  double* sig64;
  char* tc;  // the tensor-core residual products' scratch (bf16 weights)
  size_t bytes;
};

// Carves the workspace (each piece 256-byte aligned from `base`; base == NULL
// only sizes it).
CompressWs carve(char* base, long rows, long cols, long l, long r) {
  CompressWs w{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + off : nullptr;
    off += al256(bytes);
    return p;
  };
  w.y0 = (float*)take(4 * rows * l);
  w.y1 = (float*)take(4 * rows * l);
  w.z0 = (float*)take(4 * cols * l);
  w.z1 = (float*)take(4 * cols * l);
  w.Dinv = (float*)take(4 * CH_B * (l + CH_B));
  w.Wu = (float*)take(4 * l * r);
  w.Wv = (float*)take(4 * l * r);
  w.L1 = (float*)take(4 * l * l);
  w.L2 = (float*)take(4 * l * l);
  w.Mt = (float*)take(4 * l * l);
  w.Wt = (float*)take(4 * l * l);
  w.MWn = (float*)take(4 * l * l);
  w.Wn = (float*)take(4 * l * l);
  w.sig64 = (double*)take(8 * l);
  w.tc = take(res_tc_workspace(rows, cols, l));
  w.bytes = off;
  return w;
}

lx_status check_compress(int32_t rows, int32_t cols, int32_t l, int32_t r) {
  if (rows < 8 || cols < 8 || rows % 8 || cols % 8 || rows > 65536 || cols > 65536)
    return fail(LX_ERR_SHAPE, "rows and cols must be multiples of 8 in 8..65536");
  if (r < 1 || l < r || l > CP_MAX_L || l > std::min(rows, cols))
    return fail(LX_ERR_SHAPE, "need 1 <= r <= l <= min(rows, cols, 256)");
  return LX_OK;
}

template <typename TW>
lx_status run_compress(int rows, int cols, const TW* Wd, const TW* Wm, const float* omega, int l,
                       int r, int q, float* U, float* V, float* sigma, const CompressWs& w,
                       int dev, cudaStream_t s) {
  int num_sms = 0;
  LX_CUDA(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
  // bf16 weights: the residual products R X and R^T X on the tensor cores
  constexpr bool bf16_w = std::is_same<TW, __nv_bfloat16>::value;
  const bool res_tc = bf16_w && res_tc_fits(rows, cols, l);
  lx_status tc_status = LX_OK;
  bool have_wt = false;  // W^T of this call's weights lies in w.tc
  auto gemm = [&](int mode, const float* X, const float* B, float* C, int M, int N, int K) {
    const dim3 grid((N + CG_TILE - 1) / CG_TILE, (M + CG_TILE - 1) / CG_TILE);
    if constexpr (bf16_w) {
      if (res_tc && (mode == A_RES || mode == A_RES_T)) {
        const lx_status st = res_gemm_tc(mode == A_RES_T, reinterpret_cast<const __nv_bfloat16*>(Wm),
                                         reinterpret_cast<const __nv_bfloat16*>(Wd), rows, cols, B, N,
                                         C, w.tc, &have_wt, num_sms, dev, s);
        if (st != LX_OK) tc_status = st;
        return;
      }
    }
    if (mode == A_RES)
      k_cgemm<TW, A_RES><<<grid, CG_THREADS, 0, s>>>(Wm, Wd, nullptr, cols, B, C, M, N, K);
    else if (mode == A_RES_T)
      k_cgemm<TW, A_RES_T><<<grid, CG_THREADS, 0, s>>>(Wm, Wd, nullptr, cols, B, C, M, N, K);
    else
      k_cgemm<TW, A_F32><<<grid, CG_THREADS, 0, s>>>(nullptr, nullptr, X, cols, B, C, M, N, K);
  };
  // CholeskyQR pass X -> out [n][l] (X L^-T, orthonormal columns when the Gram
  // is well conditioned).  The row ranges' Gram sums lie in the residual
  // products' partials, which are idle here.
  float2* const G = reinterpret_cast<float2*>(w.tc + res_tc_part_offset(rows, cols, l));
  const int ldp = ch_ldp(l), nb = (l + CH_B - 1) / CH_B;
  const size_t ch_smem = sizeof(float) * ((((size_t)l * (l + 1) / 2 + 3) & ~(size_t)3) + (size_t)CH_B * ldp);
  const size_t ts_smem = sizeof(float) * ((size_t)ts_off(nb) + TS_ROWS * ts_ldy(nb) +
                                          (TS_ROWS + nb * CH_B) * (CH_B + 4));
  LX_CUDA(smem_cap_once((const void*)k_chol32, (int)CP_SMEM_CAP, dev, g_ch_cap));
  LX_CUDA(smem_cap_once((const void*)k_trsm, (int)CP_SMEM_CAP, dev, g_ts_cap));
  auto cholqr = [&](const float* X, float* out, int n, float shift, float* Lf) {
    const int want = gram_parts(n, l, num_sms);
    const int span = ((n + want - 1) / want + GR_KC - 1) / GR_KC * GR_KC;
    const int parts = (n + span - 1) / span;
    const dim3 grid((l + GR_T - 1) / GR_T, (l + GR_T - 1) / GR_T, parts);
    k_gram<<<grid, GR_T * GR_T, 0, s>>>(X, n, l, span, G);
    k_chol32<<<1, CH_THREADS, ch_smem, s>>>(G, parts, l, ldp, shift, Lf, w.Dinv);
    k_trsm<<<(n + TS_ROWS - 1) / TS_ROWS, TS_THREADS, ts_smem, s>>>(X, Lf, w.Dinv, n, l,
                                                                        reinterpret_cast<uintptr_t>(X) % 16 == 0, out);
  };
  // CholeskyQR (the first pass shifted by 1e-6 of the largest Gram diagonal,
  // so rank-deficient bases stay factorable).  orth2 runs it twice, X [n][l]
  // ends orthonormal and its two factors stay in L1, L2; orth1 runs the
  // shifted pass once, for the intermediate bases of the power iterations,
  // whose span is all the next product uses (the final Q and Z take orth2).
  // Both leave the result in *X; *tmp is scratch.
  auto orth1 = [&](float** X, float** tmp, int n) {
    cholqr(*X, *tmp, n, 1e-6f, w.L1);
    std::swap(*X, *tmp);
  };
  auto orth2 = [&](float** X, float** tmp, int n) {
    cholqr(*X, *tmp, n, 1e-6f, w.L1);
    cholqr(*tmp, *X, n, 0.f, w.L2);
  };
  float *yc = w.y0, *yt = w.y1, *zc = w.z0, *zt = w.z1;
  gemm(A_RES, nullptr, omega, yc, rows, l, cols);  // Y = R Omega
  if (q == 0) orth2(&yc, &yt, rows);              // Q
  else orth1(&yc, &yt, rows);
  for (int it = 0; it < q; ++it) {
    gemm(A_RES_T, nullptr, yc, zc, cols, l, rows);  // R^T Q
    orth1(&zc, &zt, cols);
    gemm(A_RES, nullptr, zc, yc, rows, l, cols);    // R Z
    if (it + 1 == q) orth2(&yc, &yt, rows);
    else orth1(&yc, &yt, rows);
  }
  // Z = R^T Q = Bs^T = Z2 (L1 L2)^T with Z2 orthonormal, so Bs = M Z2^T for
  // M = L1 L2, and the SVD of Bs follows from the small SVD of M.
  gemm(A_RES_T, nullptr, yc, zc, cols, l, rows);
  orth2(&zc, &zt, cols);
  k_trmm<<<l, 256, 0, s>>>(w.L1, w.L2, l, w.Mt);
  {
    const int b = (l + 2 * OS_P - 1) / (2 * OS_P), kv = (l + 31) / 32;
    auto launch = [&](auto kern) -> lx_status {
      const size_t smem = sizeof(float) * 2 * 2 * b * (size_t)(64 * kv);
      LX_CUDA(smem_cap_once((const void*)kern, (int)CP_SMEM_CAP, dev, g_jac_cap[kv - 1]));
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(OS_P);
      cfg.blockDim = dim3(32 * ((b + 1) / 2));
      cfg.dynamicSmemBytes = smem;
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = OS_P;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      LX_CUDA(cudaLaunchKernelEx(&cfg, kern, (const float*)w.Mt, l, b, w.Wt));
      return LX_OK;
    };
    switch (kv) {
      case 1: LX_TRY(launch(k_jacobi_cluster<1>)); break;
      case 2: LX_TRY(launch(k_jacobi_cluster<2>)); break;
      case 3: LX_TRY(launch(k_jacobi_cluster<3>)); break;
      case 4: LX_TRY(launch(k_jacobi_cluster<4>)); break;
      case 5: LX_TRY(launch(k_jacobi_cluster<5>)); break;
      case 6: LX_TRY(launch(k_jacobi_cluster<6>)); break;
      case 7: LX_TRY(launch(k_jacobi_cluster<7>)); break;
      default: LX_TRY(launch(k_jacobi_cluster<8>)); break;
    }
  }
  k_ritz<<<l, 256, 0, s>>>(w.Mt, w.Wt, l, w.MWn, w.Wn, w.sig64);
  k_finish<<<l, 256, 0, s>>>(w.sig64, w.MWn, w.Wn, l, r, w.Wu, w.Wv, sigma);
  gemm(A_F32, yc, w.Wu, U, rows, r, l);   // U_r S^(1/2)
  gemm(A_F32, zc, w.Wv, V, cols, r, l);   // V_r S^(1/2)
  k_sign<<<r, 256, 0, s>>>(U, V, rows, cols, r);
  LX_CUDA(cudaGetLastError());
  return tc_status;
}
}  // namespace
}  // namespace lx

extern "C" lx_status lx_compress_workspace(int32_t rows, int32_t cols, int32_t l, int32_t r,
                                           uint64_t* bytes) {
  using namespace lx;
  if (!bytes) return fail(LX_ERR_ARG, "bytes is NULL");
  LX_TRY(check_compress(rows, cols, l, r));
  *bytes = carve(nullptr, rows, cols, l, r).bytes;
  return LX_OK;
}

extern "C" lx_status lx_compress_factor(int32_t dtype, int32_t rows, int32_t cols,
                                        const void* w_dom, const void* w_mem, const float* omega,
                                        int32_t l, int32_t r, int32_t power_iters, float* U,
                                        float* V, float* sigma, void* workspace,
                                        uint64_t workspace_bytes, void* stream) {
  using namespace lx;
  if (dtype != LX_F32 && dtype != LX_BF16) return fail(LX_ERR_ARG, "unknown dtype");
  LX_TRY(check_compress(rows, cols, l, r));
  if (power_iters < 0 || power_iters > 16) return fail(LX_ERR_ARG, "power_iters outside 0..16");
  if (!w_dom || !w_mem || !omega || !U || !V || !sigma || !workspace)
    return fail(LX_ERR_ARG, "NULL pointer");
  if (((uintptr_t)w_dom & 15u) || ((uintptr_t)w_mem & 15u))
    return fail(LX_ERR_ARG, "w_dom and w_mem must be 16-byte aligned");
  if ((uintptr_t)workspace & 255u) return fail(LX_ERR_ARG, "workspace must be 256-byte aligned");
  const CompressWs w = carve((char*)workspace, rows, cols, l, r);
  if (workspace_bytes < w.bytes) return fail(LX_ERR_ARG, "workspace too small");
  int dev = 0;
  LX_CUDA(cudaGetDevice(&dev));
  cudaStream_t s = (cudaStream_t)stream;
  if (dtype == LX_BF16)
    return run_compress(rows, cols, (const __nv_bfloat16*)w_dom, (const __nv_bfloat16*)w_mem,
                        omega, l, r, power_iters, U, V, sigma, w, dev, s);
  return run_compress(rows, cols, (const float*)w_dom, (const float*)w_mem, omega, l, r,
                      power_iters, U, V, sigma, w, dev, s);
}
