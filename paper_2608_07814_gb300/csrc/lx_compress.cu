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
//               two-sum accumulation on the fp32 pipes), stored as the unevaluated
//               fp32 pairs of four interleaved row sets.
//   k_chol32    one CTA: Cholesky G + s I = L L^T (fp32 in shared memory,
//               blocked by 16 columns; a small relative shift in the first
//               pass keeps rank-deficient bases factorable).
//   k_tri_inverse
//               L^-T, a CTA per 16 columns of the inverse; X L^-T then has
//               orthonormal columns (CholeskyQR).
//   k_trmm      M = L1 L2 (float64 sums), the triangular factor of R^T Q = Z2 M^T.
//   k_jacobi_cluster
//               one-sided Jacobi SVD of M, M W = U S, over a thread-block
//               cluster (fp32 rotations, columns handed on through distributed
//               shared memory).
//   k_ritz      sigma_j = |M w_j| / |w_j| in float64 (Rayleigh quotients).
//   k_finish    the r largest sigma and the fp32 matrices that turn the bases
//               into the split factors.
//   k_sign      each factor column's largest-magnitude entry of U made
//               positive (U and V negated together).
// The Gram sums reach float64 accuracy by compensated fp32 arithmetic (this
// GPU's float64 rate is a small fraction of its fp32 rate); M and the Rayleigh
// quotients are summed in float64.
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
// such pairs (independent chains) take the rows in turn
// (rows 4 t + c are chain c's) and are added pairwise at the end.  A CTA takes
// 16 x 16 outputs and one of the chains (blockIdx.z), so that the tiles on or
// below the diagonal (45 at L = 136; the Cholesky reads the lower triangle
// alone) make 180 CTAs, and the Cholesky adds the chains in the same order as
// one thread with all four would: 26.9 us a launch with one, 20.1 so (L = 136,
// mean over n = 768 and 2048).  The issue rate bounds it.  Ranges of
// consecutive rows in place of the chains cost the same and round differently.
// Each chunk of 64 chain rows is staged in shared memory while the next one is
// already loading into registers.
constexpr int GR_T = 16;
constexpr int GR_KC = 64;
constexpr int GR_CH = 4;
static_assert(GR_KC * GR_T % (GR_T * GR_T) == 0, "whole staged values per thread");

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
k_gram(const float* __restrict__ X, int n, int L, float2* __restrict__ Gp) {
  constexpr int PER = GR_KC * GR_T / (GR_T * GR_T);  // staged values per thread and side
  __shared__ float Xi[GR_KC][GR_T], Xj[GR_KC][GR_T];
  if (blockIdx.x > blockIdx.y) return;  // strictly above the diagonal
  const int z = blockIdx.z;
  const int nz = n > z ? (n - z + GR_CH - 1) / GR_CH : 0;  // rows of this chain
  float2* G = Gp + (size_t)z * L * L;
  const int ti = threadIdx.x / GR_T, tj = threadIdx.x % GR_T;
  const int i0 = blockIdx.y * GR_T, j0 = blockIdx.x * GR_T;
  DF acc{0.f, 0.f};
  // the next chunk's rows are loaded into registers while this one is summed
  float ri[PER], rj[PER];
  auto fetch = [&](int m0) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int q = threadIdx.x + e * GR_T * GR_T;
      const int mr = m0 + q / GR_T, c = q % GR_T;
      const size_t at = ((size_t)GR_CH * mr + z) * L;
      ri[e] = (mr < nz && i0 + c < L) ? X[at + i0 + c] : 0.f;
      rj[e] = (mr < nz && j0 + c < L) ? X[at + j0 + c] : 0.f;
    }
  };
  fetch(0);
  for (int m0 = 0; m0 < nz; m0 += GR_KC) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int q = threadIdx.x + e * GR_T * GR_T;
      Xi[q / GR_T][q % GR_T] = ri[e];
      Xj[q / GR_T][q % GR_T] = rj[e];
    }
    __syncthreads();
    if (m0 + GR_KC < nz) fetch(m0 + GR_KC);
#pragma unroll 16
    for (int mr = 0; mr < GR_KC; ++mr) {
      const float x = Xi[mr][ti], y = Xj[mr][tj];
      const float p = __fmul_rn(x, y);
      df_add(acc, p, __fmaf_rn(x, y, -p));
    }
    __syncthreads();
  }
  if (i0 + ti < L && j0 + tj < L) G[(size_t)(i0 + ti) * L + j0 + tj] = make_float2(acc.hi, acc.lo);
}

// (chain 0 + chain 1) + (chain 2 + chain 3) of a Gram entry, each pair added as
// hi + lo
__device__ __forceinline__ DF gram_sum(const float2 (&g)[GR_CH]) {
  DF s01{g[0].x, g[0].y}, s23{g[2].x, g[2].y};
  df_add(s01, g[1].x, g[1].y);
  df_add(s23, g[3].x, g[3].y);
  df_add(s01, s23.hi, s23.lo);
  return s01;
}
static_assert(GR_CH == 4, "gram_sum adds four chains");

// One CTA (L <= 256).  Cholesky of G + s I in fp32 (the chains of G added in
// order and rounded once; s = shift_rel * max diag(G)) in a
// packed lower triangle in shared memory (L (L + 1) / 2 floats, row i from
// i (i + 1) / 2), pivots floored at 1e-30, blocked by 16 columns (right-looking).
// One SM's latency bounds it, so each part keeps its chain in registers: warp 0
// factors the diagonal block with lane i holding row i (shuffles, no shared
// memory), one thread per row below solves its 16 panel entries against it
// (vector loads of a transposed copy), and the trailing triangle takes the
// panel's rank-16 update with a warp on four rows, lanes along the columns.
// The factor goes to Lout [L][L] (zero above the diagonal) and the inverses of
// its 16 x 16 diagonal blocks to Dinv [blocks][16][16], from which the kernel
// below forms the rest of the inverse (one block is the whole of it: L <= 16 gives
// T = L^-T here, and that launch is saved).  A zero Gram gives Lout = Dinv = 0.  The
// roots and reciprocals are the correctly rounded ones: a Newton step on the
// fast reciprocal root shortens the diagonal's chain by 6 us at the cost of up to
// an ulp.  Measured at L = 136: 152 us with in-place shared-memory steps and
// the whole inverse formed here, 47 us now.
constexpr int CH_THREADS = 512;  // 16 warps: at most 16 diagonal blocks
constexpr int CH_B = 16;  // block width
__device__ __forceinline__ int tri_off(int i) { return i * (i + 1) / 2; }
inline int ch_ldp(int L) { return (L + 127) / 128 * 128; }  // panel copy: whole column chunks

__global__ void __launch_bounds__(CH_THREADS, 1)
k_chol32(const float2* __restrict__ Gp, int L, int ldp, float shift_rel, float* __restrict__ Lout,
         float* __restrict__ Dinv, float* __restrict__ T) {
  extern __shared__ __align__(16) float Ls[];
  float* Pt = Ls + ((tri_off(L) + 3) & ~3);          // [CH_B][ldp] panel, transposed
  __shared__ __align__(16) float sD[2][CH_B][CH_B];  // by block parity: sD[c][i] = l_ic of the diagonal block
  __shared__ double s_md;
  __shared__ float s_rdiag[256];  // reciprocals of the factor's diagonal
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = CH_THREADS / 32;
  const int nb = (L + CH_B - 1) / CH_B;
  // the lower triangle of G rounded to fp32, a batch's loads in flight at once
  // (rows q and L - 1 - q together hold L + 1 entries: entry e of the fold)
  const int nfold = (L + 1) / 2 * (L + 1);
  constexpr int U = 5;
  for (int e0 = tid; e0 < nfold; e0 += U * CH_THREADS) {
    float2 g[U][GR_CH];
    int at[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * CH_THREADS, q = e / (L + 1), pos = e - q * (L + 1);
      const bool low = pos < L - q;  // row L - 1 - q, else row q
      const int i = low ? L - 1 - q : q, c = low ? pos : pos - (L - q);
      const bool ok = e < nfold && (low || 2 * q != L - 1);  // (an odd L's middle row once)
      at[u] = ok ? tri_off(i) + c : -1;
#pragma unroll
      for (int z = 0; z < GR_CH; ++z)
        g[u][z] = ok ? Gp[(size_t)z * L * L + i * L + c] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      // (hi + lo rounded to fp32 at once and by way of float64 is the same: near
      // a midpoint of two fp32 values the float64 sum is exact)
      const DF t = gram_sum(g[u]);
      if (at[u] >= 0) Ls[at[u]] = __fadd_rn(t.hi, t.lo);
    }
  }
  if (warp == 0) {  // the largest diagonal entry
    double md = 0.0;
    for (int i = lane; i < L; i += 32) {
      float2 g[GR_CH];
#pragma unroll
      for (int z = 0; z < GR_CH; ++z) g[z] = Gp[(size_t)z * L * L + (size_t)i * L + i];
      const DF t = gram_sum(g);
      md = fmax(md, (double)t.hi + (double)t.lo);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
    if (lane == 0) s_md = md;
  }
  __syncthreads();
  const double md = s_md;
  if (!(md > 0.0)) {
    for (int e = tid; e < L * L; e += CH_THREADS) Lout[e] = 0.f;
    for (int e = tid; e < nb * CH_B * CH_B; e += CH_THREADS) Dinv[e] = 0.f;
    for (int e = tid; T && e < L * L; e += CH_THREADS) T[e] = 0.f;
    return;
  }
  const float shift = (float)(shift_rel * md);
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
      const float d = sqrtf(fmaxf(__shfl_sync(0xffffffffu, a[j], j), 1e-30f)), rd = 1.f / d;
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
    if (T && lane < L)
#pragma unroll
      for (int i = 0; i < CH_B; ++i)
        if (i < L) T[lane * L + i] = lane <= i ? x[i] : 0.f;
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

// T = L^-T (T[k][n] = X[n][k], X = L^-1) from the factor and its inverted
// diagonal blocks.  CTA kb forms the 16 columns of X from 16 kb on, block row by
// block row: S = sum of L_{ib,m} X_m over the earlier rows (ascending), X_ib =
// -Dinv_ib S; a thread holds one of the 16 x 16 sums.  The block columns do not
// depend on one another, so the inverse takes nb CTAs instead of more of the
// Cholesky's one (where it took 80 us at L = 136); the chain of nb block rows of
// the first bounds it: 10.9 us.  The next block row of L is on its way meanwhile.
constexpr int TI_THREADS = CH_B * CH_B;
__host__ __device__ inline int ti_ld(int nb) { return nb * CH_B + 4; }

__global__ void __launch_bounds__(TI_THREADS)
k_tri_inverse(const float* __restrict__ Lf, const float* __restrict__ Dinv, int L, float* __restrict__ T) {
  extern __shared__ __align__(16) float ti[];
  const int nb = (L + CH_B - 1) / CH_B, ld = ti_ld(nb);
  float* X = ti;                        // [rows from j0 on][CH_B]
  float* Lr = X + nb * CH_B * CH_B;     // [2][CH_B][ld]: block rows of L, columns from j0 on
  float* Dr = Lr + 2 * CH_B * ld;       // [2][CH_B][CH_B + 4]: their inverted diagonal blocks
  float* S = Dr + 2 * CH_B * (CH_B + 4);  // [CH_B][CH_B]
  const int tid = threadIdx.x, rr = tid / CH_B, cc = tid % CH_B;
  const int kb = blockIdx.x, j0 = kb * CH_B;
  auto fetch = [&](int ib) {
    if (ib < nb) {
      const int i0 = ib * CH_B, w = i0 - j0;
      float* dst = Lr + (ib & 1) * CH_B * ld;
      if (L % 4 == 0) {
        for (int q = tid; q < CH_B * w / 4; q += TI_THREADS) {
          const int r = q / (w / 4), c = 4 * (q - r * (w / 4));
          if (i0 + r < L)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(os_smem(dst + r * ld + c)),
                         "l"(Lf + (size_t)(i0 + r) * L + j0 + c)
                         : "memory");
        }
      } else {
        for (int q = tid; q < CH_B * w; q += TI_THREADS) {
          const int r = q / w, c = q - r * w;
          if (i0 + r < L)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(os_smem(dst + r * ld + c)),
                         "l"(Lf + (size_t)(i0 + r) * L + j0 + c)
                         : "memory");
        }
      }
      if (tid < CH_B * CH_B / 4) {
        const int r = tid / (CH_B / 4), c = 4 * (tid % (CH_B / 4));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         os_smem(Dr + (ib & 1) * CH_B * (CH_B + 4) + r * (CH_B + 4) + c)),
                     "l"(Dinv + (i0 + r) * CH_B + c)
                     : "memory");
      }
    }
  };
  fetch(kb + 1);
  X[rr * CH_B + cc] = Dinv[(j0 + rr) * CH_B + cc];
  for (int ib = kb + 1; ib < nb; ++ib) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // block row ib has landed; the last one's buffers are free
    fetch(ib + 1);
    const int i0 = ib * CH_B;
    const float* l = Lr + (ib & 1) * CH_B * ld + rr * ld;
    float acc = 0.f;
    if (i0 + rr < L) {
#pragma unroll 4
      for (int q = 0; q < i0 - j0; q += 4) {
        const float4 a = *reinterpret_cast<const float4*>(l + q);
        const float* x = X + q * CH_B + cc;
        acc = fmaf(a.x, x[0], acc);
        acc = fmaf(a.y, x[CH_B], acc);
        acc = fmaf(a.z, x[2 * CH_B], acc);
        acc = fmaf(a.w, x[3 * CH_B], acc);
      }
    }
    S[rr * CH_B + cc] = acc;
    __syncthreads();
    const float* d = Dr + (ib & 1) * CH_B * (CH_B + 4) + rr * (CH_B + 4);
    acc = 0.f;
#pragma unroll
    for (int p = 0; p < CH_B; p += 4) {
      const float4 a = *reinterpret_cast<const float4*>(d + p);
      acc = fmaf(a.x, S[p * CH_B + cc], acc);
      acc = fmaf(a.y, S[(p + 1) * CH_B + cc], acc);
      acc = fmaf(a.z, S[(p + 2) * CH_B + cc], acc);
      acc = fmaf(a.w, S[(p + 3) * CH_B + cc], acc);
    }
    X[(i0 - j0 + rr) * CH_B + cc] = -acc;
  }
  __syncthreads();
  for (int k = tid >> 5; k < CH_B && j0 + k < L; k += TI_THREADS / 32)
    for (int n = tid & 31; n < L; n += 32)
      T[(size_t)(j0 + k) * L + n] = n >= j0 + k ? X[(n - j0) * CH_B + k] : 0.f;
}

// Mt (column-major, Mt[j][i] = M[i][j]) of M = L1 L2 for lower-triangular
// L1, L2 [L][L] (fp32, float64 sums).  CTA i, thread j.  The float64 pipe bounds
// it (a multiply-add and a widening, 16 cycles a warp each: row i of L1 is widened
// once).  Thirty-two loads are in flight, and a warp's lanes walk the same k from
// its first column on, so that a load reads one row piece: 29 us at
// L = 136 (8 with compensated fp32 pairs, which hold 48 bits of the sum).
__global__ void __launch_bounds__(256)
k_trmm(const float* __restrict__ L1, const float* __restrict__ L2, int L, float* __restrict__ Mt) {
  __shared__ double a[256];
  const int i = blockIdx.x, j = threadIdx.x;
  if (j <= i) a[j] = (double)L1[(size_t)i * L + j];
  __syncthreads();
  if (j >= L) return;
  double acc = 0.0;
  for (int k = j & ~31; k <= i; k += 32) {
    float b[32];
#pragma unroll
    for (int u = 0; u < 32; ++u) b[u] = k + u >= j && k + u <= i ? L2[(size_t)(k + u) * L + j] : 0.f;
#pragma unroll
    for (int u = 0; u < 32; ++u)
      if (k + u >= j && k + u <= i) acc = fma(a[k + u], (double)b[u], acc);
  }
  Mt[(size_t)j * L + i] = (float)acc;
}

// One-sided Jacobi SVD of M (Hestenes): the columns of M are orthogonalised by
// plane rotations applied from the right, M W = U S, W orthogonal.  Lp = L
// rounded up to even (a zero padding column never rotates); a round pairs the
// columns by the circle method: pair g of round r is (r + g, r - g) mod Lp - 1,
// pair 0 (r, Lp - 1).  For a pair: alpha = |m_p|^2, beta = |m_q|^2, gamma =
// m_p . m_q (fp32, eight lanes with a share each, then a butterfly that leaves
// every lane the same sums), and unless |gamma| <= 1e-6 sqrt(alpha beta) (a little
// above the rounding of an fp32 dot product, so that sweeps terminate) columns
// p, q of M and of W are rotated by the angle that makes them orthogonal (zeta =
// (beta - alpha) / (2 gamma), t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)), c =
// 1 / sqrt(1 + t^2), s = c t; correctly rounded roots and divisions).  Sweeps end
// when one makes no rotation, or after OS_MAX_SWEEPS.
//
// On one SM a round moves all of M and W through shared memory: 1.44 us at
// L = 136, 1.76 ms in all.  In the circle method pair g hands its first column
// to pair g - 1 and its second to pair g + 1 (pair 0 its first to pair 1, the last
// pair its second to itself), so the pairs are cut into OS_P = 8 runs, one a CTA
// of a thread-block cluster, and only the columns at the ends of a run leave the
// SM: sixteen lanes have a pair (eight its columns of M, eight those of W), read
// the columns from one buffer and store them, rotated, where the next round
// reads them, in the other buffer of this CTA or, with st.async and the bytes
// counted by that CTA's mbarrier, of the neighbour.  A neighbour can be one round
// ahead at most, because it needs this CTA's column of every round, and it
// overwrites a slot only after the pair that read it has sent that column.  The
// order of the rotations and of every sum is that of one SM taking the rounds in
// turn, so the bits are the same.  A round's latency bounds it (a column's loads,
// the reduction, the angle, the hop to the neighbour): 0.79 us a round at L = 136,
// 970 us in all.
//
// Every wait is bounded.  A thread whose wait gave up waits no more and its CTA
// goes on with what the buffers hold, so that the neighbours get their bytes and
// every CTA reaches the end of the sweep; the CTAs then read one another's flags and
// all leave there, with LX_ERR_TIMEOUT in the call's error word.
//
// Which entries of a column a lane sums: up to 144 columns, entries 16 v + 2 u,
// + 1 (lane u, v = 0, 1, ...); above, u, u + 8, u + 16, ...; both ascending.
// Output: Wt [L][L], Wt[j][k] = W[k][j].
constexpr int OS_MAX_SWEEPS = 30;
constexpr int OS_P = 8;        // CTAs of the cluster
constexpr int OS_LANES = 16;   // of a pair: eight for M, eight for W
constexpr int OS_MAX_PAIRS = 16;  // a CTA's at L = 256
constexpr unsigned OS_ROTATED = 1, OS_GAVE_UP = 2;  // flags of a CTA's sweep
constexpr long long OS_LAND_CYCLES = 1 << 20;  // half a millisecond, for bytes in flight to land
// floats of a column's part (M or W, NV pairs of entries a lane): the parts of a
// column 16 mod 32 words apart, so that a pair's 16 lanes touch distinct banks
__host__ __device__ constexpr int os_part(int nv) { return 16 * nv + (nv % 2 == 0 ? 16 : 0); }

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
__device__ __forceinline__ void os_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// bounded wait for a phase of this CTA's mbarrier (its bytes were sent by
// CTAs that are resident beside it, so it ends)
__device__ __forceinline__ bool os_wait(uint32_t bar, uint32_t parity, unsigned long long limit) {
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
    if (clock64() - t0 > limit) return false;
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

// Rotates the columns x and y of this pair (lanes 0 .. 7 of its sixteen: M, the
// others: W); true if it did.
template <int NV>
__device__ __forceinline__ bool os_rotate(float2 (&x)[NV], float2 (&y)[NV], bool on) {
  float a = 0.f, b = 0.f, g = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    a = fmaf(x[v].x, x[v].x, a);
    a = fmaf(x[v].y, x[v].y, a);
    b = fmaf(y[v].x, y[v].x, b);
    b = fmaf(y[v].y, y[v].y, b);
    g = fmaf(x[v].x, y[v].x, g);
    g = fmaf(x[v].y, y[v].y, g);
  }
#pragma unroll
  for (int o = 4; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    g += __shfl_xor_sync(0xffffffffu, g, o);
  }
  const int from = threadIdx.x & 23;  // the M lanes' sums for the W lanes
  a = __shfl_sync(0xffffffffu, a, from);
  b = __shfl_sync(0xffffffffu, b, from);
  g = __shfl_sync(0xffffffffu, g, from);
  if (!(on && g != 0.f && fabsf(g) > 1e-6f * sqrtf(a * b))) return false;  // pair-uniform
  // (an overflowing zeta gives t = 0: no rotation, never a NaN)
  const float z = (b - a) / (2.f * g);
  const float t = (z >= 0.f ? 1.f : -1.f) / (fabsf(z) + sqrtf(fmaf(z, z, 1.f)));
  const float c = 1.f / sqrtf(fmaf(t, t, 1.f)), sn = t * c;
  const float2 c2{c, c}, s2{sn, sn}, ns2{-sn, -sn};
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const float2 p = x[v], q = y[v];
    x[v] = os_fma2(c2, p, os_mul2(ns2, q));
    y[v] = os_fma2(s2, p, os_mul2(c2, q));
  }
  return true;
}

template <int NV>
__global__ void __launch_bounds__(OS_LANES * OS_MAX_PAIRS)
k_jacobi_cluster(const float* __restrict__ Mt, int L, float* __restrict__ Wt, const CallWaits waits) {
  constexpr int PART = os_part(NV), COL = 2 * PART;  // floats of a column's part and of a column
  extern __shared__ __align__(128) float osm[];  // [2 buffers][first, second columns][nmax][COL]
  __shared__ __align__(8) uint64_t s_full[2];    // by buffer: the neighbours' columns have landed
  __shared__ unsigned s_rot[2];                  // by sweep parity: this CTA's flags
  __shared__ unsigned s_go;
  const int tid = threadIdx.x, lane16 = tid & (OS_LANES - 1), u = lane16 & 7, i = tid / OS_LANES;
  uint32_t rank_u;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
  const int rank = (int)rank_u;
  const int Lp = L + (L & 1), half = Lp / 2;
  // pairs g0 .. g0 + n - 1 of a round; a cluster has no more busy CTAs than pairs
  const int busy = min(OS_P, half), each = half / busy, more = half % busy;
  const int nmax = each + (more ? 1 : 0);
  const int n = rank < busy ? each + (rank < more ? 1 : 0) : 0;
  const int g = rank * each + min(rank, more) + i;
  const bool on = i < n;
  const uint32_t base = os_smem(osm), full0 = os_smem(s_full);
  const uint32_t buf_bytes = (uint32_t)(2 * nmax * COL) * 4u, line_bytes = (uint32_t)(nmax * COL) * 4u;
  // this lane's piece of slot `at` of line h (0: first columns) in buffer 0
  const uint32_t mine = (uint32_t)((lane16 >> 3) * PART + 2 * u) * 4u;
  auto slot = [&](int h, int at) { return (uint32_t)h * line_bytes + (uint32_t)(at * COL) * 4u + mine; };
  // where the pair's columns go for the next round: an offset, and the CTA (-1: this one)
  uint32_t xto = slot(0, 0), yto = slot(1, 0);
  int xcta = -1, ycta = -1;
  if (on && half > 1) {
    if (g == 0) {
      xto = slot(1, n > 1 ? 1 : 0);
      if (n == 1) xcta = 1;
    } else {
      if (i > 0) xto = slot(0, i - 1);
      else {
        xcta = rank - 1;
        xto = slot(0, each + (rank - 1 < more ? 1 : 0) - 1);
      }
      if (g == half - 1) yto = slot(0, n - 1);
      else if (i < n - 1) yto = slot(1, i + 1);
      else ycta = rank + 1;  // (to its slot (1, 0))
    }
  }
  // the bytes of the neighbours' columns that arrive for each round
  uint32_t incoming = (uint32_t)(n == 0 ? 0 : (rank > 0) + (rank < busy - 1)) * (uint32_t)(OS_LANES * NV * 8);
  const bool listens = on && incoming && (i == 0 || i == n - 1);
  // (test hook: the first CTA waits for bytes that nobody sends)
  if (waits.unmet == LX_WAIT_CALL_JACOBI && rank == 0 && incoming) incoming += 16;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_rot[0] = s_rot[1] = 0;
  }
  // the columns of pair g in round 0
  const int cx = g, cy = g == 0 ? Lp - 1 : Lp - 1 - g;
  const bool strided = Lp > 144;
  auto entry = [&](int v, int e) { return strided ? 16 * v + 8 * e + u : 16 * v + 2 * u + e; };
  if (on) {
    auto first = [&](int col, int k) {
      if (lane16 >= 8) return k == col ? 1.f : 0.f;
      return col < L && k < L ? Mt[(size_t)col * L + k] : 0.f;
    };
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      *reinterpret_cast<float2*>(reinterpret_cast<char*>(osm) + slot(0, i) + 64 * v) =
          make_float2(first(cx, entry(v, 0)), first(cx, entry(v, 1)));
      *reinterpret_cast<float2*>(reinterpret_cast<char*>(osm) + slot(1, i) + 64 * v) =
          make_float2(first(cy, entry(v, 0)), first(cy, entry(v, 1)));
    }
  }
  __syncthreads();
  os_cluster_sync();  // every CTA's mbarriers are initialised
  uint32_t k = 0;     // rounds done
  bool alive = true;
  for (int sweep = 0;; ++sweep) {
    bool rotated = false;
    for (int rd = 0; rd < Lp - 1; ++rd, ++k) {
      if (n == 0) continue;
      const uint32_t cur = k & 1, nxt = cur ^ 1;
      if (tid == 0 && incoming && alive)  // (thread 0 listens: the phase before is over)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full0 + 8 * nxt),
                     "r"(incoming)
                     : "memory");
      if (listens && k > 0 && alive) alive = os_wait(full0 + 8 * cur, ((k - 1) >> 1) & 1, waits.cycles);
      __syncwarp();
      float2 x[NV], y[NV];
      const char* B = reinterpret_cast<const char*>(osm) + cur * buf_bytes;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        x[v] = on ? *reinterpret_cast<const float2*>(B + slot(0, i) + 64 * v) : make_float2(0.f, 0.f);
        y[v] = on ? *reinterpret_cast<const float2*>(B + slot(1, i) + 64 * v) : make_float2(0.f, 0.f);
      }
      rotated |= os_rotate<NV>(x, y, on);
      auto put = [&](const float2 (&c)[NV], uint32_t to, int cta) {
        if (cta < 0) {
          char* D = reinterpret_cast<char*>(osm) + nxt * buf_bytes + to;
#pragma unroll
          for (int v = 0; v < NV; ++v) *reinterpret_cast<float2*>(D + 64 * v) = c[v];
        } else {
          const uint32_t dst = os_map(base + nxt * buf_bytes + to, (uint32_t)cta);
          const uint32_t bar = os_map(full0 + 8 * nxt, (uint32_t)cta);
#pragma unroll
          for (int v = 0; v < NV; ++v)
            asm volatile(
                "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                    dst + 64 * v),
                "f"(c[v].x), "f"(c[v].y), "r"(bar)
                : "memory");
        }
      };
      if (on) {
        put(x, xto, xcta);
        put(y, yto, ycta);
      }
      __syncthreads();
    }
    if (rotated || !alive) atomicOr(&s_rot[sweep & 1], (rotated ? OS_ROTATED : 0u) | (alive ? 0u : OS_GAVE_UP));
    // every CTA reads the same flags, so all leave after the same sweep
    __syncthreads();
    os_cluster_sync();
    if (tid == 0) {
      unsigned go = 0;
      for (int c = 0; c < OS_P; ++c) go |= os_ld_remote(os_map(os_smem(&s_rot[sweep & 1]), (uint32_t)c));
      s_go = go;
      s_rot[(sweep + 1) & 1] = 0;  // last read a sweep ago
    }
    __syncthreads();
    if (s_go & OS_GAVE_UP) alive = false;  // the same in every CTA
    if (s_go != OS_ROTATED || sweep + 1 == OS_MAX_SWEEPS) break;
  }
  // a sweep's rounds bring every column back to where it began
  if (listens && alive) alive = os_wait(full0 + 8 * (k & 1), ((k - 1) >> 1) & 1, waits.cycles);
  if (!alive) {
    atomicExch(waits.err, LX_ERR_TIMEOUT);
    const long long t0 = clock64();
    while (clock64() - t0 < OS_LAND_CYCLES) {
    }
  }
  if (on && lane16 >= 8) {
    const char* B = reinterpret_cast<const char*>(osm) + (k & 1) * buf_bytes;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const float2 p = *reinterpret_cast<const float2*>(B + slot(0, i) + 64 * v);
      const float2 q = *reinterpret_cast<const float2*>(B + slot(1, i) + 64 * v);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int r = entry(v, e);
        if (r >= L) continue;
        if (cx < L) Wt[(size_t)cx * L + r] = e ? p.y : p.x;
        if (cy < L) Wt[(size_t)cy * L + r] = e ? q.y : q.x;
      }
    }
  }
  __syncwarp();
  os_cluster_sync();  // no CTA leaves while its flags are read or bytes for it are in flight
}

// CTA j: v = M w_j in float64, sigma_j = |v| / |w_j| (the Rayleigh quotient of
// the converged rotation, second-order accurate in the rotation's error);
// MWn[j] = v / |w_j|, Wn[j] = w_j / |w_j| (fp32, column j stored contiguously).
__global__ void __launch_bounds__(256)
k_ritz(const float* __restrict__ Mt, const float* __restrict__ Wt, int L, float* __restrict__ MWn,
       float* __restrict__ Wn, double* __restrict__ sig64) {
  __shared__ double w[256];
  __shared__ double red[2][8];
  __shared__ double s_norm;
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < L) w[tid] = (double)Wt[(size_t)j * L + tid];
  __syncthreads();
  double v = 0.0, ww = 0.0;
  if (tid < L) {
    for (int k = 0; k < L; k += 32) {  // thirty-two loads in flight
      float m[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) m[u] = k + u < L ? Mt[(size_t)(k + u) * L + tid] : 0.f;
#pragma unroll
      for (int u = 0; u < 32; ++u)
        if (k + u < L) v = fma((double)m[u], w[k + u], v);
    }
    ww = w[tid] * w[tid];
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
  if (tid == 0) {  // the float64 roots once: they run at a fraction of the fp32 rate
    double tv = 0.0, tw = 0.0;
    for (int q = 0; q < 8; ++q) {
      tv += red[0][q];
      tw += red[1][q];
    }
    const double nw_ = sqrt(tw);
    s_norm = nw_;
    sig64[j] = nw_ > 0.0 ? sqrt(tv) / nw_ : 0.0;
  }
  __syncthreads();
  if (tid < L) {
    const double nw_ = s_norm;
    MWn[(size_t)j * L + tid] = nw_ > 0.0 ? (float)(v / nw_) : 0.f;
    Wn[(size_t)j * L + tid] = nw_ > 0.0 ? (float)(w[tid] / nw_) : 0.f;
  }
}

// CTA k (of L): the r largest sigma (ties: lower index first) and row k of the
// fp32 matrices Wu [L][r] = MWn[i_c] / sqrt(sigma_c), Wv [L][r] = Wn[i_c]
// sqrt(sigma_c) (zero for sigma_c <= 1e-6 sigma_0), so that Q Wu = U_r S_r^(1/2)
// and Z2 Wv = V_r S_r^(1/2) (Eq. factors); CTA 0 writes sig [r] fp32.  Every CTA
// ranks the sigma for itself (non-negative float64 values compare as their
// bits do), so that no single CTA takes the L r square roots and divisions:
// 87 us with one CTA, 6.7 us now at L = 136, r = 128.  All NaN if a wait of the
// call gave up (err), so that the caller sees it in every factor.
__global__ void __launch_bounds__(256)
k_finish(const double* __restrict__ sig64, const float* __restrict__ MWn,
         const float* __restrict__ Wn, int L, int r, const int* __restrict__ err,
         float* __restrict__ Wu, float* __restrict__ Wv, float* __restrict__ sig) {
  __shared__ double sv[256];
  __shared__ int order[256];
  const int tid = threadIdx.x, k = blockIdx.x;
  if (*err) {
    if (tid < r) {
      Wu[(size_t)k * r + tid] = Wv[(size_t)k * r + tid] = NAN;
      if (k == 0) sig[tid] = NAN;
    }
    return;
  }
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
bool g_ti_cap[64] = {};
bool g_jac_cap[6][64] = {};

}  // namespace
}  // namespace lx

namespace lx {
namespace {
constexpr int CP_MAX_L = 256;
constexpr size_t CP_SMEM_CAP = 200 * 1024;

size_t al256(size_t v) { return (v + 255) / 256 * 256; }

struct CompressWs {
  float *y0, *y1, *z0, *z1, *Dinv, *T, *Wu, *Wv, *L1, *L2, *Mt, *Wt, *MWn, *Wn;
  double* sig64;
  int* err;  // LX_ERR_TIMEOUT if a wait of the call gave up
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
  w.T = (float*)take(4 * l * l);
  w.Wu = (float*)take(4 * l * r);
  w.Wv = (float*)take(4 * l * r);
  w.L1 = (float*)take(4 * l * l);
  w.L2 = (float*)take(4 * l * l);
  w.Mt = (float*)take(4 * l * l);
  w.Wt = (float*)take(4 * l * l);
  w.MWn = (float*)take(4 * l * l);
  w.Wn = (float*)take(4 * l * l);
  w.sig64 = (double*)take(8 * l);
  w.err = (int*)take(4);
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
                       CallWaits waits, int dev, cudaStream_t s) {
  int num_sms = 0;
  LX_CUDA(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
  // bf16 weights: the residual products R X and R^T X on the tensor cores
  constexpr bool bf16_w = std::is_same<TW, __nv_bfloat16>::value;
  const bool res_tc = bf16_w && res_tc_fits(rows, cols, l);
  lx_status tc_status = LX_OK;
  waits.err = w.err;
  LX_CUDA(cudaMemsetAsync(w.err, 0, sizeof(int), s));
  bool have_wt = false;  // W^T of this call's weights lies in w.tc
  auto gemm = [&](int mode, const float* X, const float* B, float* C, int M, int N, int K) {
    const dim3 grid((N + CG_TILE - 1) / CG_TILE, (M + CG_TILE - 1) / CG_TILE);
    if constexpr (bf16_w) {
      if (res_tc && (mode == A_RES || mode == A_RES_T)) {
        const lx_status st = res_gemm_tc(mode == A_RES_T, reinterpret_cast<const __nv_bfloat16*>(Wm),
                                         reinterpret_cast<const __nv_bfloat16*>(Wd), rows, cols, B, N,
                                         C, w.tc, &have_wt, waits, num_sms, dev, s);
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
  // is well conditioned).  The Gram's chains lie in the residual products'
  // partials, which are idle here.
  float2* const G = reinterpret_cast<float2*>(w.tc + res_tc_part_offset(rows, cols, l));
  const int ldp = ch_ldp(l), nb = (l + CH_B - 1) / CH_B;
  const size_t ch_smem = sizeof(float) * ((((size_t)l * (l + 1) / 2 + 3) & ~(size_t)3) + (size_t)CH_B * ldp);
  const size_t ti_smem = sizeof(float) * ((size_t)nb * CH_B * CH_B + 2 * CH_B * ti_ld(nb) +
                                          2 * CH_B * (CH_B + 4) + CH_B * CH_B);
  LX_CUDA(smem_cap_once((const void*)k_chol32, (int)CP_SMEM_CAP, dev, g_ch_cap));
  LX_CUDA(smem_cap_once((const void*)k_tri_inverse, (int)CP_SMEM_CAP, dev, g_ti_cap));
  auto cholqr = [&](const float* X, float* out, int n, float shift, float* Lf) {
    const dim3 grid((l + GR_T - 1) / GR_T, (l + GR_T - 1) / GR_T, GR_CH);
    k_gram<<<grid, GR_T * GR_T, 0, s>>>(X, n, l, G);
    k_chol32<<<1, CH_THREADS, ch_smem, s>>>(G, l, ldp, shift, Lf, w.Dinv, nb == 1 ? w.T : nullptr);
    if (nb > 1) k_tri_inverse<<<nb, TI_THREADS, ti_smem, s>>>(Lf, w.Dinv, l, w.T);
    gemm(A_F32, X, w.T, out, n, l, l);
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
    const int Lp = l + (l & 1), half = Lp / 2, nmax = (half + OS_P - 1) / OS_P;
    auto launch = [&](auto kern, int slot, int col_floats) -> lx_status {
      LX_CUDA(smem_cap_once((const void*)kern, (int)CP_SMEM_CAP, dev, g_jac_cap[slot]));
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(OS_P);
      cfg.blockDim = dim3(32 * ((nmax + 1) / 2));
      cfg.dynamicSmemBytes = sizeof(float) * 2 * 2 * nmax * (size_t)col_floats;
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = OS_P;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      LX_CUDA(cudaLaunchKernelEx(&cfg, kern, (const float*)w.Mt, l, w.Wt, (const CallWaits)waits));
      return LX_OK;
    };
    if (Lp <= 32) LX_TRY(launch(k_jacobi_cluster<2>, 0, 2 * os_part(2)));
    else if (Lp <= 48) LX_TRY(launch(k_jacobi_cluster<3>, 1, 2 * os_part(3)));
    else if (Lp <= 80) LX_TRY(launch(k_jacobi_cluster<5>, 2, 2 * os_part(5)));
    else if (Lp <= 144) LX_TRY(launch(k_jacobi_cluster<9>, 3, 2 * os_part(9)));
    else if (Lp <= 192) LX_TRY(launch(k_jacobi_cluster<12>, 4, 2 * os_part(12)));
    else LX_TRY(launch(k_jacobi_cluster<16>, 5, 2 * os_part(16)));
  }
  k_ritz<<<l, 256, 0, s>>>(w.Mt, w.Wt, l, w.MWn, w.Wn, w.sig64);
  k_finish<<<l, 256, 0, s>>>(w.sig64, w.MWn, w.Wn, l, r, w.err, w.Wu, w.Wv, sigma);
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
  const CallWaits waits = take_call_waits();
  int dev = 0;
  LX_CUDA(cudaGetDevice(&dev));
  cudaStream_t s = (cudaStream_t)stream;
  if (dtype == LX_BF16)
    return run_compress(rows, cols, (const __nv_bfloat16*)w_dom, (const __nv_bfloat16*)w_mem,
                        omega, l, r, power_iters, U, V, sigma, w, waits, dev, s);
  return run_compress(rows, cols, (const float*)w_dom, (const float*)w_mem, omega, l, r,
                      power_iters, U, V, sigma, w, waits, dev, s);
}
