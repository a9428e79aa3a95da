// Router profiling statistics (Sec. 3.2 Stage 1: per-layer firing counts N_e
// read from the router; Sec. 2.2: the expert co-activation graph weighted by
// normalised pointwise mutual information, whose 1 - NPMI is Stage 2's
// Coact-NPMI clustering distance).
//
// Co-activation counts are popcounts (k_coact_bits): a CTA takes a chunk of tokens,
// records in shared memory one bit per (expert, token) of the tokens' selected
// sets, and counts for its slice of the expert pairs the tokens that have both
// (popc(bits_i & bits_j) over the chunk's words), one 64-bit atomic addition per
// non-zero pair and chunk.  Its work grows with the square of E; with many experts
// and few ids a token, a 64-bit atomic addition per pair of the token
// (k_coact_global) is less (coact_by_bits).  Integer addition is associative, so
// the counts do not depend on the form or the order.
#include <algorithm>

#include "lx_internal.cuh"

namespace lx {
namespace {

constexpr int CO_THREADS = 512;
constexpr int CO_WARPS = CO_THREADS / 32;
constexpr int CO_BIT_BYTES = 128 * 1024;  // bitmaps of a chunk
constexpr int CO_MAX_WORDS = 64;

// Words (of 32 tokens) of a chunk: 2048 tokens, fewer where E rows of bits would
// not fit, and no more than the batch has
__host__ __device__ inline int co_words(int E, int T) {
  int w = CO_MAX_WORDS;
  while (w > 1 && (size_t)w * E * 4 > CO_BIT_BYTES) w /= 2;
  const int need = T / 32 + (T % 32 != 0);
  return w < need ? w : need;
}

// CTA (c, s): tokens of chunk c, rows i = s, s + gridDim.y, ... of the pairs
// (i, j >= i).  Bits are kept [word][expert], so that the lanes of a warp
// (consecutive j) read consecutive banks.  The set of a token ignores invalid
// ids and repeats by itself.  Atomic additions bound a histogram of pairs kept in
// each CTA (every CTA flushes all its non-zero pairs): 35 us per 8192-token batch
// at E = 128, 13.5 us for this form, where a pair is added once per 2048 tokens.
__global__ void __launch_bounds__(CO_THREADS)
k_coact_bits(const int* __restrict__ ids, int T, int k, int E, int words,
             unsigned long long* __restrict__ fire, unsigned long long* __restrict__ coact) {
  extern __shared__ unsigned int cb[];  // [words][E]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int q = tid; q < words * E; q += CO_THREADS) cb[q] = 0u;
  __syncthreads();
  const int t0 = blockIdx.x * words * 32, nt = min(words * 32, T - t0);
  const int* my = ids + (size_t)t0 * k;
  constexpr int U = 8;  // ids in flight a thread
  for (int q0 = tid; q0 < nt * k; q0 += U * CO_THREADS) {  // assignment q: token q / k of the chunk
    int e[U];
#pragma unroll
    for (int u = 0; u < U; ++u) e[u] = q0 + u * CO_THREADS < nt * k ? my[q0 + u * CO_THREADS] : -1;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (e[u] >= 0 && e[u] < E) {
        const int t = (q0 + u * CO_THREADS) / k;
        atomicOr(&cb[(t >> 5) * E + e[u]], 1u << (t & 31));
      }
  }
  __syncthreads();
  // a warp per row i (dealt to the CTAs of this chunk, then to their warps)
  for (int i = blockIdx.y + gridDim.y * warp; i < E; i += gridDim.y * (CO_THREADS / 32)) {
    for (int j0 = i; j0 < E; j0 += 32) {
      const int j = j0 + lane;
      unsigned n = 0;
      if (j < E)
#pragma unroll 8
        for (int w = 0; w < words; ++w) n += __popc(cb[w * E + i] & cb[w * E + j]);
      if (!n) continue;
      if (coact) {
        atomicAdd(&coact[(size_t)i * E + j], (unsigned long long)n);
        if (i != j) atomicAdd(&coact[(size_t)j * E + i], (unsigned long long)n);
      }
      if (i == j && fire) atomicAdd(&fire[i], (unsigned long long)n);
    }
  }
}

// One warp per token: lane s holds slot s's id, selected when it is in [0, E) and
// no lower lane holds the same.
__global__ void __launch_bounds__(CO_THREADS)
k_coact_global(const int* __restrict__ ids, int T, int k, int E, unsigned long long* __restrict__ fire,
               unsigned long long* __restrict__ coact) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long t = (long)blockIdx.x * CO_WARPS + warp; t < T; t += (long)gridDim.x * CO_WARPS) {
    const int id = lane < k ? ids[(size_t)t * k + lane] : -1;
    const bool valid = id >= 0 && id < E;
    // (invalid lanes never match another lane)
    const unsigned same = __match_any_sync(0xffffffffu, valid ? id : -1 - lane);
    const bool mine = valid && lane == __ffs(same) - 1;
    const unsigned sel = __ballot_sync(0xffffffffu, mine);
    if (mine && fire) atomicAdd(&fire[id], 1ull);
    if (!coact) continue;
    for (unsigned b = sel; b; b &= b - 1) {  // warp-uniform loop over the selected lanes
      const int other = __shfl_sync(0xffffffffu, id, __ffs(b) - 1);
      if (mine) atomicAdd(&coact[(size_t)id * E + other], 1ull);
    }
  }
}

// Up to 256 experts the bits won at every size measured (the pairs kept as a
// histogram in shared memory before: 1.5 to 10 times slower).  Above, one addition a
// pair costs T k^2, the bits T E^2 / 64 and a flush of up to E^2 a chunk; measured,
// atomics against bits: E = 1024, k = 8: 2048 tokens 4.6 / 41 us, 65536 50 / 479;
// E = 512, k = 8: 65536 66 / 140, k = 32: 2048 20 / 36, 65536 466 / 188; E = 384, k =
// 8: 8192 14 / 25, 65536 88 / 78; E = 768, k = 32: 8192 64 / 48; E = 1024, k = 32:
// 65536 389 / 518.
bool coact_by_bits(int T, int k, int E) {
  return E <= 256 || (E <= 768 && E <= 48 * k && (double)T * k * k >= 4e6);
}

// p_i = C_ii / n, p_ij = C_ij / n; ln(p_ij / (p_i p_j)) / (-ln p_ij) for
// 0 < p_ij < 1, -1 for p_ij = 0, +1 for p_ij = 1 (float64).
__global__ void k_npmi(const unsigned long long* __restrict__ coact, int E,
                       unsigned long long n, double* __restrict__ npmi) {
  const long q = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (long)E * E) return;
  const int i = (int)(q / E), j = (int)(q - (long)i * E);
  const unsigned long long cij = coact[q];
  double v;
  if (cij == 0ull) {
    v = -1.0;
  } else if (cij >= n) {
    v = 1.0;
  } else {
    const double nn = (double)n;
    const double p_ij = (double)cij / nn;
    const double p_i = (double)coact[(size_t)i * E + i] / nn;
    const double p_j = (double)coact[(size_t)j * E + j] / nn;
    v = log(p_ij / (p_i * p_j)) / (-log(p_ij));
  }
  npmi[q] = v;
}

bool g_co_smem_cap[64] = {};

}  // namespace
}  // namespace lx

extern "C" lx_status lx_coact_accumulate(const int32_t* topk_id, int32_t T, int32_t k, int32_t E,
                                         uint64_t* fire, uint64_t* coact, void* stream) {
  using namespace lx;
  if (T < 0) return fail(LX_ERR_ARG, "T < 0");
  if (k < 1 || k > LX_MAX_K) return fail(LX_ERR_ARG, "k must be in 1..LX_MAX_K");
  if (E < 1 || E > LX_MAX_EXPERTS) return fail(LX_ERR_ARG, "E must be in 1..LX_MAX_EXPERTS");
  if (!fire && !coact) return fail(LX_ERR_ARG, "fire and coact are both NULL");
  if (T == 0) return LX_OK;
  if (!topk_id) return fail(LX_ERR_ARG, "topk_id is NULL");
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0, sms = 0;
  LX_CUDA(cudaGetDevice(&dev));
  LX_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  unsigned long long* f = reinterpret_cast<unsigned long long*>(fire);
  unsigned long long* c = reinterpret_cast<unsigned long long*>(coact);
  if (!coact_by_bits(T, k, E)) {
    const long grid = std::min(((long)T + CO_WARPS - 1) / CO_WARPS, 8L * sms);
    k_coact_global<<<(unsigned)grid, CO_THREADS, 0, s>>>(topk_id, T, k, E, f, c);
    LX_CUDA(cudaGetLastError());
    return LX_OK;
  }
  const int words = co_words(E, T), chunks = (int)(((long)T + 32 * words - 1) / (32 * words));
  // enough slices of the pairs for two CTAs an SM, at least a row for each
  const int slices = std::max(1, std::min(E, (2 * sms + chunks - 1) / chunks));
  LX_CUDA(smem_cap_once((const void*)k_coact_bits, CO_BIT_BYTES, dev, g_co_smem_cap));
  k_coact_bits<<<dim3(chunks, std::min(slices, 128)), CO_THREADS, sizeof(unsigned int) * (size_t)words * E, s>>>(
      topk_id, T, k, E, words, f, c);
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}

extern "C" lx_status lx_coact_npmi(const uint64_t* coact, int32_t E, int64_t n_tokens,
                                   double* npmi, void* stream) {
  using namespace lx;
  if (E < 1 || E > LX_MAX_EXPERTS) return fail(LX_ERR_ARG, "E must be in 1..LX_MAX_EXPERTS");
  if (n_tokens < 0) return fail(LX_ERR_ARG, "n_tokens < 0");
  if (!coact || !npmi) return fail(LX_ERR_ARG, "coact or npmi is NULL");
  const long n = (long)E * E;
  k_npmi<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      reinterpret_cast<const unsigned long long*>(coact), E, (unsigned long long)n_tokens, npmi);
  LX_CUDA(cudaGetLastError());
  return LX_OK;
}
