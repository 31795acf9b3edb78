// Offline planning on the GPU (Section IV, Alg. 1 grouping and placement):
//   ordermoe_similarity: H = W_r X_cal^T (Eq. 3, tcgen05 GEMM into scratch),
//     Sim = cosine of the rows of H (Eq. 4), activation counts n_j (Eq. 5);
//   ordermoe_expert_counts: the counts of Eq. 5 from given logits;
//   ordermoe_place: threshold (Eq. 6), greedy grouping (Eqs. 24-26),
//     importance (Eqs. 27-28) and mandatory placement (Eqs. 29-31);
//   ordermoe_replicate: redundant deployment (Eqs. 32-35);
//   ordermoe_coverage: local group coverage (Eq. 32).
#include <cstddef>

#include "common.cuh"

namespace om {

int logits_gemm_launch(const uint16_t* X, int N, const uint16_t* W, int C, int d, float* H,
                       cudaStream_t stream);

static __device__ unsigned long long g_err_sim = 0;

int read_clear_err_sim(unsigned long long* out) {
  unsigned long long zero = 0;
  OM_CUDA(cudaMemcpyFromSymbol(out, g_err_sim, sizeof(*out)));
  OM_CUDA(cudaMemcpyToSymbol(g_err_sim, &zero, sizeof(zero)));
  return ORDERMOE_OK;
}

constexpr int kSimChunk = 1024;  // calibration tokens per partial Gram
constexpr int kSub = 64;         // tokens staged in shared memory at a time

// grid (L, chunks), 256 threads. Partial Gram of layer l over one chunk of
// tokens in 8 x 4 blocks of experts G[8 ti .. 8 ti + 7][4 tj .. 4 tj + 3], one a
// thread in fp32 (each staged token costs three float4 shared loads per 32 FMAs:
// the loads bound it). The ceil(E / 8) ceil(E / 4) blocks leave threads over, so
// copies of them take every copies-th token (40 experts: 50 blocks, five
// copies), and the copies are added in order. 4 x 4 blocks without copies, 100
// of 256 threads at work, took 55.9 us for 32768 tokens, 8 layers of 40 experts,
// this 31.7.
__global__ void __launch_bounds__(256) gram_kernel(const float* __restrict__ H, int64_t N, int L,
                                                   int E, float* __restrict__ gpart) {
  __shared__ __align__(16) float sh[kSub][64];
  __shared__ float part[256 * 17];  // the copies' blocks (pitch 17: no bank conflicts)
  // the layers of one chunk are neighbouring blocks, so each token's record
  // of L * E logits is read from DRAM once and shared through L2
  const int l = blockIdx.x, chunk = blockIdx.y;
  const int nchunks = gridDim.y;
  const int tid = threadIdx.x;
  const int side = (E + 3) >> 2, nblk = ((E + 7) >> 3) * side;
  const int copies = 256 / nblk;  // >= 2: at most 8 x 16 blocks
  const int copy = tid / nblk, blk = tid - copy * nblk;
  const int ti = blk / side, tj = blk - ti * side;
  const bool active = copy < copies;
  const int LE = L * E;
  float acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
  const int64_t n_begin = (int64_t)chunk * kSimChunk;
  int64_t n_end = n_begin + kSimChunk;
  if (n_end > N) n_end = N;
  // the next kSub tokens are loaded into registers while these are multiplied
  const bool vec = (E & 3) == 0 && (LE & 3) == 0;
  float4 ahead[4];
  auto fetch = [&](int64_t n0) {  // 16 float4 per token row, 4 of the 1024 a thread
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int x = tid + 256 * u;
      const int c4 = (x & 15) * 4;
      const int64_t n = n0 + (x >> 4);
      ahead[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (n < n_end && c4 < E) ahead[u] = *reinterpret_cast<const float4*>(H + n * LE + (int64_t)l * E + c4);
    }
  };
  if (vec) fetch(n_begin);
  for (int64_t n0 = n_begin; n0 < n_end; n0 += kSub) {
    __syncthreads();
    if (vec) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int x = tid + 256 * u;
        *reinterpret_cast<float4*>(&sh[x >> 4][(x & 15) * 4]) = ahead[u];
      }
    } else {
      for (int x = tid; x < kSub * 64; x += 256) {
        const int r = x >> 6, c = x & 63;
        const int64_t n = n0 + r;
        sh[r][c] = (n < n_end && c < E) ? H[n * LE + (int64_t)l * E + c] : 0.0f;
      }
    }
    __syncthreads();
    if (vec && n0 + kSub < n_end) fetch(n0 + kSub);
    if (active) {
#pragma unroll 4
      for (int r = copy; r < kSub; r += copies) {
        const float4 a = *reinterpret_cast<const float4*>(&sh[r][8 * ti]);
        const float4 d = *reinterpret_cast<const float4*>(&sh[r][8 * ti + 4]);
        const float4 b = *reinterpret_cast<const float4*>(&sh[r][4 * tj]);
#define OM_GRAM_ROW(p, ap)                       \
  acc[p][0] = fmaf(ap, b.x, acc[p][0]);          \
  acc[p][1] = fmaf(ap, b.y, acc[p][1]);          \
  acc[p][2] = fmaf(ap, b.z, acc[p][2]);          \
  acc[p][3] = fmaf(ap, b.w, acc[p][3]);
        OM_GRAM_ROW(0, a.x) OM_GRAM_ROW(1, a.y) OM_GRAM_ROW(2, a.z) OM_GRAM_ROW(3, a.w)
        OM_GRAM_ROW(4, d.x) OM_GRAM_ROW(5, d.y) OM_GRAM_ROW(6, d.z) OM_GRAM_ROW(7, d.w)
#undef OM_GRAM_ROW
      }
    }
  }
  float* gp = gpart + ((size_t)l * nchunks + chunk) * 64 * 64;
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // the blocks' upper and lower four rows in turn
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 16; ++x) part[tid * 17 + x] = acc[4 * h + (x >> 2)][x & 3];
    __syncthreads();
    for (int x = tid; x < nblk * 16; x += 256) {
      const int k = x >> 4, e = x & 15;  // block and entry
      float s = part[k * 17 + e];
      for (int c = 1; c < copies; ++c) s += part[(c * nblk + k) * 17 + e];
      gp[(8 * (k / side) + 4 * h + (e >> 2)) * 64 + 4 * (k % side) + (e & 3)] = s;
    }
  }
}

// Top-kf experts of a token's E logits as a bit set (rank order: larger first,
// lower index on ties). KN > 0: a descending min/max network keeps the KN >= kf
// largest values with multiplicity, T is the kf-th of them, every logit >= T is
// taken, and where equal logits straddle the boundary the surplus equal to T
// goes back from the highest index down. KN = 0 (kf > 8), or a NaN among the
// logits: kf passes, each taking the first unused maximum (all E when kf = E: by
// the passes 1159 us of transitions for 100000 tokens, 2 layers of 64 experts).
template <int KN>
__device__ __forceinline__ unsigned long long topk_set(const float* row, int E, int kf) {
  if (kf == E) return ~0ull >> (64 - E);  // every pass takes one
  unsigned long long used = 0;
  if constexpr (KN > 0) {
    float v[KN];
#pragma unroll
    for (int p = 0; p < KN; ++p) v[p] = -INFINITY;
    bool nan = false;
#pragma unroll 8
    for (int e = 0; e < E; ++e) {
      const float c = row[e];
      nan |= c != c;
#pragma unroll
      for (int p = KN - 1; p >= 1; --p) v[p] = fminf(v[p - 1], fmaxf(v[p], c));
      v[0] = fmaxf(v[0], c);
    }
    if (!nan) {
      float T = v[0];
#pragma unroll
      for (int p = 1; p < KN; ++p) T = p < kf ? fminf(T, v[p]) : T;
      uint32_t m[2] = {0u, 0u};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int n = min(32, E - 32 * h);
#pragma unroll 8
        for (int e = 0; e < n; ++e) m[h] |= row[32 * h + e] >= T ? 1u << e : 0u;
      }
      used = (static_cast<unsigned long long>(m[1]) << 32) | m[0];
      int extra = __popcll(used) - kf;
      for (int e = E - 1; extra > 0; --e)
        if (((used >> e) & 1ull) && row[e] == T) {
          used &= ~(1ull << e);
          --extra;
        }
      return used;
    }
  }
  for (int j = 0; j < kf; ++j) {
    int best = -1;
    float bv = 0.0f;
    for (int e = 0; e < E; ++e) {
      if ((used >> e) & 1ull) continue;
      const float c = row[e];
      if (best < 0 || c > bv) {
        best = e;
        bv = c;
      }
    }
    used |= 1ull << best;
  }
  return used;
}

// The logits of a tile of kTopkTokens tokens at one layer, through shared memory
// (rows of E floats in global memory, read coalesced; an odd pitch, so that a
// thread a token reads its row without bank conflicts). Every thread of the
// block calls it; rows past n_end are left as they are.
constexpr int kTopkTokens = 256;
constexpr int kTransTiles = 8;  // tiles of a transitions block, at most
__host__ __device__ inline int topk_pitch(int E) { return E | 1; }
__device__ __forceinline__ void load_logit_tile(float* s, const float* __restrict__ logits, int64_t n0,
                                                int64_t n_end, int E, int64_t sn) {
  const int rows = static_cast<int>(n_end - n0 < kTopkTokens ? n_end - n0 : kTopkTokens);
  const int pitch = topk_pitch(E);
  const float* src = logits + n0 * sn;
  if (((E | sn) & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
    const int q = E >> 2;
#pragma unroll 4
    for (int i = threadIdx.x; i < rows * q; i += kTopkTokens) {
      const int r = i / q, c = (i - r * q) * 4;
      const float4 v = *reinterpret_cast<const float4*>(src + r * sn + c);
      float* d = s + r * pitch + c;
      d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    }
  } else {
    // Row and column are carried along: a division for each element took longer
    // than its load (counts of 20000 tokens: 31 experts 10.6 and 8.7 us, 49 12.4 and
    // 10.4, a thread reading its own row 8.6 and 12.8).
    const int step_r = kTopkTokens / E, step_c = kTopkTokens - step_r * E;
    int r = threadIdx.x / E, c = threadIdx.x - r * E;
#pragma unroll 4
    for (int i = threadIdx.x; i < rows * E; i += kTopkTokens) {
      s[r * pitch + c] = src[r * sn + c];
      r += step_r;
      c += step_c;
      if (c >= E) {
        c -= E;
        ++r;
      }
    }
  }
}

// Eq. 5 counts of layer l = blockIdx.x: logits of token n at layer l start at
// n * sn + l * sl (floats). Block totals are added with integer atomics, so the
// result does not depend on the order. Bound by the loads and the top-k's
// instructions; a thread reading its own row from global memory took 42 us for
// 32768 tokens, 8 layers of 40 experts (top-4), this 22.2.
template <int KN>
__global__ void __launch_bounds__(kTopkTokens) counts_kernel(const float* __restrict__ logits,
                                                             int64_t N, int E, int kf, int64_t sn,
                                                             int64_t sl, int32_t* __restrict__ counts) {
  extern __shared__ float s_tile[];
  __shared__ int cnt[64];
  const int l = blockIdx.x;  // layers of the same tokens run side by side (L2 reuse)
  if (threadIdx.x < 64) cnt[threadIdx.x] = 0;
  for (int64_t n0 = (int64_t)blockIdx.y * kTopkTokens; n0 < N; n0 += (int64_t)gridDim.y * kTopkTokens) {
    __syncthreads();
    load_logit_tile(s_tile, logits + l * sl, n0, N, E, sn);
    __syncthreads();
    if (n0 + threadIdx.x < N) {
      const float* row = s_tile + threadIdx.x * topk_pitch(E);
      for (unsigned long long b = topk_set<KN>(row, E, kf); b; b &= b - 1)
        atomicAdd(&cnt[__ffsll(static_cast<long long>(b)) - 1], 1);
    }
  }
  __syncthreads();
  if (threadIdx.x < E && cnt[threadIdx.x]) atomicAdd(&counts[(size_t)l * E + threadIdx.x], cnt[threadIdx.x]);
}

// Transition counts of Eq. 41 for the layer pairs (l, l + 1), l in [per *
// blockIdx.y, + per): each token adds one to n_l(k -> k') for every k in its
// top-kf at layer l and k' in its top-kf at layer l + 1 (integer atomics:
// order-independent). A block walks the layers of its tokens and keeps each
// layer's sets for the next, so that a row is read and ranked once (twice at a
// range's ends); logits of token n at layer l start at n * sn + l * sl. Ranked
// per pair, with a thread reading its own rows, it took 101 us for 32768 tokens,
// 8 layers of 40 experts (top-4), this 33.2.
template <int KN>
__global__ void __launch_bounds__(kTopkTokens) transitions_kernel(const float* __restrict__ logits,
                                                                  int64_t N, int L, int E, int kf,
                                                                  int64_t sn, int64_t sl, int per,
                                                                  int tiles,
                                                                  int32_t* __restrict__ counts) {
  extern __shared__ float s_tile[];  // the tile, then E * E counts
  __shared__ unsigned long long s_prev[kTransTiles][kTopkTokens];  // each thread's own
  int* h = reinterpret_cast<int*>(s_tile + kTopkTokens * topk_pitch(E));
  const int l0 = blockIdx.y * per, l1 = min(l0 + per, L - 1);  // pairs l0 .. l1 - 1
  const int64_t first = (int64_t)blockIdx.x * tiles * kTopkTokens;
  const float* row = s_tile + threadIdx.x * topk_pitch(E);
  for (int l = l0; l <= l1; ++l) {
    for (int i = threadIdx.x; i < E * E; i += kTopkTokens) h[i] = 0;
    for (int tl = 0; tl < tiles; ++tl) {
      const int64_t n0 = first + (int64_t)tl * kTopkTokens;
      if (n0 >= N) break;
      load_logit_tile(s_tile, logits + l * sl, n0, N, E, sn);
      __syncthreads();
      const unsigned long long set = n0 + threadIdx.x < N ? topk_set<KN>(row, E, kf) : 0ull;
      if (l > l0) {
        for (unsigned long long a = s_prev[tl][threadIdx.x]; a; a &= a - 1) {
          int* hr = h + (__ffsll(static_cast<long long>(a)) - 1) * E - 1;
          for (unsigned long long b = set; b; b &= b - 1) atomicAdd(&hr[__ffsll(static_cast<long long>(b))], 1);
        }
      }
      s_prev[tl][threadIdx.x] = set;
      __syncthreads();  // the tile is rewritten; the counts are complete
    }
    if (l > l0) {
      for (int i = threadIdx.x; i < E * E; i += kTopkTokens)
        if (h[i]) atomicAdd(&counts[(size_t)(l - 1) * E * E + i], h[i]);
      __syncthreads();
    }
  }
}

// The list length for kf (0: the passes), and dynamic shared memory.
inline int topk_list_len(int kf) { return kf <= 2 ? 2 : kf <= 4 ? 4 : kf <= 6 ? 6 : kf <= 8 ? 8 : 0; }
inline size_t topk_tile_bytes(int E) { return sizeof(float) * kTopkTokens * topk_pitch(E); }

// counts (zeroed by the caller) of L layers
static int counts_launch(const float* logits, int64_t N, int L, int E, int kf, int64_t sn, int64_t sl,
                         int32_t* counts, cudaStream_t stream) {
  static PerDevice attr;
  const cudaError_t ae = static_cast<cudaError_t>(per_device(attr, [] {
    const int most = static_cast<int>(topk_tile_bytes(64));
    cudaError_t e = cudaFuncSetAttribute(counts_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(counts_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(counts_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(counts_kernel<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(counts_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    return static_cast<int>(e);
  }));
  if (ae != cudaSuccess) return cuda_fail(ae, "cudaFuncSetAttribute(counts_kernel)");
  int64_t blocks = (N + kTopkTokens - 1) / kTopkTokens;
  const int64_t cap = (num_sms() * 6 + L - 1) / L;
  if (blocks > cap) blocks = cap;
  const dim3 grid(L, static_cast<unsigned>(blocks));
  const size_t smem = topk_tile_bytes(E);
  switch (topk_list_len(kf)) {
    case 2: counts_kernel<2><<<grid, kTopkTokens, smem, stream>>>(logits, N, E, kf, sn, sl, counts); break;
    case 4: counts_kernel<4><<<grid, kTopkTokens, smem, stream>>>(logits, N, E, kf, sn, sl, counts); break;
    case 6: counts_kernel<6><<<grid, kTopkTokens, smem, stream>>>(logits, N, E, kf, sn, sl, counts); break;
    case 8: counts_kernel<8><<<grid, kTopkTokens, smem, stream>>>(logits, N, E, kf, sn, sl, counts); break;
    default: counts_kernel<0><<<grid, kTopkTokens, smem, stream>>>(logits, N, E, kf, sn, sl, counts);
  }
  OM_LAUNCHED("counts_kernel");
  return ORDERMOE_OK;
}

// P_l(k -> k') = n / sum_k'' n (fp64, rounded once to fp32); 0 for an empty row.
// A warp a row; the counts' sum is an integer below 2^53, the same in fp64 in
// any order.
__global__ void __launch_bounds__(128) transitions_finish_kernel(const int32_t* __restrict__ counts,
                                                                 int rows, int E,
                                                                 float* __restrict__ P) {
  const int r = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const int32_t* c = counts + (size_t)r * E;
  const int c0 = lane < E ? c[lane] : 0, c1 = lane + 32 < E ? c[lane + 32] : 0;
  long long sum = (long long)c0 + c1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const double row = static_cast<double>(sum);
  float* out = P + (size_t)r * E;
  if (lane < E) out[lane] = sum > 0 ? __double2float_rn(__ddiv_rn(static_cast<double>(c0), row)) : 0.0f;
  if (lane + 32 < E)
    out[lane + 32] = sum > 0 ? __double2float_rn(__ddiv_rn(static_cast<double>(c1), row)) : 0.0f;
}

// The partial Grams of an entry summed over the chunks, in chunk order (fp64).
__device__ __forceinline__ double gram_entry(const float* __restrict__ src, int nchunks) {
  double s = 0.0;
  int c = 0;
  for (; c + 8 <= nchunks; c += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = src[(size_t)(c + u) * 4096];
#pragma unroll
    for (int u = 0; u < 8; ++u) s += static_cast<double>(v[u]);
  }
  for (; c < nchunks; ++c) s += static_cast<double>(src[(size_t)c * 4096]);
  return s;
}

// Sim(i,j) = G_ij / (sqrt(G_ii) sqrt(G_jj)) (Eq. 4), diagonal 1, zero-norm 0.
// grid (L, parts), 256 threads; block (l, b) takes the layer's entries 256 b ..
// 256 b + 255 of the E x E that there are, and first the norms it needs (all E:
// a quarter more sums than its own at E = 64). Bound by the fp64 additions, one
// in 19 cycles an SM. Reduction and quotients as two launches over 64 x 64
// entries whatever E took 24.8 + 4.0 us for 32 layers of 8 experts (37 chunks),
// 6.5 + 4.3 for 8 of 64 (75 chunks); this takes 8.3 and 10.6.
__global__ void __launch_bounds__(256) gram_sim_kernel(const float* __restrict__ gpart, int nchunks,
                                                       int E, float* __restrict__ sim) {
  __shared__ double norm[64];
  const int l = blockIdx.x;
  const float* G = gpart + (size_t)l * nchunks * 4096;
  const int x = blockIdx.y * 256 + threadIdx.x;
  const int i = x / E, j = x - i * E;
  // the last warps take the norms, so that a block's own sums run beside them
  const int d = 255 - static_cast<int>(threadIdx.x);
  if (d < E) norm[d] = sqrt(gram_entry(G + d * 65, nchunks));
  const bool mine = x < E * E && i != j;
  const double g = mine ? gram_entry(G + i * 64 + j, nchunks) : 0.0;
  __syncthreads();
  if (x >= E * E) return;
  float v = 1.0f;
  if (mine) {
    const double ni = norm[i], nj = norm[j];
    v = (ni == 0.0 || nj == 0.0) ? 0.0f : __double2float_rn(g / (ni * nj));
  }
  sim[(size_t)l * E * E + x] = v;
}

// ---------------------------------------------------------------------------
// Grouping and placement: one block of 64 threads, layers in order. Thread e
// owns expert e in the parallel parts; the greedy loops are sequential in the
// paper's order. fp64 arithmetic uses explicit round-to-nearest operations.
struct PlaceParams {
  double theta_min, theta_max, theta_single;
  double alpha_f, alpha_r, lambda1, lambda2;
};

// Integer key of an fp64 value for a descending order with NaN after every
// number: larger values get larger keys (the bits, sign-flipped for
// negatives, with -0 taken as +0), and every NaN gets 0, below them all.
__device__ __forceinline__ unsigned long long rank_key(double x) {
  if (x != x) return 0ull;
  unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x == 0.0 ? 0.0 : x));
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// One layer's scratch of the grouping (cnt is read 16 bytes at a time).
struct alignas(16) GroupSmem {
  unsigned long long kp[64];  // rank_key of p and of I, for the placement order
  unsigned long long ki[64];
  unsigned long long members[64];  // of each group
  double imp[64];
  double pls[64];
  int order[64];
  int grp[64];
  int cnt[64];
  float theta;
  int nan;  // a similarity is NaN
  int pad[2];
};
static_assert(alignof(GroupSmem) % 16 == 0 && offsetof(GroupSmem, cnt) % 16 == 0, "vector loads of cnt");
static_assert(sizeof(GroupSmem) % 16 == 0, "the similarity keys follow it in a slice");
// The similarities are kept as integer keys that order like them (-0 as +0),
// so that the greedy scan is one integer maximum per expert; 0: no value.
__device__ __forceinline__ uint32_t sim_key(float s) {
  const uint32_t u = __float_as_uint(s == 0.0f ? 0.0f : s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float sim_of_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
// Threads of a layer (a slice): a warp up to 32 experts, two above.
__host__ __device__ inline int group_slice_threads(int E) { return E <= 32 ? 32 : 64; }
__host__ __device__ inline size_t group_slice_bytes(int E) {
  return sizeof(GroupSmem) + sizeof(uint32_t) * (((size_t)E * E + 3) & ~size_t(3));
}

// Barrier of the nsync threads that group (named barrier 1: a warp that does
// something else meanwhile has no part in it).
__device__ __forceinline__ void group_sync(int nsync) {
  asm volatile("bar.sync 1, %0;" ::"r"(nsync) : "memory");
}
// Per-layer part of the plan for layer l, on the nt = group_slice_threads(E)
// threads t of a slice of the nsync that group (the layers are independent here): theta_l
// (Eq. 6), greedy cover (Eqs. 24-26), importance (Eqs. 27-28) and the
// placement order (p desc, I desc, index asc). A slice with live == false has
// no layer this time but meets every barrier.
__device__ void group_layer(GroupSmem& sm, uint32_t* K, bool live, int t, int nt, int nsync, int l,
                            const float* __restrict__ sim,
                            const int32_t* __restrict__ counts, int L, int E, PlaceParams pp,
                            const double* __restrict__ p, int32_t* __restrict__ group,
                            int32_t* __restrict__ n_groups, float* __restrict__ theta_out,
                            double* __restrict__ importance, int32_t* __restrict__ porder) {
  double* imp = sm.imp;
  double* pls = sm.pls;
  int* order = sm.order;
  int* grp = sm.grp;
  int* cnt = sm.cnt;
  const float* S = sim + (size_t)l * E * E;
  if (live && t == 0) sm.nan = 0;
  group_sync(nsync);
  if (live) {
    bool nan = false;
    if ((E & 3) == 0 && (reinterpret_cast<uintptr_t>(S) & 15u) == 0) {
#pragma unroll 8
      for (int i = t; i < E * E / 4; i += nt) {
        const float4 v = reinterpret_cast<const float4*>(S)[i];
        nan |= v.x != v.x || v.y != v.y || v.z != v.z || v.w != v.w;
        reinterpret_cast<uint4*>(K)[i] =
            make_uint4(sim_key(v.x), sim_key(v.y), sim_key(v.z), sim_key(v.w));
      }
    } else {
#pragma unroll 8
      for (int i = t; i < E * E; i += nt) {
        const float v = S[i];
        nan |= v != v;
        K[i] = sim_key(v);
      }
    }
    if (nan) sm.nan = 1;
    if (t < E) {
      sm.members[t] = 0ull;
      cnt[t] = counts[(size_t)l * E + t];
      pls[t] = p[(size_t)l * E + t];
      if (!(pls[t] >= 0.0)) report(&g_err_sim, ORDERMOE_DEV_BAD_VALUE, l * E + t);  // Eq. 29's p
    }
    if (t < 32) {  // Eq. 6 (layers numbered from 1), by one warp (fp64 is slow)
      float theta;
      if (L <= 1) {
        theta = __double2float_rn(pp.theta_single);
      } else {
        const double frac = __ddiv_rn(static_cast<double>(L - (l + 1)), static_cast<double>(L - 1));
        theta = __double2float_rn(
            __dadd_rn(pp.theta_min, __dmul_rn(__dsub_rn(pp.theta_max, pp.theta_min), frac)));
      }
      if (t == 0) sm.theta = theta;
    }
  }
  group_sync(nsync);
  const float theta = live ? sm.theta : 0.0f;
  // visiting order: count desc, index asc
  if (live && t < E) {
    const int mine = cnt[t];
    int r = 0;
    int e = 0;
#pragma unroll 4
    for (; e + 4 <= E; e += 4) {
      const int4 c = *reinterpret_cast<const int4*>(cnt + e);
      r += (c.x > mine || (c.x == mine && e < t)) ? 1 : 0;
      r += (c.y > mine || (c.y == mine && e + 1 < t)) ? 1 : 0;
      r += (c.z > mine || (c.z == mine && e + 2 < t)) ? 1 : 0;
      r += (c.w > mine || (c.w == mine && e + 3 < t)) ? 1 : 0;
    }
    for (; e < E; ++e) r += (cnt[e] > mine || (cnt[e] == mine && e < t)) ? 1 : 0;
    order[r] = t;
  }
  group_sync(nsync);
  // Eqs. 24-26 in the visiting order; warp 0 of the slice compares an expert
  // with the existing dominants in parallel (lane g has dominants g and g +
  // 32): the largest similarity, ties to the earlier dominant.
  if (live && t < 32) {
    int k = 0;
    int dom0 = 0, dom1 = 0;  // dominants t and t + 32, when there are that many
    if (!sm.nan) {
      const uint32_t low = theta != theta ? 0u : sim_key(theta);  // a NaN threshold: nothing is below
      int jn = order[0];
      for (int pos = 0; pos < E; ++pos) {
        const int j = jn;
        jn = order[min(pos + 1, E - 1)];
        const uint32_t* row = K + j * E;
        const uint32_t k0 = t < k ? row[dom0] : 0u, k1 = t + 32 < k ? row[dom1] : 0u;
        const uint32_t mk = __reduce_max_sync(0xffffffffu, max(k0, k1));
        int g;
        if (k == 0 || mk < low) {
          if (t == k) dom0 = j;
          if (t + 32 == k) dom1 = j;
          g = k++;
        } else {
          const unsigned lo32 = __ballot_sync(0xffffffffu, k0 == mk);
          g = lo32 ? __ffs(lo32) - 1 : __ffs(__ballot_sync(0xffffffffu, k1 == mk)) + 31;
        }
        if (t == 0) grp[j] = g;
      }
    } else {
      // The choice is the scan's in dominant order: the first dominant unless a
      // later one is strictly more similar. With NaN similarities that is the
      // first dominant when its similarity is NaN, else the first maximum with
      // NaN counted as -inf.
      int first = 0;
      for (int pos = 0; pos < E; ++pos) {
        const int j = order[pos];
        auto key = [&](int dom) {
          const float v = S[j * E + dom];
          return sim_key(v != v ? -INFINITY : v);
        };
        const uint32_t k0 = t < k ? key(dom0) : 0u, k1 = t + 32 < k ? key(dom1) : 0u;
        const uint32_t mk = __reduce_max_sync(0xffffffffu, max(k0, k1));
        const float s0 = k > 0 ? S[j * E + first] : 0.0f;
        int g;
        if (s0 != s0) {  // NaN first: the scan keeps dominant 0 (and NaN < theta is false)
          g = 0;
        } else if (k == 0 || sim_of_key(mk) < theta) {
          if (k == 0) first = j;
          if (t == k) dom0 = j;
          if (t + 32 == k) dom1 = j;
          g = k++;
        } else {
          const unsigned lo32 = __ballot_sync(0xffffffffu, k0 == mk);
          g = lo32 ? __ffs(lo32) - 1 : __ffs(__ballot_sync(0xffffffffu, k1 == mk)) + 31;
        }
        if (t == 0) grp[j] = g;
      }
    }
    if (t == 0) {
      n_groups[l] = k;
      theta_out[l] = theta;
    }
  }
  group_sync(nsync);
  // Eqs. 27-28; each group's members as a bit mask, so that a thread adds its
  // own group's similarities only (in ascending order)
  if (live && t < E) atomicOr(&sm.members[grp[t]], 1ull << t);
  group_sync(nsync);
  // the counts' fp64 sum in index order, formed exactly as an integer sum
  // (every partial sum is an integer below 2^53, so each fp64 addition is exact)
  long long total_i = 0;
  if (live)
    for (int e = 0; e < E; ++e) total_i += cnt[e];
  const double total = static_cast<double>(total_i);
  if (live && t < E) {
    group[(size_t)l * E + t] = grp[t];
    double sum = 0.0;
    const unsigned long long mates = sm.members[grp[t]];
    for (unsigned long long b = mates; b; b &= b - 1)
    {
      const int e = __ffsll(static_cast<long long>(b)) - 1;
      sum = __dadd_rn(sum, static_cast<double>(sm.nan ? S[t * E + e] : sim_of_key(K[t * E + e])));
    }
    const double rho = __ddiv_rn(sum, static_cast<double>(__popcll(mates)));
    const double f = total > 0.0 ? __ddiv_rn(static_cast<double>(cnt[t]), total) : 0.0;
    imp[t] = __dadd_rn(__dmul_rn(pp.alpha_f, f), __dmul_rn(pp.alpha_r, rho));
    if (importance != nullptr) importance[(size_t)l * E + t] = imp[t];
  }
  group_sync(nsync);
  // placement order: p desc, I desc, index asc, with NaN after every number
  // (a total order, so the ranks are a permutation whatever the values),
  // compared on integer keys
  if (live && t < E) {
    sm.kp[t] = rank_key(pls[t]);
    sm.ki[t] = rank_key(imp[t]);
  }
  group_sync(nsync);
  if (live && t < E) {
    const unsigned long long kpt = sm.kp[t], kit = sm.ki[t];
    int r = 0;
    for (int e = 0; e < E; ++e) {
      const unsigned long long kpe = sm.kp[e], kie = sm.ki[e];
      r += (kpe > kpt || (kpe == kpt && (kie > kit || (kie == kit && e < t)))) ? 1 : 0;
    }
    porder[(size_t)l * E + r] = t;
  }
}

// One block per layer l = l0 + blockIdx.x, group_slice_threads(E) threads.
__global__ void __launch_bounds__(64) group_kernel(
    const float* __restrict__ sim, const int32_t* __restrict__ counts, int L, int E, int l0,
    PlaceParams pp, const double* __restrict__ p, int32_t* __restrict__ group,
    int32_t* __restrict__ n_groups, float* __restrict__ theta_out, double* __restrict__ importance,
    int32_t* __restrict__ porder) {
  __shared__ GroupSmem sm;
  __shared__ __align__(16) uint32_t K[64 * 64];
  group_layer(sm, K, true, threadIdx.x, blockDim.x, blockDim.x, l0 + blockIdx.x, sim, counts, L, E, pp, p, group, n_groups,
              theta_out, importance, porder);
}

// b / C rounded to nearest by Markstein's correction step (P. Markstein, IBM J.
// Res. Dev. 34(1), 1990): with y = 1/C rounded to nearest and q = RN(b y)
// within one ulp of b / C, the residual r = b - C q is exact in one fma, and
// RN(q + r y) is the correctly rounded quotient (no underflow or overflow).
// Three dependent fp64 operations instead of a full division.
__device__ __forceinline__ double div_rn_markstein(double b, double C, double y) {
  const double q = __dmul_rn(b, y);
  const double r = __fma_rn(-q, C, b);
  return __fma_rn(r, y, q);
}

__global__ void div_selftest_kernel(const double* __restrict__ a, const double* __restrict__ b,
                                    double* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = div_rn_markstein(a[i], b[i], __drcp_rn(b[i]));
}

// Mandatory placement, Eqs. 29-31 (Alg. 1): one warp, layers and
// experts in order, b_m carried over the layers. Lane m keeps server m's
// state in registers: b_m, C_m and lambda1 * (b_m / C_m); lambda2 * eta for
// every count is a table. Per expert (experts of one size take their scores
// from tables, see below), lane m forms its score (one fp64 add of the two
// terms, as Eq. 30 states them) and, speculatively, the ratio term it
// would have after taking the expert; the argmin runs on integer keys
// (scores are non-negative, so their bit patterns order like the values; ties
// to the lower server), and the winner keeps its speculative term. A
// waiting-list expert goes to the server with the most room after its layer.
// Layers l0 .. l1 - 1: the first range starts from b_m = 0 and sets the
// status, a later range continues from b_m in used (lambda1 * (b_m / C_m) is
// recomputed from it, the same function the loop applies) and only raises the
// capacity status.
constexpr int kPlaceTable = 4096;  // (server, wins) entries
struct PlaceSmem {
  // uniform sizes: server m after n more experts, at m * depth + n
  double after_b[kPlaceTable];  // b_m
  double l2eta[65];  // lambda2 * eta for eta = 0 .. 64
  double pls[64];
  int grp[64];
  int ord[64];
  int waiting[64];
  int ready;
  int seq[64];      // experts in order with their groups
  uint8_t who[64];  // the server of each, plus one
  alignas(16) uint8_t xs[32 * 64];
  alignas(16) int eta[32 * 64];
};
static_assert(sizeof(PlaceSmem) % 16 == 0, "vector stores into xs and eta");

// Experts of one size (their memory p bitwise equal over the range's layers,
// as a model's experts are): a server's b_m and ratio term then depend on how
// many experts it has taken only, whichever they were, and a score on that and
// on eta. A producer warp tabulates b_m and the scores as ordered keys, ahead
// of the warp that places, whose loop is left without fp64 (an instruction
// holds a lone warp for 65 cycles). depth rows a server, cols scores a row
// (eta = 0 .. cols - 1; larger ones are added up when they come); ready rows of
// them are there. With the states alone tabulated, an fp64 addition an expert left
// and a branch for ties, 512 experts on 8 servers took 151 us and 256 on 4 (32
// layers) 105; this takes 101 and 79 (ncu), the second half of it per-layer work.
__host__ __device__ inline int place_depth(int M, int experts) {
  const int want = 2 * experts / M + 16, room = kPlaceTable / M;
  return want < room ? want : room;
}
// Score columns: a producer warp fills a row of all servers in M cols / 32 steps,
// and must fill rows faster than M experts are placed. Two rows more are for the
// lanes without a server. (19 columns for 8 servers: 198 us instead of 101.)
__host__ __device__ inline int place_cols(int M) { return M <= 4 ? 8 : 4; }
__host__ __device__ inline size_t place_score_bytes(int M, int experts) {
  return 8 * ((size_t)M * place_depth(M, experts) + 2) * place_cols(M);
}

// Whether n experts of one size take the tables. The placement of one expert must
// take longer than the producer's row, and a short range does not win back the
// wait for the first rows. Tables against the general loop, us of a call with one
// group and with eight groups a layer:
//   servers, experts   1, 1536          2, 1536      2, 64      3, 64      4, 1536
//                      1053 1041 / 705 694  799 667 / 842 832  92 61 / 65 53  83 63 / 67 55  507 363 / 717 705
//                      4, 64      4, 32    4, 8      8, 64      12, 64
//                      59 41 / 65 55  26 26 / 32 32  21 19 / 19 18  63 41 / 67 55  63-96 45-47 / 69 57
//                      16, 128    16, 64    32, 1536     32, 128    32, 64
//                      69 66 / 86 82  92 71 / 69 57  553 524 / 799 789  78 74 / 90 87  98 86 / 77 65
__host__ __device__ inline bool place_tabulated(int M, int n) {
  return M >= 2 && (n >= 96 || (n >= 32 && M >= 4 && M <= 8));
}

constexpr unsigned long long kNoServer = ~0ull;           // the expert does not fit
constexpr unsigned long long kOddScore = 0x7FF0ull << 48;  // not a plain non-negative number

// a score as a key: non-negative finite values order like their bit patterns
// (an infinity, a NaN, a negative score or -0 sends the layer to the general loop)
__device__ __forceinline__ unsigned long long place_key(double sc) {
  const unsigned long long k = static_cast<unsigned long long>(__double_as_longlong(sc));
  return k >= kOddScore ? kOddScore : k;
}
// The key for an eta past the columns, from the row's eta = 0 (whose score is
// the ratio term). Out of line: inlined, its fp64 is issued for every expert.
__device__ __noinline__ unsigned long long place_key_past(unsigned long long base, double l2) {
  if (base >= kOddScore) return base;
  return place_key(__dadd_rn(__longlong_as_double(static_cast<long long>(base)), l2));
}
// ready rows once there are `need` of them (at most depth), or those there after
// the limit of about 0.1 s (the producer never waits, so that is not reached).
__device__ __noinline__ int place_wait(PlaceSmem& sm, int need, int depth) {
  need = need < depth ? need : depth;
  int v = 0;
  for (int i = 0; i < (1 << 21); ++i) {
    asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(&sm.ready)) : "memory");
    if (v >= need) break;
  }
  return v;
}
// before the producer starts, the whole block: l2eta and the spare rows
__device__ void place_tables_init(PlaceSmem& sm, unsigned long long* score, int M, int depth, int cols,
                                  double lambda2, int t, int nt) {
  for (int i = t; i <= 64; i += nt) sm.l2eta[i] = __dmul_rn(lambda2, static_cast<double>(i));
  if (depth > 0)
    for (int i = t; i < 2 * cols; i += nt) score[(size_t)M * depth * cols + i] = kNoServer;
  if (t == 0) sm.ready = 0;
}
// The producer: one warp, lane m server m, b_m after 0 .. depth - 1 more
// experts of size p, the additions in the order the placement makes them, and
// the keys of placing one more then.
__device__ void place_produce(PlaceSmem& sm, unsigned long long* score, int lane, int M, int depth,
                              int cols, double p, bool first, double lambda1,
                              const double* __restrict__ C, const double* __restrict__ used) {
  const bool srv = lane < M;
  double b = (srv && !first) ? used[lane] : 0.0;
  const double cap = srv ? C[lane] : 1.0, rcap = __drcp_rn(cap);
  const int at = srv ? lane * depth : 0;
  const int e = lane & (cols - 1), m0 = lane / cols;  // cols is a power of two
  const double l2 = sm.l2eta[e];
  for (int n = 0; n < depth; ++n) {
    const double a1 = __dmul_rn(lambda1, div_rn_markstein(b, cap, rcap));
    if (srv) sm.after_b[at + n] = b;
    b = __dadd_rn(b, p);
    const int feas = __double_as_longlong(b) <= __double_as_longlong(cap);  // b <= C_m, b >= 0
    for (int mb = 0; mb < M; mb += 32 / cols) {
      const int m = mb + m0;
      const double am = __shfl_sync(0xffffffffu, a1, m & 31);
      const int fm = __shfl_sync(0xffffffffu, feas, m & 31);
      const unsigned long long key = place_key(__dadd_rn(am, l2));
      if (m < M) score[((size_t)m * depth + n) * cols + e] = fm ? key : kNoServer;
    }
    if (n < 3 || (n & 3) == 3 || n + 1 == depth) {  // four rows at a time, the first as they come
      __syncwarp();
      if (lane == 0)
        asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(&sm.ready)), "r"(n + 1) : "memory");
    }
  }
}
// whether p[0 .. n - 1] are bitwise equal (and not negative or NaN: those take
// the general loop, which reports them), for the whole block
__device__ bool place_uniform(const double* __restrict__ p, int n, int t, int nt) {
  const long long p0 = __double_as_longlong(p[0]);
  bool same = p[0] >= 0.0;
  for (int i = t; i < n; i += nt) same = same && __double_as_longlong(p[i]) == p0;
  return __syncthreads_and(same) != 0;
}

// The placement on warp 0 of a block (threadIdx.x < 32); returns 1 when a
// waiting-list expert overfilled its server.
// depth > 0: the sizes are uniform and the tables hold depth rows a server.
__device__ int place_layers(PlaceSmem& sm, const unsigned long long* score, int cols, const int32_t* __restrict__ group,
                             const int32_t* __restrict__ porder, int L, int E, int M, int l0,
                             int l1, int first, PlaceParams pp, const double* __restrict__ p,
                             const double* __restrict__ C, uint8_t* __restrict__ placement,
                             double* __restrict__ used, int depth) {
  int* grp = sm.grp;
  int* ord = sm.ord;
  double* pls = sm.pls;
  int* waiting = sm.waiting;
  uint8_t* xs = sm.xs;
  int* eta = sm.eta;
  double* l2eta = sm.l2eta;
  const int t = threadIdx.x;
  int overflow = 0;
  const bool srv = t < M;
  double b = (srv && !first) ? used[t] : 0.0;
  const double cap = srv ? C[t] : 1.0;
  const double rcap = __drcp_rn(cap);
  // non-negative finite values compare like their bit patterns
  const long long cap_bits = __double_as_longlong(cap);
  double a1 = srv ? __dmul_rn(pp.lambda1, div_rn_markstein(b, cap, rcap)) : 0.0;
  bool bad_score = srv && !(cap > 0.0 && cap <= 1.7976931348623157e308);
  int wins = 0;   // experts this server took in the range (uniform sizes)
  int avail = 0;  // rows of its tables known to be there
  // the next layer's rows, loaded a layer ahead (two experts a lane)
  int g2[2] = {0, 0}, o2[2] = {0, 0};
  double p2[2] = {0.0, 0.0};
  auto fetch = [&](int l) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (t + 32 * h < E) {
        g2[h] = group[(size_t)l * E + t + 32 * h];
        o2[h] = porder[(size_t)l * E + t + 32 * h];
        p2[h] = p[(size_t)l * E + t + 32 * h];
      }
  };
  fetch(l0);
  __syncwarp();
  for (int l = l0; l < l1; ++l) {
    for (int i = t; i < 16 * M; i += 32) {
      reinterpret_cast<uint32_t*>(xs)[i] = 0u;
      reinterpret_cast<int4*>(eta)[i] = make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (t + 32 * h < E) {
        grp[t + 32 * h] = g2[h];
        ord[t + 32 * h] = o2[h];
        pls[t + 32 * h] = p2[h];
      }
    if (l + 1 < l1) fetch(l + 1);
    __syncwarp();
    int nw = 0;
    bool general = depth == 0;
    if (!general) {
      // One pass over the experts, written to branch as little as it can (a
      // warp alone pays 20 cycles and more for each): an odd score, or a server
      // past its table, makes the layer start over below.
      const int wins0 = wins;
      // the experts in order with their groups (expert | group << 8), read ahead
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (t + 32 * h < E) sm.seq[t + 32 * h] = ord[t + 32 * h] | (grp[ord[t + 32 * h]] << 8);
        sm.who[t + 32 * h] = 0;
      }
      if (srv && wins + 1 >= avail) avail = place_wait(sm, wins + 2, depth);
      bool odd = srv && wins + 1 >= avail;
      __syncwarp();
      if (!__any_sync(0xffffffffu, odd)) {
        // this server's row, and the one after it for a further expert
        const unsigned long long* row = score + (size_t)(srv ? t * depth + wins : M * depth) * cols;
        int* my_eta = eta + (srv ? t * 64 : 0);
        int cur = sm.seq[0];
        int nxt = sm.seq[min(1, E - 1)];
        int ec = 0;  // experts of cur's group on this server
        unsigned long long key = row[0];
        for (int pos = 0; pos < E; ++pos) {
          // the next expert's count and key, if this server takes cur and if not
          const int after = sm.seq[min(pos + 2, E - 1)];
          const int en = my_eta[nxt >> 8];
          const int ew = (nxt >> 8) == (cur >> 8) ? ec + 1 : en;
          unsigned long long ks = row[min(en, cols - 1)], kw = row[cols + min(ew, cols - 1)];
          if (ew >= cols) {  // (en <= ew)
            if (en >= cols) ks = place_key_past(row[0], l2eta[min(en, 64)]);
            kw = place_key_past(row[cols], l2eta[min(ew, 64)]);
          }
          const unsigned khi = static_cast<unsigned>(key >> 32), klo = static_cast<unsigned>(key);
          odd |= key == kOddScore;
          const unsigned mhi = __reduce_min_sync(0xffffffffu, khi);
          const unsigned mlo = __reduce_min_sync(0xffffffffu, khi == mhi ? klo : 0xffffffffu);
          const unsigned win = __ballot_sync(0xffffffffu, khi == mhi && klo == mlo);
          const bool won = mhi != 0xffffffffu && t == __ffs(win) - 1;  // none: it waits
          if (won) {
            sm.who[pos] = static_cast<uint8_t>(t + 1);
            my_eta[cur >> 8] = ec + 1;
            ++wins;
            row += cols;
            if (wins + 1 >= avail) {  // seldom
              avail = place_wait(sm, wins + 2, depth);
              if (wins + 1 >= avail) {
                odd = true;
                row -= cols;  // the rows end here
              }
            }
          }
          key = won ? kw : ks;
          ec = won ? ew : en;
          cur = nxt;
          nxt = after;
        }
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, odd)) {
        general = true;
        wins = wins0;
        a1 = srv ? __dmul_rn(pp.lambda1, div_rn_markstein(b, cap, rcap)) : 0.0;
        for (int i = t; i < 16 * M; i += 32) reinterpret_cast<int4*>(eta)[i] = make_int4(0, 0, 0, 0);
        __syncwarp();
      } else {
        if (srv) b = sm.after_b[t * depth + wins];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (t + 32 * h < E) {
            const int m = sm.who[t + 32 * h];
            if (m > 0) xs[(m - 1) * 64 + (sm.seq[t + 32 * h] & 0xFF)] = 1;
          }
        // the waiting list, in order
        const unsigned w0 = __ballot_sync(0xffffffffu, t < E && sm.who[t] == 0);
        const unsigned w1 = __ballot_sync(0xffffffffu, t + 32 < E && sm.who[t + 32 < 64 ? t + 32 : 0] == 0);
        if ((w0 >> t) & 1u) waiting[__popc(w0 & ((1u << t) - 1u))] = sm.seq[t] & 0xFF;
        if ((w1 >> t) & 1u) waiting[__popc(w0) + __popc(w1 & ((1u << t) - 1u))] = sm.seq[t + 32] & 0xFF;
        nw = __popc(w0) + __popc(w1);
        __syncwarp();
      }
    }
    if (general) {
    int jn = ord[0];
    int gn = grp[jn];
    double pn = pls[jn];
    for (int pos = 0; pos < E; ++pos) {
      const int j = jn, g = gn;
      const double pj = pn;
      if (pos + 1 < E) {  // the next expert does not depend on this one's outcome
        jn = ord[pos + 1];
        gn = grp[jn];
        pn = pls[jn];
      }
      // the fp64 work on the server lanes only (the other lanes' keys are ~0)
      double bn = 0.0, a1n = 0.0;
      unsigned long long key = ~0ull;
      if (srv) {
        bn = __dadd_rn(b, pj);
        const bool feas = __double_as_longlong(bn) <= cap_bits;  // bn <= C_m, bn >= 0
        const int et = min(eta[t * 64 + g], 64);  // at most E <= 64
        const double sc = __dadd_rn(a1, l2eta[et]);
        if (feas) {
          a1n = __dmul_rn(pp.lambda1, div_rn_markstein(bn, cap, rcap));  // kept if this lane wins
          unsigned long long ks = static_cast<unsigned long long>(__double_as_longlong(sc));
          // !(sc >= 0) on the bits: a NaN, or a negative value other than -0
          const unsigned long long mag = ks & 0x7FFFFFFFFFFFFFFFull;
          bad_score |= mag > 0x7FF0000000000000ull || (ks != mag && mag != 0);
          key = (ks == 0x8000000000000000ull) ? 0ull : ks;  // -0 orders like +0
        }
      }
      // argmin of the 64-bit keys, ties to the lower server: minimum of the high
      // words, then of the low words among those lanes, then the lowest lane
      const unsigned khi = static_cast<unsigned>(key >> 32), klo = static_cast<unsigned>(key);
      const unsigned mhi = __reduce_min_sync(0xffffffffu, khi);
      const unsigned mlo = __reduce_min_sync(0xffffffffu, khi == mhi ? klo : 0xffffffffu);
      const unsigned win = __ballot_sync(0xffffffffu, khi == mhi && klo == mlo);
      int m = __ffs(win) - 1;
      if (mhi == 0xffffffffu && mlo == 0xffffffffu) m = 64;  // no feasible server
      if (m == 64) {
        if (t == 0) waiting[nw] = j;
        ++nw;
      } else if (t == m) {
        xs[m * 64 + j] = 1;
        eta[m * 64 + g] += 1;
        b = bn;
        a1 = a1n;
        ++wins;
      }
      __syncwarp();
    }
    }
    // waiting list: the server with the largest C_m - b_m (ties: lower m)
    for (int w = 0; w < nw; ++w) {
      const int j = waiting[w];
      const double room = srv ? __dsub_rn(cap, b) : -INFINITY;
      double br = room;
      int bm = srv ? t : 64;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double orr = __shfl_xor_sync(0xffffffffu, br, o);
        const int om_ = __shfl_xor_sync(0xffffffffu, bm, o);
        if (orr > br || (orr == br && om_ < bm)) {
          br = orr;
          bm = om_;
        }
      }
      if (t == bm) {
        xs[bm * 64 + j] = 1;
        b = __dadd_rn(b, pls[j]);
        a1 = __dmul_rn(pp.lambda1, div_rn_markstein(b, cap, rcap));
        ++wins;  // an expert of the same size
        if (b > cap) overflow = 1;
      }
      __syncwarp();
    }
    uint8_t* x = placement + (size_t)l * M * E;
    if ((E & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 3u) == 0) {
      for (int i = t; i < M * E / 4; i += 32) {
        const int m = i / (E / 4), e4 = i - m * (E / 4);
        reinterpret_cast<uint32_t*>(x)[i] = reinterpret_cast<const uint32_t*>(xs)[m * 16 + e4];
      }
    } else {
      for (int i = t; i < M * E; i += 32) x[i] = xs[(i / E) * 64 + (i % E)];
    }
    __syncwarp();
  }
  if (srv) used[t] = b;
  overflow = __any_sync(0xffffffffu, overflow != 0);
  if (__any_sync(0xffffffffu, bad_score) && t == 0)
    report(&g_err_sim, ORDERMOE_DEV_BAD_VALUE, 0);
  return overflow;
}

// Eq. 29's memory over all layers against the servers' total (the capacity
// status of the first range): one fp64 sum in order, the values loaded a warp
// at a time.
__device__ int demand_exceeds(const double* __restrict__ p, int n, const double* __restrict__ C,
                              int M, int lane) {
  double need = 0.0, have = 0.0;
  double v = lane < n ? p[lane] : 0.0;
  for (int i = 0; i < n; i += 32) {
    const double cur = v;
    if (i + 32 + lane < n) v = p[i + 32 + lane];
    const int m = min(32, n - i);
    for (int k = 0; k < m; ++k) need = __dadd_rn(need, __shfl_sync(0xffffffffu, cur, k));
  }
  const double c = lane < M ? C[lane] : 0.0;
  for (int m = 0; m < M; ++m) have = __dadd_rn(have, __shfl_sync(0xffffffffu, c, m));
  return need > have ? 1 : 0;
}

// Status of a placed range: the first range sets it, a later one only raises
// the capacity error.
__device__ void place_status(int first, int overflow, int32_t* __restrict__ status) {
  if (first || overflow) *status = overflow ? ORDERMOE_ERR_CAPACITY : ORDERMOE_OK;
}

// The placement of a grouped range by a block of at least four warps: the loop
// on warp 0, the capacity check of the first range beside it on warp 3 (and
// the producer of the tables on another).
__device__ void place_range(PlaceSmem& sm, const unsigned long long* score, int cols, int* s_over, const int32_t* __restrict__ group,
                            const int32_t* __restrict__ porder, int L, int E, int M, int l0, int l1,
                            int first, PlaceParams pp, const double* __restrict__ p,
                            const double* __restrict__ C, uint8_t* __restrict__ placement,
                            double* __restrict__ used, int32_t* __restrict__ status, int depth) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int over = 0;
  if (warp == 0)
    over = place_layers(sm, score, cols, group, porder, L, E, M, l0, l1, first, pp, p, C, placement, used, depth);
  else if (warp == 3 && first) {
    const int d = demand_exceeds(p, L * E, C, M, lane);
    if (lane == 0) *s_over = d;
  }
  __syncthreads();
  if (tid == 0) place_status(first, over | (first ? *s_over : 0), status);
}

constexpr int kPlaceThreads = 128;

__global__ void __launch_bounds__(kPlaceThreads) place_kernel(
    const int32_t* __restrict__ group, const int32_t* __restrict__ porder, int L, int E, int M,
    int l0, int l1, int first, PlaceParams pp, const double* __restrict__ p,
    const double* __restrict__ C, uint8_t* __restrict__ placement, double* __restrict__ used,
    int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char s_pl[];
  PlaceSmem& sm = *reinterpret_cast<PlaceSmem*>(s_pl);
  unsigned long long* score = reinterpret_cast<unsigned long long*>(s_pl + sizeof(PlaceSmem));
  __shared__ int s_over;
  const int n = (l1 - l0) * E;
  const bool tables = place_tabulated(M, n) && place_uniform(p + (size_t)l0 * E, n, threadIdx.x, blockDim.x);
  const int depth = tables ? place_depth(M, n) : 0, cols = place_cols(M);
  place_tables_init(sm, score, M, depth, cols, pp.lambda2, threadIdx.x, blockDim.x);
  __syncthreads();
  if (tables && (threadIdx.x >> 5) == 1)
    place_produce(sm, score, threadIdx.x & 31, M, depth, cols, p[(size_t)l0 * E], first, pp.lambda1, C, used);
  place_range(sm, score, cols, &s_over, group, porder, L, E, M, l0, l1, first, pp, p, C, placement, used, status,
              depth);
}

// Grouping and placement of layers l0 .. l1 - 1 in one block: the grouping
// runs several layers at a time on all warps but the last, which produces the
// placement's tables meanwhile; then warp 0 places the layers in order (one
// block, so the pipelined plan's side stream holds one SM).
// Bound: the serial chains (a group per expert, a server per expert). A layer
// of 64 experts took about 28 us to place and 10 to group (8 layers 282 us
// under ncu); with the servers' states tabulated and the integer scan 8 layers
// took 186 us, with the scores tabulated too 132.
constexpr int kGroupThreads = 256;

__host__ __device__ inline int group_slices(int E) { return kGroupThreads / group_slice_threads(E); }
static size_t group_place_smem(int E, int M, int experts) {
  return ((group_slices(E) * group_slice_bytes(E) + 15) & ~size_t(15)) + sizeof(PlaceSmem) +
         place_score_bytes(M, experts);
}
constexpr int kPlaceRange = 512;  // experts of a range
constexpr size_t kPlaceSmemMax = 200 * 1024;  // of either placing kernel, at any M
static size_t place_smem(int M, int experts) { return sizeof(PlaceSmem) + place_score_bytes(M, experts); }

__global__ void __launch_bounds__(kGroupThreads + 32) group_place_kernel(
    const float* __restrict__ sim, const int32_t* __restrict__ counts, int L, int E, int M, int l0,
    int l1, int first, PlaceParams pp, const double* __restrict__ p, const double* __restrict__ C,
    int32_t* __restrict__ group, int32_t* __restrict__ n_groups, float* __restrict__ theta_out,
    double* __restrict__ importance, int32_t* __restrict__ porder, uint8_t* __restrict__ placement,
    double* __restrict__ used, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char s_gp[];
  const int nt = group_slice_threads(E), slices = group_slices(E);
  PlaceSmem& ps = *reinterpret_cast<PlaceSmem*>(
      s_gp + ((slices * group_slice_bytes(E) + 15) & ~size_t(15)));
  unsigned long long* score = reinterpret_cast<unsigned long long*>(&ps + 1);
  __shared__ int s_over;
  const int n = (l1 - l0) * E;
  const bool tables = place_tabulated(M, n) && place_uniform(p + (size_t)l0 * E, n, threadIdx.x, blockDim.x);
  const int depth = tables ? place_depth(M, n) : 0, cols = place_cols(M);
  const int slice = threadIdx.x / nt;
  unsigned char* own = s_gp + (slice < slices ? slice : 0) * group_slice_bytes(E);
  GroupSmem& gs = *reinterpret_cast<GroupSmem*>(own);
  uint32_t* K = reinterpret_cast<uint32_t*>(own + sizeof(GroupSmem));
  place_tables_init(ps, score, M, depth, cols, pp.lambda2, threadIdx.x, blockDim.x);
  __syncthreads();
  if (slice >= slices) {  // the last warp
    if (tables)
      place_produce(ps, score, threadIdx.x & 31, M, depth, cols, p[(size_t)l0 * E], first, pp.lambda1, C, used);
  } else {
    for (int lb = l0; lb < l1; lb += slices) {
      const int l = lb + slice;
      group_layer(gs, K, l < l1, threadIdx.x % nt, nt, kGroupThreads, l, sim, counts, L, E, pp, p,
                  group, n_groups, theta_out, importance, porder);
      group_sync(kGroupThreads);  // the slices' scratch is reused; group and porder are written
    }
  }
  place_range(ps, score, cols, &s_over, group, porder, L, E, M, l0, l1, first, pp, p, C, placement, used, status,
              depth);
}

}  // namespace om

using namespace om;

namespace om {
bool sim_tc_supported(int L, int E);
int sim_tc_nsplit(int L, int E, int64_t N);
int sim_tc_max_splits();
int sim_tc_launch(const uint16_t* X, int N, const uint16_t* W, int L, int E, int d, int kf,
                  float* H, uint16_t* hi, uint16_t* lo, int ldT, int32_t* counts, float* gpart,
                  int nsplit, bool reserve_sm, cudaStream_t stream);
}  // namespace om

// Workspace: H [N][L E] fp32 | the hi/lo bf16 planes of H^T [L E][ldT] (tensor-core
// path) | partial Grams [L][parts][64][64] fp32.
static int64_t sim_ldT(int64_t N) { return (N + 7) / 8 * 8; }

// Partial Grams per layer the workspace holds: one per 1024-token chunk on
// the CUDA-core path, one per token split (at most sim_tc_max_splits, and at
// most one per 64-token step) on the tensor-core path.
static int64_t sim_parts(int L, int E, int64_t N) {
  if (!sim_tc_supported(L, E)) return (N + kSimChunk - 1) / kSimChunk;
  const int64_t kb = (N + 63) / 64;
  return kb < sim_tc_max_splits() ? kb : sim_tc_max_splits();
}

// Workspace of the similarity: H [N][L E] fp32 (with_H; the CUDA-core path
// and the logits-keeping call need it), the hi/lo planes (tensor-core path) and
// the partial Grams.
static size_t sim_ws_bytes(int L, int E, int64_t N, bool with_H) {
  if (L <= 0 || E <= 0 || E > ORDERMOE_MAX_EXPERTS || N <= 0) return 0;
  auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
  const size_t h = with_H ? up((size_t)N * L * E * sizeof(float)) : 0;
  const size_t planes = sim_tc_supported(L, E) ? 2 * up((size_t)L * E * sim_ldT(N) * 2) : 0;
  const size_t g = (size_t)L * sim_parts(L, E, N) * 64 * 64 * sizeof(float);
  return h + planes + up(g);
}

extern "C" size_t ordermoe_similarity_workspace_bytes(int L, int E, int64_t N) {
  return sim_ws_bytes(L, E, N, true);
}

// The similarity arguments a call needs (Eqs. 3-5), checked.
static int similarity_check(const uint16_t* W_r, const uint16_t* X_cal, int L, int E, int d,
                            int64_t N, int k_freq, const float* sim, const int32_t* counts,
                            const void* workspace, size_t workspace_bytes, size_t need_bytes) {
  if (L <= 0 || E <= 0 || E > ORDERMOE_MAX_EXPERTS || k_freq <= 0 || k_freq > E)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "similarity: need L >= 1, 1 <= k_freq <= E <= 64");
  if (d <= 0 || d % 64 != 0)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "similarity: d must be a positive multiple of 64");
  if (N <= 0 || N > 65535LL * kSimChunk || (int64_t)L * E > INT32_MAX || L > 65535)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "similarity: need 1 <= N <= 65535 * 1024");
  if (!W_r || !X_cal || !sim || !counts || !workspace)
    return fail(ORDERMOE_ERR_INVALID_ARG, "similarity: null pointer");
  if (!aligned16(W_r) || !aligned16(X_cal) || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return fail(ORDERMOE_ERR_INVALID_ARG, "similarity: W_r/X_cal 16-byte and workspace 256-byte aligned");
  if (workspace_bytes < need_bytes)
    return fail(ORDERMOE_ERR_INVALID_ARG, "similarity: workspace too small");
  return ORDERMOE_OK;
}

// Where the similarity's scratch lives in its workspace.
struct SimLayout {
  float* H;
  uint16_t* hi;
  uint16_t* lo;
  float* gpart;
  int64_t ldT;
  int nchunks;
  bool tc;
};

static SimLayout similarity_layout(void* workspace, int L, int E, int64_t N, bool with_H) {
  auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
  SimLayout w;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  w.H = with_H ? reinterpret_cast<float*>(ws) : nullptr;
  w.tc = sim_tc_supported(L, E);
  w.nchunks = static_cast<int>((N + kSimChunk - 1) / kSimChunk);
  w.ldT = sim_ldT(N);
  const size_t plane = up((size_t)L * E * w.ldT * 2);
  w.hi = reinterpret_cast<uint16_t*>(ws + (with_H ? up((size_t)N * L * E * sizeof(float)) : 0));
  w.lo = reinterpret_cast<uint16_t*>(reinterpret_cast<uint8_t*>(w.hi) + plane);
  w.gpart = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(w.hi) + (w.tc ? 2 * plane : 0));
  return w;
}

// keep_logits: leave the fp32 calibration logits H in the workspace (the
// input of ordermoe_transitions); the tensor-core path can skip writing them.
static int similarity_impl(const uint16_t* W_r, const uint16_t* X_cal, int L, int E, int d,
                           int64_t N, int k_freq, float* sim, int32_t* counts, void* workspace,
                           size_t workspace_bytes, bool keep_logits, cudaStream_t stream) {
  int rc0 = similarity_check(W_r, X_cal, L, E, d, N, k_freq, sim, counts, workspace, workspace_bytes,
                             ordermoe_similarity_workspace_bytes(L, E, N));
  if (rc0) return rc0;
  const SimLayout w = similarity_layout(workspace, L, E, N, true);
  float* H = w.H;
  uint16_t* hi = w.hi;
  uint16_t* lo = w.lo;
  float* gpart = w.gpart;
  const bool tc = w.tc;
  const int64_t ldT = w.ldT;
  const int nchunks = w.nchunks;
  OM_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * L * E, stream));
  if (tc) {
    // tensor-core path: logits with fused counts and hi/lo planes, then the Gram
    const int nsplit = sim_tc_nsplit(L, E, N);
    int rc = sim_tc_launch(X_cal, static_cast<int>(N), W_r, L, E, d, k_freq,
                           keep_logits ? H : nullptr, hi, lo, static_cast<int>(ldT), counts, gpart,
                           nsplit, false, stream);
    if (rc) return rc;
    gram_sim_kernel<<<dim3(L, (E * E + 255) / 256), 256, 0, stream>>>(gpart, nsplit, E, sim);
    OM_LAUNCHED("gram_sim_kernel");
    return ORDERMOE_OK;
  }
  int rc = logits_gemm_launch(X_cal, static_cast<int>(N), W_r, L * E, d, H, stream);
  if (rc) return rc;
  if ((rc = counts_launch(H, N, L, E, k_freq, (int64_t)L * E, E, counts, stream))) return rc;
  gram_kernel<<<dim3(L, nchunks), 256, 0, stream>>>(H, N, L, E, gpart);
  OM_LAUNCHED("gram_kernel");
  gram_sim_kernel<<<dim3(L, (E * E + 255) / 256), 256, 0, stream>>>(gpart, nchunks, E, sim);
  OM_LAUNCHED("gram_sim_kernel");
  return ORDERMOE_OK;
}

extern "C" int ordermoe_similarity(const uint16_t* W_r, const uint16_t* X_cal, int L, int E, int d,
                                   int64_t N, int k_freq, float* sim, int32_t* counts,
                                   void* workspace, size_t workspace_bytes,
                                   ordermoe_stream_t stream) {
  OM_TRACE();
  return similarity_impl(W_r, X_cal, L, E, d, N, k_freq, sim, counts, workspace, workspace_bytes,
                         true, stream);
}

extern "C" int ordermoe_similarity_no_logits(const uint16_t* W_r, const uint16_t* X_cal, int L,
                                             int E, int d, int64_t N, int k_freq, float* sim,
                                             int32_t* counts, void* workspace,
                                             size_t workspace_bytes, ordermoe_stream_t stream) {
  OM_TRACE();
  return similarity_impl(W_r, X_cal, L, E, d, N, k_freq, sim, counts, workspace, workspace_bytes,
                         false, stream);
}

extern "C" int ordermoe_expert_counts(const float* logits, int64_t N, int E, int k_freq,
                                      int32_t* counts, ordermoe_stream_t stream) {
  OM_TRACE();
  if (E <= 0 || E > ORDERMOE_MAX_EXPERTS || k_freq <= 0 || k_freq > E || N < 0)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "expert_counts: need 1 <= k_freq <= E <= 64");
  if (!counts || (N > 0 && !logits)) return fail(ORDERMOE_ERR_INVALID_ARG, "expert_counts: null pointer");
  OM_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * E, stream));
  if (N == 0) return ORDERMOE_OK;
  return counts_launch(logits, N, 1, E, k_freq, E, 0, counts, stream);
}

namespace om {

constexpr int kRepThreads = 512;
// Counting against sorting: 32 candidates 6.6 and 8.3 us, 128 12.2 and 11.2, 448
// 39 and 19 (a graph of calls, with the copies that reset their state).
constexpr int kRepCount = 64;
constexpr int kRepMaxCand = 16384;
constexpr int kRepMaxLayers = 1024;

// Redundant deployment for one server (blockIdx.x = m), Eqs. 32-35: the
// candidates (l, j) are deployed in the order (benefit desc, candidate id asc)
// while the group is uncovered and the replica fits. Benefits are positive
// fp64 values, so their bit patterns order like the values; non-positive and
// NaN benefits are never taken.
//
// Only candidates that can be taken are ordered. The server's load b_m never
// falls (p > 0, and rounding is monotone) and its covered groups stay covered,
// so a candidate that fails against the initial state fails always. Of two
// candidates of one group, the later is never taken when its p is at least the
// earlier's: when the earlier was taken the group is covered, and when it did
// not fit the later does not either. Up to kRepCount candidates are ordered by
// counting those before each, more by a bitonic sort in shared memory. One warp
// then tests 32 at a time against the current state and takes the first that
// passes: every candidate it passes over failed under the same state it would
// have met one at a time.
//
// Bound: latency of one block a server (barriers of the sort, fp64 chain of the
// takes). In a graph of calls with the two copies that reset its state: layers x
// experts, groups a layer, servers, all candidates in one sort with a window read
// again after each take against this: 24 x 64, 8 groups, 8 servers with room for as
// many again 54.1 and 7.9 us; 32 x 8, 4, 4 24.8 and 17.1; 24 x 64, 16, 8 91.3 and
// 40.5; every expert its own group, 8 x 64 on 32 servers 22.1 and 20.2. (Candidates
// compared with the whole layer instead of their group's, and up to 512 of them
// ordered by counting those before each: 65.5 and 48.8 us for the last two.)
__global__ void __launch_bounds__(kRepThreads) replicate_kernel(
    const int32_t* __restrict__ group, const double* __restrict__ importance,
    const double* __restrict__ p, const double* __restrict__ C, const double* __restrict__ pi,
    int L, int E, int M, int Np, uint8_t* __restrict__ placement, double* __restrict__ used,
    int32_t* __restrict__ replicas) {
  extern __shared__ __align__(16) unsigned char s_rep[];
  unsigned long long* key = reinterpret_cast<unsigned long long*>(s_rep);
  unsigned long long* cov = key + Np;  // [L]: bit g = group g covered (Eq. 32)
  uint32_t* cid = reinterpret_cast<uint32_t*>(cov + L);
  __shared__ int n_cand;
  __shared__ unsigned long long mates[kRepThreads / 32][64];  // a layer's candidates by group
  const int m = blockIdx.x;
  const int t = threadIdx.x;
  const int lane = t & 31;
  const unsigned full = 0xffffffffu;
  const int N = L * E;
  if (t == 0) n_cand = 0;
  for (int l = t; l < L; l += kRepThreads) cov[l] = 0ull;
  __syncthreads();
  for (int i = t; i < N; i += kRepThreads) {
    const int g = group[i], l = i / E;
    const bool here = placement[((size_t)l * M + m) * E + (i - l * E)] != 0;
    if (here && g >= 0 && g < E) atomicOr(&cov[l], 1ull << g);
  }
  const double pim = pi[m];
  const double b0 = used[m], cap = C[m];
  __syncthreads();
  // benefits of the candidates that pass the initial state (0: none), their groups
  for (int i = t; i < N; i += kRepThreads) {
    unsigned long long k = 0;
    const int g = group[i];
    const double pj = p[i];
    if (g < 0 || g >= E) {
      if (m == 0) report(&g_err_sim, ORDERMOE_DEV_BAD_INDEX, i);
    } else if (!(pj > 0.0)) {
      if (m == 0) report(&g_err_sim, ORDERMOE_DEV_BAD_VALUE, i);
    } else if (!((cov[i / E] >> g) & 1ull) && __dadd_rn(b0, pj) <= cap) {  // Eqs. 32, 35
      const double ben = __ddiv_rn(__dmul_rn(pim, importance[i]), pj);     // Eq. 33, y = 0
      if (ben > 0.0) k = static_cast<unsigned long long>(__double_as_longlong(ben));
    }
    key[i] = k;
    cid[i] = static_cast<uint32_t>(g);
  }
  __syncthreads();
  // kept: not after another of its group that asks for no more memory. A warp a
  // layer, an expert against the candidates of its own group
  for (int l = t >> 5; l < L; l += kRepThreads / 32) {
    unsigned long long* const mate = mates[t >> 5];
    const unsigned long long own[2] = {lane < E ? key[l * E + lane] : 0ull,
                                       lane + 32 < E ? key[l * E + lane + 32] : 0ull};
    if (!__any_sync(full, (own[0] | own[1]) != 0)) continue;
    mate[lane] = mate[lane + 32] = 0ull;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (own[h] != 0) atomicOr(&mate[cid[l * E + lane + 32 * h]], 1ull << (lane + 32 * h));
    __syncwarp();
    uint32_t drop = 0;  // of this lane's two experts
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = lane + 32 * h, i = l * E + e;
      const unsigned long long k = own[h];
      if (k == 0) continue;
      const double pj = p[i];
      for (unsigned long long b = mate[cid[i]] & ~(1ull << e); b; b &= b - 1) {
        const int o = l * E + __ffsll(static_cast<long long>(b)) - 1;
        if ((key[o] > k || (key[o] == k && o < i)) && p[o] <= pj) {
          drop |= 1u << h;
          break;
        }
      }
    }
    __syncwarp();  // the layer's keys are read
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if ((drop >> h) & 1u) key[l * E + lane + 32 * h] = 0ull;
  }
  __syncthreads();
  // their keys and ids moved to the front, kRepThreads candidates at a time (a
  // round writes only where it and the rounds before it have been read)
  for (int r = 0; r * kRepThreads < N; ++r) {
    const int i = r * kRepThreads + t;
    const unsigned long long k = i < N ? key[i] : 0ull;
    const bool mine = k != 0;
    const unsigned bal = __ballot_sync(full, mine);
    int at = 0;
    if (lane == 0 && bal != 0u) at = atomicAdd(&n_cand, __popc(bal));
    at = __shfl_sync(full, at, 0) + __popc(bal & ((1u << lane) - 1u));
    __syncthreads();
    if (mine) {
      key[at] = k;
      cid[at] = static_cast<uint32_t>(i);
    }
    __syncthreads();
  }
  const int nc = n_cand;
  if (nc > kRepCount) {
    int ns = 1;
    while (ns < nc) ns <<= 1;  // <= Np
    for (int i = nc + t; i < ns; i += kRepThreads) {
      key[i] = 0ull;
      cid[i] = 0xFFFFFFFFu;
    }
    __syncthreads();
    // bitonic sort into (key desc, cid asc)
    for (int size = 2; size <= ns; size <<= 1) {
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int i = t; i < ns; i += kRepThreads) {
          const int o = i ^ stride;
          if (o > i) {
            const unsigned long long ki = key[i], ko = key[o];
            const uint32_t ci = cid[i], co = cid[o];
            const bool o_first = ko > ki || (ko == ki && co < ci);
            const bool i_first = ki > ko || (ki == ko && ci < co);
            if ((i & size) == 0 ? o_first : i_first) {
              key[i] = ko; key[o] = ki;
              cid[i] = co; cid[o] = ci;
            }
          }
        }
        __syncthreads();
      }
    }
  }
  // each sorted slot holds (l, g, j) and the bits of p_{l,j}
  if (nc <= kRepCount) {
    int rank = 0, i = 0;
    if (t < nc) {
      const unsigned long long k = key[t];
      i = static_cast<int>(cid[t]);
#pragma unroll 4
      for (int o = 0; o < nc; ++o) {
        const unsigned long long ko = key[o];
        rank += ko > k || (ko == k && cid[o] < static_cast<uint32_t>(i)) ? 1 : 0;
      }
    }
    __syncthreads();
    if (t < nc) {
      const int l = i / E;
      cid[rank] = (static_cast<uint32_t>(l) << 12) | (static_cast<uint32_t>(group[i]) << 6) |
                  static_cast<uint32_t>(i - l * E);
      key[rank] = static_cast<unsigned long long>(__double_as_longlong(p[i]));
    }
  } else {
    for (int s = t; s < nc; s += kRepThreads) {
      const int i = static_cast<int>(cid[s]), l = i / E;
      cid[s] = (static_cast<uint32_t>(l) << 12) | (static_cast<uint32_t>(group[i]) << 6) |
               static_cast<uint32_t>(i - l * E);
      key[s] = static_cast<unsigned long long>(__double_as_longlong(p[i]));
    }
  }
  __syncthreads();
  if (t < 32) {
    double b = b0;
    int count = 0;
    for (int base = 0; base < nc; base += 32) {
      const int s = base + lane;
      const uint32_t rec = s < nc ? cid[s] : 0u;
      const double pj = s < nc ? __longlong_as_double(static_cast<long long>(key[s])) : 0.0;
      const uint32_t lg = rec >> 6;  // layer and group
      bool open = s < nc && !((cov[lg >> 6] >> (lg & 63u)) & 1ull);  // B = 0 once the group is local
      __syncwarp();  // read before a lane below sets a bit
      for (;;) {
        const double b1 = __dadd_rn(b, pj);
        const unsigned bal = __ballot_sync(full, open && b1 <= cap);  // Eq. 35
        if (bal == 0) break;
        const int w = __ffs(bal) - 1;
        b = __shfl_sync(full, b1, w);
        const uint32_t taken = __shfl_sync(full, lg, w);
        open = open && lane > w && lg != taken;
        if (lane == w) {
          placement[((size_t)(lg >> 6) * M + m) * E + static_cast<int>(rec & 63u)] = 1;
          cov[lg >> 6] |= 1ull << (lg & 63u);
        }
        ++count;
        __syncwarp();  // the next take may set a bit of the same word, and the next 32 read it
      }
    }
    if (lane == 0) {
      used[m] = b;
      replicas[m] = count;
    }
  }
}

// Eq. 32 for one layer (blockIdx.x = l): thread m ORs its server's groups.
__global__ void __launch_bounds__(32) coverage_kernel(const int32_t* __restrict__ group,
                                                      const uint8_t* __restrict__ placement, int L,
                                                      int E, int M, uint8_t* __restrict__ cover,
                                                      int32_t* __restrict__ covered) {
  const int l = blockIdx.x;
  const int m = threadIdx.x;
  // the layer's groups, checked once (-1: out of range, reported)
  __shared__ int gsh[64];
  for (int j = m; j < E; j += 32) {
    int g = group[(size_t)l * E + j];
    if (g < 0 || g >= E) {
      report(&g_err_sim, ORDERMOE_DEV_BAD_INDEX, l * E + j);
      g = -1;
    }
    gsh[j] = g;
  }
  __syncwarp();
  // server m's row of the layer's placement: 16-byte loads where it allows,
  // all issued before they are used
  unsigned long long bits = 0;
  if (m < M) {
    const uint8_t* row = placement + ((size_t)l * M + m) * E;
    if ((E & 15) == 0 && (reinterpret_cast<uintptr_t>(row) & 15u) == 0) {
      uint4 v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < E / 16) v[c] = reinterpret_cast<const uint4*>(row)[c];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (c >= E / 16) break;
        const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const int g = gsh[c * 16 + q];
          if (((w[q >> 2] >> (8 * (q & 3))) & 0xFFu) != 0u && g >= 0) bits |= 1ull << g;
        }
      }
    } else {
#pragma unroll 16
      for (int j = 0; j < E; ++j) {
        const int g = gsh[j];
        if (row[j] && g >= 0) bits |= 1ull << g;
      }
    }
  }
  if (m < M && cover != nullptr)
    for (int g = 0; g < E; ++g) cover[((size_t)l * M + m) * E + g] = (bits >> g) & 1ull;
  int n = __popcll(bits);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if (m == 0 && covered != nullptr) covered[l] = n;
}

}  // namespace om

extern "C" size_t ordermoe_place_workspace_bytes(int L, int E) {
  if (L <= 0 || E <= 0 || E > ORDERMOE_MAX_EXPERTS) return 0;
  return ((size_t)L * E * sizeof(int32_t) + 255) & ~size_t(255);
}

static cudaError_t place_attr() {
  return cudaFuncSetAttribute(place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kPlaceSmemMax));
}

// The placement of grouped layers l0 .. l1 - 1 in ranges of at most 512 experts
// (a range's tables hold its servers' states).
static cudaError_t place_launch(const int32_t* group, const int32_t* porder, int L, int E, int M, int l0,
                                int l1, const PlaceParams& pp, const double* p, const double* C,
                                uint8_t* placement, double* used, int32_t* status, cudaStream_t stream) {
  const int part = kPlaceRange / E;
  for (int a = l0; a < l1; a += part) {
    const int b = a + part < l1 ? a + part : l1;
    place_kernel<<<1, kPlaceThreads, place_smem(M, (b - a) * E), stream>>>(
        group, porder, L, E, M, a, b, a == 0 ? 1 : 0, pp, p, C, placement, used, status);
  }
  return cudaGetLastError();
}

extern "C" int ordermoe_place(const float* sim, const int32_t* counts, int L, int E, int M,
                              double theta_min, double theta_max, double theta_single,
                              double alpha_f, double alpha_r, double lambda1, double lambda2,
                              const double* p, const double* C, int32_t* group, int32_t* n_groups,
                              float* theta, double* importance, uint8_t* placement, double* used,
                              int32_t* status, void* workspace, size_t workspace_bytes,
                              ordermoe_stream_t stream) {
  OM_TRACE();
  if (L <= 0 || E <= 0 || E > ORDERMOE_MAX_EXPERTS || M <= 0 || M > ORDERMOE_MAX_SERVERS)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "place: need L >= 1, 1 <= E <= 64, 1 <= M <= 32");
  if (!sim || !counts || !p || !C || !group || !n_groups || !theta || !placement || !used || !status)
    return fail(ORDERMOE_ERR_INVALID_ARG, "place: null pointer");
  if (!workspace || workspace_bytes < ordermoe_place_workspace_bytes(L, E))
    return fail(ORDERMOE_ERR_INVALID_ARG, "place: workspace missing or too small");
  int32_t* porder_scratch = static_cast<int32_t*>(workspace);
  PlaceParams pp{theta_min, theta_max, theta_single, alpha_f, alpha_r, lambda1, lambda2};
  group_kernel<<<L, group_slice_threads(E), 0, stream>>>(sim, counts, L, E, 0, pp, p, group, n_groups, theta, importance,
                                     porder_scratch);
  OM_LAUNCHED("group_kernel");
  static PerDevice attr;
  const cudaError_t ae =
      static_cast<cudaError_t>(per_device(attr, [] { return static_cast<int>(place_attr()); }));
  if (ae != cudaSuccess) return cuda_fail(ae, "cudaFuncSetAttribute(place_kernel)");
  const cudaError_t e = place_launch(group, porder_scratch, L, E, M, 0, L, pp, p, C, placement, used, status, stream);
  if (e != cudaSuccess) return cuda_fail(e, "place_kernel");
  return ORDERMOE_OK;
}

static int transitions_launch(const char* who, const float* logits, int64_t N, int L, int E,
                              int k_freq, int64_t sn, int64_t sl, int32_t* counts, float* P,
                              cudaStream_t stream) {
  if (L < 2 || E <= 0 || E > ORDERMOE_MAX_EXPERTS || k_freq <= 0 || k_freq > E || N < 0)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "%s: need L >= 2, 1 <= k_freq <= E <= 64", who);
  if (!counts || !P || (N > 0 && !logits)) return fail(ORDERMOE_ERR_INVALID_ARG, "%s: null pointer", who);
  OM_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * (size_t)(L - 1) * E * E, stream));
  if (N > 0) {
    static PerDevice attr;
    const cudaError_t ae = static_cast<cudaError_t>(per_device(attr, [] {
      const int most = static_cast<int>(topk_tile_bytes(64) + sizeof(int) * 64 * 64);
      cudaError_t e = cudaFuncSetAttribute(transitions_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(transitions_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(transitions_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(transitions_kernel<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(transitions_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      return static_cast<int>(e);
    }));
    if (ae != cudaSuccess) return cuda_fail(ae, "cudaFuncSetAttribute(transitions_kernel)");
    const int64_t tiles = (N + kTopkTokens - 1) / kTopkTokens;
    if (tiles > INT32_MAX) return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "%s: too many tokens", who);
    // tiles a block counts before it adds its E * E counts to memory, and layer
    // pairs it walks: as many as leave two blocks an SM
    int64_t tb = tiles / num_sms();
    if (tb < 1) tb = 1;
    if (tb > kTransTiles) tb = kTransTiles;
    const int64_t cols = (tiles + tb - 1) / tb;
    int64_t ranges = (2 * num_sms() + cols - 1) / cols;
    if (ranges > L - 1) ranges = L - 1;
    int per = static_cast<int>((L - 1 + ranges - 1) / ranges);
    if ((L - 1 + per - 1) / per > 65535) per = (L - 1 + 65534) / 65535;  // the grid's y limit
    const dim3 grid(static_cast<unsigned>(cols), (L - 1 + per - 1) / per);
    const size_t smem = topk_tile_bytes(E) + sizeof(int) * E * E;
    switch (topk_list_len(k_freq)) {
      case 2: transitions_kernel<2><<<grid, kTopkTokens, smem, stream>>>(logits, N, L, E, k_freq, sn, sl, per, static_cast<int>(tb), counts); break;
      case 4: transitions_kernel<4><<<grid, kTopkTokens, smem, stream>>>(logits, N, L, E, k_freq, sn, sl, per, static_cast<int>(tb), counts); break;
      case 6: transitions_kernel<6><<<grid, kTopkTokens, smem, stream>>>(logits, N, L, E, k_freq, sn, sl, per, static_cast<int>(tb), counts); break;
      case 8: transitions_kernel<8><<<grid, kTopkTokens, smem, stream>>>(logits, N, L, E, k_freq, sn, sl, per, static_cast<int>(tb), counts); break;
      default: transitions_kernel<0><<<grid, kTopkTokens, smem, stream>>>(logits, N, L, E, k_freq, sn, sl, per, static_cast<int>(tb), counts);
    }
    OM_LAUNCHED("transitions_kernel");
  }
  const int rows = (L - 1) * E;
  transitions_finish_kernel<<<(rows + 3) / 4, 128, 0, stream>>>(counts, rows, E, P);
  OM_LAUNCHED("transitions_finish_kernel");
  return ORDERMOE_OK;
}

extern "C" int ordermoe_transitions(const float* logits, int64_t N, int L, int E, int k_freq,
                                    int32_t* counts, float* P, ordermoe_stream_t stream) {
  OM_TRACE();
  return transitions_launch("transitions", logits, N, L, E, k_freq, (int64_t)L * E, E, counts, P,
                            stream);
}

extern "C" int ordermoe_transitions_strided(const float* logits, int64_t N, int L, int E,
                                            int k_freq, int64_t token_stride, int64_t layer_stride,
                                            int32_t* counts, float* P, ordermoe_stream_t stream) {
  OM_TRACE();
  if (token_stride < E || layer_stride < E)
    return fail(ORDERMOE_ERR_INVALID_ARG, "transitions_strided: strides must be >= E");
  return transitions_launch("transitions_strided", logits, N, L, E, k_freq, token_stride,
                            layer_stride, counts, P, stream);
}

extern "C" int ordermoe_replicate(const int32_t* group, const double* importance, const double* p,
                                  const double* C, const double* pi, int L, int E, int M,
                                  uint8_t* placement, double* used, int32_t* replicas,
                                  ordermoe_stream_t stream) {
  OM_TRACE();
  if (L <= 0 || L > kRepMaxLayers || E <= 0 || E > ORDERMOE_MAX_EXPERTS || M <= 0 ||
      M > ORDERMOE_MAX_SERVERS || (long long)L * E > kRepMaxCand)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE,
                "replicate: need 1 <= L <= 1024, 1 <= E <= 64, L * E <= 16384, 1 <= M <= 32");
  if (!group || !importance || !p || !C || !pi || !placement || !used || !replicas)
    return fail(ORDERMOE_ERR_INVALID_ARG, "replicate: null pointer");
  int Np = 1;
  while (Np < L * E) Np <<= 1;
  const size_t smem = (size_t)Np * (sizeof(unsigned long long) + sizeof(uint32_t)) +
                      (size_t)L * sizeof(unsigned long long);
  // once per device, for the largest sort (no attribute call per launch, so
  // the call can be captured into a CUDA graph)
  static PerDevice attr;
  const cudaError_t ae = static_cast<cudaError_t>(per_device(attr, [] {
    const size_t most = (size_t)kRepMaxCand * (sizeof(unsigned long long) + sizeof(uint32_t)) +
                        (size_t)kRepMaxLayers * sizeof(unsigned long long);
    return static_cast<int>(cudaFuncSetAttribute(
        replicate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
  }));
  if (ae != cudaSuccess) return cuda_fail(ae, "cudaFuncSetAttribute(replicate_kernel)");
  replicate_kernel<<<M, kRepThreads, smem, stream>>>(group, importance, p, C, pi, L, E, M, Np,
                                                     placement, used, replicas);
  OM_LAUNCHED("replicate_kernel");
  return ORDERMOE_OK;
}

extern "C" int ordermoe_coverage(const int32_t* group, const uint8_t* placement, int L, int E,
                                 int M, uint8_t* cover, int32_t* covered,
                                 ordermoe_stream_t stream) {
  OM_TRACE();
  if (L <= 0 || E <= 0 || E > ORDERMOE_MAX_EXPERTS || M <= 0 || M > ORDERMOE_MAX_SERVERS)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "coverage: need L >= 1, 1 <= E <= 64, 1 <= M <= 32");
  if (!group || !placement) return fail(ORDERMOE_ERR_INVALID_ARG, "coverage: null pointer");
  coverage_kernel<<<L, 32, 0, stream>>>(group, placement, L, E, M, cover, covered);
  OM_LAUNCHED("coverage_kernel");
  return ORDERMOE_OK;
}

extern "C" int ordermoe_selftest_div_rn(const double* a, const double* b, double* out, int64_t n,
                                        ordermoe_stream_t stream) {
  OM_TRACE();
  if (n < 0) return fail(ORDERMOE_ERR_INVALID_ARG, "selftest_div_rn: n < 0");
  if (n == 0) return ORDERMOE_OK;
  if (!a || !b || !out) return fail(ORDERMOE_ERR_INVALID_ARG, "selftest_div_rn: null pointer");
  int64_t blocks = (n + 255) / 256;
  if (blocks > num_sms() * 8) blocks = num_sms() * 8;
  div_selftest_kernel<<<static_cast<int>(blocks), 256, 0, stream>>>(a, b, out, n);
  OM_LAUNCHED("div_selftest_kernel");
  return ORDERMOE_OK;
}

// ----------------------------------------------------------------------------
// The whole offline plan in one call (Alg. 1): similarity (Eqs. 3-5), grouping
// (Eqs. 6, 24-28), mandatory placement (Eqs. 29-31), redundant deployment
// (Eqs. 32-35) and coverage (Eq. 32). On the tensor-core path the layers go in
// blocks of 512 logit columns: the caller's stream runs a block's logits GEMM,
// Gram and similarities, and a side stream, behind an event, runs that
// block's grouping and placement while the next block's GEMM runs. The
// placement carries b_m from block to block in `used`; its layers stay in
// order because the side stream runs the blocks in order. The results are
// those of ordermoe_similarity_no_logits, ordermoe_place, ordermoe_replicate
// and ordermoe_coverage called one after the other.
namespace om {

int sim_tc_part_layers(int E);

// One side stream and its events per device, shared by every call: a call
// holds `mu` while it enqueues, so calls from several host threads cannot
// interleave their event records (a stream wait takes the event as it was
// when the wait was enqueued).
struct PlanSync {
  std::mutex mu;
  cudaStream_t side;
  cudaEvent_t ev[4];
};
static PlanSync g_plan_sync[64];
static PerDevice g_plan_sync_once;

static int plan_sync(PlanSync** out) {
  int dev = 0;
  OM_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "plan: device index above 63");
  const int e = per_device(g_plan_sync_once, [dev] {
    PlanSync& ps = g_plan_sync[dev];
    cudaError_t err = cudaFuncSetAttribute(group_place_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           static_cast<int>(kPlaceSmemMax));
    if (err == cudaSuccess) err = place_attr();
    if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&ps.side, cudaStreamNonBlocking);
    for (int i = 0; i < 4 && err == cudaSuccess; ++i)
      err = cudaEventCreateWithFlags(&ps.ev[i], cudaEventDisableTiming);
    return static_cast<int>(err);
  });
  if (e != cudaSuccess) return cuda_fail(static_cast<cudaError_t>(e), "plan: side stream and events");
  *out = &g_plan_sync[dev];
  return ORDERMOE_OK;
}

static int launched(const char* what) {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ORDERMOE_OK : cuda_fail(e, what);
}

}  // namespace om

// The similarity part of the plan's workspace: without H on the tensor-core
// path (the plan keeps no logits), the whole similarity workspace otherwise.
static size_t plan_sim_bytes(int L, int E, int64_t N) {
  return sim_ws_bytes(L, E, N, !sim_tc_supported(L, E));
}

extern "C" size_t ordermoe_plan_workspace_bytes(int L, int E, int64_t N) {
  const size_t a = plan_sim_bytes(L, E, N);  // a multiple of 256
  const size_t b = ordermoe_place_workspace_bytes(L, E);
  return (a == 0 || b == 0) ? 0 : a + b;
}

extern "C" int ordermoe_plan(const uint16_t* W_r, const uint16_t* X_cal, int L, int E, int d,
                             int64_t N, int k_freq, int M, double theta_min, double theta_max,
                             double theta_single, double alpha_f, double alpha_r, double lambda1,
                             double lambda2, const double* p, const double* C, const double* pi,
                             float* sim, int32_t* counts, int32_t* group, int32_t* n_groups,
                             float* theta, double* importance, uint8_t* placement, double* used,
                             int32_t* status, int32_t* replicas, uint8_t* cover, int32_t* covered,
                             void* workspace, size_t workspace_bytes, ordermoe_stream_t stream) {
  OM_TRACE();
  const size_t sim_ws = plan_sim_bytes(L, E, N);
  int rc = similarity_check(W_r, X_cal, L, E, d, N, k_freq, sim, counts, workspace, sim_ws, sim_ws);
  if (rc) return rc;
  if (M <= 0 || M > ORDERMOE_MAX_SERVERS || L > kRepMaxLayers || (long long)L * E > kRepMaxCand)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE,
                "plan: need 1 <= M <= 32, L <= 1024 and L * E <= 16384");
  if (!p || !C || !pi || !group || !n_groups || !theta || !importance || !placement || !used ||
      !status || !replicas)
    return fail(ORDERMOE_ERR_INVALID_ARG, "plan: null pointer");
  if (workspace_bytes < ordermoe_plan_workspace_bytes(L, E, N))
    return fail(ORDERMOE_ERR_INVALID_ARG, "plan: workspace too small");
  int32_t* porder = reinterpret_cast<int32_t*>(static_cast<uint8_t*>(workspace) + sim_ws);
  const size_t porder_bytes = workspace_bytes - sim_ws;
  cudaStream_t S = static_cast<cudaStream_t>(stream);
  const SimLayout w = similarity_layout(workspace, L, E, N, !sim_tc_supported(L, E));
  if (!w.tc) {  // the CUDA-core similarity needs every layer's logits at once
    rc = similarity_impl(W_r, X_cal, L, E, d, N, k_freq, sim, counts, workspace, sim_ws, false, S);
    if (!rc)
      rc = ordermoe_place(sim, counts, L, E, M, theta_min, theta_max, theta_single, alpha_f, alpha_r,
                          lambda1, lambda2, p, C, group, n_groups, theta, importance, placement,
                          used, status, porder, porder_bytes, stream);
  } else {
    PlanSync* ps = nullptr;
    if ((rc = plan_sync(&ps))) return rc;
    std::lock_guard<std::mutex> hold(ps->mu);
    OM_CUDA(cudaMemsetAsync(counts, 0, sizeof(int32_t) * L * E, S));
    OM_CUDA(cudaEventRecord(ps->ev[0], S));
    OM_CUDA(cudaStreamWaitEvent(ps->side, ps->ev[0], 0));
    const PlaceParams pp{theta_min, theta_max, theta_single, alpha_f, alpha_r, lambda1, lambda2};
    const int part = sim_tc_part_layers(E);
    const int nsplit = sim_tc_nsplit(L, E, N);
    for (int l0 = 0, k = 0; l0 < L && !rc; ++k) {
      const int lp = L - l0 < part ? L - l0 : part;
      const size_t rows = (size_t)l0 * E;
      float* gpart = w.gpart + (size_t)l0 * nsplit * 4096;
      rc = sim_tc_launch(X_cal, static_cast<int>(N), W_r + rows * d, lp, E, d, k_freq, nullptr,
                         w.hi + rows * w.ldT, w.lo + rows * w.ldT, static_cast<int>(w.ldT),
                         counts + rows, gpart, nsplit, true, S);
      if (rc) break;
      gram_sim_kernel<<<dim3(lp, (E * E + 255) / 256), 256, 0, S>>>(gpart, nsplit, E, sim + rows * E);
      if ((rc = launched("gram_sim_kernel"))) break;
      cudaEvent_t ev = ps->ev[1 + (k & 1)];
      cudaError_t e = cudaEventRecord(ev, S);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(ps->side, ev, 0);
      if (e != cudaSuccess) {
        rc = cuda_fail(e, "plan: block event");
        break;
      }
      if (l0 + lp < L) {
        group_place_kernel<<<1, kGroupThreads + 32, group_place_smem(E, M, lp * E), ps->side>>>(
            sim, counts, L, E, M, l0, l0 + lp, l0 == 0 ? 1 : 0, pp, p, C, group, n_groups, theta,
            importance, porder, placement, used, status);
        if ((rc = launched("group_place_kernel"))) break;
      } else {
        // no GEMM runs beside the last block: a block a layer groups it. (Cut in
        // two halves, so that less is left to group and place, the last block
        // streams X_cal once more: 1613 against 1569 us for the whole plan.)
        group_kernel<<<lp, group_slice_threads(E), 0, ps->side>>>(
            sim, counts, L, E, l0, pp, p, group, n_groups, theta, importance, porder);
        if ((rc = launched("group_kernel"))) break;
        const cudaError_t pe = place_launch(group, porder, L, E, M, l0, L, pp, p, C, placement, used, status, ps->side);
        if (pe != cudaSuccess) {
          rc = cuda_fail(pe, "place_kernel");
          break;
        }
      }
      l0 += lp;
    }
    // every exit after the fork joins the side stream back into the caller's
    cudaError_t e = cudaEventRecord(ps->ev[3], ps->side);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(S, ps->ev[3], 0);
    if (!rc && e != cudaSuccess) rc = cuda_fail(e, "plan: join");
  }
  if (!rc)
    rc = ordermoe_replicate(group, importance, p, C, pi, L, E, M, placement, used, replicas, stream);
  if (!rc) rc = ordermoe_coverage(group, placement, L, E, M, cover, covered, stream);
  return rc;
}
