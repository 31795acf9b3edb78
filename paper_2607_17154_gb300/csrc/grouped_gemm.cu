// Grouped SwiGLU expert FFN on sm_103a tensor cores (tcgen05 + TMEM + TMA).
//
// ffn_gemm_kernel: persistent warp-specialised kernels over the
// expert-contiguous rows of ordermoe_dispatch, with the per-expert row ranges
// read on the device: the weights on the MMA's M side, on CTA pairs for large
// batches and on single CTAs for small ones (its own section below).
//   gate/up: H = bf16(silu(X W1_e^T) * (X W3_e^T)), fused in the epilogue;
//   down:    Y = bf16(H W2_e^T).
// logits_gemm_kernel: the router logits of the offline similarity where the
// tensor-core path of sim_gemm.cu does not apply. Tile = 128 rows x 256
// accumulator columns, K step 64 (one 128-byte swizzled TMA box per operand
// row), 4-stage shared-memory ring, two TMEM accumulators (2 x 256 columns =
// all 512) so the epilogue of one tile overlaps the main loop of the next.
// Warp roles: warp 0 = TMA producer, warp 1 = MMA issuer and TMEM owner, the
// others = epilogue (warp w reads TMEM lanes 32 (w % 4) ...).
// Every wait is bounded (globaltimer); a wait that runs out reports
// ORDERMOE_DEV_WAIT_TIMEOUT, makes the other roles stop, drains the copies
// and MMAs in flight (bounded too), frees TMEM and returns.
#include <initializer_list>
#include <mutex>

#include "common.cuh"

namespace om {

static __device__ unsigned long long g_err_gemm = 0;

int read_clear_err_gemm(unsigned long long* out) {
  unsigned long long zero = 0;
  OM_CUDA(cudaMemcpyFromSymbol(out, g_err_gemm, sizeof(*out)));
  OM_CUDA(cudaMemcpyToSymbol(g_err_gemm, &zero, sizeof(zero)));
  return ORDERMOE_OK;
}

namespace gg {

constexpr int BM = 128;
constexpr int BN = 256;  // accumulator columns per tile
constexpr int BK = 64;   // bf16 elements = 128 bytes
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;
constexpr int B_BYTES = BN * BK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int THREADS = 192;
constexpr int TMEM_COLS = 512;

struct Smem {
  uint64_t full[STAGES];
  uint64_t empty[STAGES];
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
  int zero;
};
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + static_cast<int>(sizeof(Smem));

enum { GATEUP = 0, DOWN = 1 };

struct Args {
  const int32_t* offsets;  // FFN: [E+1] row ranges (0 <= ... <= rows)
  int rows;
  int n_valid;       // LOGITS: number of valid output columns
  float* out_f32;    // LOGITS: H [rows][n_valid] fp32
  int E;
  int K;             // reduction length
  int n_tiles;       // N slices per expert
  int b_rows;        // weight rows per expert (d_ff or d); logits: columns of a slice
  uint16_t* out;     // H [R][d_ff] or Y [R][d]
  int ldo;           // row length of out
  uint64_t limit_ns; // bounded-wait limit
  int fast_div;      // gate/up: SwiGLU's quotient by the fast reciprocal
};

struct Tile {
  int e, m0, m_end, n;
};

// The experts' row ranges and first row tiles (of bm rows) into s.offs and
// s.mt_start, by one warp: two experts a lane, all loads in flight together.
// (One thread reading the offsets in turn took 3.4 us of a 64-expert launch:
// gate/up of 128 tokens, top-6, d 2048, d_ff 1408: 124.3 -> 120.9 us.)
// No tiles, and a report, when the offsets do not run 0 <= ... <= rows.
template <class S>
__device__ __forceinline__ void load_row_tiles(S& s, const Args& args, int bm, int lane) {
  const int E = args.E;
  auto off = [&](int e) { return args.offsets[min(e, E)]; };
  const int o0 = off(lane), o1 = off(lane + 32), o2 = off(64);
  const int top = __shfl_sync(0xffffffffu, o1, 0);
  int n0 = __shfl_down_sync(0xffffffffu, o0, 1), n1 = __shfl_down_sync(0xffffffffu, o1, 1);
  if (lane == 31) {
    n0 = top;
    n1 = o2;
  }
  const bool bad = __any_sync(0xffffffffu, n0 < o0 || n1 < o1 || (lane == 0 && o0 != 0) || o2 > args.rows);
  const int t0 = (n0 - o0 + bm - 1) / bm, t1 = (n1 - o1 + bm - 1) / bm;
  int i0 = t0, i1 = t1;  // inclusive sums of experts 0-31 and 32-63
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u0 = __shfl_up_sync(0xffffffffu, i0, o), u1 = __shfl_up_sync(0xffffffffu, i1, o);
    if (lane >= o) {
      i0 += u0;
      i1 += u1;
    }
  }
  i1 += __shfl_sync(0xffffffffu, i0, 31);
  if (bad) i0 = i1 = 0;
  const int most = __reduce_max_sync(0xffffffffu, max(n0 - o0, n1 - o1));
  if (lane == 0) s.max_rows = bad ? 0 : min(most, bm);
  if (lane <= E) {
    s.offs[lane] = o0;
    s.mt_start[lane] = bad ? 0 : i0 - t0;
  }
  if (lane + 32 <= E) {
    s.offs[lane + 32] = o1;
    s.mt_start[lane + 32] = bad ? 0 : i1 - t1;
  }
  if (lane == 31 && E == 64) {
    s.offs[64] = o2;
    s.mt_start[64] = i1;
  }
  if (bad && lane == 0 && blockIdx.x == 0) report(&g_err_gemm, ORDERMOE_DEV_BAD_INDEX, -2);
}

// A tile of the logits: all column slices of a row tile back to back, so that the
// rows are read once from HBM (the stacked router rows stay in L2).
__device__ __forceinline__ Tile decode(int tile, const Args& args) {
  const int mt = tile / args.n_tiles;
  return Tile{0, mt * BM, args.rows, tile - mt * args.n_tiles};
}

__global__ void __launch_bounds__(THREADS, 1)
    logits_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB0,
                       Args args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  Smem& s = *reinterpret_cast<Smem*>(tiles + STAGES * STAGE_BYTES);
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  // launched with launch_pdl: barriers, TMEM and tensor-map prefetches are set
  // up while the previous kernel finishes; global memory only after pdl_wait
  pdl_trigger();
  if (warp == 0 && lane == 0) {
    tma_prefetch_map(&mapA);
    tma_prefetch_map(&mapB0);
  }

  if (tid == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s.tfull[i], 1);
      mbar_init(&s.tempty[i], 128);
    }
    mbar_init(&s.drain, 1);
    s.abort = 0;
    s.zero = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&s.tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();  // every thread: the previous kernel's outputs are visible
  const uint32_t tmem_base = s.tmem_base;
  const int total = (args.rows + BM - 1) / BM * args.n_tiles;
  const int kblocks = args.K / BK;
  volatile int* abort = &s.abort;

  // per-role bookkeeping for the drain after an abort
  uint32_t issued_mask = 0, last_phase_bits = 0;
  bool mma_issued = false;
  bool leader = false;  // the MMA warp's issuing lane

  const int width = args.b_rows;  // columns of a slice, its weight rows in two boxes
  const int box_bytes = width / 2 * BK * 2;
  if (warp == 0) {
    // producer and MMA issuer walk the stages converged, one elected lane issues
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
      const Tile t = decode(tile, args);
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(&s.empty[stage], phase ^ 1u, args.limit_ns, abort))) {
          if (issuer && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 1);
          *abort = 1;
          ok = false;
          break;
        }
        uint8_t* sa = tiles + stage * STAGE_BYTES;
        uint8_t* sb = sa + A_BYTES;
        if (issuer) {
          mbar_arrive_expect_tx(&s.full[stage], A_BYTES + 2 * box_bytes);
          tma_load_2d(sa, &mapA, &s.full[stage], kb * BK, t.m0);
          tma_load_2d(sb, &mapB0, &s.full[stage], kb * BK, t.n * width);
          tma_load_2d(sb + box_bytes, &mapB0, &s.full[stage], kb * BK, t.n * width + width / 2);
        }
        issued_mask |= 1u << stage;
        last_phase_bits = (last_phase_bits & ~(1u << stage)) | (phase << stage);
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    leader = elect_one();
    const uint64_t desc0 = sdesc_kmajor_sw128(smem_u32(tiles));
    const uint32_t idesc = idesc_bf16_f32(BM, width);
    int stage = 0;
    uint32_t phase = 0;
    int it = 0;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, ++it) {
      const int slot = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&s.tempty[slot], acc_phase ^ 1u, args.limit_ns, abort))) {
        if (leader && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 2);
        *abort = 1;
        break;
      }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + slot * BN;
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(&s.full[stage], phase, args.limit_ns, abort))) {
          if (leader && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 3);
          *abort = 1;
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t da = desc0 + static_cast<uint64_t>((stage * STAGE_BYTES) >> 4);
        const uint64_t db = da + (A_BYTES >> 4);
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)  // 16 elements = 32 bytes on
            mma_bf16(d_tmem, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          mma_commit(&s.empty[stage]);
        }
        mma_issued = true;
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      if (leader) mma_commit(&s.tfull[slot]);
      __syncwarp();
    }
  } else {
    // epilogue: warps 2..5 -> TMEM lane quarter (warp % 4)
    const int q = warp & 3;
    const int lrow = q * 32 + lane;
    int it = 0;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, ++it) {
      // warp-uniform control flow: tcgen05.ld below is .sync.aligned
      if (__any_sync(0xffffffffu, *abort != 0)) break;
      const int slot = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&s.tfull[slot], acc_phase, args.limit_ns, abort));
      if (!ok) {
        if (lane == 0 && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 4);
        *abort = 1;
        break;
      }
      tc_fence_after();
      const Tile t = decode(tile, args);
      const int row = t.m0 + lrow;
      const bool valid = row < t.m_end;
      const uint32_t tb = tmem_base + slot * BN + (static_cast<uint32_t>(q * 32) << 16);
      const int col0 = t.n * width, col1 = min(col0 + width, args.n_valid);
      float* orow = args.out_f32 + (size_t)row * args.n_valid;
      const bool vec = (args.n_valid & 3) == 0;
#pragma unroll 1
      for (int c = 0; c < 8; ++c) {
        if (col0 + c * 32 >= col1) break;  // warp-uniform
        uint32_t v[32];
        tmem_ld32(tb + c * 32, v);
        tmem_ld_wait();
        if (valid) {
          const int cb = col0 + c * 32;
          if (vec && cb + 32 <= col1) {
            float4* dst = reinterpret_cast<float4*>(orow + cb);
#pragma unroll
            for (int i = 0; i < 8; ++i)
              dst[i] = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]),
                                   __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (cb + i < col1) orow[cb + i] = __uint_as_float(v[i]);
          }
        }
      }
      tc_fence_before();
      mbar_arrive(&s.tempty[slot]);
    }
  }

  __syncthreads();
  if (s.abort) {
    volatile int* never = &s.zero;
    if (warp == 0 && lane == 0) {
      // wait for every TMA copy this CTA issued (bounded)
      for (int st = 0; st < STAGES; ++st)
        if ((issued_mask >> st) & 1u)
          mbar_wait(&s.full[st], (last_phase_bits >> st) & 1u, args.limit_ns, never);
    }
    if (leader && mma_issued) {  // the lane that issued the MMAs
      mma_commit(&s.drain);
      mbar_wait(&s.drain, 0, args.limit_ns, never);
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// ------------------------------------------------------------- gate/up and down
//
// Pairs (PAIR): a pair of CTAs on 2 SMs computes, with tcgen05.mma.cta_group::2 issued
// by the even CTA, a tile of 256 weight rows (the MMA's M side; 128 in each
// CTA's shared memory and TMEM lanes) by up to 256 permuted rows of one expert
// (the N side, split evenly between the two CTAs' shared memory). The weight
// side is always full; an expert's rows are cut into even tiles of a multiple of
// 16 rows (the N granularity of the instruction), so at most 15 padding rows
// are computed per expert instead of up to 255 for a 256-row M tile. Each CTA
// loads its N/2 rows as one TMA box: a stage of 5-6 boxes starved the tensor
// pipe.
//   gate/up: CTA r holds W1_e rows f..f+63 (TMEM lanes 0..63) and the same
//            rows of W3_e (lanes 64..127), f = 128 n + 64 r; the epilogue
//            warps of the gate and up lanes exchange half of their values
//            through shared memory and each forms SwiGLU for half the rows.
//   down:    CTA r holds W2_e rows 256 n + 128 r + 0..127 (all 128 lanes).
// The accumulator is transposed (lane = output column, TMEM column = row);
// the epilogue writes it row-major through a shared-memory tile with 16-byte
// coalesced stores, skipping rows beyond the expert's range.
// Each cluster is one CTA pair, and each CTA loads its own operand boxes from
// this GPU's memory (no multicast loads).
// Single CTAs: the same tile halved, 128 weight rows by up to 128 permuted
// rows, with cta_group::1 MMAs, for batches whose weights are streamed once:
// bound by HBM. A tile moves 16 KB of weights and the expert's own rows (16 to
// 128) a K step; rows on the M side moved 128 row boxes whatever the expert
// had and 256 columns a tile: gate/up of 1 token on 8 experts 126 against 72
// us, of 128 tokens 285 against 275; 64 experts x 8 tokens 74 and 62 us.
// Barriers: full[s] (even CTA, one arrive with the pair's bytes; both CTAs'
// TMA loads complete on it), empty[s] and tfull[b] (both CTAs, arrived by the
// even CTA's MMA commits signalled to the pair), tempty[b] (even CTA, one
// arrive per epilogue warp of either CTA). The gate/up epilogue runs on two
// groups of four warps that take alternate 32-row chunks, so two chunks are
// in flight (short-K tiles are otherwise epilogue-bound); down runs one group.
// Named barriers 1 and 2 (the 128 threads of a group) order each group's
// shared-memory exchange, and the decision to stop is a barrier reduction over
// all epilogue warps (barrier 3), so they always leave together.
constexpr int P_BM = 256;            // permuted rows (N side) per tile
constexpr int P_W_BYTES = 128 * BK * 2;   // 128 weight rows per CTA and K block
constexpr int P_T_BYTES = 128 * BK * 2;   // one box of 128 permuted rows per CTA
constexpr int P_STAGE_BYTES = P_W_BYTES + P_T_BYTES;
// the most stages a ring has: a single CTA's with boxes of 16 rows, in the space of six of 128
constexpr int P_MAX_STAGES = 6 * P_STAGE_BYTES / (P_W_BYTES + 16 * BK * 2);
constexpr int P_X_PITCH = 17;             // floats per exchange row (odd: no bank conflicts)
constexpr int P_XBUF_FLOATS = 128 * P_X_PITCH;
constexpr int P_EPI_GROUP_BYTES = 2 * (P_XBUF_FLOATS * 4 + 32 * 64 * 2);  // gate/up, double-buffered
static_assert(P_EPI_GROUP_BYTES >= 2 * 32 * 128 * 2, "down staging fits");


struct PSmem {
  uint64_t full[P_MAX_STAGES];
  uint64_t empty[P_MAX_STAGES];
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
  int zero;
  int max_rows;  // the largest row tile
  int mt_start[ORDERMOE_MAX_EXPERTS + 1];
  int offs[ORDERMOE_MAX_EXPERTS + 1];
};
// Per projection: a pair's gate/up (SwiGLU exchange in the epilogue) runs two
// epilogue groups of four warps and five stages; down (a plain conversion) one
// group and six stages. Five stages time the same as six for gate/up, and a
// second group made down slower. A single CTA, bound by the weights' bytes,
// runs one group and six stages.
template <int MODE, bool PAIR>
struct PCfg {
  static constexpr int GROUPS = MODE == GATEUP && PAIR ? 2 : 1;
  static constexpr int EPI_WARPS = 4 * GROUPS;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;
  static constexpr int STAGES = MODE == GATEUP && PAIR ? 5 : 6;  // stages of full rows
  static constexpr int MAX_STAGES = PAIR ? STAGES : P_MAX_STAGES;
  static constexpr int ROWS = PAIR ? P_BM : P_BM / 2;  // permuted rows per tile
  static constexpr int EPI_BYTES = GROUPS * P_EPI_GROUP_BYTES;
  static constexpr int SMEM_BYTES =
      STAGES * P_STAGE_BYTES + EPI_BYTES + 1024 + static_cast<int>(sizeof(PSmem));
  static_assert(MAX_STAGES <= P_MAX_STAGES, "stage barriers");
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of the FFN kernels");
};

__device__ __forceinline__ Tile decode_pair(int tile, const PSmem& s, int E, int n_tiles) {
  // the last expert whose first tile is <= tile (binary search: the row-tile
  // starts never decrease; empty experts share their successor's start)
  int e = 0, hi = E - 1;
  while (e < hi) {
    const int mid = (e + hi + 1) >> 1;
    if (s.mt_start[mid] * n_tiles <= tile) e = mid;
    else hi = mid - 1;
  }
  const int local = tile - s.mt_start[e] * n_tiles;
  const int n_mt = s.mt_start[e + 1] - s.mt_start[e];
  Tile t;
  t.e = e;
  t.n = local / n_mt;
  // an expert's rows in even shares: tiles of one expert take the same time, so
  // the CTAs that share its weights stay at the same K and find them in L2.
  // (Full tiles and a small last one: 2.47 and 2.23 GB of DRAM reads in the wide
  // layer's gate/up and down, 4096 tokens x 8 experts, against 1.97 and 1.81.)
  const int rows = s.offs[e + 1] - s.offs[e];
  const int per = ((rows + n_mt - 1) / n_mt + 15) & ~15;  // <= bm, and (n_mt - 1) per < rows
  const int first = (local - t.n * n_mt) * per;
  t.m0 = s.offs[e] + first;
  t.m_end = s.offs[e] + min(first + per, rows);
  return t;
}

// rows of the tile rounded up to the MMA's N granularity (16)
__device__ __forceinline__ int tile_n(const Tile& t) { return (t.m_end - t.m0 + 15) & ~15; }

// the 128 threads of epilogue group grp (named barriers 1 and 2)
__device__ __forceinline__ void epi_sync(int grp) {
  asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
}
// true in every epilogue thread iff p holds in all N of them (named barrier 3)
template <int N>
__device__ __forceinline__ bool epi_all(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.and.pred po, 3, %2, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(p)), "n"(N)
      : "memory");
  return r != 0;
}

// Tensor maps of the permuted rows with boxes of 16, 32, ..., 128 rows: a
// tile of N rows loads N/2 rows per CTA (rounded up to 16) instead of a full
// 128-row box.
struct RowMaps {
  CUtensorMap m[8];  // m[i]: box of 16 (i + 1) rows; single CTAs: m[0..3], 16 << i rows
};
// A single CTA's box for n rows (16 .. 128): the next power of two, so that a
// launch prepares four maps (each costs about 0.1 us of the host's time).
__device__ __forceinline__ int single_box(int n) { return n <= 16 ? 16 : 1 << (32 - __clz(n - 1)); }
// PAIR: one cluster = one CTA pair. Otherwise a CTA alone computes the tile's
// 128 weight rows by up to 128 permuted rows with cta_group::1 MMAs.
template <int MODE, bool PAIR>
__global__ void __launch_bounds__(PCfg<MODE, PAIR>::THREADS, 1)
    ffn_gemm_kernel(const __grid_constant__ CUtensorMap mapW0,
                    const __grid_constant__ CUtensorMap mapW1,
                    const __grid_constant__ RowMaps mapT, Args args) {
  using Cfg = PCfg<MODE, PAIR>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* epi = tiles + Cfg::STAGES * P_STAGE_BYTES;
  PSmem& s = *reinterpret_cast<PSmem*>(epi + Cfg::EPI_BYTES);
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  const uint32_t rp = PAIR ? cluster_ctarank() & 1u : 0u;  // rank within the pair
  const uint32_t lead = 0;                                  // the pair's even CTA (MMA issuer)
  const bool even = (rp == 0);
  const int cluster = PAIR ? blockIdx.x / 2 : blockIdx.x;
  const int n_clusters = PAIR ? gridDim.x / 2 : gridDim.x;
  // launched with launch_pdl: barriers, TMEM and tensor-map prefetches are set
  // up while the previous kernel finishes; global memory only after pdl_wait
  pdl_trigger();
  if (warp == 0 && lane == 0) {
    tma_prefetch_map(&mapW0);
    if (MODE == GATEUP) tma_prefetch_map(&mapW1);
#pragma unroll
    for (int i = 0; i < (PAIR ? 8 : 4); ++i) tma_prefetch_map(&mapT.m[i]);
  }

  if (tid == 0) {
    for (int i = 0; i < Cfg::MAX_STAGES; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 1);  // one MMA commit of the pair
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s.tfull[i], 1);
      mbar_init(&s.tempty[i], (PAIR ? 2 : 1) * Cfg::EPI_WARPS);  // every epilogue warp (of both CTAs)
    }
    mbar_init(&s.drain, 1);
    s.abort = 0;
    s.zero = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(&s.tmem_base, TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(&s.tmem_base, TMEM_COLS);
      tmem_relinquish();
    }
  }
  if (warp == 2) {
    pdl_wait();  // the offsets come from the permutation
    load_row_tiles(s, args, Cfg::ROWS, lane);
  }
  tc_fence_before();
  if (PAIR) cluster_sync();  // barriers of both CTAs initialised, TMEM allocated
  else __syncthreads();
  tc_fence_after();
  pdl_wait();  // every thread: the previous kernel's outputs are visible
  const uint32_t tmem_base = s.tmem_base;
  // A single CTA's ring holds as many stages as its largest row tile leaves
  // room for: it is bound by the weights' bytes, and the fewer the rows, the
  // more of the weights are in flight. (Wide gate/up of 128 tokens, 8 experts,
  // d 4096, d_ff 14336: 286 us with six stages of 128 rows, 273 with nine of
  // 48; 64 experts, d 2048, d_ff 1408: 120.8 and 117.0 us.)
  const int stage_bytes = PAIR ? P_STAGE_BYTES : P_W_BYTES + single_box(s.max_rows) * BK * 2;
  const int n_stages = PAIR ? Cfg::STAGES : min(Cfg::MAX_STAGES, Cfg::STAGES * P_STAGE_BYTES / stage_bytes);
  const int total = s.mt_start[args.E] * args.n_tiles;
  const int kblocks = args.K / BK;
  volatile int* abort = &s.abort;
  uint32_t issued_mask = 0, last_phase_bits = 0;
  bool mma_issued = false;
  bool leader = false;  // the MMA warp's issuing lane
  // tile -> (expert, column slice, row range)
  auto tile_of = [&](int tile) { return decode_pair(tile, s, args.E, args.n_tiles); };

  if (warp == 0) {
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    for (int tile = cluster; tile < total; tile += n_clusters) {
      const Tile t = tile_of(tile);
      const int nr = tile_n(t) >> (PAIR ? 1 : 0);  // N/2 rows per CTA of a pair
      const int trow = t.m0 + static_cast<int>(rp) * nr;
      const int hb = PAIR ? (nr + 15) & ~15 : single_box(nr);  // rows per CTA's box (16 .. 128)
      const CUtensorMap* mrow = &mapT.m[PAIR ? (hb >> 4) - 1 : 27 - __clz(hb)];
      const uint32_t stage_tx = (PAIR ? 2u : 1u) * static_cast<uint32_t>(P_W_BYTES + hb * BK * 2);
      // the CTA's rows of the weights: 64 of W1 and of W3, or 128 of W2
      const int wrow = t.e * args.b_rows +
                       (PAIR ? 2 * t.n + static_cast<int>(rp) : t.n) * (MODE == GATEUP ? 64 : 128);
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(&s.empty[stage], phase ^ 1u, args.limit_ns, abort))) {
          if (issuer && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 11);
          *abort = 1;
          ok = false;
          break;
        }
        uint8_t* sw = tiles + stage * stage_bytes;
        uint8_t* st = sw + P_W_BYTES;
        if (issuer) {
          if (even) mbar_arrive_expect_tx(&s.full[stage], stage_tx);
          if (PAIR) {
            const uint32_t full_even = mapa_shared(smem_u32(&s.full[stage]), lead);
            tma_load_2d_pair(sw, &mapW0, full_even, kb * BK, wrow);  // gate/up: W1, lanes 0..63
            if (MODE == GATEUP) tma_load_2d_pair(sw + P_W_BYTES / 2, &mapW1, full_even, kb * BK, wrow);  // W3: 64..127
            tma_load_2d_pair(st, mrow, full_even, kb * BK, trow);
          } else {
            tma_load_2d(sw, &mapW0, &s.full[stage], kb * BK, wrow);
            if (MODE == GATEUP) tma_load_2d(sw + P_W_BYTES / 2, &mapW1, &s.full[stage], kb * BK, wrow);
            tma_load_2d(st, mrow, &s.full[stage], kb * BK, trow);
          }
        }
        issued_mask |= 1u << stage;
        last_phase_bits = (last_phase_bits & ~(1u << stage)) | (phase << stage);
        if (++stage == n_stages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
    }
  } else if (warp == 1) {
    // The whole warp walks the stages, so that its control flow and the
    // descriptors stay uniform, and one elected lane issues (the producer warp
    // alike). A lane walking them alone held the issue back, whatever the tile:
    // gate/up of 8192 tokens x 64 experts (top-6, d 2048, d_ff 1408) 372 -> 347
    // us, down 197 -> 180; of 4096 x 8 (top-2, d 4096, d_ff 14336) gate/up 1144
    // -> 1030 (ncu, with even row tiles); single CTAs' down of 1 token x 8 experts 65 -> 46, of 128 152 ->
    // 146 us.
    if (even) {
      leader = elect_one();
      const uint64_t desc0 = sdesc_kmajor_sw128(smem_u32(tiles));
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      for (int tile = cluster; tile < total; tile += n_clusters, ++it) {
        const int slot = it & 1;
        const uint32_t acc_phase = (it >> 1) & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&s.tempty[slot], acc_phase ^ 1u, args.limit_ns, abort))) {
          if (leader && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 12);
          *abort = 1;
          break;
        }
        tc_fence_after();
        const Tile t = tile_of(tile);
        const uint32_t idesc = idesc_bf16_f32(PAIR ? 256 : 128, tile_n(t));
        const uint32_t d_tmem = tmem_base + slot * BN;
        bool ok = true;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!__all_sync(0xffffffffu, mbar_wait(&s.full[stage], phase, args.limit_ns, abort))) {
            if (leader && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 13);
            *abort = 1;
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = desc0 + static_cast<uint64_t>((stage * stage_bytes) >> 4);
          const uint64_t db = da + (P_W_BYTES >> 4);
          if (leader) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {  // 16 elements = 32 bytes on
              if (PAIR) mma_bf16_pair(d_tmem, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
              else mma_bf16(d_tmem, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
            }
            if (PAIR) mma_commit_pair(&s.empty[stage], 0x3);
            else mma_commit(&s.empty[stage]);
          }
          mma_issued = true;
          if (++stage == n_stages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (leader) {
          if (PAIR) mma_commit_pair(&s.tfull[slot], 0x3);
          else mma_commit(&s.tfull[slot]);
        }
        __syncwarp();
      }
    }
  } else {
    // epilogue: warps 2..9 in two groups of four; TMEM lane quarter q = warp % 4;
    // group grp takes the 32-row chunks grp, grp + 2, ... of every tile
    const int q = warp & 3;
    const int grp = (warp - 2) >> 2;  // 0 .. GROUPS - 1
    const int et = tid - 64 - 128 * grp;  // 0..127 within the group
    uint8_t* ge = epi + grp * P_EPI_GROUP_BYTES;
    float* xbuf = reinterpret_cast<float*>(ge);                          // [2][128][P_X_PITCH]
    uint16_t* obuf = reinterpret_cast<uint16_t*>(ge + 2 * P_XBUF_FLOATS * 4);  // gate/up [2][32][64]
    uint16_t* ybuf = reinterpret_cast<uint16_t*>(ge);                    // down [2][32][128]
    int it = 0;
    for (int tile = cluster; tile < total; tile += n_clusters, ++it) {
      const int slot = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      const bool waited = (*abort == 0) && mbar_wait(&s.tfull[slot], acc_phase, args.limit_ns, abort);
      if (!epi_all<Cfg::EPI_WARPS * 32>(waited)) {  // the same decision in every epilogue warp
        if (!waited && lane == 0 && !*abort) report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 14);
        *abort = 1;
        break;
      }
      tc_fence_after();
      const Tile t = tile_of(tile);
      const int rows = t.m_end - t.m0;
      const int nchunks = (rows + 31) >> 5;
      const uint32_t tb = tmem_base + slot * BN + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll 1
      for (int c = grp; c < nchunks; c += Cfg::GROUPS) {
        const int buf = (c / Cfg::GROUPS) & 1;
        uint32_t v[32];
        tmem_ld32(tb + c * 32, v);  // TMEM column = row c*32 + i of the tile
        tmem_ld_wait();
        if (MODE == GATEUP) {
          // gate lanes (q 0, 1) keep rows 0..15 of the chunk and hand 16..31
          // to the up lanes (q 2, 3) of the same columns, which hand back 0..15
          const bool gate = q < 2;
          const int keep = gate ? 0 : 16;
          float* xb = xbuf + buf * P_XBUF_FLOATS;
          float* mine = xb + (q * 32 + lane) * P_X_PITCH;
#pragma unroll
          for (int i = 0; i < 16; ++i) mine[i] = __uint_as_float(gate ? v[16 + i] : v[i]);
          epi_sync(grp);
          const float* other = xb + ((q ^ 2) * 32 + lane) * P_X_PITCH;
          uint16_t* ob = obuf + buf * (32 * 64);
          const int col = (q & 1) * 32 + lane;
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            float h[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const float own = __uint_as_float(gate ? v[i + j] : v[16 + i + j]);
              const float oth = other[i + j];
              const float g = gate ? own : oth;
              const float u = gate ? oth : own;
              // silu(g) u = g u / (1 + e^-g); for full row tiles, whose epilogue
              // the MMAs wait for, the quotient by the fast reciprocal (2 ulp in
              // fp32, far below the bf16 rounding of h)
              h[j] = PAIR && args.fast_div ? __fdividef(g * u, 1.0f + __expf(-g))
                                           : g / (1.0f + __expf(-g)) * u;
            }
            const uint32_t pk = pack_bf16x2(h[0], h[1]);
            ob[(keep + i) * 64 + col] = static_cast<uint16_t>(pk & 0xFFFFu);
            ob[(keep + i + 1) * 64 + col] = static_cast<uint16_t>(pk >> 16);
          }
          epi_sync(grp);
          uint16_t* gcol = args.out + (PAIR ? 2 * t.n + static_cast<int>(rp) : t.n) * 64 + (et & 7) * 8;
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const int r = p * 16 + (et >> 3);
            const int row = c * 32 + r;
            if (row < rows)
              *reinterpret_cast<uint4*>(gcol + (size_t)(t.m0 + row) * args.ldo) =
                  *reinterpret_cast<const uint4*>(ob + r * 64 + (et & 7) * 8);
          }
        } else {
          uint16_t* yb = ybuf + buf * (32 * 128);
          const int col = q * 32 + lane;
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const uint32_t pk = pack_bf16x2(__uint_as_float(v[i]), __uint_as_float(v[i + 1]));
            yb[i * 128 + col] = static_cast<uint16_t>(pk & 0xFFFFu);
            yb[(i + 1) * 128 + col] = static_cast<uint16_t>(pk >> 16);
          }
          epi_sync(grp);
          uint16_t* gcol = args.out + (PAIR ? 2 * t.n + static_cast<int>(rp) : t.n) * 128 + (et & 15) * 8;
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const int r = p * 8 + (et >> 4);
            const int row = c * 32 + r;
            if (row < rows)
              *reinterpret_cast<uint4*>(gcol + (size_t)(t.m0 + row) * args.ldo) =
                  *reinterpret_cast<const uint4*>(yb + r * 128 + (et & 15) * 8);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_remote(mapa_shared(smem_u32(&s.tempty[slot]), lead));
        else mbar_arrive(&s.tempty[slot]);
      }
    }
  }

  __syncthreads();
  if (s.abort) {
    volatile int* never = &s.zero;
    if (warp == 0 && lane == 0 && even) {
      for (int st = 0; st < n_stages; ++st)
        if ((issued_mask >> st) & 1u)
          mbar_wait(&s.full[st], (last_phase_bits >> st) & 1u, args.limit_ns, never);
    }
    if (leader && mma_issued) {  // the lane that issued the MMAs
      if (PAIR) mma_commit_pair(&s.drain, 0x1);
      else mma_commit(&s.drain);
      mbar_wait(&s.drain, 0, args.limit_ns, never);
    }
  }
  tc_fence_before();
  if (PAIR) cluster_sync();  // every CTA finished: no more arrivals or copies into any
  else __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    if (PAIR) tmem_dealloc_pair(tmem_base, TMEM_COLS);
    else tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// ------------------------------------------------------------------- host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// 2-D bf16 row-major [rows][cols] map with a 64 x 128 box and 128-byte swizzle.
int make_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols) {
  return make_tmap_bf16(map, base, rows, cols, 128);
}

}  // namespace gg

int make_tmap_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols,
                   uint32_t box_rows) {
  gg::EncodeTiledFn enc = gg::encode_fn();
  if (!enc) return fail(ORDERMOE_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {gg::BK, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(ORDERMOE_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return ORDERMOE_OK;
}

template <int MODE, bool PAIR>
static cudaError_t ffn_attr() {
  return cudaFuncSetAttribute(gg::ffn_gemm_kernel<MODE, PAIR>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              gg::PCfg<MODE, PAIR>::SMEM_BYTES);
}

static int ffn_attrs() {
  using namespace gg;
  static PerDevice cache;
  const cudaError_t attr_err = static_cast<cudaError_t>(per_device(cache, [] {
    cudaError_t e = ffn_attr<GATEUP, true>();
    if (e == cudaSuccess) e = ffn_attr<DOWN, true>();
    if (e == cudaSuccess) e = ffn_attr<GATEUP, false>();
    if (e == cudaSuccess) e = ffn_attr<DOWN, false>();
    return static_cast<int>(e);
  }));
  if (attr_err != cudaSuccess) return cuda_fail(attr_err, "cudaFuncSetAttribute(ffn_gemm_kernel)");
  return ORDERMOE_OK;
}

template <int MODE, bool PAIR>
static cudaLaunchConfig_t ffn_config(int grid, cudaStream_t stream, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(gg::PCfg<MODE, PAIR>::THREADS, 1, 1);
  cfg.dynamicSmemBytes = gg::PCfg<MODE, PAIR>::SMEM_BYTES;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = PAIR ? 2 : 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // waits in the kernel
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_on(stream) ? 2 : 1;
  return cfg;
}

// CTA pairs that can be resident at once (not every SM finds a partner in its
// GPC: 76 pairs on GB300); the persistent grid never exceeds it, so no
// cluster waits for another.
template <int MODE>
static int max_resident_clusters() {
  static PerDevice cache;
  return per_device(cache, [] {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = ffn_config<MODE, true>(2 * (num_sms() / 2), nullptr, attr);
    cfg.numAttrs = 1;  // the cluster shape alone decides residency
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gg::ffn_gemm_kernel<MODE, true>, &cfg) != cudaSuccess ||
        n <= 0) {
      cudaGetLastError();
      n = num_sms() / 2;
    }
    return n < num_sms() / 2 ? n : num_sms() / 2;
  });
}

// One launch over the row tiles of R permuted rows; a.n_tiles weight tiles
// (of a pair, or of a CTA) per expert.
template <int MODE, bool PAIR>
static int launch_ffn(const CUtensorMap& w0, const CUtensorMap& w1, const gg::RowMaps& t,
                      const gg::Args& a, int R, cudaStream_t stream, const char* what) {
  constexpr int rows = gg::PCfg<MODE, PAIR>::ROWS;
  const long long row_tiles = (long long)R / rows + (R < a.E ? R : a.E);  // at least as many as there are
  const long long tiles = row_tiles * a.n_tiles;
  const long long most = PAIR ? max_resident_clusters<MODE>() : num_sms();
  const int units = static_cast<int>(tiles < most ? tiles : most);
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = ffn_config<MODE, PAIR>(PAIR ? 2 * units : units, stream, attr);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, gg::ffn_gemm_kernel<MODE, PAIR>, w0, w1, t, a);
  if (e != cudaSuccess) return cuda_fail(e, what);
  OM_LAUNCHED(what);
  return ORDERMOE_OK;
}

// The row maps of a [rows][cols] bf16 tensor, boxes of 16 .. 128 rows.
static int make_row_maps(gg::RowMaps* rm, const void* base, uint64_t rows, uint64_t cols, bool pairs) {
  for (int i = 0; i < (pairs ? 8 : 4); ++i) {
    const int rc = make_tmap_bf16(&rm->m[i], base, rows, cols,
                                  static_cast<uint32_t>(pairs ? 16 * (i + 1) : 16 << i));
    if (rc) return rc;
  }
  return ORDERMOE_OK;
}

// Tile shape: CTA pairs when experts average at least kPairRows rows, single
// CTAs of up to 128 rows below, where an expert is one row tile and the
// weights are read once. Measured, single against pairs (gate/up + down, us):
// 64 experts, d 2048, d_ff 1408: 96 rows an expert on average (at most 122)
// 128 + 67 against 133 + 69, 112 rows (139) 125 + 73 against 135 + 70, 131
// rows (156) 157 + 85 against 136 + 72; 8 experts, d 4096, d_ff 14336: 107
// rows (119) 287 + 155 against 302 + 161, 127 rows (142) 370 + 210 against
// 305 + 162: the line is where the fuller experts pass 128 rows. (It sees the
// average: with every row on one expert, single tiles of 128 x 128 move more of
// the rows than the 256-column tiles they took the place of: gate/up + down of 64
// experts, 96 rows on average, 100 against 91 us, of 16 experts, d 1024, d_ff 4096,
// 111 rows, 66 against 57. By zipf 1.1 101 against 96 there, faster elsewhere.)
constexpr int kPairRows = 112;
static bool use_pairs(int R, int E) { return (long long)R >= (long long)kPairRows * E; }

// H = SwiGLU(X_perm W1^T, X_perm W3^T) over the expert row ranges.
int gate_up_launch(const uint16_t* X_perm, const int32_t* offsets, int R, const uint16_t* W1,
                   const uint16_t* W3, int E, int d, int dff, uint16_t* H, cudaStream_t stream) {
  using namespace gg;
  int rc;
  if ((rc = ffn_attrs())) return rc;
  const bool pairs = use_pairs(R, E);
  Args a{};
  a.offsets = offsets; a.rows = R; a.E = E; a.limit_ns = wait_limit_ns();
  a.K = d; a.n_tiles = dff / (pairs ? 128 : 64); a.b_rows = dff; a.out = H; a.ldo = dff;
  a.fast_div = (long long)R >= (long long)P_BM * E;  // row tiles full on average
  CUtensorMap mW1, mW3;
  RowMaps mX;
  if ((rc = make_tmap_bf16(&mW1, W1, (uint64_t)E * dff, d, 64))) return rc;
  if ((rc = make_tmap_bf16(&mW3, W3, (uint64_t)E * dff, d, 64))) return rc;
  if ((rc = make_row_maps(&mX, X_perm, R, d, pairs))) return rc;
  return pairs ? launch_ffn<GATEUP, true>(mW1, mW3, mX, a, R, stream, "ffn_gemm_kernel<gate_up, pair>")
               : launch_ffn<GATEUP, false>(mW1, mW3, mX, a, R, stream, "ffn_gemm_kernel<gate_up>");
}

// Y_perm = H W2^T over the expert row ranges.
int down_launch(const uint16_t* H, const int32_t* offsets, int R, const uint16_t* W2, int E, int d,
                int dff, uint16_t* Y, cudaStream_t stream) {
  using namespace gg;
  int rc;
  if ((rc = ffn_attrs())) return rc;
  const bool pairs = use_pairs(R, E);
  Args a{};
  a.offsets = offsets; a.rows = R; a.E = E; a.limit_ns = wait_limit_ns();
  a.K = dff; a.n_tiles = d / (pairs ? 256 : 128); a.b_rows = d; a.out = Y; a.ldo = d;
  CUtensorMap mW2;
  RowMaps mH;
  if ((rc = make_tmap_bf16(&mW2, W2, (uint64_t)E * d, dff, 128))) return rc;
  if ((rc = make_row_maps(&mH, H, R, dff, pairs))) return rc;
  return pairs ? launch_ffn<DOWN, true>(mW2, mW2, mH, a, R, stream, "ffn_gemm_kernel<down, pair>")
               : launch_ffn<DOWN, false>(mW2, mW2, mH, a, R, stream, "ffn_gemm_kernel<down>");
}

int ffn_launch(const uint16_t* X_perm, const int32_t* offsets, int R, const uint16_t* W1,
               const uint16_t* W3, const uint16_t* W2, int E, int d, int dff, uint16_t* H,
               uint16_t* Y, cudaStream_t stream) {
  int rc = gate_up_launch(X_perm, offsets, R, W1, W3, E, d, dff, H, stream);
  if (rc) return rc;
  return down_launch(H, offsets, R, W2, E, d, dff, Y, stream);
}

// H[n][c] = sum_k X[n][k] W[c][k] in fp32 for n < N, c < C (C = L*E stacked
// router rows): the router-logit contraction of Eq. 3 over calibration tokens.
int logits_gemm_launch(const uint16_t* X, int N, const uint16_t* W, int C, int d, float* H,
                       cudaStream_t stream) {
  using namespace gg;
  static PerDevice cache;
  const cudaError_t attr_err = static_cast<cudaError_t>(per_device(cache, [] {
    return static_cast<int>(cudaFuncSetAttribute(logits_gemm_kernel,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 SMEM_BYTES));
  }));
  if (attr_err != cudaSuccess) return cuda_fail(attr_err, "cudaFuncSetAttribute(logits)");
  CUtensorMap mX, mW;
  int rc;
  if ((rc = make_map(&mX, X, N, d))) return rc;
  // column slices of one width, so that every tile costs the same (with 256 and
  // a rest, CTAs of one parity got all the full tiles: 45.7 against 33.2 us
  // for 32768 tokens x 320 columns, d 1024)
  const int n_tiles = (C + BN - 1) / BN;
  const int width = ((C + n_tiles - 1) / n_tiles + 15) & ~15;
  if ((rc = make_tmap_bf16(&mW, W, C, d, width / 2))) return rc;
  Args a{};
  a.offsets = nullptr;
  a.rows = N;
  a.n_valid = C;
  a.out_f32 = H;
  a.K = d;
  a.n_tiles = n_tiles;
  a.b_rows = width;
  a.limit_ns = wait_limit_ns();
  const long long tiles = (long long)((N + BM - 1) / BM) * a.n_tiles;
  const int sms = num_sms();
  const int grid = static_cast<int>(tiles < sms ? tiles : sms);
  logits_gemm_kernel<<<grid, THREADS, SMEM_BYTES, stream>>>(mX, mW, a);
  OM_LAUNCHED("logits_gemm_kernel");
  return ORDERMOE_OK;
}

// ---------------------------------------------------------- wait self-test
__global__ void wait_timeout_kernel(uint64_t limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // nothing ever arrives on `bar`: the wait must run out
    if (!mbar_wait(&bar, 0, limit_ns, reinterpret_cast<volatile int*>(&abort_flag)))
      report(&g_err_gemm, ORDERMOE_DEV_WAIT_TIMEOUT, 99);
  }
}

int selftest_wait_timeout(uint64_t limit_ns, cudaStream_t stream) {
  wait_timeout_kernel<<<1, 32, 0, stream>>>(limit_ns);
  OM_LAUNCHED("wait_timeout_kernel");
  return ORDERMOE_OK;
}

}  // namespace om

using namespace om;

static int ffn_check(const char* who, int R, int E, int d, int dff) {
  if (R < 0 || E <= 0 || E > ORDERMOE_MAX_EXPERTS)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "%s: need R >= 0 and 1 <= E <= 64", who);
  if (d <= 0 || d % 256 != 0 || dff <= 0 || dff % 128 != 0)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "%s: need d %% 256 == 0 and dff %% 128 == 0", who);
  if ((long long)E * dff > INT32_MAX || (long long)E * d > INT32_MAX || (long long)R * dff > INT32_MAX * 4LL)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "%s: sizes too large", who);
  return ORDERMOE_OK;
}

static bool all_aligned(std::initializer_list<const void*> ps) {
  for (const void* p : ps)
    if (!p || !aligned16(p)) return false;
  return true;
}

extern "C" int ordermoe_expert_ffn(const uint16_t* X_perm, const int32_t* offsets, int R,
                                   const uint16_t* W1, const uint16_t* W3, const uint16_t* W2,
                                   int E, int d, int dff, uint16_t* H, uint16_t* Y_perm,
                                   ordermoe_stream_t stream) {
  OM_TRACE();
  int rc = ffn_check("expert_ffn", R, E, d, dff);
  if (rc || R == 0) return rc;
  if (!offsets || !all_aligned({X_perm, W1, W3, W2, H, Y_perm}))
    return fail(ORDERMOE_ERR_INVALID_ARG, "expert_ffn: null or not 16-byte aligned pointer");
  return ffn_launch(X_perm, offsets, R, W1, W3, W2, E, d, dff, H, Y_perm, stream);
}

extern "C" int ordermoe_expert_gate_up(const uint16_t* X_perm, const int32_t* offsets, int R,
                                       const uint16_t* W1, const uint16_t* W3, int E, int d, int dff,
                                       uint16_t* H, ordermoe_stream_t stream) {
  OM_TRACE();
  int rc = ffn_check("expert_gate_up", R, E, d, dff);
  if (rc || R == 0) return rc;
  if (!offsets || !all_aligned({X_perm, W1, W3, H}))
    return fail(ORDERMOE_ERR_INVALID_ARG, "expert_gate_up: null or not 16-byte aligned pointer");
  return gate_up_launch(X_perm, offsets, R, W1, W3, E, d, dff, H, stream);
}

extern "C" int ordermoe_expert_down(const uint16_t* H, const int32_t* offsets, int R,
                                    const uint16_t* W2, int E, int d, int dff, uint16_t* Y_perm,
                                    ordermoe_stream_t stream) {
  OM_TRACE();
  int rc = ffn_check("expert_down", R, E, d, dff);
  if (rc || R == 0) return rc;
  if (!offsets || !all_aligned({H, W2, Y_perm}))
    return fail(ORDERMOE_ERR_INVALID_ARG, "expert_down: null or not 16-byte aligned pointer");
  return down_launch(H, offsets, R, W2, E, d, dff, Y_perm, stream);
}
