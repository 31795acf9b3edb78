// Router + softmax + top-k + server-expert selection (Alg. 2, H = 1), and the
// per-layer selection tables it reads (Eqs. 7, 18, 37, 38).
#include <cstring>

#include "common.cuh"

namespace om {

static __device__ unsigned long long g_err_route = 0;

int read_clear_err_route(unsigned long long* out) {
  unsigned long long zero = 0;
  OM_CUDA(cudaMemcpyFromSymbol(out, g_err_route, sizeof(*out)));
  OM_CUDA(cudaMemcpyToSymbol(g_err_route, &zero, sizeof(zero)));
  return ORDERMOE_OK;
}

// Byte layout of the tables buffer (documented in ordermoe.h).
constexpr int kTabMagic = 0x4f4d5442;
constexpr size_t kOffPmask = 64, kOffSubst = 320, kOffQtab = 832;
__host__ __device__ inline size_t off_cq(int E) { return kOffQtab + sizeof(float) * E * E; }
__host__ __device__ inline size_t off_a(int E) { return off_cq(E) + sizeof(float) * E * E; }
__host__ __device__ inline size_t tables_bytes(int E, int M) {
  size_t b = off_a(E) + sizeof(float) * (size_t)M * M * M;
  return (b + 255) & ~size_t(255);
}

// ---------------------------------------------------------------------------
// Tables. One block; fp64 terms use explicit round-to-nearest operations so
// that no multiply-add is fused.
__global__ void build_tables_kernel(const float* __restrict__ sim, const int32_t* __restrict__ group,
                                    const uint8_t* __restrict__ placement, int E, int M,
                                    float theta, float qbar, const double* __restrict__ F,
                                    const double* __restrict__ B, const double* __restrict__ tau,
                                    double z, double c, double omega_T, double omega_Q,
                                    uint8_t* __restrict__ tab) {
  int32_t* hdr = reinterpret_cast<int32_t*>(tab);
  float* hdrf = reinterpret_cast<float*>(tab);
  uint32_t* pmask = reinterpret_cast<uint32_t*>(tab + kOffPmask);
  unsigned long long* subst = reinterpret_cast<unsigned long long*>(tab + kOffSubst);
  float* Qtab = reinterpret_cast<float*>(tab + kOffQtab);
  float* Cq = reinterpret_cast<float*>(tab + off_cq(E));
  float* A = reinterpret_cast<float*>(tab + off_a(E));
  const int tid = threadIdx.x;
  if (tid == 0) {
    hdr[0] = kTabMagic; hdr[1] = E; hdr[2] = M; hdr[3] = 0;
    hdrf[4] = theta; hdrf[5] = qbar;
  }
  for (int e = tid; e < 64; e += blockDim.x) {
    uint32_t pm = 0;
    unsigned long long sb = 0;
    if (e < E) {
      for (int m = 0; m < M; ++m)
        if (placement[m * E + e]) pm |= 1u << m;
      for (int k = 0; k < E; ++k) {
        const float s = sim[e * E + k];
        if (k != e && group[k] == group[e] && s >= theta) sb |= 1ull << k;
      }
    }
    pmask[e] = pm;
    subst[e] = sb;
  }
  for (int i = tid; i < E * E; i += blockDim.x) {
    const int r = i / E, k = i % E;
    const float s = sim[i];
    float q = 0.0f;
    if (k != r) q = __fmul_rn(0.5f, __fsub_rn(1.0f, (1.0f < s) ? 1.0f : s));  // Eq. 18
    Qtab[i] = q;
    float cq = 0.0f;
    if (q != 0.0f)
      cq = __double2float_rn(__ddiv_rn(__dmul_rn(omega_Q, static_cast<double>(q)),
                                       static_cast<double>(qbar)));
    Cq[i] = cq;
  }
  for (int i = tid; i < M * M * M; i += blockDim.x) {
    const int a = i / (M * M), s = (i / M) % M, m = i % M;
    const double dref = __ddiv_rn(c, F[a]);
    const double comp = __ddiv_rn(c, F[m]);
    double dl = comp;
    if (s != m) {
      const double trans = __dadd_rn(__ddiv_rn(z, B[s * M + m]), tau[s * M + m]);  // Eq. 37
      dl = __dadd_rn(trans, comp);
    }
    A[i] = __double2float_rn(__ddiv_rn(__dmul_rn(omega_T, dl), dref));  // Eq. 38, delay term
  }
}

// ---------------------------------------------------------------------------
// Selection tables staged in shared memory (one copy per CTA).
struct SelSmem {
  uint32_t pmask[64];
  int nsub[64];
  int kind[4];
  uint8_t sublist[64 * 64];
};

// Threads t0, t0 + nt (nt >= 64) ... of the block load the layer's tables
// into shared memory. The header, masks and the first E x E entries are
// loaded before any of them is used, so that their latencies overlap; the
// E x E tables are copied with 16-byte loads where sizes and addresses
// allow.
__device__ bool load_tables_range(const uint8_t* __restrict__ tab, int E, SelSmem& sm, float* s_Q,
                                  float* s_Cq, int t0, int nt) {
  const float* gQ = reinterpret_cast<const float*>(tab + kOffQtab);
  const float* gCq = reinterpret_cast<const float*>(tab + off_cq(E));
  const int n = E * E;
  const bool vec = (n & 3) == 0 && ((reinterpret_cast<uintptr_t>(gQ) | reinterpret_cast<uintptr_t>(gCq) |
                                     reinterpret_cast<uintptr_t>(s_Q) | reinterpret_cast<uintptr_t>(s_Cq)) &
                                    15u) == 0;
  const int Eh = reinterpret_cast<const int32_t*>(tab)[1];
  const int M = reinterpret_cast<const int32_t*>(tab)[2];
  uint32_t pm = 0;
  unsigned long long sb = 0;
  if (t0 < 64) {
    pm = reinterpret_cast<const uint32_t*>(tab + kOffPmask)[t0];
    sb = reinterpret_cast<const unsigned long long*>(tab + kOffSubst)[t0];
  }
  constexpr int kFirst = 4;  // 16-byte chunks of each table a thread loads up front
  float4 q_first[kFirst], c_first[kFirst];
  if (vec) {
    const float4* q4 = reinterpret_cast<const float4*>(gQ);
    const float4* c4 = reinterpret_cast<const float4*>(gCq);
#pragma unroll
    for (int u = 0; u < kFirst; ++u) {
      const int i = t0 + u * nt;
      if (i < n / 4) {
        q_first[u] = __ldg(q4 + i);
        c_first[u] = __ldg(c4 + i);
      }
    }
  }
  if (Eh != E || M <= 0 || M > 32) {
    if (blockIdx.x == 0 && t0 == 0) report(&g_err_route, ORDERMOE_DEV_BAD_INDEX, -1);
    return false;
  }
  if (t0 < 64) {
    sm.pmask[t0] = pm;
    int cnt = 0;
    while (sb) {
      const int b = __ffsll(static_cast<long long>(sb)) - 1;
      sm.sublist[t0 * 64 + cnt++] = static_cast<uint8_t>(b);
      sb &= sb - 1;
    }
    sm.nsub[t0] = cnt;
  }
  if (vec) {
    const float4* q4 = reinterpret_cast<const float4*>(gQ);
    const float4* c4 = reinterpret_cast<const float4*>(gCq);
#pragma unroll
    for (int u = 0; u < kFirst; ++u) {
      const int i = t0 + u * nt;
      if (i < n / 4) {
        reinterpret_cast<float4*>(s_Q)[i] = q_first[u];
        reinterpret_cast<float4*>(s_Cq)[i] = c_first[u];
      }
    }
#pragma unroll 4
    for (int i = t0 + kFirst * nt; i < n / 4; i += nt) {
      const float4 x = __ldg(q4 + i), y = __ldg(c4 + i);
      reinterpret_cast<float4*>(s_Q)[i] = x;
      reinterpret_cast<float4*>(s_Cq)[i] = y;
    }
  } else {
#pragma unroll 4
    for (int i = t0; i < n; i += nt) {
      s_Q[i] = gQ[i];
      s_Cq[i] = gCq[i];
    }
  }
  for (int i = t0; i < 4; i += nt) sm.kind[i] = 0;
  return true;
}

// Loads the layer's tables into shared memory (whole block). Returns false
// if the header does not match E (reported once).
__device__ bool load_tables(const uint8_t* __restrict__ tab, int E, SelSmem& sm, float* s_Q,
                            float* s_Cq) {
  return load_tables_range(tab, E, sm, s_Q, s_Cq, threadIdx.x, blockDim.x);  // blockDim.x >= 64
}

// The delay table A[a][s][m] of Eq. 38 (M^3 floats) is read once per
// candidate (expert, server) of every slot, so the selection keeps it in
// shared memory when it has at most kDelayStage entries (M <= 16);
// larger tables stay in global memory. Threads t0, t0 + nt, ... copy it;
// every thread gets the same pointer back, the one the selection reads.
constexpr int kDelayStage = 4096;
__device__ const float* load_delay_range(const uint8_t* __restrict__ tab, int E, float* s_A,
                                         int t0, int nt) {
  const int M = reinterpret_cast<const int32_t*>(tab)[2];
  const float* gA = reinterpret_cast<const float*>(tab + off_a(E));
  if (M <= 0 || M > 16) return gA;
  const int n = M * M * M;
  for (int i = t0; i < n; i += nt) s_A[i] = gA[i];
  return s_A;
}

// Look-ahead context (Eqs. 41-43): the tables of the next layers follow the
// current layer's at a fixed byte stride; P holds P_l .. P_{l+H-2}.
struct Lookahead {
  int H;                 // horizon; 1 = myopic (Phi = 0)
  size_t stride;         // bytes between consecutive layers' tables
  const float* P;        // [H-1][E][E]
  int topk_only;         // H = 1 with many experts: the router writes the targets and weights,
                         // select_lanes_kernel selects
};

// A token's logits in shared memory as 16-byte chunks: chunk c holds
// logits 4c .. 4c + 3 (-inf past E), at p[128 c] (one thread's column of a
// [chunk][128 tokens] array, so the 32 tokens of a warp read consecutive
// chunks: no bank conflicts).
struct ColLogits {
  const float4* p;
  __device__ __forceinline__ float4 chunk(int c) const { return p[c * 128]; }
};

// The KN largest of the token's nc chunks of logits by (logit desc, index
// asc) into v[0..KN), ix[0..KN), as a sorted list built by inserting the
// logits in index order: logit e goes to the first position whose value it
// exceeds, so an equal value stays behind the earlier index, and the entries
// from that position on move down one. The positions it exceeds form a
// suffix of the list (g[p] implies g[p+1]), which makes every position one
// select of its own value, the new logit or its predecessor; positions
// p >= e are still empty when logit e arrives. The list stays in registers
// (compile-time positions), nothing branches inside a chunk, and the loop
// over chunks keeps the code short (a long unrolled form stalled on
// instruction fetch). The -inf logits past E go behind every real one, so
// the first k <= E entries are real. Returns whether a logit was NaN.
template <int KN, class Src>
__device__ __forceinline__ bool topk_list(const Src& src, int nc, float (&v)[ORDERMOE_MAX_TOPK],
                                          int (&ix)[ORDERMOE_MAX_TOPK]) {
#pragma unroll
  for (int p = 0; p < ORDERMOE_MAX_TOPK; ++p) {
    v[p] = -INFINITY;
    ix[p] = -1;
  }
  bool nan = false;
#pragma unroll 1
  for (int c4 = 0; c4 < nc; ++c4) {
    const float4 x4 = src.chunk(c4);
    const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float c = xs[u];
      const int e = 4 * c4 + u;
      nan |= isnan(c);
      bool g[KN];
#pragma unroll
      for (int p = 0; p < KN; ++p) g[p] = (p >= e) | (c > v[p]);
#pragma unroll
      for (int p = KN - 1; p >= 1; --p) {
        const float tv = g[p] ? c : v[p];
        const int ti = g[p] ? e : ix[p];
        v[p] = g[p - 1] ? v[p - 1] : tv;
        ix[p] = g[p - 1] ? ix[p - 1] : ti;
      }
      v[0] = g[0] ? c : v[0];
      ix[0] = g[0] ? e : ix[0];
    }
  }
  return nan;
}

// One token: softmax over E, top-k, then Alg. 2 (H = 1) per slot in rank
// order (Eqs. 36-44). src gives the logits in 16-byte chunks (ColLogits).
// The caller loads the token's home a, location s (Eq. 36: a on the first
// layer) and accumulated loss q. Atab is the delay table of Eq. 38, in
// shared or global memory. The argmin of Eq. 43 packs (fp32 cost bits,
// substitute, away, server, expert) into a 64-bit key and keeps the
// smallest; costs are never negative, so the bit pattern orders them like
// the values.
template <class Src>
__device__ __forceinline__ void select_token(
    int t, const Src& src, int E, int k, int renorm, int M, float qbar,
    const float* Atab, const SelSmem& sm, const float* s_Q, const float* s_Cq, int a, int s, float q,
    uint8_t* __restrict__ loc, float* __restrict__ qhat,
    int32_t* __restrict__ topk_idx, float* __restrict__ topk_w, int32_t* __restrict__ chosen_expert,
    uint8_t* __restrict__ chosen_server, uint8_t* __restrict__ kind_out, int (&kind_count)[4],
    bool topk_only = false) {
  // top-k by (logit desc, index asc): a sorted list of 2, 4, 6 or 8 >= k
  float vtop[ORDERMOE_MAX_TOPK];
  int itop[ORDERMOE_MAX_TOPK];
  const int nc = (E + 3) / 4;
  bool nan;
  if (k <= 2) nan = topk_list<2>(src, nc, vtop, itop);
  else if (k <= 4) nan = topk_list<4>(src, nc, vtop, itop);
  else if (k <= 6) nan = topk_list<6>(src, nc, vtop, itop);
  else nan = topk_list<8>(src, nc, vtop, itop);
  if (nan) {
    report(&g_err_route, ORDERMOE_DEV_NAN_LOGIT, t);
    for (int j = 0; j < k; ++j) {  // no targets: a later pass skips this token
      topk_idx[(size_t)t * k + j] = -1;
      topk_w[(size_t)t * k + j] = 0.0f;
    }
    return;
  }
  // softmax over all E in fp32, summed in index order (the maximum is the
  // list's head; the -inf logits past E add exact zeros after the real
  // terms); gate weights of the k slots
  const float lmax = vtop[0];
  float denom = 0.0f;
#pragma unroll 1
  for (int c4 = 0; c4 < nc; ++c4) {
    const float4 x4 = src.chunk(c4);
    denom += expf(x4.x - lmax);
    denom += expf(x4.y - lmax);
    denom += expf(x4.z - lmax);
    denom += expf(x4.w - lmax);
  }
  float wsel[ORDERMOE_MAX_TOPK];
  float ssel = 0.0f;
#pragma unroll
  for (int j = 0; j < ORDERMOE_MAX_TOPK; ++j)
    if (j < k) {
      wsel[j] = expf(vtop[j] - lmax) / denom;
      ssel += wsel[j];
    }
  int idx[ORDERMOE_MAX_TOPK];
  unsigned long long used_targets = 0;
#pragma unroll
  for (int j = 0; j < ORDERMOE_MAX_TOPK; ++j) {
    idx[j] = itop[j];
    if (j < k) {
      topk_idx[(size_t)t * k + j] = itop[j];
      topk_w[(size_t)t * k + j] = renorm ? wsel[j] / ssel : wsel[j];
      used_targets |= 1ull << itop[j];
    }
  }
  if (topk_only) return;
  // selection
  if (a >= M || s >= M) {
    report(&g_err_route, ORDERMOE_DEV_BAD_INDEX, t);
    return;
  }
  const float* Aas = Atab + (a * M + s) * M;
  unsigned long long taken = used_targets;
  int first_server = s;
  for (int j = 0; j < k; ++j) {
    const int r = idx[j];
    const int nsub = sm.nsub[r];
    unsigned long long best = ~0ull;
    for (int ki = 0; ki <= nsub; ++ki) {
      const int kk = (ki == 0) ? r : sm.sublist[r * 64 + ki - 1];
      const bool sub = (ki != 0);
      float cq = 0.0f;
      if (sub) {
        if ((taken >> kk) & 1ull) continue;
        if (!(__fadd_rn(q, s_Q[r * E + kk]) <= qbar)) continue;  // Eq. 40 budget
        cq = s_Cq[r * E + kk];
      }
      uint32_t pm = sm.pmask[kk];
      while (pm) {
        const int m = __ffs(pm) - 1;
        pm &= pm - 1;
        const float cost = __fadd_rn(Aas[m], cq);
        const unsigned long long key =
            (static_cast<unsigned long long>(__float_as_uint(cost)) << 32) |
            (static_cast<unsigned long long>(sub ? 1u : 0u) << 31) |
            (static_cast<unsigned long long>(m != s ? 1u : 0u) << 30) |
            (static_cast<unsigned long long>(m) << 8) | static_cast<unsigned long long>(kk);
        best = key < best ? key : best;
      }
    }
    int kstar, mstar, kd;
    if (best == ~0ull) {
      report(&g_err_route, ORDERMOE_DEV_NO_CANDIDATE, t);
      kstar = r; mstar = s; kd = 0;
    } else {
      kstar = static_cast<int>(best & 0xFFu);
      mstar = static_cast<int>((best >> 8) & 0xFFu);
      const int sub = static_cast<int>((best >> 31) & 1u);
      const int away = static_cast<int>((best >> 30) & 1u);
      kd = 2 * away + sub;
      if (sub) {
        taken |= 1ull << kstar;
        q = __fadd_rn(q, s_Q[r * E + kstar]);
      }
    }
    if (j == 0) first_server = mstar;
    chosen_expert[(size_t)t * k + j] = kstar;
    chosen_server[(size_t)t * k + j] = static_cast<uint8_t>(mstar);
    kind_out[(size_t)t * k + j] = static_cast<uint8_t>(kd);
    if (kd == 0) ++kind_count[0];  // constant indices: kind_count[] stays in registers
    else if (kd == 1) ++kind_count[1];
    else if (kd == 2) ++kind_count[2];
    else ++kind_count[3];
  }
  if (loc != nullptr) {
    loc[t] = static_cast<uint8_t>(first_server);
    qhat[t] = q;
  }
}

__device__ __forceinline__ void flush_kind_counts(SelSmem& sm, const int (&kind_count)[4],
                                                  int32_t* counters) {
  if (counters == nullptr) return;
  for (int i = 0; i < 4; ++i)
    if (kind_count[i]) atomicAdd(&sm.kind[i], kind_count[i]);
}

// Selection from given logits: one thread per token.
template <int EMAX>
__global__ void __launch_bounds__(128) select_kernel(
    const float* __restrict__ logits_in, int T, int E, int k, int renorm,
    const uint8_t* __restrict__ tab, const uint8_t* __restrict__ home, uint8_t* __restrict__ loc,
    float* __restrict__ qhat, float* __restrict__ logits_out, int32_t* __restrict__ topk_idx,
    float* __restrict__ topk_w, int32_t* __restrict__ chosen_expert,
    uint8_t* __restrict__ chosen_server, uint8_t* __restrict__ kind_out,
    int32_t* __restrict__ counters, Lookahead la) {
  pdl_trigger();  // launched with launch_pdl: no global access before pdl_wait
  pdl_wait();
  __shared__ SelSmem sm;
  extern __shared__ __align__(16) float s_dyn[];
  float4* s_lg = reinterpret_cast<float4*>(s_dyn);  // [EMAX / 4][128] chunks of logits
  float* s_Q = s_dyn + EMAX * 128;
  float* s_Cq = s_Q + E * E;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  // the token's state first: its loads overlap the tables'
  int a = 0, sl = 0;
  float q0 = 0.0f;
  if (t < T && la.H == 1) {
    a = home[t];
    sl = (loc != nullptr) ? loc[t] : a;  // no state given: first layer (Eq. 36)
    q0 = (qhat != nullptr) ? qhat[t] : 0.0f;
  }
  if (!load_tables(tab, E, sm, s_Q, s_Cq)) return;
  const float* Atab = load_delay_range(tab, E, s_Cq + E * E, threadIdx.x, blockDim.x);
  __syncthreads();
  const int M = reinterpret_cast<const int32_t*>(tab)[2];
  const float qbar = reinterpret_cast<const float*>(tab)[5];
  int kind_count[4] = {0, 0, 0, 0};
  if (t < T) {
    float lg[EMAX];
#pragma unroll
    for (int e = 0; e < EMAX; ++e) lg[e] = (e < E) ? logits_in[(size_t)t * E + e] : -INFINITY;
    if (logits_out != nullptr) {
#pragma unroll
      for (int e = 0; e < EMAX; ++e)  // constant indices keep lg[] in registers
        if (e < E) logits_out[(size_t)t * E + e] = lg[e];
    }
#pragma unroll
    for (int c = 0; c < EMAX; c += 4)
      s_lg[(c / 4) * 128 + threadIdx.x] = make_float4(lg[c], lg[c + 1], lg[c + 2], lg[c + 3]);
    select_token(t, ColLogits{s_lg + threadIdx.x}, E, k, renorm, M, qbar, Atab, sm, s_Q, s_Cq,
                 a, sl, q0, loc, qhat, topk_idx, topk_w, chosen_expert, chosen_server,
                 kind_out, kind_count, la.H > 1);
  }
  flush_kind_counts(sm, kind_count, counters);
  __syncthreads();
  if (counters != nullptr && threadIdx.x < 4 && sm.kind[threadIdx.x])
    atomicAdd(&counters[threadIdx.x], sm.kind[threadIdx.x]);
}

// ---------------------------------------------------------------------------
// Alg. 2 with H = 1 from the targets topk_idx, eight lanes per token: for
// each slot the lanes split the target and its substitutes (lane j takes
// candidates j, j + 8, ... of the list), each keeps the smallest 64-bit key
// of select_token (cost bits, substitute, away, server, expert: a total
// order, so the minimum over any split is the same), and three butterfly
// steps over the eight lanes give the slot's argmin to all of them; they
// then update the taken set and the loss identically. Used for many experts,
// where one thread per token walks a long serial chain of candidates.
constexpr int kLaneTokens = 4;   // tokens per warp (eight lanes each)
constexpr int kLaneThreads = 256;

// The slots of one token whose targets are idx, on eight lanes (sub 0 .. 7); Aas:
// its row A[a][s][.] of the delay table (valid when a, s < M). Every lane of the
// warp calls it (the butterflies need them all), inactive tokens (past T, a NaN
// token) write nothing.
__device__ __forceinline__ void select_slots(
    int t, bool active, int sub, const int (&idx)[ORDERMOE_MAX_TOPK], int E, int k, int M, float qbar,
    const float* Aas, const SelSmem& sm, const float* s_Q, const float* s_Cq, int a, int s, float q,
    uint8_t* __restrict__ loc, float* __restrict__ qhat, int32_t* __restrict__ chosen_expert,
    uint8_t* __restrict__ chosen_server, uint8_t* __restrict__ kind_out, int (&kind_count)[4]) {
  unsigned long long taken = 0;
#pragma unroll
  for (int j = 0; j < ORDERMOE_MAX_TOPK; ++j)
    if (j < k && active) {
      if (idx[j] < 0 || idx[j] >= E) active = false;
      else taken |= 1ull << idx[j];
    }
  if (active && (a >= M || s >= M)) {
    if (sub == 0) report(&g_err_route, ORDERMOE_DEV_BAD_INDEX, t);
    active = false;
  }
  int first_server = s;
#pragma unroll
  for (int j = 0; j < ORDERMOE_MAX_TOPK; ++j) {
    if (j >= k) break;  // k is the same for every lane
    const int r = idx[j];
    const int nsub = active ? sm.nsub[r] : -1;
    unsigned long long best = ~0ull;
    for (int ki = sub; ki <= nsub; ki += 8) {
      const int kk = (ki == 0) ? r : sm.sublist[r * 64 + ki - 1];
      const bool issub = (ki != 0);
      float cq = 0.0f;
      if (issub) {
        if ((taken >> kk) & 1ull) continue;
        if (!(__fadd_rn(q, s_Q[r * E + kk]) <= qbar)) continue;  // Eq. 40 budget
        cq = s_Cq[r * E + kk];
      }
      uint32_t pm = sm.pmask[kk];
      while (pm) {
        const int m = __ffs(pm) - 1;
        pm &= pm - 1;
        const float cost = __fadd_rn(Aas[m], cq);
        const unsigned long long key =
            (static_cast<unsigned long long>(__float_as_uint(cost)) << 32) |
            (static_cast<unsigned long long>(issub ? 1u : 0u) << 31) |
            (static_cast<unsigned long long>(m != s ? 1u : 0u) << 30) |
            (static_cast<unsigned long long>(m) << 8) | static_cast<unsigned long long>(kk);
        best = key < best ? key : best;
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
      best = other < best ? other : best;
    }
    if (!active) continue;
    int kstar, mstar, kd;
    if (best == ~0ull) {
      if (sub == 0) report(&g_err_route, ORDERMOE_DEV_NO_CANDIDATE, t);
      kstar = r; mstar = s; kd = 0;
    } else {
      kstar = static_cast<int>(best & 0xFFu);
      mstar = static_cast<int>((best >> 8) & 0xFFu);
      const int bsub = static_cast<int>((best >> 31) & 1u);
      const int away = static_cast<int>((best >> 30) & 1u);
      kd = 2 * away + bsub;
      if (bsub) {
        taken |= 1ull << kstar;
        q = __fadd_rn(q, s_Q[r * E + kstar]);
      }
    }
    if (j == 0) first_server = mstar;
    if (sub == 0) {
      chosen_expert[(size_t)t * k + j] = kstar;
      chosen_server[(size_t)t * k + j] = static_cast<uint8_t>(mstar);
      kind_out[(size_t)t * k + j] = static_cast<uint8_t>(kd);
      if (kd == 0) ++kind_count[0];  // constant indices: kind_count[] stays in registers
      else if (kd == 1) ++kind_count[1];
      else if (kd == 2) ++kind_count[2];
      else ++kind_count[3];
    }
  }
  if (active && sub == 0 && loc != nullptr) {
    loc[t] = static_cast<uint8_t>(first_server);
    qhat[t] = q;
  }
}

__global__ void __launch_bounds__(kLaneThreads) select_lanes_kernel(
    const int32_t* __restrict__ topk_idx, int T, int E, int k, const uint8_t* __restrict__ tab,
    const uint8_t* __restrict__ home, uint8_t* __restrict__ loc, float* __restrict__ qhat,
    int32_t* __restrict__ chosen_expert, uint8_t* __restrict__ chosen_server,
    uint8_t* __restrict__ kind_out, int32_t* __restrict__ counters) {
  pdl_trigger();  // launched with launch_pdl: no global access before pdl_wait
  pdl_wait();
  __shared__ SelSmem sm;
  extern __shared__ __align__(16) float s_dyn[];
  float* s_Q = s_dyn;
  float* s_Cq = s_dyn + E * E;
  if (!load_tables(tab, E, sm, s_Q, s_Cq)) return;
  // the delay table stays in global memory here: staging it took longer
  // than the reads it saves (one per candidate, eight lanes at a time)
  const float* Atab = reinterpret_cast<const float*>(tab + off_a(E));
  __syncthreads();
  const int M = reinterpret_cast<const int32_t*>(tab)[2];
  const float qbar = reinterpret_cast<const float*>(tab)[5];
  const int lane = threadIdx.x & 31;
  const int sub = lane & 7;       // lane within the token's group of eight
  const int grp = lane >> 3;
  const int warps_total = gridDim.x * (kLaneThreads / 32);
  int kind_count[4] = {0, 0, 0, 0};
  for (int base = (blockIdx.x * (kLaneThreads / 32) + (threadIdx.x >> 5)) * kLaneTokens; base < T;
       base += warps_total * kLaneTokens) {
    const int t = base + grp;
    const bool active = t < T;
    // the token's state and targets, loaded together
    int a = 0, s = 0;
    float q = 0.0f;
    if (active) {
      a = home[t];
      s = (loc != nullptr) ? loc[t] : a;
      q = (qhat != nullptr) ? qhat[t] : 0.0f;
    }
    int idx[ORDERMOE_MAX_TOPK];
#pragma unroll
    for (int j = 0; j < ORDERMOE_MAX_TOPK; ++j) idx[j] = (j < k && active) ? topk_idx[(size_t)t * k + j] : 0;
    const float* Aas = Atab + (active && a < M && s < M ? (a * M + s) * M : 0);
    select_slots(t, active, sub, idx, E, k, M, qbar, Aas, sm, s_Q, s_Cq, a, s, q, loc, qhat,
                 chosen_expert, chosen_server, kind_out, kind_count);
  }
  flush_kind_counts(sm, kind_count, counters);
  __syncthreads();
  if (counters != nullptr && threadIdx.x < 4 && sm.kind[threadIdx.x])
    atomicAdd(&counters[threadIdx.x], sm.kind[threadIdx.x]);
}

// ---------------------------------------------------------------------------
// Alg. 2 with horizon H = D + 1 > 1 (Eq. 43) from the targets topk_idx.
//
// Phi^(D)(m, kx, q) depends on the token through its home a and its loss q
// only, and on q only through the budget checks it makes. Level d counts the
// layers left (d = D: the next layer, d = 1: the last one looked at), and
//   Phi^(d)(m, kx, q) = sum over k' of P(kx -> k') V^(d)_q(m, k'),
//   V^(d)_q(m, k')    = min over the feasible (m', k'') of target k' of
//                       A[a][m][m'] + Cq[k'][k''] + Phi^(d-1)(m', k'', q'),
// where V does not depend on kx. So a block takes tokens of one home and
// builds, once, Phi^(d) for the two cases that most losses fall into: every
// check below passes (Ua) and every check fails (Un, exact experts only).
//   all pass: q plus the largest loss of each level in turn stays within Qbar;
//   all fail: at every level q plus its smallest loss exceeds Qbar.
// Both follow for every check from these because fadd is monotone and losses
// are not negative, so the table holds the same fp32 value as the recursion,
// which adds its terms in ascending k' as the tables do. A candidate in
// neither case is listed and evaluated by a warp, k' over the lanes (with more
// levels and experts by the block, k' and its substitutes over the threads),
// with the tables read again one level down. V_q itself is read from rows that hold, for each
// target and server, the minima over its substitutes in order of loss (the
// ones that fit are a prefix of that order); a pair in neither case one level
// down is evaluated by its lane, unless the bounds Ua <= Phi <= Un already
// show that it cannot be the minimum.
//
// A warp a token and slot, blocks of NW warps; the block finds its home and
// tokens by ranking home[] (every block ranks the same way, so the blocks
// partition the tokens without scratch memory or a sort kernel).
//
// Bound: latency. A block's set-up is a chain of L2 reads and block barriers,
// a slot's argmin a chain of shared-memory reads, and a token whose loss falls
// between the two cases slot after slot would end the launch long after the
// rest (one warp takes 40 us for such an evaluation at H = 3), so the tokens
// of a block go slot by slot and all its warps share what is open.
// One block a token, with the tables rebuilt for each and V folded into every
// term, took 15.7 ms for 2048 tokens of 64 experts, 8 servers, top-6, H = 3,
// and 14.6 us for 128 tokens of 8 experts, 4 servers, top-2 (ncu); this takes
// 84 us and 11.5 us (351 us with every token's evaluations left to its warp).
constexpr int kLaMaxTok = 512;   // tokens of a block
constexpr int kLaTasks = 512;    // evaluations listed in a step
// Losses of the last level that the class table takes: 37 KB at 64 experts, beside
// which the rows of groups of 8 on 8 servers fit at H = 3 (beside a table for 1024,
// 74 KB, they do not). Where the rows or the classes have no room the open
// evaluations go by direct minima. Calls with logits given, 2048 tokens of 64
// experts: H = 3, 8 servers, groups of 4 103 us and of 8 157 (in the tables), of 16
// 72 ms; groups of 8 on 16 servers 14.9 ms, on 32 12.2; H = 2, groups of 16, 52 us
// on 8 servers, 85 on 32. (One block a token: 10.2, 27.4, 108, 28.4, 30.6, 3.7 and
// 2.3 ms.)
constexpr int kLaMaxLoss = 512;
// Up to 16 experts a block has 8 warps and no class table: its set-up (2 us)
// is longer than the few evaluations it would shorten (14.5 against 12.4 us
// for 128 tokens of 8 experts). For 64 experts the table took the 2048-token
// call above from 4620 to 351 us, a token's evaluations still one after another.
constexpr int kLaNarrow = 16;
// bytes of a class's row of counts, one a target: an odd number of words, so
// that lanes reading one word of different rows hit distinct banks
__host__ __device__ inline int la_class_pitch(int E) { return 4 * (((E + 3) / 4) | 1); }
__host__ __device__ inline int la_max_loss(int E) {
  return E <= kLaNarrow ? 0 : E * (E - 1) < kLaMaxLoss ? E * (E - 1) : kLaMaxLoss;
}

// A level's tables in global memory (layout in ordermoe.h).
struct LaLevel {
  const uint32_t* pmask;
  const unsigned long long* subst;
  const float* Q;
  const float* Cq;
  const float* A;  // home a's [M][M]
};

__device__ __forceinline__ LaLevel la_level(const uint8_t* tab, int E, int M, int a) {
  LaLevel v;
  v.pmask = reinterpret_cast<const uint32_t*>(tab + kOffPmask);
  v.subst = reinterpret_cast<const unsigned long long*>(tab + kOffSubst);
  v.Q = reinterpret_cast<const float*>(tab + kOffQtab);
  v.Cq = reinterpret_cast<const float*>(tab + off_cq(E));
  v.A = reinterpret_cast<const float*>(tab + off_a(E)) + (size_t)a * M * M;
  return v;
}

// Everything the evaluation of Phi reads: dynamic shared memory and the
// levels' tables. Index d - 1 is level d. A level's rows: for target k' the
// exact expert, then its n substitutes in order of loss (equal losses by
// expert), M entries each, at woff[k'].
template <int D>
struct LaCtx {
  int E, M, pitch;      // pitch: of P and sQ rows (odd: lanes down a column hit distinct banks)
  float qbar;
  LaLevel lev[D];
  const float* P[D];    // shared [E][pitch]
  const float* Ua[D];   // shared [M][E]: Phi^(d), every check passing
  const float* Un[D];   //                         every check failing
  float qmax[D], qmin[D];
  bool has[D];          // the level has substitutes at all
  bool prune;           // no transition is negative: Phi lies between Ua and Un
  bool rows;            // the rows below fit in shared memory
  const float* sQ[D];   // shared [E][pitch]: the losses of each target's substitutes, ascending
  const float* Wa[D];   // shared rows: minima over the row's entries so far, Phi^(d-1) from Ua
  const float* Cn[D];   // shared rows (d > 1): each entry alone, Phi^(d-1) from Un
  const int* woff[D];
  const int* nsub[D];
  const uint8_t* ord[D];  // shared [E][64]: the substitutes in that order
  // level 1's losses of all targets in ascending order, and for every number
  // of them that fit (the class of a loss q) how many of each target's do
  bool classes;
  int n_loss;
  const float* loss;
  const uint8_t* fits;  // [n_loss + 1][la_class_pitch(E)]
};

// every budget check of levels d .. 1 passes for a loss of q
template <int D>
__device__ __forceinline__ bool la_all(const LaCtx<D>& c, int d, float q) {
#pragma unroll
  for (int i = D - 1; i >= 0; --i)
    if (i < d && c.has[i]) {
      q = __fadd_rn(q, c.qmax[i]);
      if (!(q <= c.qbar)) return false;
    }
  return true;
}
// every budget check of levels d .. 1 fails for a loss of q
template <int D>
__device__ __forceinline__ bool la_none(const LaCtx<D>& c, int d, float q) {
#pragma unroll
  for (int i = D - 1; i >= 0; --i)
    if (i < d && c.has[i] && __fadd_rn(q, c.qmin[i]) <= c.qbar) return false;
  return true;
}

template <int D, int d>
__device__ __forceinline__ float la_phi(const LaCtx<D>& c, int m, int kx, float q);

// V^(d)_q(m, kt). From the rows: the substitutes whose deeper checks all pass
// are a prefix of the row (and the exact expert with them, its loss being
// smaller), those that fit at all a longer one. A pair in neither case is
// evaluated unless its cost cannot be the minimum: Phi^(d-1) lies between Ua
// and Un, since every operation of the recursion is monotone.
template <int D, int d>
__device__ __forceinline__ float la_value(const LaCtx<D>& c, int m, int kt, float q) {
  const LaLevel& v = c.lev[d - 1];
  float best = INFINITY;
  if (c.rows) {
    const float* s = c.sQ[d - 1] + kt * c.pitch;
    const float* wa = c.Wa[d - 1] + c.woff[d - 1][kt] + m;
    const int n = c.nsub[d - 1][kt];
    if constexpr (d == 1) {
      int lo = 0, hi = n;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__fadd_rn(q, s[mid]) <= c.qbar) lo = mid + 1;
        else hi = mid;
      }
      return wa[lo * c.M];
    } else {
      const float* cn = c.Cn[d - 1] + c.woff[d - 1][kt] + m;
      int na = 0, first = n + 1, last = -1;  // entries of neither case lie in first .. last
      float bound = INFINITY;                // some entry's cost is at most this
      for (int i = 0; i <= n; ++i) {
        const float q2 = i == 0 ? q : __fadd_rn(q, s[i - 1]);
        if (i > 0 && !(q2 <= c.qbar)) break;
        if (la_all<D>(c, d - 1, q2)) {
          na = i + 1;
          continue;
        }
        const float x = cn[i * c.M];
        if (la_none<D>(c, d - 1, q2)) {
          best = fminf(best, x);
        } else {
          bound = fminf(bound, x);
          first = min(first, i);
          last = i;
        }
      }
      if (na > 0) best = fminf(best, wa[(na - 1) * c.M]);
      for (int i = first; i <= last; ++i) {
        const float q2 = i == 0 ? q : __fadd_rn(q, s[i - 1]);
        const int kk = i == 0 ? kt : c.ord[d - 1][kt * 64 + i - 1];
        const float cq = i == 0 ? 0.0f : v.Cq[kt * c.E + kk];
        for (uint32_t pm = v.pmask[kk]; pm; pm &= pm - 1) {
          const int m2 = __ffs(pm) - 1;
          const float base = __fadd_rn(v.A[m * c.M + m2], cq);
          const float least = __fadd_rn(base, c.Ua[d - 2][m2 * c.E + kk]);
          if (c.prune && (least >= best || least > bound)) continue;
          best = fminf(best, __fadd_rn(base, la_phi<D, d - 1>(c, m2, kk, q2)));
        }
      }
      return best;
    }
  }
  unsigned long long cand = v.subst[kt] | (1ull << kt);
  while (cand) {
    const int kk = __ffsll(static_cast<long long>(cand)) - 1;
    cand &= cand - 1;
    float cq = 0.0f, q2 = q;
    if (kk != kt) {
      q2 = __fadd_rn(q, v.Q[kt * c.E + kk]);
      if (!(q2 <= c.qbar)) continue;
      cq = v.Cq[kt * c.E + kk];
    }
    for (uint32_t pm = v.pmask[kk]; pm; pm &= pm - 1) {
      const int m2 = __ffs(pm) - 1;
      float cost = __fadd_rn(v.A[m * c.M + m2], cq);
      if constexpr (d > 1) cost = __fadd_rn(cost, la_phi<D, d - 1>(c, m2, kk, q2));
      best = fminf(best, cost);
    }
  }
  return best;
}

// The class of a loss of q: how many of level 1's losses fit.
template <int D>
__device__ __forceinline__ int la_class(const LaCtx<D>& c, float q) {
  int lo = 0, hi = c.n_loss;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (__fadd_rn(q, c.loss[mid]) <= c.qbar) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}
// Phi^(1)(m, kx, .) of a loss of class cl, from the counts of substitutes that
// fit, four targets' counts and row offsets a load (with the class found once an
// entry 166 -> 139 us for 2048 tokens of 64 experts whose worst token has many).
template <int D>
__device__ __forceinline__ float la_phi_class(const LaCtx<D>& c, int m, int kx, int cl) {
  const float* Pr = c.P[0] + kx * c.pitch;
  const uint8_t* fits = c.fits + cl * la_class_pitch(c.E);
  const float* wa = c.Wa[0] + m;
  float acc = 0.0f;
#pragma unroll 2
  for (int k4 = 0; k4 < c.E; k4 += 4) {
    const uint32_t n4 = *reinterpret_cast<const uint32_t*>(fits + k4);
    const int4 w4 = *reinterpret_cast<const int4*>(c.woff[0] + k4);
    const int w[4] = {w4.x, w4.y, w4.z, w4.w};
    float p[4], x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool real = k4 + u < c.E;
      p[u] = real ? Pr[k4 + u] : 0.0f;
      x[u] = real ? wa[w[u] + static_cast<int>((n4 >> (8 * u)) & 0xFFu) * c.M] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p[u] != 0.0f) acc = __fadd_rn(acc, __fmul_rn(p[u], x[u]));
  }
  return acc;
}

// Phi^(d)(m, kx, q) by one thread
template <int D, int d>
__device__ __forceinline__ float la_phi(const LaCtx<D>& c, int m, int kx, float q) {
  if (la_all<D>(c, d, q)) return c.Ua[d - 1][m * c.E + kx];
  if (la_none<D>(c, d, q)) return c.Un[d - 1][m * c.E + kx];
  if (d == 1 && c.rows && c.classes) return la_phi_class<D>(c, m, kx, la_class<D>(c, q));
  const float* Pr = c.P[d - 1] + kx * c.pitch;
  float acc = 0.0f;
  for (int kt = 0; kt < c.E; ++kt) {
    const float p = Pr[kt];
    if (p != 0.0f) acc = __fadd_rn(acc, __fmul_rn(p, la_value<D, d>(c, m, kt, q)));
  }
  return acc;
}

// Phi^(D)(m, kx, q) by the whole warp, k' over the lanes; the same value in
// every lane. The terms are added in ascending k' (a term with P = 0 adds an
// exact 0, which leaves the sum as it is). term: 64 floats of the warp's own.
template <int D>
__device__ __forceinline__ float la_phi_warp(const LaCtx<D>& c, float* term, int lane, int m, int kx,
                                             float q) {
  const float* Prow = c.P[D - 1] + kx * c.pitch;
#pragma unroll 1
  for (int kt = lane; kt < 64; kt += 32) {
    const float p = kt < c.E ? Prow[kt] : 0.0f;
    term[kt] = p != 0.0f ? __fmul_rn(p, la_value<D, D>(c, m, kt, q)) : 0.0f;
  }
  __syncwarp();
  float acc = 0.0f;
  const float4* t4 = reinterpret_cast<const float4*>(term);
#pragma unroll 4
  for (int i = 0; i < (c.E + 3) / 4; ++i) {
    const float4 x = t4[i];
    acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc, x.x), x.y), x.z), x.w);
  }
  __syncwarp();  // the terms are rewritten by the next evaluation
  return acc;
}

// V^(D)_q(m, kt) by `width` neighbouring lanes (a power of two), lane `sub` of
// them taking every width-th substitute; the same value in all of them. Called
// by whole warps. (The minimum does not depend on the order.)
template <int D>
__device__ __forceinline__ float la_value_lanes(const LaCtx<D>& c, int m, int kt, float q, int sub,
                                                int width) {
  auto all_min = [&](float x) {
    for (int o = width >> 1; o; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
  };
  const LaLevel& v = c.lev[D - 1];
  float best = INFINITY;
  // entry i of the target's row: expert kk at a loss of q2
  auto entry = [&](int kk, float cq, float q2, float bound) {
    const bool by_class = D == 2 && c.rows && c.classes;  // (the entry is in neither case)
    const int cl = by_class ? la_class<D>(c, q2) : 0;
#pragma unroll 1
    for (uint32_t pm = v.pmask[kk]; pm; pm &= pm - 1) {
      const int m2 = __ffs(pm) - 1;
      const float base = __fadd_rn(v.A[m * c.M + m2], cq);
      const float least = __fadd_rn(base, c.Ua[D - 2][m2 * c.E + kk]);
      if (c.prune && (least >= best || least > bound)) continue;
      const float phi = by_class ? la_phi_class<D>(c, m2, kk, cl) : la_phi<D, D - 1>(c, m2, kk, q2);
      best = fminf(best, __fadd_rn(base, phi));
    }
  };
  if (c.rows) {
    const float* s = c.sQ[D - 1] + kt * c.pitch;
    const float* wa = c.Wa[D - 1] + c.woff[D - 1][kt] + m;
    const float* cn = c.Cn[D - 1] + c.woff[D - 1][kt] + m;
    const int n = c.nsub[D - 1][kt];
    unsigned long long neither = 0;  // of this lane's entries
    float bound = INFINITY;          // some entry's cost is at most this
    int na = 0;
    for (int i = sub; i <= n; i += width) {
      const float q2 = i == 0 ? q : __fadd_rn(q, s[i - 1]);
      if (i > 0 && !(q2 <= c.qbar)) break;
      if (la_all<D>(c, D - 1, q2)) {
        na = i + 1;
      } else if (la_none<D>(c, D - 1, q2)) {
        best = fminf(best, cn[i * c.M]);
      } else {
        bound = fminf(bound, cn[i * c.M]);
        neither |= 1ull << i;
      }
    }
    if (na > 0) best = fminf(best, wa[(na - 1) * c.M]);
    best = all_min(best);
    bound = all_min(bound);
#pragma unroll 1
    for (; neither; neither &= neither - 1) {
      const int i = __ffsll(static_cast<long long>(neither)) - 1;
      const int kk = i == 0 ? kt : c.ord[D - 1][kt * 64 + i - 1];
      entry(kk, i == 0 ? 0.0f : v.Cq[kt * c.E + kk], i == 0 ? q : __fadd_rn(q, s[i - 1]), bound);
    }
  } else {
    int i = 0;
#pragma unroll 1
    for (unsigned long long sb = v.subst[kt] | (1ull << kt); sb; sb &= sb - 1, ++i) {
      if ((i & (width - 1)) != sub) continue;
      const int kk = __ffsll(static_cast<long long>(sb)) - 1;
      const float q2 = kk == kt ? q : __fadd_rn(q, v.Q[kt * c.E + kk]);
      if (kk != kt && !(q2 <= c.qbar)) continue;
      entry(kk, kk == kt ? 0.0f : v.Cq[kt * c.E + kk], q2, INFINITY);
    }
  }
  return all_min(best);
}

// Dynamic shared memory for M servers and NW warps: what every block needs, the
// class table, and the levels' rows where none is shorter than it can be (Wa of
// every level, Cn of all but the last).
__host__ __device__ constexpr size_t la_smem_fixed(int E, int D, int M, int NW) {
  return sizeof(float) * ((size_t)64 * NW + 2 * D * E * (E | 1) + (size_t)(2 * D + 2) * M * E);
}
__host__ __device__ inline size_t la_smem_classes(int E) {
  return la_max_loss(E) == 0 ? 0
                             : sizeof(float) * la_max_loss(E) + (size_t)(la_max_loss(E) + 1) * la_class_pitch(E);
}
__host__ __device__ inline size_t la_smem_rows(int E, int D, int M) {
  return sizeof(float) * (size_t)(2 * D - 1) * E * ((E * M) | 1);
}
// The most a block asks for: the launch gives what the servers that the table
// stride has room for can use, up to this, and the block lays it out for the
// servers that there are: the class table where it fits beside the fixed part,
// the rows in what is left where theirs fit.
constexpr size_t kLaSmem = 200 * 1024;
constexpr size_t kLaStatic = 27 * 1024;  // of the 227 KB a block can have; checked at the first launch
static_assert(la_smem_fixed(64, 3, 32, 16) <= kLaSmem && kLaSmem + kLaStatic <= 227 * 1024,
              "every shape that is taken can be launched");

template <int D, int NW>
__global__ void __launch_bounds__(32 * NW, 1) lookahead_select_kernel(
    const int32_t* __restrict__ topk_idx, int t0, int T, int E, int k, const uint8_t* __restrict__ tab,
    Lookahead la, int Mcap, int smem, int tpb, const uint8_t* __restrict__ home,
    uint8_t* __restrict__ loc, float* __restrict__ qhat, int32_t* __restrict__ chosen_expert,
    uint8_t* __restrict__ chosen_server, uint8_t* __restrict__ kind_out,
    int32_t* __restrict__ counters) {
  constexpr int kThreads = 32 * NW;
  constexpr int kEmax = NW > 8 ? 64 : kLaNarrow;    // experts that this many warps take
  constexpr int kRowsPer = (kEmax + NW - 1) / NW;   // rows of a level a warp
  constexpr int kElems = (kEmax * kEmax + kThreads - 1) / kThreads;  // elements of P a thread
  pdl_trigger();  // launched with launch_pdl: no global access before pdl_wait
  pdl_wait();
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ uint8_t s_ord[D][64 * 64];
  // the losses' ranks while the tables are built, then the listed evaluations
  __shared__ __align__(16) unsigned char s_scratch[64 * 64 * 2];
  static_assert(sizeof(uint4) * kLaTasks <= sizeof(s_scratch), "task list");
  uint16_t* s_rank = reinterpret_cast<uint16_t*>(s_scratch);
  uint4* s_task = reinterpret_cast<uint4*>(s_scratch);  // cost0, q, key's low word, warp
  __shared__ unsigned long long s_best[NW];
  __shared__ float s_As[NW][32];  // a warp's own row of A
  __shared__ int s_task_n[2][2];
  __shared__ int s_cnt[32], s_nsub[D][64], s_tok[kLaMaxTok];
  __shared__ __align__(16) int s_woff[D][68];
  __shared__ int s_part[NW], s_kind[4];
  __shared__ int s_home, s_chunk, s_qmax[D], s_qmin[D];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t* hdr = reinterpret_cast<const int32_t*>(tab);
  const int M = hdr[2];
  const float qbar = reinterpret_cast<const float*>(tab)[5];
  if (hdr[1] != E || E > kEmax || M <= 0 || M > Mcap) {
    if (blockIdx.x == 0 && tid == 0) report(&g_err_route, ORDERMOE_DEV_BAD_INDEX, -1);
    return;
  }
  // ---- this block's home and tokens: home a has ceil(count / tpb) blocks
  if (tid < 32) s_cnt[tid] = 0;
  if (tid < 4) {
    s_kind[tid] = 0;
    s_task_n[tid >> 1][tid & 1] = 0;
  }
  if (tid < D) {
    s_qmax[tid] = -1;  // no substitute (losses are not negative: their bits order like values)
    s_qmin[tid] = 0x7FFFFFFF;
  }
  LaCtx<D> c;
  c.E = E;
  c.M = M;
  c.pitch = E | 1;
  c.qbar = qbar;
  float* sp = reinterpret_cast<float*>(s_raw);
  float* s_term = sp + 64 * warp;
  sp += 64 * NW;
  float *U[2 * D], *Wa[D], *Cn[D];
  bool bad_p = false;
  float* sQ[D];
  float pv[D][kElems];  // every load in flight before the first store
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const float* g = la.P + (size_t)(D - 1 - i) * E * E;
#pragma unroll
    for (int u = 0; u < kElems; ++u) {
      const int x = tid + u * kThreads;
      pv[i][u] = x < E * E ? g[x] : 0.0f;
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    // level i + 1: layer l + D - i, entered from the layer before it by P_{l + D - i - 1}
#pragma unroll
    for (int u = 0; u < kElems; ++u) {
      const int x = tid + u * kThreads;
      if (x >= E * E) break;
      sp[x + (x / E) * (c.pitch - E)] = pv[i][u];
      bad_p |= !(pv[i][u] >= 0.0f);
    }
    c.P[i] = sp;
    sp += E * c.pitch;
    c.sQ[i] = sQ[i] = sp;
    sp += E * c.pitch;
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    c.Ua[i] = U[2 * i] = sp;
    c.Un[i] = U[2 * i + 1] = sp + M * E;
    sp += 2 * M * E;
  }
  float* Va = sp;
  float* Vn = Va + M * E;
  sp = Vn + M * E;
  // what is left: the class table, then rows of wcap floats
  const int left = smem - static_cast<int>(la_smem_fixed(E, D, M, NW));
  const int class_bytes = static_cast<int>(la_smem_classes(E));
  const bool class_room = kEmax > kLaNarrow && class_bytes > 0 && class_bytes <= left;
  const int wcap = (left - (class_room ? class_bytes : 0)) / ((2 * D - 1) * static_cast<int>(sizeof(float)));
#pragma unroll
  for (int i = 0; i < D; ++i) {
    c.Wa[i] = Wa[i] = sp;
    sp += wcap;
    c.Cn[i] = Cn[i] = nullptr;
    if (i > 0) {
      c.Cn[i] = Cn[i] = sp;
      sp += wcap;
    }
    c.woff[i] = s_woff[i];
    c.nsub[i] = s_nsub[i];
    c.ord[i] = s_ord[i];
  }
  float* s_loss = sp;
  uint8_t* s_fits = reinterpret_cast<uint8_t*>(sp + la_max_loss(E));
  c.loss = s_loss;
  c.fits = s_fits;
  __syncthreads();
  // thread i looks at tokens i, i + kThreads, ..., kScan of them loaded at a time
  constexpr int kScan = 8;
  auto scan_homes = [&](auto&& take) {
    for (int b = 0; b < T; b += kScan * kThreads) {
      int h[kScan];
#pragma unroll
      for (int u = 0; u < kScan; ++u) {
        const int t = b + u * kThreads + tid;
        h[u] = t < T ? home[t] : -1;
      }
#pragma unroll
      for (int u = 0; u < kScan; ++u) {
        if (b + u * kThreads >= T) break;  // the same for the block
        take(b + u * kThreads + tid, h[u]);
      }
    }
  };
  scan_homes([&](int t, int a) {
    const unsigned peers = __match_any_sync(0xffffffffu, a);
    if (a >= 0 && a < M && lane == __ffs(peers) - 1) atomicAdd(&s_cnt[a], __popc(peers));
    if (a >= M && blockIdx.x == 0) report(&g_err_route, ORDERMOE_DEV_BAD_INDEX, t0 + t);
  });
  __syncthreads();
  if (warp == 0) {
    const int nb = lane < M ? (s_cnt[lane] + tpb - 1) / tpb : 0;
    int incl = nb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    const int b = static_cast<int>(blockIdx.x);
    const unsigned here = __ballot_sync(0xffffffffu, b >= incl - nb && b < incl);
    if (here == 0) {
      if (lane == 0) s_home = -1;
    } else if (lane == __ffs(here) - 1) {
      s_home = lane;
      s_chunk = b - (incl - nb);
    }
  }
  __syncthreads();
  const int a = s_home;
  if (a < 0) return;  // more blocks than the homes need
  const int lo = s_chunk * tpb;
  const int ntok = min(tpb, s_cnt[a] - lo);
  int mine = 0;
  scan_homes([&](int, int h) { mine += h == a ? 1 : 0; });
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_part[warp] = incl;

  // ---- the tables of home a. A warp a row: the losses in order, their extremes.
  // The rows' sets are loaded together, then their losses.
  {
    unsigned long long sets[D][kRowsPer];
    int loss0[D][kRowsPer], loss1[D][kRowsPer];
#pragma unroll
    for (int i = 0; i < D; ++i) {
      c.lev[i] = la_level(tab + (size_t)(D - i) * la.stride, E, M, a);
#pragma unroll
      for (int u = 0; u < kRowsPer; ++u) {
        const int kt = warp + u * NW;
        sets[i][u] = kt < E ? c.lev[i].subst[kt] : 0ull;
      }
    }
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int u = 0; u < kRowsPer; ++u) {
        const float* Q = c.lev[i].Q + (warp + u * NW) * E;
        loss0[i][u] = (sets[i][u] >> lane) & 1ull ? __float_as_int(Q[lane]) : -1;
        loss1[i][u] = kEmax > 32 && ((sets[i][u] >> (lane + 32)) & 1ull) ? __float_as_int(Q[lane + 32]) : -1;
      }
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int u = 0; u < kRowsPer; ++u) {
        const int kt = warp + u * NW;
        if (kt >= E) break;
        const unsigned long long sb = sets[i][u];
        if (lane == 0) s_nsub[i][kt] = __popcll(sb);
        if (sb == 0ull) continue;
        const int q0 = loss0[i][u], q1 = loss1[i][u];
        const int mx = __reduce_max_sync(0xffffffffu, max(q0, q1));
        const unsigned mn = __reduce_min_sync(0xffffffffu, min(static_cast<unsigned>(q0), static_cast<unsigned>(q1)));
        if (lane == 0) {
          atomicMax(&s_qmax[i], mx);
          atomicMin(&s_qmin[i], static_cast<int>(mn));
        }
        int r0 = 0, r1 = 0;
        for (unsigned long long b = sb; b; b &= b - 1) {
          const int e = __ffsll(static_cast<long long>(b)) - 1;
          const int o = __shfl_sync(0xffffffffu, e < 32 ? q0 : q1, e & 31);
          r0 += (o < q0 || (o == q0 && e < lane)) ? 1 : 0;
          r1 += (o < q1 || (o == q1 && e < lane + 32)) ? 1 : 0;
        }
        if (q0 >= 0) {
          sQ[i][kt * c.pitch + r0] = __int_as_float(q0);
          s_ord[i][kt * 64 + r0] = static_cast<uint8_t>(lane);
        }
        if (q1 >= 0) {
          sQ[i][kt * c.pitch + r1] = __int_as_float(q1);
          s_ord[i][kt * 64 + r1] = static_cast<uint8_t>(lane + 32);
        }
      }
  }
  __syncthreads();
  {  // the tokens of this block, by their rank among home a's
    int rank = incl - mine;
    for (int i = 0; i < warp; ++i) rank += s_part[i];
    scan_homes([&](int t, int h) {
      if (h != a) return;
      if (rank >= lo && rank < lo + ntok) s_tok[rank - lo] = t;
      ++rank;
    });
  }
  // The classes of level 1: every loss is put at its rank among all of them
  // (equal losses by target and place), read as one list, which lies where the
  // counts go once all ranks are known. (A row of counts between equal losses
  // is never asked for: both fit or neither does.)
  int first0, first1;  // where targets 2 lane and 2 lane + 1 start in the list
  {
    const int n0 = 2 * lane < E ? s_nsub[0][2 * lane] : 0;
    const int n1 = 2 * lane + 1 < E ? s_nsub[0][2 * lane + 1] : 0;
    int in = n0 + n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, in, o);
      if (lane >= o) in += u;
    }
    first0 = in - n0 - n1;
    first1 = in - n1;
    c.n_loss = __shfl_sync(0xffffffffu, in, 31);
    c.classes = class_room && c.n_loss > 0 && c.n_loss <= la_max_loss(E);
  }
  auto first_of = [&](int kt) { return __shfl_sync(0xffffffffu, kt & 1 ? first1 : first0, kt >> 1); };
  if (c.classes) {
    float* list = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(s_fits) + 15) & ~uintptr_t(15));
    for (int kt = warp; kt < E; kt += NW) {
      const int f = first_of(kt);
      for (int n = lane; n < s_nsub[0][kt]; n += 32) list[f + n] = c.sQ[0][kt * c.pitch + n];
    }
    if (tid < 4) list[c.n_loss + tid] = __int_as_float(0x7FFFFFFF);  // the last four's rest: after every loss
    __syncthreads();
    for (int x = tid; x < c.n_loss; x += kThreads) {
      // losses are not negative: their bits order like values. Before the four
      // that hold x an equal loss counts, after them it does not.
      const int q = __float_as_int(list[x]), x4 = x & ~3;
      const int4* l4 = reinterpret_cast<const int4*>(list);
      int r = 0;
#pragma unroll 4
      for (int y = 0; y < c.n_loss; y += 4) {
        const int4 o = l4[y >> 2];
        const int below = y < x4 ? q + 1 : q;
        r += (o.x < below ? 1 : 0) + (o.y < below ? 1 : 0) + (o.z < below ? 1 : 0) + (o.w < below ? 1 : 0);
      }
      for (int y = x4; y < x; ++y) r += __float_as_int(list[y]) == q ? 1 : 0;
      s_loss[r] = __int_as_float(q);
      s_rank[x] = static_cast<uint16_t>(r);
    }
  }
  // where each target's row starts: (1 + substitutes) M entries, an odd length
  // (rows of equal length start in distinct banks), two targets a lane
  if (warp < D) {
    int* off = s_woff[warp];
    const int* ns = s_nsub[warp];
    const int n0 = 2 * lane < E ? ((ns[2 * lane] + 1) * M) | 1 : 0;
    const int n1 = 2 * lane + 1 < E ? ((ns[2 * lane + 1] + 1) * M) | 1 : 0;
    int in = n0 + n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, in, o);
      if (lane >= o) in += u;
    }
    if (2 * lane < E) off[2 * lane] = in - n0 - n1;
    if (2 * lane + 1 < E) off[2 * lane + 1] = in - n1;
    if (lane == 31) off[64] = in;
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    c.has[i] = s_qmax[i] >= 0;
    c.qmax[i] = __int_as_float(s_qmax[i]);
    c.qmin[i] = __int_as_float(s_qmin[i]);
  }
  c.prune = __syncthreads_or(bad_p) == 0;
  c.rows = true;
#pragma unroll
  for (int i = 0; i < D; ++i) c.rows = c.rows && s_woff[i][64] <= wcap;
  if (c.classes) {
    // a target a warp, classes lane, lane + 32, ... a lane: the losses below each
    const int pitch = la_class_pitch(E);
    constexpr int kPer = kLaMaxLoss / 32 + 1;
    for (int kt = warp; kt < E; kt += NW) {
      const int ns = s_nsub[0][kt], f0 = first_of(kt);
      int f[kPer];
#pragma unroll
      for (int u = 0; u < kPer; ++u) f[u] = 0;
      for (int n = 0; n < ns; ++n) {
        const int r = s_rank[f0 + n];
#pragma unroll
        for (int u = 0; u < kPer; ++u) f[u] += r < lane + 32 * u ? 1 : 0;
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (lane + 32 * u <= c.n_loss) s_fits[(lane + 32 * u) * pitch + kt] = static_cast<uint8_t>(f[u]);
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const LaLevel& v = c.lev[i];
    const float* ua = i > 0 ? c.Ua[i - (i > 0)] : nullptr;
    const float* un = i > 0 ? c.Un[i - (i > 0)] : nullptr;
    if (c.rows) {
      // a warp a row, an entry (the exact expert or a substitute) and m a lane;
      // then a lane an m takes the minima along the row
      for (int kt = warp; kt < E; kt += NW) {
        const int ns = s_nsub[i][kt];
        float* wa = Wa[i] + s_woff[i][kt];
        float* cn = i > 0 ? Cn[i] + s_woff[i][kt] : nullptr;
        for (int x = lane; x < (ns + 1) * M; x += 32) {
          const int n = x / M, m = x - n * M;
          const int kk = n == 0 ? kt : s_ord[i][kt * 64 + n - 1];
          const float cq = n == 0 ? 0.0f : v.Cq[kt * E + kk];
          float all = INFINITY, none = INFINITY;
          for (uint32_t pm = v.pmask[kk]; pm; pm &= pm - 1) {
            const int m2 = __ffs(pm) - 1;
            const float base = __fadd_rn(v.A[m * M + m2], cq);
            if (i == 0) {
              all = fminf(all, base);
            } else {
              all = fminf(all, __fadd_rn(base, ua[m2 * E + kk]));
              none = fminf(none, __fadd_rn(base, un[m2 * E + kk]));
            }
          }
          wa[x] = all;
          if (i > 0) cn[x] = none;
        }
        __syncwarp();
        for (int m = lane; m < M; m += 32) {
          float best = wa[m];
          Vn[m * E + kt] = i > 0 ? cn[m] : best;
          for (int n = 1; n <= ns; ++n) {
            best = fminf(best, wa[n * M + m]);
            wa[n * M + m] = best;
          }
          Va[m * E + kt] = best;
        }
      }
    } else {
      // V of level i + 1, one (k', m) a thread
      for (int x = tid; x < E * M; x += kThreads) {
        const int kt = x / M, m = x - kt * M;
        float all = INFINITY, none = INFINITY;
        for (unsigned long long sb = v.subst[kt] | (1ull << kt); sb; sb &= sb - 1) {
          const int kk = __ffsll(static_cast<long long>(sb)) - 1;
          const float cq = kk == kt ? 0.0f : v.Cq[kt * E + kk];
          for (uint32_t pm = v.pmask[kk]; pm; pm &= pm - 1) {
            const int m2 = __ffs(pm) - 1;
            const float base = __fadd_rn(v.A[m * M + m2], cq);
            all = fminf(all, i > 0 ? __fadd_rn(base, ua[m2 * E + kk]) : base);
            if (kk == kt) none = fminf(none, i > 0 ? __fadd_rn(base, un[m2 * E + kk]) : base);
          }
        }
        Va[m * E + kt] = all;
        Vn[m * E + kt] = none;
      }
    }
    __syncthreads();
    // Phi of level i + 1 in both cases, one (m, kx) a thread
    for (int x = tid; x < M * E; x += kThreads) {
      const int m = x / E, kx = x - m * E;
      const float* Pr = c.P[i] + kx * c.pitch;
      float pa = 0.0f, pn = 0.0f;
#pragma unroll 8
      for (int kt = 0; kt < E; ++kt) {
        const float p = Pr[kt];
        if (p != 0.0f) {
          pa = __fadd_rn(pa, __fmul_rn(p, Va[m * E + kt]));
          pn = __fadd_rn(pn, __fmul_rn(p, Vn[m * E + kt]));
        }
      }
      U[2 * i][x] = pa;
      U[2 * i + 1][x] = pn;
    }
    __syncthreads();
  }

  // ---- the tokens, one a warp
  const LaLevel own = la_level(tab, E, M, a);
  // the servers of experts lane and lane + 32
  const uint32_t pmask0 = lane < E ? own.pmask[lane] : 0u;
  const uint32_t pmask1 = lane + 32 < E ? own.pmask[lane + 32] : 0u;
  int kind_count[4] = {0, 0, 0, 0};
  // NW tokens at a time, one a warp, slot by slot: each warp takes its token's
  // candidates in the two cases and lists the others, then the warps share the
  // listed evaluations (a few tokens have most of them), then each updates its
  // token. Counters of a step are cleared a step ahead.
  int step = 0;
  for (int base = 0; base < ntok; base += NW) {
    bool live = base + warp < ntok;
    const int t = live ? s_tok[base + warp] : 0;
    const int s = live && loc != nullptr ? loc[t] : a;
    float q = live && qhat != nullptr ? qhat[t] : 0.0f;
    const int idx = live && lane < k ? topk_idx[(size_t)t * k + lane] : 0;
    if (live && s >= M) {
      if (lane == 0) report(&g_err_route, ORDERMOE_DEV_BAD_INDEX, t0 + t);
      live = false;
    }
    if (__any_sync(0xffffffffu, idx < 0 || idx >= E)) live = false;  // -1: a NaN token (reported)
    unsigned long long taken = 0;
    for (int j = 0; j < k; ++j) taken |= 1ull << (__shfl_sync(0xffffffffu, idx, j) & 63);
    const float* As = s_As[warp];
    if (live && lane < M) s_As[warp][lane] = own.A[s * M + lane];
    __syncwarp();
    // the target's set and rows, loaded a slot ahead
    unsigned long long sb_next = 0;
    float q_next[2] = {0.0f, 0.0f}, cq_next[2] = {0.0f, 0.0f};
    auto load_slot = [&](int j) {
      const int r = __shfl_sync(0xffffffffu, idx, j);
      if (!live) return;
      sb_next = own.subst[r];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int e = lane + 32 * h;
        if (e < E) {
          q_next[h] = own.Q[r * E + e];
          cq_next[h] = own.Cq[r * E + e];
        }
      }
    };
    load_slot(0);
    int first_server = s;
    for (int j = 0; j < k; ++j, ++step) {
      const int r = __shfl_sync(0xffffffffu, idx, j);
      const unsigned long long sb_r = sb_next;
      const float q_r[2] = {q_next[0], q_next[1]}, cq_r[2] = {cq_next[0], cq_next[1]};
      if (j + 1 < k) load_slot(j + 1);
      int* n_task = &s_task_n[step & 1][0];  // listed, taken
      unsigned long long best = ~0ull;
      if (live) {
        const unsigned long long sb = sb_r & ~taken;
#pragma unroll
        for (int h = 0; h < kEmax / 32 + (kEmax < 32); ++h) {
          const int e = lane + 32 * h;
          const bool sub = (sb >> e) & 1ull;
          float cq = 0.0f, qn = q;
          uint32_t pm = (sub || e == r) ? (h ? pmask1 : pmask0) : 0u;
          if (sub) {
            qn = __fadd_rn(q, q_r[h]);
            cq = cq_r[h];
            if (!(qn <= qbar)) pm = 0u;  // Eq. 40 budget
          }
          const float* Ut = la_all<D>(c, D, qn) ? c.Ua[D - 1] : la_none<D>(c, D, qn) ? c.Un[D - 1] : nullptr;
          // the key's low word: substitute, away, server, expert
          auto low_of = [&](int m) {
            return (sub ? 0x80000000u : 0u) | (m != s ? 0x40000000u : 0u) |
                   (static_cast<uint32_t>(m) << 8) | static_cast<uint32_t>(e);
          };
          uint32_t left = 0u;  // not listed for want of room
          for (; pm; pm &= pm - 1) {
            const int m = __ffs(pm) - 1;
            const float cost0 = __fadd_rn(As[m], cq);
            if (Ut != nullptr) {
              const unsigned long long key =
                  (static_cast<unsigned long long>(__float_as_uint(__fadd_rn(cost0, Ut[m * E + e]))) << 32) | low_of(m);
              best = key < best ? key : best;
              continue;
            }
            const int i = atomicAdd(n_task, 1);
            if (i < kLaTasks) s_task[i] = make_uint4(__float_as_uint(cost0), __float_as_uint(qn), low_of(m), warp);
            else left |= 1u << m;
          }
          for (unsigned todo = __ballot_sync(0xffffffffu, left != 0u); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const float qs = __shfl_sync(0xffffffffu, qn, src);
            for (uint32_t x = __shfl_sync(0xffffffffu, left, src); x; x &= x - 1) {
              const int m = __ffs(x) - 1;
              const float phi = la_phi_warp<D>(c, s_term, lane, m, src + 32 * h, qs);
              if (lane == src) {
                const unsigned long long key =
                    (static_cast<unsigned long long>(__float_as_uint(__fadd_rn(__fadd_rn(As[m], cq), phi))) << 32) | low_of(m);
                best = key < best ? key : best;
              }
            }
          }
        }
        // the smallest key of the warp: high words, then the low words among those
        const unsigned hi = static_cast<unsigned>(best >> 32);
        const unsigned mhi = __reduce_min_sync(0xffffffffu, hi);
        const unsigned mlo = __reduce_min_sync(0xffffffffu, hi == mhi ? static_cast<unsigned>(best) : 0xffffffffu);
        if (lane == 0) s_best[warp] = (static_cast<unsigned long long>(mhi) << 32) | mlo;
      }
      __syncthreads();
      if (tid == 0) s_task_n[(step + 1) & 1][0] = s_task_n[(step + 1) & 1][1] = 0;
      const int nt = min(n_task[0], kLaTasks);
      // passed over when it costs more than another at best (Ua is the least of Phi)
      auto passed_over = [&](float cost0, uint32_t low, unsigned long long so_far) {
        const int m = static_cast<int>((low >> 8) & 0xFFu), e = static_cast<int>(low & 0xFFu);
        return c.prune && so_far != ~0ull &&
               __fadd_rn(cost0, c.Ua[D - 1][m * E + e]) > __uint_as_float(static_cast<unsigned>(so_far >> 32));
      };
      if constexpr (D > 1 && NW > 8) {
        // all warps on one evaluation: a group of lanes a target
        int width = 1;
        while (2 * width * E <= kThreads && width < 8) width *= 2;
#pragma unroll 1
        for (int i = 0; i < nt; ++i) {
          const uint4 task = s_task[i];
          const float cost0 = __uint_as_float(task.x), qn = __uint_as_float(task.y);
          if (passed_over(cost0, task.z, s_best[task.w])) continue;  // the same for the block
          const int m = static_cast<int>((task.z >> 8) & 0xFFu), e = static_cast<int>(task.z & 0xFFu);
          float* term = reinterpret_cast<float*>(s_raw);
          const int sub = tid & (width - 1), kt = tid / width;
          for (int k0 = 0; k0 < E; k0 += kThreads / width) {
            const int kv = min(k0 + kt, E - 1);
            const float p = c.P[D - 1][e * c.pitch + kv];
            const float x = la_value_lanes<D>(c, m, kv, qn, sub, width);
            if (sub == 0 && k0 + kt < E) term[k0 + kt] = p != 0.0f ? __fmul_rn(p, x) : 0.0f;
          }
          __syncthreads();
          if (tid == 0) {
            float phi = 0.0f;
#pragma unroll 8
            for (int kv = 0; kv < E; ++kv) phi = __fadd_rn(phi, term[kv]);
            const unsigned long long key =
                (static_cast<unsigned long long>(__float_as_uint(__fadd_rn(cost0, phi))) << 32) | task.z;
            if (key < s_best[task.w]) s_best[task.w] = key;
          }
          __syncthreads();
        }
      } else {
        // an evaluation a warp
        while (nt > 0) {
          int i = 0;
          if (lane == 0) i = atomicAdd(n_task + 1, 1);
          i = __shfl_sync(0xffffffffu, i, 0);
          if (i >= nt) break;
          const uint4 task = s_task[i];
          const float cost0 = __uint_as_float(task.x);
          const unsigned long long so_far = *static_cast<volatile unsigned long long*>(&s_best[task.w]);
          if (__any_sync(0xffffffffu, passed_over(cost0, task.z, so_far))) continue;
          const float phi = la_phi_warp<D>(c, s_term, lane, static_cast<int>((task.z >> 8) & 0xFFu),
                                           static_cast<int>(task.z & 0xFFu), __uint_as_float(task.y));
          if (lane == 0)
            atomicMin(&s_best[task.w],
                      (static_cast<unsigned long long>(__float_as_uint(__fadd_rn(cost0, phi))) << 32) | task.z);
        }
      }
      __syncthreads();
      if (!live) continue;
      best = s_best[warp];
      int kstar, mstar, kd;
      if (best == ~0ull) {
        if (lane == 0) report(&g_err_route, ORDERMOE_DEV_NO_CANDIDATE, t0 + t);
        kstar = r; mstar = s; kd = 0;
      } else {
        const uint32_t mlo = static_cast<uint32_t>(best);
        kstar = static_cast<int>(mlo & 0xFFu);
        mstar = static_cast<int>((mlo >> 8) & 0xFFu);
        const int sub = static_cast<int>((mlo >> 31) & 1u);
        kd = 2 * static_cast<int>((mlo >> 30) & 1u) + sub;
        if (sub) {
          taken |= 1ull << kstar;
          q = __fadd_rn(q, own.Q[r * E + kstar]);
        }
      }
      if (j == 0) first_server = mstar;
      if (lane == 0) {
        chosen_expert[(size_t)t * k + j] = kstar;
        chosen_server[(size_t)t * k + j] = static_cast<uint8_t>(mstar);
        kind_out[(size_t)t * k + j] = static_cast<uint8_t>(kd);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) kind_count[x] += kd == x ? 1 : 0;
    }
    if (live && lane == 0 && loc != nullptr) {
      loc[t] = static_cast<uint8_t>(first_server);
      qhat[t] = q;
    }
  }
  if (counters == nullptr) return;
  if (lane == 0)
    for (int x = 0; x < 4; ++x)
      if (kind_count[x]) atomicAdd(&s_kind[x], kind_count[x]);
  __syncthreads();
  if (tid < 4 && s_kind[tid]) atomicAdd(&counters[tid], s_kind[tid]);
}

// ---------------------------------------------------------------------------
// Router on tcgen05 + selection. A cluster of S CTAs (S = 1..8) handles 128
// tokens: CTA r of the cluster accumulates logits = X W_r^T over its share of
// the K blocks (M = 128 tokens, N = NE >= E padded to 16/32/64) in TMEM. Its
// epilogue thread i of warp w (w = 2..5) reads TMEM lane 32 (w % 4) + i (token
// 32 (w % 4) + i); ranks > 0 store their partial logits into rank 0's shared
// memory (distributed shared memory), and after a cluster barrier rank 0 adds
// the partials in rank order (deterministic) and runs select_token. Splitting
// K lets a few hundred tokens (decode) still stream X over many SMs. The
// partials are laid out [rank - 1][NE / 4][128 tokens][4], so that the 32
// tokens of a warp store and load 16-byte vectors at consecutive addresses
// (no bank conflicts). While the TMA and MMA warps run, rank 0's epilogue
// warps load the selection tables (the delay table too, when small) and
// each token's home, location and loss.
// Warp 0 issues the TMA loads (X: 128 x 64 box; W_r: NE x 64 box, rows >= E
// zero-filled), warp 1 the MMAs; mbarrier ring; bounded waits.
namespace rt {
constexpr int BK = 64;
constexpr int A_BYTES = 128 * BK * 2;
constexpr int THREADS = 192;
// Only layers of up to 16 experts (NE = 16) select inside the router; for
// more experts it writes the targets and a selection kernel selects, so the
// wider instantiations keep no tables and give that space to the X ring.
template <int NE>
constexpr bool selects() { return NE <= 16; }
// stages of (16 KB + NE x 128 B) in flight per CTA, and the largest cluster,
// sized so the ring, the partial logits of ranks 1..S-1 and (NE = 16) the
// tables and the staged delay table fit in 227 KB beside the static
// selection tables
template <int NE>
constexpr int stages() { return NE <= 16 ? 8 : (NE <= 32 ? 8 : 7); }
template <int NE>
constexpr int max_split() { return NE <= 16 ? 8 : (NE <= 32 ? 4 : 2); }
template <int NE>
constexpr int smem_bytes(int E) {
  return 1024 + stages<NE>() * (A_BYTES + NE * BK * 2) + 256 +
         (max_split<NE>() - 1) * 128 * NE * 4 + (selects<NE>() ? 8 * E * E + 4 * kDelayStage : 0);
}
static_assert(smem_bytes<16>(16) + sizeof(SelSmem) <= 227 * 1024, "router shared memory");
static_assert(smem_bytes<32>(32) + sizeof(SelSmem) <= 227 * 1024, "router shared memory");
static_assert(smem_bytes<64>(64) + sizeof(SelSmem) <= 227 * 1024, "router shared memory");
}  // namespace rt

template <int NE>
struct RouterSmem {
  uint64_t full[rt::stages<NE>()];
  uint64_t empty[rt::stages<NE>()];
  uint64_t tfull;
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
  int zero;
};

template <int NE>
__global__ void __launch_bounds__(rt::THREADS, 1) router_select_kernel(
    const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW, int T,
    int E, int d, int k, int renorm, const uint8_t* __restrict__ tab,
    const uint8_t* __restrict__ home, uint8_t* __restrict__ loc, float* __restrict__ qhat,
    float* __restrict__ logits_out, int32_t* __restrict__ topk_idx, float* __restrict__ topk_w,
    int32_t* __restrict__ chosen_expert, uint8_t* __restrict__ chosen_server,
    uint8_t* __restrict__ kind_out, int32_t* __restrict__ counters, uint64_t limit_ns, int split,
    Lookahead la) {
  pdl_trigger();  // launched with launch_pdl: shared memory, barrier and TMEM set-up first
  constexpr int B_BYTES = NE * rt::BK * 2;
  constexpr int STAGE_BYTES = rt::A_BYTES + B_BYTES;
  constexpr int STAGES = rt::stages<NE>();
  constexpr int TMEM_COLS = NE <= 32 ? 32 : NE;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  RouterSmem<NE>& s = *reinterpret_cast<RouterSmem<NE>*>(tiles + STAGES * STAGE_BYTES);
  // partials of ranks 1..split-1: [split - 1][NE / 4][128][4]
  float* red = reinterpret_cast<float*>(tiles + STAGES * STAGE_BYTES + 256);
  float* s_Q = red + (rt::max_split<NE>() - 1) * 128 * NE;
  float* s_Cq = s_Q + E * E;
  float* s_A = s_Cq + E * E;
  __shared__ SelSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = split > 1 ? cluster_ctarank() : 0;
  const int tile = blockIdx.x / split;
  const int m0 = tile * 128;
  const int kblocks_all = d / rt::BK;
  const int per = (kblocks_all + split - 1) / split;
  const int kb_begin = static_cast<int>(rank) * per;
  const int kb_end = min(kblocks_all, kb_begin + per);
  const int kblocks = kb_end > kb_begin ? kb_end - kb_begin : 0;

  if (tid == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 1);
    }
    mbar_init(&s.tfull, 1);
    mbar_init(&s.drain, 1);
    s.abort = 0;
    s.zero = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_map(&mapX);
    tma_prefetch_map(&mapW);
  }
  if (warp == 1) {
    tmem_alloc(&s.tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  bool tables_ok = true;  // rank 0's epilogue warps load the tables during the main loop
  const float* Atab = nullptr;
  int pre_a = 0, pre_s = 0;  // the token's home and location, loaded during the main loop
  float pre_q = 0.0f;
  tc_fence_before();
  if (split > 1) cluster_sync();  // rank 0 runs: its shared memory may be written
  else __syncthreads();
  tc_fence_after();
  pdl_wait();  // the previous kernel's outputs (X, tables, state) are ready
  const uint32_t tmem_base = s.tmem_base;
  volatile int* abort = &s.abort;
  uint32_t issued_mask = 0, last_phase_bits = 0;
  bool mma_issued = false, leader = false;
  float lg[NE];
  int kind_count[4] = {0, 0, 0, 0};

  // Producer and MMA warps walk the stages converged, one elected lane issues: a
  // lane walking them alone held the stream back (4096 tokens of 8 experts, d
  // 4096, 14.9 us; so 12.9; 8192 of 64, d 2048, 20.5 and 19.4; 128 tokens 8.9 and
  // 8.1, ncu).
  if (warp == 0) {
    const bool issuer = elect_one();
    for (int i = 0; i < kblocks; ++i) {
      const int stage = i % STAGES;
      const uint32_t phase = (i / STAGES) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&s.empty[stage], phase ^ 1u, limit_ns, abort))) {
        if (issuer && !*abort) report(&g_err_route, ORDERMOE_DEV_WAIT_TIMEOUT, 21);
        *abort = 1;
        break;
      }
      if (issuer) {
        uint8_t* sa = tiles + stage * STAGE_BYTES;
        mbar_arrive_expect_tx(&s.full[stage], STAGE_BYTES);
        tma_load_2d(sa, &mapX, &s.full[stage], (kb_begin + i) * rt::BK, m0);
        tma_load_2d(sa + rt::A_BYTES, &mapW, &s.full[stage], (kb_begin + i) * rt::BK, 0);
      }
      issued_mask |= 1u << stage;
      last_phase_bits = (last_phase_bits & ~(1u << stage)) | (phase << stage);
    }
  } else if (warp == 1) {
    constexpr uint32_t IDESC = idesc_bf16_f32(128, NE);
    leader = elect_one();
    const uint64_t desc0 = sdesc_kmajor_sw128(smem_u32(tiles));
    bool ok = true;
    for (int i = 0; i < kblocks; ++i) {
      const int stage = i % STAGES;
      const uint32_t phase = (i / STAGES) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&s.full[stage], phase, limit_ns, abort))) {
        if (leader && !*abort) report(&g_err_route, ORDERMOE_DEV_WAIT_TIMEOUT, 22);
        *abort = 1;
        ok = false;
        break;
      }
      tc_fence_after();
      const uint64_t da = desc0 + static_cast<uint64_t>((stage * STAGE_BYTES) >> 4);
      const uint64_t db = da + (rt::A_BYTES >> 4);
      if (leader) {
#pragma unroll
        for (int kk = 0; kk < rt::BK / 16; ++kk)  // 16 elements = 32 bytes on
          mma_bf16(tmem_base, da + 2 * kk, db + 2 * kk, IDESC, (i | kk) != 0 ? 1u : 0u);
        mma_commit(&s.empty[stage]);
      }
      mma_issued = true;
    }
    if (ok && leader) {
      if (mma_issued) mma_commit(&s.tfull);
      else mbar_arrive(&s.tfull);  // empty K share: nothing to wait for
    }
  } else {
    // the selection tables, while the TMA and MMA warps run (named barrier 1:
    // the 128 epilogue threads)
    if (rank == 0) {
      if (!rt::selects<NE>() || la.H > 1 || la.topk_only) {  // targets only: a selection kernel reads the tables
        if (tid - 64 < 4) sm.kind[tid - 64] = 0;
      } else {
        const int t = m0 + (warp & 3) * 32 + lane;
        if (t < T) {
          pre_a = home[t];
          pre_s = (loc != nullptr) ? loc[t] : pre_a;  // no state given: first layer (Eq. 36)
          pre_q = (qhat != nullptr) ? qhat[t] : 0.0f;
        }
        tables_ok = load_tables_range(tab, E, sm, s_Q, s_Cq, tid - 64, 128);
        Atab = load_delay_range(tab, E, s_A, tid - 64, 128);
      }
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    // epilogue part 1: this CTA's partial logits
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(&s.tfull, 0, limit_ns, abort));
    if (!ok) {
      if (lane == 0 && !*abort) report(&g_err_route, ORDERMOE_DEV_WAIT_TIMEOUT, 23);
      *abort = 1;
    } else {
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < NE; c += 32) {
        uint32_t v[32];
        tmem_ld32(tmem_base + (static_cast<uint32_t>(q * 32) << 16) + c, v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (c + i < NE) lg[c + i] = kblocks > 0 ? __uint_as_float(v[i]) : 0.0f;
      }
      tc_fence_before();
      if (rank > 0) {
        // partial logits of this rank -> red[rank - 1][c / 4][row][c % 4] in rank 0's
        // shared memory
        const uint32_t dst =
            mapa_shared(smem_u32(red + ((size_t)(rank - 1) * (NE / 4) * 128 + row) * 4), 0);
#pragma unroll
        for (int c = 0; c < NE; c += 4)
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + c * 128 * 4),
                       "f"(lg[c]), "f"(lg[c + 1]), "f"(lg[c + 2]), "f"(lg[c + 3])
                       : "memory");
      }
    }
  }
  if (split > 1) cluster_sync();  // partials visible in rank 0
  if (warp >= 2 && rank == 0 && !*abort) {
    // epilogue part 2: full logits (partials in rank order) and the selection
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const int t = m0 + row;
    for (int r = 1; r < split; ++r) {
      const float4* src = reinterpret_cast<const float4*>(red) + (size_t)(r - 1) * (NE / 4) * 128 + row;
#pragma unroll
      for (int c = 0; c < NE; c += 4) {
        const float4 p = src[(c / 4) * 128];
        lg[c] += p.x;
        lg[c + 1] += p.y;
        lg[c + 2] += p.z;
        lg[c + 3] += p.w;
      }
    }
#pragma unroll
    for (int e = 0; e < NE; ++e)  // padding past E for select_token
      if (e >= E) lg[e] = -INFINITY;
    if (t < T && tables_ok) {
      if (logits_out != nullptr) {
#pragma unroll
        for (int e = 0; e < NE; ++e)  // constant indices keep lg[] in registers
          if (e < E) logits_out[(size_t)t * E + e] = lg[e];
      }
      // the token's logits into this thread's column of partial slot 0 (read above)
      float4* col = reinterpret_cast<float4*>(red) + row;
#pragma unroll
      for (int c = 0; c < NE; c += 4)
        col[(c / 4) * 128] = make_float4(lg[c], lg[c + 1], lg[c + 2], lg[c + 3]);
      const int M = reinterpret_cast<const int32_t*>(tab)[2];
      const float qbar = reinterpret_cast<const float*>(tab)[5];
      select_token(t, ColLogits{col}, E, k, renorm, M, qbar, Atab, sm, s_Q, s_Cq, pre_a, pre_s,
                   pre_q, loc, qhat, topk_idx, topk_w, chosen_expert, chosen_server,
                   kind_out, kind_count, !rt::selects<NE>() || la.H > 1 || la.topk_only);
    }
    flush_kind_counts(sm, kind_count, counters);
  }

  __syncthreads();
  if (s.abort) {
    volatile int* never = &s.zero;
    if (warp == 0 && lane == 0)
      for (int st = 0; st < STAGES; ++st)
        if ((issued_mask >> st) & 1u) mbar_wait(&s.full[st], (last_phase_bits >> st) & 1u, limit_ns, never);
    if (leader && mma_issued) {  // the lane that issued the MMAs
      mma_commit(&s.drain);
      mbar_wait(&s.drain, 0, limit_ns, never);
    }
    __syncthreads();
  }
  if (rank == 0 && counters != nullptr && tid < 4 && sm.kind[tid]) atomicAdd(&counters[tid], sm.kind[tid]);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// Small batches of 17 to 64 experts: router, top-k and selection in one launch.
// A cluster of S CTAs (two for more than 32 experts, else four) handles 16 S
// tokens, CTA r the r-th of S shares of the K blocks, and then the tokens 16 r ..
// 16 r + 15: every CTA stores its partial logits of a token into the shared memory
// of the CTA that owns it, which adds them in rank order and gives the token eight
// lanes for the top-k, the softmax and the slots of Alg. 2 (select_slots, as
// select_lanes_kernel). The shares are router_select_kernel's at its largest
// split, so a token's logits are the same bits from either kernel.
// The MMA's M side is 128 rows, of which the tokens' 16 S are loaded; it reads the
// rest from the stage's own weights and from padding that nothing writes, and
// those rows of the accumulator are not read.
// Bound by latency: the K share's loads, two cluster barriers and the slots'
// serial argmins. In a graph of calls, tokens x experts, d 2048: one CTA of two
// with all 128 tokens, a thread each, and the selection in a launch of its own took
// 19.5 us for 33 x 64 and 20.2 for 1021 x 64, this takes 11.6 and 12.0 (d 4096:
// 27.0 and 15.9); 12.4 and 8.5 for 33 x 24, d 1024. Stages of one K block, ten of
// them: 12.1 and 12.5. (Eight shares of K for 128 tokens took 11.1 and 11.4 us, but
// their logits differ from the other kernel's in the last bits.)
namespace rl {
constexpr int ROWS = 16;  // tokens of a CTA
constexpr int STAGES = 5;  // of two K blocks each
constexpr int THREADS = 192;
template <int NE>
constexpr int split() { return rt::max_split<NE>(); }
template <int NE>
constexpr int a_bytes() { return split<NE>() * ROWS * rt::BK * 2; }  // the tokens' rows
constexpr int BLOCK_BYTES = rt::A_BYTES;  // what an MMA's 128 rows span
// partials of one rank: [NE / 4 chunks][ROWS + 1][4] floats (the odd pitch spreads
// the chunks that the eight lanes of a token read over the banks)
template <int NE>
constexpr int part_floats() { return NE / 4 * (ROWS + 1) * 4; }
constexpr int LG_PITCH = 68;  // floats a token's exponentials take
template <int NE>
constexpr int smem_bytes(int E) {
  return 1024 + STAGES * 2 * BLOCK_BYTES + 256 + split<NE>() * part_floats<NE>() * 4 + ROWS * LG_PITCH * 4 +
         8 * E * E;
}
static_assert(smem_bytes<32>(32) + sizeof(SelSmem) <= 227 * 1024, "router shared memory");
static_assert(smem_bytes<64>(64) + sizeof(SelSmem) <= 227 * 1024, "router shared memory");
static_assert(a_bytes<32>() + 32 * rt::BK * 2 <= BLOCK_BYTES, "rows and weights of a K block");
static_assert(a_bytes<64>() + 64 * rt::BK * 2 <= BLOCK_BYTES, "rows and weights of a K block");
}  // namespace rl

struct RouterLanesSmem {
  uint64_t full[rl::STAGES];
  uint64_t empty[rl::STAGES];
  uint64_t tfull;
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
  int zero;
};

template <int NE>
__global__ void __launch_bounds__(rl::THREADS, 1)
    router_lanes_kernel(const __grid_constant__ CUtensorMap mapX,
                        const __grid_constant__ CUtensorMap mapW, int T, int E, int d, int k,
                        int renorm, const uint8_t* __restrict__ tab,
                        const uint8_t* __restrict__ home, uint8_t* __restrict__ loc,
                        float* __restrict__ qhat, float* __restrict__ logits_out,
                        int32_t* __restrict__ topk_idx, float* __restrict__ topk_w,
                        int32_t* __restrict__ chosen_expert, uint8_t* __restrict__ chosen_server,
                        uint8_t* __restrict__ kind_out, int32_t* __restrict__ counters,
                        uint64_t limit_ns, int topk_only) {
  pdl_trigger();  // launched with programmatic serialization: set-up first
  constexpr int SPLIT = rl::split<NE>();
  constexpr int TILE = SPLIT * rl::ROWS;  // tokens of the cluster
  constexpr int BLOCK_BYTES = rl::BLOCK_BYTES, STAGE_BYTES = 2 * BLOCK_BYTES;
  constexpr int A_BYTES = rl::a_bytes<NE>(), B_BYTES = NE * rt::BK * 2;
  constexpr int TMEM_COLS = NE;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  RouterLanesSmem& s = *reinterpret_cast<RouterLanesSmem*>(tiles + rl::STAGES * STAGE_BYTES);
  float* part = reinterpret_cast<float*>(tiles + rl::STAGES * STAGE_BYTES + 256);
  float* s_ex = part + SPLIT * rl::part_floats<NE>();  // [ROWS][LG_PITCH] the logits' exponentials
  float* s_Q = s_ex + rl::ROWS * rl::LG_PITCH;
  float* s_Cq = s_Q + E * E;
  __shared__ SelSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int m0 = static_cast<int>(blockIdx.x / SPLIT) * TILE;
  const int kblocks_all = d / rt::BK;
  const int per = (kblocks_all + SPLIT - 1) / SPLIT;
  const int kb_begin = min(kblocks_all, rank * per);
  const int kblocks = min(kblocks_all, kb_begin + per) - kb_begin;

  if (tid == 0) {
    for (int i = 0; i < rl::STAGES; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 1);
    }
    mbar_init(&s.tfull, 1);
    mbar_init(&s.drain, 1);
    s.abort = 0;
    s.zero = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_map(&mapX);
    tma_prefetch_map(&mapW);
  }
  if (warp == 1) {
    tmem_alloc(&s.tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  cluster_sync();  // every CTA of the cluster runs: its shared memory may be written
  tc_fence_after();
  pdl_wait();  // the previous kernel's outputs (X, tables, state) are ready
  const uint32_t tmem_base = s.tmem_base;
  volatile int* abort = &s.abort;
  uint32_t issued_mask = 0, last_phase_bits = 0;
  bool mma_issued = false, leader = false;
  bool tables_ok = true;
  // the epilogue thread's token (eight lanes each) and its state
  const int et = tid - 64;
  const int row = et >> 3, sub = lane & 7;
  const int t = m0 + rank * rl::ROWS + row;
  int a = 0, loc0 = 0;
  float q0 = 0.0f;

  if (warp == 0) {
    const bool issuer = elect_one();
    for (int kb = 0, i = 0; kb < kblocks; kb += 2, ++i) {
      const int stage = i % rl::STAGES, n = min(2, kblocks - kb);
      const uint32_t phase = (i / rl::STAGES) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&s.empty[stage], phase ^ 1u, limit_ns, abort))) {
        if (issuer && !*abort) report(&g_err_route, ORDERMOE_DEV_WAIT_TIMEOUT, 24);
        *abort = 1;
        break;
      }
      if (issuer) {
        uint8_t* sa = tiles + stage * STAGE_BYTES;
        mbar_arrive_expect_tx(&s.full[stage], n * (A_BYTES + B_BYTES));
        for (int j = 0; j < n; ++j, sa += BLOCK_BYTES) {
          tma_load_2d(sa, &mapX, &s.full[stage], (kb_begin + kb + j) * rt::BK, m0);
          tma_load_2d(sa + A_BYTES, &mapW, &s.full[stage], (kb_begin + kb + j) * rt::BK, 0);
        }
      }
      issued_mask |= 1u << stage;
      last_phase_bits = (last_phase_bits & ~(1u << stage)) | (phase << stage);
    }
  } else if (warp == 1) {
    constexpr uint32_t IDESC = idesc_bf16_f32(128, NE);
    leader = elect_one();
    const uint64_t desc0 = sdesc_kmajor_sw128(smem_u32(tiles));
    bool ok = true;
    for (int kb = 0, i = 0; kb < kblocks; kb += 2, ++i) {
      const int stage = i % rl::STAGES, n = min(2, kblocks - kb);
      const uint32_t phase = (i / rl::STAGES) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&s.full[stage], phase, limit_ns, abort))) {
        if (leader && !*abort) report(&g_err_route, ORDERMOE_DEV_WAIT_TIMEOUT, 25);
        *abort = 1;
        ok = false;
        break;
      }
      tc_fence_after();
      const uint64_t da0 = desc0 + static_cast<uint64_t>((stage * STAGE_BYTES) >> 4);
      if (leader) {
        for (int j = 0; j < n; ++j) {
          const uint64_t da = da0 + static_cast<uint64_t>((j * BLOCK_BYTES) >> 4), db = da + (A_BYTES >> 4);
#pragma unroll
          for (int kk = 0; kk < rt::BK / 16; ++kk)  // 16 elements = 32 bytes on
            mma_bf16(tmem_base, da + 2 * kk, db + 2 * kk, IDESC, (kb | j | kk) != 0 ? 1u : 0u);
        }
        mma_commit(&s.empty[stage]);
      }
      mma_issued = true;
    }
    if (ok && leader) {
      if (mma_issued) mma_commit(&s.tfull);
      else mbar_arrive(&s.tfull);  // empty K share: nothing to wait for
    }
  } else {
    // the selection tables and the token's state, while the TMA and MMA warps run
    if (et < 4) sm.kind[et] = 0;
    if (!topk_only) {
      if (t < T) {
        a = home[t];
        loc0 = (loc != nullptr) ? loc[t] : a;  // no state given: first layer (Eq. 36)
        q0 = (qhat != nullptr) ? qhat[t] : 0.0f;
      }
      tables_ok = load_tables_range(tab, E, sm, s_Q, s_Cq, et, 128);
    }
    // this CTA's partial logits to the tokens' owners
    const int q = warp & 3;
    const int r = q * 32 + lane;  // TMEM lane: row of the tile
    const bool ok = q * 32 >= TILE || __all_sync(0xffffffffu, mbar_wait(&s.tfull, 0, limit_ns, abort));
    if (!ok) {
      if (lane == 0 && !*abort) report(&g_err_route, ORDERMOE_DEV_WAIT_TIMEOUT, 26);
      *abort = 1;
    } else if (q * 32 < TILE) {
      tc_fence_after();
      const uint32_t dst = mapa_shared(
          smem_u32(part + rank * rl::part_floats<NE>() + (r % rl::ROWS) * 4), r / rl::ROWS);
#pragma unroll
      for (int c = 0; c < NE; c += 32) {
        uint32_t v[32];
        tmem_ld32(tmem_base + (static_cast<uint32_t>(q * 32) << 16) + c, v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const bool any = kblocks > 0;
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(
                           dst + static_cast<uint32_t>((c + i) / 4 * (rl::ROWS + 1) * 16)),
                       "f"(any ? __uint_as_float(v[i]) : 0.0f), "f"(any ? __uint_as_float(v[i + 1]) : 0.0f),
                       "f"(any ? __uint_as_float(v[i + 2]) : 0.0f), "f"(any ? __uint_as_float(v[i + 3]) : 0.0f)
                       : "memory");
        }
      }
      tc_fence_before();
    }
  }
  cluster_sync();  // the partials of every CTA are there (and the tables, in the block)
  if (warp >= 2 && !*abort) {
    // the token's logits: chunks of four experts over its lanes, ranks in order
    float* ex = s_ex + row * rl::LG_PITCH;
    bool nan = false;
    float v[NE / 8];
#pragma unroll
    for (int h = 0; h < NE / 32; ++h) {
      const int c = sub + 8 * h;  // chunk
      const float* src = part + (c * (rl::ROWS + 1) + row) * 4;
      float4 x = *reinterpret_cast<const float4*>(src);
#pragma unroll
      for (int r = 1; r < SPLIT; ++r) {
        const float4 y = *reinterpret_cast<const float4*>(src + r * rl::part_floats<NE>());
        x.x += y.x;
        x.y += y.y;
        x.z += y.z;
        x.w += y.w;
      }
      float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = 4 * c + u;
        if (e >= E) xs[u] = -INFINITY;
        else if (logits_out != nullptr && t < T) logits_out[(size_t)t * E + e] = xs[u];
        nan |= xs[u] != xs[u];
        v[4 * h + u] = xs[u];
      }
    }
    const unsigned group = 0xFFu << (lane & 24);  // the token's lanes
    nan = (__ballot_sync(0xffffffffu, nan) & group) != 0u;
    bool active = t < T && !nan;
    if (t < T && nan && sub == 0) {
      report(&g_err_route, ORDERMOE_DEV_NAN_LOGIT, t);
      for (int j = 0; j < k; ++j) {  // no targets: a later pass skips this token
        topk_idx[(size_t)t * k + j] = -1;
        topk_w[(size_t)t * k + j] = 0.0f;
      }
    }
    // top-k by (logit desc, index asc): each pass takes the largest left, found
    // among a lane's eight and then across the token's lanes. Lane j keeps slot j.
    float my_v = -INFINITY, lmax = -INFINITY;
    int my_e = 0;
    uint32_t used = 0;  // of this lane's experts
    int idx[ORDERMOE_MAX_TOPK];
#pragma unroll
    for (int j = 0; j < ORDERMOE_MAX_TOPK; ++j) {
      idx[j] = 0;
      if (j >= k) continue;  // the same for every lane
      float bv = -INFINITY;
      int be = 1 << 20, bi = 0;
#pragma unroll
      for (int i = 0; i < NE / 8; ++i) {
        const int e = 4 * (sub + 8 * (i >> 2)) + (i & 3);
        // an unused expert, a real one before the padding past E
        if (!((used >> i) & 1u) && e < E && (be == (1 << 20) || v[i] > bv)) {
          bv = v[i];
          be = e;
          bi = i;
        }
      }
      const int own = be;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oe = __shfl_xor_sync(0xffffffffu, be, o);
        if (oe != (1 << 20) && (be == (1 << 20) || ov > bv || (ov == bv && oe < be))) {
          bv = ov;
          be = oe;
        }
      }
      if (own == be && own != (1 << 20)) used |= 1u << bi;
      idx[j] = active ? be : 0;
      if (j == 0) lmax = bv;
      if (sub == j) {
        my_v = bv;
        my_e = be;
      }
    }
    // softmax over all E in fp32, summed in index order (the -inf logits past E
    // add exact zeros); gate weights of the k slots
#pragma unroll
    for (int h = 0; h < NE / 32; ++h) {
      const int c = sub + 8 * h;
      *reinterpret_cast<float4*>(ex + 4 * c) =
          make_float4(expf(v[4 * h] - lmax), expf(v[4 * h + 1] - lmax), expf(v[4 * h + 2] - lmax),
                      expf(v[4 * h + 3] - lmax));
    }
    __syncwarp();
    float denom = 0.0f;
    for (int c = 0; c < (E + 3) / 4; ++c) {
      const float4 x = *reinterpret_cast<const float4*>(ex + 4 * c);
      denom += x.x;
      denom += x.y;
      denom += x.z;
      denom += x.w;
    }
    const float wsel = sub < k ? expf(my_v - lmax) / denom : 0.0f;
    float ssel = 0.0f;
    for (int j = 0; j < k; ++j) ssel += __shfl_sync(0xffffffffu, wsel, (lane & 24) + j);
    if (active && sub < k) {
      topk_idx[(size_t)t * k + sub] = my_e;
      topk_w[(size_t)t * k + sub] = renorm ? wsel / ssel : wsel;
    }
    if (!topk_only && tables_ok) {  // the same for the warp
      const int M = reinterpret_cast<const int32_t*>(tab)[2];
      const float qbar = reinterpret_cast<const float*>(tab)[5];
      const float* Aas = reinterpret_cast<const float*>(tab + off_a(E)) +
                         (active && a < M && loc0 < M ? (a * M + loc0) * M : 0);
      int kind_count[4] = {0, 0, 0, 0};
      select_slots(t, active, sub, idx, E, k, M, qbar, Aas, sm, s_Q, s_Cq, a, loc0, q0, loc, qhat,
                   chosen_expert, chosen_server, kind_out, kind_count);
      flush_kind_counts(sm, kind_count, counters);
    }
  }

  __syncthreads();
  if (s.abort) {
    volatile int* never = &s.zero;
    if (warp == 0 && lane == 0)
      for (int st = 0; st < rl::STAGES; ++st)
        if ((issued_mask >> st) & 1u) mbar_wait(&s.full[st], (last_phase_bits >> st) & 1u, limit_ns, never);
    if (leader && mma_issued) {  // the lane that issued the MMAs
      mma_commit(&s.drain);
      mbar_wait(&s.drain, 0, limit_ns, never);
    }
    __syncthreads();
  }
  if (counters != nullptr && tid < 4 && sm.kind[tid]) atomicAdd(&counters[tid], sm.kind[tid]);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

}  // namespace om

using namespace om;

extern "C" size_t ordermoe_tables_bytes(int E, int M) {
  if (E <= 0 || E > ORDERMOE_MAX_EXPERTS || M <= 0 || M > ORDERMOE_MAX_SERVERS) return 0;
  return om::tables_bytes(E, M);
}

extern "C" int ordermoe_build_tables(const float* sim, const int32_t* group,
                                     const uint8_t* placement, int E, int M, float theta,
                                     float qbar, const double* F, const double* B,
                                     const double* tau, double z, double c, double omega_T,
                                     double omega_Q, void* tables, size_t tables_bytes_,
                                     ordermoe_stream_t stream) {
  OM_TRACE();
  if (!sim || !group || !placement || !F || !B || !tau || !tables)
    return fail(ORDERMOE_ERR_INVALID_ARG, "build_tables: null pointer");
  if (E <= 0 || E > ORDERMOE_MAX_EXPERTS || M <= 0 || M > ORDERMOE_MAX_SERVERS)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "build_tables: need 1 <= E <= 64, 1 <= M <= 32");
  if (tables_bytes_ < om::tables_bytes(E, M))
    return fail(ORDERMOE_ERR_INVALID_ARG, "build_tables: tables buffer too small");
  if (!(qbar >= 0.0f)) return fail(ORDERMOE_ERR_INVALID_ARG, "build_tables: qbar must be >= 0");
  if (!(c > 0.0) || !(z >= 0.0) || !(omega_T >= 0.0) || !(omega_Q >= 0.0))
    return fail(ORDERMOE_ERR_INVALID_ARG, "build_tables: need c > 0, z >= 0, omega >= 0");
  if ((reinterpret_cast<uintptr_t>(tables) & 15u) != 0)
    return fail(ORDERMOE_ERR_INVALID_ARG, "build_tables: tables must be 16-byte aligned");
  build_tables_kernel<<<1, 256, 0, stream>>>(sim, group, placement, E, M, theta, qbar, F, B, tau,
                                             z, c, omega_T, omega_Q,
                                             static_cast<uint8_t*>(tables));
  OM_LAUNCHED("build_tables_kernel");
  return ORDERMOE_OK;
}

template <int D, int NW>
static cudaError_t lookahead_launch(int t0, int T, int E, int Mcap, int k, const int32_t* topk_idx,
                                    const uint8_t* tb, const Lookahead& la, const uint8_t* home,
                                    uint8_t* loc, float* qhat, int32_t* chosen_expert,
                                    uint8_t* chosen_server, uint8_t* kind, int32_t* counters,
                                    cudaStream_t stream) {
  const size_t full = la_smem_fixed(E, D, Mcap, NW) + la_smem_classes(E) + la_smem_rows(E, D, Mcap);
  const size_t smem = full < kLaSmem ? full : kLaSmem;
  static PerDevice attr;
  const int ae = per_device(attr, [] {
    return static_cast<int>(cudaFuncSetAttribute(lookahead_select_kernel<D, NW>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(kLaSmem)));
  });
  if (ae != cudaSuccess) return static_cast<cudaError_t>(ae);
  // a token a warp until the blocks of one wave (one an SM) are full, then
  // more tokens a block, which share its tables
  const long long wave = (long long)num_sms() * NW;
  long long tpb = NW * ((T + wave - 1) / wave);
  if (tpb > kLaMaxTok) tpb = kLaMaxTok;
  // a home's last block may be partly filled: at most one more block a home
  const long long blocks = T / tpb + Mcap;
  return launch_pdl(lookahead_select_kernel<D, NW>, dim3(static_cast<unsigned>(blocks)),
                    dim3(32 * NW), smem, stream, topk_idx, t0, T, E, k, tb, la, Mcap,
                    static_cast<int>(smem), static_cast<int>(tpb), home, loc, qhat, chosen_expert,
                    chosen_server, kind, counters);
}

static int launch_lookahead_select(const int32_t* topk_idx, int T, int E, int k,
                                   const uint8_t* tb, Lookahead la, const uint8_t* home,
                                   uint8_t* loc, float* qhat, int32_t* chosen_expert,
                                   uint8_t* chosen_server, uint8_t* kind, int32_t* counters,
                                   cudaStream_t stream) {
  if (T <= 0) return ORDERMOE_OK;
  // the most servers whose tables fit the stride (the device header has the
  // number; one that does not fit is reported)
  int Mcap = 1;
  while (Mcap < ORDERMOE_MAX_SERVERS && om::tables_bytes(E, Mcap + 1) <= la.stride) ++Mcap;
  // Every block ranks the homes of all tokens of its launch, so the tokens go in
  // launches of at most kLaTokens: 1000000 tokens of 8 experts, 4 servers, H = 2
  // took 8.5 ms in one, 2.3 so (300000 of 64, 8 servers: 1.92 and 1.68).
  constexpr int kLaTokens = 131072;
  for (int t0 = 0; t0 < T; t0 += kLaTokens) {
    const int n = T - t0 < kLaTokens ? T - t0 : kLaTokens;
    const size_t at = (size_t)t0 * k;
    const bool wide = E > kLaNarrow;
    const auto launch = la.H == 2 ? (wide ? lookahead_launch<1, 16> : lookahead_launch<1, 8>)
                        : la.H == 3 ? (wide ? lookahead_launch<2, 16> : lookahead_launch<2, 8>)
                                    : (wide ? lookahead_launch<3, 16> : lookahead_launch<3, 8>);
    const cudaError_t e = launch(t0, n, E, Mcap, k, topk_idx + at, tb, la, home + t0,
                                 loc != nullptr ? loc + t0 : nullptr, qhat != nullptr ? qhat + t0 : nullptr,
                                 chosen_expert + at, chosen_server + at, kind + at, counters, stream);
    if (e != cudaSuccess) return cuda_fail(e, "lookahead_select_kernel");
  }
  return ORDERMOE_OK;
}

static int launch_select_lanes(const int32_t* topk_idx, int T, int E, int k, const uint8_t* tb,
                               const uint8_t* home, uint8_t* loc, float* qhat,
                               int32_t* chosen_expert, uint8_t* chosen_server, uint8_t* kind,
                               int32_t* counters, size_t tab_smem, cudaStream_t stream) {
  if (T <= 0) return ORDERMOE_OK;
  const int per_block = (kLaneThreads / 32) * kLaneTokens;
  long long blocks = (T + per_block - 1) / per_block;
  const long long cap = 4LL * num_sms();
  if (blocks > cap) blocks = cap;
  OM_LAUNCH_PDL("select_lanes_kernel", select_lanes_kernel, dim3(static_cast<int>(blocks)),
                dim3(kLaneThreads), tab_smem, stream, topk_idx, T, E, k, tb, home, loc, qhat,
                chosen_expert, chosen_server, kind, counters);
  return ORDERMOE_OK;
}

// Selection from given logits: the tables, the staged delay table and the
// logits' chunks in shared memory.
template <int EM>
constexpr size_t select_smem(int E) {
  return sizeof(float) * (2 * (size_t)E * E + kDelayStage + EM * 128);
}

template <int EM>
static cudaError_t launch_select(const float* logits_in, int T, int E, int k, int renorm,
                                 const uint8_t* tb, const Lookahead& la, const uint8_t* home,
                                 uint8_t* loc, float* qhat, float* logits_out, int32_t* topk_idx,
                                 float* topk_w, int32_t* chosen_expert, uint8_t* chosen_server,
                                 uint8_t* kind, int32_t* counters, cudaStream_t stream) {
  static PerDevice attr;
  const int ae = per_device(attr, [] {
    return static_cast<int>(cudaFuncSetAttribute(select_kernel<EM>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(select_smem<EM>(EM))));
  });
  if (ae != cudaSuccess) return static_cast<cudaError_t>(ae);
  return launch_pdl(select_kernel<EM>, dim3((T + 127) / 128), dim3(128), select_smem<EM>(E), stream,
                    logits_in, T, E, k, renorm, tb, home, loc, qhat, logits_out, topk_idx, topk_w,
                    chosen_expert, chosen_server, kind, counters, la);
}

template <int NE>
static cudaError_t router_attr() {
  return cudaFuncSetAttribute(router_select_kernel<NE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              rt::smem_bytes<NE>(NE));
}

template <int NE>
static cudaError_t router_lanes_attr() {
  return cudaFuncSetAttribute(router_lanes_kernel<NE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              rl::smem_bytes<NE>(NE));
}

static int route_select_impl(const uint16_t* X, const uint16_t* W_r, const float* logits_in, int T,
                             int E, int d, int k, int renorm, const void* tables,
                             size_t tables_bytes_, Lookahead la, const uint8_t* home, uint8_t* loc,
                             float* qhat, float* logits_out, int32_t* topk_idx, float* topk_w,
                             int32_t* chosen_expert, uint8_t* chosen_server, uint8_t* kind,
                             int32_t* counters, cudaStream_t stream) {
  if (T < 0) return fail(ORDERMOE_ERR_INVALID_ARG, "route_select: T < 0");
  if (E <= 0 || E > ORDERMOE_MAX_EXPERTS || k <= 0 || k > ORDERMOE_MAX_TOPK || k > E)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "route_select: need 1 <= k <= min(E, 8), E <= 64");
  if (!tables || !home || !topk_idx || !topk_w || !chosen_expert || !chosen_server || !kind)
    return fail(ORDERMOE_ERR_INVALID_ARG, "route_select: null pointer");
  if ((loc == nullptr) != (qhat == nullptr))
    return fail(ORDERMOE_ERR_INVALID_ARG, "route_select: give both loc and qhat, or neither");
  if (logits_in == nullptr) {
    if (!X || !W_r) return fail(ORDERMOE_ERR_INVALID_ARG, "route_select: X/W_r null without logits_in");
    if (d <= 0 || d % 64 != 0)
      return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "route_select: d must be a positive multiple of 64");
    if (!aligned16(X) || !aligned16(W_r))
      return fail(ORDERMOE_ERR_INVALID_ARG, "route_select: X and W_r must be 16-byte aligned");
  }
  if (tables_bytes_ < om::tables_bytes(E, 1))
    return fail(ORDERMOE_ERR_INVALID_ARG, "route_select: tables buffer smaller than E needs");
  if (T == 0) return ORDERMOE_OK;
  const uint8_t* tb = static_cast<const uint8_t*>(tables);
  const size_t tab_smem = sizeof(float) * 2 * E * E;  // the lane kernel's
  static_assert(sizeof(float) * 2 * 64 * 64 + sizeof(SelSmem) <= 48 * 1024, "launches without an attribute");
  const int blocks = (T + 127) / 128;
  if (logits_in != nullptr) {
    const auto launch = E <= 8 ? launch_select<8> : E <= 16 ? launch_select<16>
                        : E <= 32 ? launch_select<32> : launch_select<64>;
    const cudaError_t sel_err = launch(logits_in, T, E, k, renorm, tb, la, home, loc, qhat, logits_out,
                                       topk_idx, topk_w, chosen_expert, chosen_server, kind, counters,
                                       stream);
    if (sel_err != cudaSuccess) return cuda_fail(sel_err, "select_kernel");
    return la.H > 1 ? launch_lookahead_select(topk_idx, T, E, k, tb, la, home, loc, qhat,
                                              chosen_expert, chosen_server, kind, counters, stream)
                    : ORDERMOE_OK;
  }
  // many experts (long candidate lists per slot): the router writes the
  // targets and select_lanes_kernel selects with eight lanes per token
  const bool lanes = la.H == 1 && E > 16;
  if (lanes) la.topk_only = 1;
  CUtensorMap mX, mW;
  int rc;
  const int NE = E <= 16 ? 16 : (E <= 32 ? 32 : 64);
  const uint64_t lim = wait_limit_ns();
  const int kblocks = d / rt::BK;
  // Small batches of many experts: one CTA for every 16 tokens, all resident at
  // once (up to 2432 tokens on 152 SMs). Larger ones fill the SMs with the tokens,
  // and the selection in rounds would be longer than a launch over all SMs.
  // (d >= 512: narrower routers are a few K blocks.)
  const int rl_split = NE == 32 ? rl::split<32>() : rl::split<64>();
  const int rl_tile = rl_split * rl::ROWS;
  const long long rl_tiles = (T + rl_tile - 1) / rl_tile;
  const bool small = E > 16 && rl_tiles * rl_split <= num_sms() && kblocks >= 8;
  if ((rc = make_tmap_bf16(&mX, X, T, d, small ? rl_tile : 128))) return rc;
  if ((rc = make_tmap_bf16(&mW, W_r, E, d, NE))) return rc;
  // split K over a cluster so that about one CTA per SM streams X
  const int smax = NE == 16 ? rt::max_split<16>() : (NE == 32 ? rt::max_split<32>() : rt::max_split<64>());
  int split = 1;
  while (split * 2 <= smax && (long long)blocks * split * 2 <= num_sms() && split * 2 <= kblocks)
    split *= 2;
  // once per device, for the most experts of each width (not at every launch)
  static PerDevice attr_cache;
  const cudaError_t ae = static_cast<cudaError_t>(per_device(attr_cache, [] {
    cudaError_t e = router_attr<16>();
    if (e == cudaSuccess) e = router_attr<32>();
    if (e == cudaSuccess) e = router_attr<64>();
    if (e == cudaSuccess) e = router_lanes_attr<32>();
    if (e == cudaSuccess) e = router_lanes_attr<64>();
    return static_cast<int>(e);
  }));
  if (ae != cudaSuccess) return cuda_fail(ae, "cudaFuncSetAttribute(router_select_kernel)");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks * split, 1, 1);
  cfg.blockDim = dim3(rt::THREADS, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // waits in the kernel
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_on(stream) ? 2 : 1;
  cudaError_t le;
  if (small) {
    cfg.gridDim = dim3(static_cast<unsigned>(rl_tiles * rl_split), 1, 1);
    cfg.blockDim = dim3(rl::THREADS, 1, 1);
    attr[0].val.clusterDim.x = rl_split;
    const int only = la.H > 1 ? 1 : 0;
    if (NE == 32) {
      cfg.dynamicSmemBytes = rl::smem_bytes<32>(E);
      OM_CUDA(cudaLaunchKernelEx(&cfg, router_lanes_kernel<32>, mX, mW, T, E, d, k, renorm, tb, home, loc,
                                 qhat, logits_out, topk_idx, topk_w, chosen_expert, chosen_server, kind,
                                 counters, lim, only));
    } else {
      cfg.dynamicSmemBytes = rl::smem_bytes<64>(E);
      OM_CUDA(cudaLaunchKernelEx(&cfg, router_lanes_kernel<64>, mX, mW, T, E, d, k, renorm, tb, home, loc,
                                 qhat, logits_out, topk_idx, topk_w, chosen_expert, chosen_server, kind,
                                 counters, lim, only));
    }
    return only ? launch_lookahead_select(topk_idx, T, E, k, tb, la, home, loc, qhat, chosen_expert,
                                          chosen_server, kind, counters, stream)
                : ORDERMOE_OK;
  }
#define OM_RT_LAUNCH(N)                                                                          \
  do {                                                                                           \
    cfg.dynamicSmemBytes = rt::smem_bytes<N>(E);                                                 \
    le = cudaLaunchKernelEx(&cfg, router_select_kernel<N>, mX, mW, T, E, d, k, renorm, tb, home, \
                            loc, qhat, logits_out, topk_idx, topk_w, chosen_expert,              \
                            chosen_server, kind, counters, lim, split, la);                      \
  } while (0)
  if (NE == 16) OM_RT_LAUNCH(16);
  else if (NE == 32) OM_RT_LAUNCH(32);
  else OM_RT_LAUNCH(64);
#undef OM_RT_LAUNCH
  if (le != cudaSuccess) return cuda_fail(le, "router_select_kernel launch");
  OM_LAUNCHED("router_select_kernel");
  if (la.H > 1)
    return launch_lookahead_select(topk_idx, T, E, k, tb, la, home, loc, qhat, chosen_expert,
                                   chosen_server, kind, counters, stream);
  if (lanes)
    return launch_select_lanes(topk_idx, T, E, k, tb, home, loc, qhat, chosen_expert,
                               chosen_server, kind, counters, tab_smem, stream);
  return ORDERMOE_OK;
}

extern "C" int ordermoe_route_select(const uint16_t* X, const uint16_t* W_r, const float* logits_in,
                                     int T, int E, int d, int k, int renorm, const void* tables,
                                     size_t tables_bytes_, const uint8_t* home, uint8_t* loc,
                                     float* qhat, float* logits_out, int32_t* topk_idx,
                                     float* topk_w, int32_t* chosen_expert,
                                     uint8_t* chosen_server, uint8_t* kind, int32_t* counters,
                                     ordermoe_stream_t stream) {
  OM_TRACE();
  Lookahead la{1, 0, nullptr};
  return route_select_impl(X, W_r, logits_in, T, E, d, k, renorm, tables, tables_bytes_, la, home,
                           loc, qhat, logits_out, topk_idx, topk_w, chosen_expert, chosen_server,
                           kind, counters, stream);
}

extern "C" int ordermoe_route_select_lookahead(
    const uint16_t* X, const uint16_t* W_r, const float* logits_in, int T, int E, int d, int k,
    int renorm, const void* tables, size_t tables_stride, int H, const float* P,
    const uint8_t* home, uint8_t* loc, float* qhat, float* logits_out, int32_t* topk_idx,
    float* topk_w, int32_t* chosen_expert, uint8_t* chosen_server, uint8_t* kind,
    int32_t* counters, ordermoe_stream_t stream) {
  OM_TRACE();
  if (H < 1 || H > 4) return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "route_select_lookahead: need 1 <= H <= 4");
  if (E <= 0 || E > ORDERMOE_MAX_EXPERTS)
    return fail(ORDERMOE_ERR_UNSUPPORTED_SHAPE, "route_select_lookahead: need 1 <= E <= 64");
  if (H > 1 && (!P || tables_stride < om::tables_bytes(E, 1) || (tables_stride & 15u)))
    return fail(ORDERMOE_ERR_INVALID_ARG,
                "route_select_lookahead: need P and a 16-byte multiple table stride for H > 1");
  Lookahead la{H, tables_stride, P};
  return route_select_impl(X, W_r, logits_in, T, E, d, k, renorm, tables, tables_stride, la, home,
                           loc, qhat, logits_out, topk_idx, topk_w, chosen_expert, chosen_server,
                           kind, counters, stream);
}
