// Persistent drafter: the whole K-step draft rollout of one environment (Sec. 3.2 "Draft Generation
// Procedure", Eq. (3)) in ONE kernel launch, for small batches where the rollout is latency-bound.
//
// One thread-block cluster of cs = 8 or 4 CTAs serves one environment at a time; the sequence is one 16-row tile of mma.sync
// m16n8k16.  The work is split so that little has to travel and nothing is computed twice that matters:
//   * the residual stream belongs to rows: a CTA keeps 16 / cs token rows in registers (16 cs threads a row) and does everything
//     that is local to a token -- embedding, LayerNorms, the folded cross-attention, output head, scheduler step;
//   * the weights belong to columns: CTA r computes queries and keys of its head, the d / cs value columns and the MLP
//     columns [4 r d / cs, +4 d / cs) for all 16 rows, and the products that follow (attention projection, MLP down) over
//     just those columns as k: cs partial sums per output, added by the row's owner in a fixed order.
// So a block exchanges four times: normalised rows to everyone (1 KB per CTA and peer at d = 256, cs = 8), partial sums to their row
// owners (2 KB), and the same again for the MLP; queries, keys, values and MLP activations never leave a CTA.
// An exchange costs about 770 clocks plus 390 per KB (measured); the layout before this one (every activation
// replicated in every CTA, LayerNorms and the cross-attention recomputed by all) exchanged 2.4 KB four times on average
// and needed 33 k clocks per d = 256 block against 17 k now (9.3 us with the block's share of a draft step, cs = 8).
// cs = 4 takes longer (12.2 us for the same) and serves 33 environments at a time instead of 15.  Both give the same bits: what is summed
// over CTAs is summed pairwise, and a CTA of four forms its two halves' sums apart (dc_kloop); what is summed over a row is summed in
// four groups of columns.
//
// Weights are laid out once, when they are loaded, in the order in which the lanes of a warp consume them (dc_pack_kernel):
// a lane's operand of two MMAs is one 16-byte word, a warp reads 512 contiguous bytes, and a CTA's slice of a matrix is
// one contiguous piece.  A producer warp brings the pieces to shared memory by bulk copies: all of them once per launch
// where a CTA's share of the whole network fits, otherwise in 16 KB chunks through a ring that runs ahead of the
// computation across layers and forwards (the weights do not depend on it), so that a linear layer rarely waits for the L2.
// Each layer's LayerNorm parameters and biases and the memory tokens' folded tables travel the same way.  Eight warps compute.
//
// What a stage exchanges travels as 16-byte st.async stores that also count their bytes on an mbarrier of the receiving
// CTA; a CTA goes on as soon as the bytes of all CTAs of the cluster have arrived (a bounded mbarrier wait), with no
// release fence and no cluster-wide barrier per stage.  Two mbarriers alternate between consecutive stages: a CTA
// can run at most one stage ahead of the slowest one (it needs everybody's bytes of the previous stage), so the
// bytes of stage s + 1 never land on the barrier that still counts stage s.  The same reasoning covers the
// buffers: what a fast CTA writes remotely in stage s + 1 is never what a slower one still reads in stage s.
// (TSDP_NO_ASYNC_BCAST selects plain distributed-shared-memory stores and one remote arrival per CTA and stage.)
// All CTAs of a cluster make the same sequence of stages because the control flow depends only on (t[b], k).
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"
#include "gemm_tcgen05.cuh"
#include "net_kernels.cuh"

namespace tsdp {
namespace cg = cooperative_groups;

// CTAs per cluster: 8 (the portable maximum), or 4 where more environments wait than clusters of 8 run at once
constexpr int DC_COMPUTE = 256;   // compute threads; one producer warp behind them
constexpr int DC_THREADS = DC_COMPUTE + 32;
constexpr int DC_WARPS = DC_COMPUTE / 32;
constexpr int DC_ROWS = 16;       // one m16 tile: H <= 16
__host__ __device__ constexpr int dc_own(int cs) { return DC_ROWS / cs; }   // token rows a CTA owns
constexpr int DC_MAX_LAYERS = 8;
constexpr int DC_MAX_NK = 4;      // memory tokens: time token + at most 3 observation tokens
constexpr int DC_MAX_NKH = 16;    // folded cross-attention: (memory token, head) pairs
constexpr int DC_CHUNK = 16384;   // bytes of a ring slot
constexpr int DC_MAX_SLOTS = 8;

__device__ __forceinline__ uint32_t dc_mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void dc_st_async16(uint32_t remote, const uint4& v, uint32_t remote_bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];"
               ::"r"(remote), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(remote_bar) : "memory");
}
__device__ __forceinline__ void dc_st_cluster16(uint32_t remote, const uint4& v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(remote), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void dc_bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void dc_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }      // the compute warps

template <int CS>
__device__ __forceinline__ void dc_row_sync(int row) { asm volatile("bar.sync %0, %1;" ::"r"(2 + row), "n"(16 * CS) : "memory"); }      // the warps of an owned row

// ---- weight layout.  A CTA's share of a layer, one piece ("slab") behind the other (dh = head width, v = d / cs columns, cs CTAs):
//   0 [query dh | key dh of its head | its value columns v] x d | 1 attention projection, d x (its v columns, padded to 32) |
//   2 MLP up m x d | 3 MLP down d x (its m columns), m = 4 d / cs | not needed when the cross-attention is folded: 4 its query dh x d |
//   5 output projection, d x (its v columns, padded to 32)
// and a slab [n x K] is [K / KC][n / 8 column tiles][KC / 32][32 lanes] 16-byte words, KC = min(K, 256): the word of lane
// (g, tg) = (lane / 4, lane % 4) holds W[8 tile + g][k0 + {0, 8, 16, 24} + 2 tg .. + 1], the B operands of two MMAs.
__host__ __device__ constexpr int dc_kv(int d, int cs) { return d / cs < 32 ? 32 : d / cs; }
__host__ __device__ constexpr int dc_slab_rows(int d, int dh, int s, int cs) {
  return s == 0 ? 2 * dh + d / cs : (s == 2 ? 4 * d / cs : (s == 4 ? dh : d));
}
__host__ __device__ constexpr int dc_slab_k(int d, int s, int cs) { return s == 1 || s == 5 ? dc_kv(d, cs) : (s == 3 ? 4 * d / cs : d); }
__host__ __device__ constexpr int dc_slab_bytes(int d, int dh, int s, int cs) { return dc_slab_rows(d, dh, s, cs) * dc_slab_k(d, s, cs) * 2; }
__host__ __device__ constexpr int dc_slab_off(int d, int dh, int s, int cs) { int o = 0; for (int i = 0; i < s; ++i) o += dc_slab_bytes(d, dh, i, cs); return o; }
__host__ __device__ constexpr int dc_layer_bytes(int d, int dh, int cs) { return dc_slab_off(d, dh, 6, cs); }
// floats of a layer's parameters in a CTA: 6 LayerNorm vectors, bo, bo2, b2 (whole), its biases of slab 0, of slab 2, of slab 4
__host__ __device__ constexpr int dc_par_floats(int d, int dh, int cs) { return 9 * d + 2 * dh + d / cs + 4 * d / cs + dh; }
// column tiles of a slab that a warp takes in one pass over it: all of them where that is at most 4 tiles of 128 k or 3 of 256 (the
// accumulators, and the chunks of a pass, which are resident together)
__host__ __device__ constexpr int dc_tiles_per_warp(int d, int dh, int s, int cs) {
  const int per = (dc_slab_rows(d, dh, s, cs) / 8 + DC_WARPS - 1) / DC_WARPS, most = dc_slab_k(d, s, cs) <= 128 ? 4 : 3;
  return per <= most ? per : (most == 3 ? 2 : most);
}
__host__ __device__ constexpr int dc_min_slots(int d, int dh, int cs) {      // chunks of the largest pass
  int most = 0;
  for (int s = 0; s < 6; ++s) {
    const int nt = dc_slab_rows(d, dh, s, cs) / 8, pt = dc_tiles_per_warp(d, dh, s, cs) * DC_WARPS;
    const int n = ((nt < pt ? nt : pt) * dc_slab_k(d, s, cs) * 16 + DC_CHUNK - 1) / DC_CHUNK;
    most = n > most ? n : most;
  }
  return most;
}
// element offset of weight (n, k) inside its slab
__host__ __device__ inline int dc_frag_index(int n, int k, int rows, int K) {
  const int KC = K < 256 ? K : 256, kc = k / KC, kk = k % KC, tile = n >> 3, g = n & 7, kb = kk >> 5, r = kk & 31;
  const int tg = (r & 7) >> 1;
  return (((kc * (rows >> 3) + tile) * (KC >> 5) + kb) * 32 + (g * 4 + tg)) * 8 + ((r >> 3) << 1) + (r & 1);
}
// where element (n, k) of slab s of CTA `rank` comes from: row and column of the full matrix [out, in]; false: padding
__host__ __device__ inline bool dc_slab_source(int d, int dh, int cs, int rank, int s, int n, int k, int* row, int* col) {
  const int heads = d / dh, hd = rank * heads / cs, v = d / cs, m = 4 * d / cs;      // cs / heads CTAs share a head
  *row = n; *col = k;
  if (s == 0) *row = n < dh ? hd * dh + n : (n < 2 * dh ? d + hd * dh + (n - dh) : 2 * d + rank * v + (n - 2 * dh));
  else if (s == 1 || s == 5) { *col = rank * v + k; return k < v; }
  else if (s == 2) *row = rank * m + n;
  else if (s == 3) *col = rank * m + k;
  else *row = hd * dh + n;
  return true;
}
// W [out, in] bf16 of row pitch ld -> slab `s` of every CTA's share of a layer
__global__ void dc_pack_kernel(const __nv_bfloat16* __restrict__ W, int ld, __nv_bfloat16* __restrict__ layer, int d, int dh, int s, int cs) {
  const int rows = dc_slab_rows(d, dh, s, cs), K = dc_slab_k(d, s, cs);
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)rows * K * cs) return;
  const int rank = (int)(i / ((long long)rows * K)), n = (int)(i / K % rows), k = (int)(i % K);
  int row, col;
  const bool real = dc_slab_source(d, dh, cs, rank, s, n, k, &row, &col);
  layer[(size_t)rank * (dc_layer_bytes(d, dh, cs) / 2) + dc_slab_off(d, dh, s, cs) / 2 + dc_frag_index(n, k, rows, K)] =
      real ? W[(size_t)row * ld + col] : __float2bfloat16_rn(0.f);
}
struct DcParSrc { const float* whole[9]; const float *bqkv, *b1, *bq2; };      // ln1 g, b, ln2 g, b, ln3 g, b, bo, bo2, b2
__global__ void dc_pack_par_kernel(DcParSrc src, float* __restrict__ layer, int d, int dh, int cs) {
  const int rank = blockIdx.x;
  float* o = layer + (size_t)rank * dc_par_floats(d, dh, cs);
  for (int j = 0; j < 9; ++j, o += d)
    for (int i = threadIdx.x; i < d; i += blockDim.x) o[i] = src.whole[j][i];
  const int slabs[3] = {0, 2, 4};
  const float* bias[3] = {src.bqkv, src.b1, src.bq2};
  for (int j = 0; j < 3; ++j) {
    const int n = dc_slab_rows(d, dh, slabs[j], cs);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      int row, col;
      dc_slab_source(d, dh, cs, rank, slabs[j], i, 0, &row, &col);
      o[i] = bias[j][row];
    }
    o += n;
  }
}

struct DcParams {
  const __nv_bfloat16* Wf;                                   // [layers][cs ranks][dc_layer_bytes] in fragment order
  const float* parf;                                         // [layers][cs ranks][dc_par_floats]
  int layers, heads, H, A, To, T;
  const float *W_in, *b_in, *pos;                            // [A, d], [d], [H, d]
  const float *lnf_g, *lnf_b, *W_outT, *b_out;               // W_outT [A, d]
  const float *kv_time, *kv_obs;                             // [T, L*2d], [B*To, L*2d]
  // cross-attention folded into the memory tokens (xattn_fold.cuh): per-token tables kq [L][heads][d],
  // ut [L][heads/2][d][2] (bf16) and c [L][heads] (fp32); fold = 0 runs the projections and the attention instead
  const __nv_bfloat16 *kq_time, *ut_time, *kq_obs, *ut_obs;
  const float *c_time, *c_obs;
  int fold;
  int async_bcast;                                           // 1: slices travel by st.async and are counted by the receivers' mbarriers
  int* status;                                               // set to 5 if a wait gives up
  DdpmTables S;
  float* xt; long long xs_b;                                 // candidates [B, Kmax+1, D]
  float* muhat; long long ms_b;                              // drafter means [B, Kmax, D]
  const int* t;
  const uint64_t* seed;
  int resident, n_slots;                                     // weights in shared memory for the whole launch, or slots of the ring
  // mode 0: draft rollout (K steps per slot, writes xt / muhat).  mode 1: verification -- one forward per
  // (slot, candidate c < C) at timestep t[slot] - c, reading xt[slot, c] and writing eps[slot, c].
  int mode, C;
  float* eps; long long es_b;
  const EnvParams* envp;                                     // per-request draft cap, or null
  const int* item;                                           // slot -> request it serves, or null
  int B, K;
};

// Shared-memory plan of one CTA (bytes), for model width d and head width dh.
struct DcSmem {
  int n_slots;      // ring slots (0: resident)
  int off_w, off_par, off_xa, off_q, off_o, off_f, off_recv, off_kq, off_u, off_x, off_xr, off_red, off_head, off_bar, total;
};
__host__ __device__ inline DcSmem dc_smem_plan(int d, int dh, int cs, int layers, int A, bool resident, int limit) {
  DcSmem p{};
  int o = 0;
  auto take = [&](int bytes) { int r = o; o += (bytes + 127) & ~127; return r; };
  p.off_xa = take(DC_ROWS * (d + 8) * 2);                        // normalised rows of everyone
  p.off_q = take(DC_ROWS * (2 * dh + d / cs + 8) * 2);        // queries, keys of the head, value columns (all 16 rows)
  p.off_o = take(DC_ROWS * (dc_kv(d, cs) + 8) * 2);                  // attention output, this CTA's columns
  p.off_f = take(DC_ROWS * (4 * d / cs + 8) * 2);                     // MLP activations, this CTA's columns
  p.off_recv = take(DC_ROWS * d * 4);                     // partial sums of the owned rows
  p.off_kq = take(DC_MAX_NKH * d * 2);                           // folded cross-attention: kq rows; otherwise keys, values of the head
  p.off_u = take(DC_MAX_NKH / 2 * d * 4);                        // u rows (head pairs in one word)
  p.off_x = take(dc_own(cs) * ((A + 3) & ~3) * 4 * 4);               // latent, eps, noise and sigma of the owned rows
  p.off_xr = take(dc_own(cs) * d * 4);                               // an owned row's normalised values, fp32
  p.off_red = take(512);                                         // row statistics [2 uses][own][4 groups of d / 4 columns] (mean, M2), scores [own][16]
  p.off_head = take((2 * d + A * d + 64) * 4);
  p.off_par = take((resident ? layers : 2) * dc_par_floats(d, dh, cs) * 4);
  p.off_bar = take(256);
  p.off_w = o;
  if (resident) { p.total = o + layers * dc_layer_bytes(d, dh, cs); return p; }
  const int n = (limit - o) / DC_CHUNK;
  p.n_slots = n > DC_MAX_SLOTS ? DC_MAX_SLOTS : n;
  p.total = p.n_slots >= dc_min_slots(d, dh, cs) ? o + p.n_slots * DC_CHUNK : limit + 1;
  return p;
}

template <int I, int N, typename F>
__device__ __forceinline__ void dc_passes(F f) {      // f(0), f(1), .. f(N - 1) with compile-time arguments
  if constexpr (I < N) { f(std::integral_constant<int, I>{}); dc_passes<I + 1, N>(f); }
}
// One warp's k loop of a linear layer: c[t] = X[16, k32 blocks 0 .. NKB) * (its tile t)^T, two accumulator chains per
// tile; base[t] is the shared-memory address of this lane's words of the tile.  All warps read all of X, so the loop is bound by
// shared-memory reads (d = 256, 16 tiles: 64 KB of X and 64 KB of weights, 1024 clocks at 128 B per clock); `ready` says when X
// may be read, and the first half of the weights is fetched before that, while X is still on its way from the other CTAs.
// HALVES = 2: the two halves of k are summed apart and then added, as two CTAs of a larger cluster would have.
__device__ __forceinline__ uint4 dc_lds16(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
template <int TPW, int NKB, int HALVES, typename Ready>
__device__ __forceinline__ void dc_kloop(const __nv_bfloat16* X, int px, float (&c)[TPW][4], const uint32_t (&base)[TPW], Ready ready) {
  constexpr int PRE = NKB < 4 ? NKB : 4;
  const int lane = threadIdx.x & 31;
  float e[TPW][4], first[HALVES == 2 ? TPW : 1][4];
  uint4 pre[TPW][PRE];
#pragma unroll
  for (int t = 0; t < TPW; ++t) {
    c[t][0] = c[t][1] = c[t][2] = c[t][3] = 0.f; e[t][0] = e[t][1] = e[t][2] = e[t][3] = 0.f;
#pragma unroll
    for (int kb = 0; kb < PRE; ++kb) pre[t][kb] = dc_lds16(base[t] + kb * 512);
  }
  ready();
  const __nv_bfloat16* xa = X + (lane & 15) * px + 8 * (lane >> 4);
#pragma unroll
  for (int kb = 0; kb < NKB; ++kb) {
    uint32_t a1[4], a2[4];
    ldmatrix_x4(a1, xa + kb * 32);
    ldmatrix_x4(a2, xa + kb * 32 + 16);
#pragma unroll
    for (int t = 0; t < TPW; ++t) {
      const uint4 w = kb < PRE ? pre[t][kb < PRE ? kb : 0] : dc_lds16(base[t] + kb * 512);
      mma_bf16_16816(c[t], a1, w.x, w.y);
      mma_bf16_16816(e[t], a2, w.z, w.w);
    }
    if (HALVES == 2 && kb == NKB / 2 - 1) {
#pragma unroll
      for (int t = 0; t < TPW; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) { first[t][i] = c[t][i] + e[t][i]; c[t][i] = e[t][i] = 0.f; }
    }
  }
#pragma unroll
  for (int t = 0; t < TPW; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) c[t][i] = HALVES == 2 ? first[t][i] + (c[t][i] + e[t][i]) : c[t][i] + e[t][i];
}

template <int D_MODEL, int DH, int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(DC_THREADS, 1)
drafter_cluster_kernel(const __grid_constant__ DcParams P) {
  extern __shared__ __align__(128) uint8_t dc_smem[];
  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int cid = blockIdx.x / CS, ncl = gridDim.x / CS;
  // An owned row is four groups of d / 4 columns; a warp holds VG of them, a lane V2 neighbouring columns of each.  What is summed over a row is
  // summed group by group, so that it does not depend on the cluster's size.
  constexpr int d = D_MODEL, OWN = dc_own(CS), WPR = DC_WARPS / OWN, VG = 4 / WPR, V2 = d / 128;
  constexpr int VW = d / CS, MW = 4 * d / CS, NQ = 2 * DH + VW;                // value and MLP columns of this CTA; columns of slab 0
  constexpr int PX = d + 8, PQ = NQ + 8, PO = dc_kv(d, CS) + 8, PF = MW + 8;
  constexpr int PL = dc_par_floats(d, DH, CS), HEADS = d / DH;
  static_assert(WPR >= 1 && HEADS <= CS && VW / 16 <= 4, "a CTA works on one head, its first warps on the attention");
  const bool resident = P.resident != 0, use_async = P.async_bcast != 0;
  const DcSmem pl = dc_smem_plan(d, DH, CS, P.layers, P.A, resident, DC_CHUNK * 1024);      // (offsets only: the number of slots is the host's)
  const int n_slots = P.n_slots;
  __nv_bfloat16* xa = reinterpret_cast<__nv_bfloat16*>(dc_smem + pl.off_xa);
  __nv_bfloat16* qs = reinterpret_cast<__nv_bfloat16*>(dc_smem + pl.off_q);
  __nv_bfloat16* os = reinterpret_cast<__nv_bfloat16*>(dc_smem + pl.off_o);
  __nv_bfloat16* fs = reinterpret_cast<__nv_bfloat16*>(dc_smem + pl.off_f);
  float* recv = reinterpret_cast<float*>(dc_smem + pl.off_recv);
  const __nv_bfloat16* skq = reinterpret_cast<const __nv_bfloat16*>(dc_smem + pl.off_kq);
  const uint32_t* su = reinterpret_cast<const uint32_t*>(dc_smem + pl.off_u);
  const int H = P.H, A = P.A, AP = (A + 3) & ~3, D = H * A, L = P.layers, NK = 1 + P.To, NKH = NK * HEADS;
  float* sx = reinterpret_cast<float*>(dc_smem + pl.off_x);          // [OWN][AP]
  float* seps = sx + OWN * AP;                                       // [OWN][AP]
  float* sxr = reinterpret_cast<float*>(dc_smem + pl.off_xr);        // [OWN][d]
  float2* sstat = reinterpret_cast<float2*>(dc_smem + pl.off_red);   // [2 uses][OWN][4 groups]
  float* sscore = reinterpret_cast<float*>(dc_smem + pl.off_red + 64 * OWN);   // [OWN][16]
  float* shead = reinterpret_cast<float*>(dc_smem + pl.off_head);
  float* spar = reinterpret_cast<float*>(dc_smem + pl.off_par);
  const uint32_t sbase = ptx::smem_u32(dc_smem), bar0 = sbase + pl.off_bar, ring = sbase + pl.off_w;
  // barriers: stage hand-over 0, 1 | resident weights 2 | parameters full 3, 4, empty 5, 6 | tables full 7, empty 24 |
  // ring full 8 .., empty 16 ..
  auto bar_of = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) ptx::mbar_init(bar_of(i), use_async ? 1 : CS);
    for (int i : {2, 3, 4, 7}) ptx::mbar_init(bar_of(i), 1);
    for (int i : {5, 6, 24}) ptx::mbar_init(bar_of(i), DC_WARPS);
    for (int i = 0; i < DC_MAX_SLOTS; ++i) { ptx::mbar_init(bar_of(8 + i), 1); ptx::mbar_init(bar_of(16 + i), DC_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  bool failed = false;      // a wait has given up (reported): the rest of the launch does not wait again
  auto wait_bar = [&](uint32_t bar, uint32_t parity) {
    if (failed) return;
    if (!ptx::mbar_wait_thread(bar, parity)) { failed = true; atomicExch(P.status, 5); }
  };
  const int n_slabs = P.fold ? 4 : 6;
  int chunks_layer = 0;
#pragma unroll
  for (int s = 0; s < 6; ++s)
    if (s < 4 || n_slabs == 6) chunks_layer += (dc_slab_bytes(d, DH, s, CS) + DC_CHUNK - 1) / DC_CHUNK;

  // ---- once per launch (compute warps): head parameters; zeroed activations
  if (warp < DC_WARPS) {
    for (int i = threadIdx.x; i < d; i += DC_COMPUTE) { shead[i] = P.lnf_g[i]; shead[d + i] = P.lnf_b[i]; }
    for (int i = threadIdx.x; i < A * d; i += DC_COMPUTE) shead[2 * d + i] = P.W_outT[i];
    for (int i = threadIdx.x; i < A; i += DC_COMPUTE) shead[2 * d + A * d + i] = P.b_out[i];
    uint32_t* z = reinterpret_cast<uint32_t*>(dc_smem);              // xa, q, o, f: one behind the other
    for (int i = threadIdx.x; i < pl.off_recv / 4; i += DC_COMPUTE) z[i] = 0u;
    for (int i = threadIdx.x; i < 4 * OWN * AP; i += DC_COMPUTE) sx[i] = 0.f;
  }
  cluster.sync();
  const float *lnf_g = shead, *lnf_b = shead + d, *woutT = shead + 2 * d, *bout = shead + 2 * d + A * d;

  // forwards this cluster runs (the same for every CTA and every warp)
  const int C = P.mode == 1 ? P.C : 1;
  auto steps = [&](int slot, int cand) {       // forwards of a work item: 0 for a finished slot or a candidate beyond t = 0
    const int tb = P.t[slot];
    if (P.mode == 1) return tb >= 0 && cand <= tb ? 1 : 0;
    return tb < 0 ? 0 : min(min(P.K, env_draft_cap(P.envp, item_of(P.item, slot), tb, P.K, P.T)), tb);
  };

  if (warp == DC_WARPS) {
    // ================================================================ producer: weights, parameters, tables, ahead of the computation
    if (ptx::elect_one()) {
      auto wsrc = [&](int l) { return reinterpret_cast<const uint8_t*>(P.Wf) + ((size_t)l * CS + rank) * dc_layer_bytes(d, DH, CS); };
      auto psrc = [&](int l) { return P.parf + ((size_t)l * CS + rank) * PL; };
      int slot = 0, pre_chunks = 0;
      uint32_t round = 0, n_layer = 0;          // rounds through the ring; layers whose parameters have been asked for
      auto par_load = [&](int l) {
        const uint32_t n = n_layer++, b = n & 1u;
        if (n >= 2) wait_bar(bar_of(5 + (int)b), ((n >> 1) - 1u) & 1u);
        if (failed) return;
        ptx::mbar_expect_tx(bar_of(3 + (int)b), PL * 4u);
        dc_bulk_load(sbase + pl.off_par + b * PL * 4u, psrc(l), PL * 4u, bar_of(3 + (int)b));
      };
      auto chunk_load = [&](const uint8_t* src, int bytes) {
        if (round > 0) wait_bar(bar_of(16 + slot), (round - 1) & 1u);
        if (failed) return;
        ptx::mbar_expect_tx(bar_of(8 + slot), (uint32_t)bytes);
        dc_bulk_load(ring + (uint32_t)slot * DC_CHUNK, src, (uint32_t)bytes, bar_of(8 + slot));
        if (++slot == n_slots) { slot = 0; ++round; }
      };
      auto layer_load = [&](int l, int skip, int most) {      // chunks skip .. of layer l, at most `most` of them, in the order of use
        int at = 0;
#pragma unroll 1
        for (int i = 0; i < 6; ++i) {
          const int s = i < 2 ? i : (i < 4 ? i + 2 : i - 2);      // 0, 1, (4, 5,) 2, 3
          if (s >= n_slabs) continue;
          const uint8_t* src = wsrc(l) + dc_slab_off(d, DH, s, CS);
          const int bytes = dc_slab_bytes(d, DH, s, CS);
#pragma unroll 1
          for (int o = 0; o < bytes; o += DC_CHUNK, ++at)
            if (at >= skip && at < skip + most) chunk_load(src + o, min(DC_CHUNK, bytes - o));
        }
      };
      if (resident) {
        const uint32_t wb = (uint32_t)(P.fold ? dc_slab_off(d, DH, 4, CS) : dc_layer_bytes(d, DH, CS));
        ptx::mbar_expect_tx(bar_of(2), (uint32_t)L * (wb + PL * 4u));
        for (int l = 0; l < L; ++l) {
          dc_bulk_load(ring + (uint32_t)(l * dc_layer_bytes(d, DH, CS)), wsrc(l), wb, bar_of(2));
          dc_bulk_load(sbase + pl.off_par + (uint32_t)l * PL * 4u, psrc(l), PL * 4u, bar_of(2));
        }
      } else {      // the first layer's pieces are on their way before the predecessor has finished
        par_load(0);
        pre_chunks = min(n_slots, chunks_layer);
        layer_load(0, 0, pre_chunks);
      }
      pdl_wait();
      uint32_t n_tab = 0;
      bool first = true;
      for (int w = cid; w < P.B * C && !failed; w += ncl) {
        const int slot_w = w / C, cand = w - slot_w * C, ke = steps(slot_w, cand), env = item_of(P.item, slot_w);
        for (int k = 1; k <= ke && !failed; ++k) {
          const int tau = P.t[slot_w] - cand - k + 1;
          for (int l = 0; l < L && !failed; ++l) {      // everything one forward consumes
            if (!resident && !first) par_load(l);
            if (P.fold) {
              if (n_tab > 0) wait_bar(bar_of(24), (n_tab - 1) & 1u);
              if (failed) break;
              ++n_tab;
              const uint32_t tok = (uint32_t)(HEADS * d * 2);      // bytes of a memory token's kq rows, and of its u rows
              const size_t stride = (size_t)L * HEADS * d, lay = (size_t)l * HEADS * d;
              ptx::mbar_expect_tx(bar_of(7), 2u * (uint32_t)NK * tok);
#pragma unroll 1
              for (int j = 0; j < NK; ++j) {
                const size_t at = (j == 0 ? (size_t)tau : (size_t)env * P.To + (j - 1)) * stride + lay;
                dc_bulk_load(sbase + pl.off_kq + (uint32_t)j * tok, (j == 0 ? P.kq_time : P.kq_obs) + at, tok, bar_of(7));
                dc_bulk_load(sbase + pl.off_u + (uint32_t)j * tok, (j == 0 ? P.ut_time : P.ut_obs) + at, tok, bar_of(7));
              }
            }
            if (!resident) layer_load(l, first ? pre_chunks : 0, chunks_layer);
            first = false;
          }
        }
      }
      if (first && !resident) {                 // nothing to do: let the copies land
        wait_bar(bar_of(3), 0);
        for (int i = 0; i < pre_chunks; ++i) wait_bar(bar_of(8 + i), 0);
      }
      if (first && resident) wait_bar(bar_of(2), 0);
      if (failed) { const long long t0 = clock64(); while (clock64() - t0 < 400000ll) { } }
    }
    __syncwarp();
    cluster.sync();
    return;
  }

  // ================================================================== compute warps
  pdl_wait();      // t, the latents and the obs K/V come from earlier kernels
  const uint64_t seed = *P.seed;
  const int g = lane >> 2, tg = lane & 3;
  const int row = warp / WPR, grp = (warp % WPR) * VG, c0 = (grp * 32 + lane) * V2;      // owned row of this thread, its first group, its columns there
  constexpr int GC = 32 * V2;                                    // from a column to the same one of the warp's next group
  uint32_t stage_no = 0, stage_phase = 0;      // stages so far; bit b = parity this CTA waits for next on barrier b
  auto stage_begin = [&](uint32_t bytes) {     // thread 0 announces the bytes this CTA will receive in the stage that begins
    if (use_async && threadIdx.x == 0) ptx::mbar_expect_tx(bar_of((int)(stage_no & 1u)), bytes);
  };
  // 16 bytes to shared-memory offset `off` of the CTA whose shared memory starts at `r`
  auto send16 = [&](uint32_t r, uint32_t off, const uint4& v) {
    if (use_async) dc_st_async16(r + off, v, r + (uint32_t)pl.off_bar + 8u * (stage_no & 1u));
    else dc_st_cluster16(r + off, v);
  };
  // everything of the stage has arrived in this CTA (bounded wait)
  auto stage_end = [&]() {
    const uint32_t b = stage_no & 1u;
    if (!use_async) {
      asm volatile("fence.acq_rel.cluster;" ::: "memory");
      dc_sync();
      if (threadIdx.x < CS) ptx::mbar_arrive_cluster(dc_mapa(bar_of((int)b), threadIdx.x));
    }
    wait_bar(bar_of((int)b), (stage_phase >> b) & 1u);
    if (!use_async) asm volatile("fence.acq_rel.cluster;" ::: "memory");
    stage_phase ^= 1u << b;
    ++stage_no;
  };
  // ---- all-gather of the owned rows' values (as bf16) into everyone's xa: 8 columns of a row are 8 / V2 neighbouring lanes,
  // which share out the CTAs that get the 16 bytes
  constexpr int GL = 8 / V2, NS = CS / GL > 0 ? CS / GL : 1;
  const bool sends = (lane % GL) * NS < CS;
  uint32_t gdst[NS];
#pragma unroll
  for (int j = 0; j < NS; ++j) gdst[j] = dc_mapa(sbase, (uint32_t)min((lane % GL) * NS + j, CS - 1));
  auto gather_rows = [&](const float (&v)[VG][V2]) {
#pragma unroll
    for (int u = 0; u < VG; ++u) {
      const float up = V2 == 1 ? __shfl_down_sync(0xffffffffu, v[u][0], 1) : v[u][V2 - 1];
      const uint32_t w = pack_bf16x2(v[u][0], up);                       // V2 = 1: even lanes hold a pair
      uint4 o;
      uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
      for (int j = 0; j < 4; ++j) ow[j] = __shfl_sync(0xffffffffu, w, (lane & ~(GL - 1)) | (j * (GL / 4)));
      const uint32_t off = (uint32_t)pl.off_xa + (uint32_t)((OWN * rank + row) * PX + ((c0 + u * GC) & ~7)) * 2u;
#pragma unroll
      for (int j = 0; j < NS; ++j)
        if (sends) send16(gdst[j], off, o);
    }
  };
  // ---- partial sums of an output tile (8 columns, 16 rows) to the owners of the rows: lanes pair up, the even one sends four
  // columns of row g, the odd one of row g + 8
  const uint32_t pdst = dc_mapa(sbase, (uint32_t)(((tg & 1) * 8 + g) / OWN));
  const uint32_t poff = (uint32_t)pl.off_recv + (uint32_t)((rank * OWN + g % OWN) * d + 4 * (tg >> 1)) * 4u;
  auto send_partial = [&](int tile, const float (&c)[4]) {
    const bool odd = tg & 1;
    const float r0 = __shfl_xor_sync(0xffffffffu, odd ? c[0] : c[2], 1), r1 = __shfl_xor_sync(0xffffffffu, odd ? c[1] : c[3], 1);
    const uint4 o = odd ? make_uint4(__float_as_uint(r0), __float_as_uint(r1), __float_as_uint(c[2]), __float_as_uint(c[3]))
                        : make_uint4(__float_as_uint(c[0]), __float_as_uint(c[1]), __float_as_uint(r0), __float_as_uint(r1));
    send16(pdst, poff + (uint32_t)tile * 32u, o);
  };
  float hv[VG][V2];      // the stream: this thread's columns of its row
  auto add_partials = [&](const float* bias) {      // stream += sum of the CTAs' parts (in pairs, pairs of pairs, ..) + bias
#pragma unroll
    for (int u = 0; u < VG; ++u)
#pragma unroll
      for (int j = 0; j < V2; ++j) {
        const int c = c0 + u * GC + j;
        float p[CS];
#pragma unroll
        for (int r = 0; r < CS; ++r) p[r] = recv[(r * OWN + row) * d + c];
#pragma unroll
        for (int n = CS; n > 1; n >>= 1)
#pragma unroll
          for (int r = 0; r < n / 2; ++r) p[r] = p[2 * r] + p[2 * r + 1];
        hv[u][j] += p[0] + bias[c];
      }
  };
  // LayerNorm of the owned rows without the affine part: mean and squared deviations per group, then combined over the row's four
  uint32_t n_stat = 0;
  auto normalise = [&](float (&x)[VG][V2]) {
    float2* st = sstat + ((n_stat & 1u) * OWN + row) * 4;
    float s[VG], q[VG];
#pragma unroll
    for (int u = 0; u < VG; ++u) {
      s[u] = 0.f; q[u] = 0.f;
#pragma unroll
      for (int j = 0; j < V2; ++j) s[u] += hv[u][j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < VG; ++u) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
#pragma unroll
    for (int u = 0; u < VG; ++u) {
      s[u] *= 1.0f / (32 * V2);
#pragma unroll
      for (int j = 0; j < V2; ++j) { const float e = hv[u][j] - s[u]; q[u] += e * e; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < VG; ++u) q[u] += __shfl_xor_sync(0xffffffffu, q[u], o);
    if (lane == 0) {
#pragma unroll
      for (int u = 0; u < VG; ++u) st[grp + u] = make_float2(s[u], q[u]);
    }
    ++n_stat;
    dc_row_sync<CS>(row);
    const float2 a0 = st[0], a1 = st[1], a2 = st[2], a3 = st[3];
    const float mean = 0.25f * ((a0.x + a1.x) + (a2.x + a3.x));
    const float e0 = a0.x - mean, e1 = a1.x - mean, e2 = a2.x - mean, e3 = a3.x - mean;
    const float m2 = ((a0.y + a1.y) + (a2.y + a3.y)) + (32 * V2) * ((e0 * e0 + e1 * e1) + (e2 * e2 + e3 * e3));
    const float rstd = rsqrtf(m2 / d + 1e-5f);
#pragma unroll
    for (int u = 0; u < VG; ++u)
#pragma unroll
      for (int j = 0; j < V2; ++j) x[u][j] = (hv[u][j] - mean) * rstd;
  };
  auto affine = [&](float (&x)[VG][V2], const float* gam, const float* bet) {
#pragma unroll
    for (int u = 0; u < VG; ++u)
#pragma unroll
      for (int j = 0; j < V2; ++j) x[u][j] = x[u][j] * gam[c0 + u * GC + j] + bet[c0 + u * GC + j];
  };
  // ---- ring, consumer side: chunk i of the pass that begins sits in slot (cslot + i) % n_slots
  const uint32_t ring_end = resident ? 0xffffffffu : ring + (uint32_t)n_slots * DC_CHUNK;
  int cslot = 0;
  uint32_t cround = 0;
  auto slot_of = [&](int i) { const int s = cslot + i; return s >= n_slots ? s - n_slots : s; };
  auto chunks_wait = [&](int n) {              // the pass's n chunks are there (one lane each)
    if (lane < n) wait_bar(bar_of(8 + slot_of(lane)), (cround + (cslot + lane >= n_slots ? 1u : 0u)) & 1u);
    __syncwarp();
  };
  auto chunks_release = [&](int n) {           // this warp is done with them
    __syncwarp();
    if (lane < n) ptx::mbar_arrive(bar_of(16 + slot_of(lane)));
    cslot += n;
    if (cslot >= n_slots) { cslot -= n_slots; ++cround; }
  };
  // Y = X W^T for slab S of layer l, tile warp + 8 t of a pass; X may be read after `ready()`, which every warp runs once; `done(tile, accumulators)`
  // per finished tile
  auto linear = [&](auto slab_c, int l, const __nv_bfloat16* X, int px, auto ready, auto done) {
    constexpr int S = decltype(slab_c)::value;
    constexpr int K = dc_slab_k(d, S, CS), NT = dc_slab_rows(d, DH, S, CS) / 8, NKB = K / 32, TB = K * 16;      // TB: bytes of a tile
    constexpr int HALVES = CS < 8 && (S & 1) && NKB > 1 ? 2 : 1;      // partial sums over the CTAs' columns
    constexpr int TPW = dc_tiles_per_warp(d, DH, S, CS), PT = TPW * DC_WARPS;                               // tiles of a pass
    dc_passes<0, (NT + PT - 1) / PT>([&](auto pass_c) {
      constexpr int t0 = decltype(pass_c)::value * PT, N = NT - t0 < PT ? NT - t0 : PT, NCH = (N * TB + DC_CHUNK - 1) / DC_CHUNK;
      constexpr int T1 = (N + DC_WARPS - 1) / DC_WARPS;      // tiles of the busiest warps; the others have one less
      if (!resident) chunks_wait(NCH);
      auto run = [&](auto tiles_c) {
        constexpr int T = decltype(tiles_c)::value;
        if constexpr (T > 0) {
          // a resident slab lies in one piece; a pass in the ring may wrap
          const uint32_t first = ring + (uint32_t)(warp * TB + lane * 16) +
                                 (resident ? (uint32_t)(l * dc_layer_bytes(d, DH, CS) + dc_slab_off(d, DH, S, CS) + t0 * TB) : (uint32_t)cslot * DC_CHUNK);
          uint32_t base[T];
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const uint32_t at = first + t * DC_WARPS * TB;
            base[t] = at >= ring_end ? at - (uint32_t)n_slots * DC_CHUNK : at;
          }
          float c[T][4];
          dc_kloop<T, NKB, HALVES>(X, px, c, base, [&] { if constexpr (t0 == 0) ready(); });
          if (!resident) chunks_release(NCH);
#pragma unroll
          for (int t = 0; t < T; ++t) done(t0 + warp + t * DC_WARPS, c[t]);
        } else {
          if constexpr (t0 == 0) ready();
          if (!resident) chunks_release(NCH);
        }
      };
      if constexpr (N % DC_WARPS == 0) run(std::integral_constant<int, T1>{});
      else if (warp < N - (T1 - 1) * DC_WARPS) run(std::integral_constant<int, T1>{});
      else run(std::integral_constant<int, T1 - 1>{});
    });
  };
  // a finished tile with bias (and GELU) as bf16 into a local buffer
  auto keep = [&](__nv_bfloat16* dst, int pitch, int tile, const float (&c)[4], const float* bias, bool gelu) {
    const float2 bb = *reinterpret_cast<const float2*>(bias + tile * 8 + 2 * tg);
    float v0 = c[0] + bb.x, v1 = c[1] + bb.y, v2 = c[2] + bb.x, v3 = c[3] + bb.y;
    if (gelu) { v0 = ptx::gelu_fast(v0); v1 = ptx::gelu_fast(v1); v2 = ptx::gelu_fast(v2); v3 = ptx::gelu_fast(v3); }
    *reinterpret_cast<uint32_t*>(dst + g * pitch + tile * 8 + 2 * tg) = pack_bf16x2(v0, v1);
    *reinterpret_cast<uint32_t*>(dst + (g + 8) * pitch + tile * 8 + 2 * tg) = pack_bf16x2(v2, v3);
  };
  // dot products of the owned rows' fp32 values (sxr) with `n` vectors per row, one per warp and turn: out(row, i, value) in the lane of the pair's turn
  auto row_dots = [&](int n, auto load4, auto out) {
    for (int p0 = warp; p0 < OWN * n; p0 += 4 * DC_WARPS) {
      float acc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = min(p0 + u * DC_WARPS, OWN * n - 1), r = p % OWN, i = p / OWN;
        acc[u] = 0.f;
#pragma unroll
        for (int j = 0; j < d / 128; ++j) {
          const int c = j * 128 + lane * 4;
          const float4 x = *reinterpret_cast<const float4*>(sxr + r * d + c), w = load4(i, c);
          acc[u] += (x.x * w.x + x.y * w.y) + (x.z * w.z + x.w * w.w);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = p0 + u * DC_WARPS;
        if (lane == p / DC_WARPS && p < OWN * n) out(p % OWN, p / OWN, acc[u]);
      }
    }
  };
  auto put_rows = [&](const float (&x)[VG][V2]) {
#pragma unroll
    for (int u = 0; u < VG; ++u)
#pragma unroll
      for (int j = 0; j < V2; ++j) sxr[row * d + c0 + u * GC + j] = x[u][j];
  };

  uint32_t n_layer = 0, n_tab = 0;      // layers so far (parameter buffers), tables so far
  if (resident) wait_bar(bar_of(2), 0);
  // One forward of the network on the owned rows' latent in sx at timestep tau for request env; leaves their eps in seps.  `rest`
  // is run once, by the upper four warps, which have nothing to do during the first layer's attention.
  auto forward = [&](int tau, int env, auto rest) {
    {   // token embedding into the residual stream
      const int tok = OWN * rank + row;
      const bool live = tok < H;
#pragma unroll
      for (int u = 0; u < VG; ++u) {
        const int c = c0 + u * GC;
#pragma unroll
        for (int j = 0; j < V2; ++j) hv[u][j] = live ? __ldg(P.b_in + c + j) + __ldg(P.pos + tok * d + c + j) : 0.f;
        if (live)
#pragma unroll 4
          for (int i = 0; i < A; ++i) {
            const float xv = sx[row * AP + i];
#pragma unroll
            for (int j = 0; j < V2; ++j) hv[u][j] = __fmaf_rn(xv, __ldg(P.W_in + i * d + c + j), hv[u][j]);
          }
      }
    }
    for (int l = 0; l < L; ++l) {
      if (!resident) wait_bar(bar_of(3 + (int)(n_layer & 1u)), (n_layer >> 1) & 1u);
      const float* pb = spar + (size_t)(resident ? l : (int)(n_layer & 1u)) * PL;
      const float *ln1 = pb, *ln2 = pb + 2 * d, *ln3 = pb + 4 * d, *bo = pb + 6 * d, *bo2 = pb + 7 * d, *b2 = pb + 8 * d,
                  *bqkv = pb + 9 * d, *b1 = bqkv + NQ, *bq2 = b1 + MW;
      float x[VG][V2];
      // ---- causal self-attention of this CTA's head
      normalise(x);
      affine(x, ln1, ln1 + d);
      stage_begin(DC_ROWS * d * 2);
      gather_rows(x);
      linear(std::integral_constant<int, 0>{}, l, xa, PX, stage_end, [&](int tile, const float (&c)[4]) { keep(qs, PQ, tile, c, bqkv, false); });
      dc_sync();
      if (warp < VW / 16) {
        // scores of all 16 rows by each of these warps, then 16 of the CTA's value columns
        const float scale = rsqrtf((float)DH);
        float s[2][4];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
          uint32_t a4[4], b4[4];
          ldmatrix_x4(a4, qs + (lane & 15) * PQ + ks * 16 + 8 * (lane >> 4));
          ldmatrix_x4(b4, qs + ((lane & 7) + 8 * (lane >> 4)) * PQ + DH + ks * 16 + 8 * ((lane >> 3) & 1));
          mma_bf16_16816(s[0], a4, b4[0], b4[1]);
          mma_bf16_16816(s[1], a4, b4[2], b4[3]);
        }
        const int r0 = g, r1 = g + 8;
        float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const int col = nt * 8 + 2 * tg;
          s[nt][0] = (col <= r0 && col < H) ? s[nt][0] * scale : -INFINITY;
          s[nt][1] = (col + 1 <= r0 && col + 1 < H) ? s[nt][1] * scale : -INFINITY;
          s[nt][2] = (col <= r1 && col < H) ? s[nt][2] * scale : -INFINITY;
          s[nt][3] = (col + 1 <= r1 && col + 1 < H) ? s[nt][3] * scale : -INFINITY;
          m0 = fmaxf(m0, fmaxf(s[nt][0], s[nt][1]));
          m1 = fmaxf(m1, fmaxf(s[nt][2], s[nt][3]));
        }
        m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 1)); m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 1));
        m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 2)); m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 2));
        float l0 = 0.f, l1 = 0.f;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          s[nt][0] = __expf(s[nt][0] - m0); s[nt][1] = __expf(s[nt][1] - m0);
          s[nt][2] = __expf(s[nt][2] - m1); s[nt][3] = __expf(s[nt][3] - m1);
          l0 += s[nt][0] + s[nt][1]; l1 += s[nt][2] + s[nt][3];
        }
        l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
        l0 += __shfl_xor_sync(0xffffffffu, l0, 2); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
        const float inv0 = 1.0f / l0, inv1 = 1.0f / l1;      // every row sees at least key 0 (H >= 1)
        uint32_t pa[4];
        pa[0] = pack_bf16x2(s[0][0], s[0][1]); pa[1] = pack_bf16x2(s[0][2], s[0][3]);
        pa[2] = pack_bf16x2(s[1][0], s[1][1]); pa[3] = pack_bf16x2(s[1][2], s[1][3]);
        float o0[4] = {0.f, 0.f, 0.f, 0.f}, o1[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t b4[4];
        ldmatrix_x4_trans(b4, qs + ((lane & 7) + 8 * ((lane >> 3) & 1)) * PQ + 2 * DH + warp * 16 + 8 * (lane >> 4));
        mma_bf16_16816(o0, pa, b4[0], b4[1]);
        mma_bf16_16816(o1, pa, b4[2], b4[3]);
        __nv_bfloat16* o = os + warp * 16 + 2 * tg;
        *reinterpret_cast<uint32_t*>(o + r0 * PO) = pack_bf16x2(o0[0] * inv0, o0[1] * inv0);
        *reinterpret_cast<uint32_t*>(o + r1 * PO) = pack_bf16x2(o0[2] * inv1, o0[3] * inv1);
        *reinterpret_cast<uint32_t*>(o + r0 * PO + 8) = pack_bf16x2(o1[0] * inv0, o1[1] * inv0);
        *reinterpret_cast<uint32_t*>(o + r1 * PO + 8) = pack_bf16x2(o1[2] * inv1, o1[3] * inv1);
      } else if (l == 0 && warp >= 4) rest();
      dc_sync();
      stage_begin(DC_ROWS * d * 4);
      linear(std::integral_constant<int, 1>{}, l, os, PO, [] {}, [&](int tile, const float (&c)[4]) { send_partial(tile, c); });
      float cst = 0.f;      // constant of the score that this lane will finish (16 OWN scores at most, 2 OWN per warp)
      if (P.fold) {
        const int p = warp + lane * DC_WARPS, n = p / OWN, j = n / HEADS;
        if (p < OWN * NKH)
          cst = (j == 0 ? P.c_time + (size_t)tau * L * HEADS : P.c_obs + ((size_t)env * P.To + (j - 1)) * L * HEADS)[(size_t)l * HEADS + n % HEADS];
      } else {      // keys and value columns of the memory tokens for this CTA's head
        float* skv = reinterpret_cast<float*>(dc_smem + pl.off_kq);      // [NK][DH + VW]
        const size_t ldkv = (size_t)L * 2 * d;
        for (int i = threadIdx.x; i < NK * (DH + VW); i += DC_COMPUTE) {
          const int kx = i / (DH + VW), c = i % (DH + VW);
          const float* src = (kx == 0 ? P.kv_time + (size_t)tau * ldkv : P.kv_obs + ((size_t)env * P.To + (kx - 1)) * ldkv) + (size_t)l * 2 * d;
          skv[i] = src[c < DH ? rank * HEADS / CS * DH + c : d + rank * VW + (c - DH)];
        }
      }
      stage_end();
      add_partials(bo);
      // ---- cross-attention to [time token | obs tokens]
      normalise(x);
      if (P.fold) {
        // Folded form, on the owned rows alone: scores = xhat . kq + c, out = P . u + bo2 (fp32)
        put_rows(x);
        wait_bar(bar_of(7), n_tab & 1u);
        ++n_tab;
        dc_sync();
        row_dots(NKH, [&](int n, int c) {
          const uint2 w = *reinterpret_cast<const uint2*>(skq + n * d + c);
          const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x)), hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
          return make_float4(lo.x, lo.y, hi.x, hi.y);
        }, [&](int r, int n, float v) { sscore[r * DC_MAX_NKH + n] = v + cst; });
        dc_sync();
        // softmax over the memory tokens of each head, lane n (and n + 16) for (token, head) pair n of the warp's row
        float p = (lane & 15) < NKH ? sscore[row * DC_MAX_NKH + (lane & 15)] : -INFINITY, m = p;
#pragma unroll
        for (int o = HEADS; o < DC_MAX_NKH; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        p = __expf(p - m);
        float sum = p;
#pragma unroll
        for (int o = HEADS; o < DC_MAX_NKH; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        p /= sum;
        float o[VG][V2];
#pragma unroll
        for (int u = 0; u < VG; ++u)
#pragma unroll
          for (int j = 0; j < V2; ++j) o[u][j] = 0.f;
#pragma unroll
        for (int q = 0; q < DC_MAX_NKH / 2; ++q)
          if (2 * q < NKH) {
            const float p0 = __shfl_sync(0xffffffffu, p, 2 * q), p1 = __shfl_sync(0xffffffffu, p, 2 * q + 1);
#pragma unroll
            for (int u = 0; u < VG; ++u)
#pragma unroll
              for (int j = 0; j < V2; ++j) {
                const float2 u2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(su + q * d + c0 + u * GC + j));
                o[u][j] = __fmaf_rn(p0, u2.x, __fmaf_rn(p1, u2.y, o[u][j]));
              }
          }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar_of(24));      // this warp is done with the tables
#pragma unroll
        for (int u = 0; u < VG; ++u)
#pragma unroll
          for (int j = 0; j < V2; ++j) hv[u][j] += o[u][j] + bo2[c0 + u * GC + j];
      } else {
        affine(x, ln2, ln2 + d);
        stage_begin(DC_ROWS * d * 2);
        gather_rows(x);
        linear(std::integral_constant<int, 4>{}, l, xa, PX, stage_end, [&](int tile, const float (&c)[4]) { keep(qs, PQ, tile, c, bq2, false); });
        dc_sync();
        if (threadIdx.x < 4 * DC_ROWS) {                   // four lanes per query row, each a quarter of the head and of the value columns
          const float* skv = reinterpret_cast<const float*>(dc_smem + pl.off_kq);
          const int r = threadIdx.x >> 2, sub = threadIdx.x & 3;
          const float scale = rsqrtf((float)DH);
          float sc[DC_MAX_NK], m = -INFINITY, s = 0.f;
#pragma unroll
          for (int j = 0; j < DC_MAX_NK; ++j) {
            float v = 0.f;
            if (j < NK)
              for (int i = sub * (DH / 4); i < (sub + 1) * (DH / 4); ++i) v += __bfloat162float(qs[r * PQ + i]) * skv[j * (DH + VW) + i];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            sc[j] = j < NK ? v * scale : -INFINITY;
            m = fmaxf(m, sc[j]);
          }
#pragma unroll
          for (int j = 0; j < DC_MAX_NK; ++j) { sc[j] = __expf(sc[j] - m); s += sc[j]; }
          const float inv = 1.0f / s;
          for (int i = sub * (VW / 4); i < (sub + 1) * (VW / 4); ++i) {
            float v = 0.f;
#pragma unroll
            for (int j = 0; j < DC_MAX_NK; ++j)
              if (j < NK) v += sc[j] * skv[j * (DH + VW) + DH + i];
            os[r * PO + i] = __float2bfloat16_rn(v * inv);
          }
        }
        dc_sync();
        stage_begin(DC_ROWS * d * 4);
        linear(std::integral_constant<int, 5>{}, l, os, PO, [] {}, [&](int tile, const float (&c)[4]) { send_partial(tile, c); });
        stage_end();
        add_partials(bo2);
      }
      // ---- MLP
      normalise(x);
      affine(x, ln3, ln3 + d);
      stage_begin(DC_ROWS * d * 2);
      gather_rows(x);
      linear(std::integral_constant<int, 2>{}, l, xa, PX, stage_end, [&](int tile, const float (&c)[4]) { keep(fs, PF, tile, c, b1, true); });
      stage_begin(DC_ROWS * d * 4);
      linear(std::integral_constant<int, 3>{}, l, fs, PF, dc_sync, [&](int tile, const float (&c)[4]) { send_partial(tile, c); });
      stage_end();
      add_partials(b2);
      if (!resident) { __syncwarp(); if (lane == 0) ptx::mbar_arrive(bar_of(5 + (int)(n_layer & 1u))); }
      ++n_layer;
    }
    // ---- head: eps = LN_f(h) W_out + b_out of the owned rows
    float x[VG][V2];
    normalise(x);
    affine(x, lnf_g, lnf_b);
    put_rows(x);
    dc_sync();
    row_dots(A, [&](int i, int c) { return *reinterpret_cast<const float4*>(woutT + (size_t)i * d + c); },
             [&](int r, int i, float v) { seps[r * AP + i] = v + bout[i]; });
    dc_sync();
  };
  // one element of the owned rows per thread of the upper four warps (OWN A <= 128): its index in the latent, -1 if there is none
  const int e_own = (int)threadIdx.x - 128, e_row = e_own >= 0 ? e_own / A : 0;
  const int e_idx = e_own >= 0 && e_row < OWN && OWN * rank + e_row < H ? (OWN * rank + e_row) * A + e_own % A : -1;
  float* e_x = sx + e_row * AP + (e_own >= 0 ? e_own % A : 0);
  const int e_eps = OWN * AP, e_z = 2 * e_eps, e_sig = 3 * e_eps;      // from there to its eps, noise, sigma

  // drafting: one slot after the other, K steps each; verification: one forward per (slot, candidate)
  const bool verify = P.mode == 1;
  for (int w = cid; w < P.B * C; w += ncl) {
    const int slot = w / C, cand = w - slot * C, ke = steps(slot, cand), tb = P.t[slot] - cand;
    const int env = item_of(P.item, slot);       // request served by this slot: its noise streams, obs K/V, parameters
    float* xt_b = P.xt + slot * P.xs_b + (long long)cand * D;
    float* mh_b = P.muhat + slot * P.ms_b;
    float xv = 0.f;
    if (e_idx >= 0) { xv = xt_b[e_idx]; *e_x = xv; }
    dc_sync();
    for (int k = 1; k <= ke; ++k) {
      const int tau = tb - k + 1;
      forward(tau, env, [&] {
        if (e_idx >= 0 && !verify) {
          float z4[4];
          normal4(seed, (uint32_t)env, STREAM_XI, (uint32_t)tau, (uint32_t)(e_idx >> 2), z4);
          const int j = e_idx & 3;
          e_x[e_z] = j == 0 ? z4[0] : (j == 1 ? z4[1] : (j == 2 ? z4[2] : z4[3]));
          e_x[e_sig] = P.S.sigma[tau];
        }
      });
      if (e_idx >= 0) {
        if (verify) P.eps[slot * P.es_b + (long long)cand * D + e_idx] = e_x[e_eps];
        else {                                   // scheduler step: mu^_k, x~_k = mu^_k + sigma_tau xi_tau
          const float m = posterior_mean(P.S, xv, e_x[e_eps], tau);
          xv = ddpm_sample(m, e_x[e_sig], e_x[e_z]);
          *e_x = xv;
          mh_b[(size_t)(k - 1) * D + e_idx] = m;
          xt_b[(size_t)k * D + e_idx] = xv;
        }
      }
      dc_sync();
    }
    if (!verify && e_idx >= 0)                   // beyond K_eff: carry the latent along
      for (int k = ke + 1; k <= P.K; ++k) { mh_b[(size_t)(k - 1) * D + e_idx] = xv; xt_b[(size_t)k * D + e_idx] = xv; }
  }
  if (failed) { const long long t0 = clock64(); while (clock64() - t0 < 400000ll) { } }      // copies in flight land first
  cluster.sync();      // no CTA leaves while another may still write into its shared memory
}
}  // namespace tsdp
