// Network kernels other than the tensor-core GEMM: the fp32 check-mode GEMM, token embedding,
// LayerNorm, the two small attentions, the output head and the closed-form Gaussian denoiser.  T is the activation type: float in the fp32 check mode, bf16 in the production mode.
#pragma once
#include "common.cuh"
#include "gemm_tcgen05.cuh"

namespace tsdp {

// ------------------------------------------------------------------------------------------------
// fp32 check-mode GEMM (CUDA cores): C[M,N] = A[M,K] W[N,K]^T, same epilogues as the tensor-core one.
// ------------------------------------------------------------------------------------------------
template <int EPI>
__global__ void __launch_bounds__(256)
gemm_simt_kernel(const float* A, const float* __restrict__ W, GemmArgs g) {
  pdl_trigger();
  pdl_wait();
  __shared__ float As[16][65], Ws[16][65];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  g.M = live_rows(g.live, g.M);
  if (m0 >= g.M) return;
  float acc[4][4] = {};
  const int lr = threadIdx.x >> 4, lk = threadIdx.x & 15;      // this thread loads rows lr, lr + 16, .. at k = lk
  size_t arow[4];                                              // where they start (kept out of the k loop: a convolution's take a division)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int row = m0 + lr + 16 * j;
    arow[j] = (g.conv_c ? (size_t)(row / g.conv_l) * (g.conv_l + 4) + row % g.conv_l + g.conv_off : (size_t)row) * g.lda;
  }
  for (int k0 = 0; k0 < g.K; k0 += 16) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = lr + 16 * j;
      As[lk][r] = (m0 + r < g.M && k0 + lk < g.K) ? A[arow[j] + k0 + lk] : 0.f;
      Ws[lk][r] = (n0 + r < g.N && k0 + lk < g.K) ? W[(size_t)(n0 + r) * g.K + k0 + lk] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      float a[4], w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = As[k][ty * 4 + i]; w[i] = Ws[k][tx * 4 + i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * w[j];
    }
    __syncthreads();
  }
  for (int i = 0; i < 4; ++i) {
    const int row = m0 + ty * 4 + i;
    if (row >= g.M) continue;
    for (int j = 0; j < 4; ++j) {
      const int col = n0 + tx * 4 + j;
      if (col >= g.N) continue;
      float v = acc[i][j] + (g.bias ? g.bias[col] : 0.f);
      if (EPI == EPI_GELU) v = gelu_tanh(v);
      if (EPI == EPI_SILU) v = v / (1.0f + expf(-v));
      if (EPI == EPI_MISH) v = v * tanhf(v > 20.f ? v : log1pf(expf(v)));
      if (EPI == EPI_GATE) v *= gate_row(g, row)[col];
      float* o = reinterpret_cast<float*>(g.out) + (size_t)row * g.ldo + col;
      if (EPI == EPI_RESID || EPI == EPI_GATE) v += *o;
      *o = v;
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Token embedding: h[n*H + i, :] = x[n, i, :] W_in + b_in + pos[i, :]      (fp32 residual stream)
// ------------------------------------------------------------------------------------------------
__global__ void embed_kernel(CandMap cm, const float* __restrict__ W_in, const float* __restrict__ b_in,
                             const float* __restrict__ pos, float* __restrict__ h, int H, int A, int d) {
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x;
  const int n = row / H, i = row % H;
  if (n >= cand_count(cm, gridDim.x / H)) return;
  int b, c;
  cand_decode(cm, n, b, c);
  const float* x = cm.xin + b * cm.x_stride_b + (long long)c * H * A + (long long)i * A;
  for (int col = threadIdx.x; col < d; col += blockDim.x) {
    float v = b_in[col] + pos[i * d + col];
    for (int a = 0; a < A; ++a) v += x[a] * W_in[a * d + col];
    h[(size_t)row * d + col] = v;
  }
}

// 16 bytes from global to shared memory, past the L1.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Time tokens, at load time: out[r, :] = in[r, :] + cpos[0] (in = the sinusoidal table).
template <typename T>
__global__ void timetok_kernel(const float* __restrict__ in, const float* __restrict__ cpos, T* __restrict__ out, int d) {
  const size_t r = blockIdx.x;
  for (int col = threadIdx.x; col < d; col += blockDim.x) out[r * d + col] = from_f<T>(in[r * d + col] + cpos[col]);
}

// Memory tokens of the observations, once per chunk: out[r, :] = in[r, :] W[Din, d] + bias + cpos[cpos_off + r % cpos_mod], fp32 as
// the observations are.  A product on the CUDA cores: a block owns TM x 64 outputs and walks k in steps of 32, the next step's operands
// on their way in registers while the current one is multiplied from shared memory (packed fp32).  16-row tiles where 64-row
// ones would leave most SMs idle; every output sums over k in order either way.  The kernel before it gave a row to each
// block, with one load in flight per multiply; before and after: 16384 x 1024 x 1024 4950 -> 1071 us, 768 x 1024 x 1024 685 -> 85,
// 2 x 256 x 512 93 -> 20.
constexpr int MT_BK = 32, MT_N = 64, MT_THREADS = 256;
template <typename T, int TM>
__global__ void __launch_bounds__(MT_THREADS)
memtok_kernel(const float* in, int rows, int Din, const float* __restrict__ W, const float* __restrict__ bias,
              const float* __restrict__ cpos, int cpos_mod, int cpos_off, T* __restrict__ out, int d) {
  constexpr int RT = TM / 16, NA = TM * MT_BK / MT_THREADS, NB = MT_BK * MT_N / MT_THREADS, PA = TM + 4;      // rows a thread, loads a step
  __shared__ __align__(16) float As[MT_BK * PA];
  __shared__ __align__(16) float Bs[MT_BK * MT_N];
  pdl_trigger();
  pdl_wait();
  const int nt = d / MT_N, r0 = (int)(blockIdx.x / nt) * TM, c0 = (int)(blockIdx.x % nt) * MT_N;      // (a long queue has more row tiles than grid.y may)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tid & 15, ty = tid >> 4;
  float ra[NA], rb[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      const int r = r0 + warp + 8 * j, k = k0 + lane;
      ra[j] = r < rows && k < Din ? in[(size_t)r * Din + k] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int k = k0 + (tid >> 6) + 4 * j;
      rb[j] = k < Din ? __ldg(W + (size_t)k * d + c0 + (tid & 63)) : 0.f;
    }
  };
  float2 acc[RT][2];
#pragma unroll
  for (int i = 0; i < RT; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
  fetch(0);
  for (int k0 = 0; k0 < Din; k0 += MT_BK) {
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NA; ++j) As[lane * PA + warp + 8 * j] = ra[j];
#pragma unroll
    for (int j = 0; j < NB; ++j) Bs[((tid >> 6) + 4 * j) * MT_N + (tid & 63)] = rb[j];
    __syncthreads();
    if (k0 + MT_BK < Din) fetch(k0 + MT_BK);
#pragma unroll 8
    for (int k = 0; k < MT_BK; ++k) {
      const float4 b = *reinterpret_cast<const float4*>(Bs + k * MT_N + 4 * tx);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const float a = As[k * PA + ty * RT + i];
        acc[i][0] = __ffma2_rn(make_float2(a, a), make_float2(b.x, b.y), acc[i][0]);
        acc[i][1] = __ffma2_rn(make_float2(a, a), make_float2(b.z, b.w), acc[i][1]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int r = r0 + ty * RT + i, c = c0 + 4 * tx;
    if (r < rows) {
      const float* cp = cpos + (size_t)(cpos_off + r % cpos_mod) * d + c;
      const float v[4] = {acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y};
#pragma unroll
      for (int j = 0; j < 4; ++j) out[(size_t)r * d + c + j] = from_f<T>(v[j] + (cp[j] + bias[c + j]));
    }
  }
}

// ------------------------------------------------------------------------------------------------
// LayerNorm over d (multiple of 128), one warp per row, fp32 in, T out.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void store4(float* o, float a, float b, float c, float e) {
  *reinterpret_cast<float4*>(o) = make_float4(a, b, c, e);
}
__device__ __forceinline__ void store4(__nv_bfloat16* o, float a, float b, float c, float e) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, e);
  uint2 p;
  p.x = *reinterpret_cast<uint32_t*>(&lo); p.y = *reinterpret_cast<uint32_t*>(&hi);
  *reinterpret_cast<uint2*>(o) = p;
}

template <typename T, int VEC>
__global__ void ln_kernel(const float* h, const float* __restrict__ gam, const float* __restrict__ bet,
                          T* __restrict__ out, int M, LiveRows lv) {
  pdl_trigger(std::is_same<T, __nv_bfloat16>::value);
  pdl_wait();
  constexpr int d = VEC * 128;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= live_rows(lv, M)) return;
  float4 v[VEC];
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    v[j] = reinterpret_cast<const float4*>(h + (size_t)row * d)[j * 32 + lane];
    s += v[j].x + v[j].y + v[j].z + v[j].w;
  }
  const float mean = warp_sum(s) / d;
  float q = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    v[j].x -= mean; v[j].y -= mean; v[j].z -= mean; v[j].w -= mean;
    q += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
  }
  const float rstd = rsqrtf(warp_sum(q) / d + 1e-5f);
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    const int c = (j * 32 + lane) * 4;
    const float4 gg = reinterpret_cast<const float4*>(gam)[j * 32 + lane];
    const float4 bb = reinterpret_cast<const float4*>(bet)[j * 32 + lane];
    store4(out + (size_t)row * d + c, v[j].x * rstd * gg.x + bb.x, v[j].y * rstd * gg.y + bb.y,
           v[j].z * rstd * gg.z + bb.z, v[j].w * rstd * gg.w + bb.w);
  }
}

// Token embedding and the first block's LayerNorm of one token row by one warp:
//   h_row[:] = x[0..A) W_in + b_in + pos_row[:]   (fp32 residual stream),   out_row[:] = LN(h_row[:])
// x_of(a) returns the a-th input value (the same in every lane).
template <typename T, int VEC, typename XF>
__device__ __forceinline__ void embed_ln_row(XF x_of, int A, const float* __restrict__ W_in, const float* __restrict__ b_in,
                                             const float* __restrict__ pos_row, float* __restrict__ h_row,
                                             const float* __restrict__ gam, const float* __restrict__ bet, T* __restrict__ out_row,
                                             int lane) {
  constexpr int d = VEC * 128;
  float4 v[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    const float4 bi = reinterpret_cast<const float4*>(b_in)[j * 32 + lane];
    const float4 po = reinterpret_cast<const float4*>(pos_row)[j * 32 + lane];
    v[j] = make_float4(bi.x + po.x, bi.y + po.y, bi.z + po.z, bi.w + po.w);
  }
  for (int a = 0; a < A; ++a) {
    const float xa = x_of(a);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const float4 w = reinterpret_cast<const float4*>(W_in + (size_t)a * d)[j * 32 + lane];
      v[j].x = __fmaf_rn(xa, w.x, v[j].x); v[j].y = __fmaf_rn(xa, w.y, v[j].y);
      v[j].z = __fmaf_rn(xa, w.z, v[j].z); v[j].w = __fmaf_rn(xa, w.w, v[j].w);
    }
  }
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    reinterpret_cast<float4*>(h_row)[j * 32 + lane] = v[j];
    s += v[j].x + v[j].y + v[j].z + v[j].w;
  }
  const float mean = warp_sum(s) / d;
  float q = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    v[j].x -= mean; v[j].y -= mean; v[j].z -= mean; v[j].w -= mean;
    q += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
  }
  const float rstd = rsqrtf(warp_sum(q) / d + 1e-5f);
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    const int col = (j * 32 + lane) * 4;
    const float4 gg = reinterpret_cast<const float4*>(gam)[j * 32 + lane];
    const float4 bb = reinterpret_cast<const float4*>(bet)[j * 32 + lane];
    store4(out_row + col, v[j].x * rstd * gg.x + bb.x, v[j].y * rstd * gg.y + bb.y,
           v[j].z * rstd * gg.z + bb.z, v[j].w * rstd * gg.w + bb.w);
  }
}

template <typename T, int VEC>
__global__ void embed_ln_kernel(CandMap cm, const float* __restrict__ W_in, const float* __restrict__ b_in,
                                const float* __restrict__ pos, float* __restrict__ h, const float* __restrict__ gam,
                                const float* __restrict__ bet, T* __restrict__ out, int M, int H, int A) {
  pdl_trigger(std::is_same<T, __nv_bfloat16>::value);
  pdl_wait();
  constexpr int d = VEC * 128;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const int n = row / H, i = row % H;
  if (n >= cand_count(cm, M / H)) return;
  int b, c;
  cand_decode(cm, n, b, c);
  const float* x = cm.xin + b * cm.x_stride_b + (long long)c * H * A + (long long)i * A;
  embed_ln_row<T, VEC>([&](int a) { return x[a]; }, A, W_in, b_in, pos + (size_t)i * d, h + (size_t)row * d, gam, bet,
                       out + (size_t)row * d, lane);
}

// ------------------------------------------------------------------------------------------------
// Causal self-attention over the H action tokens of one candidate; one warp per (candidate, head).
// qkv [M, 3d] -> out [M, d].  H <= 64, dh = d / heads a multiple of 32 and <= 128.
// ------------------------------------------------------------------------------------------------
template <typename T>
__global__ void self_attn_kernel(const T* qkv, T* __restrict__ out, int n_cand, int H, int d,
                                 int heads, int causal, LiveRows lv) {
  pdl_trigger();
  pdl_wait();
  n_cand = live_rows(lv, n_cand);
  extern __shared__ float sm[];
  const int dh = d / heads;
  const int wpb = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = blockIdx.x * wpb + warp;
  if (gid >= n_cand * heads) return;
  const int n = gid / heads, hd = gid % heads;
  float* Q = sm + (size_t)warp * (H * dh + 2 * H * (dh + 1));
  float* Kt = Q + H * dh;
  float* V = Kt + H * (dh + 1);
  const T* base = qkv + (size_t)n * H * 3 * d + hd * dh;
  for (int i = lane; i < H * dh; i += 32) {
    const int r = i / dh, c = i % dh;
    const T* p = base + (size_t)r * 3 * d + c;
    Q[r * dh + c] = to_f(p[0]);
    Kt[r * (dh + 1) + c] = to_f(p[d]);
    V[r * (dh + 1) + c] = to_f(p[2 * d]);
  }
  __syncwarp();
  const float scale = rsqrtf((float)dh);
  for (int r = 0; r < H; ++r) {
    const int last = causal ? r : H - 1;            // last key this query sees
    float s0 = -INFINITY, s1 = -INFINITY;
    if (lane <= last) {
      float a = 0.f;
      for (int i = 0; i < dh; ++i) a += Q[r * dh + i] * Kt[lane * (dh + 1) + i];
      s0 = a * scale;
    }
    if (lane + 32 <= last) {
      float a = 0.f;
      for (int i = 0; i < dh; ++i) a += Q[r * dh + i] * Kt[(lane + 32) * (dh + 1) + i];
      s1 = a * scale;
    }
    const float m = warp_max(fmaxf(s0, s1));
    const float p0 = (lane <= last) ? __expf(s0 - m) : 0.f;
    const float p1 = (lane + 32 <= last) ? __expf(s1 - m) : 0.f;
    const float inv = 1.0f / warp_sum(p0 + p1);
    for (int c0 = 0; c0 < dh; c0 += 32) {
      float o = 0.f;
      for (int c = 0; c <= last; ++c) {
        const float p = __shfl_sync(0xffffffffu, c < 32 ? p0 : p1, c & 31);
        o += p * V[c * (dh + 1) + c0 + lane];
      }
      out[((size_t)n * H + r) * d + hd * dh + c0 + lane] = from_f<T>(o * inv);
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Cross-attention to the memory [time token(tau) | obs tokens]; one warp per token row.
// Keys/values are precomputed: kv_time [T, L*2d] (a function of tau only, built at weight load) and
// kv_obs [B*To, L*2d] (built once per chunk); layer l occupies columns [l*2d, (l+1)*2d) = [K | V].
// ------------------------------------------------------------------------------------------------
template <typename T>
__global__ void cross_attn_kernel(const T* q, T* __restrict__ out, const float* __restrict__ kv_time,
                                  const float* kv_obs, CandMap cm, int M, int H, int d, int heads,
                                  int To, int layer, int L, int Tsteps) {
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const int n = row / H;
  if (n >= cand_count(cm, M / H)) return;
  int b, c;
  cand_decode(cm, n, b, c);
  int tau = cm.t[b] - cm.koff - c;
  tau = max(0, min(Tsteps - 1, tau));
  const int dh = d / heads;
  const size_t ld = (size_t)L * 2 * d;
  const float* kt = kv_time + (size_t)tau * ld + (size_t)layer * 2 * d;
  const float* ko = kv_obs + (size_t)item_of(cm.item, b) * To * ld + (size_t)layer * 2 * d;
  const float scale = rsqrtf((float)dh);
  const int NK = 1 + To;
  for (int hd = 0; hd < heads; ++hd) {
    float sc[9];
    float m = -INFINITY;
    for (int kx = 0; kx < NK; ++kx) {
      const float* kp = (kx == 0 ? kt : ko + (size_t)(kx - 1) * ld) + hd * dh;
      float a = 0.f;
      for (int i = lane; i < dh; i += 32) a += to_f(q[(size_t)row * d + hd * dh + i]) * kp[i];
      sc[kx] = warp_sum(a) * scale;
      m = fmaxf(m, sc[kx]);
    }
    float l = 0.f;
    for (int kx = 0; kx < NK; ++kx) { sc[kx] = __expf(sc[kx] - m); l += sc[kx]; }
    const float inv = 1.0f / l;
    for (int i = lane; i < dh; i += 32) {
      float o = 0.f;
      for (int kx = 0; kx < NK; ++kx) {
        const float* vp = (kx == 0 ? kt : ko + (size_t)(kx - 1) * ld) + d + hd * dh;
        o += sc[kx] * vp[i];
      }
      out[(size_t)row * d + hd * dh + i] = from_f<T>(o * inv);
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Tensor-core causal self-attention for bf16 activations: one warp per (candidate, head, 16-query
// tile).  S = Q K^T and O = P V run on mma.sync m16n8k16 (the sequence has at most 64 tokens, so
// one warp-level tile covers it; a tcgen05 tile would be 8x too tall).  Operand fragments are read
// straight from qkv [M, 3d]; the softmax lives in the accumulator registers; the output tile is
// staged in shared memory so that every lane stores 16 contiguous bytes.
// ------------------------------------------------------------------------------------------------
constexpr int SA_WARPS = 4;

template <int DH>
__global__ void __launch_bounds__(SA_WARPS * 32)
self_attn_mma_kernel(const __nv_bfloat16* qkv, __nv_bfloat16* __restrict__ out, int n_cand, int H, int d,
                     int heads, int causal, LiveRows lv) {
  pdl_trigger(true);
  pdl_wait();
  n_cand = live_rows(lv, n_cand);
  constexpr int KS = DH / 16;        // k-steps of Q K^T
  constexpr int NO = DH / 8;         // n-tiles of the output
  constexpr int LDS = DH + 8;        // staging row pitch (elements); keeps 16-byte alignment
  __shared__ __align__(16) __nv_bfloat16 stage[SA_WARPS][16 * LDS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int QT = (H + 15) >> 4;
  const int wg = blockIdx.x * SA_WARPS + warp;
  if (wg >= n_cand * heads * QT) return;
  const int qt = wg % QT, hd = (wg / QT) % heads, n = wg / (QT * heads);
  const int g = lane >> 2, tg = lane & 3;
  const size_t ld = (size_t)3 * d;
  const __nv_bfloat16* base = qkv + (size_t)n * H * ld + (size_t)hd * DH;
  const int r0 = qt * 16 + g, r1 = r0 + 8;
  auto ld32 = [&](int row, int col) -> uint32_t {
    return row < H ? *reinterpret_cast<const uint32_t*>(base + (size_t)row * ld + col) : 0u;
  };
  uint32_t qa[KS][4];
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const int c = ks * 16 + 2 * tg;
    qa[ks][0] = ld32(r0, c); qa[ks][1] = ld32(r1, c); qa[ks][2] = ld32(r0, c + 8); qa[ks][3] = ld32(r1, c + 8);
  }
  // keys 0 .. 16 (qt+1) - 1 are the only ones a causal query of this tile can see; a bidirectional one sees all H
  const int nkt = causal ? 2 * (qt + 1) : (H + 7) >> 3;
  const int kst = causal ? qt + 1 : (H + 15) >> 4;
  float s[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
    if (nt < nkt) {
      const int key = nt * 8 + g;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const int c = d + ks * 16 + 2 * tg;
        mma_bf16_16816(s[nt], qa[ks], ld32(key, c), ld32(key, c + 8));
      }
    }
  }
  const float scale = rsqrtf((float)DH);
  float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    if (nt < nkt) {
      const int col = nt * 8 + 2 * tg;
      const int lim0 = causal ? r0 : H, lim1 = causal ? r1 : H;
      s[nt][0] = (col <= lim0 && col < H) ? s[nt][0] * scale : -INFINITY;
      s[nt][1] = (col + 1 <= lim0 && col + 1 < H) ? s[nt][1] * scale : -INFINITY;
      s[nt][2] = (col <= lim1 && col < H) ? s[nt][2] * scale : -INFINITY;
      s[nt][3] = (col + 1 <= lim1 && col + 1 < H) ? s[nt][3] * scale : -INFINITY;
      m0 = fmaxf(m0, fmaxf(s[nt][0], s[nt][1]));
      m1 = fmaxf(m1, fmaxf(s[nt][2], s[nt][3]));
    }
  }
  m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 1)); m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 2));
  m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 1)); m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 2));
  // rows beyond H have no visible key: keep the arithmetic finite, their output is never stored
  if (m0 == -INFINITY) m0 = 0.f;
  if (m1 == -INFINITY) m1 = 0.f;
  float l0 = 0.f, l1 = 0.f;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    if (nt < nkt) {
      s[nt][0] = __expf(s[nt][0] - m0); s[nt][1] = __expf(s[nt][1] - m0);
      s[nt][2] = __expf(s[nt][2] - m1); s[nt][3] = __expf(s[nt][3] - m1);
      l0 += s[nt][0] + s[nt][1]; l1 += s[nt][2] + s[nt][3];
    }
  }
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  const float inv0 = l0 > 0.f ? 1.0f / l0 : 0.f, inv1 = l1 > 0.f ? 1.0f / l1 : 0.f;
  // O = P V; the accumulator layout of two adjacent key tiles is the A-operand layout of one k-step
  float o[NO][4];
#pragma unroll
  for (int no = 0; no < NO; ++no) o[no][0] = o[no][1] = o[no][2] = o[no][3] = 0.f;
  const __nv_bfloat16* vbase = base + 2 * d;
  const unsigned short* vraw = reinterpret_cast<const unsigned short*>(vbase);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (j < kst) {
      uint32_t pa[4];
      pa[0] = pack_bf16(s[2 * j][0], s[2 * j][1]); pa[1] = pack_bf16(s[2 * j][2], s[2 * j][3]);
      pa[2] = pack_bf16(s[2 * j + 1][0], s[2 * j + 1][1]); pa[3] = pack_bf16(s[2 * j + 1][2], s[2 * j + 1][3]);
      const int k0 = 16 * j + 2 * tg;
#pragma unroll
      for (int no = 0; no < NO; ++no) {
        const int col = no * 8 + g;
        auto v16 = [&](int key) -> uint32_t {
          return key < H ? (uint32_t)vraw[(size_t)key * ld + col] : 0u;
        };
        const uint32_t b0 = v16(k0) | (v16(k0 + 1) << 16);
        const uint32_t b1 = v16(k0 + 8) | (v16(k0 + 9) << 16);
        mma_bf16_16816(o[no], pa, b0, b1);
      }
    }
  }
  __nv_bfloat16* st = stage[warp];
#pragma unroll
  for (int no = 0; no < NO; ++no) {
    const int col = no * 8 + 2 * tg;
    *reinterpret_cast<uint32_t*>(st + g * LDS + col) = pack_bf16(o[no][0] * inv0, o[no][1] * inv0);
    *reinterpret_cast<uint32_t*>(st + (g + 8) * LDS + col) = pack_bf16(o[no][2] * inv1, o[no][3] * inv1);
  }
  __syncwarp();
  constexpr int VPR = DH / 8;        // 16-byte vectors per row
  for (int i = lane; i < 16 * VPR; i += 32) {
    const int r = i / VPR, v = i % VPR;
    const int row = qt * 16 + r;
    if (row < H)
      *reinterpret_cast<uint4*>(out + ((size_t)n * H + row) * d + (size_t)hd * DH + v * 8) =
          *reinterpret_cast<const uint4*>(st + r * LDS + v * 8);
  }
}

// ------------------------------------------------------------------------------------------------
// Self-attention for sequences of at most 16 tokens, bf16: one warp per (candidate, head).  The warp
// copies the head's Q, K and V rows into its own piece of shared memory with 16-byte loads (a
// lane-by-lane gather of fragments from global memory costs one L1 tag look-up per 16 bytes) and takes
// the mma operands from there: Q with 4-byte loads, K through ldmatrix, V through ldmatrix.trans.
// ------------------------------------------------------------------------------------------------
template <int DH>
__global__ void __launch_bounds__((DH > 64 ? 2 : 4) * 32)
self_attn_tile_kernel(const __nv_bfloat16* qkv, __nv_bfloat16* __restrict__ out, int n_cand, int H, int d,
                      int heads, int causal, LiveRows lv) {
  pdl_trigger(true);
  pdl_wait();
  n_cand = live_rows(lv, n_cand);
  constexpr int TW = DH > 64 ? 2 : 4;
  constexpr int KS = DH / 16, NO = DH / 8, P = DH + 8, VPR = DH / 8;
  __shared__ __align__(16) __nv_bfloat16 sm[TW][3][16 * P];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
  const int wg = blockIdx.x * TW + warp;
  if (wg >= n_cand * heads) return;
  const int hd = wg % heads, n = wg / heads;
  const size_t ld = (size_t)3 * d;
  const __nv_bfloat16* base = qkv + (size_t)n * H * ld + (size_t)hd * DH;
  __nv_bfloat16* sQ = sm[warp][0];
  __nv_bfloat16* sK = sm[warp][1];
  __nv_bfloat16* sV = sm[warp][2];
  constexpr int NV = 3 * 16 * VPR / 32;          // 16-byte vectors per lane
  constexpr int CH = NV > 12 ? NV / 2 : NV;      // in flight at a time
#pragma unroll
  for (int c0 = 0; c0 < NV; c0 += CH) {
    uint4 buf[CH];
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int idx = (c0 + i) * 32 + lane;
      const int which = idx / (16 * VPR), rem = idx % (16 * VPR), r = rem / VPR, v = rem % VPR;
      buf[i] = r < H ? reinterpret_cast<const uint4*>(base + (size_t)r * ld + (size_t)which * d)[v] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int idx = (c0 + i) * 32 + lane;
      const int which = idx / (16 * VPR), rem = idx % (16 * VPR), r = rem / VPR, v = rem % VPR;
      *reinterpret_cast<uint4*>(sm[warp][which] + r * P + v * 8) = buf[i];
    }
  }
  __syncwarp();
  attn16_from_smem<DH>(sQ, sK, sV, H, causal, lane);
  __syncwarp();
  for (int i = lane; i < 16 * VPR; i += 32) {
    const int r = i / VPR, v = i % VPR;
    if (r < H)
      *reinterpret_cast<uint4*>(out + ((size_t)n * H + r) * d + (size_t)hd * DH + v * 8) =
          *reinterpret_cast<const uint4*>(sQ + r * P + v * 8);
  }
}

// ------------------------------------------------------------------------------------------------
// Self-attention for sequences longer than one 16-row tile (17..64 tokens), bf16: one block per
// (candidate, head), one warp per 16-query tile.  Bound by memory where it matters (q, k, v in, o out: 54 400 rows of width 1024
// 445 MB), so everything moves in whole 16-byte words of whole rows and at once: queries, keys and values come by cp.async into shared
// memory and become mma operands through ldmatrix (values transposed), a warp's output leaves through its own (dead) query
// rows.  Before, queries and outputs went as 4-byte words per lane and the queries behind the barrier: 54 400 x 1024, 16 heads 176 -> 155 us,
// 150 x 512, 8 heads 5.2 -> 4.8.  (Eight blocks an SM instead of six cost registers that spill: 172.)  causal = 0 gives the bidirectional attention of the DiT blocks.
// ------------------------------------------------------------------------------------------------
template <int DH>
__host__ __device__ constexpr int sa_smem_bytes() { return 3 * 64 * (DH + 8) * 2; }
template <int DH>
__global__ void __launch_bounds__(128)
self_attn_staged_kernel(const __nv_bfloat16* qkv, __nv_bfloat16* __restrict__ out, int n_cand, int H, int d,
                        int heads, int causal, LiveRows lv) {
  pdl_trigger(true);
  pdl_wait();
  constexpr int KS = DH / 16, NO = DH / 8, P = DH + 8, VPR = DH / 8;
  extern __shared__ __align__(16) uint8_t sa_raw[];
  __nv_bfloat16 *Qs = reinterpret_cast<__nv_bfloat16*>(sa_raw), *Ks = Qs + 64 * P, *Vs = Ks + 64 * P;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
  const int n = blockIdx.x / heads, hd = blockIdx.x % heads;
  if (n >= live_rows(lv, n_cand)) return;
  const size_t ld = (size_t)3 * d;
  const __nv_bfloat16* base = qkv + (size_t)n * H * ld + (size_t)hd * DH;
  for (int i = threadIdx.x; i < 64 * VPR; i += blockDim.x) {
    const int r = i / VPR, v = (i % VPR) * 8;
    if (r < H) {
      const __nv_bfloat16* src = base + (size_t)r * ld + v;
      cp_async16(Qs + r * P + v, src);
      cp_async16(Ks + r * P + v, src + d);
      cp_async16(Vs + r * P + v, src + 2 * d);
    } else {      // rows past H: weights of zero must not meet what happens to lie there
      const uint4 z = make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(Qs + r * P + v) = z; *reinterpret_cast<uint4*>(Ks + r * P + v) = z; *reinterpret_cast<uint4*>(Vs + r * P + v) = z;
    }
  }
  cp_async_wait_all();
  __syncthreads();
  const int qt = warp;
  if (qt * 16 >= H) return;
  const int r0 = qt * 16 + g, r1 = r0 + 8;
  uint32_t qa[KS][4];
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) ldmatrix_x4(qa[ks], Qs + (qt * 16 + (lane & 15)) * P + ks * 16 + 8 * (lane >> 4));
  const int nkt = causal ? 2 * (qt + 1) : (H + 7) >> 3;
  const int kst = causal ? qt + 1 : (H + 15) >> 4;
  float s[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
    if (nt < nkt) {
#pragma unroll
      for (int ks = 0; ks < KS; ks += 2) {
        uint32_t b[4];
        ldmatrix_x4(b, Ks + (nt * 8 + (lane & 7)) * P + ks * 16 + 8 * (lane >> 3));
        mma_bf16_16816(s[nt], qa[ks], b[0], b[1]);
        mma_bf16_16816(s[nt], qa[ks + 1], b[2], b[3]);
      }
    }
  }
  const float scale = rsqrtf((float)DH);
  float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    if (nt < nkt) {
      const int col = nt * 8 + 2 * tg;
      const int lim0 = causal ? r0 : H, lim1 = causal ? r1 : H;
      s[nt][0] = (col <= lim0 && col < H) ? s[nt][0] * scale : -INFINITY;
      s[nt][1] = (col + 1 <= lim0 && col + 1 < H) ? s[nt][1] * scale : -INFINITY;
      s[nt][2] = (col <= lim1 && col < H) ? s[nt][2] * scale : -INFINITY;
      s[nt][3] = (col + 1 <= lim1 && col + 1 < H) ? s[nt][3] * scale : -INFINITY;
      m0 = fmaxf(m0, fmaxf(s[nt][0], s[nt][1]));
      m1 = fmaxf(m1, fmaxf(s[nt][2], s[nt][3]));
    }
  }
  m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 1)); m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, 2));
  m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 1)); m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, 2));
  if (m0 == -INFINITY) m0 = 0.f;
  if (m1 == -INFINITY) m1 = 0.f;
  float l0 = 0.f, l1 = 0.f;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    if (nt < nkt) {
      s[nt][0] = __expf(s[nt][0] - m0); s[nt][1] = __expf(s[nt][1] - m0);
      s[nt][2] = __expf(s[nt][2] - m1); s[nt][3] = __expf(s[nt][3] - m1);
      l0 += s[nt][0] + s[nt][1]; l1 += s[nt][2] + s[nt][3];
    }
  }
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  const float inv0 = l0 > 0.f ? 1.0f / l0 : 0.f, inv1 = l1 > 0.f ? 1.0f / l1 : 0.f;
  float o[NO][4];
#pragma unroll
  for (int no = 0; no < NO; ++no) o[no][0] = o[no][1] = o[no][2] = o[no][3] = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (j < kst) {
      uint32_t pa[4];
      pa[0] = pack_bf16(s[2 * j][0], s[2 * j][1]); pa[1] = pack_bf16(s[2 * j][2], s[2 * j][3]);
      pa[2] = pack_bf16(s[2 * j + 1][0], s[2 * j + 1][1]); pa[3] = pack_bf16(s[2 * j + 1][2], s[2 * j + 1][3]);
#pragma unroll
      for (int no = 0; no < NO; no += 2) {
        uint32_t b[4];
        ldmatrix_x4_trans(b, Vs + (16 * j + (lane & 7) + 8 * ((lane >> 3) & 1)) * P + no * 8 + 8 * (lane >> 4));
        mma_bf16_16816(o[no], pa, b[0], b[1]);
        mma_bf16_16816(o[no + 1], pa, b[2], b[3]);
      }
    }
  }
  __nv_bfloat16* ow = Qs + qt * 16 * P;      // this warp's query rows: nobody else reads them
  __syncwarp();
#pragma unroll
  for (int no = 0; no < NO; ++no) {
    *reinterpret_cast<uint32_t*>(ow + g * P + no * 8 + 2 * tg) = pack_bf16(o[no][0] * inv0, o[no][1] * inv0);
    *reinterpret_cast<uint32_t*>(ow + (g + 8) * P + no * 8 + 2 * tg) = pack_bf16(o[no][2] * inv1, o[no][3] * inv1);
  }
  __syncwarp();
  __nv_bfloat16* og = out + ((size_t)n * H + qt * 16) * d + (size_t)hd * DH;
  for (int i = lane; i < 16 * VPR; i += 32) {
    const int r = i / VPR, v = (i % VPR) * 8;
    if (qt * 16 + r < H) *reinterpret_cast<uint4*>(og + (size_t)r * d + v) = *reinterpret_cast<const uint4*>(ow + r * P + v);
  }
}

// ------------------------------------------------------------------------------------------------
// Cross-attention for bf16 activations with at most 4 memory tokens: DH/8 lanes own one (candidate,
// head); they load that head's keys and values once into registers (they are the same for all H
// query rows of the candidate) and then stream the H query rows, 16 bytes per lane per row.
// ------------------------------------------------------------------------------------------------
constexpr int CA_MAXNK = 4;
constexpr int CA_ROWS = 4;

template <int DH>
__global__ void __launch_bounds__(256)
cross_attn_group_kernel(const __nv_bfloat16* q, __nv_bfloat16* __restrict__ out,
                        const float* __restrict__ kv_time, const float* kv_obs, CandMap cm, int n_cand,
                        int H, int d, int heads, int To, int layer, int L, int Tsteps) {
  pdl_trigger();
  pdl_wait();
  constexpr int LG = DH / 8;
  const int gid_raw = (blockIdx.x * blockDim.x + threadIdx.x) / LG;
  const int sub = threadIdx.x % LG;
  // a group works on CA_ROWS consecutive query rows of its (candidate, head): more groups in flight than
  // one per (candidate, head) would give, at the price of re-reading the few keys / values from cache
  const int row_chunks = (H + CA_ROWS - 1) / CA_ROWS;
  n_cand = cand_count(cm, n_cand);
  if (n_cand <= 0) return;
  const bool live = gid_raw < n_cand * heads * row_chunks;
  const int gid_c = live ? gid_raw : n_cand * heads * row_chunks - 1;
  const int rc = gid_c % row_chunks, gid = gid_c / row_chunks;
  const int n = gid / heads, hd = gid % heads;
  int b, c;
  cand_decode(cm, n, b, c);
  int tau = cm.t[b] - cm.koff - c;
  tau = max(0, min(Tsteps - 1, tau));
  const size_t ldkv = (size_t)L * 2 * d;
  const int NK = 1 + To;
  float kreg[CA_MAXNK][8], vreg[CA_MAXNK][8];
#pragma unroll
  for (int kx = 0; kx < CA_MAXNK; ++kx) {
    if (kx < NK) {
      const float* kp = (kx == 0 ? kv_time + (size_t)tau * ldkv : kv_obs + ((size_t)item_of(cm.item, b) * To + (kx - 1)) * ldkv) +
                        (size_t)layer * 2 * d + hd * DH + sub * 8;
      const float4 k0 = reinterpret_cast<const float4*>(kp)[0], k1 = reinterpret_cast<const float4*>(kp)[1];
      const float4 v0 = reinterpret_cast<const float4*>(kp + d)[0], v1 = reinterpret_cast<const float4*>(kp + d)[1];
      kreg[kx][0] = k0.x; kreg[kx][1] = k0.y; kreg[kx][2] = k0.z; kreg[kx][3] = k0.w;
      kreg[kx][4] = k1.x; kreg[kx][5] = k1.y; kreg[kx][6] = k1.z; kreg[kx][7] = k1.w;
      vreg[kx][0] = v0.x; vreg[kx][1] = v0.y; vreg[kx][2] = v0.z; vreg[kx][3] = v0.w;
      vreg[kx][4] = v1.x; vreg[kx][5] = v1.y; vreg[kx][6] = v1.z; vreg[kx][7] = v1.w;
    }
  }
  const float scale = rsqrtf((float)DH);
  const __nv_bfloat16* qp = q + (size_t)n * H * d + (size_t)hd * DH + sub * 8;
  __nv_bfloat16* op = out + (size_t)n * H * d + (size_t)hd * DH + sub * 8;
#pragma unroll
  for (int rr = 0; rr < CA_ROWS; ++rr) {
    const int r = min(rc * CA_ROWS + rr, H - 1);       // a ragged last chunk repeats its last row
    const uint4 qv = *reinterpret_cast<const uint4*>(qp + (size_t)r * d);
    const __nv_bfloat162* q2 = reinterpret_cast<const __nv_bfloat162*>(&qv);
    float qf[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 f = __bfloat1622float2(q2[i]); qf[2 * i] = f.x; qf[2 * i + 1] = f.y; }
    float sc[CA_MAXNK];
    float m = -INFINITY;
#pragma unroll
    for (int kx = 0; kx < CA_MAXNK; ++kx) {
      if (kx < NK) {
        float a = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) a += qf[i] * kreg[kx][i];
#pragma unroll
        for (int o = LG / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        sc[kx] = a * scale;
        m = fmaxf(m, sc[kx]);
      }
    }
    float l = 0.f;
#pragma unroll
    for (int kx = 0; kx < CA_MAXNK; ++kx)
      if (kx < NK) { sc[kx] = __expf(sc[kx] - m); l += sc[kx]; }
    const float inv = 1.0f / l;
    float o8[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) o8[i] = 0.f;
#pragma unroll
    for (int kx = 0; kx < CA_MAXNK; ++kx)
      if (kx < NK) {
#pragma unroll
        for (int i = 0; i < 8; ++i) o8[i] += sc[kx] * vreg[kx][i];
      }
    uint4 ov;
    ov.x = pack_bf16(o8[0] * inv, o8[1] * inv); ov.y = pack_bf16(o8[2] * inv, o8[3] * inv);
    ov.z = pack_bf16(o8[4] * inv, o8[5] * inv); ov.w = pack_bf16(o8[6] * inv, o8[7] * inv);
    if (live) *reinterpret_cast<uint4*>(op + (size_t)r * d) = ov;
  }
}

// ------------------------------------------------------------------------------------------------
// Output head: eps[n, i, :] = LN_f(h[row]) W_out + b_out, one warp per row; W_outT is [A, d] fp32.
// ------------------------------------------------------------------------------------------------
// Final LayerNorm of one row by one warp, result left in v (lane owns columns (j*32 + lane)*4 .. +3).
template <int VEC>
__device__ __forceinline__ void head_ln_row(const float* h_row, const float* __restrict__ gam,
                                            const float* __restrict__ bet, float4 (&v)[VEC], int lane) {
  constexpr int d = VEC * 128;
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    v[j] = reinterpret_cast<const float4*>(h_row)[j * 32 + lane];
    s += v[j].x + v[j].y + v[j].z + v[j].w;
  }
  const float mean = warp_sum(s) / d;
  float q = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    v[j].x -= mean; v[j].y -= mean; v[j].z -= mean; v[j].w -= mean;
    q += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
  }
  const float rstd = rsqrtf(warp_sum(q) / d + 1e-5f);
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    const float4 gg = reinterpret_cast<const float4*>(gam)[j * 32 + lane];
    const float4 bb = reinterpret_cast<const float4*>(bet)[j * 32 + lane];
    v[j].x = v[j].x * rstd * gg.x + bb.x; v[j].y = v[j].y * rstd * gg.y + bb.y;
    v[j].z = v[j].z * rstd * gg.z + bb.z; v[j].w = v[j].w * rstd * gg.w + bb.w;
  }
}
// eps of action a for that row (the same value in every lane); products and sums spelled out so that every
// kernel that computes it gets the same bits.
template <int VEC>
__device__ __forceinline__ float head_out(const float4 (&v)[VEC], const float* __restrict__ w_row, float bias, int lane) {
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    const float4 w = reinterpret_cast<const float4*>(w_row)[j * 32 + lane];
    acc = __fmaf_rn(v[j].x, w.x, acc); acc = __fmaf_rn(v[j].y, w.y, acc);
    acc = __fmaf_rn(v[j].z, w.z, acc); acc = __fmaf_rn(v[j].w, w.w, acc);
  }
  return __fadd_rn(warp_sum(acc), bias);
}

template <int VEC>
__global__ void head_kernel(const float* h, const float* __restrict__ gam, const float* __restrict__ bet,
                            const float* __restrict__ W_outT, const float* __restrict__ b_out, CandMap cm, int M,
                            int H, int A) {
  pdl_trigger();
  pdl_wait();
  constexpr int d = VEC * 128;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const int n = row / H, i = row % H;
  if (n >= cand_count(cm, M / H)) return;
  float4 v[VEC];
  head_ln_row<VEC>(h + (size_t)row * d, gam, bet, v, lane);
  int b, c;
  cand_decode(cm, n, b, c);
  float* o = cm.eout + b * cm.e_stride_b + (long long)c * H * A + (long long)i * A;
  for (int a = 0; a < A; ++a) {
    const float e = head_out<VEC>(v, W_outT + (size_t)a * d, b_out[a], lane);
    if (lane == 0) o[a] = e;
  }
}

// Closed-form denoiser of iid N(m0, s0^2) data: eps = sqrt(1-abar)(x - sqrt(abar) m0)/(abar s0^2 + 1 - abar).
__global__ void gauss_forward_kernel(DdpmTables S, float m0, float s0, CandMap cm, int n_cand, int D) {
  pdl_trigger();
  pdl_wait();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n_cand * D) return;
  const int n = (int)(idx / D), i = (int)(idx % D);
  if (n >= cand_count(cm, n_cand)) return;
  int b, c;
  cand_decode(cm, n, b, c);
  int tau = cm.t[b] - cm.koff - c;
  tau = max(0, min(S.T - 1, tau));
  const float sab = S.sqrt_ab[tau], s1 = S.sqrt_1mab[tau];
  const float ab = sab * sab;
  const float x = cm.xin[b * cm.x_stride_b + (long long)c * D + i];
  cm.eout[b * cm.e_stride_b + (long long)c * D + i] = s1 * (x - sab * m0) / (ab * s0 * s0 + s1 * s1);
}

}  // namespace tsdp
