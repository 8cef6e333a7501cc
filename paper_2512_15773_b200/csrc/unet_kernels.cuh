// Kernels of the 1-D temporal conv UNet around its convolutions.  Activations are channels-last and
// zero-padded along the sequence: a tensor of L positions and C channels of n candidates is stored as
// [n, L + 4, C] with two zero rows before and after the L valid ones.  In that layout the im2col
// matrix of a kernel-5 "same" convolution is a VIEW: row (n, l) starts at element ((n (L+4) + l) C)
// and is 5 C elements long (rows overlap), so every convolution runs on the tensor-core GEMM through a
// three-dimensional tensor map (channel, position, candidate) whose boxes hold the L valid positions of several
// candidates.  Its output rows are dense, r = n L + l.
// The kernels here write only valid rows, so the padding rows stay zero for the lifetime of a buffer.
#pragma once
#include "common.cuh"
#include "net_kernels.cuh"
#include "dit_kernels.cuh"

namespace tsdp {

__device__ __forceinline__ float mish_f(float v) {
  const float sp = v > 20.f ? v : log1pf(expf(v));       // softplus
  return v * tanhf(sp);
}

__global__ void mish_kernel(const float* in, float* out, long long n) {
  pdl_trigger();
  pdl_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = mish_f(in[i]);
}

// v tanh(softplus(v)) = v n / m with n = e^v (e^v + 2), m = n + 2: one exponential and one division in place of log1p, exp
// and tanh.  The quotient is taken of the smaller side, n / m = 1 - 2 / m above zero and
// e^v (1 - (e^2v + e^v) / m) below, where it is at most 0.4, so that the error of the fast division weighs 2/3 at most.
// Against 64 bits, in units of 2^-24 of the result, largest and rms over [-30, 25]: 4.2 and 0.70; v tanhf(log1pf(expf(v))) 5.4
// and 0.72, v * __fdividef(n, m) 5.6 and 0.93 (calls of the UNet workload with that one: 0.3 % faster at most).
__device__ __forceinline__ float mish_fast(float v) {
  if (v > 20.f) return v;
  const float e = expf(v), m = __fmaf_rn(e, e, e + e) + 2.f;
  const float c = 1.f - __fdividef(v > 0.f ? 2.f : __fmaf_rn(e, e, e), m);
  return v * (v > 0.f ? c : e * c);
}

// Input projection: X[n, l + 2, :] = x[n, l, :] W_in + b_in   (pointwise, A -> C channels).  A block takes the H rows of one
// candidate: a thread owns four channels of UE_ROWS rows at a time, so a weight is read once for all of them.
// 288 candidates, 10 -> 256 channels: one block per row (9.4 us) did nothing but wait for its weights.
constexpr int UE_ROWS = 4;
template <typename T>
__global__ void __launch_bounds__(256)
unet_embed_kernel(CandMap cm, const float* __restrict__ W_in, const float* __restrict__ b_in,
                  T* __restrict__ X, int H, int A, int C) {
  pdl_trigger(std::is_same<T, __nv_bfloat16>::value);
  pdl_wait();
  const int n = blockIdx.x;
  if (n >= cand_count(cm, gridDim.x)) return;
  int b, c;
  cand_decode(cm, n, b, c);
  const float* x = cm.xin + b * cm.x_stride_b + (long long)c * H * A;
  const int quads = C >> 2, groups = (H + UE_ROWS - 1) / UE_ROWS;
  for (int u = threadIdx.x; u < quads * groups; u += blockDim.x) {
    const int col = (u % quads) * 4, l0 = (u / quads) * UE_ROWS;
    const float4 bi = *reinterpret_cast<const float4*>(b_in + col);
    float4 acc[UE_ROWS];
#pragma unroll
    for (int r = 0; r < UE_ROWS; ++r) acc[r] = bi;
#pragma unroll 5
    for (int a = 0; a < A; ++a) {
      const float4 w = __ldg(reinterpret_cast<const float4*>(W_in + (size_t)a * C + col));
#pragma unroll
      for (int r = 0; r < UE_ROWS; ++r) {
        const float xv = x[min(l0 + r, H - 1) * A + a];
        acc[r].x += xv * w.x; acc[r].y += xv * w.y; acc[r].z += xv * w.z; acc[r].w += xv * w.w;
      }
    }
#pragma unroll
    for (int r = 0; r < UE_ROWS; ++r)
      if (l0 + r < H) store4(X + ((size_t)n * (H + 4) + l0 + r + 2) * C + col, acc[r].x, acc[r].y, acc[r].z, acc[r].w);
  }
}

// FiLM term of the observations: out[n, f] = sum_k x[n, k] W[f, k] (fp32).  A block holds UF_N rows of x in shared memory,
// a warp takes UF_F features at a time: lanes along k, 16-byte loads of the weight rows, one reduction per output.
// 14336 features of 1024 inputs: the weights are 59 MB, read once per UF_N rows; the general fp32 GEMM took 214 us whatever
// the number of rows (64 x 64 tiles with a serial loop over k).
constexpr int UF_N = 8, UF_F = 4;
constexpr size_t UF_MAX_SMEM = 200 * 1024;
__global__ void __launch_bounds__(256)
film_obs_kernel(const float* x, const float* __restrict__ W, float* __restrict__ out, int N, int F, int K) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) float sx_film[];      // [UF_N][Kp], zero beyond K and N
  const int fx = (F + 8 * UF_F - 1) / (8 * UF_F);      // blocks along the features (row blocks of a long queue exceed grid.y)
  const int Kp = (K + 3) & ~3, n0 = (int)(blockIdx.x / fx) * UF_N, nn = min(UF_N, N - n0);
  for (int i = threadIdx.x; i < UF_N * Kp; i += blockDim.x) {
    const int r = i / Kp, k = i - r * Kp;
    sx_film[i] = (r < nn && k < K) ? x[(size_t)(n0 + r) * K + k] : 0.f;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool vec = (K & 3) == 0;
  const int f0 = ((int)(blockIdx.x % fx) * 8 + warp) * UF_F;
  if (f0 < F) {
    float acc[UF_F][UF_N];
#pragma unroll
    for (int i = 0; i < UF_F; ++i)
#pragma unroll
      for (int r = 0; r < UF_N; ++r) acc[i][r] = 0.f;
    for (int k = lane * 4; k < Kp; k += 128) {
      float4 w[UF_F];
#pragma unroll
      for (int i = 0; i < UF_F; ++i) {
        const float* wr = W + (size_t)min(f0 + i, F - 1) * K + k;
        if (vec) w[i] = __ldg(reinterpret_cast<const float4*>(wr));
        else w[i] = make_float4(__ldg(wr), k + 1 < K ? __ldg(wr + 1) : 0.f, k + 2 < K ? __ldg(wr + 2) : 0.f, k + 3 < K ? __ldg(wr + 3) : 0.f);
      }
#pragma unroll
      for (int r = 0; r < UF_N; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(sx_film + r * Kp + k);
#pragma unroll
        for (int i = 0; i < UF_F; ++i) {
          acc[i][r] = __fmaf_rn(v.x, w[i].x, acc[i][r]); acc[i][r] = __fmaf_rn(v.y, w[i].y, acc[i][r]);
          acc[i][r] = __fmaf_rn(v.z, w[i].z, acc[i][r]); acc[i][r] = __fmaf_rn(v.w, w[i].w, acc[i][r]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < UF_F; ++i)
#pragma unroll
      for (int r = 0; r < UF_N; ++r) {
        const float s = warp_sum(acc[i][r]);
        if (lane == 0 && f0 + i < F && r < nn) out[(size_t)(n0 + r) * F + f0 + i] = s;
      }
  }
}

// GroupNorm + Mish (+ FiLM) (+ residual) over one (candidate, group) of a convolution's fp32 output Y, dense rows n L + l:
//   v = Mish(GN(Y)) ; v = scale v + bias (film_time != null) ; v += residual
// FiLM vectors of candidate n: film_time[tau(n)] + film_obs[item(n)], this block's scale at column foff, its bias at
// foff + C.  Residual: res_t (activation type, padded [n, L+4, res_pitch], channels 0..C-1) or res_f (fp32 dense
// rows, pitch C); at most one of them.  Y may arrive as n_split partial sums of the convolution's reduction, split_stride
// elements apart: added in the order of the parts, whichever CTA produced which.
// The result goes to any of: dst [n, L+4, dst_pitch] at channel coff; up [n, 2L+4, up_pitch] with every position repeated
// (the 2x repetition on the way up, channels from 0); pool [n, L/2+4, C] as means of neighbouring positions (of the
// rounded values), so that neither needs a pass of its own.
struct GnArgs {
  const float* Y; long long split_stride; int n_split;
  const float *gam, *bet; int groups;
  const float *film_time, *film_obs; int F, foff;
  int Tsteps;
  const void* res_t; int res_pitch; const float* res_f;
  void* dst; int dst_pitch, coff;
  void* up; int up_pitch;
  void* pool;
  int L, C;
};
__device__ __forceinline__ void gn_film_rows(const GnArgs& g, const CandMap& cm, int n, const float*& ft, const float*& fo) {
  int b, cc;
  cand_decode(cm, n, b, cc);
  const int tau = max(0, min(g.Tsteps - 1, cm.t[b] - cm.koff - cc));
  ft = g.film_time + (size_t)tau * g.F + g.foff;
  fo = g.film_obs + (size_t)item_of(cm.item, b) * g.F + g.foff;
}
__device__ __forceinline__ float4 gn_load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 gn_load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// TPG threads per (candidate, group), up to GN_ITEMS float4 of it in each thread's registers: Y is read once (all parts and
// all values in flight together), statistics in two steps in registers, 8-byte bf16 stores.  One warp per group (no
// block barrier) where there are enough groups to fill the chip, four where there are not.  MAXS: parts.
// 288 candidates x 8 groups of 512 values: 12.6 us with 256 scalar threads per group and two passes over Y.
// PRE: the sums (those of a candidate past the live ones exist) are on their way beside the live count and the candidate, whose timestep and
// request follow and then, beside the statistics, the affine and FiLM vectors, in place of one behind the other.  64 registers a thread
// in place of 56: eight blocks an SM in place of nine.  Chains of launches of 16 x 256 values in 8 groups a candidate, residual / FiLM form, us a
// launch without and with it: 2 groups per SM 4.19 / 4.38 -> 3.43 / 3.42, 4 4.73 / 4.97 -> 3.69 / 3.74, 8 4.91 / 5.16 -> 4.71 / 4.86, 10 6.39 / 6.45 -> 6.60 / 6.81,
// 16 7.78 / 8.03 -> 8.29 / 8.46, 32 13.8 / 14.4 -> 15.3 / 15.5.  With a warp per group it loses on one form what it wins on the other (32 groups per SM
// 8.70 / 8.96 -> 8.80 / 8.65, 64 16.9 / 16.3 -> 17.2 / 15.6) and spills.
constexpr int GN_ITEMS = 4;
constexpr int GN_PRE_BLOCKS = 8;      // of the PRE form on an SM
template <typename T, int TPG, int MAXS, bool PRE>
__global__ void __launch_bounds__(TPG == 32 ? 256 : TPG, MAXS == 2 ? (TPG == 32 ? 4 : (PRE ? GN_PRE_BLOCKS : 9)) : 1)
gn_mish_kernel(GnArgs g, CandMap cm, int n_static) {
  pdl_trigger(std::is_same<T, __nv_bfloat16>::value);
  pdl_wait();
  constexpr int GPB = TPG == 32 ? 8 : 1;                  // groups per block
  __shared__ float s_red[2][TPG / 32];
  __shared__ float4 s_pool[GPB][GN_ITEMS * TPG];
  const int sub = TPG == 32 ? (threadIdx.x >> 5) : 0, t = TPG == 32 ? (threadIdx.x & 31) : threadIdx.x;
  const int gid = blockIdx.x * GPB + sub, n = gid / g.groups, grp = gid - n * g.groups;
  if (n >= (PRE ? n_static : cand_count(cm, n_static))) return;      // the whole warp (TPG 32) or block
  const int Cg = g.C / g.groups, quads = Cg >> 2, items = g.L * quads, cnt = g.L * Cg;
  const int q_step = TPG % quads, l_step = TPG / quads;
  int lj[GN_ITEMS], qj[GN_ITEMS];
  lj[0] = t / quads; qj[0] = t - lj[0] * quads;
#pragma unroll
  for (int j = 1; j < GN_ITEMS; ++j) {
    lj[j] = lj[j - 1] + l_step; qj[j] = qj[j - 1] + q_step;
    if (qj[j] >= quads) { qj[j] -= quads; ++lj[j]; }
  }
  float4 v[GN_ITEMS];
#pragma unroll
  for (int j = 0; j < GN_ITEMS; ++j) {
    v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j * TPG + t < items) {
      const float* y = g.Y + ((size_t)n * g.L + lj[j]) * g.C + grp * Cg + 4 * qj[j];
      float4 p[MAXS];
#pragma unroll
      for (int s = 0; s < MAXS; ++s) if (s < g.n_split) p[s] = load_now(y + (size_t)s * (size_t)g.split_stride);
      v[j] = p[0];
#pragma unroll
      for (int s = 1; s < MAXS; ++s) if (s < g.n_split) { v[j].x += p[s].x; v[j].y += p[s].y; v[j].z += p[s].z; v[j].w += p[s].w; }
    }
  }
  int cb, cc;
  cand_decode(cm, n, cb, cc);
  if (PRE && n >= cand_count(cm, n_static)) return;
  const float *ft = nullptr, *fo = nullptr;
  if (g.film_time) {
    ft = g.film_time + (size_t)max(0, min(g.Tsteps - 1, cm.t[cb] - cm.koff - cc)) * g.F + g.foff;
    fo = g.film_obs + (size_t)item_of(cm.item, cb) * g.F + g.foff;
  }
  // (PRE: where a lane's values are all of the same four channels, the thread count being a multiple of the group's quads)
  const bool same = PRE && q_step == 0;
  float4 ga0, be0, fs0, fs1, fb0, fb1;
  auto vectors = [&](int c) {
    ga0 = load_now(g.gam + c); be0 = load_now(g.bet + c);
    if (ft) { fs0 = load_now(ft + c); fs1 = load_now(fo + c); fb0 = load_now(ft + g.C + c); fb1 = load_now(fo + g.C + c); }
  };
  if (same) vectors(grp * Cg + 4 * qj[0]);
  auto group_sum = [&](float x, int slot) {
    x = warp_sum(x);
    if (TPG == 32) return x;
    if ((threadIdx.x & 31) == 0) s_red[slot][threadIdx.x >> 5] = x;
    __syncthreads();
    float r = 0.f;
#pragma unroll
    for (int w = 0; w < TPG / 32; ++w) r += s_red[slot][w];
    return r;
  };
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < GN_ITEMS; ++j) s += (v[j].x + v[j].y) + (v[j].z + v[j].w);
  const float mean = group_sum(s, 0) / cnt;
  float q = 0.f;
#pragma unroll
  for (int j = 0; j < GN_ITEMS; ++j)
    if (j * TPG + t < items) {
      v[j].x -= mean; v[j].y -= mean; v[j].z -= mean; v[j].w -= mean;
      q += (v[j].x * v[j].x + v[j].y * v[j].y) + (v[j].z * v[j].z + v[j].w * v[j].w);
    }
  const float rstd = rsqrtf(group_sum(q, 1) / cnt + 1e-5f);
#pragma unroll
  for (int j = 0; j < GN_ITEMS; ++j) {
    if (j * TPG + t >= items) continue;
    const int l = lj[j], c = grp * Cg + 4 * qj[j];
    if (!same) vectors(c);
    float4 o;
    o.x = mish_fast(v[j].x * rstd * ga0.x + be0.x); o.y = mish_fast(v[j].y * rstd * ga0.y + be0.y);
    o.z = mish_fast(v[j].z * rstd * ga0.z + be0.z); o.w = mish_fast(v[j].w * rstd * ga0.w + be0.w);
    if (ft) {
      o.x = (fs0.x + fs1.x) * o.x + (fb0.x + fb1.x); o.y = (fs0.y + fs1.y) * o.y + (fb0.y + fb1.y);
      o.z = (fs0.z + fs1.z) * o.z + (fb0.z + fb1.z); o.w = (fs0.w + fs1.w) * o.w + (fb0.w + fb1.w);
    }
    const size_t prow = (size_t)n * (g.L + 4) + l + 2;
    if (g.res_t) {
      const float4 r = gn_load4(reinterpret_cast<const T*>(g.res_t) + prow * g.res_pitch + c);
      o.x += r.x; o.y += r.y; o.z += r.z; o.w += r.w;
    }
    if (g.res_f) {
      const float4 r = *reinterpret_cast<const float4*>(g.res_f + ((size_t)n * g.L + l) * g.C + c);
      o.x += r.x; o.y += r.y; o.z += r.z; o.w += r.w;
    }
    if (g.dst) store4(reinterpret_cast<T*>(g.dst) + prow * g.dst_pitch + g.coff + c, o.x, o.y, o.z, o.w);
    if (g.up) {
      T* u = reinterpret_cast<T*>(g.up) + ((size_t)n * (2 * g.L + 4) + 2 * l + 2) * g.up_pitch + c;
      store4(u, o.x, o.y, o.z, o.w);
      store4(u + g.up_pitch, o.x, o.y, o.z, o.w);
    }
    if (g.pool) s_pool[sub][j * TPG + t] = make_float4(to_f(from_f<T>(o.x)), to_f(from_f<T>(o.y)), to_f(from_f<T>(o.z)), to_f(from_f<T>(o.w)));
  }
  if (g.pool) {
    if (TPG == 32) __syncwarp(); else __syncthreads();
    for (int i = t; i < (g.L / 2) * quads; i += TPG) {
      const int l = i / quads, qd = i - l * quads;
      const float4 a = s_pool[sub][2 * l * quads + qd], b = s_pool[sub][(2 * l + 1) * quads + qd];
      store4(reinterpret_cast<T*>(g.pool) + ((size_t)n * (g.L / 2 + 4) + l + 2) * g.C + grp * Cg + 4 * qd,
             0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
    }
  }
}

// The same for groups that do not fit the registers of four warps or whose channels do not come in fours: one block per
// (candidate, group), value by value, Y read again in the second pass.
template <typename T>
__global__ void __launch_bounds__(256)
gn_mish_any_kernel(GnArgs g, CandMap cm, int n_static) {
  pdl_trigger();
  pdl_wait();
  __shared__ float red[2][8];
  const int n = blockIdx.x / g.groups, grp = blockIdx.x % g.groups;
  if (n >= cand_count(cm, n_static)) return;
  const int Cg = g.C / g.groups, cnt = g.L * Cg;
  auto y_at = [&](int l, int c) {
    const size_t idx = ((size_t)n * g.L + l) * g.C + c;
    float v = g.Y[idx];
    for (int s = 1; s < g.n_split; ++s) v += g.Y[idx + (size_t)s * (size_t)g.split_stride];
    return v;
  };
  float s = 0.f, q = 0.f;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const float v = y_at(i / Cg, grp * Cg + i % Cg);
    s += v; q += v * v;
  }
  s = warp_sum(s); q = warp_sum(q);
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = s; red[1][threadIdx.x >> 5] = q; }
  __syncthreads();
  float ts = 0.f, tq = 0.f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { ts += red[0][w]; tq += red[1][w]; }
  const float mean = ts / cnt;
  const float rstd = rsqrtf(fmaxf(tq / cnt - mean * mean, 0.f) + 1e-5f);
  const float *ft = nullptr, *fo = nullptr;
  if (g.film_time) gn_film_rows(g, cm, n, ft, fo);
  auto value = [&](int l, int c) {
    float v = mish_fast((y_at(l, c) - mean) * rstd * g.gam[c] + g.bet[c]);
    if (ft) v = (ft[c] + fo[c]) * v + (ft[g.C + c] + fo[g.C + c]);
    if (g.res_t) v += to_f(reinterpret_cast<const T*>(g.res_t)[((size_t)n * (g.L + 4) + l + 2) * g.res_pitch + c]);
    if (g.res_f) v += g.res_f[((size_t)n * g.L + l) * g.C + c];
    return from_f<T>(v);
  };
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const int l = i / Cg, c = grp * Cg + i % Cg;
    const T v = value(l, c);
    if (g.dst) reinterpret_cast<T*>(g.dst)[((size_t)n * (g.L + 4) + l + 2) * g.dst_pitch + g.coff + c] = v;
    if (g.up) {
      T* u = reinterpret_cast<T*>(g.up) + ((size_t)n * (2 * g.L + 4) + 2 * l + 2) * g.up_pitch + c;
      u[0] = v; u[g.up_pitch] = v;
    }
    if (g.pool && (l & 1) == 0)
      reinterpret_cast<T*>(g.pool)[((size_t)n * (g.L / 2 + 4) + l / 2 + 2) * g.C + c] = from_f<T>(0.5f * (to_f(v) + to_f(value(l + 1, c))));
  }
}

// Output projection: eps[n, l, :] = X[n, l + 2, :] W_out + b_out; one warp per position, UH_A outputs at a time (their
// loads and reductions overlap); W_outT [A, C] fp32, C a multiple of 128.
constexpr int UH_A = 5;
template <typename T>
__global__ void __launch_bounds__(256)
unet_head_kernel(const T* X, const float* __restrict__ W_outT, const float* __restrict__ b_out,
                 CandMap cm, int M, int H, int A, int C) {
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const int n = row / H, l = row % H;
  if (n >= cand_count(cm, M / H)) return;
  int b, c;
  cand_decode(cm, n, b, c);
  const T* x = X + ((size_t)n * (H + 4) + l + 2) * C;
  float* o = cm.eout + b * cm.e_stride_b + (long long)c * H * A + (long long)l * A;
  for (int a0 = 0; a0 < A; a0 += UH_A) {
    float acc[UH_A] = {};
#pragma unroll 2
    for (int i = lane * 4; i < C; i += 128) {
      const float4 xv = gn_load4(x + i);
#pragma unroll
      for (int j = 0; j < UH_A; ++j) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(W_outT + (size_t)min(a0 + j, A - 1) * C + i));
        acc[j] += (xv.x * w.x + xv.y * w.y) + (xv.z * w.z + xv.w * w.w);
      }
    }
#pragma unroll
    for (int j = 0; j < UH_A; ++j) acc[j] = warp_sum(acc[j]);
#pragma unroll
    for (int j = 0; j < UH_A; ++j)
      if (lane == j && a0 + j < A) o[a0 + j] = acc[j] + b_out[a0 + j];
  }
}

}  // namespace tsdp
