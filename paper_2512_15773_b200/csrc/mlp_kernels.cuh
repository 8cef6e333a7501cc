// Toy MLP denoiser (fp32): input [latent | sinusoidal(tau) | obs], SiLU hidden layers, linear head.
//
// A forward on one latent is a chain of matrix-vector products over a few hundred kilobytes of weights that sit in the
// L2, so what counts is how many loads are in flight and how many SMs pull weights.  A thread-block cluster of `cs`
// CTAs works on R candidates: every CTA owns a block of output columns of every layer, splits the inputs of a column
// into MLP_PARTS parts that run side by side (each with all of its 16-byte weight loads in flight), adds the parts in
// order and writes its outputs into the shared memory of all CTAs of the cluster.  The order of the sums is the same
// whatever R and cs are, so results do not depend on the batch.
// Measured: a chunk of one environment with the 3 x 256 base and the 64-wide drafter, K = 4, takes 0.88 ms; 2.08 ms with one
// block of 256 threads per latent, one serial sum per thread (40 us per base forward, 8 us and a draft-step launch per
// drafted step).
#pragma once
#include "common.cuh"
#include "gemm_tcgen05.cuh"

namespace tsdp {

constexpr int MLP_MAX_LAYERS = 8;
constexpr int MLP_THREADS = 512;
constexpr int MLP_PARTS = 16;          // parts of an output's sum over its inputs
constexpr int MLP_COLS = 256;          // output columns of a CTA per pass
constexpr int MLP_MAX_SMEM = 200 * 1024;
struct MlpWeights {
  int n_lin;                 // hidden layers + 1
  int dims[MLP_MAX_LAYERS + 2];
  const float* W[MLP_MAX_LAYERS + 1];
  const float* b[MLP_MAX_LAYERS + 1];
  int temb;
  const float* temb_table;   // [T, temb]
};
__host__ __device__ inline int mlp_max_width(const MlpWeights& w) {
  int m = 0;
  for (int l = 0; l <= w.n_lin; ++l) m = w.dims[l] > m ? w.dims[l] : m;
  return m;
}
// activations (two buffers of R rows) and the partial sums
__host__ __device__ inline size_t mlp_smem_bytes(int max_width, int R) {
  return ((size_t)2 * R * ((max_width + 3) & ~3) + (size_t)MLP_PARTS * R * MLP_COLS) * sizeof(float);
}

__device__ __forceinline__ void mlp_sync(int cs) {
  if (cs > 1) ptx::cluster_sync_all(); else __syncthreads();
}

// One layer for R rows: nxt[r][j] = act(b[j] + sum_i cur[r][i] W[i][j]), this CTA's columns, into every CTA of the cluster.
template <int R>
__device__ __forceinline__ void mlp_layer(const float* __restrict__ W, const float* __restrict__ b, int nin, int nout, bool hidden,
                                          const float* cur, float* nxt, int ld, float* part, int cs, int rank) {
  const int quads = (nout + 3) >> 2, per = (quads + cs - 1) / cs;        // columns in groups of four
  const int q_end = min(quads, (rank + 1) * per);
  const bool vec = (nout & 3) == 0;                                      // rows of W start on 16-byte boundaries
  const int chunk = (nin + MLP_PARTS - 1) / MLP_PARTS;
  for (int q0 = rank * per; q0 < q_end; q0 += MLP_COLS / 4) {
    const int nq = min(MLP_COLS / 4, q_end - q0);
    for (int u = threadIdx.x; u < nq * MLP_PARTS; u += MLP_THREADS) {
      const int q = u % nq, p = u / nq, col = 4 * (q0 + q);
      const int i0 = p * chunk, i1 = min(nin, i0 + chunk);
      float4 acc[R];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
      const float* wp = W + col;
      auto step = [&](int i, const float4& w) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float x = cur[r * ld + i];
          acc[r].x = __fmaf_rn(x, w.x, acc[r].x); acc[r].y = __fmaf_rn(x, w.y, acc[r].y);
          acc[r].z = __fmaf_rn(x, w.z, acc[r].z); acc[r].w = __fmaf_rn(x, w.w, acc[r].w);
        }
      };
      if (vec) {
        int i = i0;
        for (; i + 8 <= i1; i += 8) {
          float4 w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) w[j] = __ldg(reinterpret_cast<const float4*>(wp + (size_t)(i + j) * nout));
#pragma unroll
          for (int j = 0; j < 8; ++j) step(i + j, w[j]);
        }
        for (; i < i1; ++i) step(i, __ldg(reinterpret_cast<const float4*>(wp + (size_t)i * nout)));
      } else {
        for (int i = i0; i < i1; ++i) {
          const float* wr = wp + (size_t)i * nout;
          step(i, make_float4(__ldg(wr), col + 1 < nout ? __ldg(wr + 1) : 0.f, col + 2 < nout ? __ldg(wr + 2) : 0.f,
                              col + 3 < nout ? __ldg(wr + 3) : 0.f));
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) *reinterpret_cast<float4*>(part + ((size_t)p * R + r) * MLP_COLS + 4 * q) = acc[r];
    }
    __syncthreads();
    for (int o = threadIdx.x; o < R * 4 * nq; o += MLP_THREADS) {
      const int r = o / (4 * nq), c = o % (4 * nq), col = 4 * q0 + c;
      if (col >= nout) continue;
      float v = b[col];
#pragma unroll
      for (int p = 0; p < MLP_PARTS; ++p) v += part[((size_t)p * R + r) * MLP_COLS + c];
      if (hidden) v = silu(v);
      float* d = nxt + r * ld + col;
      if (cs == 1) *d = v;
      else {
        const uint32_t a = ptx::smem_u32(d);
        for (int k = 0; k < cs; ++k)
          asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ptx::mapa_rank(a, (uint32_t)k)), "f"(v) : "memory");
      }
    }
    if (q0 + MLP_COLS / 4 < q_end) __syncthreads();                      // the partial sums are written again
  }
  mlp_sync(cs);
}

// Input row r of the network: [latent (latent(i)) | time embedding | observation].
template <typename F>
__device__ __forceinline__ void mlp_input(const MlpWeights& w, float* row, int D, int tau, const float* __restrict__ obs, F latent) {
  for (int i = threadIdx.x; i < w.dims[0]; i += MLP_THREADS) {
    float v;
    if (i < D) v = latent(i);
    else if (i < D + w.temb) v = w.temb_table[tau * w.temb + (i - D)];
    else v = obs[i - D - w.temb];
    row[i] = v;
  }
}

// All layers for the R input rows in buf[0]; returns the buffer that holds the outputs.
template <int R>
__device__ __forceinline__ float* mlp_forward_rows(const MlpWeights& w, float* buf0, float* buf1, int ld, float* part, int cs, int rank) {
  mlp_sync(cs);            // the inputs are complete, and in a cluster nobody still reads a buffer that a peer writes into
  float *cur = buf0, *nxt = buf1;
  for (int l = 0; l < w.n_lin; ++l) {
    mlp_layer<R>(w.W[l], w.b[l], w.dims[l], w.dims[l + 1], l + 1 < w.n_lin, cur, nxt, ld, part, cs, rank);
    float* tmp = cur; cur = nxt; nxt = tmp;
  }
  return cur;
}

template <int R>
__global__ void __launch_bounds__(MLP_THREADS)
mlp_forward_kernel(const __grid_constant__ MlpWeights w, CandMap cm, const float* __restrict__ obs, int obs_len, int D, int Tsteps,
                   int n_static, int cs) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) float mlp_sm[];
  const int rank = blockIdx.x % cs, n0 = (blockIdx.x / cs) * R;
  const int count = cand_count(cm, n_static);
  if (n0 >= count) return;                                   // the same for every CTA of the cluster
  const int ld = (mlp_max_width(w) + 3) & ~3;
  float *buf0 = mlp_sm, *buf1 = buf0 + R * ld, *part = buf1 + R * ld;
  for (int r = 0; r < R; ++r) {
    int b, c;
    cand_decode(cm, min(n0 + r, count - 1), b, c);
    const int tau = max(0, min(Tsteps - 1, cm.t[b] - cm.koff - c));
    const float* x = cm.xin + b * cm.x_stride_b + (long long)c * D;
    mlp_input(w, buf0 + r * ld, D, tau, obs + (size_t)item_of(cm.item, b) * obs_len, [&](int i) { return x[i]; });
  }
  const float* res = mlp_forward_rows<R>(w, buf0, buf1, ld, part, cs, rank);
  if (rank != 0) return;
  for (int r = 0; r < R && n0 + r < count; ++r) {
    int b, c;
    cand_decode(cm, n0 + r, b, c);
    float* o = cm.eout + b * cm.e_stride_b + (long long)c * D;
    for (int i = threadIdx.x; i < D; i += MLP_THREADS) o[i] = res[r * ld + i];
  }
}

// The whole K-step draft rollout of R slots (Sec. 3.2, Eq. (3)) in one launch: forward, posterior mean, noise, next
// latent; the arithmetic of mlp_forward_kernel and draft_step_kernel (the same device functions).  Steps beyond a
// slot's window carry the latent along, as draft_step_kernel does.
template <int R>
__global__ void __launch_bounds__(MLP_THREADS)
mlp_rollout_kernel(const __grid_constant__ MlpWeights w, DdpmTables S, float* __restrict__ xt, long long xs_b, float* __restrict__ muhat,
                   long long ms_b, const int* t, const uint64_t* __restrict__ seedp, const EnvParams* envp,
                   const int* item, const float* __restrict__ obs, int obs_len, int D, int B, int K, int Tsteps, int cs) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) float mlp_sm[];
  const int rank = blockIdx.x % cs, b0 = (blockIdx.x / cs) * R;
  const int ld = (mlp_max_width(w) + 3) & ~3;
  float *buf0 = mlp_sm, *buf1 = buf0 + R * ld, *part = buf1 + R * ld, *sx = part + MLP_PARTS * R * MLP_COLS;      // sx [R][D]
  const uint64_t seed = *seedp;
  int tb[R], env[R], ke[R], ke_max = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int b = min(b0 + r, B - 1);
    tb[r] = b0 + r < B ? t[b] : -1;
    env[r] = item_of(item, b);
    ke[r] = tb[r] >= 0 ? min(env_draft_cap(envp, env[r], tb[r], K, Tsteps), tb[r]) : 0;
    ke_max = max(ke_max, ke[r]);
    for (int i = threadIdx.x; i < D; i += MLP_THREADS) sx[r * D + i] = xt[b * xs_b + i];
  }
  __syncthreads();
  const int nq = (D + 3) >> 2;
  for (int k = 1; k <= K; ++k) {
    const float* res = nullptr;
    if (k <= ke_max) {                                       // the same for every CTA of the cluster
#pragma unroll
      for (int r = 0; r < R; ++r)
        mlp_input(w, buf0 + r * ld, D, max(0, tb[r] - k + 1), obs + (size_t)env[r] * obs_len, [&](int i) { return sx[r * D + i]; });
      res = mlp_forward_rows<R>(w, buf0, buf1, ld, part, cs, rank);
    }
    for (int u = threadIdx.x; u < R * nq; u += MLP_THREADS) {
      const int r = u / nq, q = u - r * nq;
      int tbr = 0, envr = 0, ker = 0;
#pragma unroll
      for (int s = 0; s < R; ++s) if (s == r) { tbr = tb[s]; envr = env[s]; ker = ke[s]; }
      const bool valid = k <= ker;
      const int tau = tbr - k + 1;
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      if (valid) normal4(seed, (uint32_t)envr, STREAM_XI, (uint32_t)tau, (uint32_t)q, z);
      float* xg = xt + (b0 + r) * xs_b + (long long)k * D;
      float* mg = muhat + (b0 + r) * ms_b + (long long)(k - 1) * D;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = 4 * q + j;
        if (i >= D) break;
        const float x = sx[r * D + i];
        float m = x, xn = x;
        if (valid) {
          m = posterior_mean(S, x, res[r * ld + i], tau);
          xn = ddpm_sample(m, S.sigma[tau], z[j]);
          sx[r * D + i] = xn;
        }
        if (rank == 0 && b0 + r < B) { mg[i] = m; xg[i] = xn; }
      }
    }
    __syncthreads();
  }
  if (cs > 1) ptx::cluster_sync_all();       // nobody leaves while a peer may still write into its shared memory
}

}  // namespace tsdp
