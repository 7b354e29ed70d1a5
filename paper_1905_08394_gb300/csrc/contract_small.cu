// K4 + K5 + K6 for small lattices in one persistent launch: every column
// absorption of one bitstring's sweep (supplementary "exact computation of
// the overlap", the generic scheme transposed to columns) runs inside one
// block, with the running tensor held in shared memory from the scalar 1 to
// the final 1 x 1 tensor.  Blocks walk the bitstrings (block b takes
// b, b + gridDim.x, ...), so a call is one launch whatever the number of
// bitstrings and steps.
//
// Step s: out[M x N] = in[M x K] * Ec[K x N] in complex FP32 with the same
// permute-fused store as the step-by-step kernels (row m = m_hi (M / P) +
// m_lo, column n = h' dv' + v' goes to ((m_lo dh' + h') P + m_hi) dv' + v'),
// and the same power-of-two renormalisation: the output is multiplied by 2^x
// with x from the input's max |entry| and the operand's column bound, so that
// it stays at most 1; the exponents add up exactly and the amplitude is
// m 2^-S in FP64, added to the call's accumulator (a sum over slices when the
// call has several).
#include "common.h"
#include "format.cuh"

namespace peps {

namespace {

constexpr int SW_THREADS = 256;
constexpr int kPre = 4;   // operand entries per thread loaded a step ahead

// A thread computes rt x ct outputs (rows M / rt apart, neighbouring columns):
// one output per thread reads two entries from shared memory per
// multiply-add, which bound the sweep (5x5 (1+16+1), 1024 bitstrings: 495 us, 10.7
// TFLOP/s; 251 us so).  Running tensors are read down k by lanes of neighbouring
// rows, K entries apart: entry i lies at swz(i), which spreads those over the
// banks for every power-of-two K.
__device__ __forceinline__ int swz(int i) { return (i & ~15) | ((i ^ (i >> 4) ^ (i >> 6)) & 15); }

template <int RT, int CT>
__device__ __forceinline__ float small_tiles(const SmallStep &st, const float2 *__restrict__ in,
                                             float2 *__restrict__ out,
                                             const float2 *__restrict__ E, float sc, int tid) {
  const int M = (int)st.sh.M, K = st.sh.K, N = st.sh.N, P = (int)st.sh.P;
  const int rows = M / RT, tn = (int)st.d_tn.d, T = rows * tn;
  const int dv = st.sh.dv_out, dh = st.sh.dh_out;
  float vmax = 0.f;
  for (int t = tid; t < T; t += SW_THREADS) {
    const int mt = (int)st.d_tn.q(t), n0 = (t - mt * tn) * CT;
    float re[RT][CT], im[RT][CT];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int c = 0; c < CT; ++c) re[i][c] = im[i][c] = 0.f;
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      float2 w[CT];
      if (CT == 4) {
        const float4 w0 = *reinterpret_cast<const float4 *>(E + k * N + n0);
        const float4 w1 = *reinterpret_cast<const float4 *>(E + k * N + n0 + 2);
        w[0] = make_float2(w0.x, w0.y);
        w[1 % CT] = make_float2(w0.z, w0.w);
        w[2 % CT] = make_float2(w1.x, w1.y);
        w[3 % CT] = make_float2(w1.z, w1.w);
      } else {
#pragma unroll
        for (int c = 0; c < CT; ++c) w[c] = E[k * N + n0 + c];
      }
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const float2 u = in[swz((mt + i * rows) * K + k)];
#pragma unroll
        for (int c = 0; c < CT; ++c) {
          re[i][c] = fmaf(u.x, w[c].x, re[i][c]);
          re[i][c] = fmaf(-u.y, w[c].y, re[i][c]);
          im[i][c] = fmaf(u.x, w[c].y, im[i][c]);
          im[i][c] = fmaf(u.y, w[c].x, im[i][c]);
        }
      }
    }
    const int q0 = (int)st.d_R.q(n0), r0 = n0 - q0 * st.R;
    const int col = q0 * st.stride_q + r0 * st.stride_r;
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int m = mt + i * rows;
      const int m_hi = (int)st.d_Mlo.q(m), m_lo = m - m_hi * (int)st.d_Mlo.d;
      int dest = (m_lo * dh * P + m_hi) * dv + col, r = r0;
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        const float x = re[i][c] * sc, y = im[i][c] * sc;
        out[swz(dest)] = make_float2(x, y);
        vmax = fmaxf(vmax, fmaxf(fabsf(x), fabsf(y)));
        dest += st.stride_r;
        if (++r == st.R) {
          r = 0;
          dest += st.stride_q - st.R * st.stride_r;
        }
      }
    }
  }
  return vmax;
}

__global__ void __launch_bounds__(SW_THREADS) k_sweep_small(const SmallSweep p) {
  extern __shared__ __align__(16) float2 sm[];
  float2 *const E = sm;
  float2 *const buf0 = sm + ((p.cap_e + 1) & ~1);
  float2 *const buf1 = buf0 + ((p.cap_g + 15) & ~15);
  __shared__ float red[SW_THREADS / 32];
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int64_t i = blockIdx.x; i < p.n; i += gridDim.x) {
    const uint64_t bits = p.bits[i];
    float2 *in = buf0, *out = buf1;
    if (tid == 0) in[0] = make_float2(1.f, 0.f);
    float mu = 1.f;   // max |entry| of the stored input
    int S = 0;        // stored G = true G * 2^S
    // the step's operand: its first kPre 256 entries are loaded a step ahead
    float2 pre[kPre];
    const float2 *Ec = nullptr;
    int kn = 0;
    float beta = 0.f;
    auto fetch = [&](int s) {
      const StepShape &sh = p.steps[s].sh;
      const OpDesc &op = p.ops[p.op_base[s] + block_variant(bits, sh)];
      Ec = op.Ec;
      kn = sh.K * sh.N;
      beta = __uint_as_float(op.beta_c_bits);
#pragma unroll
      for (int j = 0; j < kPre; ++j)
        if (tid + j * SW_THREADS < kn) pre[j] = Ec[tid + j * SW_THREADS];
    };
    fetch(0);
    for (int s = 0; s < p.n_steps; ++s) {
      const SmallStep &st = p.steps[s];
#pragma unroll
      for (int j = 0; j < kPre; ++j)
        if (tid + j * SW_THREADS < kn) E[tid + j * SW_THREADS] = pre[j];
      for (int e = tid + kPre * SW_THREADS; e < kn; e += SW_THREADS) E[e] = Ec[e];
      const int x = step_scale_exp(mu, beta, 0);
      const float sc = pow2f(x);
      __syncthreads();   // E loaded; the previous step's output complete
      if (s + 1 < p.n_steps) fetch(s + 1);
      float vmax;
      if (st.ct == 4) {
        if (st.rt == 4) vmax = small_tiles<4, 4>(st, in, out, E, sc, tid);
        else if (st.rt == 2) vmax = small_tiles<2, 4>(st, in, out, E, sc, tid);
        else vmax = small_tiles<1, 4>(st, in, out, E, sc, tid);
      } else {
        if (st.rt == 4) vmax = small_tiles<4, 1>(st, in, out, E, sc, tid);
        else vmax = small_tiles<1, 1>(st, in, out, E, sc, tid);
      }
      const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
      if (lane == 0) red[warp] = __uint_as_float(mx);
      __syncthreads();   // output and partial maxima complete; E free
      vmax = red[0];
#pragma unroll
      for (int w = 1; w < SW_THREADS / 32; ++w) vmax = fmaxf(vmax, red[w]);
      mu = vmax;
      S += x;
      float2 *t = in;
      in = out;
      out = t;
    }
    if (tid == 0) {
      const float2 g = in[0];
      double2 a = p.acc[i];
      a.x += ldexp((double)g.x, -S);
      a.y += ldexp((double)g.y, -S);
      p.acc[i] = a;
    }
    __syncthreads();   // red and the buffers are reused by the next bitstring
  }
}

}  // namespace

size_t small_sweep_smem(int cap_g, int cap_e) {
  const int g = (cap_g + 15) & ~15;   // whole blocks of 16 (swz)
  return (size_t)(2 * g + ((cap_e + 1) & ~1)) * sizeof(float2);
}

// The thread tile of a step: 4 x 4 outputs down to one, so that at least 256
// tiles are left; four columns only where N has them.
SmallStep small_step(const StepShape &sh) {
  SmallStep st{};
  st.sh = sh;
  const int64_t out = sh.M * sh.N;
  st.ct = sh.N % 4 == 0 && out >= 4 * SW_THREADS ? 4 : 1;
  st.rt = 1;
  if (sh.M % 4 == 0 && out >= 4 * st.ct * SW_THREADS) st.rt = 4;
  else if (st.ct == 4 && sh.M % 2 == 0 && out >= 2 * st.ct * SW_THREADS) st.rt = 2;
  st.d_tn = make_div(sh.N / st.ct);
  st.d_Mlo = make_div(sh.M / sh.P);
  // column n = h' dv' + v' lies h' P dv' + v' after its row's first entry
  const bool flat = sh.dv_out == 1;
  st.R = flat ? sh.N : sh.dv_out;
  st.d_R = make_div(st.R);
  st.stride_q = flat ? 0 : (int32_t)(sh.P * sh.dv_out);
  st.stride_r = flat ? (int32_t)sh.P : 1;
  return st;
}

cudaError_t launch_sweep_small(const SmallSweep &p, int sm_count, cudaStream_t s) {
  if (p.n <= 0) return cudaSuccess;
  const size_t smem = small_sweep_smem(p.cap_g, p.cap_e);
  static PerDevice allowed;   // (padding of the parts)
  const cudaError_t e = allow_smem(allowed, k_sweep_small, kSmallSweepMaxSmem + 512);
  if (e != cudaSuccess) return e;
  if (smem > kSmallSweepMaxSmem + 512) return cudaErrorInvalidValue;
  // blocks resident per SM (about 220 KiB of shared memory), at most 4
  const int per_sm = (int)((220u * 1024u) / (smem > 0 ? smem : 1));
  int64_t blocks = (int64_t)sm_count * (per_sm < 1 ? 1 : (per_sm > 4 ? 4 : per_sm));
  if (blocks > p.n) blocks = p.n;
  return launch_dependent(k_sweep_small, dim3((unsigned)blocks), dim3(SW_THREADS), smem, s, p);
}

}  // namespace peps
