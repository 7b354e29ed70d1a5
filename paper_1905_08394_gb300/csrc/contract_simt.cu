// K4 (CUDA-core form): one site absorption of the column sweep for a batch
// of lanes,
//   G'[rest, h'_r, v'] = sum_{h_r, v} G[rest, h_r, v] * E[h_r, v, h'_r, v']
// (supplementary "exact computation of the overlap", the absorption of one
// tensor into the running tensor, transposed to sweep columns).  As a matrix
// product: out[M x N] = G[M x K] * Ec[K x N] in complex FP32, with
//   M = product of the untouched h legs (slowest leg P first),
//   K = dim(h_r) * dim(v), N = dim(h'_r) * dim(v').
// The store is permute-fused: row m = b * Mr + m_hi * (Mr / P) + m_lo, column
// n = h' * dv' + v' goes to b Mr N + ((m_lo * dh' + h') * P + m_hi) * dv' + v'
// (StepShape::Mr gives the open-leg form), which moves the slowest untouched
// leg next to v' so that the next step's contracted legs are again the two
// fastest.
//
// Every output is multiplied by the step's power-of-two scale 2^x (exact), and
// the block's max |stored entry| goes to the lane's record for the next step.
//
// A block takes rows in the order of their destinations (m_hi fastest), one
// row per lane, so that a warp's stores are contiguous whatever P and dv' are;
// the input rows are then gathered, K entries (a whole sector or more) each.  It
// walks several row tiles of its item with the next pass's loads in flight, so
// that the chain item -> bitstring -> operand -> data is paid once.  A thread
// holds RT rows x CT neighbouring columns; products are formed two columns at a
// time with packed FP32 multiply-adds, each half the same chain of IEEE
// operations as a scalar one (re += a.x b.x, re += a.y (-b.y); im += a.x b.y, im
// += a.y b.x, k ascending).  The packed form halves the issue slots: with
// distinct operands it reaches 60 TFLOP/s on its own, and this kernel is 14 %
// faster with it than with scalar multiply-adds.  Large K is bound by that rate,
// small K by memory, launches of few tiles by latency.  The 4 x 8 tiles (42 to
// 51 TFLOP/s on the square partition's large steps at 64 lanes) keep 64 sums per
// thread: at the 128 registers that two blocks per SM leave, ptxas spills 92 to
// 204 bytes a thread, and the operand lies in three planes in shared memory (b.y
// and -b.y both).  What either costs has not been measured apart; the 2 x 8 tile
// with K passes of 16, which spills nothing, reaches 47.
#include "common.h"
#include "format.cuh"

namespace peps {

namespace {

constexpr int THREADS = 256;

struct SimtParams {
  StepShape sh;
  Div d_P, d_Mlo, d_R;     // rows in destination order, columns (run length)
  uint32_t R;              // columns per run (dv', or dh' / N; see below)
  int32_t W;               // entries per store: 8 or 4 (contiguous runs), or 1
  int32_t vec;             // 1: K is a multiple of 4 (16-byte loads)
  int32_t wide;            // 1: buffers 32-byte aligned
  int64_t stride_q, stride_r;   // of a run, of a column within it
  int64_t row_b, row_lo, row_hi;  // of b, m_lo, m_hi
  int64_t Mlo;             // input rows from one m_hi to the next
};

// two FP32 lanes of one multiply-add
__device__ __forceinline__ void fma2(unsigned long long &c, unsigned long long a,
                                     unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// C pairs of neighbouring floats from shared memory, 16 bytes at a time.
template <int C>
__device__ __forceinline__ void load_pairs(const float *s, unsigned long long (&v)[C]) {
  if (C % 2 == 0) {
#pragma unroll
    for (int c = 0; c + 1 < C; c += 2) {
      const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(s + 2 * c);
      v[c] = w.x;
      v[c + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = *reinterpret_cast<const unsigned long long *>(s + 2 * c);
  }
}

// Four entries e .. e+3 of G (e % 4 == 0): raw words, then values.
struct Raw4 {
  uint4 w[2];
};
template <int FMT>
__device__ __forceinline__ void load4_raw(const void *base, int64_t e, int64_t plane, Raw4 &r) {
  if (FMT == FMT_F32 || FMT == FMT_TF32) {
    const uint4 *s = reinterpret_cast<const uint4 *>(reinterpret_cast<const float2 *>(base) + e);
    r.w[0] = s[0];
    r.w[1] = s[1];
  } else {
    const uint32_t *p = reinterpret_cast<const uint32_t *>(base);
    r.w[0] = *reinterpret_cast<const uint4 *>(p + e);
    if (FMT == FMT_BF16X2 || FMT == FMT_FP16X2)
      r.w[1] = *reinterpret_cast<const uint4 *>(p + plane / 2 + e);
  }
}
// The first n (< 4, or 4) of them one by one, the rest left as they are.
template <int FMT>
__device__ __forceinline__ void load4_some(const void *base, int64_t e, int64_t plane, int n,
                                           Raw4 &r) {
  uint32_t *w = reinterpret_cast<uint32_t *>(r.w);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (j >= n) continue;
    if (FMT == FMT_F32 || FMT == FMT_TF32) {
      const uint2 v = reinterpret_cast<const uint2 *>(base)[e + j];
      w[2 * j] = v.x;
      w[2 * j + 1] = v.y;
    } else {
      w[j] = reinterpret_cast<const uint32_t *>(base)[e + j];
      if (FMT == FMT_BF16X2 || FMT == FMT_FP16X2)
        w[4 + j] = reinterpret_cast<const uint32_t *>(base)[plane / 2 + e + j];
    }
  }
}
template <int FMT>
__device__ __forceinline__ void unpack4(const Raw4 &r, float2 (&f)[4]) {
  const uint32_t *w = reinterpret_cast<const uint32_t *>(r.w);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (FMT == FMT_F32 || FMT == FMT_TF32) {
      f[j] = make_float2(__uint_as_float(w[2 * j]), __uint_as_float(w[2 * j + 1]));
    } else {
      constexpr bool BF = FMT == FMT_BF16 || FMT == FMT_BF16X2;
      f[j] = BF ? unpack_bf16(w[j]) : unpack_f16(w[j]);
      if (FMT == FMT_BF16X2 || FMT == FMT_FP16X2) {
        const float2 l = BF ? unpack_bf16(w[4 + j]) : unpack_f16(w[4 + j]);
        f[j] = make_float2(f[j].x + l.x, f[j].y + l.y);
      }
    }
  }
}

// (The unit scalar, the input of a sweep's first step with M = K = 1, is the
// rows kernel's.)
// RT rows (32 apart) x CT columns per thread; WN warps side by side cover the
// block's WN CT columns, the other 8 / WN its rows; BK entries of K per pass.
template <int FMT, int RT, int CT, int WN, int BK>
__global__ void __launch_bounds__(THREADS, RT * CT >= 16 ? 2 : 3)
k_contract_simt(const __grid_constant__ SimtParams p, const StepItem *__restrict__ items,
                const OpDesc *__restrict__ ops, Rec *__restrict__ recs) {
  constexpr int WM = 8 / WN, ROWS = WM * 32 * RT, COLS = WN * CT;
  constexpr int LDA = BK + 2;                         // padded row of A (entries)
  constexpr int GA = ROWS * BK / 4 / THREADS;         // groups of 4 entries of A per thread
  constexpr int GB = (BK * COLS + THREADS - 1) / THREADS;  // entries of B per thread
  static_assert(GA >= 1 && GA * 4 * THREADS == ROWS * BK, "A tile and threads");
  extern __shared__ __align__(16) float simt_sm[];
  float2 *As = reinterpret_cast<float2 *>(simt_sm);                      // [2][ROWS][LDA]
  float *Bs = reinterpret_cast<float *>(As + 2 * ROWS * LDA);            // [2][3][BK][COLS]

  pdl_trigger();
  const StepItem it = items[blockIdx.z];
  const OpDesc &op = ops[it.op_base + block_variant(*it.bits, p.sh)];
  pdl_wait();
  const float2 *__restrict__ Ec = op.Ec;
  const int64_t M = p.sh.M;
  const int K = p.sh.K, N = p.sh.N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wn = warp % WN, wm = warp / WN;
  const int n0 = blockIdx.y * COLS;
  const int64_t Mr = p.sh.Mr > 0 ? p.sh.Mr : M;
  const int tiles = (int)((M + ROWS - 1) / ROWS);   // at most 2^31 - 1
  const bool narrow = M < 0x7fffff00LL;   // 32-bit row arithmetic
  // the step's scale (the records and the bound are loaded ahead of their use)
  const float mu = __uint_as_float(recs[it.in_rec].maxbits);
  const int s_in = recs[it.in_rec].exp;
  const float beta = __uint_as_float(op.beta_c_bits);

  // destination-order row s -> b, m_lo, m_hi
  auto split_row = [&](int64_t s, int64_t &b, int64_t &m_lo, int64_t &m_hi) {
    if (narrow) {
      const uint32_t t = p.d_P.q((uint32_t)s), bb = p.d_Mlo.q(t);
      m_hi = (uint32_t)s - t * p.d_P.d;
      m_lo = t - bb * p.d_Mlo.d;
      b = bb;
    } else {
      const int64_t P = p.sh.P, Mlo = Mr / P;
      const int64_t t = s / P;
      m_hi = s - t * P;
      b = t / Mlo;
      m_lo = t - b * Mlo;
    }
  };

  // A: group g is row (tid + 256 g) / (BK / 4) of the tile, entries 4 kq .. 4 kq + 3
  const int kq = tid % (BK / 4);
  int64_t a_off[GA];   // the row's first entry, -1 past the end
  Raw4 ra[GA];
  float2 rb[GB];
  auto rows_of = [&](int tile) {
#pragma unroll
    for (int g = 0; g < GA; ++g) {
      const int64_t s = (int64_t)tile * ROWS + (tid + THREADS * g) / (BK / 4);
      a_off[g] = -1;
      if (s < M) {
        int64_t b, lo, hi;
        split_row(s, b, lo, hi);
        a_off[g] = (b * Mr + hi * p.Mlo + lo) * K;
      }
    }
  };
  auto fetch = [&](int k0, bool with_b) {
#pragma unroll
    for (int g = 0; g < GA; ++g) {
      const int k = k0 + 4 * kq;
      ra[g].w[0] = ra[g].w[1] = make_uint4(0u, 0u, 0u, 0u);
      if (a_off[g] >= 0 && k < K) {
        if (p.vec) load4_raw<FMT>(it.A, a_off[g] + k, p.sh.plane, ra[g]);
        else load4_some<FMT>(it.A, a_off[g] + k, p.sh.plane, K - k, ra[g]);
      }
    }
    if (with_b) {
#pragma unroll
      for (int g = 0; g < GB; ++g) {
        const int e = tid + THREADS * g, k = k0 + e / COLS, n = n0 + e % COLS;
        rb[g] = (e < BK * COLS && k < K && n < N) ? Ec[(int64_t)k * N + n] : make_float2(0.f, 0.f);
      }
    }
  };
  auto put = [&](int buf, bool with_b) {
#pragma unroll
    for (int g = 0; g < GA; ++g) {
      const int row = (tid + THREADS * g) / (BK / 4);
      float2 f[4];
      unpack4<FMT>(ra[g], f);
      float4 *d = reinterpret_cast<float4 *>(As + (buf * ROWS + row) * LDA + 4 * kq);
      d[0] = make_float4(f[0].x, f[0].y, f[1].x, f[1].y);
      d[1] = make_float4(f[2].x, f[2].y, f[3].x, f[3].y);
    }
    if (with_b) {
#pragma unroll
      for (int g = 0; g < GB; ++g) {
        const int e = tid + THREADS * g;
        if (e < BK * COLS) {
          float *d = Bs + buf * 3 * BK * COLS + e;
          d[0] = rb[g].x;
          d[BK * COLS] = rb[g].y;
          d[2 * BK * COLS] = -rb[g].y;
        }
      }
    }
  };

  unsigned long long re[RT][CT / 2], im[RT][CT / 2];   // columns 2c, 2c + 1
  const int nk = (K + BK - 1) / BK;
  const int nc = n0 + wn * CT;
  // column nc: run q, place r in it; entry = row + q stride_q + r stride_r
  const uint32_t q0 = p.d_R.q((uint32_t)nc), r0 = (uint32_t)nc - q0 * p.R;
  const int64_t col = q0 * p.stride_q + r0 * p.stride_r;
  float vmax = 0.f;
  rows_of(blockIdx.x);
  fetch(0, true);
  put(0, true);
  const int x = step_scale_exp(mu, beta, p.sh.target);
  const float sc = pow2f(x);
  __syncthreads();
  // passes (tile, t) in order; pass i's data is in buffer i & 1.  With one pass
  // per tile the operand stays in buffer 0.
  int cur = 0;
  for (int tile = blockIdx.x;; tile += gridDim.x) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int c = 0; c < CT / 2; ++c) re[i][c] = im[i][c] = 0ull;
    for (int t = 0; t < nk; ++t) {
      const bool last = t + 1 == nk, more = !last || tiles - tile > (int)gridDim.x;
      if (more) {
        if (last) rows_of(tile + gridDim.x);
        fetch(last ? 0 : (t + 1) * BK, nk > 1);
      }
      const int kmax = K - t * BK;
      const float2 *a = As + (cur * ROWS + wm * 32 * RT + lane) * LDA;
      const float *b = Bs + (nk > 1 ? cur : 0) * 3 * BK * COLS + wn * CT;
#pragma unroll
      for (int kk = 0; kk < BK; kk += 2) {
        if (kk % 4 == 0 && kk > 0 && kk >= kmax) break;   // the rest are zeros
        float4 av[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) av[i] = *reinterpret_cast<const float4 *>(a + 32 * i * LDA + kk);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          unsigned long long bx[CT / 2], by[CT / 2], bn[CT / 2];
          load_pairs<CT / 2>(b + (kk + h) * COLS, bx);
          load_pairs<CT / 2>(b + (BK + kk + h) * COLS, by);
          load_pairs<CT / 2>(b + (2 * BK + kk + h) * COLS, bn);
#pragma unroll
          for (int i = 0; i < RT; ++i) {
            const float ax = h ? av[i].z : av[i].x, ay = h ? av[i].w : av[i].y;
            const unsigned long long xx = pack2(ax, ax), yy = pack2(ay, ay);
#pragma unroll
            for (int c = 0; c < CT / 2; ++c) {
              fma2(re[i][c], xx, bx[c]);
              fma2(im[i][c], xx, by[c]);
            }
#pragma unroll
            for (int c = 0; c < CT / 2; ++c) {
              fma2(re[i][c], yy, bn[c]);
              fma2(im[i][c], yy, bx[c]);
            }
          }
        }
      }
      if (more) put(cur ^ 1, nk > 1);
      cur ^= 1;
      if (last) {
        // scale, permuted store, max
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const int64_t s = (int64_t)tile * ROWS + (wm * RT + i) * 32 + lane;
          if (s >= M || nc >= N) continue;
          int64_t b_, lo, hi;
          split_row(s, b_, lo, hi);
          int64_t dest = b_ * p.row_b + lo * p.row_lo + hi * p.row_hi + col;
          float o[16];
#pragma unroll
          for (int c = 0; c < CT / 2; ++c) {
            const float2 xr = unpack2(re[i][c]), xi = unpack2(im[i][c]);
            o[4 * c] = xr.x;
            o[4 * c + 1] = xi.x;
            o[4 * c + 2] = xr.y;
            o[4 * c + 3] = xi.y;
          }
          if (CT == 8 && p.W >= 4) {   // runs of 8 or 4 (N is a multiple of 4)
            if (p.W == 8 || nc + 8 <= N) {
              Packed8<FMT> w;
              vmax = fmaxf(vmax, pack8<FMT>(o, sc, w));
              if (p.W == 8) {
                if (p.wide) store_run8_wide<FMT>(it.D, dest, p.sh.plane, w);
                else store_run<FMT, 8>(it.D, dest, p.sh.plane, w, 0);
              } else {
                store_run<FMT, 4>(it.D, dest, p.sh.plane, w, 0);
                dest += 4;
                if (r0 + 4 == p.R) dest += p.stride_q - p.R;
                store_run<FMT, 4>(it.D, dest, p.sh.plane, w, 4);
              }
              continue;
            }
          }
          uint32_t r = r0;
#pragma unroll
          for (int j = 0; j < CT; ++j) {
            if (nc + j >= N) continue;
            const float2 v = make_float2(o[2 * j] * sc, o[2 * j + 1] * sc);
            store_g<FMT>(it.D, dest, p.sh.plane, v);
            vmax = fmaxf(vmax, max_abs2(v));
            dest += p.stride_r;
            if (++r == p.R) {
              r = 0;
              dest += p.stride_q - (int64_t)p.R * p.stride_r;
            }
          }
        }
      }
      __syncthreads();
    }
    if (tiles - tile <= (int)gridDim.x) break;
  }
  const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
  if (lane == 0) atomicMax(&recs[it.out_rec].maxbits, mx);
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) recs[it.out_rec].exp = s_in + x + op.e_c;
}

// The same step for a running tensor of at most a few rows (the first steps
// of a sweep, M = 1 .. 8): one thread per output entry, no tiling.
template <int FMT>
__global__ void __launch_bounds__(256)
k_contract_rows(const StepShape sh, const StepItem *__restrict__ items,
                const OpDesc *__restrict__ ops, Rec *__restrict__ recs) {
  pdl_trigger();
  const StepItem it = items[blockIdx.y];
  const uint64_t bits = *it.bits;
  const OpDesc &op = ops[it.op_base + block_variant(bits, sh)];
  pdl_wait();
  const int M = (int)sh.M, K = sh.K, N = sh.N;
  const bool unit_in = it.in_rec < 0;
  const float mu = unit_in ? 1.f : __uint_as_float(recs[it.in_rec].maxbits);
  const int s_in = unit_in ? 0 : recs[it.in_rec].exp;
  const int x = step_scale_exp(mu, __uint_as_float(op.beta_c_bits), sh.target);
  const float sc = pow2f(x);
  const int64_t Mr = sh.Mr > 0 ? sh.Mr : sh.M;
  const bool batched = Mr != sh.M;
  const int64_t Mlo = Mr / sh.P;
  const int dv = sh.dv_out, dh = sh.dh_out;
  float vmax = 0.f;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < M * N) {
    const int m = e / N, n = e - m * N;
    float re = 0.f, im = 0.f;
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
      float2 a;
      if (unit_in) a = (m == 0 && k == 0) ? make_float2(1.f, 0.f) : make_float2(0.f, 0.f);
      else a = load_g<FMT>(it.A, (int64_t)m * K + k, sh.plane);
      const float2 w = op.Ec[(int64_t)k * N + n];
      re = fmaf(a.x, w.x, fmaf(-a.y, w.y, re));
      im = fmaf(a.x, w.y, fmaf(a.y, w.x, im));
    }
    const int64_t b = batched ? m / Mr : 0, mr = m - b * Mr;
    const int64_t m_hi = mr / Mlo, m_lo = mr - m_hi * Mlo;
    const int hh = sh.nvs ? n % dh : n / dv, vv = sh.nvs ? n / dh : n % dv;
    const int64_t rot = (m_lo * dh + hh) * sh.P + m_hi;
    const int64_t dest = sh.vb ? (b * dv + vv) * (Mr * dh) + rot : b * (Mr * N) + rot * dv + vv;
    const float2 v = make_float2(re * sc, im * sc);
    store_g<FMT>(it.D, dest, sh.plane, v);
    vmax = max_abs2(v);
  }
  for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&recs[it.out_rec].maxbits, __float_as_uint(vmax));
  if (blockIdx.x == 0 && threadIdx.x == 0) recs[it.out_rec].exp = s_in + x + op.e_c;
}

template <int FMT, int RT, int CT, int WN, int BK>
cudaError_t launch_cfg(const SimtParams &p, const StepItem *items, int n_items, const OpDesc *ops,
                       Rec *recs, cudaStream_t s) {
  constexpr int ROWS = 8 / WN * 32 * RT, COLS = WN * CT;
  constexpr size_t smem = 2 * ROWS * (BK + 2) * sizeof(float2) + 2 * 3 * BK * COLS * sizeof(float);
  auto kern = k_contract_simt<FMT, RT, CT, WN, BK>;
  if (smem > 48 * 1024) {
    static PerDevice allowed;
    const cudaError_t e = allow_smem(allowed, kern, smem);
    if (e != cudaSuccess) return e;
  }
  int64_t mt = (p.sh.M + ROWS - 1) / ROWS;
  const int nt = (p.sh.N + COLS - 1) / COLS;
  if (mt > 0x7fffffffLL || nt > 65535 || n_items > 65535) return cudaErrorInvalidValue;
  // row tiles per block: as many as leave the chip about eight blocks per SM
  const int64_t per = mt * nt * (int64_t)n_items / (8 * 152);
  if (per > 1) mt = (mt + per - 1) / per;
  return launch_dependent(kern, dim3((unsigned)mt, nt, n_items), dim3(THREADS), smem, s, p, items, ops,
                          recs);
}

// The tile of a launch: 128 rows x 64 columns where that gives two waves of two
// blocks per SM, 64 x 64 down to one such wave (16 lanes of 1024 x 1024 x 256:
// 716 against 781 us; 4096 x 64 x 256: 212 against 203), 32 x 64 with long K
// passes below it; narrower and taller ones for few columns (a block reads its
// rows once: 32 lanes of 32768 x 8 x 32 on 256 x 32 tiles 157 us, on 128 x 32
// 199); and 32 x 16 for launches of few tiles, whose time is the chain of K
// passes of one block.  Against the 128 x 64 tile with rows in input order that
// this replaces (FP16X3 unless noted): 32 lanes of 32768 x 8 x 32 369 -> 108 us
// (2.9 TB/s), 32768 x 8 x 16 319 -> 58, 16384 x 4 x 64 251 -> 80; FP32, 16 lanes
// of 1024 x 1024 x 256 893 -> 728 us (47 TFLOP/s).
template <int FMT>
cudaError_t launch_tiles(const StepShape &sh, const StepItem *items, int n_items,
                         const OpDesc *ops, Rec *recs, bool aligned32, cudaStream_t s) {
  SimtParams p{};
  p.sh = sh;
  const int64_t M = sh.M, Mr = sh.Mr > 0 ? sh.Mr : M, P = sh.P, dv = sh.dv_out, dh = sh.dh_out;
  p.d_P = make_div(P < 0x7fffffffLL ? P : 1);
  p.d_Mlo = make_div(Mr / P < 0x7fffffffLL ? Mr / P : 1);
  // destination of row (b, m_lo, m_hi) and column n:
  //   vb = 0: b Mr N + ((m_lo dh + h') P + m_hi) dv + v'
  //   vb = 1: (b dv + v') Mr dh + (m_lo dh + h') P + m_hi
  // with n = h' dv + v' (nvs = 0) or v' dh + h' (nvs = 1)
  const int64_t st_h = sh.vb ? P : P * dv, st_v = sh.vb ? Mr * dh : 1;
  p.row_b = sh.vb ? dv * Mr * dh : Mr * (int64_t)sh.N;
  p.row_lo = dh * st_h;
  p.row_hi = sh.vb ? 1 : dv;
  p.R = (uint32_t)(sh.nvs ? dh : dv);
  p.stride_q = sh.nvs ? st_v : st_h;
  p.stride_r = sh.nvs ? st_h : st_v;
  if (p.R == 1) {   // one run over the other leg
    p.R = (uint32_t)sh.N;
    p.stride_r = p.stride_q;
    p.stride_q = 0;
  }
  p.d_R = make_div(p.R);
  p.W = p.stride_r != 1 ? 1 : (p.R % 8 == 0 ? 8 : (p.R % 4 == 0 ? 4 : 1));
  p.Mlo = Mr / P;
  p.vec = sh.K % 4 == 0 ? 1 : 0;
  p.wide = aligned32 ? 1 : 0;
  const int N = sh.N;
  auto tiles = [&](int rows, int cols) {
    return ((M + rows - 1) / rows) * ((N + cols - 1) / cols) * (int64_t)n_items;
  };
  const bool few_ok = N <= 16 * 65535;
#define PEPS_SIMT_CFG(...) return launch_cfg<FMT, __VA_ARGS__>(p, items, n_items, ops, recs, s)
  if (N > 32) {
    if (tiles(128, 64) >= 608 || !few_ok) PEPS_SIMT_CFG(4, 8, 8, 8);
    if (tiles(64, 64) >= 304) PEPS_SIMT_CFG(2, 8, 8, 16);
    if (tiles(32, 64) >= 100) PEPS_SIMT_CFG(1, 8, 8, 32);
  } else if (N > 16) {
    if (tiles(256, 32) >= 304) PEPS_SIMT_CFG(4, 8, 4, 8);
    if (tiles(64, 32) >= 100) PEPS_SIMT_CFG(1, 8, 4, 32);
  } else if (N > 8) {
    if (tiles(256, 16) >= 304) PEPS_SIMT_CFG(2, 8, 2, 8);
    if (tiles(128, 16) >= 100) PEPS_SIMT_CFG(1, 8, 2, 8);
  } else if (N > 4) {
    if (tiles(256, 8) >= 304) PEPS_SIMT_CFG(1, 8, 1, 8);
  } else if (tiles(256, 4) >= 152) {
    PEPS_SIMT_CFG(1, 4, 1, 8);
  }
  PEPS_SIMT_CFG(1, 2, 8, 32);
#undef PEPS_SIMT_CFG
}

}  // namespace

cudaError_t launch_contract_simt(const StepShape &sh, const StepItem *d_items, int n_items,
                                 const OpDesc *d_ops, Rec *d_recs, const DeviceStatus *st,
                                 cudaStream_t s, bool aligned32) {
  (void)st;
  if (n_items <= 0) return cudaSuccess;
  if (sh.M <= 8 && n_items <= 65535) {
    const int64_t blocks = (sh.M * sh.N + 255) / 256;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    dim3 grid((unsigned)blocks, n_items);
    switch (sh.fmt) {
      case FMT_F32: return launch_dependent(k_contract_rows<FMT_F32>, grid, dim3(256), 0, s, sh, d_items, d_ops, d_recs);
      case FMT_TF32: return launch_dependent(k_contract_rows<FMT_TF32>, grid, dim3(256), 0, s, sh, d_items, d_ops, d_recs);
      case FMT_BF16: return launch_dependent(k_contract_rows<FMT_BF16>, grid, dim3(256), 0, s, sh, d_items, d_ops, d_recs);
      case FMT_FP16: return launch_dependent(k_contract_rows<FMT_FP16>, grid, dim3(256), 0, s, sh, d_items, d_ops, d_recs);
      case FMT_BF16X2: return launch_dependent(k_contract_rows<FMT_BF16X2>, grid, dim3(256), 0, s, sh, d_items, d_ops, d_recs);
      case FMT_FP16X2: return launch_dependent(k_contract_rows<FMT_FP16X2>, grid, dim3(256), 0, s, sh, d_items, d_ops, d_recs);
    }
    return cudaErrorInvalidValue;
  }
  switch (sh.fmt) {
    case FMT_F32: return launch_tiles<FMT_F32>(sh, d_items, n_items, d_ops, d_recs, aligned32, s);
    case FMT_TF32: return launch_tiles<FMT_TF32>(sh, d_items, n_items, d_ops, d_recs, aligned32, s);
    case FMT_BF16: return launch_tiles<FMT_BF16>(sh, d_items, n_items, d_ops, d_recs, aligned32, s);
    case FMT_FP16: return launch_tiles<FMT_FP16>(sh, d_items, n_items, d_ops, d_recs, aligned32, s);
    case FMT_BF16X2: return launch_tiles<FMT_BF16X2>(sh, d_items, n_items, d_ops, d_recs, aligned32, s);
    case FMT_FP16X2: return launch_tiles<FMT_FP16X2>(sh, d_items, n_items, d_ops, d_recs, aligned32, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace peps
