// Jet-trajectory surrogate behind include/lbm_mlp.h: a multilayer perceptron
// trained and evaluated on the device.  Matrix products run on the tensor
// cores with bfloat16 operands and FP32 accumulation (mma.sync m16n8k16: a
// batch tile of 16 or 32 rows is below the 64 rows of the asynchronous tensor-core
// pipeline's smallest tile, and the products are bound by streaming the weights from L2);
// epilogues fuse bias, SiLU and its derivative; every reduction has a fixed order, so results are
// reproducible.
//
// Networks whose width is a multiple of 64 up to 256 (n_in <= 64, n_out <= 256: the surrogate's
// own size) run fused: one kernel takes a tile of rows through every layer with the activations in
// shared memory, and in training on through the loss and the backward pass of those rows
// (k_rows); the weight gradients of all layers follow in one launch (k_wgrad), their reduction and
// the optimiser in a third (k_update).  Other networks run layer by layer (k_gemm).  One kernel per
// layer and direction took 176 us for a batch of 4096 and 440 us for a training step of 64 rows,
// nearly all of it launch latency and the gaps between launches of a few microseconds; fused they
// take 29 and 63 us through the C ABI (host arrays in, loss out).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <vector>

#include "../../include/lbm_mlp.h"
#include "lbm_mlp_buffers.h"

namespace {

constexpr int TM = 64, TN = 64, TK = 32, GEMM_THREADS = 128;
constexpr int SK = TK + 8;  // padded shared row (bf16): conflict-free fragment loads
constexpr int KSPLIT = 256;  // batch rows per split of a weight-gradient product

enum { EPI_SILU = 0, EPI_LINEAR = 1, EPI_DSILU = 2, EPI_PARTIAL = 3 };

// C(m, n) = sum_k A(m, k) B(n, k); A(m, k) = A[m sAm + k sAk], B(n, k) = B[n sBn + k sBk]
struct GemmArgs {
  const __nv_bfloat16* A;
  long long sAm, sAk;
  const __nv_bfloat16* B;
  long long sBn, sBk;
  int M, N, K;
  int kps;            // K range per blockIdx.z (multiple of TK)
  const float* bias;  // EPI_SILU, EPI_LINEAR
  float* out;         // SILU: z; LINEAR: y; DSILU: dz; PARTIAL: [split][M][N]
  long long ldo;
  __nv_bfloat16* outb;  // SILU: silu(z); DSILU: dz
  long long ldb;
  const float* zsave;  // DSILU: pre-activations
  long long ldz;
};

// 1 / (1 + exp(-z)).  The reciprocal by the hardware estimate and one Newton step, of a quarter of the
// denominator (rounded as the whole), so that the estimate of no finite one is subnormal.  Compared with the
// rounded division for every float exp(-z) >= 0: the same bits wherever the quotient is normal (z > -87.3), within
// 2^-149 below.  The evaluations are most of k_rows: 29 us for a batch of 4096, 31.5 us with a division.
__device__ __forceinline__ float sigmoid_(float z) {
  const float e = expf(-z), d = fmaf(0.25f, e, 0.25f);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  r = fmaf(r, fmaf(-d, r, 1.0f), r);
  return e > 3.402823466e38f ? 0.0f : 0.25f * r;
}
// derivative of z s, s = sigmoid_(z)
__device__ __forceinline__ float silu_slope(float z, float s) { return s * (1.0f + z * (1.0f - s)); }

__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// stage a ROWS x TK tile X(r, k) = P[(r0 + r) sr + (k0 + k) sk] (zero outside rows < R, k < kend)
template <int ROWS>
__device__ __forceinline__ void stage(__nv_bfloat16* S, const __nv_bfloat16* P, long long sr, long long sk, int r0,
                                      int R, int k0, int kend) {
  const __nv_bfloat16 zero = __float2bfloat16(0.0f);
  for (int e = threadIdx.x; e < ROWS * TK; e += GEMM_THREADS) {
    int r, c;
    if (sk == 1) {  // consecutive threads along the contiguous index
      r = e / TK;
      c = e % TK;
    } else {
      c = e / ROWS;
      r = e % ROWS;
    }
    const int gr = r0 + r, gk = k0 + c;
    S[r * SK + c] = (gr < R && gk < kend) ? P[gr * sr + gk * sk] : zero;
  }
}

template <int EPI>
__global__ void __launch_bounds__(GEMM_THREADS) k_gemm(const GemmArgs g) {
  __shared__ __align__(16) __nv_bfloat16 As[TM * SK];
  __shared__ __align__(16) __nv_bfloat16 Bs[TN * SK];
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int kbeg = blockIdx.z * g.kps;
  const int kend = min(g.K, kbeg + g.kps);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const int gid = lane >> 2, tig = lane & 3;
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][j][c] = 0.0f;

  for (int k0 = kbeg; k0 < kend; k0 += TK) {
    stage<TM>(As, g.A, g.sAm, g.sAk, m0, g.M, k0, kend);
    stage<TN>(Bs, g.B, g.sBn, g.sBk, n0, g.N, k0, kend);
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; kk += 16) {
      uint32_t a[2][4], b[4][2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const __nv_bfloat16* p = As + (wm + i * 16 + gid) * SK + kk + 2 * tig;
        a[i][0] = ld_pair(p);
        a[i][1] = ld_pair(p + 8 * SK);
        a[i][2] = ld_pair(p + 8);
        a[i][3] = ld_pair(p + 8 * SK + 8);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __nv_bfloat16* p = Bs + (wn + j * 8 + gid) * SK + kk + 2 * tig;
        b[j][0] = ld_pair(p);
        b[j][1] = ld_pair(p + 8);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int m = m0 + wm + i * 16 + gid + (c >= 2 ? 8 : 0);
        const int n = n0 + wn + j * 8 + 2 * tig + (c & 1);
        if (m >= g.M || n >= g.N) continue;
        const float v = acc[i][j][c];
        if constexpr (EPI == EPI_SILU) {
          const float z = v + g.bias[n];
          g.out[m * g.ldo + n] = z;
          g.outb[m * g.ldb + n] = __float2bfloat16(z * sigmoid_(z));
        } else if constexpr (EPI == EPI_LINEAR) {
          g.out[m * g.ldo + n] = v + g.bias[n];
        } else if constexpr (EPI == EPI_DSILU) {
          const float z = g.zsave[m * g.ldz + n];
          const float s = sigmoid_(z);
          const float d = v * silu_slope(z, s);
          g.out[m * g.ldo + n] = d;
          g.outb[m * g.ldb + n] = __float2bfloat16(d);
        } else {
          g.out[((long long)blockIdx.z * g.M + m) * g.N + n] = v;
        }
      }
}

__global__ void k_to_bf16(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) y[i] = __float2bfloat16(x[i]);
}

// per row: squared error of the positions and cross-entropy of the logits, and dL/dy
__global__ void k_loss(const float* __restrict__ y, const float* __restrict__ target, const int* __restrict__ label,
                       int B, int n_pos, int n_cls, float w_pos, float w_cls, float* __restrict__ dy,
                       __nv_bfloat16* __restrict__ dyb, float* __restrict__ row_loss, int* __restrict__ bad) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int n_out = n_pos + n_cls;
  const float* yr = y + (long long)b * n_out;
  float* dr = dy + (long long)b * n_out;
  __nv_bfloat16* dbr = dyb + (long long)b * n_out;
  float lp = 0.0f;
  for (int k = 0; k < n_pos; ++k) {
    const float d = yr[k] - target[(long long)b * n_pos + k];
    lp += d * d;
    dr[k] = w_pos * 2.0f * d / (float)(B * n_pos);
  }
  float lc = 0.0f;
  if (n_cls > 0) {
    int lab = label[b];
    if (lab < 0 || lab >= n_cls) {
      atomicOr(bad, 1);
      lab = 0;
    }
    float mx = yr[n_pos];
    for (int k = 1; k < n_cls; ++k) mx = fmaxf(mx, yr[n_pos + k]);
    float se = 0.0f;
    for (int k = 0; k < n_cls; ++k) se += expf(yr[n_pos + k] - mx);
    lc = logf(se) - (yr[n_pos + lab] - mx);
    for (int k = 0; k < n_cls; ++k) {
      const float p = expf(yr[n_pos + k] - mx) / se;
      dr[n_pos + k] = w_cls * (p - (k == lab ? 1.0f : 0.0f)) / (float)B;
    }
  }
  for (int k = 0; k < n_out; ++k) dbr[k] = __float2bfloat16(dr[k]);
  row_loss[b] = (n_pos > 0 ? w_pos * lp / (float)(B * n_pos) : 0.0f) + w_cls * lc / (float)B;
}

// fixed-order sum of n values by one block of 256 threads
__global__ void k_sum(const float* __restrict__ v, int n, float* __restrict__ out) {
  __shared__ float s[256];
  float a = 0.0f;
  for (int i = threadIdx.x; i < n; i += 256) a += v[i];
  s[threadIdx.x] = a;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = s[0];
}

// out[n] = sum_b g[b][n] (bias gradients), one thread per column, fixed order
__global__ void k_colsum(const float* __restrict__ g, int B, int N, float* __restrict__ out) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  float a = 0.0f;
  for (int b = 0; b < B; ++b) a += g[(long long)b * N + n];
  out[n] = a;
}

// out[e] = sum_s part[s][e], fixed order
__global__ void k_reduce_splits(const float* __restrict__ part, int splits, long long n, float* __restrict__ out) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  float a = 0.0f;
  for (int s = 0; s < splits; ++s) a += part[s * n + e];
  out[e] = a;
}

// Adam with bias correction; refreshes the bfloat16 copy of the parameters
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, __nv_bfloat16* __restrict__ pb, long long n, float lr, float c1,
                       float c2) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
  p[i] = pi;
  pb[i] = __float2bfloat16(pi);
}

// ---------------------------------------------------------------------------
// fused path

constexpr int MAX_L = 9;          // layers: depth + 1
constexpr int FR_WARPS = 16;      // warps of k_rows; a warp owns up to FR_NT tiles of 8 output features
constexpr int FR_NT = 2;
constexpr int FR_KC = 4;           // chunks of 64 inputs of a layer
constexpr int WG_ROWS = 256;      // batch rows per split of k_wgrad

struct NetShape {
  int L, n_in, width, n_out, n_pos, n_cls;
  int kp;                          // n_out rounded up to 64 (transposed head weights are zero padded)
  long long w_off[MAX_L], b_off[MAX_L], P;
  int c_off[MAX_L], nbias;         // the layer's place among all biases, and their number
  long long t_off[MAX_L];          // transposed weights of layers 1.. : [fan_in][fan_out rounded up to 64]
  // row lengths of the stored layer inputs and dL/dz: multiples of 64, zero padded
  __host__ __device__ int ld_h(int l) const { return l == 0 ? 64 : width; }
  __host__ __device__ int ld_d(int l) const { return l == L - 1 ? kp : width; }
  __host__ __device__ int fan_in(int l) const { return l == 0 ? n_in : width; }
  __host__ __device__ int fan_out(int l) const { return l == L - 1 ? n_out : width; }
};

struct RowsArgs {
  const float* x;
  const float* target;             // training
  const int* label;
  float* y;                        // inference
  const float* p;                  // FP32 parameters (biases)
  const __nv_bfloat16 *pb, *pt;    // bfloat16 parameters, transposed weights
  __nv_bfloat16* h[MAX_L];         // training: layer inputs [batch][ld_h]
  __nv_bfloat16* d[MAX_L];         // training: dL/dz of layer l [batch][ld_d]
  float* bias_part;                // training: per block, column sums of dL/dz [blocks][nbias]
  float* row_loss;
  int* bad;
  float w_pos, w_cls;
  int batch;
};

// shared-memory row strides: 8 bytes past a multiple of 128 keeps the 8-byte fragment loads of
// 4 rows x 4 column groups on distinct banks
__host__ __device__ constexpr int act_stride(int width) { return width * 2 + 8; }  // bytes
__host__ __device__ constexpr int z_stride(int width) { return width + 8; }        // floats

// One layer's weights as a warp needs them: n_rows x (64 KC), row stride ld, the warp's nt tiles of 8
// rows from tile0
struct WarpWeights {
  const __nv_bfloat16* W;
  long long ld;
  int n_rows, tile0, nt, KC;
};

// Weights of one 64-wide chunk of k for a warp's tiles of 8 output features: lane (gid, tig) takes the 16
// consecutive elements k0 + 16 tig .. of row n0 + gid (two 16-byte loads).  The order of k inside
// a product is free as long as both operands agree: step s of the chunk multiplies the elements
// 16 tig + 4 s .. + 3, so no shared-memory transpose is needed.
__device__ __forceinline__ void load_weights(uint4 q[FR_NT][2], const WarpWeights& w, int kc, int lane) {
  const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int j = 0; j < FR_NT; ++j) {
    const int n = (w.tile0 + j) * 8 + gid;
    if (kc < w.KC && j < w.nt && n < w.n_rows) {
      const uint4* src = reinterpret_cast<const uint4*>(w.W + n * w.ld + kc * 64 + 16 * tig);
      q[j][0] = __ldg(src);
      q[j][1] = __ldg(src + 1);
    } else {
      q[j][0] = q[j][1] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
}

// acc = act (16 MT rows, row stride in bytes) x W^T.  q holds this layer's weights; each chunk's
// registers take the same chunk of the next layer as soon as it has been multiplied, so the loads have
// a whole layer, its epilogue and barrier included, to arrive (with one chunk of lookahead the kernel
// waited for L2 four times a layer: 34 us for a batch of 4096, 28 us like this, cold caches).
template <int MT>
__device__ __forceinline__ void rows_gemm(float acc[MT][FR_NT][4], const unsigned char* act, int stride,
                                          const WarpWeights& w, const WarpWeights& next, uint4 q[FR_KC][FR_NT][2],
                                          int lane) {
  const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < FR_NT; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][j][c] = 0.0f;
#pragma unroll
  for (int kc = 0; kc < FR_KC; ++kc) {
    if (kc < w.KC) {
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        uint32_t a[MT][4];
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          const unsigned char* r = act + (i * 16 + gid) * stride + (kc * 64 + 16 * tig + 4 * s) * 2;
          const uint2 lo = *reinterpret_cast<const uint2*>(r), hi = *reinterpret_cast<const uint2*>(r + 8 * stride);
          a[i][0] = lo.x;
          a[i][1] = hi.x;
          a[i][2] = lo.y;
          a[i][3] = hi.y;
        }
#pragma unroll
        for (int j = 0; j < FR_NT; ++j) {
          if (j < w.nt) {
            const uint4 v = q[kc][j][s >> 1];
            const uint32_t b[2] = {s & 1 ? v.z : v.x, s & 1 ? v.w : v.y};
#pragma unroll
            for (int i = 0; i < MT; ++i) mma_bf16(acc[i][j], a[i], b);
          }
        }
      }
    }
    load_weights(q[kc], next, kc, lane);
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// One tile of 16 MT rows through the whole network, and in training back again.  A block streams
// the bfloat16 weights once from L2 (433 KB each way for 5 -> 4 x 256 -> 68).  Bound by instruction
// issue and latency: a block has 16 warps, and a third of their instructions evaluate exp and SiLU.
// 22 us for a batch of 4096 (128 blocks), 50 us with the backward pass, 35 us for a training batch of 64
// (4 blocks), cold caches.
template <int MT, bool TRAIN>
__global__ void __launch_bounds__(FR_WARPS * 32) k_rows(const __grid_constant__ NetShape S,
                                                        const __grid_constant__ RowsArgs A) {
  constexpr int RT = 16 * MT, NTHR = FR_WARPS * 32;
  extern __shared__ __align__(16) unsigned char fr_smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int W = S.width, as = act_stride(W > S.kp ? W : S.kp), zs = z_stride(W);
  unsigned char* act[2] = {fr_smem, fr_smem + RT * as};
  float* const ys = reinterpret_cast<float*>(fr_smem + 2 * RT * as);  // [RT][n_out]
  float* const xs = ys + RT * S.n_out;                                // [RT][n_in], bfloat16 values
  float* const bs = xs + RT * S.n_in;                                 // the biases of every layer
  __nv_bfloat16* const w0 = reinterpret_cast<__nv_bfloat16*>(bs + S.nbias);  // [width][n_in]
  // training: the slopes silu'(z) of the hidden layers, [L-1][RT][zs]
  float* const slope = bs + ((RT * (S.n_out + S.n_in) + S.nbias + (W * S.n_in + 1) / 2 + 1) & ~1) - RT * (S.n_out + S.n_in);
  const int row0 = blockIdx.x * RT, rows = min(RT, A.batch - row0);

  for (int e = tid; e < RT * S.n_in; e += NTHR) {
    const int r = e / S.n_in, k = e - r * S.n_in;
    const __nv_bfloat16 v = __float2bfloat16(r < rows ? A.x[(long long)(row0 + r) * S.n_in + k] : 0.0f);
    xs[e] = __bfloat162float(v);
  }
  if (TRAIN) {
    for (int e = tid; e < rows * 64; e += NTHR) {
      const int r = e >> 6, k = e & 63;
      A.h[0][(long long)(row0 + r) * 64 + k] =
          __float2bfloat16(k < S.n_in ? A.x[(long long)(row0 + r) * S.n_in + k] : 0.0f);
    }
  }
  for (int e = tid; e < W * S.n_in; e += NTHR) w0[e] = A.pb[S.w_off[0] + e];
  for (int l = 0; l < S.L; ++l)
    for (int n = tid; n < S.fan_out(l); n += NTHR) bs[S.c_off[l] + n] = A.p[S.b_off[l] + n];
  uint4 q[FR_KC][FR_NT][2];
  float acc[MT][FR_NT][4];
  // the warp's share of layer l forwards, and of the product with the transposed weights backwards
  const auto fwd = [&](int l) {
    const bool head = l == S.L - 1;
    const int nt = ((head ? S.kp : W) / 8 + FR_WARPS - 1) / FR_WARPS;
    return WarpWeights{A.pb + S.w_off[l], W, S.fan_out(l), warp * nt, nt, W / 64};
  };
  const auto bwd = [&](int l) {
    const int K = l == S.L - 1 ? S.kp : W;
    const int nt = (W / 8 + FR_WARPS - 1) / FR_WARPS;
    return WarpWeights{A.pt + S.t_off[l], K, W, warp * nt, nt, K / 64};
  };
  WarpWeights ww = fwd(1);
#pragma unroll
  for (int kc = 0; kc < FR_KC; ++kc) load_weights(q[kc], ww, kc, lane);
  __syncthreads();

  // layer 0: n_in inputs; a thread takes one output feature for half of the rows
  constexpr int RH = RT / 2;
  for (int e = tid; e < 2 * W; e += NTHR) {
    const int n = e % W, r0 = e / W * RH;
    const __nv_bfloat16* w = w0 + n * S.n_in;
    const float b = bs[n];
    float z[RH];
#pragma unroll
    for (int r = 0; r < RH; ++r) z[r] = 0.0f;
    for (int k = 0; k < S.n_in; ++k) {
      const float wk = __bfloat162float(w[k]);
#pragma unroll
      for (int r = 0; r < RH; ++r) z[r] = fmaf(xs[(r0 + r) * S.n_in + k], wk, z[r]);
    }
#pragma unroll
    for (int r = 0; r < RH; ++r) {
      const float zr = z[r] + b, sr = sigmoid_(zr);
      const __nv_bfloat16 h = __float2bfloat16(zr * sr);
      *reinterpret_cast<__nv_bfloat16*>(act[0] + (r0 + r) * as + n * 2) = h;
      if (TRAIN) {
        slope[(r0 + r) * zs + n] = silu_slope(zr, sr);
        if (r0 + r < rows) A.h[1][(long long)(row0 + r0 + r) * W + n] = h;
      }
    }
  }
  __syncthreads();

  int cur = 0;
  for (int l = 1; l < S.L; ++l) {
    const bool head = l == S.L - 1;
    const int nt = ww.nt, t0 = ww.tile0, N = S.fan_out(l);
    WarpWeights next = ww;
    next.KC = 0;
    if (!head) next = fwd(l + 1);
    else if (TRAIN) next = bwd(l);
    rows_gemm<MT>(acc, act[cur], as, ww, next, q, lane);
    ww = next;
#pragma unroll
    for (int j = 0; j < FR_NT; ++j) {
      const int n = (t0 + j) * 8 + 2 * tig;
      if (j >= nt || n >= N) continue;
      const float b0 = bs[S.c_off[l] + n], b1 = n + 1 < N ? bs[S.c_off[l] + n + 1] : 0.0f;
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int hrow = 0; hrow < 2; ++hrow) {
          const int r = i * 16 + gid + 8 * hrow;
          const float z0 = acc[i][j][2 * hrow] + b0, z1 = acc[i][j][2 * hrow + 1] + b1;
          if (head) {
            if (TRAIN) {
              ys[r * S.n_out + n] = z0;
              if (n + 1 < N) ys[r * S.n_out + n + 1] = z1;
            } else if (r < rows) {
              float* yr = A.y + (long long)(row0 + r) * S.n_out + n;
              yr[0] = z0;
              if (n + 1 < N) yr[1] = z1;
            }
          } else {
            const float s0 = sigmoid_(z0), s1 = sigmoid_(z1);
            const uint32_t h = pack_bf16(z0 * s0, z1 * s1);
            *reinterpret_cast<uint32_t*>(act[cur ^ 1] + r * as + n * 2) = h;
            if (TRAIN) {
              *reinterpret_cast<float2*>(slope + (l * RT + r) * zs + n) =
                  make_float2(silu_slope(z0, s0), silu_slope(z1, s1));
              if (r < rows) *reinterpret_cast<uint32_t*>(A.h[l + 1] + (long long)(row0 + r) * W + n) = h;
            }
          }
        }
    }
    cur ^= 1;
    if (TRAIN || !head) __syncthreads();
  }
  if (!TRAIN) return;

  // loss of the rows and dL/dy: TPR threads per row, their sums by a butterfly
  constexpr int TPR = NTHR / RT;
  {
    const int r = tid / TPR, t = tid % TPR, B = A.batch, n_pos = S.n_pos, n_cls = S.n_cls;
    const bool live = r < rows;
    float* const yr = ys + r * S.n_out;
    const long long gr = row0 + r;
    float lp = 0.0f;
    for (int k = t; k < n_pos; k += TPR) {
      const float d = live ? yr[k] - A.target[gr * n_pos + k] : 0.0f;
      lp += d * d;
      yr[k] = A.w_pos * 2.0f * d / (float)(B * n_pos);
    }
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1) lp += __shfl_xor_sync(0xffffffffu, lp, o);
    if (t == 0) {
      float lc = 0.0f;
      if (n_cls > 0) {
        int lab = live ? A.label[gr] : 0;
        if (lab < 0 || lab >= n_cls) {
          atomicOr(A.bad, 1);
          lab = 0;
        }
        float mx = yr[n_pos];
        for (int k = 1; k < n_cls; ++k) mx = fmaxf(mx, yr[n_pos + k]);
        float se = 0.0f;
        for (int k = 0; k < n_cls; ++k) se += expf(yr[n_pos + k] - mx);
        lc = logf(se) - (yr[n_pos + lab] - mx);
        for (int k = 0; k < n_cls; ++k) {
          const float pk = expf(yr[n_pos + k] - mx) / se;
          yr[n_pos + k] = live ? A.w_cls * (pk - (k == lab ? 1.0f : 0.0f)) / (float)B : 0.0f;
        }
      }
      if (live) A.row_loss[gr] = (n_pos > 0 ? A.w_pos * lp / (float)(B * n_pos) : 0.0f) + A.w_cls * lc / (float)B;
    }
  }
  __syncthreads();
  // dL/dz of the head: bfloat16 operand (zero padded), bias column sums
  float* const bp = A.bias_part + (long long)blockIdx.x * S.nbias;
  for (int e = tid; e < RT * S.kp; e += NTHR) {
    const int r = e / S.kp, n = e - r * S.kp;
    const __nv_bfloat16 v = __float2bfloat16(n < S.n_out ? ys[r * S.n_out + n] : 0.0f);
    *reinterpret_cast<__nv_bfloat16*>(act[cur] + r * as + n * 2) = v;
    if (r < rows) A.d[S.L - 1][(long long)(row0 + r) * S.kp + n] = v;
  }
  for (int n = tid; n < S.n_out; n += NTHR) {
    float a = 0.0f;
    for (int r = 0; r < RT; ++r) a += ys[r * S.n_out + n];
    bp[S.c_off[S.L - 1] + n] = a;
  }
  __syncthreads();

  // dL/dz_{l-1} = (dL/dz_l W_l) silu'(z_{l-1})
  for (int l = S.L - 1; l >= 1; --l) {
    WarpWeights next = ww;
    next.KC = 0;
    if (l > 1) next = bwd(l - 1);
    rows_gemm<MT>(acc, act[cur], as, ww, next, q, lane);
    const int hid_nt = ww.nt, hid_t0 = ww.tile0;
    ww = next;
#pragma unroll
    for (int j = 0; j < FR_NT; ++j) {
      const int n = (hid_t0 + j) * 8 + 2 * tig;
      if (j >= hid_nt || n >= W) continue;  // whole warps
      float c0 = 0.0f, c1 = 0.0f;  // column sums over the tile's rows
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int hrow = 0; hrow < 2; ++hrow) {
          const int r = i * 16 + gid + 8 * hrow;
          const float2 sl = *reinterpret_cast<const float2*>(slope + ((l - 1) * RT + r) * zs + n);
          const float d0 = acc[i][j][2 * hrow] * sl.x, d1 = acc[i][j][2 * hrow + 1] * sl.y;
          c0 += d0;
          c1 += d1;
          const uint32_t v = pack_bf16(d0, d1);
          *reinterpret_cast<uint32_t*>(act[cur ^ 1] + r * as + n * 2) = v;
          if (r < rows) *reinterpret_cast<uint32_t*>(A.d[l - 1] + (long long)(row0 + r) * W + n) = v;
        }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {  // over gid: rows past the batch hold zeros
        c0 += __shfl_xor_sync(0xffffffffu, c0, o);
        c1 += __shfl_xor_sync(0xffffffffu, c1, o);
      }
      if (gid == 0) {
        bp[S.c_off[l - 1] + n] = c0;
        bp[S.c_off[l - 1] + n + 1] = c1;
      }
    }
    cur ^= 1;
    __syncthreads();
  }
}

// Weight gradients of every layer in one launch: dW_l(o, i) = sum_b dz_l(b, o) h_l(b, i), one 64 x 64
// tile of one layer and one split of WG_ROWS batch rows per block, partial sums in FP32 at
// part[split][w_off + o fan_in + i].  Both operands lie with their features contiguous; ldmatrix.trans
// turns them into fragments.
constexpr int WG_T = 64, WG_K = 64, WG_LD = WG_T + 8;

struct WgradArgs {
  const __nv_bfloat16* h[MAX_L];
  const __nv_bfloat16* d[MAX_L];
  float* part;
  int batch;
  int tile0[MAX_L + 1];  // first tile of each layer
};

__device__ __forceinline__ void wg_load(uint4 v[4], const __nv_bfloat16* src, int ld, int c0, int b0, int bend) {
  // rows b0 .. b0+63 (zeros from bend on), columns c0 .. c0+63
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int e = threadIdx.x + k * GEMM_THREADS, r = e >> 3, c = (e & 7) * 8;
    v[k] = b0 + r < bend ? __ldg(reinterpret_cast<const uint4*>(src + (long long)(b0 + r) * ld + c0 + c))
                         : make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ void wg_put(__nv_bfloat16* T, const uint4 v[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int e = threadIdx.x + k * GEMM_THREADS;
    *reinterpret_cast<uint4*>(T + (e >> 3) * WG_LD + (e & 7) * 8) = v[k];
  }
}
static_assert(WG_K * WG_T == 4 * 8 * GEMM_THREADS, "four 16-byte loads per thread and operand");
__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__global__ void __launch_bounds__(GEMM_THREADS) k_wgrad(const __grid_constant__ NetShape S,
                                                        const __grid_constant__ WgradArgs A) {
  __shared__ __align__(16) __nv_bfloat16 Ds[WG_K * WG_LD], Hs[WG_K * WG_LD];
  int l = 0;
  while ((int)blockIdx.x >= A.tile0[l + 1]) ++l;
  const int K = S.fan_in(l), N = S.fan_out(l), tiles_i = (K + WG_T - 1) / WG_T;
  const int tile = blockIdx.x - A.tile0[l];
  const int o0 = tile / tiles_i * WG_T, i0 = tile % tiles_i * WG_T;
  const int bbeg = blockIdx.y * WG_ROWS, bend = min(A.batch, bbeg + WG_ROWS);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][j][c] = 0.0f;
  uint4 vd[4], vh[4];  // the next chunk of rows travels while this one is multiplied
  wg_load(vd, A.d[l], S.ld_d(l), o0, bbeg, bend);
  wg_load(vh, A.h[l], S.ld_h(l), i0, bbeg, bend);
  for (int b0 = bbeg; b0 < bend; b0 += WG_K) {
    wg_put(Ds, vd);
    wg_put(Hs, vh);
    __syncthreads();
    if (b0 + WG_K < bend) {
      wg_load(vd, A.d[l], S.ld_d(l), o0, b0 + WG_K, bend);
      wg_load(vh, A.h[l], S.ld_h(l), i0, b0 + WG_K, bend);
    }
    // lane -> row (k) and column group of the four 8 x 8 matrices of one ldmatrix
    const int lr = lane & 7, lq = lane >> 3;
#pragma unroll
    for (int kk = 0; kk < WG_K; kk += 16) {
      uint32_t a[2][4], b[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)  // matrices (k lo, m lo), (k lo, m hi), (k hi, m lo), (k hi, m hi)
        ldsm_x4_t(a[i], Ds + (kk + lr + (lq >> 1) * 8) * WG_LD + wm + i * 16 + (lq & 1) * 8);
#pragma unroll
      for (int j = 0; j < 2; ++j)  // matrices (k lo, n lo), (k hi, n lo), (k lo, n hi), (k hi, n hi)
        ldsm_x4_t(b[j], Hs + (kk + lr + (lq & 1) * 8) * WG_LD + wn + j * 16 + (lq >> 1) * 8);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], &b[j >> 1][(j & 1) * 2]);
    }
    __syncthreads();
  }
  float* const out = A.part + (long long)blockIdx.y * S.P + S.w_off[l];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int o = o0 + wm + i * 16 + gid + (c >= 2 ? 8 : 0), k = i0 + wn + j * 8 + 2 * tig + (c & 1);
        if (o < N && k < K) out[(long long)o * K + k] = acc[i][j][c];
      }
}

// bfloat16 copies of parameter e: the plain one and, for the weights of layers 1.., the transposed
__device__ __forceinline__ void put_bf16(const NetShape& S, __nv_bfloat16* pb, __nv_bfloat16* pt, long long e, float v) {
  const __nv_bfloat16 h = __float2bfloat16(v);
  pb[e] = h;
  int l = S.L - 1;
  while (e < S.w_off[l]) --l;
  if (l == 0 || e >= S.b_off[l]) return;
  const unsigned K = (unsigned)S.width, r = (unsigned)(e - S.w_off[l]), o = r / K, i = r - o * K;
  const int ld = l == S.L - 1 ? S.kp : S.width;
  pt[S.t_off[l] + (long long)i * ld + o] = h;
}
__global__ void k_refresh(const __grid_constant__ NetShape S, const float* __restrict__ p,
                          __nv_bfloat16* __restrict__ pb, __nv_bfloat16* __restrict__ pt) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e < S.P) put_bf16(S, pb, pt, e, p[e]);
}

// Gradient of parameter e from the partial sums (weights: splits of k_wgrad; biases: blocks of
// k_rows), in a fixed order; with lr >= 0 the Adam update, else the gradient to g.  The last block sums the
// row losses.
__global__ void __launch_bounds__(256) k_update(const __grid_constant__ NetShape S, const float* __restrict__ part,
                                                int splits, const float* __restrict__ bias_part, int row_blocks,
                                                float* __restrict__ g, float* __restrict__ p, float* __restrict__ m,
                                                float* __restrict__ v, __nv_bfloat16* __restrict__ pb,
                                                __nv_bfloat16* __restrict__ pt, float lr, float c1, float c2,
                                                const float* __restrict__ row_loss, int batch,
                                                float* __restrict__ loss) {
  if (blockIdx.x == gridDim.x - 1) {  // as k_sum
    __shared__ float s[256];
    float a = 0.0f;
    for (int i = threadIdx.x; i < batch; i += 256) a += row_loss[i];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = s[0];
    return;
  }
  const long long e = blockIdx.x * 256LL + threadIdx.x;
  if (e >= S.P) return;
  int l = S.L - 1;
  while (e < S.w_off[l]) --l;
  float a = 0.0f;
  if (e >= S.b_off[l])
    for (int k = 0; k < row_blocks; ++k) a += bias_part[(long long)k * S.nbias + S.c_off[l] + (e - S.b_off[l])];
  else
    for (int k = 0; k < splits; ++k) a += part[k * S.P + e];
  if (lr < 0.0f) {
    g[e] = a;
    return;
  }
  const float mi = 0.9f * m[e] + 0.1f * a;
  const float vi = 0.999f * v[e] + 0.001f * a * a;
  m[e] = mi;
  v[e] = vi;
  const float pi = p[e] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
  p[e] = pi;
  put_bf16(S, pb, pt, e, pi);
}

// rows per block: 16 where that already gives every SM a block at most (a smaller tile has the shorter
// chain), else 32
template <bool TRAIN>
size_t rows_smem(const NetShape& S, int mt) {
  const size_t rt = 16 * (size_t)mt;
  size_t b = 2 * rt * act_stride(S.width > S.kp ? S.width : S.kp) +
             4 * (rt * S.n_out + rt * S.n_in + S.nbias + (S.width * S.n_in + 1) / 2 + 2);
  if (TRAIN) b += 4 * (size_t)(S.L - 1) * rt * z_stride(S.width);
  return b;
}
constexpr size_t ROWS_SMEM_MAX = 220 * 1024;
constexpr size_t STAGE_BYTES = 128 * 1024;

template <int MT, bool TRAIN>
cudaError_t launch_rows_mt(const NetShape& S, const RowsArgs& A, cudaStream_t s) {
  k_rows<MT, TRAIN><<<(A.batch + 16 * MT - 1) / (16 * MT), FR_WARPS * 32, rows_smem<TRAIN>(S, MT), s>>>(S, A);
  return cudaGetLastError();
}
// let k_rows have its shared memory on the current device (the attribute is per device)
bool allow_rows() {
  const auto allow = [](auto* kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ROWS_SMEM_MAX) == cudaSuccess;
  };
  if (allow(k_rows<1, false>) && allow(k_rows<2, false>) && allow(k_rows<1, true>) && allow(k_rows<2, true>)) return true;
  cudaGetLastError();
  return false;
}
template <bool TRAIN>
int rows_mt(const NetShape& S, int batch) {
  return batch > 16 * 152 && rows_smem<TRAIN>(S, 2) <= ROWS_SMEM_MAX ? 2 : 1;
}
template <bool TRAIN>
cudaError_t launch_rows(const NetShape& S, const RowsArgs& A, cudaStream_t s) {
  return rows_mt<TRAIN>(S, A.batch) == 2 ? launch_rows_mt<2, TRAIN>(S, A, s) : launch_rows_mt<1, TRAIN>(S, A, s);
}

bool is_device_ptr(const void* ptr) {
  if (!ptr) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

struct lbm_mlp {
  int n_in, width, depth, n_pos, n_cls, n_out, max_batch;
  int device;
  cudaStream_t stream;
  std::vector<int> fan_in, fan_out;  // per layer
  std::vector<size_t> w_off, b_off;  // flat offsets
  size_t P;
  long long step;
  char* mem;
  float *p, *g, *m, *v;          // parameters, gradient, Adam moments (flat FP32)
  __nv_bfloat16* pb;             // bfloat16 copy of the parameters
  float* x32;                    // staged input [max_batch][n_in]
  __nv_bfloat16* h[9];           // layer inputs: h[0] = x, h[l] = silu(z_l), bf16
  float* z[9];                   // pre-activations z_l, l = 1..depth (FP32)
  float* y;                      // output [max_batch][n_out]
  float *d32[2];                 // backward: dL/dz (FP32), ping-pong
  __nv_bfloat16* d16[2];         // backward: dL/dz (bf16)
  float* part;                   // weight-gradient split partials
  float *tgt, *row_loss, *loss;  // staged targets, per-row loss, total
  int *lab, *bad;
  // fused path (fused: the network's shape allows it)
  bool fused;
  NetShape S;
  __nv_bfloat16* pt;             // transposed bfloat16 weights
  __nv_bfloat16* dl[MAX_L];      // dL/dz per layer
  float* bias_part;
  char* stage_dev;               // a training batch from the host arrives here in one copy
  char* pinned;                  // page-locked: that batch (STAGE_BYTES), then loss and bad
};

namespace {

template <int EPI>
cudaError_t gemm(const GemmArgs& a, int splits, cudaStream_t s) {
  dim3 grid((unsigned)((a.N + TN - 1) / TN), (unsigned)((a.M + TM - 1) / TM), (unsigned)splits);
  k_gemm<EPI><<<grid, GEMM_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

GemmArgs args(const __nv_bfloat16* A, long long sAm, long long sAk, const __nv_bfloat16* B, long long sBn,
              long long sBk, int M, int N, int K) {
  GemmArgs a;
  memset(&a, 0, sizeof a);
  a.A = A;
  a.sAm = sAm;
  a.sAk = sAk;
  a.B = B;
  a.sBn = sBn;
  a.sBk = sBk;
  a.M = M;
  a.N = N;
  a.K = K;
  a.kps = (K + TK - 1) / TK * TK;
  return a;
}

#define MLP_CUDA(call)                              \
  do {                                              \
    if ((call) != cudaSuccess) {                    \
      cudaGetLastError();                           \
      return LBM_ECUDA;                             \
    }                                               \
  } while (0)

// forward pass of `batch` rows already staged in m->x32
lbm_status forward(lbm_mlp* m, int batch) {
  MLP_CUDA((k_to_bf16<<<blocks((long long)batch * m->n_in, 256), 256, 0, m->stream>>>(m->x32, m->h[0],
                                                                                     (long long)batch * m->n_in),
            cudaGetLastError()));
  const int L = m->depth + 1;
  for (int l = 0; l < L; ++l) {
    const int K = m->fan_in[l], N = m->fan_out[l];
    GemmArgs a = args(m->h[l], K, 1, m->pb + m->w_off[l], K, 1, batch, N, K);
    a.bias = m->p + m->b_off[l];
    if (l < L - 1) {
      a.out = m->z[l + 1];
      a.ldo = N;
      a.outb = m->h[l + 1];
      a.ldb = N;
      MLP_CUDA(gemm<EPI_SILU>(a, 1, m->stream));
    } else {
      a.out = m->y;
      a.ldo = N;
      MLP_CUDA(gemm<EPI_LINEAR>(a, 1, m->stream));
    }
  }
  return LBM_OK;
}

// loss and gradient (into m->g) of `batch` rows staged in x32 / tgt / lab
lbm_status backward(lbm_mlp* m, int batch, float w_pos, float w_cls) {
  lbm_status st = forward(m, batch);
  if (st != LBM_OK) return st;
  const int L = m->depth + 1;
  k_loss<<<blocks(batch, 128), 128, 0, m->stream>>>(m->y, m->tgt, m->lab, batch, m->n_pos, m->n_cls, w_pos, w_cls,
                                                     m->d32[0], m->d16[0], m->row_loss, m->bad);
  MLP_CUDA(cudaGetLastError());
  k_sum<<<1, 256, 0, m->stream>>>(m->row_loss, batch, m->loss);
  MLP_CUDA(cudaGetLastError());
  int cur = 0;
  for (int l = L - 1; l >= 0; --l) {
    const int K = m->fan_in[l], N = m->fan_out[l];
    // dW_l(o, i) = sum_b g(b, o) h_{l-1}(b, i): split over the batch, reduced in a fixed order
    const int splits = (batch + KSPLIT - 1) / KSPLIT;
    GemmArgs a = args(m->d16[cur], 1, N, m->h[l], 1, K, N, K, batch);
    a.kps = KSPLIT;
    a.out = m->part;
    MLP_CUDA(gemm<EPI_PARTIAL>(a, splits, m->stream));
    k_reduce_splits<<<blocks((long long)N * K, 256), 256, 0, m->stream>>>(m->part, splits, (long long)N * K,
                                                                         m->g + m->w_off[l]);
    MLP_CUDA(cudaGetLastError());
    k_colsum<<<blocks(N, 128), 128, 0, m->stream>>>(m->d32[cur], batch, N, m->g + m->b_off[l]);
    MLP_CUDA(cudaGetLastError());
    if (l > 0) {
      // dL/dz_{l-1}(b, i) = sum_o g(b, o) W_l(o, i) * silu'(z_{l-1}(b, i))
      GemmArgs d = args(m->d16[cur], N, 1, m->pb + m->w_off[l], 1, K, batch, K, N);
      d.out = m->d32[cur ^ 1];
      d.ldo = K;
      d.outb = m->d16[cur ^ 1];
      d.ldb = K;
      d.zsave = m->z[l];
      d.ldz = K;
      MLP_CUDA(gemm<EPI_DSILU>(d, 1, m->stream));
      cur ^= 1;
    }
  }
  return LBM_OK;
}

lbm_status stage_inputs(lbm_mlp* m, const float* x, const float* target, const int* label, int batch) {
  const cudaMemcpyKind kx = is_device_ptr(x) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  MLP_CUDA(cudaMemcpyAsync(m->x32, x, sizeof(float) * batch * m->n_in, kx, m->stream));
  if (target && m->n_pos > 0) {
    const cudaMemcpyKind kt = is_device_ptr(target) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    MLP_CUDA(cudaMemcpyAsync(m->tgt, target, sizeof(float) * batch * m->n_pos, kt, m->stream));
  }
  if (label && m->n_cls > 0) {
    const cudaMemcpyKind kl = is_device_ptr(label) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    MLP_CUDA(cudaMemcpyAsync(m->lab, label, sizeof(int) * batch, kl, m->stream));
  }
  return LBM_OK;
}

// where a caller's buffer lies (one query each): on the host, on a device but to be staged, or where the
// kernels use it themselves
enum Place { ON_HOST, ON_DEVICE, IN_PLACE };
Place place_of(const lbm_mlp* m, const void* ptr) {
  cudaPointerAttributes a;
  if (!ptr) return ON_HOST;
  if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
    cudaGetLastError();
    return ON_HOST;
  }
  const bool dev = a.type == cudaMemoryTypeDevice, managed = a.type == cudaMemoryTypeManaged;
  if (mlpbuf::in_place(dev, managed, a.device, m->device, reinterpret_cast<uintptr_t>(ptr))) return IN_PLACE;
  return dev || managed ? ON_DEVICE : ON_HOST;
}

// device pointer of an input: the caller's own where the kernels may use it and it stays as it is while
// they run, else a copy at `staged`
template <typename V>
lbm_status on_device(lbm_mlp* m, const V* src, Place at, V* staged, size_t n, const V** out, bool stays = true) {
  if (stays && at == IN_PLACE) {
    *out = src;
    return LBM_OK;
  }
  const cudaMemcpyKind k = at == ON_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  MLP_CUDA(cudaMemcpyAsync(staged, src, sizeof(V) * n, k, m->stream));
  *out = staged;
  return LBM_OK;
}

// fused forward pass; y: memory that the kernels may use.  An x that y overlaps is staged: a block
// writes the outputs of its rows while others have yet to read theirs.
lbm_status fused_forward(lbm_mlp* m, const float* x, int batch, float* y) {
  RowsArgs A;
  memset(&A, 0, sizeof A);
  const size_t nx = (size_t)batch * m->n_in, ny = (size_t)batch * m->n_out;
  const bool apart = !mlpbuf::overlap(reinterpret_cast<uintptr_t>(x), sizeof(float) * nx,
                                      reinterpret_cast<uintptr_t>(y), sizeof(float) * ny);
  lbm_status st = on_device(m, x, place_of(m, x), m->x32, nx, &A.x, apart);
  if (st != LBM_OK) return st;
  A.y = y;
  A.p = m->p;
  A.pb = m->pb;
  A.batch = batch;
  MLP_CUDA(launch_rows<false>(m->S, A, m->stream));
  return LBM_OK;
}

// fused loss and gradient; lr >= 0: and the Adam step, else the gradient to m->g
lbm_status fused_backward(lbm_mlp* m, const float* x, const float* target, const int* label, int batch, float w_pos,
                          float w_cls, float lr, float c1, float c2) {
  RowsArgs A;
  memset(&A, 0, sizeof A);
  const size_t nx = (size_t)batch * m->n_in, nt = (size_t)batch * m->n_pos, nl = m->n_cls > 0 ? (size_t)batch : 0;
  const Place px = place_of(m, x), pt = nt ? place_of(m, target) : ON_HOST, pl = nl ? place_of(m, label) : ON_HOST;
  if (m->pinned && 4 * (nx + nt + nl) <= STAGE_BYTES && px == ON_HOST && pt == ON_HOST && pl == ON_HOST) {
    // a small host batch: through page-locked memory in one copy (every call waits for its stream
    // before it returns, so the buffer is free again by the next)
    memcpy(m->pinned, x, 4 * nx);
    if (nt) memcpy(m->pinned + 4 * nx, target, 4 * nt);
    if (nl) memcpy(m->pinned + 4 * (nx + nt), label, 4 * nl);
    MLP_CUDA(cudaMemcpyAsync(m->stage_dev, m->pinned, 4 * (nx + nt + nl), cudaMemcpyHostToDevice, m->stream));
    A.x = reinterpret_cast<const float*>(m->stage_dev);
    A.target = A.x + nx;
    A.label = reinterpret_cast<const int*>(A.target + nt);
  } else {
    lbm_status st = on_device(m, x, px, m->x32, nx, &A.x);
    if (st == LBM_OK && nt) st = on_device(m, target, pt, m->tgt, nt, &A.target);
    if (st == LBM_OK && nl) st = on_device(m, label, pl, m->lab, nl, &A.label);
    if (st != LBM_OK) return st;
  }
  WgradArgs G;
  memset(&G, 0, sizeof G);
  const NetShape& S = m->S;
  for (int l = 0; l < S.L; ++l) {
    A.h[l] = m->h[l];
    A.d[l] = m->dl[l];
    G.h[l] = m->h[l];
    G.d[l] = m->dl[l];
    G.tile0[l + 1] = G.tile0[l] + ((S.fan_in(l) + WG_T - 1) / WG_T) * ((S.fan_out(l) + WG_T - 1) / WG_T);
  }
  A.p = m->p;
  A.pb = m->pb;
  A.pt = m->pt;
  A.bias_part = m->bias_part;
  A.row_loss = m->row_loss;
  A.bad = m->bad;
  A.w_pos = w_pos;
  A.w_cls = w_cls;
  A.batch = G.batch = batch;
  G.part = m->part;
  MLP_CUDA(launch_rows<true>(S, A, m->stream));
  const int splits = (batch + WG_ROWS - 1) / WG_ROWS, rt = 16 * rows_mt<true>(S, batch);
  k_wgrad<<<dim3((unsigned)G.tile0[S.L], (unsigned)splits), GEMM_THREADS, 0, m->stream>>>(S, G);
  MLP_CUDA(cudaGetLastError());
  k_update<<<blocks(S.P, 256) + 1, 256, 0, m->stream>>>(S, m->part, splits, m->bias_part, (batch + rt - 1) / rt, m->g,
                                                        m->p, m->m, m->v, m->pb, m->pt, lr, c1, c2, m->row_loss, batch,
                                                        m->loss);
  MLP_CUDA(cudaGetLastError());
  return LBM_OK;
}

lbm_status copy_out(lbm_mlp* m, void* dst, const void* src, size_t bytes) {
  const cudaMemcpyKind k = is_device_ptr(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  MLP_CUDA(cudaMemcpyAsync(dst, src, bytes, k, m->stream));
  return LBM_OK;
}

// wait for a loss / training call: its loss to the caller, LBM_EINVAL if a label was out of range
lbm_status finish_loss(lbm_mlp* m, float* loss) {
  struct {
    float loss;
    int bad;
  } r, *out = m->pinned ? reinterpret_cast<decltype(r)*>(m->pinned + STAGE_BYTES) : &r;
  const bool dev = loss && is_device_ptr(loss);
  if (dev) MLP_CUDA(cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  MLP_CUDA(cudaMemcpyAsync(out, m->loss, sizeof r, cudaMemcpyDeviceToHost, m->stream));
  MLP_CUDA(cudaStreamSynchronize(m->stream));
  if (loss && !dev) *loss = out->loss;
  if (!out->bad) return LBM_OK;
  MLP_CUDA(cudaMemsetAsync(m->bad, 0, sizeof(int), m->stream));  // for the next call
  return LBM_EINVAL;
}

uint64_t splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

extern "C" {

lbm_status lbm_mlp_create(int n_in, int width, int depth, int n_pos, int n_cls, int max_batch,
                          unsigned long long seed, void* cuda_stream, lbm_mlp** out) {
  if (!out) return LBM_EINVAL;
  *out = nullptr;
  if (n_in < 1 || width < 1 || width > 4096 || depth < 1 || depth > 8 || n_pos < 0 || n_cls < 0 || n_cls > 64 ||
      n_pos + n_cls < 1 || max_batch < 1 || max_batch > (1 << 20))
    return LBM_EINVAL;
  lbm_mlp* m = new (std::nothrow) lbm_mlp();
  if (!m) return LBM_ENOMEM;
  m->n_in = n_in;
  m->width = width;
  m->depth = depth;
  m->n_pos = n_pos;
  m->n_cls = n_cls;
  m->n_out = n_pos + n_cls;
  m->max_batch = max_batch;
  m->stream = static_cast<cudaStream_t>(cuda_stream);
  m->step = 0;
  if (cudaGetDevice(&m->device) != cudaSuccess) {
    cudaGetLastError();
    delete m;
    return LBM_ECUDA;
  }
  const int L = depth + 1;
  size_t o = 0;
  for (int l = 0; l < L; ++l) {
    const int fi = l == 0 ? n_in : width, fo = l == L - 1 ? m->n_out : width;
    m->fan_in.push_back(fi);
    m->fan_out.push_back(fo);
    m->w_off.push_back(o);
    o += (size_t)fi * fo;
    m->b_off.push_back(o);
    o += (size_t)fo;
  }
  m->P = o;
  const size_t B = (size_t)max_batch, W = (size_t)width, wide = (size_t)(width > m->n_out ? width : m->n_out);
  // fused path: the widths its tiles fit, and a training tile of 16 rows that fits in shared memory
  NetShape& S = m->S;
  memset(&S, 0, sizeof S);
  S.L = L;
  S.n_in = n_in;
  S.width = width;
  S.n_out = m->n_out;
  S.n_pos = n_pos;
  S.n_cls = n_cls;
  S.kp = (m->n_out + 63) / 64 * 64;
  S.P = (long long)m->P;
  long long toff = 0;
  for (int l = 0; l < L; ++l) {
    S.w_off[l] = (long long)m->w_off[l];
    S.b_off[l] = (long long)m->b_off[l];
    S.t_off[l] = toff;
    S.c_off[l] = S.nbias;
    S.nbias += m->fan_out[l];
    if (l > 0) toff += (long long)width * (l == L - 1 ? S.kp : width);
  }
  m->fused = width % 64 == 0 && width <= 256 && n_in <= 64 && m->n_out <= 256 &&
             rows_smem<true>(S, 1) <= ROWS_SMEM_MAX && allow_rows();
  size_t max_part = 0;
  for (int l = 0; l < L; ++l) {
    const size_t s = (size_t)((max_batch + KSPLIT - 1) / KSPLIT) * m->fan_in[l] * m->fan_out[l];
    if (s > max_part) max_part = s;
  }
  if (m->fused) max_part = (size_t)((max_batch + WG_ROWS - 1) / WG_ROWS) * m->P;
  // one device allocation, carved into 256-byte aligned pieces
  std::vector<std::pair<void**, size_t>> parts;
  parts.push_back({(void**)&m->p, 4 * m->P});
  parts.push_back({(void**)&m->g, 4 * m->P});
  parts.push_back({(void**)&m->m, 4 * m->P});
  parts.push_back({(void**)&m->v, 4 * m->P});
  parts.push_back({(void**)&m->pb, 2 * m->P});
  if (m->fused) {
    parts.push_back({(void**)&m->pt, 2 * (size_t)toff});
    for (int l = 0; l < L; ++l) parts.push_back({(void**)&m->dl[l], 2 * B * S.ld_d(l)});
    parts.push_back({(void**)&m->bias_part, 4 * ((B + 15) / 16) * (size_t)S.nbias});
    parts.push_back({(void**)&m->stage_dev, STAGE_BYTES});
  }
  parts.push_back({(void**)&m->x32, 4 * B * n_in});
  parts.push_back({(void**)&m->h[0], 2 * B * (m->fused ? 64 : n_in)});
  for (int l = 1; l <= depth; ++l) {
    parts.push_back({(void**)&m->h[l], 2 * B * W});
    if (!m->fused) parts.push_back({(void**)&m->z[l], 4 * B * W});
  }
  parts.push_back({(void**)&m->y, 4 * B * m->n_out});
  for (int k = 0; k < 2 && !m->fused; ++k) {
    parts.push_back({(void**)&m->d32[k], 4 * B * wide});
    parts.push_back({(void**)&m->d16[k], 2 * B * wide});
  }
  parts.push_back({(void**)&m->part, 4 * max_part});
  parts.push_back({(void**)&m->tgt, 4 * B * (n_pos > 0 ? n_pos : 1)});
  parts.push_back({(void**)&m->row_loss, 4 * B});
  parts.push_back({(void**)&m->loss, 8});  // and bad, one word after it
  parts.push_back({(void**)&m->lab, 4 * B});
  size_t total = 0;
  for (auto& pr : parts) total += (pr.second + 255) / 256 * 256;
  if (cudaMalloc(&m->mem, total) != cudaSuccess) {
    cudaGetLastError();
    delete m;
    return LBM_ENOMEM;
  }
  size_t off = 0;
  for (auto& pr : parts) {
    *pr.first = m->mem + off;
    off += (pr.second + 255) / 256 * 256;
  }
  m->bad = reinterpret_cast<int*>(m->loss) + 1;
  if (cudaMemsetAsync(m->loss, 0, 8, m->stream) != cudaSuccess) {
    cudaGetLastError();
    lbm_mlp_free(m);
    return LBM_ECUDA;
  }
  if (cudaMallocHost(&m->pinned, STAGE_BYTES + 8) != cudaSuccess) {  // only saves copies: go on without it
    cudaGetLastError();
    m->pinned = nullptr;
  }
  // parameters: uniform in +-1/sqrt(fan_in) (SplitMix64 stream from seed)
  std::vector<float> init(m->P);
  uint64_t s = seed;
  for (int l = 0; l < L; ++l) {
    const double a = 1.0 / sqrt((double)m->fan_in[l]);
    const size_t n = (size_t)m->fan_in[l] * m->fan_out[l] + m->fan_out[l];
    for (size_t i = 0; i < n; ++i)
      init[m->w_off[l] + i] = (float)(a * (2.0 * ((double)(splitmix(s) >> 11) * (1.0 / 9007199254740992.0)) - 1.0));
  }
  lbm_status st = lbm_mlp_set_params(m, init.data());
  if (st != LBM_OK) {
    lbm_mlp_free(m);
    return st;
  }
  *out = m;
  return LBM_OK;
}

size_t lbm_mlp_param_count(const lbm_mlp* m) { return m ? m->P : 0; }

lbm_status lbm_mlp_set_params(lbm_mlp* m, const float* params) {
  if (!m || !params) return LBM_EINVAL;
  const cudaMemcpyKind k = is_device_ptr(params) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  MLP_CUDA(cudaMemcpyAsync(m->p, params, 4 * m->P, k, m->stream));
  MLP_CUDA(cudaMemsetAsync(m->m, 0, 4 * m->P, m->stream));
  MLP_CUDA(cudaMemsetAsync(m->v, 0, 4 * m->P, m->stream));
  if (m->fused) {
    const NetShape& S = m->S;
    const int last = S.L - 1;  // the padding of the transposed head weights stays zero
    MLP_CUDA(cudaMemsetAsync(m->pt + S.t_off[last], 0, sizeof(__nv_bfloat16) * S.width * S.kp, m->stream));
    k_refresh<<<blocks(S.P, 256), 256, 0, m->stream>>>(S, m->p, m->pb, m->pt);
  } else {
    k_to_bf16<<<blocks((long long)m->P, 256), 256, 0, m->stream>>>(m->p, m->pb, (long long)m->P);
  }
  MLP_CUDA(cudaGetLastError());
  m->step = 0;
  MLP_CUDA(cudaStreamSynchronize(m->stream));
  return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp* m, float* params) {
  if (!m || !params) return LBM_EINVAL;
  lbm_status st = copy_out(m, params, m->p, 4 * m->P);
  if (st != LBM_OK) return st;
  MLP_CUDA(cudaStreamSynchronize(m->stream));
  return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp* m, const float* x, int batch, float* y) {
  if (!m || !x || !y || batch < 1 || batch > m->max_batch) return LBM_EINVAL;
  lbm_status st;
  if (m->fused) {
    const bool own = place_of(m, y) == IN_PLACE;  // the answers go straight to the caller's device memory
    st = fused_forward(m, x, batch, own ? y : m->y);
    if (st == LBM_OK && !own) st = copy_out(m, y, m->y, sizeof(float) * batch * m->n_out);
  } else {
    st = stage_inputs(m, x, nullptr, nullptr, batch);
    if (st == LBM_OK) st = forward(m, batch);
    if (st == LBM_OK) st = copy_out(m, y, m->y, sizeof(float) * batch * m->n_out);
  }
  if (st != LBM_OK) return st;
  MLP_CUDA(cudaStreamSynchronize(m->stream));
  return LBM_OK;
}

lbm_status lbm_mlp_loss_grad(lbm_mlp* m, const float* x, const float* target, const int* label, int batch,
                             float w_pos, float w_cls, float* loss, float* grad) {
  if (!m || !x || batch < 1 || batch > m->max_batch) return LBM_EINVAL;
  if ((m->n_pos > 0 && !target) || (m->n_cls > 0 && !label)) return LBM_EINVAL;
  lbm_status st;
  if (m->fused) {
    st = fused_backward(m, x, target, label, batch, w_pos, w_cls, -1.0f, 1.0f, 1.0f);
  } else {
    st = stage_inputs(m, x, target, label, batch);
    if (st == LBM_OK) st = backward(m, batch, w_pos, w_cls);
  }
  if (st == LBM_OK && grad) st = copy_out(m, grad, m->g, 4 * m->P);
  if (st != LBM_OK) return st;
  return finish_loss(m, loss);
}

lbm_status lbm_mlp_train_step(lbm_mlp* m, const float* x, const float* target, const int* label, int batch,
                              float w_pos, float w_cls, float lr, float* loss) {
  if (!m || !x || batch < 1 || batch > m->max_batch || !(lr >= 0.0f)) return LBM_EINVAL;
  if ((m->n_pos > 0 && !target) || (m->n_cls > 0 && !label)) return LBM_EINVAL;
  const long long step = m->step + 1;
  const float c1 = (float)(1.0 - pow(0.9, (double)step)), c2 = (float)(1.0 - pow(0.999, (double)step));
  lbm_status st;
  if (m->fused) {
    st = fused_backward(m, x, target, label, batch, w_pos, w_cls, lr, c1, c2);
    if (st != LBM_OK) return st;
    m->step = step;
  } else {
    st = stage_inputs(m, x, target, label, batch);
    if (st == LBM_OK) st = backward(m, batch, w_pos, w_cls);
    if (st != LBM_OK) return st;
    m->step = step;
    k_adam<<<blocks((long long)m->P, 256), 256, 0, m->stream>>>(m->p, m->g, m->m, m->v, m->pb, (long long)m->P, lr, c1,
                                                                 c2);
    MLP_CUDA(cudaGetLastError());
  }
  return finish_loss(m, loss);
}

void lbm_mlp_free(lbm_mlp* m) {
  if (!m) return;
  if (m->mem) cudaFree(m->mem);
  if (m->pinned) cudaFreeHost(m->pinned);
  delete m;
}

}  // extern "C"
