// Warm-rain surrogate network: 12 -> 256 -> 256 -> 256 -> 4, tanh hidden
// layers, BF16 weights and GEMM operands, FP32 accumulation on the tensor
// cores.  Training (forward, backward, Adam) and inference run on the
// kernels below; the step takes the network's rates where its inputs lie in
// the box spanned by the training data and the scheme's rates elsewhere.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "casim_device.cuh"
#include "casim_batch.cuh"
#include "casim_umma.cuh"

namespace casim_dev {

constexpr int kNin = 12, kNinPad = 16, kNh = 256, kNout = 4, kNoutPad = 16;
constexpr int kNParam = kNin * kNh + kNh + 2 * (kNh * kNh + kNh) + kNh * kNout + kNout;
// offsets of the layers in the flat parameter vector (oracle order)
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kNin * kNh, kOffW2 = kOffB1 + kNh, kOffB2 = kOffW2 + kNh * kNh,
              kOffW3 = kOffB2 + kNh, kOffB3 = kOffW3 + kNh * kNh, kOffW4 = kOffB3 + kNh,
              kOffB4 = kOffW4 + kNh * kNout;

// ------------------------------------------------------------ tensor-core GEMM
// C[m][n] = sum_k A(m, k) B(n, k) with A(m, k) = A[m*sam + k*sak] and
// B(n, k) = B[n*sbn + k*sbk] (BF16), FP32 accumulation by mma.sync
// m16n8k16.  Tiles of 64x64 over a 2x2 arrangement of warps; operands are
// gathered with arbitrary strides into k-contiguous shared-memory tiles, so
// one kernel serves the forward pass (W^T), the data gradient (W) and the
// weight gradient (both operands transposed).  The epilogue receives
// (m, n, acc) for m < M, n < N.
struct GemmArgs {
  const __nv_bfloat16 *A;
  long long sam, sak;
  const __nv_bfloat16 *B;
  long long sbn, sbk;
  int M, N, K;
  int kchunk;            // split K: block z sums k in [z kchunk, (z+1) kchunk)
};

constexpr int kGBM = 64, kGBN = 64, kGBK = 32, kGPad = 8;

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <class Epi>
__global__ void __launch_bounds__(128) k_gemm(const GemmArgs g, const Epi epi) {
  __shared__ __align__(16) __nv_bfloat16 As[kGBM][kGBK + kGPad];
  __shared__ __align__(16) __nv_bfloat16 Bs[kGBN][kGBK + kGPad];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 1, wn = warp & 1;
  const int m0 = blockIdx.y * kGBM, n0 = blockIdx.x * kGBN;
  const int gq = lane >> 2, tq = lane & 3;
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
  const __nv_bfloat16 zero = __float2bfloat16(0.f);
  const int kb = blockIdx.z * g.kchunk, ke = min(g.K, kb + g.kchunk);
  // gather order: consecutive threads along the operand's unit-stride index
  const bool a_rows = g.sam == 1 && g.sak != 1, b_rows = g.sbn == 1 && g.sbk != 1;
  for (int k0 = kb; k0 < ke; k0 += kGBK) {
#pragma unroll 4
    for (int i = tid; i < kGBM * kGBK; i += 128) {
      const int r = a_rows ? i % kGBM : i / kGBK, kk = a_rows ? i / kGBM : i % kGBK;
      const int m = m0 + r, k = k0 + kk;
      As[r][kk] = (m < g.M && k < ke) ? g.A[(long long)m * g.sam + (long long)k * g.sak] : zero;
    }
#pragma unroll 4
    for (int i = tid; i < kGBN * kGBK; i += 128) {
      const int r = b_rows ? i % kGBN : i / kGBK, kk = b_rows ? i / kGBN : i % kGBK;
      const int n = n0 + r, k = k0 + kk;
      Bs[r][kk] = (n < g.N && k < ke) ? g.B[(long long)n * g.sbn + (long long)k * g.sbk] : zero;
    }
    __syncthreads();
#pragma unroll
    for (int ks = 0; ks < kGBK; ks += 16) {
      uint32_t af[2][4], bf[4][2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = wm * 32 + i * 16 + gq;
        af[i][0] = *reinterpret_cast<const uint32_t *>(&As[r][ks + 2 * tq]);
        af[i][1] = *reinterpret_cast<const uint32_t *>(&As[r + 8][ks + 2 * tq]);
        af[i][2] = *reinterpret_cast<const uint32_t *>(&As[r][ks + 2 * tq + 8]);
        af[i][3] = *reinterpret_cast<const uint32_t *>(&As[r + 8][ks + 2 * tq + 8]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = wn * 32 + j * 8 + gq;
        bf[j][0] = *reinterpret_cast<const uint32_t *>(&Bs[r][ks + 2 * tq]);
        bf[j][1] = *reinterpret_cast<const uint32_t *>(&Bs[r][ks + 2 * tq + 8]);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int m = m0 + wm * 32 + i * 16 + gq + (r >> 1) * 8;
        const int n = n0 + wn * 32 + j * 8 + 2 * tq + (r & 1);
        if (m < g.M && n < g.N) epi(m, n, acc[i][j][r]);
      }
}

// Epilogues receive (m, n, acc) for m < M, n < N.  One with kLoad = true
// also reads a value per element (load(m, n)); the tensor-core GEMM issues
// those reads for a block of rows before it applies the epilogue
// (apply(m, n, acc, loaded)), so their latencies overlap.

// hidden layer: a = tanh(acc + b); keeps a (FP32, for the backward pass) and
// its BF16 copy (the next layer's input)
struct EpiHidden {
  static constexpr bool kLoad = false;
  const float *bias;
  float *a;              // [M][ld] or null
  __nv_bfloat16 *h;      // [M][ld]
  int ld;
  __device__ __forceinline__ void operator()(int m, int n, float acc) const {
    const float v = tanhf(acc + bias[n]);
    if (a) a[(long long)m * ld + n] = v;
    h[(long long)m * ld + n] = __float2bfloat16(v);
  }
};

// output layer: y = acc + b
struct EpiOut {
  static constexpr bool kLoad = false;
  const float *bias;
  float *y;              // [M][ld]
  int ld;
  __device__ __forceinline__ void operator()(int m, int n, float acc) const { y[(long long)m * ld + n] = acc + bias[n]; }
};

// masked squared error of one output: the gradient to dz (FP32 [n][4] and BF16
// [n][16]), the loss term returned.  Columns 4.. of the BF16 copy meet the zero
// columns of w4k in the data gradient; the kernels that write a row write them
// as zeros too, on the stream that reads them.
__device__ __forceinline__ double mlp_loss_term(float y, float t, float m, float cnt, float &g) {
  const float inv = 1.f / fmaxf(cnt, 1.f);
  const float d = (y - t) * m;
  g = 2.f * d * inv;
  return (double)d * d * inv;
}

// output layer of a training pass: y = acc + b, its loss term (summed over
// the rows by the GEMM) and gradient; y itself is not kept
struct EpiOutLoss {
  static constexpr bool kLoad = false;
  const float *bias, *T, *Mk, *cnt;
  double *loss;
  float *dz;
  __nv_bfloat16 *dzb;
  // the outputs of one row
  __device__ __forceinline__ double row(int m, const float *acc) const {
    const float4 t = reinterpret_cast<const float4 *>(T)[m], k = reinterpret_cast<const float4 *>(Mk)[m];
    const float tv[kNout] = {t.x, t.y, t.z, t.w}, kv[kNout] = {k.x, k.y, k.z, k.w}, c = *cnt;
    float g[kNout];
    __nv_bfloat16 h[kNout];
    double part = 0.0;
#pragma unroll
    for (int n = 0; n < kNout; ++n) {
      part += mlp_loss_term(acc[n] + bias[n], tv[n], kv[n], c, g[n]);
      h[n] = __float2bfloat16(g[n]);
    }
    reinterpret_cast<float4 *>(dz)[m] = make_float4(g[0], g[1], g[2], g[3]);
    __nv_bfloat162 lo, hi;
    lo.x = h[0]; lo.y = h[1]; hi.x = h[2]; hi.y = h[3];
    uint4 *d = reinterpret_cast<uint4 *>(dzb + (long long)m * kNoutPad);   // 32 bytes a row
    d[0] = make_uint4(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi), 0u, 0u);
    d[1] = make_uint4(0u, 0u, 0u, 0u);
    return part;
  }
};

// one chunk's partial weight gradient: c[m][n] = acc
struct EpiStore {
  static constexpr bool kLoad = false;
  float *c;
  int ld;
  __device__ __forceinline__ void operator()(int m, int n, float acc) const { c[(long long)m * ld + n] = acc; }
};

// split-K partial sums: ws[z][m][n] for block z
struct EpiPartial {
  static constexpr bool kLoad = false;
  float *ws;
  int ld;
  long long zstride;
  __device__ __forceinline__ void operator()(int m, int n, float acc) const {
    ws[blockIdx.z * zstride + (long long)m * ld + n] = acc;
  }
};

// data gradient through tanh: dz = acc (1 - a^2); FP32 for the bias sums,
// BF16 for the next GEMMs
struct EpiBackTanh {
  static constexpr bool kLoad = true;
  const float *a;        // [M][ld] activations of the layer below
  float *dz;
  __nv_bfloat16 *dzb;
  int ld;
  __device__ __forceinline__ float load(int m, int n) const { return __ldg(a + (long long)m * ld + n); }
  __device__ __forceinline__ void apply(int m, int n, float acc, float av) const {
    const long long i = (long long)m * ld + n;
    const float v = acc * (1.f - av * av);
    dz[i] = v;
    dzb[i] = __float2bfloat16(v);
  }
  __device__ __forceinline__ void operator()(int m, int n, float acc) const { apply(m, n, acc, load(m, n)); }
};

// ---------------------------------------------------------- elementwise kernels
// master FP32 parameters -> BF16 weight copies in both layouts:
//   Wt[l]: [N][K] (K padded with zeros) for the forward GEMM,
//   Wk[l]: [K][Npad] for the data gradient.
struct MlpBf16 {
  __nv_bfloat16 *w1t, *w2t, *w3t, *w4t;   // [256][16], [256][256], [256][256], [16][256]
  __nv_bfloat16 *w2k, *w3k, *w4k;         // [256][256], [256][256], [256][16]
};

__global__ void k_mlp_cast(const float *theta, MlpBf16 w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const __nv_bfloat16 z = __float2bfloat16(0.f);
  if (i < kNh * kNinPad) {   // w1t[n][k]
    const int n = i / kNinPad, k = i % kNinPad;
    w.w1t[i] = k < kNin ? __float2bfloat16(theta[kOffW1 + k * kNh + n]) : z;
  }
  if (i < kNh * kNh) {
    const int n = i / kNh, k = i % kNh;   // t-layout index i = n*256 + k
    w.w2t[i] = __float2bfloat16(theta[kOffW2 + k * kNh + n]);
    w.w3t[i] = __float2bfloat16(theta[kOffW3 + k * kNh + n]);
    w.w2k[i] = __float2bfloat16(theta[kOffW2 + i]);   // natural [k][n]
    w.w3k[i] = __float2bfloat16(theta[kOffW3 + i]);
  }
  if (i < kNoutPad * kNh) {  // w4t[n][k], n < 16 (rows >= 4 zero)
    const int n = i / kNh, k = i % kNh;
    w.w4t[i] = n < kNout ? __float2bfloat16(theta[kOffW4 + k * kNout + n]) : z;
  }
  if (i < kNh * kNoutPad) {  // w4k[k][n]
    const int k = i / kNoutPad, n = i % kNoutPad;
    w.w4k[i] = n < kNout ? __float2bfloat16(theta[kOffW4 + k * kNout + n]) : z;
  }
}

// FP32 inputs [n][12] -> BF16 [n][16] (zero padded)
__global__ void k_mlp_inputs(const float *X, int n, __nv_bfloat16 *h0) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)n * kNinPad) return;
  const long long r = i / kNinPad;
  const int k = (int)(i % kNinPad);
  h0[i] = __float2bfloat16(k < kNin ? X[r * kNin + k] : 0.f);
}

// masked squared error of the mma.sync engine's pass: loss += sum (y - t)^2 m / cnt and its gradient
__global__ void k_mlp_loss(const float *Y, const float *T, const float *Mk, int n, const float *cnt, double *loss,
                           float *dz, __nv_bfloat16 *dzb) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  double part = 0.0;
  if (i < (long long)n * kNout) {
    float g;
    part = mlp_loss_term(Y[i], T[i], Mk[i], *cnt, g);
    dz[i] = g;
    __nv_bfloat16 *row = dzb + i / kNout * kNoutPad + i % kNout;
    row[0] = __float2bfloat16(g);
#pragma unroll
    for (int j = kNout; j < kNoutPad; j += kNout) row[j] = __float2bfloat16(0.f);
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0 && part != 0.0) atomicAdd(loss, part);
}

__global__ void k_sum(const float *x, long long n, float *out) {
  float part = 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    part += x[i];
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, part);
}

// Weight gradients are summed over chunks of the batch (split K): chunk z of
// layer l's [M][N] gradient at ws[split * off[l] + z M N + i].  Bias
// gradients are column sums of dz over kColsumChunks row chunks.
constexpr int kSplitMax = 64;
constexpr int kColsumY = 32, kColsumChunks = 16;
constexpr int kColsumLen = 3 * kNh + kNout;   // columns of dz1, dz2, dz3, dz4
struct MlpGradWs {
  float *ws;       // [kSplitMax][kNin + 2 kNh + kNout][..]: W1, W2, W3, W4 one after another
  float *part;     // [kColsumChunks][kColsumLen]
  int nsplit;
};
// first element of layer l's partial sums, in units of one chunk of it
__host__ __device__ constexpr long long grad_ws_off(int l) {
  return l == 0 ? 0 : l == 1 ? kNin * kNh : l == 2 ? kNin * kNh + kNh * kNh : kNin * kNh + 2 * kNh * kNh;
}
constexpr long long kGradWsLen = kNin * kNh + 2 * kNh * kNh + kNh * kNout;

// Bias column sums, one block of 256 threads per 32 columns and row chunk:
// lane x is a column (coalesced rows), and each warp takes four of the
// chunk's 32 row phases; the 32 phase sums are added in a fixed order into
// part[chunk][column]; k_mlp_update adds the chunks in order (deterministic).
struct ColsumArgs {
  const float *dz[4];   // [n][256] of layers 1-3, [n][4] of layer 4
  int n;
  float *part;
};
constexpr int kColsumBlocks = (3 * kNh / 32 + 1) * kColsumChunks;
__global__ void __launch_bounds__(256) k_colsum(const ColsumArgs a) {
  __shared__ float s_part[kColsumY][33];
  pdl_trigger();
  pdl_wait();
  const int block = blockIdx.x;
  const int cb = block / kColsumChunks, chunk = block % kColsumChunks;
  const int l = cb / (kNh / 32), ld = l < 3 ? kNh : kNout;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, c = (l < 3 ? cb % (kNh / 32) * 32 : 0) + x;
  const float *dz = l == 0 ? a.dz[0] : l == 1 ? a.dz[1] : l == 2 ? a.dz[2] : a.dz[3];
  const int per = (a.n + kColsumChunks - 1) / kColsumChunks, r0 = chunk * per, r1 = min(a.n, r0 + per);
  float part[4] = {0.f, 0.f, 0.f, 0.f};
  if (c < ld) {
    const float *p = dz + c;
#pragma unroll 4
    for (int r = r0 + y; r < r1; r += kColsumY) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (r + 8 * j < r1) part[j] += p[(long long)(r + 8 * j) * ld];
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) s_part[y + 8 * j][x] = part[j];
  __syncthreads();
  if (y == 0 && c < ld) {
    float s = 0.f;
    for (int i = 0; i < kColsumY; ++i) s += s_part[i][x];
    a.part[(long long)chunk * kColsumLen + l * kNh + c] = s;
  }
}
struct AdamArgs {
  float *theta, *m1, *m2;   // theta null: the gradient only
  float lr, b1, b2, eps, c1, c2;
  MlpBf16 w;
  float *cnt, *hist;        // hist: this step's loss, or null
  double *loss;
};

// One parameter per thread: its gradient from the partial sums, in order
// (deterministic), then with Adam its new value and BF16 copies; the loss and
// the mask count are handed over and cleared for the next step.
__global__ void k_mlp_update(const MlpGradWs g, float *grad, const AdamArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (i == 0 && a.theta) {
    if (a.hist) *a.hist = (float)*a.loss;
    *a.loss = 0.0;
    *a.cnt = 0.f;
  }
  if (i >= kNParam) return;
  const int off[8] = {kOffW1, kOffB1, kOffW2, kOffB2, kOffW3, kOffB3, kOffW4, kOffB4};
  int t = 0, base = 0;   // 2 l: weights of layer l + 1, 2 l + 1: its biases
#pragma unroll
  for (int j = 1; j < 8; ++j)
    if (i >= off[j]) {
      t = j;
      base = off[j];
    }
  const int e = i - base, l = t >> 1;
  float s = 0.f;
  if (t & 1) {
    for (int y = 0; y < kColsumChunks; ++y) s += g.part[(long long)y * kColsumLen + l * kNh + e];
  } else {
    const long long len = l == 0 ? kNin * kNh : l == 3 ? kNh * kNout : kNh * kNh;
    const float *ws = g.ws + g.nsplit * (l == 0 ? grad_ws_off(0) : l == 1 ? grad_ws_off(1) : l == 2 ? grad_ws_off(2)
                                                                                                     : grad_ws_off(3)) + e;
#pragma unroll 32
    for (int z = 0; z < g.nsplit; ++z) s += ws[z * len];
  }
  grad[i] = s;
  if (!a.theta) return;
  const float x = a.b1 * a.m1[i] + (1.f - a.b1) * s;
  const float v = a.b2 * a.m2[i] + (1.f - a.b2) * s * s;
  a.m1[i] = x;
  a.m2[i] = v;
  const float th = a.theta[i] - a.lr * (x / a.c1) / (sqrtf(v / a.c2) + a.eps);
  a.theta[i] = th;
  if (t & 1) return;
  const __nv_bfloat16 h = __float2bfloat16(th);
  if (t == 0) {
    a.w.w1t[e % kNh * kNinPad + e / kNh] = h;
  } else if (t == 6) {
    a.w.w4t[e % kNout * kNh + e / kNout] = h;
    a.w.w4k[e / kNout * kNoutPad + e % kNout] = h;
  } else {
    (t == 2 ? a.w.w2t : a.w.w3t)[e % kNh * kNh + e / kNh] = h;
    (t == 2 ? a.w.w2k : a.w.w3k)[e] = h;
  }
}

// counter-based mini-batch sampling: row r of batch `step` is
// hash(seed, step, r) mod n (splitmix64 finaliser)
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// gather a standardised mini-batch from the raw data: 16 threads per row (the
// rows lie anywhere in the data; each is read by neighbouring threads), its
// BF16 inputs [B][16], targets, masks and the sum of the masks
__global__ void __launch_bounds__(256) k_mlp_batch(const float *X, const float *Y, const float *Mk, long long n,
                                                   unsigned long long seed, long long step, int B, const float *norm,
                                                   __nv_bfloat16 *h0, float *Tn, float *Mb, float *cnt) {
  __shared__ float s_cnt[256 / 32];
  pdl_trigger();
  pdl_wait();
  const long long i = blockIdx.x * 256ll + threadIdx.x;
  const int r = (int)(i / kNinPad), k = (int)(i % kNinPad);
  const float *mu = norm, *sd = norm + kNin, *muy = norm + 2 * kNin, *sdy = norm + 2 * kNin + kNout;
  float m = 0.f;
  if (r < B) {
    const long long src = (long long)(mix64(seed ^ mix64((unsigned long long)step * 0x100000001b3ull + r)) % (unsigned long long)n);
    h0[i] = __float2bfloat16(k < kNin ? (X[src * kNin + k] - mu[k]) / sd[k] : 0.f);
    if (k < kNout) {
      m = Mk[src * kNout + k];
      Mb[(long long)r * kNout + k] = m;
      Tn[(long long)r * kNout + k] = m > 0.f ? (Y[src * kNout + k] - muy[k]) / sdy[k] : 0.f;
    }
  }
  for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < 256 / 32; ++w) t += s_cnt[w];
    atomicAdd(cnt, t);
  }
}

// per-feature mean and standard deviation, per-target (masked) mean and
// standard deviation, per-feature min and max (the box of the training data)
__global__ void __launch_bounds__(256) k_mlp_stats(const float *X, const float *Y, const float *Mk, long long n, double *acc) {
  // acc: [12 sum][12 sumsq][4 sum][4 sumsq][4 count] then min/max as ordered ints elsewhere
  double s[kNin] = {0}, q[kNin] = {0}, sy[kNout] = {0}, qy[kNout] = {0}, cy[kNout] = {0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int k = 0; k < kNin; ++k) {
      const double v = X[i * kNin + k];
      s[k] += v;
      q[k] += v * v;
    }
#pragma unroll
    for (int c = 0; c < kNout; ++c)
      if (Mk[i * kNout + c] > 0.f) {
        const double v = Y[i * kNout + c];
        sy[c] += v;
        qy[c] += v * v;
        cy[c] += 1.0;
      }
  }
  // the block's sums, one atomic per block and sum: with one per thread,
  // 65 536 of them queued on each of the 36 addresses, and the kernel took
  // 1.54 ms for 262 144 rows
  __shared__ double s_sum[256 / 32][2 * kNin + 3 * kNout];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto put = [&](int at, double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_sum[warp][at] = v;
  };
#pragma unroll
  for (int k = 0; k < kNin; ++k) {
    put(k, s[k]);
    put(kNin + k, q[k]);
  }
#pragma unroll
  for (int c = 0; c < kNout; ++c) {
    put(2 * kNin + c, sy[c]);
    put(2 * kNin + kNout + c, qy[c]);
    put(2 * kNin + 2 * kNout + c, cy[c]);
  }
  __syncthreads();
  if (threadIdx.x < 2 * kNin + 3 * kNout) {
    double v = 0.0;
    for (int w = 0; w < 256 / 32; ++w) v += s_sum[w][threadIdx.x];
    atomicAdd(&acc[threadIdx.x], v);
  }
}

// order-preserving float <-> int mapping for atomic min/max
__device__ __forceinline__ int f2ord(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float ord2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__global__ void k_mlp_box(const float *X, long long n, int *lo, int *hi) {
  int l[kNin], h[kNin];
#pragma unroll
  for (int k = 0; k < kNin; ++k) {
    l[k] = 0x7fffffff;
    h[k] = -0x7fffffff;
  }
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
#pragma unroll
    for (int k = 0; k < kNin; ++k) {
      const int v = f2ord(X[i * kNin + k]);
      l[k] = min(l[k], v);
      h[k] = max(h[k], v);
    }
#pragma unroll
  for (int k = 0; k < kNin; ++k) {
    atomicMin(&lo[k], l[k]);
    atomicMax(&hi[k], h[k]);
  }
}

// ------------------------------------------------------ features and targets
// The 12 features of a post-activation point (natural logarithms).
__device__ __forceinline__ void mlp_features(const ConstK<float> &K, const W<float> &w, float na, float wv,
                                             float f[kNin]) {
  const float ln2 = 0.693147180559945309f;
  f[0] = lg2a(fmaxf(w.qc, K.qmin)) * ln2;
  f[1] = lg2a(fmaxf(w.qr, K.qmin)) * ln2;
  f[2] = lg2a(fmaxf(w.nc, 1.f)) * ln2;
  f[3] = lg2a(fmaxf(w.nr, 1e-3f)) * ln2;
  f[4] = lg2a(w.rho) * ln2;
  f[5] = w.tc;
  f[6] = lg2a(w.p) * ln2;
  f[7] = lg2a(fmaxf(w.qv, 1e-10f)) * ln2;
  f[8] = wv;
  f[9] = lg2a(fmaxf(na, 1.f)) * ln2;
  f[10] = w.qc > K.qmin ? 1.f : 0.f;
  f[11] = w.qr > K.qmin ? 1.f : 0.f;
}

struct FeatArgs {
  int mode;               // 0: training data (raw features, log-rates, masks); 1: inference rows
  long long cap;          // rows available
  unsigned long long *rows;   // row counter
  float *X, *Y, *M;       // mode 0: [cap][12], [cap][4], [cap][4]
  __nv_bfloat16 *xb;      // mode 1: [cap][16] standardised BF16 features
  long long *rowpt;       // point index (k * pitch + c) of each row (mode 0: optional)
  float4 *surr;           // mode 1: [nlev][pitch]; NaN written where the point is outside the box
  const float *norm;      // mode 1: means and deviations of the features
  const float *box;       // mode 1: [12 lo][12 hi]
};

// The features of one point (index pt of its domain's [nlev][pitch] grid;
// gpt: its index in the rates array, which is pt for one domain): adjustment
// and activation as the mixed step does them, then the point's features (and,
// for training data, the scheme's four log-rates).  warm: the point gets a row.
__device__ __forceinline__ void feature_point(const KArgs &a, const KParams &P, const FeatArgs &fa, long long pt,
                                              long long gpt, bool &warm, float f[kNin], float y[kNout],
                                              float mk[kNout]) {
  const long long np = (long long)a.nlev * a.pitch;
  if (pt < np) {
    const int c = (int)(pt % a.pitch);
    if (c < a.ncols) {
      const ConstK<float> &K = P.f;
      Pt s;
      const double *b = a.fld + pt;
      const size_t fs = (size_t)a.nlev * (size_t)a.pitch;
      s.T = b[0]; s.qv = b[1 * fs]; s.qc = b[2 * fs]; s.qr = b[3 * fs];
      s.qi = b[4 * fs]; s.qs = b[5 * fs]; s.qg = b[6 * fs];
      s.p = b[13 * fs];
      W<float> w;
      float es0, qs0;
      if (Mix::active(K, s, P.T0, w, es0, qs0)) {
        s.nc = b[7 * fs]; s.nr = b[8 * fs]; s.ni = b[9 * fs]; s.ns = b[10 * fs]; s.ng = b[11 * fs];
        s.na = b[12 * fs]; s.rho = b[14 * fs]; s.w = b[15 * fs];
        MixInc o;
        const float dn = Mix::pre(K, s, w, es0, qs0, o);
        warm = w.qc > K.qmin || w.qr > K.qmin;
        if (warm) {
          mlp_features(K, w, d2f(s.na) - dn, d2f(s.w), f);
          if (fa.mode == 0) {
            Rt<float> r;
            Phys<PolicyMix>::rates(K, w, a.dt, r);
            const bool hc = w.qc > K.qmin, hr = w.qr > K.qmin;
            const float v[kNout] = {r.aut, r.acc, r.scc, r.scr};
            const bool def[kNout] = {hc, hc && hr, hc, hr};
#pragma unroll
            for (int j = 0; j < kNout; ++j)
              if (def[j] && v[j] > 0.f) {
                y[j] = lg2a(v[j]) * 0.693147180559945309f;
                mk[j] = 1.f;
              }
          } else {
            bool inbox = true;
#pragma unroll
            for (int j = 0; j < kNin; ++j) inbox &= f[j] >= fa.box[j] && f[j] <= fa.box[kNin + j];
            if (!inbox) {
              fa.surr[gpt] = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
              warm = false;
            }
          }
        }
      }
    }
  }
}

// Block-aggregated append of the rows: one atomic on the row counter per
// block (a counter that every warp hits serialises in L2), the warps' offsets
// from a prefix sum of their counts; rows come in no set order (each carries
// its point, gpt).  Every thread of the block calls it.
__device__ __forceinline__ void feature_append(const FeatArgs &fa, bool warm, long long gpt, const float f[kNin],
                                               const float y[kNout], const float mk[kNout]) {
  __shared__ unsigned s_off[256 / 32];
  __shared__ unsigned long long s_base;
  const unsigned ball = __ballot_sync(0xffffffffu, warm);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) s_off[wid] = __popc(ball);
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned tot = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
      const unsigned t = s_off[i];
      s_off[i] = tot;
      tot += t;
    }
    s_base = tot ? atomicAdd(fa.rows, (unsigned long long)tot) : 0ull;
  }
  __syncthreads();
  if (!warm) return;
  const long long row = (long long)(s_base + s_off[wid]) + __popc(ball & ((1u << lane) - 1u));
  if (row >= fa.cap) return;   // the caller sees rows > cap and reports it
  if (fa.mode == 0) {
    if (fa.rowpt) fa.rowpt[row] = gpt;
#pragma unroll
    for (int j = 0; j < kNin; ++j) fa.X[row * kNin + j] = f[j];
#pragma unroll
    for (int j = 0; j < kNout; ++j) {
      fa.Y[row * kNout + j] = y[j];
      fa.M[row * kNout + j] = mk[j];
    }
  } else {
    __align__(16) __nv_bfloat16 hb[kNinPad];
#pragma unroll
    for (int j = 0; j < kNinPad; ++j)
      hb[j] = __float2bfloat16(j < kNin ? (f[j] - fa.norm[j]) / fa.norm[kNin + j] : 0.f);
    uint4 *dst = reinterpret_cast<uint4 *>(fa.xb + row * kNinPad);
    dst[0] = reinterpret_cast<const uint4 *>(hb)[0];
    dst[1] = reinterpret_cast<const uint4 *>(hb)[1];
    fa.rowpt[row] = gpt;
  }
}

// One thread per point of a domain.
__global__ void __launch_bounds__(256) k_mlp_features(const KArgs a, const KParams P, const FeatArgs fa) {
  const long long pt = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  bool warm = false;
  float f[kNin];
  float y[kNout] = {0, 0, 0, 0}, mk[kNout] = {0, 0, 0, 0};
  feature_point(a, P, fa, pt, pt, warm, f, y, mk);
  feature_append(fa, warm, pt, f, y, mk);
}

// One thread per point of every domain of a batch: the points of domain d
// are [dom[d].pt_off, dom[d].pt_off + nlev pitch) of the batch's rates array
// (a binary search over the domains' offsets finds a thread's domain).
__global__ void __launch_bounds__(256) k_mlp_features_batch(const DomDesc *dom, int ndom, long long total,
                                                            double dt, const KParams P, const FeatArgs fa) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  bool warm = false;
  float f[kNin];
  float y[kNout] = {0, 0, 0, 0}, mk[kNout] = {0, 0, 0, 0};
  if (g < total) {
    int lo = 0, hi = ndom - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (dom[mid].pt_off <= g) lo = mid;
      else hi = mid - 1;
    }
    const DomDesc d = dom[lo];
    KArgs a;
    a.fld = d.fld;
    a.pitch = d.pitch;
    a.dz = d.dz;
    a.precip = d.precip;
    a.err = nullptr;
    a.ncols = d.ncols;
    a.nlev = d.nlev;
    a.dt = dt;
    a.surr = nullptr;
    a.stats = nullptr;
    a.segs = 1;
    feature_point(a, P, fa, g - d.pt_off, g, warm, f, y, mk);
  }
  feature_append(fa, warm, g, f, y, mk);
}

// network outputs (standardised log-rates) -> rates at the rows' points
__global__ void k_mlp_scatter(const float *Yn, long long rows, const long long *rowpt, const float *norm,
                              float4 *surr, long long npts, unsigned *err) {
  const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (r >= rows) return;
  if (!CASIM_INDEX_OK(rowpt[r] >= 0 && rowpt[r] < npts, err)) return;
  const float *muy = norm + 2 * kNin, *sdy = norm + 2 * kNin + kNout;
  float v[kNout];
#pragma unroll
  for (int j = 0; j < kNout; ++j) v[j] = __expf(Yn[r * kNout + j] * sdy[j] + muy[j]);
  surr[rowpt[r]] = make_float4(v[0], v[1], v[2], v[3]);
}

}  // namespace casim_dev

// ------------------------------------------------ tcgen05 inference kernel

namespace casim_dev {

// Weight images in global memory, already in the swizzled shared-memory
// layout, so that 1-D bulk copies land them ready for the tensor cores:
//   W1: [256 rows][16] (k >= 12 zero), 32-byte swizzle               8 KB
//   W2, W3: per K-step of 16 an image like W1's, 16 steps each      8 KB a step
//   W4: [16 rows][256] (rows >= 4 zero)                               8 KB
// K-steps per ring stage: two (16 KB, four stages).  On the rows stated at the
// kernel: 1020 us with two, 1090 with four (two stages only: a copy of
// 32 KB is not covered), 1440 with one (a wait and a commit for every MMA).
constexpr int kUmmaSteps = 2;
constexpr uint32_t kImgStep = 256 * 32;
constexpr uint32_t kImgW1 = 256 * 32, kImgChunk = kUmmaSteps * kImgStep, kImgW4 = 16 * 4 * 128;
constexpr int kImgChunks = 32 / kUmmaSteps;
constexpr uint32_t kImgBytes = kImgW1 + kImgChunks * kImgChunk + kImgW4;

__global__ void k_mlp_images(const float *theta, unsigned char *img) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const __nv_bfloat16 z = __float2bfloat16(0.f);
  if (i < 256 * 16) {   // W1 (n, k)
    const int n = i / 16, k = i % 16;
    *reinterpret_cast<__nv_bfloat16 *>(img + sw32_offset(n, k)) =
        k < kNin ? __float2bfloat16(theta[kOffW1 + k * kNh + n]) : z;
  }
  if (i < 256 * 256) {  // W2, W3 (n, k)
    const int n = i / 256, k = i % 256;
    const uint32_t off = (uint32_t)(k >> 4) * kImgStep + sw32_offset(n, k & 15);
    *reinterpret_cast<__nv_bfloat16 *>(img + kImgW1 + off) = __float2bfloat16(theta[kOffW2 + k * kNh + n]);
    *reinterpret_cast<__nv_bfloat16 *>(img + kImgW1 + 16 * kImgStep + off) = __float2bfloat16(theta[kOffW3 + k * kNh + n]);
  }
  if (i < 16 * 256) {   // W4 (n, k)
    const int n = i / 256, k = i % 256;
    *reinterpret_cast<__nv_bfloat16 *>(img + kImgW1 + kImgChunks * kImgChunk + sw128_offset(16, n, k)) =
        n < kNout ? __float2bfloat16(theta[kOffW4 + k * kNout + n]) : z;
  }
}

struct UmmaArgs {
  const __nv_bfloat16 *xb;     // [rows][16] standardised features
  long long rows;              // rows, or the capacity when rows_dev is set
  const unsigned long long *rows_dev;   // if set: the row count, read on the device (at most rows)
  const long long *rowpt;      // point of each row (null: write Y rows instead)
  const unsigned char *img;    // weight images
  const float *theta;          // biases are read from the flat parameters
  const float *norm;           // output standardisation
  float4 *surr;                // rates at the points
  long long npts;              // points of surr (the rows' point indices are below it)
  float *y;                    // [rows][4] standardised outputs when rowpt is null
  unsigned *err;
};

constexpr unsigned kUmmaSpins = 1u << 22;
constexpr int kUmmaEpiWarps = 16;                       // 4 per TMEM lane quarter
constexpr int kUmmaMmaWarp = kUmmaEpiWarps;             // issues the MMAs, owns TMEM
constexpr int kUmmaProdWarp = kUmmaEpiWarps + 1;        // streams the weight chunks
constexpr int kUmmaThreads = (kUmmaEpiWarps + 2) * 32;
constexpr int kUmmaStages = 8 / kUmmaSteps;                          // weight-chunk ring
// dynamic shared memory (1024-byte aligned): resident W1 and W4, the features
// and activations of two tiles, the chunk ring
constexpr uint32_t kUmmaFeat = 128 * 32, kUmmaAct = 4 * 128 * 128;
constexpr uint32_t kSmW1 = 0, kSmW4 = kSmW1 + kImgW1, kSmFeat = kSmW4 + kImgW4, kSmAct = kSmFeat + 2 * kUmmaFeat,
                   kSmRing = kSmAct + 2 * kUmmaAct;
constexpr int kUmmaSmem = 1024 + kSmRing + kUmmaStages * kImgChunk;
static_assert(kUmmaSmem + 4096 <= 232448, "shared memory of the tensor-core kernel");

// Persistent, one CTA (18 warps) per SM, 128-row tiles, two in flight.
//
// What bounds it is tanh: 98 304 per 128-row tile at 16 per SM and clock are
// 6.1 k cycles; the MMAs need 4.4 k.  Each tile has a 256-column FP32
// accumulator of its own in tensor memory; the BF16 activations go to shared
// memory, so that the next layer's sums can replace this layer's in the same
// columns.  While the epilogue warps work on one tile's layer, the other
// tile's next layer is multiplied:
//  * epilogue warps (16): for each layer, tile by tile, warp w reads lanes
//    32(w%4).. (its rows) and the 64 columns of slab w/4: bias, tanh, BF16
//    pack, to the activation slab; then one arrival on the tile's act barrier;
//  * MMA warp (one thread): once a tile's activations are complete, the next
//    layer's MMAs (N = 256, A and B in shared memory, weights from the ring)
//    into the same accumulator, then a commit to the tile's acc barrier;
//  * producer warp (one thread): streams the weights of layers 2-3 for each
//    tile through the ring (full/free barriers), 256 KB of L2 reads per tile.
// 3.6 million rows (28 k tiles, 186 per SM): 1.02 ms; one tile in flight, with the activations in tensor memory
// and the next layer's MMAs behind the epilogue slab by slab, took 1.20 ms.
// The epilogue alone takes 0.88 ms, the MMAs alone 0.51.  Tried and slower:
// eight warps for each tile instead of all for one (1.10), the second tile two
// layers behind the first (1.17).
// Every wait is bounded and gives up once any thread of the CTA has set the
// abort flag; before the tensor memory is released and the CTA leaves, all
// MMAs, copies and arrivals from or to this CTA have completed.
__global__ void __launch_bounds__(kUmmaThreads, 1) k_mlp_umma(const UmmaArgs u) {
  extern __shared__ __align__(16) unsigned char sraw[];
  unsigned char *sm = sraw + ((1024 - (smem_addr(sraw) & 1023)) & 1023);
  __shared__ float s_bias[3 * kNh + kNout];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) unsigned long long s_bar[8 + 2 * kUmmaStages];
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long nrows = u.rows_dev ? min((long long)*u.rows_dev, u.rows) : u.rows;
  const long long ntiles = (nrows + 127) / 128;
  const long long cta = blockIdx.x, ncta = gridDim.x;
  const long long my_tiles = cta < ntiles ? (ntiles - 1 - cta) / ncta + 1 : 0;   // tiles cta, cta + ncta, ..
  const uint32_t sb = smem_addr(sm);
  volatile int *abort = &s_abort;
  // per tile slot t = 0, 1: features ready, accumulator ready, activations ready
  enum { B_W = 0, B_FEAT = 1, B_ACC = 3, B_ACT = 5, B_FULL = 7, B_FREE = 7 + kUmmaStages, B_DRAIN = 7 + 2 * kUmmaStages };
  const uint32_t bar0 = smem_addr(&s_bar[0]);
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  auto fail = [&]() {
    *abort = 1;
    atomicOr(u.err, 4u);
  };

  for (int i = tid; i < kNh; i += kUmmaThreads) {
    s_bias[i] = u.theta[kOffB1 + i];
    s_bias[kNh + i] = u.theta[kOffB2 + i];
    s_bias[2 * kNh + i] = u.theta[kOffB3 + i];
  }
  if (tid < kNout) s_bias[3 * kNh + tid] = u.theta[kOffB4 + tid];
  if (warp == kUmmaMmaWarp) {
    tmem_alloc(smem_addr(&s_tmem), 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    bar_init(bar(B_W), 1);
    for (int t = 0; t < 2; ++t) {
      // all warps, so that none can be a whole phase of ACC behind when the
      // next tile's layer 1 is issued
      bar_init(bar(B_FEAT + t), kUmmaEpiWarps);
      bar_init(bar(B_ACC + t), 1);
      bar_init(bar(B_ACT + t), kUmmaEpiWarps);
    }
    for (int s = 0; s < kUmmaStages; ++s) {
      bar_init(bar(B_FULL + s), 1);
      bar_init(bar(B_FREE + s), 1);
    }
    bar_init(bar(B_DRAIN), 1);
    bar_fence_init();
    s_abort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = s_tmem;

  if (warp == kUmmaProdWarp) {
    if (lane == 0) {
      bar_expect_tx(bar(B_W), kImgW1 + kImgW4);
      bulk_load(sb + kSmW1, u.img, kImgW1, bar(B_W));
      bulk_load(sb + kSmW4, u.img + kImgW1 + kImgChunks * kImgChunk, kImgW4, bar(B_W));
      // the MMA warp takes, per pair of tiles, layer 2's four chunks for each
      // tile and then layer 3's.  Load i goes to stage i % S as that stage's
      // (i / S)-th fill; from the second fill on it waits until the MMAs of
      // the previous fill have completed
      constexpr int kL = kImgChunks / 2;   // chunks per layer
      uint32_t i = 0;
      bool ok = true;
      for (long long it = 0; ok && it < my_tiles; it += 2) {
        const int ntp = my_tiles - it >= 2 ? 2 : 1;
        for (int l = 0; ok && l < 2; ++l)
          for (int t = 0; ok && t < ntp; ++t) {
            const unsigned char *src = u.img + kImgW1 + (uint32_t)l * (kL * kImgChunk);
#pragma unroll
            for (int s = 0; s < kL; ++s, ++i) {
              const uint32_t st = i % kUmmaStages, fill = i / kUmmaStages;
              ok = ok && (fill == 0 || bar_wait_or_abort(bar(B_FREE + (int)st), (fill - 1) & 1u, kUmmaSpins, abort));
              if (!ok) break;
              bar_expect_tx(bar(B_FULL + (int)st), kImgChunk);
              bulk_load(sb + kSmRing + st * kImgChunk, src + (uint32_t)s * kImgChunk, kImgChunk, bar(B_FULL + (int)st));
            }
          }
      }
      if (!ok) fail();
      // drain: the copies into this CTA have landed (last fill of each
      // stage), and so have the commits of those fills
      bar_wait(bar(B_W), 0, kUmmaSpins);
      for (uint32_t st = 0; st < kUmmaStages && st < i; ++st) {
        const uint32_t fills = (i - st + kUmmaStages - 1) / kUmmaStages;
        bar_wait(bar(B_FULL + (int)st), (fills - 1) & 1u, kUmmaSpins);
        bar_wait_or_abort(bar(B_FREE + (int)st), (fills - 1) & 1u, kUmmaSpins, abort);
      }
    }
    __syncwarp();
  } else if (warp == kUmmaMmaWarp) {
    if (lane == 0) {
      const uint32_t id256 = umma_idesc_bf16(128, 256), id16 = umma_idesc_bf16(128, 16);
      bool ok = bar_wait_or_abort(bar(B_W), 0, kUmmaSpins, abort);
      uint32_t nfeat[2] = {0, 0}, nact[2] = {0, 0};
      uint32_t chunk = 0;
      // the descriptors' addresses are in units of 16 bytes and shared memory
      // ends below 2^18: an offset is a plain addition
      const uint64_t dact = umma_desc_sw128(sb + kSmAct), dring = umma_desc_sw32(sb + kSmRing);
      for (long long it = 0; ok && it < my_tiles; it += 2) {
        const int ntp = my_tiles - it >= 2 ? 2 : 1;
        // layer 1: features x W1
        for (int t = 0; ok && t < ntp; ++t) {
          ok = bar_wait_or_abort(bar(B_FEAT + t), nfeat[t]++ & 1u, kUmmaSpins, abort);
          if (!ok) break;
          tc_fence_after();
          umma_bf16(taddr + 256u * (uint32_t)t, umma_desc_sw32(sb + kSmFeat + (uint32_t)t * kUmmaFeat),
                    umma_desc_sw32(sb + kSmW1), id256, 0u);
          umma_commit(bar(B_ACC + t));
        }
        // layers 2 and 3, K-slab by K-slab as the weights land
        for (int l = 0; ok && l < 2; ++l)
          for (int t = 0; ok && t < ntp; ++t) {
            ok = bar_wait_or_abort(bar(B_ACT + t), nact[t]++ & 1u, kUmmaSpins, abort);
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = dact + (uint64_t)(t * (kUmmaAct >> 4));
#pragma unroll
            for (int s = 0; s < 16; s += kUmmaSteps, ++chunk) {
              const uint32_t st = chunk % kUmmaStages;
              ok = ok && bar_wait_or_abort(bar(B_FULL + (int)st), (chunk / kUmmaStages) & 1u, kUmmaSpins, abort);
              if (!ok) break;
              tc_fence_after();
              const uint64_t dw = dring + (uint64_t)(st * (kImgChunk >> 4));
#pragma unroll
              for (int sub = 0; sub < kUmmaSteps; ++sub) {
                const int k = s + sub;   // K elements 16 k ..
                umma_bf16(taddr + 256u * (uint32_t)t, da + (uint64_t)((16384 * (k >> 2) + 32 * (k & 3)) >> 4),
                          dw + (uint64_t)((kImgStep * sub) >> 4), id256, k ? 1u : 0u);
              }
              umma_commit(bar(B_FREE + (int)st));
            }
            if (ok) umma_commit(bar(B_ACC + t));
          }
        // layer 4: columns 0..15 of the tile's accumulator
        for (int t = 0; ok && t < ntp; ++t) {
          ok = bar_wait_or_abort(bar(B_ACT + t), nact[t]++ & 1u, kUmmaSpins, abort);
          if (!ok) break;
          tc_fence_after();
          const uint64_t da = dact + (uint64_t)(t * (kUmmaAct >> 4)), dw = umma_desc_sw128(sb + kSmW4);
#pragma unroll
          for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int sub = 0; sub < 4; ++sub)
              umma_bf16(taddr + 256u * (uint32_t)t, da + (uint64_t)((16384 * s + 32 * sub) >> 4),
                        dw + (uint64_t)((2048 * s + 32 * sub) >> 4), id16,
                        (s | sub) ? 1u : 0u);
          umma_commit(bar(B_ACC + t));
        }
      }
      if (!ok) fail();
      // drain: every MMA this thread issued has completed
      umma_commit(bar(B_DRAIN));
      bar_wait(bar(B_DRAIN), 0, kUmmaSpins);
    }
    __syncwarp();
  } else {
    // epilogue warps
    const int q = warp & 3, j = warp >> 2;
    const int row = 32 * q + lane;
    const uint32_t rowx = (uint32_t)(row & 7) << 4;   // the 128-byte swizzle of this row
    uint32_t nacc[2] = {0, 0};
    bool ok = true;
    uint4 f0[2], f1[2];
    // tile n of this CTA: its rows' features into registers, then (put) shared memory
    auto load_features = [&](long long n, int t) {
      f0[t] = make_uint4(0, 0, 0, 0);
      f1[t] = f0[t];
      const long long r = (cta + n * ncta) * 128 + row;
      if (n < my_tiles && r < nrows) {
        const uint4 *src = reinterpret_cast<const uint4 *>(u.xb + r * kNinPad);
        f0[t] = src[0];
        f1[t] = src[1];
      }
    };
    auto put_features = [&](int t) {
      if (j == 0) {
        unsigned char *p = sm + kSmFeat + (uint32_t)t * kUmmaFeat;
        *reinterpret_cast<uint4 *>(p + sw32_offset(row, 0)) = f0[t];
        *reinterpret_cast<uint4 *>(p + sw32_offset(row, 8)) = f1[t];
        fence_async_smem();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(bar(B_FEAT + t));
    };
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (j == 0) load_features(t, t);
      if (t < my_tiles) put_features(t);
    }
    for (long long it = 0; ok && it < my_tiles; it += 2) {
      const int ntp = my_tiles - it >= 2 ? 2 : 1;
      if (j == 0) {
#pragma unroll
        for (int t = 0; t < 2; ++t) load_features(it + 2 + t, t);
      }
      for (int l = 0; ok && l < 3; ++l) {
        const float *b = s_bias + l * kNh;
        for (int t = 0; t < ntp; ++t) {
          const uint32_t ph = t == 0 ? nacc[0]++ : nacc[1]++;
          ok = bar_wait_or_abort(bar(B_ACC + t), ph & 1u, kUmmaSpins, abort);
          if (!ok) break;
          tc_fence_after();
          // this warp's slab, 32 columns at a time: the second load is in
          // flight while the first half is worked on
          const uint32_t tacc = taddr + 256u * (uint32_t)t + ((uint32_t)(32 * q) << 16) + 64u * (uint32_t)j;
          unsigned char *act = sm + kSmAct + (uint32_t)t * kUmmaAct + 16384u * (uint32_t)j + 128u * (uint32_t)row;
          uint32_t v[2][32];
          tmem_ld32(tacc, v[0]);
          tmem_wait32(v[0]);
          tmem_ld32(tacc + 32u, v[1]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (h == 1) tmem_wait32(v[1]);
#pragma unroll
            for (int c = 0; c < 4; ++c) {   // 8 columns, one 16-byte chunk of the row
              const float *bc = b + 64 * j + 32 * h + 8 * c;
              uint32_t hb[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 p =
                    __floats2bfloat162_rn(tanh_approx(__uint_as_float(v[h][8 * c + 2 * i]) + bc[2 * i]),
                                          tanh_approx(__uint_as_float(v[h][8 * c + 2 * i + 1]) + bc[2 * i + 1]));
                hb[i] = *reinterpret_cast<const uint32_t *>(&p);
              }
              *reinterpret_cast<uint4 *>(act + ((uint32_t)((4 * h + c) << 4) ^ rowx)) =
                  make_uint4(hb[0], hb[1], hb[2], hb[3]);
            }
          }
          fence_async_smem();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) bar_arrive(bar(B_ACT + t));
        }
      }
      if (!ok) break;
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (t >= ntp) break;
        ok = bar_wait_or_abort(bar(B_ACC + t), (t == 0 ? nacc[0]++ : nacc[1]++) & 1u, kUmmaSpins, abort);
        if (!ok) break;
        tc_fence_after();
        float v[16];
        if (j == 0) tmem_ld16(taddr + 256u * (uint32_t)t + ((uint32_t)(32 * q) << 16), v);
        if (it + 2 + t < my_tiles) put_features(t);   // the accumulator is free: the slot's next tile
        if (j == 0) {
          const long long r = (cta + (it + t) * ncta) * 128 + row;
          if (r < nrows) {
            float y[kNout];
#pragma unroll
            for (int i = 0; i < kNout; ++i) y[i] = v[i] + s_bias[3 * kNh + i];
            if (u.rowpt && CASIM_INDEX_OK(u.rowpt[r] >= 0 && u.rowpt[r] < u.npts, u.err)) {
              const float *muy = u.norm + 2 * kNin, *sdy = u.norm + 2 * kNin + kNout;
              u.surr[u.rowpt[r]] = make_float4(__expf(y[0] * sdy[0] + muy[0]), __expf(y[1] * sdy[1] + muy[1]),
                                               __expf(y[2] * sdy[2] + muy[2]), __expf(y[3] * sdy[3] + muy[3]));
            } else {
#pragma unroll
              for (int i = 0; i < kNout; ++i) u.y[r * kNout + i] = y[i];
            }
          }
        }
      }
    }
    if (!ok) fail();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kUmmaMmaWarp) tmem_dealloc(taddr, 512);
}


// ------------------------------------------------ tcgen05 training GEMM
// The training GEMMs of the network on the fifth-generation tensor cores:
// C[m][n] = sum_k A(m, k) B(n, k), operands BF16 with the strides of
// GemmArgs, FP32 accumulators in tensor memory, the same fused epilogues as
// k_gemm.  Each operand is K-major (unit stride along k: the forward pass and
// the data gradients) or MN-major (unit stride along m or n: the weight
// gradients, whose k runs over the batch); both are staged by 16-byte
// asynchronous copies in the 128-byte-swizzled slabs of that major-ness, which
// the MMA reads as they are.
//
// A tile is 128 x 64, one CTA of 8 warps, two CTAs per SM.  These GEMMs are a
// microsecond of tensor work behind a chain of latencies (operands, MMAs,
// epilogue), so the whole depth of up to 256 is loaded at once, in slabs of 64
// whose MMAs follow as they land, and small tiles put every SM to work: with
// 128 x 128 tiles of 4 warps and two slabs in flight a hidden layer took 24 us
// on 8192 rows and a data gradient 36 us, now 12 us each; the weight
// gradients, one launch of 23 us per layer with 128 x 128 tiles transposed
// through registers, take 18 us in one launch for all four (all by ncu, cold
// caches).  A training step on 8192 rows: 0.33 -> 0.094 ms.
// One thread issues the MMAs (M = 128, N = the
// tile's columns rounded up to 16, K = 16 each).  Epilogue: warp w reads
// tensor-memory lanes 32 (w % 4).. (its rows) and 32 columns, and passes the
// 32 x 32 block through shared memory (the operand slabs, free once the last
// MMA completed) so that the epilogue's loads and stores run along n,
// coalesced.  A wait that gives up sets error bit 4, waits again for the MMAs
// it issued and releases the tensor memory.
constexpr int kTcBM = 128, kTcBN = 64, kTcBK = 64, kTcSlabs = 4;
constexpr int kTcThreads = 256;
constexpr uint32_t kTcSlabA = kTcBM * kTcBK * 2, kTcSlabB = kTcBN * kTcBK * 2;   // 16 KB, 8 KB
constexpr int kTcSmem = 1024 + kTcSlabs * (int)(kTcSlabA + kTcSlabB);            // 1024-byte alignment
constexpr unsigned kTcSpins = 1u << 24;

// 16-byte asynchronous copy global -> shared; ok false: zeros (src not read)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// slab `s` (k0 .. k0 + 63 of [.., ke)) of a K-major operand of R rows r0..: asynchronous copies
template <int R>
__device__ __forceinline__ void tc_load_kmajor(uint32_t dst, const __nv_bfloat16 *P, long long srow, int nrows, int r0,
                                               int k0, int ke, int tid) {
#pragma unroll
  for (int j = 0; j < R * 8 / kTcThreads; ++j) {
    const int i = tid + kTcThreads * j, r = i >> 3, ch = i & 7;
    const int row = r0 + r, k = k0 + 8 * ch;
    const bool ok = row < nrows && k < ke;   // every K-major depth is a multiple of 8
    cp_async16(dst + sw128_offset(R, r, 8 * ch), ok ? P + (long long)row * srow + k : P, ok);
  }
}

// the same of an MN-major operand (rows in whole chunks of 8)
template <int R>
__device__ __forceinline__ void tc_load_mn(uint32_t dst, const __nv_bfloat16 *P, long long sk, int nrows, int r0, int k0,
                                           int ke, int tid) {
#pragma unroll
  for (int j = 0; j < R * 8 / kTcThreads; ++j) {
    const int i = tid + kTcThreads * j, kk = i / (R / 8), rr = 8 * (i % (R / 8));
    const int row = r0 + rr, k = k0 + kk;
    const bool ok = row < nrows && k < ke;
    cp_async16(dst + sw128_mn_offset(rr, kk), ok ? P + (long long)k * sk + row : P, ok);
  }
}

// the tile at (m0, n0) over k in [kb, ke), then the epilogue.  kMN: both
// operands MN-major, with rows in memory up to ra and rb (multiples of 8)
template <bool kMN, class Epi>
__device__ __forceinline__ void gemm_tile(const GemmArgs &g, int m0, int n0, int kb, int ke, const Epi &epi,
                                          unsigned *err, int ra = 0, int rb = 0) {
  extern __shared__ __align__(16) unsigned char sraw[];
  unsigned char *sm = sraw + ((1024 - (smem_addr(sraw) & 1023)) & 1023);
  unsigned char *smB = sm + kTcSlabs * kTcSlabA;
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) unsigned long long s_bar;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ncols = min(kTcBN, ((g.N - n0) + 15) / 16 * 16);   // MMA N: the tile's columns, multiple of 16
  const uint32_t idesc = umma_idesc_bf16(kTcBM, ncols, kMN);
  const uint32_t bar = smem_addr(&s_bar), sa = smem_addr(sm), sbb = smem_addr(smB);
  if (warp == 0) {
    tmem_alloc(smem_addr(&s_tmem), kTcBN);
    tmem_relinquish();
  }
  if (tid == 0) {
    bar_init(bar, 1);
    bar_fence_init();
  }
  pdl_wait();
  bool ok = true;
  int round = 0;   // depths of 256
  uint32_t taddr = 0;
  for (int k0 = kb; k0 < ke; k0 += kTcSlabs * kTcBK, ++round) {
    // the MMAs that read the slabs of the round before have completed
    if (round > 0 && ok) ok = bar_wait(bar, (uint32_t)((round - 1) & 1), kTcSpins);
    const int nst = min(kTcSlabs, (ke - k0 + kTcBK - 1) / kTcBK);
    if (ok) {
#pragma unroll
      for (int s = 0; s < kTcSlabs; ++s) {
        const int ks = k0 + s * kTcBK;
        if (s < nst) {
          if constexpr (kMN) {
            tc_load_mn<kTcBM>(sa + s * kTcSlabA, g.A, g.sak, ra, m0, ks, ke, tid);
            tc_load_mn<kTcBN>(sbb + s * kTcSlabB, g.B, g.sbk, rb, n0, ks, ke, tid);
          } else {
            tc_load_kmajor<kTcBM>(sa + s * kTcSlabA, g.A, g.sam, g.M, m0, ks, ke, tid);
            tc_load_kmajor<kTcBN>(sbb + s * kTcSlabB, g.B, g.sbn, g.N, n0, ks, ke, tid);
          }
        }
        cp_async_commit();
      }
    }
#pragma unroll
    for (int s = 0; s < kTcSlabs; ++s) {
      if (s == 0) cp_async_wait<3>();
      else if (s == 1) cp_async_wait<2>();
      else if (s == 2) cp_async_wait<1>();
      else cp_async_wait<0>();
      fence_async_smem();
      tc_fence_before();
      __syncthreads();   // slab s (and, the first time, the tensor memory and the barrier) is ready
      if (s >= nst) continue;
      if (tid == 0) {
        tc_fence_after();
        const int nsub = (min(kTcBK, ke - k0 - s * kTcBK) + 15) / 16;
        for (int sub = 0; sub < nsub; ++sub) {
          const uint32_t pa = sa + s * kTcSlabA + (kMN ? 2048u : 32u) * (uint32_t)sub,
                         pb = sbb + s * kTcSlabB + (kMN ? 2048u : 32u) * (uint32_t)sub;
          umma_bf16(s_tmem, kMN ? umma_desc_mn_sw128(pa) : umma_desc_sw128(pa),
                    kMN ? umma_desc_mn_sw128(pb) : umma_desc_sw128(pb), idesc, (round | s | sub) ? 1u : 0u);
        }
        if (s == nst - 1) umma_commit(bar);
      }
    }
  }
  if (round == 0) {
    tc_fence_before();
    __syncthreads();
  }
  tc_fence_after();
  taddr = s_tmem;
  if (round > 0 && !bar_wait(bar, (uint32_t)((round - 1) & 1), kTcSpins)) ok = false;
  tc_fence_after();
  if (!__all_sync(0xffffffffu, ok)) ok = false;
  const int q = warp & 3, c0 = 32 * (warp >> 2);
  if (ok) {
    if (c0 < ncols) {
      float *blk = reinterpret_cast<float *>(sm) + warp * (32 * 33);
      float v[32];
      if (round > 0) {
        tmem_ld32(taddr + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, v);
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = 0.f;
      }
      if constexpr (std::is_same<Epi, EpiOutLoss>::value) {
        // a lane holds a row: its few outputs straight from there
        const int m = m0 + 32 * q + lane;
        double part = m < g.M ? epi.row(m, v) : 0.0;
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0 && part != 0.0) atomicAdd(epi.loss, part);
      } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) blk[lane * 33 + i] = v[i];   // row lane, column i
      __syncwarp();
      const int n = n0 + c0 + lane;
      if (c0 + lane < ncols && n < g.N) {
        if constexpr (Epi::kLoad) {
          // 16 rows at a time: their reads first, then the epilogue
#pragma unroll
          for (int h = 0; h < 32; h += 16) {
            float ld[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
              const int m = m0 + 32 * q + h + r;
              ld[r] = m < g.M ? epi.load(m, n) : 0.f;
            }
#pragma unroll
            for (int r = 0; r < 16; ++r) {
              const int m = m0 + 32 * q + h + r;
              if (m < g.M) epi.apply(m, n, blk[(h + r) * 33 + lane], ld[r]);
            }
          }
        } else {
#pragma unroll 8
          for (int r = 0; r < 32; ++r) {
            const int m = m0 + 32 * q + r;
            if (m < g.M) epi(m, n, blk[r * 33 + lane]);
          }
        }
      }
      }
    }
  } else if (lane == 0) {
    atomicOr(err, 4u);
  }
  tc_fence_before();
  __syncthreads();
  // drain: every MMA this CTA issued has completed before its tensor memory
  // is released (bounded as every wait)
  if (!ok && tid == 0 && round > 0) bar_wait(bar, (uint32_t)((round - 1) & 1), kTcSpins);
  __syncthreads();
  if (warp == 0) tmem_dealloc(taddr, kTcBN);
}

template <class Epi>
__global__ void __launch_bounds__(kTcThreads, 2) k_gemm_tc(const GemmArgs g, const Epi epi, unsigned *err) {
  pdl_trigger();
  gemm_tile<false>(g, blockIdx.y * kTcBM, blockIdx.x * kTcBN, 0, g.K, epi, err);
}

// Every layer's weight gradient in one launch: tiles of all layers times
// chunks of the batch, each CTA one tile of one chunk's partial sum.
struct WgradArgs {
  const __nv_bfloat16 *h[4], *dz[4];   // inputs and output gradients of layers 1-4
  int n, kchunk;
  MlpGradWs ws;
};
constexpr int kWgradTiles1 = kNh / kTcBN, kWgradTiles2 = (kNh / kTcBM) * (kNh / kTcBN), kWgradTiles4 = kNh / kTcBM;
constexpr int kWgradTiles = kWgradTiles1 + 2 * kWgradTiles2 + kWgradTiles4;
__global__ void __launch_bounds__(kTcThreads, 2) k_wgrad_tc(const WgradArgs a, unsigned *err) {
  pdl_trigger();
  int t = blockIdx.x % kWgradTiles, l = 0;
  const int z = blockIdx.x / kWgradTiles;
  if (t >= kWgradTiles1) {
    t -= kWgradTiles1;
    l = 1 + t / kWgradTiles2;
    t -= (l - 1) * kWgradTiles2;
  }
  const int nt = l == 3 ? 1 : kNh / kTcBN;   // tiles along n
  GemmArgs g;
  g.A = l == 0 ? a.h[0] : l == 1 ? a.h[1] : l == 2 ? a.h[2] : a.h[3];
  g.B = l == 0 ? a.dz[0] : l == 1 ? a.dz[1] : l == 2 ? a.dz[2] : a.dz[3];
  g.sam = g.sbn = 1;
  g.sak = l == 0 ? kNinPad : kNh;
  g.sbk = l == 3 ? kNoutPad : kNh;
  g.M = l == 0 ? kNin : kNh;
  g.N = l == 3 ? kNout : kNh;
  g.K = a.n;
  g.kchunk = a.kchunk;
  const long long len = (long long)g.M * g.N;
  const long long off = l == 0 ? grad_ws_off(0) : l == 1 ? grad_ws_off(1) : l == 2 ? grad_ws_off(2) : grad_ws_off(3);
  const int kb = z * a.kchunk;
  gemm_tile<true>(g, t / nt * kTcBM, t % nt * kTcBN, kb, min(a.n, kb + a.kchunk),
                  EpiStore{a.ws.ws + a.ws.nsplit * off + z * len, g.N}, err, l == 0 ? kNinPad : kNh,
                  l == 3 ? kNoutPad : kNh);
}

}  // namespace casim_dev
