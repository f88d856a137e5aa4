// Learned proposal network: kernels and the C ABI of the omp_proposal object.
//
// The network maps the first correlation of a signal to per-atom logits:
//   x = (A^T y)_n / (||a_n|| ||y||)              features, BF16 (the first OMP correlation)
//   h = GELU(W1 x + b1)                          W1: hidden x N, exact GELU x Phi(x) via erff
//   o = W2 h + b2 + beta |x|                     W2: N x hidden, beta a learned scalar (skip term:
//                                                the hidden width is far below N, so the
//                                                per-atom magnitude |x_n| enters directly)
// and proposes, per signal, the `topk` atoms with the largest logits (lowest index on ties).
// Training minimises the mean binary cross-entropy with logits against the support that plain
// OMP picked, with a positive-class weight, using AdamW on FP32 master weights.
//
// Every GEMM runs on the tcgen05 mainloop of tcgemm.cuh with BF16 operands and FP32
// accumulation; operands are K-major, so the epilogues also write the transposed copies the
// backward GEMMs need (Xt, Ht, dOt, dZ1t):
//   features  X   = Yq A16^T            (rows: signals, K = Mp)
//   fwd1      H   = GELU(X W1^T + b1)   (K = N)          also Z1 (FP32) and Ht for training
//   fwd2      O   = H W2^T + b2         (K = hidden)     inference: FP32 logits;
//                                                         training: dO = dBCE/dO, and dOt
//   bwd       dH  = dO W2 = dO (W2t)^T  (K = N)          dZ1t = (dH * GELU'(Z1))^T
//   grads     dW2 = dOt (Ht)^T          (K = batch)      dW1 = dZ1t (Xt)^T
//   biases    db2 = row sums of dOt,    db1 = row sums of dZ1t
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "tcgemm.cuh"

namespace ompk {
namespace {

using namespace tcg;

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x) {
  const float cdf = 0.5f * (1.f + erff(x * 0.70710678118654752f));
  const float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
  return cdf + x * pdf;
}

// log(1 + e^-|o|) from E = e^-o, so that the sigmoid's exponential serves the loss too and no logarithm is
// taken: 2 atanh(s), s = e / (2 + e) <= 1/3 with e = e^-|o|, by the odd series of atanh (seven terms leave
// 1.5e-8 relative). What the denominator, its reciprocal and the quotient round off comes back in by ds:
// against 64 bits the largest error and the root mean square are then no more than those of
// log1pf(expf(-|o|)) (o from -16 to 0: 1.82e-7 for 1.94e-7, 4.64e-8 for 4.66e-8; from -6 to 30: 1.93e-7 both,
// 4.42e-8 for 4.43e-8), without it 2.6e-7. A step at batch 4096, 8192 -> 1024 -> 8192: 633 us; without the
// correction 618, with expf and log1pf 677.
__device__ __forceinline__ float log1p_exp_neg_abs(float E) {
  const bool big = E >= 1.f;  // o <= 0: e = 1 / E
  const float w = fminf(E, 0x1p124f);
  const float a = big ? 1.f : w, two = big ? 2.f * w : 2.f, x = big ? 1.f : w;
  const float b = two + x, be = x - (b - two);
  const float rb = __fdividef(1.f, b);
  const float s = a * rb;
  const float ds = fmaf(-s, be, fmaf(-s, b, a)) * rb;
  const float q = s * s;
  float p = 1.f / 13.f;
  p = fmaf(p, q, 1.f / 11.f);
  p = fmaf(p, q, 1.f / 9.f);
  p = fmaf(p, q, 1.f / 7.f);
  p = fmaf(p, q, 1.f / 5.f);
  p = fmaf(p, q, 1.f / 3.f);
  return 2.f * (s + fmaf(s, p * q, fmaf(ds, q, ds)));
}

// two BF16 values of a word (the lower index in the low half) as FP32
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// ---------------------------------------------------------------------------- epilogues
// The widths here (N and the hidden width) are multiples of 64, so a 32-column chunk lies wholly
// inside the matrix or wholly outside, and its row piece starts on a 64-byte boundary. Each thread
// owns one row of the tile: what it reads and writes of row-major matrices goes in 16-byte
// pieces, a transposed store puts a warp's 32 consecutive rows side by side. Scalar row-major
// accesses (32 sectors per instruction) bounded these kernels by their epilogue: at batch 4096,
// 8192 -> 1024 -> 8192 (MMAs of about 40 us each) the features and the hidden layer in training took
// 157 us on average and take 64 us now, the loss kernel 856 us and now 149 us, the GELU backward
// 102 us and now 60 us.

// The warp's EPI_COLS columns of a vector over the columns (bias or scale) of column tile t, staged in
// its shared scratch at each unit (16 bytes a lane): the chunks read them there.
__device__ __forceinline__ void stage_columns(float* scratch, const float* x, int t, int part, int cols, int lane) {
  static_assert(EPI_COLS == 128 && EPI_SCRATCH >= 128, "one float4 per lane");
  const int c = t * BN + part * EPI_COLS + 4 * lane;
  const float4 v = c < cols ? __ldg(reinterpret_cast<const float4*>(x + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
  __syncwarp();  // every lane has finished with the previous unit's
  reinterpret_cast<float4*>(scratch)[lane] = v;
  __syncwarp();
}

// value = acc * rowscale[r] * colscale[c] + bias[c], optional GELU; BF16 store (row-major and
// optionally transposed into a matrix with leading dimension ldT) and optional FP32 store of the
// pre-activation.
struct EpiAct {
  int rows, cols, ldT, gelu;
  const float* rowscale;
  const float* colscale;
  const float* bias;
  float* pre;
  __nv_bfloat16* out;
  __nv_bfloat16* outT;
  int row, part;
  float* scr;
  __device__ void begin(int, int, int, int row_, int part_, float* scratch, unsigned long long*) {
    row = row_;
    part = part_;
    scr = scratch;
  }
  // (a scale or a bias is given, not both)
  __device__ void unit(int, int t) { stage_columns(scr, colscale ? colscale : bias, t, part, cols, row & 31); }
  __device__ void chunk(int s, int t, int c0, const uint32_t (&v)[32]) {
    const int r = s * BM + row;
    const int cb = t * BN + c0;
    if (r >= rows || cb >= cols) return;
    const float rs = rowscale ? __ldg(rowscale + r) : 1.f;
    const float4* cv = reinterpret_cast<const float4*>(scr + (c0 - part * EPI_COLS));
    uint4* dst = reinterpret_cast<uint4*>(out + static_cast<size_t>(r) * cols + cb);
    float4* pdst = reinterpret_cast<float4*>(pre + static_cast<size_t>(r) * cols + cb);
    __nv_bfloat16* tdst = outT + static_cast<size_t>(cb) * ldT + r;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t ow[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 8 * q + 4 * h;
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = __uint_as_float(v[j + e]) * rs;
        if (colscale) {
          const float4 c = cv[j >> 2];
          x[0] *= c.x;
          x[1] *= c.y;
          x[2] *= c.z;
          x[3] *= c.w;
        } else {
          const float4 c = cv[j >> 2];
          x[0] += c.x;
          x[1] += c.y;
          x[2] += c.z;
          x[3] += c.w;
        }
        if (pre) pdst[j >> 2] = make_float4(x[0], x[1], x[2], x[3]);
        if (gelu) {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = gelu_f(x[e]);
        }
        ow[2 * h] = pack_bf16(x[0], x[1]);
        ow[2 * h + 1] = pack_bf16(x[2], x[3]);
        if (outT) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            tdst[static_cast<size_t>(j + e) * ldT] = __ushort_as_bfloat16(
                static_cast<unsigned short>((e & 1) ? ow[2 * h + (e >> 1)] >> 16 : ow[2 * h + (e >> 1)]));
        }
      }
      dst[q] = make_uint4(ow[0], ow[1], ow[2], ow[3]);
    }
  }
  __device__ void end(bool) {}
};

// FP32 store of acc (+ bias): logits at inference, weight gradients in training.
struct EpiF32 {
  int rows, cols;
  const float* bias;
  const __nv_bfloat16* skipX;  // optional skip term beta * |x| (x: rows x cols features)
  const float* beta;
  float* out;
  int row;
  __device__ void begin(int, int, int, int row_, int, float*, unsigned long long*) { row = row_; }
  __device__ void unit(int, int) {}
  __device__ void chunk(int s, int t, int c0, const uint32_t (&v)[32]) {
    const int r = s * BM + row;
    const int cb = t * BN + c0;
    if (r >= rows || cb >= cols) return;
    const float bt = skipX ? *beta : 0.f;
    float4* dst = reinterpret_cast<float4*>(out + static_cast<size_t>(r) * cols + cb);
    const uint4* xsrc = reinterpret_cast<const uint4*>(skipX + static_cast<size_t>(r) * cols + cb);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint4 xw = make_uint4(0u, 0u, 0u, 0u);
      if (skipX) xw = __ldg(xsrc + q);
      const uint32_t xs[4] = {xw.x, xw.y, xw.z, xw.w};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 8 * q + 4 * h;
        float4 o = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]),
                               __uint_as_float(v[j + 3]));
        if (bias) {
          const float4 c = __ldg(reinterpret_cast<const float4*>(bias + cb + j));
          o.x += c.x;
          o.y += c.y;
          o.z += c.z;
          o.w += c.w;
        }
        if (skipX) {
          o.x = fmaf(bt, fabsf(bf_lo(xs[2 * h])), o.x);
          o.y = fmaf(bt, fabsf(bf_hi(xs[2 * h])), o.y);
          o.z = fmaf(bt, fabsf(bf_lo(xs[2 * h + 1])), o.z);
          o.w = fmaf(bt, fabsf(bf_hi(xs[2 * h + 1])), o.w);
        }
        dst[j >> 2] = o;
      }
    }
  }
  __device__ void end(bool) {}
};

// Gradient of the mean weighted BCE with logits o = acc + b2 and labels from a bit matrix
// (row r, column c at bit c % 32 of word r * (cols / 32) + c / 32):
//   loss = pw y softplus(-o) + (1 - y) softplus(o),  dloss/do = sigma(o) (1 - y + pw y) - pw y,
// both divided by rows * cols. Stores dO (row-major) and dOt (transposed, leading dim ldT) in
// BF16 and adds the loss to *loss.
struct EpiBCE {
  int rows, cols, ldT;
  float pos_weight, inv_count;
  const float* bias;
  const uint32_t* labels;
  const __nv_bfloat16* skipX;  // features x: the logit has the skip term beta * |x|
  const float* beta;
  float* dbeta;                // accumulates sum dO * |x|
  __nv_bfloat16* dO;
  __nv_bfloat16* dOT;
  float* loss;
  int row, part;
  float* scr;
  float lsum, bsum;
  __device__ void begin(int, int, int, int row_, int part_, float* scratch, unsigned long long*) {
    row = row_;
    part = part_;
    scr = scratch;
    lsum = 0.f;
    bsum = 0.f;
  }
  __device__ void unit(int, int t) { stage_columns(scr, bias, t, part, cols, row & 31); }
  __device__ void chunk(int s, int t, int c0, const uint32_t (&v)[32]) {
    const int r = s * BM + row;
    const int cb = t * BN + c0;
    if (r >= rows || cb >= cols) return;
    const uint32_t bits = __ldg(labels + static_cast<size_t>(r) * (cols >> 5) + (cb >> 5));
    const float bt = *beta;
    const uint4* xsrc = reinterpret_cast<const uint4*>(skipX + static_cast<size_t>(r) * cols + cb);
    uint4* dst = reinterpret_cast<uint4*>(dO + static_cast<size_t>(r) * cols + cb);
    __nv_bfloat16* tdst = dOT + static_cast<size_t>(cb) * ldT + r;
    const float4* cv = reinterpret_cast<const float4*>(scr + (c0 - part * EPI_COLS));
    uint4 xq[4];  // the row's 32 features, in flight together
#pragma unroll
    for (int q = 0; q < 4; ++q) xq[q] = __ldg(xsrc + q);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 xw = xq[q];
      const uint32_t xs[4] = {xw.x, xw.y, xw.z, xw.w};
      uint32_t ow[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 8 * q + 4 * h;
        const float4 c = cv[j >> 2];
        const float bc[4] = {c.x, c.y, c.z, c.w};
        float g[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t xp = xs[2 * h + (e >> 1)];
          const float ax = fabsf((e & 1) ? bf_hi(xp) : bf_lo(xp));
          const float o = fmaf(bt, ax, __uint_as_float(v[j + e]) + bc[e]);
          const bool y = (bits >> (j + e)) & 1u;
          const float E = expf(-o);
          const float sg = 1.f / (1.f + E);
          // y 1: pw sigma(o) - pw and pw softplus(-o); y 0: sigma(o) and softplus(o)
          g[e] = (y ? fmaf(sg, pos_weight, -pos_weight) : sg) * inv_count;
          const float sp = fmaxf(y ? -o : o, 0.f) + log1p_exp_neg_abs(E);
          lsum += (y ? pos_weight * sp : sp) * inv_count;
          bsum = fmaf(g[e], ax, bsum);
        }
        ow[2 * h] = pack_bf16(g[0], g[1]);
        ow[2 * h + 1] = pack_bf16(g[2], g[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          tdst[static_cast<size_t>(j + e) * ldT] = __ushort_as_bfloat16(
              static_cast<unsigned short>((e & 1) ? ow[2 * h + (e >> 1)] >> 16 : ow[2 * h + (e >> 1)]));
      }
      dst[q] = make_uint4(ow[0], ow[1], ow[2], ow[3]);
    }
  }
  __device__ void end(bool) {
    float v = lsum, w = bsum;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, o);
      w += __shfl_xor_sync(0xffffffffu, w, o);
    }
    if ((threadIdx.x & 31) == 0) {
      if (loss) atomicAdd(loss, v);
      atomicAdd(dbeta, w);
    }
  }
};

// dZ1 = dH * GELU'(Z1), stored transposed (hidden x batch, leading dim ldT) in BF16.
struct EpiGeluBwd {
  int rows, cols, ldT;
  const float* Z1;
  __nv_bfloat16* dZT;
  int row;
  __device__ void begin(int, int, int, int row_, int, float*, unsigned long long*) { row = row_; }
  __device__ void unit(int, int) {}
  __device__ void chunk(int s, int t, int c0, const uint32_t (&v)[32]) {
    const int r = s * BM + row;
    const int cb = t * BN + c0;
    if (r >= rows || cb >= cols) return;
    const float4* zsrc = reinterpret_cast<const float4*>(Z1 + static_cast<size_t>(r) * cols + cb);
    __nv_bfloat16* tdst = dZT + static_cast<size_t>(cb) * ldT + r;
    float4 zq[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) zq[q] = __ldg(zsrc + q);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 z = zq[q];
      const float zz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        tdst[static_cast<size_t>(4 * q + e) * ldT] =
            __float2bfloat16_rn(__uint_as_float(v[4 * q + e]) * gelu_grad_f(zz[e]));
    }
  }
  __device__ void end(bool) {}
};

template <class Epi>
__global__ void __launch_bounds__(THREADS, 1)
    mlp_gemm_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                    int rows, int cols, int K, unsigned int* err, Epi epi) {
  gemm_body<OMP_PREC_BF16>(&ta, &tb, (rows + BM - 1) / BM, (cols + BN - 1) / BN, K / 64, 1, err, epi);
}

// ------------------------------------------------------------------------ small kernels
// Feature input: y in BF16 (zero padded to Mp) and 1/||y|| (0 for y == 0 or non-finite y). One warp
// per signal, the row read once, 16 loads in flight a lane.
__global__ void __launch_bounds__(256) feat_prep_kernel(const float* __restrict__ Y, int M, int Mp, int B,
                                                        __nv_bfloat16* Yq, float* inv_ynorm) {
  constexpr int R = 16;
  const int lane = threadIdx.x & 31;
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= B) return;
  const float* y = Y + static_cast<size_t>(b) * M;
  SquareSum sq;
  bool finite = true;
  for (int m0 = 0; m0 < Mp; m0 += 32 * R) {
    float v[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int m = m0 + 32 * i + lane;
      v[i] = m < M ? __ldg(y + m) : 0.f;
    }
    auto take = [&](int i) {
      finite = finite && isfinite(v[i]);
      square_in(sq, v[i]);
    };
    if (m0 + 32 * R <= Mp) {
#pragma unroll
      for (int i = 0; i < R; ++i) take(i);
    } else {  // no chain over zeros past the end of the row
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (m0 + 32 * i < Mp) take(i);
    }
    // written as if finite; a signal with a NaN or Inf is cleared below
    __nv_bfloat16* q = Yq + static_cast<size_t>(b) * Mp;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int m = m0 + 32 * i + lane;
      if (m < Mp) q[m] = __float2bfloat16_rn(v[i]);
    }
  }
  double s = warp_sum(total(sq));
  if (!squares_ok(s)) {  // zero, tiny or huge signals (or a NaN)
    s = 0.0;
    for (int m = lane; m < M; m += 32) s += static_cast<double>(y[m]) * y[m];
    s = warp_sum(s);
  }
  finite = __all_sync(0xffffffffu, finite);
  if (!finite)
    for (int m = lane; m < Mp; m += 32) Yq[static_cast<size_t>(b) * Mp + m] = __float2bfloat16_rn(0.f);
  if (lane == 0) inv_ynorm[b] = finite && s > 0.0 ? static_cast<float>(1.0 / sqrt(s)) : 0.f;
}

// Label bit matrix from supports (B x S, -1 padded): bit c of row b is set if c is in the row.
__global__ void labels_kernel(const int* __restrict__ sup, int B, int S, int N, uint32_t* bits) {
  const int b = blockIdx.x;
  uint32_t* row = bits + static_cast<size_t>(b) * (N >> 5);
  for (int w = threadIdx.x; w < (N >> 5); w += blockDim.x) row[w] = 0u;
  __syncthreads();
  for (int j = threadIdx.x; j < S; j += blockDim.x) {
    const int c = sup[static_cast<size_t>(b) * S + j];
    if (c >= 0 && c < N) atomicOr(row + (c >> 5), 1u << (c & 31));
  }
}

// out[i] = sum_j in[i * ld + j], j < n (one warp per row, FP32 accumulation, lane l over
// j = l, l + 32, ...), 16 loads in flight per lane: bound by the row's round trips
__global__ void __launch_bounds__(256) row_sum_kernel(const __nv_bfloat16* __restrict__ in, int rows, int n,
                                                      int ld, float* out) {
  constexpr int R = 16;
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const __nv_bfloat16* p = in + static_cast<size_t>(r) * ld;
  float s = 0.f;
  for (int j0 = lane; j0 < n; j0 += 32 * R) {
    __nv_bfloat16 w[R];
#pragma unroll
    for (int i = 0; i < R; ++i) w[i] = j0 + 32 * i < n ? p[j0 + 32 * i] : __nv_bfloat16(0.f);
#pragma unroll
    for (int i = 0; i < R; ++i) s += __bfloat162float(w[i]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[r] = s;
}

struct AdamParams {
  float lr, beta1, beta2, eps, wd, c1, c2;  // c1 = 1 / (1 - beta1^t), c2 = 1 / (1 - beta2^t)
};

__device__ __forceinline__ void adamw_one(float& w, float& m, float& v, float g, const AdamParams& a) {
  m = a.beta1 * m + (1.f - a.beta1) * g;
  v = a.beta2 * v + (1.f - a.beta2) * g * g;
  const float upd = (m * a.c1) / (sqrtf(v * a.c2) + a.eps) + a.wd * w;
  w = w - a.lr * upd;
}

// AdamW step on FP32 master weights (rows x cols, both multiples of 64) that also writes the BF16
// copy and, with wbT, its transpose: a 64 x 64 tile per 256-thread block, four rows of 16-byte
// loads per thread in flight. Bound by HBM: 30 bytes an element (32 with the transpose, which a
// kernel of its own read the weights again for): 38 us for 8.4 million weights, 6.6 TB/s, against
// 52 us with 4-byte accesses and 18 us more for the transpose.
__global__ void __launch_bounds__(256) adamw_matrix_kernel(float* __restrict__ w, float* __restrict__ m,
                                                           float* __restrict__ v, const float* __restrict__ g,
                                                           int rows, int cols, AdamParams a,
                                                           __nv_bfloat16* __restrict__ wb,
                                                           __nv_bfloat16* __restrict__ wbT) {
  __shared__ __nv_bfloat16 tile[64][66];
  const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
  const int tc = threadIdx.x & 15, tr = threadIdx.x >> 4;
  size_t at[4];
  float4 gv[4], wv[4], mv[4], vv[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    at[i] = static_cast<size_t>(r0 + tr + 16 * i) * cols + c0 + 4 * tc;
    gv[i] = *reinterpret_cast<const float4*>(g + at[i]);
    wv[i] = *reinterpret_cast<const float4*>(w + at[i]);
    mv[i] = *reinterpret_cast<const float4*>(m + at[i]);
    vv[i] = *reinterpret_cast<const float4*>(v + at[i]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    adamw_one(wv[i].x, mv[i].x, vv[i].x, gv[i].x, a);
    adamw_one(wv[i].y, mv[i].y, vv[i].y, gv[i].y, a);
    adamw_one(wv[i].z, mv[i].z, vv[i].z, gv[i].z, a);
    adamw_one(wv[i].w, mv[i].w, vv[i].w, gv[i].w, a);
    *reinterpret_cast<float4*>(w + at[i]) = wv[i];
    *reinterpret_cast<float4*>(m + at[i]) = mv[i];
    *reinterpret_cast<float4*>(v + at[i]) = vv[i];
    const uint32_t lo = pack_bf16(wv[i].x, wv[i].y), hi = pack_bf16(wv[i].z, wv[i].w);
    *reinterpret_cast<uint2*>(wb + at[i]) = make_uint2(lo, hi);
    if (wbT) {  // 66 BF16 a row: the 4-byte words of a column walk all banks
      *reinterpret_cast<uint32_t*>(&tile[tr + 16 * i][4 * tc]) = lo;
      *reinterpret_cast<uint32_t*>(&tile[tr + 16 * i][4 * tc + 2]) = hi;
    }
  }
  if (!wbT) return;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int c = warp + 8 * i;
    const __nv_bfloat162 h{tile[2 * lane][c], tile[2 * lane + 1][c]};
    *reinterpret_cast<__nv_bfloat162*>(wbT + static_cast<size_t>(c0 + c) * rows + r0 + 2 * lane) = h;
  }
}

// AdamW step of a short vector (the biases and the skip scale: one launch for all three)
struct AdamVec {
  float *w, *m, *v;
  const float* g;
  int n;
};
__global__ void __launch_bounds__(256) adamw_vectors_kernel(AdamVec x0, AdamVec x1, AdamVec x2, AdamParams a) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  AdamVec x = x0;
  if (i >= x.n) {
    i -= x.n;
    x = x1;
    if (i >= x.n) {
      i -= x.n;
      x = x2;
    }
  }
  if (i < x.n) adamw_one(x.w[i], x.m[i], x.v[i], x.g[i], a);
}

__global__ void abs_bf16_kernel(const __nv_bfloat16* __restrict__ x, size_t n, float* out) {
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x)
    out[i] = fabsf(__bfloat162float(x[i]));
}

__global__ void to_bf16_kernel(const float* __restrict__ w, size_t n, __nv_bfloat16* wb) {
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x)
    wb[i] = __float2bfloat16_rn(w[i]);
}

// out (cols x rows, BF16) = transpose of in (rows x cols, FP32), 32 x 32 tiles through smem
__global__ void transpose_bf16_kernel(const float* __restrict__ in, int rows, int cols, __nv_bfloat16* out) {
  __shared__ float tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    tile[i][threadIdx.x] = (r < rows && c < cols) ? in[static_cast<size_t>(r) * cols + c] : 0.f;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (c < cols && r < rows) out[static_cast<size_t>(c) * rows + r] = __float2bfloat16_rn(tile[threadIdx.x][i]);
  }
}

// Per row of logits (N values): the K largest, lowest index first among equal values, written
// in ascending index order. One 256-thread block per row: a bitwise search over the
// order-preserving integer image of the floats finds the K-th largest value t, then every
// element > t is kept and the elements == t fill the remaining slots in index order.
__device__ __forceinline__ uint32_t orderable(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// SMEM: the row's orderable keys are staged in dynamic shared memory once (N x 4 bytes). The keys'
// range is then cut into 2048 equal bins: their counts give the bin of the K-th largest key, and that
// bin's few keys its exact value. (Logits share their leading bits, so a radix histogram meets the
// same few bins over and over, and 4 passes of it with match-any took 171 us for 4096 rows of 8192;
// equal pieces of the row's own range spread them: 100 us.) A bin that holds too many keys is
// searched bit by bit.
constexpr int kBins = 2048, kBinList = 512;

template <bool SMEM>
__global__ void __launch_bounds__(256) topk_rows_kernel(const float* __restrict__ logits, int N, int K,
                                                         int* __restrict__ out) {
  __shared__ int red[8];
  __shared__ int wcnt_gt[8], wcnt_eq[8];
  __shared__ uint32_t lo_s[8], hi_s[8];
  __shared__ int hist[SMEM ? kBins : 1];
  __shared__ uint32_t list[SMEM ? kBinList : 1];
  __shared__ int sel_s[3];       // the bin found, the rank still to find within it, keys listed
  __shared__ uint32_t thr_s;
  extern __shared__ uint32_t keys_s[];
  const int row = blockIdx.x;
  const float* x = logits + static_cast<size_t>(row) * N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  if (SMEM) {
    for (int i0 = tid; i0 < N; i0 += 8 * 256) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = i0 + 256 * u < N ? __ldg(x + i0 + 256 * u) : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + 256 * u < N) {
          const uint32_t kv = orderable(v[u]);
          keys_s[i0 + 256 * u] = kv;
          kmin = min(kmin, kv);
          kmax = max(kmax, kv);
        }
    }
    for (int i = tid; i < kBins; i += 256) hist[i] = 0;
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
      lo_s[warp] = kmin;
      hi_s[warp] = kmax;
    }
    if (tid == 0) sel_s[2] = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      kmin = min(kmin, lo_s[w]);
      kmax = max(kmax, hi_s[w]);
    }
  }
  auto key = [&](int i) -> uint32_t { return SMEM ? keys_s[i] : orderable(x[i]); };
  // T = the K-th largest key: the largest threshold with count(key >= T) >= K
  uint32_t T = 0;
  bool found = false;
  if (SMEM) {
    // bin = floor((key - kmin) m / 2^32), m the largest factor that keeps every bin below kBins:
    // increasing with the key
    const uint32_t span = kmax - kmin;
    const uint32_t m = span < kBins ? 0u
                                    : static_cast<uint32_t>((static_cast<unsigned long long>(kBins) << 32) /
                                                            (static_cast<unsigned long long>(span) + 1ull));
    auto bin_of = [&](uint32_t kv) -> int {
      return span < kBins ? static_cast<int>(kv - kmin) : static_cast<int>(__umulhi(kv - kmin, m));
    };
    for (int i = tid; i < N; i += 256) atomicAdd(&hist[bin_of(keys_s[i])], 1);
    __syncthreads();
    // thread t owns bins 8t .. 8t + 7; counts above a bin come from the higher threads
    int cnt[8], tot = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      cnt[j] = hist[8 * tid + j];
      tot += cnt[j];
    }
    int inc = tot;  // over this thread and the higher lanes of its warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_down_sync(0xffffffffu, inc, o);
      if (lane + o < 32) inc += v;
    }
    if (lane == 0) red[warp] = inc;
    __syncthreads();
    int above = inc - tot;
    for (int w = warp + 1; w < 8; ++w) above += red[w];
#pragma unroll
    for (int j = 7; j >= 0; --j) {
      if (above < K && above + cnt[j] >= K) {
        sel_s[0] = 8 * tid + j;
        sel_s[1] = K - above;
      }
      above += cnt[j];
    }
    __syncthreads();
    const int sb = sel_s[0], rank = sel_s[1];
    if (hist[sb] <= kBinList) {
      for (int i = tid; i < N; i += 256) {
        const uint32_t kv = keys_s[i];
        if (bin_of(kv) == sb) list[atomicAdd(&sel_s[2], 1)] = kv;
      }
      __syncthreads();
      const int n = sel_s[2];
      // the rank-th largest of the list: fewer than rank keys above it, at least rank at or above
      for (int i = tid; i < n; i += 256) {
        const uint32_t kv = list[i];
        int gt = 0, ge = 0;
        for (int j = 0; j < n; ++j) {
          gt += list[j] > kv ? 1 : 0;
          ge += list[j] >= kv ? 1 : 0;
        }
        if (gt < rank && ge >= rank) thr_s = kv;
      }
      __syncthreads();
      T = thr_s;
      found = true;
    }
  }
  if (!found) {
    // bitwise search over the row
    for (int bit = 31; bit >= 0; --bit) {
      const uint32_t cand = T | (1u << bit);
      int c = 0;
      for (int i = tid; i < N; i += 256) c += key(i) >= cand ? 1 : 0;
      c = warp_sum_int(c);
      if (lane == 0) red[warp] = c;
      __syncthreads();
      int tot = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) tot += red[w];
      __syncthreads();
      if (tot >= K) T = cand;
    }
  }
  // Output: the > T elements and the first K - count(> T) elements == T, in index order. Each
  // warp owns a contiguous index range: one pass counts its > T and == T elements, one barrier
  // gives every warp the counts of the ranges before it, and each warp then writes its selected
  // indices in order (ballots within the warp, no further barriers).
  const int per = (N + 7) / 8;
  const int lo = min(N, warp * per), hi = min(N, lo + per);
  int cg = 0, ce = 0;
  for (int i = lo + lane; i < hi; i += 32) {
    const uint32_t kv = key(i);
    cg += kv > T ? 1 : 0;
    ce += kv == T ? 1 : 0;
  }
  cg = warp_sum_int(cg);
  ce = warp_sum_int(ce);
  if (lane == 0) {
    wcnt_gt[warp] = cg;
    wcnt_eq[warp] = ce;
  }
  __syncthreads();
  int total_gt = 0, base_gt = 0, base_eq = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    total_gt += wcnt_gt[w];
    if (w < warp) {
      base_gt += wcnt_gt[w];
      base_eq += wcnt_eq[w];
    }
  }
  const int need_eq = K - total_gt;
  int* o = out + static_cast<size_t>(row) * K;
  const unsigned below = (1u << lane) - 1u;
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t kv = i < hi ? key(i) : 0u;
    const bool gt = i < hi && kv > T;
    const bool eq = i < hi && kv == T;
    const unsigned mg = __ballot_sync(0xffffffffu, gt);
    const unsigned me = __ballot_sync(0xffffffffu, eq);
    const int rg = base_gt + __popc(mg & below);
    const int re = base_eq + __popc(me & below);
    if (gt || (eq && re < need_eq)) {
      const int slot = rg + min(re, need_eq);
      if (slot < K) o[slot] = i;
    }
    base_gt += __popc(mg);
    base_eq += __popc(me);
  }
}

// The rows' K largest entries (see topk_rows_kernel); shared-memory keys when a row fits.
bool launch_topk_rows(const float* logits, int rows, int N, int K, int* out, cudaStream_t s) {
  const size_t bytes = static_cast<size_t>(N) * 4;
  if (bytes <= 160 * 1024 &&
      raise_smem_limit(reinterpret_cast<const void*>(topk_rows_kernel<true>), bytes) == cudaSuccess) {
    topk_rows_kernel<true><<<rows, 256, bytes, s>>>(logits, N, K, out);
  } else {
    cudaGetLastError();
    topk_rows_kernel<false><<<rows, 256, 0, s>>>(logits, N, K, out);
  }
  return cudaGetLastError() == cudaSuccess;
}

// tau[k] = the q-quantile (the floor(q * n)-th smallest, 0-based) of the positive entries of
// column k of a B x S matrix; 0 if the column has none. One block per column; a bitwise search
// over the IEEE bits of the (positive) values.
__global__ void __launch_bounds__(256) quantile_cols_kernel(const float* __restrict__ v, int B, int S, float q,
                                                            float* __restrict__ tau) {
  __shared__ int red[8];
  const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto block_count = [&](auto pred) {
    int c = 0;
    for (int b = tid; b < B; b += 256) {
      const float x = v[static_cast<size_t>(b) * S + k];
      c += (x > 0.f && pred(__float_as_uint(x))) ? 1 : 0;
    }
    c = warp_sum_int(c);
    if (lane == 0) red[warp] = c;
    __syncthreads();
    int t = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[w];
    __syncthreads();
    return t;
  };
  const int n = block_count([](uint32_t) { return true; });
  if (n == 0) {
    if (tid == 0) tau[k] = 0.f;
    return;
  }
  int m = static_cast<int>(q * static_cast<float>(n));
  if (m > n - 1) m = n - 1;
  uint32_t T = 0;
  for (int bit = 30; bit >= 0; --bit) {
    const uint32_t cand = T | (1u << bit);
    const int below = block_count([cand](uint32_t u) { return u < cand; });
    if (below <= m) T = cand;
  }
  if (tid == 0) tau[k] = __uint_as_float(T);
}

}  // namespace
}  // namespace ompk

// =============================================================================== C ABI
using namespace ompk;

struct omp_proposal_s {
  omp_proposal_desc d{};
  int dev = 0;
  int N = 0, M = 0, Mp = 0, H = 0, Bi = 0, Bt = 0;
  int grid = 0;
  long long step = 0;
  std::vector<void*> allocs;
  // parameters (FP32 masters, Adam moments, BF16 copies)
  float *W1 = nullptr, *b1 = nullptr, *W2 = nullptr, *b2 = nullptr;
  float *beta = nullptr, *mbeta = nullptr, *vbeta = nullptr, *dbeta = nullptr;  // skip-term scale
  float *mW1 = nullptr, *vW1 = nullptr, *mb1 = nullptr, *vb1 = nullptr;
  float *mW2 = nullptr, *vW2 = nullptr, *mb2 = nullptr, *vb2 = nullptr;
  __nv_bfloat16 *W1b = nullptr, *W2b = nullptr, *W2Tb = nullptr;
  // dictionary copy (BF16) and scales used by the feature GEMM
  __nv_bfloat16* A16 = nullptr;
  float* escale = nullptr;
  const float* prepared_A = nullptr;
  // activations
  __nv_bfloat16 *Yq = nullptr, *X = nullptr, *XT = nullptr, *Hh = nullptr, *HT = nullptr;
  float *inv_yn = nullptr, *Z1 = nullptr, *logits = nullptr;
  __nv_bfloat16 *dO = nullptr, *dOT = nullptr, *dZT = nullptr;
  float *dW1 = nullptr, *db1 = nullptr, *dW2 = nullptr, *db2 = nullptr;
  uint32_t* labels = nullptr;
  float* loss = nullptr;
  float* tau = nullptr;
  int* cand = nullptr;
  int Smax_tau = 0;
  unsigned int* err = nullptr;
};

namespace ompk {
namespace mlpd {

using namespace tcg;

template <class T>
bool palloc(omp_proposal_s* p, T** ptr, size_t count) {
  *ptr = nullptr;
  if (count == 0) return true;
  void* q = nullptr;
  if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  p->allocs.push_back(q);
  *ptr = static_cast<T*>(q);
  return true;
}

void pfree(omp_proposal_s* p) {
  for (void* q : p->allocs) cudaFree(q);
  p->allocs.clear();
}

int blocks_for(size_t n) {
  const size_t b = (n + 255) / 256;
  return static_cast<int>(b < 4096 ? b : 4096);
}

template <class Epi>
bool gemm(const omp_proposal_s* p, const void* a, int a_rows, const void* b, int b_rows, int K,
          const Epi& epi, cudaStream_t s, int ld = 0) {
  CUtensorMap ta, tb;
  if (!make_kmajor_map(&ta, a, OMP_PREC_BF16, a_rows, K, BM, ld) ||
      !make_kmajor_map(&tb, b, OMP_PREC_BF16, b_rows, K, BN, ld))
    return false;
  static bool attr_done = false;  // per epilogue type
  if (!attr_done) {
    if (set_smem_attr(reinterpret_cast<const void*>(mlp_gemm_kernel<Epi>)) != cudaSuccess) return false;
    attr_done = true;
  }
  mlp_gemm_kernel<Epi><<<p->grid, THREADS, SMEM_BYTES, s>>>(ta, tb, a_rows, b_rows, K, p->err, epi);
  return cudaGetLastError() == cudaSuccess;
}

// Dictionary copy for the feature GEMM: BF16 rows zero-padded to Mp and escale = 1/||a_n||.
__global__ void dict_bf16_kernel(const float* __restrict__ A, int M, int Mp, int N, __nv_bfloat16* A16,
                                 float* escale) {
  const int lane = threadIdx.x & 31;
  const int n = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (n >= N) return;
  const float* a = A + static_cast<size_t>(n) * M;
  double s = 0.0;
  for (int m = lane; m < Mp; m += 32) {
    const float v = m < M ? a[m] : 0.f;
    A16[static_cast<size_t>(n) * Mp + m] = __float2bfloat16_rn(v);
    s += static_cast<double>(v) * v;
  }
  s = warp_sum(s);
  if (lane == 0) escale[n] = s > 0.0 ? static_cast<float>(1.0 / sqrt(s)) : 0.f;
}

bool features(omp_proposal_s* p, const float* A, const float* Y, int B, bool transposed,
              cudaStream_t s) {
  if (A != p->prepared_A) {
    dict_bf16_kernel<<<(p->N + 7) / 8, 256, 0, s>>>(A, p->M, p->Mp, p->N, p->A16, p->escale);
    p->prepared_A = A;
  }
  feat_prep_kernel<<<(B + 7) / 8, 256, 0, s>>>(Y, p->M, p->Mp, B, p->Yq, p->inv_yn);
  EpiAct e{};
  e.rows = B;
  e.cols = p->N;
  e.ldT = p->Bt;
  e.gelu = 0;
  e.rowscale = p->inv_yn;
  e.colscale = p->escale;
  e.out = p->X;
  e.outT = transposed ? p->XT : nullptr;
  return gemm(p, p->Yq, B, p->A16, p->N, p->Mp, e, s);
}

bool forward_hidden(omp_proposal_s* p, int B, bool training, cudaStream_t s) {
  EpiAct e{};
  e.rows = B;
  e.cols = p->H;
  e.ldT = p->Bt;
  e.gelu = 1;
  e.bias = p->b1;
  e.pre = training ? p->Z1 : nullptr;
  e.out = p->Hh;
  e.outT = training ? p->HT : nullptr;
  return gemm(p, p->X, B, p->W1b, p->H, p->N, e, s);
}

bool gradients(omp_proposal_s* p, const float* A, const float* Y, const int* labels_sup, int B, int S,
               cudaStream_t s) {
  if (!features(p, A, Y, B, true, s)) return false;
  if (!forward_hidden(p, B, true, s)) return false;
  labels_kernel<<<B, 256, 0, s>>>(labels_sup, B, S, p->N, p->labels);
  cudaMemsetAsync(p->loss, 0, sizeof(float), s);
  cudaMemsetAsync(p->dbeta, 0, sizeof(float), s);
  EpiBCE eb{};
  eb.skipX = p->X;
  eb.beta = p->beta;
  eb.dbeta = p->dbeta;
  eb.rows = B;
  eb.cols = p->N;
  eb.ldT = p->Bt;
  eb.pos_weight = p->d.pos_weight;
  eb.inv_count = 1.f / (static_cast<float>(B) * static_cast<float>(p->N));
  eb.bias = p->b2;
  eb.labels = p->labels;
  eb.dO = p->dO;
  eb.dOT = p->dOT;
  eb.loss = p->loss;
  if (!gemm(p, p->Hh, B, p->W2b, p->N, p->H, eb, s)) return false;
  EpiGeluBwd eg{};
  eg.rows = B;
  eg.cols = p->H;
  eg.ldT = p->Bt;
  eg.Z1 = p->Z1;
  eg.dZT = p->dZT;
  if (!gemm(p, p->dO, B, p->W2Tb, p->H, p->N, eg, s)) return false;
  EpiF32 e2{};
  e2.rows = p->N;
  e2.cols = p->H;
  e2.out = p->dW2;
  if (!gemm(p, p->dOT, p->N, p->HT, p->H, B, e2, s, p->Bt)) return false;
  EpiF32 e1{};
  e1.rows = p->H;
  e1.cols = p->N;
  e1.out = p->dW1;
  if (!gemm(p, p->dZT, p->H, p->XT, p->N, B, e1, s, p->Bt)) return false;
  row_sum_kernel<<<(p->N + 7) / 8, 256, 0, s>>>(p->dOT, p->N, B, p->Bt, p->db2);
  row_sum_kernel<<<(p->H + 7) / 8, 256, 0, s>>>(p->dZT, p->H, B, p->Bt, p->db1);
  return cudaGetLastError() == cudaSuccess;
}

void refresh_bf16(omp_proposal_s* p, cudaStream_t s) {
  const size_t n1 = static_cast<size_t>(p->H) * p->N;
  to_bf16_kernel<<<blocks_for(n1), 256, 0, s>>>(p->W1, n1, p->W1b);
  to_bf16_kernel<<<blocks_for(n1), 256, 0, s>>>(p->W2, n1, p->W2b);
  dim3 grid((p->H + 31) / 32, (p->N + 31) / 32);
  transpose_bf16_kernel<<<grid, dim3(32, 8), 0, s>>>(p->W2, p->N, p->H, p->W2Tb);
}

}  // namespace mlpd
}  // namespace ompk

using namespace ompk::mlpd;

extern "C" {

void omp_proposal_desc_default(omp_proposal_desc* d) {
  if (!d) return;
  std::memset(d, 0, sizeof(*d));
  d->hidden = 1024;
  d->topk = 256;
  d->max_batch = 16384;
  d->train_batch = 4096;
  d->lr = 1e-3f;
  d->beta1 = 0.9f;
  d->beta2 = 0.999f;
  d->weight_decay = 0.f;
  d->adam_eps = 1e-8f;
  d->pos_weight = 1.f;
}

omp_status omp_proposal_create(omp_handle h, const omp_proposal_desc* desc, omp_proposal* out) {
  if (!h || !desc || !out) return OMP_ERR_INVALID_ARGUMENT;
  *out = nullptr;
  omp_desc hd{};
  int dev = 0, sms = 0;
  if (omp_handle_info(h, &hd, &sms) != OMP_OK) return OMP_ERR_INVALID_ARGUMENT;
  dev = hd.device;
  const omp_proposal_desc d = *desc;
  if (d.hidden < 64 || d.hidden % 64 || hd.N % 64 || d.topk < 1 || d.topk > hd.N || d.max_batch < 1 ||
      d.max_batch > hd.max_batch || d.train_batch < 64 || d.train_batch % 64 || d.topk > 256)
    return OMP_ERR_INVALID_ARGUMENT;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(dev);
  omp_proposal_s* p = new (std::nothrow) omp_proposal_s();
  if (!p) return OMP_ERR_OUT_OF_MEMORY;
  p->d = d;
  p->dev = dev;
  p->N = static_cast<int>(hd.N);
  p->M = static_cast<int>(hd.M);
  p->Mp = static_cast<int>((hd.M + 63) / 64 * 64);
  p->H = d.hidden;
  p->Bi = (d.max_batch + 127) / 128 * 128;
  p->Bt = d.train_batch;
  p->grid = sms;
  p->Smax_tau = hd.max_iters;
  const size_t N = p->N, H = p->H, Bx = p->Bi > p->Bt ? p->Bi : p->Bt, Bt = p->Bt, Mp = p->Mp;
  bool ok = palloc(p, &p->W1, H * N) && palloc(p, &p->b1, H) && palloc(p, &p->W2, N * H) && palloc(p, &p->b2, N);
  ok = ok && palloc(p, &p->beta, 1) && palloc(p, &p->mbeta, 1) && palloc(p, &p->vbeta, 1) && palloc(p, &p->dbeta, 1);
  ok = ok && palloc(p, &p->mW1, H * N) && palloc(p, &p->vW1, H * N) && palloc(p, &p->mb1, H) && palloc(p, &p->vb1, H);
  ok = ok && palloc(p, &p->mW2, N * H) && palloc(p, &p->vW2, N * H) && palloc(p, &p->mb2, N) && palloc(p, &p->vb2, N);
  ok = ok && palloc(p, &p->W1b, H * N) && palloc(p, &p->W2b, N * H) && palloc(p, &p->W2Tb, H * N);
  ok = ok && palloc(p, &p->A16, N * Mp) && palloc(p, &p->escale, N);
  ok = ok && palloc(p, &p->Yq, Bx * Mp) && palloc(p, &p->inv_yn, Bx) && palloc(p, &p->X, Bx * N) &&
       palloc(p, &p->Hh, Bx * H) && palloc(p, &p->logits, static_cast<size_t>(p->Bi) * N) &&
       palloc(p, &p->cand, static_cast<size_t>(p->Bi) * d.topk);
  ok = ok && palloc(p, &p->XT, N * Bt) && palloc(p, &p->HT, H * Bt) && palloc(p, &p->Z1, Bt * H) &&
       palloc(p, &p->dO, Bt * N) && palloc(p, &p->dOT, N * Bt) && palloc(p, &p->dZT, H * Bt) &&
       palloc(p, &p->dW1, H * N) && palloc(p, &p->db1, H) && palloc(p, &p->dW2, N * H) &&
       palloc(p, &p->db2, N) && palloc(p, &p->labels, Bt * (N / 32)) && palloc(p, &p->loss, 1) &&
       palloc(p, &p->tau, static_cast<size_t>(p->Smax_tau)) && palloc(p, &p->err, 1);
  bool cuda_ok = ok;
  if (ok) {
    const size_t n1 = H * N;
    cuda_ok = cudaMemset(p->W1, 0, n1 * 4) == cudaSuccess && cudaMemset(p->W2, 0, n1 * 4) == cudaSuccess &&
              cudaMemset(p->b1, 0, H * 4) == cudaSuccess && cudaMemset(p->b2, 0, N * 4) == cudaSuccess &&
              cudaMemset(p->mW1, 0, n1 * 4) == cudaSuccess && cudaMemset(p->vW1, 0, n1 * 4) == cudaSuccess &&
              cudaMemset(p->mW2, 0, n1 * 4) == cudaSuccess && cudaMemset(p->vW2, 0, n1 * 4) == cudaSuccess &&
              cudaMemset(p->mb1, 0, H * 4) == cudaSuccess && cudaMemset(p->vb1, 0, H * 4) == cudaSuccess &&
              cudaMemset(p->mb2, 0, N * 4) == cudaSuccess && cudaMemset(p->vb2, 0, N * 4) == cudaSuccess &&
              cudaMemset(p->tau, 0, p->Smax_tau * 4) == cudaSuccess && cudaMemset(p->err, 0, 4) == cudaSuccess &&
              cudaMemset(p->beta, 0, 4) == cudaSuccess && cudaMemset(p->mbeta, 0, 4) == cudaSuccess &&
              cudaMemset(p->vbeta, 0, 4) == cudaSuccess &&
              cudaDeviceSynchronize() == cudaSuccess;
  }
  if (prev >= 0) cudaSetDevice(prev);
  if (!ok || !cuda_ok) {
    pfree(p);
    delete p;
    return ok ? OMP_ERR_CUDA : OMP_ERR_OUT_OF_MEMORY;
  }
  *out = p;
  return OMP_OK;
}

omp_status omp_proposal_destroy(omp_proposal p) {
  if (!p) return OMP_OK;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(p->dev);
  cudaDeviceSynchronize();
  pfree(p);
  if (prev >= 0) cudaSetDevice(prev);
  delete p;
  return OMP_OK;
}

omp_status omp_proposal_set_weights(omp_proposal p, const float* W1, const float* b1, const float* W2,
                                    const float* b2, const float* beta, void* stream) {
  if (!p || !W1 || !b1 || !W2 || !b2 || !beta) return OMP_ERR_INVALID_ARGUMENT;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t n1 = static_cast<size_t>(p->H) * p->N;
  bool ok = cudaMemcpyAsync(p->beta, beta, 4, cudaMemcpyDefault, s) == cudaSuccess &&
            cudaMemsetAsync(p->mbeta, 0, 4, s) == cudaSuccess && cudaMemsetAsync(p->vbeta, 0, 4, s) == cudaSuccess &&
            cudaMemcpyAsync(p->W1, W1, n1 * 4, cudaMemcpyDefault, s) == cudaSuccess &&
            cudaMemcpyAsync(p->W2, W2, n1 * 4, cudaMemcpyDefault, s) == cudaSuccess &&
            cudaMemcpyAsync(p->b1, b1, p->H * 4, cudaMemcpyDefault, s) == cudaSuccess &&
            cudaMemcpyAsync(p->b2, b2, p->N * 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (!ok) return OMP_ERR_CUDA;
  refresh_bf16(p, s);
  p->step = 0;
  const size_t z1 = n1 * 4;
  ok = cudaMemsetAsync(p->mW1, 0, z1, s) == cudaSuccess && cudaMemsetAsync(p->vW1, 0, z1, s) == cudaSuccess &&
       cudaMemsetAsync(p->mW2, 0, z1, s) == cudaSuccess && cudaMemsetAsync(p->vW2, 0, z1, s) == cudaSuccess &&
       cudaMemsetAsync(p->mb1, 0, p->H * 4, s) == cudaSuccess && cudaMemsetAsync(p->vb1, 0, p->H * 4, s) == cudaSuccess &&
       cudaMemsetAsync(p->mb2, 0, p->N * 4, s) == cudaSuccess && cudaMemsetAsync(p->vb2, 0, p->N * 4, s) == cudaSuccess;
  return ok && cudaGetLastError() == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
}

omp_status omp_proposal_get_weights(omp_proposal p, float* W1, float* b1, float* W2, float* b2, float* beta,
                                    void* stream) {
  if (!p || !W1 || !b1 || !W2 || !b2 || !beta) return OMP_ERR_INVALID_ARGUMENT;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t n1 = static_cast<size_t>(p->H) * p->N;
  const bool ok = cudaMemcpyAsync(beta, p->beta, 4, cudaMemcpyDefault, s) == cudaSuccess &&
                  cudaMemcpyAsync(W1, p->W1, n1 * 4, cudaMemcpyDefault, s) == cudaSuccess &&
                  cudaMemcpyAsync(W2, p->W2, n1 * 4, cudaMemcpyDefault, s) == cudaSuccess &&
                  cudaMemcpyAsync(b1, p->b1, p->H * 4, cudaMemcpyDefault, s) == cudaSuccess &&
                  cudaMemcpyAsync(b2, p->b2, p->N * 4, cudaMemcpyDefault, s) == cudaSuccess &&
                  cudaStreamSynchronize(s) == cudaSuccess;
  return ok ? OMP_OK : OMP_ERR_CUDA;
}

omp_status omp_proposal_gradients(omp_proposal p, const float* A, const float* Y, const int32_t* labels,
                                  int64_t B, int32_t S, float* dW1, float* db1, float* dW2, float* db2,
                                  float* dbeta, float* loss_out, void* stream) {
  if (!p || !A || !Y || !labels || B < 64 || B % 64 || B > p->Bt || S < 1) return OMP_ERR_INVALID_ARGUMENT;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!gradients(p, A, Y, labels, static_cast<int>(B), S, s)) return OMP_ERR_CUDA;
  const size_t n1 = static_cast<size_t>(p->H) * p->N;
  bool ok = true;
  if (dW1) ok = ok && cudaMemcpyAsync(dW1, p->dW1, n1 * 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (dW2) ok = ok && cudaMemcpyAsync(dW2, p->dW2, n1 * 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (db1) ok = ok && cudaMemcpyAsync(db1, p->db1, p->H * 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (db2) ok = ok && cudaMemcpyAsync(db2, p->db2, p->N * 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (dbeta) ok = ok && cudaMemcpyAsync(dbeta, p->dbeta, 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (loss_out) ok = ok && cudaMemcpyAsync(loss_out, p->loss, 4, cudaMemcpyDefault, s) == cudaSuccess;
  return ok ? OMP_OK : OMP_ERR_CUDA;
}

omp_status omp_proposal_train_step(omp_proposal p, const float* A, const float* Y, const int32_t* labels,
                                   int64_t B, int32_t S, float* loss_out, void* stream) {
  if (!p || !A || !Y || !labels || B < 64 || B % 64 || B > p->Bt || S < 1) return OMP_ERR_INVALID_ARGUMENT;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!gradients(p, A, Y, labels, static_cast<int>(B), S, s)) return OMP_ERR_CUDA;
  p->step += 1;
  AdamParams a;
  a.lr = p->d.lr;
  a.beta1 = p->d.beta1;
  a.beta2 = p->d.beta2;
  a.eps = p->d.adam_eps;
  a.wd = p->d.weight_decay;
  a.c1 = static_cast<float>(1.0 / (1.0 - std::pow(static_cast<double>(a.beta1), static_cast<double>(p->step))));
  a.c2 = static_cast<float>(1.0 / (1.0 - std::pow(static_cast<double>(a.beta2), static_cast<double>(p->step))));
  adamw_matrix_kernel<<<dim3(p->N / 64, p->H / 64), 256, 0, s>>>(p->W1, p->mW1, p->vW1, p->dW1, p->H, p->N, a,
                                                                 p->W1b, nullptr);
  adamw_matrix_kernel<<<dim3(p->H / 64, p->N / 64), 256, 0, s>>>(p->W2, p->mW2, p->vW2, p->dW2, p->N, p->H, a,
                                                                 p->W2b, p->W2Tb);
  adamw_vectors_kernel<<<(p->H + p->N + 1 + 255) / 256, 256, 0, s>>>(
      AdamVec{p->b1, p->mb1, p->vb1, p->db1, p->H}, AdamVec{p->b2, p->mb2, p->vb2, p->db2, p->N},
      AdamVec{p->beta, p->mbeta, p->vbeta, p->dbeta, 1}, a);
  if (loss_out && cudaMemcpyAsync(loss_out, p->loss, 4, cudaMemcpyDefault, s) != cudaSuccess) return OMP_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
}

omp_status omp_proposal_infer(omp_proposal p, const float* A, const float* Y, int64_t B, int32_t* cand_out,
                              float* logits_out, void* stream) {
  if (!p || !A || !Y || B < 1 || B > p->d.max_batch) return OMP_ERR_INVALID_ARGUMENT;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int b = static_cast<int>(B);
  if (!features(p, A, Y, b, false, s) || !forward_hidden(p, b, false, s)) return OMP_ERR_CUDA;
  EpiF32 e{};
  e.rows = b;
  e.cols = p->N;
  e.bias = p->b2;
  e.skipX = p->X;
  e.beta = p->beta;
  e.out = p->logits;
  if (!gemm(p, p->Hh, b, p->W2b, p->N, p->H, e, s)) return OMP_ERR_CUDA;
  bool ok = launch_topk_rows(p->logits, b, p->N, p->d.topk, p->cand, s);
  if (cand_out)
    ok = ok && cudaMemcpyAsync(cand_out, p->cand, static_cast<size_t>(b) * p->d.topk * 4, cudaMemcpyDefault, s) == cudaSuccess;
  if (logits_out)
    ok = ok && cudaMemcpyAsync(logits_out, p->logits, static_cast<size_t>(b) * p->N * 4, cudaMemcpyDefault, s) == cudaSuccess;
  return ok && cudaGetLastError() == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
}

// Candidates of the method without the network: the top-K atoms of |x| = |A^T y| / (||a|| ||y||).
omp_status omp_proposal_baseline_candidates(omp_proposal p, const float* A, const float* Y, int64_t B,
                                            int32_t* cand_out, void* stream) {
  if (!p || !A || !Y || !cand_out || B < 1 || B > p->d.max_batch) return OMP_ERR_INVALID_ARGUMENT;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int b = static_cast<int>(B);
  if (!features(p, A, Y, b, false, s)) return OMP_ERR_CUDA;
  const size_t n = static_cast<size_t>(b) * p->N;
  abs_bf16_kernel<<<blocks_for(n), 256, 0, s>>>(p->X, n, p->logits);
  return launch_topk_rows(p->logits, b, p->N, p->d.topk, cand_out, s) ? OMP_OK : OMP_ERR_CUDA;
}

omp_status omp_proposal_set_thresholds(omp_proposal p, const float* tau_host, int32_t S) {
  if (!p || !tau_host || S < 1 || S > p->Smax_tau) return OMP_ERR_INVALID_ARGUMENT;
  return cudaMemcpy(p->tau, tau_host, static_cast<size_t>(S) * 4, cudaMemcpyHostToDevice) == cudaSuccess
             ? OMP_OK
             : OMP_ERR_CUDA;
}

omp_status omp_proposal_get_thresholds(omp_proposal p, float* tau_host, int32_t S) {
  if (!p || !tau_host || S < 1 || S > p->Smax_tau) return OMP_ERR_INVALID_ARGUMENT;
  return cudaMemcpy(tau_host, p->tau, static_cast<size_t>(S) * 4, cudaMemcpyDeviceToHost) == cudaSuccess
             ? OMP_OK
             : OMP_ERR_CUDA;
}

// ------------------------------------------------------------------------------ save / load
// File layout (little-endian): the 8 bytes "OMPPROP1"; int32 N, hidden, topk, S (thresholds);
// FP32 W1 (hidden x N), b1 (hidden), W2 (N x hidden), b2 (N), beta (1), tau (S); then a 64-bit
// FNV-1a hash of every byte before it, so a truncated or altered file is refused.
namespace {
constexpr char kPropMagic[8] = {'O', 'M', 'P', 'P', 'R', 'O', 'P', '1'};

uint64_t fnv1a(const unsigned char* data, size_t n, uint64_t h = 1469598103934665603ull) {
  for (size_t i = 0; i < n; ++i) {
    h ^= data[i];
    h *= 1099511628211ull;
  }
  return h;
}

struct PropFile {
  int32_t hdr[4];  // N, hidden, topk, S
  std::vector<float> W1, b1, W2, b2, beta, tau;
};

size_t prop_payload_floats(const int32_t* hdr) {
  const size_t N = static_cast<size_t>(hdr[0]), H = static_cast<size_t>(hdr[1]);
  return 2 * N * H + H + N + 1 + static_cast<size_t>(hdr[3]);
}
}  // namespace

omp_status omp_proposal_save(omp_proposal p, const char* path) {
  if (!p || !path) return OMP_ERR_INVALID_ARGUMENT;
  const int32_t hdr[4] = {p->N, p->H, p->d.topk, p->Smax_tau};
  const size_t n1 = static_cast<size_t>(p->H) * p->N;
  std::vector<float> buf(prop_payload_floats(hdr));
  float* W1 = buf.data();
  float* W2 = W1 + n1;
  float* b1 = W2 + n1;
  float* b2 = b1 + p->H;
  float* beta = b2 + p->N;
  float* tau = beta + 1;
  omp_status st = omp_proposal_get_weights(p, W1, b1, W2, b2, beta, nullptr);
  if (st == OMP_OK) st = omp_proposal_get_thresholds(p, tau, p->Smax_tau);
  if (st != OMP_OK) return st;
  // written in the file's order: W1, b1, W2, b2, beta, tau
  std::vector<unsigned char> out(sizeof(kPropMagic) + sizeof(hdr) + buf.size() * 4);
  unsigned char* o = out.data();
  std::memcpy(o, kPropMagic, sizeof(kPropMagic));
  o += sizeof(kPropMagic);
  std::memcpy(o, hdr, sizeof(hdr));
  o += sizeof(hdr);
  const std::pair<const float*, size_t> parts[] = {{W1, n1}, {b1, static_cast<size_t>(p->H)}, {W2, n1},
                                                   {b2, static_cast<size_t>(p->N)}, {beta, 1},
                                                   {tau, static_cast<size_t>(p->Smax_tau)}};
  for (const auto& part : parts) {
    std::memcpy(o, part.first, part.second * 4);
    o += part.second * 4;
  }
  const uint64_t h = fnv1a(out.data(), out.size());
  FILE* f = std::fopen(path, "wb");
  if (!f) return OMP_ERR_INVALID_ARGUMENT;
  const bool ok = std::fwrite(out.data(), 1, out.size(), f) == out.size() &&
                  std::fwrite(&h, sizeof(h), 1, f) == 1;
  return (std::fclose(f) == 0 && ok) ? OMP_OK : OMP_ERR_INVALID_ARGUMENT;
}

omp_status omp_proposal_load(omp_proposal p, const char* path) {
  if (!p || !path) return OMP_ERR_INVALID_ARGUMENT;
  FILE* f = std::fopen(path, "rb");
  if (!f) return OMP_ERR_INVALID_ARGUMENT;
  std::vector<unsigned char> in;
  unsigned char chunk[1 << 16];
  size_t got;
  while ((got = std::fread(chunk, 1, sizeof(chunk), f)) > 0) in.insert(in.end(), chunk, chunk + got);
  std::fclose(f);
  const size_t head = sizeof(kPropMagic) + 4 * sizeof(int32_t);
  if (in.size() < head + sizeof(uint64_t) || std::memcmp(in.data(), kPropMagic, sizeof(kPropMagic)) != 0)
    return OMP_ERR_INVALID_ARGUMENT;
  int32_t hdr[4];
  std::memcpy(hdr, in.data() + sizeof(kPropMagic), sizeof(hdr));
  if (hdr[0] != p->N || hdr[1] != p->H || hdr[3] < 1 || hdr[3] > 4096) return OMP_ERR_INVALID_ARGUMENT;
  const size_t nf = prop_payload_floats(hdr);
  if (in.size() != head + nf * 4 + sizeof(uint64_t)) return OMP_ERR_INVALID_ARGUMENT;
  uint64_t h = 0;
  std::memcpy(&h, in.data() + head + nf * 4, sizeof(h));
  if (h != fnv1a(in.data(), head + nf * 4)) return OMP_ERR_INVALID_ARGUMENT;
  std::vector<float> buf(nf);
  std::memcpy(buf.data(), in.data() + head, nf * 4);
  const size_t n1 = static_cast<size_t>(p->H) * p->N;
  const float* W1 = buf.data();
  const float* b1 = W1 + n1;
  const float* W2 = b1 + p->H;
  const float* b2 = W2 + n1;
  const float* beta = b2 + p->N;
  const float* tau = beta + 1;
  omp_status st = omp_proposal_set_weights(p, W1, b1, W2, b2, beta, nullptr);
  if (st == OMP_OK && cudaDeviceSynchronize() != cudaSuccess) st = OMP_ERR_CUDA;
  // thresholds: as many as both the file and the proposal hold; the rest accept every step
  const int S = hdr[3] < p->Smax_tau ? hdr[3] : p->Smax_tau;
  std::vector<float> t(static_cast<size_t>(p->Smax_tau), 0.f);
  std::memcpy(t.data(), tau, static_cast<size_t>(S) * 4);
  if (st == OMP_OK) st = omp_proposal_set_thresholds(p, t.data(), p->Smax_tau);
  return st;
}

omp_status omp_proposal_calibrate(omp_proposal p, const float* drops, int64_t B, int32_t S, float quantile,
                                  void* stream) {
  if (!p || !drops || B < 1 || S < 1 || S > p->Smax_tau || !(quantile >= 0.f && quantile <= 1.f))
    return OMP_ERR_INVALID_ARGUMENT;
  quantile_cols_kernel<<<S, 256, 0, static_cast<cudaStream_t>(stream)>>>(drops, static_cast<int>(B), S,
                                                                           quantile, p->tau);
  return cudaGetLastError() == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
}

omp_status omp_topk_rows(const float* logits, int64_t rows, int64_t N, int32_t K, int32_t* idx_out, void* stream) {
  if (!logits || !idx_out || rows < 1 || N < 1 || K < 1 || K > N || N > (1 << 30)) return OMP_ERR_INVALID_ARGUMENT;
  return launch_topk_rows(logits, static_cast<int>(rows), static_cast<int>(N), K, idx_out,
                          static_cast<cudaStream_t>(stream))
             ? OMP_OK
             : OMP_ERR_CUDA;
}

}  // extern "C"

namespace ompk {
bool proposal_run_inference(omp_proposal p, const float* A, const float* Y, int B, cudaStream_t s) {
  if (B > p->d.max_batch) return false;
  if (!features(p, A, Y, B, false, s) || !forward_hidden(p, B, false, s)) return false;
  EpiF32 e{};
  e.rows = B;
  e.cols = p->N;
  e.bias = p->b2;
  e.skipX = p->X;
  e.beta = p->beta;
  e.out = p->logits;
  if (!gemm(p, p->Hh, B, p->W2b, p->N, p->H, e, s)) return false;
  return launch_topk_rows(p->logits, B, p->N, p->d.topk, p->cand, s);
}

// accessors used by the learned solve (runtime.cu)
const int* proposal_candidates(omp_proposal p) { return p->cand; }
int proposal_topk(omp_proposal p) { return p->d.topk; }
const float* proposal_tau(omp_proposal p) { return p->tau; }
int proposal_tau_len(omp_proposal p) { return p->Smax_tau; }
float* proposal_tau_mut(omp_proposal p) { return p->tau; }
}  // namespace ompk
