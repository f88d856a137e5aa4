// The FP32 path's selection behind the tensor cores. A BF16 correlation (corr_tc.cu) leaves per
// position the lists of its best columns; |BF16 score - FP32 score| <= eps ||r||, with eps from the
// actual rounding errors of the atoms and of the residual row plus both accumulations (data_bound),
// so only columns within 2 eps ||r|| of the best BF16 score can have the best FP32 score. Here a
// warp per position takes those: one alone is the pick; up to seven are scored in FP32 exactly as
// corr_simt.cu scores them (one chain of FMAs over m), so the pick is the one a full FP32 correlation
// makes. A position with more (the lists may then lack some), or whose norm leaves FP32's normal
// range, goes on a list for which every atom is scored in FP32 (launch_corr_overflow). After a step that
// left most positions on that list the next ones up to a multiple of four do without the filter: the BF16
// correlation returns at once and the list holds every position (filter_rests).
//
// The full FP32 correlation of 1000 signals with 8192 atoms of length 1024 takes 309 us a step, the
// BF16 one 20, this kernel 9.7 and the overflow launch 3.4 on average (1.7 where empty). This kernel is bound by the
// latency of a position's round trips and of its chain (four cycles an element at best); with chunks of
// 256 elements it takes 9.4 there, but 122 registers a thread instead of 80 cost a large batch residency.
#include "common.cuh"

namespace ompk {
namespace {

constexpr int kWarpsF = 4;   // warps (positions) per block
constexpr int kMaxC = 7;     // candidates scored here
constexpr int kCh = 128;     // elements of a row staged at a time
constexpr int kBatch = 4;   // 16-byte reads ahead of a chain
constexpr int kLd = kCh + 4; // padded: the lanes' 16-byte reads of different rows meet no bank twice

__global__ void __launch_bounds__(32 * kWarpsF) filter_select_kernel(Ws ws, int k) {
  __shared__ __align__(16) float stage[kWarpsF][(kMaxC + 1) * kLd];
  k = iter_of(ws, k);
  const bool rests = filter_rests(ws, k);
  const int L = ws.cnt[k + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int p = blockIdx.x * kWarpsF + warp;
  if (p >= L) return;  // the whole warp
  if (rests) {
    if (lane == 0) ws.ovf[p] = p;
    if (p == 0 && lane == 0) ws.ovf_cnt[k] = L;
    return;
  }
  Lists l;
  const int total = tc_piece_count(ws, L, p) * kMaxTopk;
  load_lists(ws, total, p, lane, l);
  const int id = ws.live[k & 1][p];
  const float win = ws.win_pos[p];
  const float rn = ws.rnorm[id];
  settle_lists(ws, total, p, lane, l);
  // The window's candidates, best first; lane c < n keeps candidate c. win is three bounds: two of
  // them, rounded up, below the best.
  int n = 0, mine = -1;
  float best = -1.f, thr = 0.f;
  while (n <= kMaxC) {
    int idx;
    const float v = take_best(l, idx);
    if (n == 0) {
      best = v;
      thr = best - 0.66667f * win;
    }
    if (!(v >= 0.f) || v < thr) break;
    if (lane == n) mine = idx;
    ++n;
  }
  const bool ranged = rn > 1e-12f && rn < 1e12f && win < 1e30f;  // false for a NaN
  if (!ranged || n == 0 || n > kMaxC) {
    if (lane == 0) ws.ovf[atomicAdd(ws.ovf_cnt + k, 1)] = p;
    return;
  }
  if (n == 1) {
    if (lane == 0) ws.cand1[p] = pack_key(best, mine);
    return;
  }
  // rows of the candidates and the residual, kCh elements at a time: loaded a chunk ahead, side by
  // side by the warp, then read by the lane whose chain it is
  float* st = stage[warp];
  const int M4 = ws.Mp >> 2;
  const float4* src[kMaxC + 1];
#pragma unroll
  for (int c = 0; c < kMaxC; ++c) {
    const int idx = __shfl_sync(0xffffffffu, mine, c);
    src[c] = reinterpret_cast<const float4*>(ws.A32 + static_cast<size_t>(c < n ? idx : 0) * ws.Mp);
  }
  src[kMaxC] = reinterpret_cast<const float4*>(ws.R32 + static_cast<size_t>(id) * ws.Mp);
  float4 v[kMaxC + 1];
  auto load = [&](int s0) {
#pragma unroll
    for (int c = 0; c <= kMaxC; ++c)
      v[c] = (c < n || c == kMaxC) && s0 + lane < M4 ? src[c][s0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  load(0);
  float acc = 0.f;
  for (int s0 = 0; s0 < M4; s0 += 32) {
    __syncwarp();  // the previous chunk has been read
#pragma unroll
    for (int c = 0; c <= kMaxC; ++c) *reinterpret_cast<float4*>(st + c * kLd + 4 * lane) = v[c];
    __syncwarp();
    if (s0 + 32 < M4) load(s0 + 32);
    if (lane < n) {
      const float4* a = reinterpret_cast<const float4*>(st + lane * kLd);
      const float4* r = reinterpret_cast<const float4*>(st + kMaxC * kLd);
      // past Mp both are zero, which adds nothing; the reads go a batch ahead of the chain, which
      // waited for each before (13.7 cycles an element, 9 now: the next chunk's loads are the rest)
      float4 x[2][kBatch], y[2][kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        x[0][q] = a[q];
        y[0][q] = r[q];
      }
#pragma unroll
      for (int s = 0; s < kCh / 4; s += kBatch) {
        const int cur = s / kBatch & 1;
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
          if (s + kBatch < kCh / 4) {
            x[cur ^ 1][q] = a[s + kBatch + q];
            y[cur ^ 1][q] = r[s + kBatch + q];
          }
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
          acc = fmaf(y[cur][q].x, x[cur][q].x, acc);
          acc = fmaf(y[cur][q].y, x[cur][q].y, acc);
          acc = fmaf(y[cur][q].z, x[cur][q].z, acc);
          acc = fmaf(y[cur][q].w, x[cur][q].w, acc);
        }
      }
    }
  }
  float sc = -1.f;
  int ix = 0x7fffffff;
  if (lane < n) {
    sc = fabsf(acc) * __ldg(ws.inv_norm + mine);
    ix = mine;
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {  // lanes 0..7
    const float os = __shfl_xor_sync(0xffffffffu, sc, o);
    const int oi = __shfl_xor_sync(0xffffffffu, ix, o);
    if (better(os, oi, sc, ix)) {
      sc = os;
      ix = oi;
    }
  }
  if (lane == 0) ws.cand1[p] = pack_key(sc, ix);
}

}  // namespace

void launch_filter_select(const Ws& ws, int k, int B, cudaStream_t s) {
  filter_select_kernel<<<(B + kWarpsF - 1) / kWarpsF, 32 * kWarpsF, 0, s>>>(ws, k);
}

}  // namespace ompk
