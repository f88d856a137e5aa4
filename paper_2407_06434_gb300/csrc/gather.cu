// q = A_{S+n*} F[:,k] for dictionaries that L2 does not hold, between the head and the tail of a step
// (append.cuh).
//
// A step of a large batch reads each atom row several times over (4096 signals with 33 atoms each
// gather 135 thousand rows of 32768): in one kernel, signal by signal, nearly all of it from HBM. Here
// the row length is cut into pieces and the blocks of all signals' first pieces come before any second,
// so that a piece of the dictionary stays in L2 while the whole batch reads it: HBM then reads the
// dictionary about once a step. 4096 signals, 4096 x 32768, FP8, 64 steps (us a step on average): one
// kernel 463; head 127, gather 157, tail 35 (60 steps; the first four, in one kernel, 234). (A head of one
// warp per signal took 190: its rescoring reads up to eight rows of 16 KB one warp at a time.)
//
// q's rows are summed in the same order as in the one kernel: the same bits.
#include "append.cuh"

namespace ompk {
namespace {

// A dictionary up to this many bytes stays in L2 as a whole, or nearly: at 134 MB (2048 x 16384, two
// warps a signal) the three launches took 191 us a step against 193 for one. Of a larger one, a piece.
constexpr size_t kWholeBytes = 160u << 20;
constexpr size_t kPieceBytes = 72u << 20;
constexpr int kApartMinB = 1024;  // fewer signals do not read a row often enough

// q += sum_a f[a] row_a over the rows sup[0..na), in order, for this thread's slots s0 + t * stride
template <int V, bool G24>
__device__ __forceinline__ void gather_rows(const Ws& ws, const float* f, const int* sup, int na, int s0, int stride,
                                            int lim, float4 (&q)[V]) {
  constexpr int R = 6;  // rows in flight
  auto add = [&](float c, int t, const Slot4<G24>& w) {
    const float4 v = widen<G24>(w);
    q[t].x = fmaf(c, v.x, q[t].x);
    q[t].y = fmaf(c, v.y, q[t].y);
    q[t].z = fmaf(c, v.z, q[t].z);
    q[t].w = fmaf(c, v.w, q[t].w);
  };
  int a = 0;
  for (; a + R <= na; a += R) {
    Slot4<G24> w[R][V];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int n = sup[a + i];
#pragma unroll
      for (int t = 0; t < V; ++t) {
        const int s = s0 + t * stride;
        w[i][t] = s < lim ? gather4<G24>(ws, n, s) : zero4<G24>();
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float c = f[a + i];
#pragma unroll
      for (int t = 0; t < V; ++t) add(c, t, w[i][t]);
    }
  }
  if (a < na) {  // the rest, side by side too
    Slot4<G24> w[R - 1][V];
#pragma unroll
    for (int i = 0; i < R - 1; ++i) {
      const int n = sup[min(a + i, na - 1)];
#pragma unroll
      for (int t = 0; t < V; ++t) {
        const int s = s0 + t * stride;
        w[i][t] = a + i < na && s < lim ? gather4<G24>(ws, n, s) : zero4<G24>();
      }
    }
#pragma unroll
    for (int i = 0; i < R - 1; ++i)
      if (a + i < na) {
        const float c = f[a + i];
#pragma unroll
        for (int t = 0; t < V; ++t) add(c, t, w[i][t]);
      }
  }
}

// q of every live position over slots [c cs, (c + 1) cs) of the rows, c = blockIdx.y: the blocks of a
// piece are consecutive, so the whole batch reads one piece of the dictionary before the next
template <bool G24>
__global__ void __launch_bounds__(128, 6) gather_piece_kernel(Ws ws, int k, int cs) {
  k = iter_of(ws, k);
  const int p = blockIdx.x;
  if (p >= ws.cnt[k + 1]) return;
  __shared__ float f[32 * kMaxBlk + 1];
  __shared__ int sup[32 * kMaxBlk + 1];
  const int4 sel = ws.sel[p];
  const int id = ws.live[k & 1][p], kk = ws.livek[k & 1][p];
  if (sel.x < 0) return;
  const float* fg = ws.F32 + static_cast<size_t>(id) * ws.Fstride + static_cast<size_t>(kk) * (kk + 1) / 2;
  const int* sg = ws.sup + static_cast<size_t>(id) * ws.Smax;
  for (int i = threadIdx.x; i <= kk; i += blockDim.x) {
    f[i] = fg[i];
    sup[i] = sg[i];
  }
  __syncthreads();
  const int base = blockIdx.y * cs, lim = min(ws.Mp >> 2, base + cs);
  float4* qg = reinterpret_cast<float4*>(ws.Q + static_cast<size_t>(p) * ws.Mp);
  for (int s0 = base + threadIdx.x; s0 < lim; s0 += 2 * blockDim.x) {
    float4 q[2];
    q[0] = q[1] = make_float4(0.f, 0.f, 0.f, 0.f);
    gather_rows<2, G24>(ws, f, sup, kk + 1, s0, blockDim.x, lim, q);
    qg[s0] = q[0];
    if (s0 + static_cast<int>(blockDim.x) < lim) qg[s0 + blockDim.x] = q[1];
  }
}

int pieces_of(const Ws& ws) {
  const size_t bytes = static_cast<size_t>(ws.N) * ws.Mp * 4;
  return static_cast<int>((bytes + kPieceBytes - 1) / kPieceBytes);
}

}  // namespace

bool gather_apart_shape(int64_t N, int64_t Mp, int64_t Bmax) {
  return static_cast<size_t>(N) * Mp * 4 > kWholeBytes && Bmax >= kApartMinB;
}
// Two launches more and q's way through memory cost about as much at every step, while the rows that
// are read from L2 and not from HBM grow with the step. So the first steps are one kernel; from which
// step on three are faster depends on the row length (warps a signal), the batch and on what the head
// carries besides (BF16: two candidate rows in shared memory for the threshold). Measured, us a step on
// average over solves of 12, 48 and 100 steps, one kernel / three: 1024 x 60000, FP8, 4096 signals 235 /
// 243, 290 / 284, 390 / 353, 1024 signals 84 / 93, 100 / 108, 146 / 149; 2048 x 24576, 4096 signals, FP8
// 239 / 242, 329 / 296, 448 / 366, BF16 329 / 348, 394 / 391, 510 / 455, FP32 (48) 417 / 401; 2048 x 24576,
// 1024 signals, FP8 90 / 98, 106 / 115, 137 / 139; 4096 x 16384, 4096 signals, FP8 334 / 341, 517 / 438, 751 /
// 557, BF16 464 / 492, 592 / 569, 821 / 667, FP32 (48) 645 / 593; 1024 signals, FP8 114 / 115, 160 / 144,
// 222 / 178, BF16 147 / 157, 180 / 184, 245 / 215.
bool gather_apart(const Ws& ws, int B, int k, int S) {
  if (!ws.Q || B < kApartMinB) return false;
  const bool many = B >= 2048, bf16 = ws.prec == OMP_PREC_BF16, fp8 = ws.prec == OMP_PREC_FP8_E4M3;
  int from;
  if (ws.Mp <= 1024)
    from = many ? 24 : 64;
  else if (ws.Mp <= 2048)
    from = bf16 ? (many ? 24 : 40) : fp8 ? (many ? 7 : 48) : (many ? 18 : 28);
  else
    from = bf16 ? (many ? 19 : 28) : fp8 ? 4 : 12;
  return (k >= 0 ? k : S / 2) >= from;
}

void launch_gather(const Ws& ws, int k, int B, cudaStream_t s) {
  const int M4 = ws.Mp / 4;
  const int nc = pieces_of(ws);
  const int cs = ((M4 + nc - 1) / nc + 31) / 32 * 32;  // whole 512-byte pieces of a row
  const int T = cs / 2 < 128 ? (cs / 2 + 31) / 32 * 32 : 128;
  const dim3 grid(B, (M4 + cs - 1) / cs);
  if (ws.A24h)
    gather_piece_kernel<true><<<grid, T, 0, s>>>(ws, k, cs);
  else
    gather_piece_kernel<false><<<grid, T, 0, s>>>(ws, k, cs);
}

}  // namespace ompk
