// FP32 correlation on the CUDA cores (the plain-FP32 path) and the FP32 Gram matrix.
//
// Both are the contraction C = X A^T over the padded signal length Mp with both operands stored
// K-major (rows of Mp contiguous floats): for the correlation X holds the live residuals
// (batched as one GEMM, Sec. 3.2 eq:bmm), for the Gram matrix X = A^T itself (Sec. 2.2), of which
// only the upper triangle is computed (the lower is its mirror image, bit for bit).
// A tile of 128 rows x 8 TN atoms per 128-thread block, 8 x TN outputs per thread, K chunks of 32
// staged through double-buffered shared memory, transposed. Every output is one FMA chain over m
// in order, two outputs to an FFMA2. What bounds it: 8 x 8 outputs a thread read shared memory as
// long as they multiply (a 16-byte read takes four cycles of the SM's 128 bytes whatever it
// broadcasts), 8 x 16 three quarters of that; the chunks come as whole 128-byte lines, since loads
// of 64 or 32 bytes a row cost more than the products could hide (Gram matrix of 8192 atoms of
// length 1024: 2764 us for both triangles with 8 x 8 outputs and FMAs, 1301 us for one with FFMA2,
// 1252 us with 8 x 16 outputs, 1148 us with whole lines: 61 TFLOP/s of 80.5 nominal).
//
// A third form stores C = Y A^T for signals 0..B-1 (rows of R32 in signal order) into the c0
// workspace: the exact first correlation the Gram-space solve starts from.
//
// The correlation never writes C: the epilogue forms the score |c| / ||a_n|| (Alg. 1), takes
// each thread's best atom in ascending index order (strict '>', so the lowest index keeps a
// tie), reduces across the 8 threads that share a signal with warp shuffles, and merges the
// tile's winner into the signal's packed (score, ~index) key with one 64-bit atomicMax: the
// maximum key is the highest score and, among equal scores, the lowest index, whatever order
// the tiles finish in.
#include "common.cuh"

namespace ompk {

namespace {
constexpr int kCorrelate = 0, kGram = 1, kStoreC = 2, kOverflow = 3;

// Two FP32 FMAs in one instruction (each rounded as fmaf): d.lo += x.lo a.lo, d.hi += x.hi a.hi
__device__ __forceinline__ void ffma2(unsigned long long& d, unsigned long long x, unsigned long long a) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(x), "l"(a));
}
__device__ __forceinline__ float lo2(unsigned long long v) { return __uint_as_float(static_cast<uint32_t>(v)); }
__device__ __forceinline__ float hi2(unsigned long long v) { return __uint_as_float(static_cast<uint32_t>(v >> 32)); }

__device__ __forceinline__ unsigned long long dup2(float x) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}

constexpr int BM = 128, BK = 32;
constexpr int TX = 8, THREADS = 128;  // threads along the atoms; 16 along the rows, 8 rows each

// kOverflow: a block holds two groups of threads, each with tiles, shared memory and barrier of its own
template <int MODE>
constexpr int kGroups = MODE == kOverflow ? 2 : 1;
template <int MODE>
__device__ __forceinline__ void tile_sync() {
  if (MODE == kOverflow)
    asm volatile("bar.sync %0, %1;" ::"r"(static_cast<int>(threadIdx.x) / THREADS + 1), "r"(THREADS) : "memory");
  else
    __syncthreads();
}

// One tile: rows by * 128 .., atoms bx * 8 TN ..; L rows in all
template <int MODE, int TN>
__device__ __forceinline__ void simt_tile(const Ws& ws, int bx, int by, int L, const int* live, const int* ovf) {
  constexpr bool GRAM = MODE == kGram;
  constexpr int BN = TX * TN;
  constexpr int RS = THREADS / (BK / 4);             // rows apart of a thread's loads (16)
  constexpr int LX = BM / RS / 2, LA = BN / RS / 2;  // loads per thread and half chunk
  extern __shared__ __align__(16) float smem_f[];
  float* Xs = smem_f + (kGroups<MODE> > 1 ? threadIdx.x / THREADS * (2 * BK * (BM + BN)) : 0);  // 2 x BK x BM
  float* As = Xs + 2 * BK * BM;                                                                // 2 x BK x BN
  const int tid = kGroups<MODE> > 1 ? threadIdx.x % THREADS : threadIdx.x;
  const int n0 = bx * BN;
  const int p0 = by * BM;
  // a warp loads 4 rows x 128 bytes (whole lines); element (k, r) of a chunk is stored at column
  // r ^ 4 ((k / 4) % 8) of its row k, so that the transposed stores of a warp meet every bank once
  // and four consecutive rows stay one aligned float4
  const int lrow = tid >> 3, lq = tid & 7;
  const float* xsrc[2 * LX];
  const float* asrc[2 * LA];
#pragma unroll
  for (int i = 0; i < 2 * LX; ++i) {
    const int p = p0 + lrow + RS * i;
    const int row = p >= L ? -1 : (GRAM || MODE == kStoreC) ? p : live[MODE == kOverflow ? ovf[p] : p];
    xsrc[i] = row < 0 ? nullptr : (GRAM ? ws.A32 : ws.R32) + static_cast<size_t>(row) * ws.Mp + 4 * lq;
  }
#pragma unroll
  for (int i = 0; i < 2 * LA; ++i) {
    const int n = n0 + lrow + RS * i;
    asrc[i] = n < ws.N ? ws.A32 + static_cast<size_t>(n) * ws.Mp + 4 * lq : nullptr;
  }
  float4 xr[LX], ar[LA];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto gload = [&](int kc, int h) {
#pragma unroll
    for (int i = 0; i < LX; ++i)
      xr[i] = xsrc[h * LX + i] ? __ldg(reinterpret_cast<const float4*>(xsrc[h * LX + i] + kc)) : zero;
#pragma unroll
    for (int i = 0; i < LA; ++i)
      ar[i] = asrc[h * LA + i] ? __ldg(reinterpret_cast<const float4*>(asrc[h * LA + i] + kc)) : zero;
  };
  auto sstore = [&](int buf, int h) {
#pragma unroll
    for (int i = 0; i < LX; ++i) {
      float* d = Xs + (buf * BK + 4 * lq) * BM + ((lrow + RS * (h * LX + i)) ^ (4 * lq));
      d[0] = xr[i].x;
      d[BM] = xr[i].y;
      d[2 * BM] = xr[i].z;
      d[3 * BM] = xr[i].w;
    }
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      float* d = As + (buf * BK + 4 * lq) * BN + ((lrow + RS * (h * LA + i)) ^ (4 * lq));
      d[0] = ar[i].x;
      d[BN] = ar[i].y;
      d[2 * BN] = ar[i].z;
      d[3 * BN] = ar[i].w;
    }
  };

  // acc2[i][j2]: outputs (row i, atoms 2 j2 and 2 j2 + 1); every output is one chain of FMAs over
  // m = 0, 1, ..., Mp - 1
  unsigned long long acc2[8][TN / 2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc2[i][j] = 0ull;

  const int tx = tid % TX, ty = tid / TX;
  const int nk = ws.Mp / BK;
  // the fragments of step kk + 1 are read while the products of step kk run
  float4 xf[2][2];
  ulonglong2 af[2][TN / 4];
  auto frag = [&](int f, int buf, int kk) {
    const int w = 4 * (kk >> 2);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      xf[f][h] = *reinterpret_cast<const float4*>(Xs + (buf * BK + kk) * BM + h * (BM / 2) + ((ty * 4) ^ w));
#pragma unroll
    for (int h = 0; h < TN / 4; ++h)
      af[f][h] = *reinterpret_cast<const ulonglong2*>(As + (buf * BK + kk) * BN + h * (4 * TX) + ((tx * 4) ^ w));
  };
  gload(0, 0);
  sstore(0, 0);
  gload(0, 1);
  sstore(0, 1);
  tile_sync<MODE>();
  for (int kt = 0; kt < nk; ++kt) {
    const int buf = kt & 1;
    const bool more = kt + 1 < nk;
    if (more) gload((kt + 1) * BK, 0);
    frag(0, buf, 0);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const int f = kk & 1;
      if (kk == BK / 2 && more) {  // the next chunk comes in halves, half the registers in flight
        sstore(buf ^ 1, 0);
        gload((kt + 1) * BK, 1);
      }
      if (kk + 1 < BK) frag(f ^ 1, buf, kk + 1);
      const float xs[8] = {xf[f][0].x, xf[f][0].y, xf[f][0].z, xf[f][0].w,
                           xf[f][1].x, xf[f][1].y, xf[f][1].z, xf[f][1].w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long xx = dup2(xs[i]);
#pragma unroll
        for (int h = 0; h < TN / 4; ++h) {
          ffma2(acc2[i][2 * h], xx, af[f][h].x);
          ffma2(acc2[i][2 * h + 1], xx, af[f][h].y);
        }
      }
    }
    if (more) sstore(buf ^ 1, 1);
    tile_sync<MODE>();
  }
  auto acc = [&](int i, int j) { return (j & 1) ? hi2(acc2[i][j >> 1]) : lo2(acc2[i][j >> 1]); };

  // atoms of this thread, ascending: n0 + 32 h + 4 tx + {0..3}; rows p0 + 64 h + 4 ty + {0..3}
  auto ncol = [&](int j) { return n0 + (j >> 2) * (4 * TX) + tx * 4 + (j & 3); };
  auto prows = [&](int i) { return p0 + (i >> 2) * (BM / 2) + ty * 4 + (i & 3); };

  if (GRAM || MODE == kStoreC) {
    // C row-major in rows of ldg, 16 bytes at a time (the products past N are zeros); the Gram form
    // stores the mirror image G[n][p] as well
    float* C = GRAM ? ws.gram : ws.c0;
    auto store4 = [&](int row, int col, float a, float b, float c, float d) {
      if (col < ws.ldg)
        *reinterpret_cast<float4*>(C + static_cast<size_t>(row) * ws.ldg + col) = make_float4(a, b, c, d);
    };
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < TN; j += 4)
        if (prows(i) < L) store4(prows(i), ncol(j), acc(i, j), acc(i, j + 1), acc(i, j + 2), acc(i, j + 3));
    if (GRAM) {
#pragma unroll
      for (int j = 0; j < TN; ++j)
#pragma unroll
        for (int i = 0; i < 8; i += 4)
          if (ncol(j) < ws.N) store4(ncol(j), prows(i), acc(i, j), acc(i + 1, j), acc(i + 2, j), acc(i + 3, j));
    }
    return;
  }

  float inv[TN];
#pragma unroll
  for (int j = 0; j < TN; ++j) inv[j] = ncol(j) < ws.N ? __ldg(ws.inv_norm + ncol(j)) : 0.f;
  if (MODE == kCorrelate && ws.cand2) {
    // Margins recorded: each row's best two atoms of the tile (same scan and ties), then
    // cand1 keeps the global best as before and cand2 receives every key that loses a merge
    // (the smaller of the old and the new key of each atomicMax) and each tile's second best,
    // so that it ends with the largest key other than the best: the runner-up.
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int prow = prows(i);
      float b1 = -1.f, b2 = -1.f;
      int i1 = 0x7fffffff, i2 = 0x7fffffff;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        if (ncol(j) < ws.N) {
          const float sc = fabsf(acc(i, j)) * inv[j];
          if (better(sc, ncol(j), b1, i1)) {
            b2 = b1;
            i2 = i1;
            b1 = sc;
            i1 = ncol(j);
          } else if (better(sc, ncol(j), b2, i2)) {
            b2 = sc;
            i2 = ncol(j);
          }
        }
      }
#pragma unroll
      for (int o = 1; o < TX; o <<= 1) {
        const float o1 = __shfl_xor_sync(0xffffffffu, b1, o);
        const int oi1 = __shfl_xor_sync(0xffffffffu, i1, o);
        const float o2 = __shfl_xor_sync(0xffffffffu, b2, o);
        const int oi2 = __shfl_xor_sync(0xffffffffu, i2, o);
        if (better(o1, oi1, b1, i1)) {
          if (!better(b1, i1, o2, oi2)) {
            b1 = o2;  // the partner holds both: (o1, o2)
            i1 = oi2;
          }
          b2 = b1;
          i2 = i1;
          b1 = o1;
          i1 = oi1;
        } else if (better(o1, oi1, b2, i2)) {
          b2 = o1;
          i2 = oi1;
        }
      }
      if (tx == 0 && prow < L && i1 < ws.N) {
        const unsigned long long k1 = pack_key(b1, i1);
        const unsigned long long old = atomicMax(ws.cand1 + prow, k1);
        atomicMax(ws.cand2 + prow, old < k1 ? old : k1);
        if (i2 < ws.N) atomicMax(ws.cand2 + prow, pack_key(b2, i2));
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int prow = prows(i);
    float best = -1.f;
    int bidx = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      if (ncol(j) < ws.N) {
        const float s = fabsf(acc(i, j)) * inv[j];
        if (s > best) {
          best = s;
          bidx = ncol(j);
        }
      }
    }
#pragma unroll
    for (int o = 1; o < TX; o <<= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
      if (better(ob, oi, best, bidx)) {
        best = ob;
        bidx = oi;
      }
    }
    if (tx == 0 && prow < L && bidx < ws.N)
      atomicMax(ws.cand1 + (MODE == kOverflow ? ovf[prow] : prow), pack_key(best, bidx));
  }
}

// MODE kCorrelate: k is the iteration; kGram: k unused; kStoreC: k is the number of signals;
// kOverflow: as kCorrelate for the positions that the filter could not decide (their number is not
// known at the launch: a grid that fills the SMs strides over the tiles).
// TN atoms per thread: a tile of 128 rows x 8 TN atoms.
template <int MODE, int TN>
__global__ void __launch_bounds__(THREADS * kGroups<MODE>, 2 / kGroups<MODE>) simt_tile_kernel(Ws ws, int k) {
  constexpr bool GRAM = MODE == kGram;
  constexpr int BN = TX * TN;
  const int bx = blockIdx.x, by = blockIdx.y;  // (kOverflow: the grid is one row)
  // G is symmetric and every entry's products and sums are the same in both orders, so only tiles
  // that reach the diagonal or lie above it are computed, and each stores its mirror image too
  if (GRAM && bx * BN + BN <= by * BM) return;
  int L;
  const int* live = nullptr;
  const int* ovf = nullptr;
  if (GRAM) {
    L = ws.N;
  } else if (MODE == kStoreC) {
    L = k;
  } else {
    k = iter_of(ws, k);
    L = MODE == kOverflow ? ws.ovf_cnt[k] : ws.cnt[k + 1];
    live = ws.live[k & 1];
    ovf = ws.ovf;
  }
  if (MODE == kOverflow) {
    const int cols = (ws.N + BN - 1) / BN, tiles = (L + BM - 1) / BM * cols;
    const int grp = threadIdx.x / THREADS;  // (no tile for the second group before every block has one)
    for (int t = blockIdx.x + grp * gridDim.x; t < tiles; t += 2 * gridDim.x) {
      simt_tile<MODE, TN>(ws, t % cols, t / cols, L, live, ovf);
      tile_sync<MODE>();  // the next tile overwrites the chunks
    }
    return;
  }
  if (by * BM >= L) return;
  simt_tile<MODE, TN>(ws, bx, by, L, live, ovf);
}

template <int TN>
constexpr size_t tile_bytes() {
  return 2 * BK * (BM + TX * TN) * sizeof(float);
}

template <int MODE, int TN>
void launch_one(const Ws& ws, int rows, int k, cudaStream_t s) {
  const dim3 grid((ws.N + TX * TN - 1) / (TX * TN), (rows + BM - 1) / BM);
  simt_tile_kernel<MODE, TN><<<grid, THREADS, tile_bytes<TN>(), s>>>(ws, k);
}

// Output tiles of 128 rows x 128, 96 or 64 atoms: the width whose rounds over the SMs (a lone
// round counts 1.25, one block's four warps leave an SM's latencies exposed) times its area are
// least, the widest on a tie (it reads the least from shared memory per product). Measured, us at
// widths 128 / 96 / 64: correlation of 1000 signals x 8192 atoms x 1024 365 / 322 / 309; first
// correlation of 1200 x 1207 x 8064 1015 / 644 / 752; Gram matrix of 2048 atoms of length 512
// 99 / 70 / 50, of 8192 of length 1024 1148 / 1180 / 1192.
template <int MODE>
void launch_tiles(const Ws& ws, int rows, int k, cudaStream_t s) {
  int best = 16;
  double least = 0.0;
  for (int tn = 16; tn >= 8; tn -= 4) {
    const int cols = (ws.N + TX * tn - 1) / (TX * tn), rts = (rows + BM - 1) / BM;
    long long tiles = static_cast<long long>(cols) * rts;
    if (MODE == kGram) {  // the tiles that simt_tile_kernel does not skip
      tiles = 0;
      for (int by = 0; by < rts; ++by) tiles += cols - (by * BM) / (TX * tn);
    }
    const double rounds = tiles <= ws.sms ? 1.25 : static_cast<double>((tiles + ws.sms - 1) / ws.sms);
    if (least == 0.0 || rounds * tn < least) {
      least = rounds * tn;
      best = tn;
    }
  }
  if (best == 16)
    launch_one<MODE, 16>(ws, rows, k, s);
  else if (best == 12)
    launch_one<MODE, 12>(ws, rows, k, s);
  else
    launch_one<MODE, 8>(ws, rows, k, s);
}

template <int MODE>
cudaError_t set_tile_limits() {
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(simt_tile_kernel<MODE, 16>), tile_bytes<16>());
  if (e == cudaSuccess)
    e = raise_smem_limit(reinterpret_cast<const void*>(simt_tile_kernel<MODE, 12>), tile_bytes<12>());
  if (e == cudaSuccess)
    e = raise_smem_limit(reinterpret_cast<const void*>(simt_tile_kernel<MODE, 8>), tile_bytes<8>());
  return e;
}
}  // namespace

cudaError_t configure_corr_simt(const Ws& ws) {
  cudaError_t e = set_tile_limits<kGram>();
  if (e == cudaSuccess && ws.prec == OMP_PREC_FP32) e = set_tile_limits<kCorrelate>();
  if (e == cudaSuccess && ws.filt)
    e = raise_smem_limit(reinterpret_cast<const void*>(simt_tile_kernel<kOverflow, 8>), 2 * tile_bytes<8>());
  return e;
}
cudaError_t configure_c0_simt() { return set_tile_limits<kStoreC>(); }

void launch_corr_simt(const Ws& ws, int k, int B, cudaStream_t s) { launch_tiles<kCorrelate>(ws, B, k, s); }

// Mostly no position is left over, and the blocks return at once (1.7 us). Where a few are, each block
// has one tile of its own SM; where many are (near copies, long rows at the noise floor), two, side by
// side, which hide each other's latency as two blocks do. (A grid of two blocks an SM puts some first
// tiles on one SM: 1000 signals x 8192 atoms x 1024, a step 52.2 us for 50.2.) Every position, us a step
// here / one row of blocks / without the filter: 40 near copies of each atom, 256 x 1024, 5000 signals
// 113 / 804 / 80; 1024 x 8192, 1000 signals 368 / 552 / 322; noise floor, 8064 x 1207, 1200 signals
// 723 / 4352 / 723.
void launch_corr_overflow(const Ws& ws, int k, int B, cudaStream_t s) {
  const long long tiles = static_cast<long long>((ws.N + 8 * TX - 1) / (8 * TX)) * ((B + BM - 1) / BM);
  simt_tile_kernel<kOverflow, 8><<<tiles < ws.sms ? static_cast<int>(tiles) : ws.sms, 2 * THREADS, 2 * tile_bytes<8>(), s>>>(ws, k);
}

void launch_c0_simt(const Ws& ws, int B, cudaStream_t s) { launch_tiles<kStoreC>(ws, B, B, s); }

void launch_gram_simt(const Ws& ws, cudaStream_t s) { launch_tiles<kGram>(ws, ws.N, 0, s); }

}  // namespace ompk
