// Solves of few signals: the same iteration (Sec. 2.3, as in append.cuh) arranged for latency.
//
// A batch that does not fill the tensor-core tiles leaves the batched kernels waiting: one signal
// over 8192 atoms of length 1024 took 39 us a step (the correlation 23 on 10 CTAs, one warp's
// append and update 13, the compaction and three launches the rest), 16 signals over 64 x 256
// 16 to 20 us. Here nothing is compacted and a signal has a block of eight warps:
//   solo   a small dictionary: one block per signal runs every step in one launch, the residual,
//          the scores and the factor in shared memory
//   wide   a large dictionary and up to 8 signals: per step one launch scores every atom with the
//          whole GPU (bound by reading the FP32 atom rows from L2), one does the rest with a block
//          per signal
// One signal over 1024 x 8192 then takes 13 us a step, 16 signals over 64 x 256 7 us: a chain of
// short dependent phases, of which the append's FP64 part is 1900 cycles.
// Scores here are FP32 dot products in an order of their own. An atom can only be the pick if its
// score is within two error bounds of the best, so those atoms -- mostly one -- are scored again
// as the batched path of the handle does it (FP32: one chain of FMAs over m; BF16: the rescoring's
// order), and b and ||r|| are summed in the batched update's order: the same picks and bits as the
// batched kernels, but for BF16 signals with more than eight atoms in the window (near copies). The
// batched path rescores the eight best by BF16 score; here all of them are, so the pick is FP32's.
#include <type_traits>

#include "append.cuh"

namespace ompk {
namespace {

// One float4 slot's part of a dot product, rounded as the batched kernels (append.cuh) round it
__device__ __forceinline__ float dot4(const float4& a, const float4& b, int V0) {
  return V0 == 1 ? slot_dot<true>(a, b) : slot_dot<false>(a, b);
}
constexpr int kT = 256, kWarps = kT / 32;
constexpr int kList = 32;                          // atoms of a pick's window that are listed
constexpr int kGS = 4;                             // wide: scores per recorded maximum
constexpr int kSmallMaxB = 8;                      // wide: signals that share one pass over A
constexpr int64_t kWideMaxElems = 24ll << 20;      // wide: FP32 rows of at most 96 MB stay in L2
constexpr int64_t kWideMaxRows = 48 * 1024;         // wide: residuals in shared memory (192 KB)
constexpr int64_t kWideMaxWork = 144ll << 20;       // wide: products of a step; past it the tile kernel, for
constexpr int64_t kWideMaxWork16 = 96ll << 20;      //   BF16 handles the tensor cores, score faster
constexpr int64_t kSoloMaxElems = 1ll << 18;       // solo: at most 1 MB of atom rows a step and block
constexpr int64_t kSoloMaxTotal = 24ll << 20;      // solo: at most 96 MB a step over all signals
constexpr size_t kSmallMaxSmem = 100 * 1024;       // solo: two blocks an SM at least
constexpr size_t kWideMaxSmem = 216 * 1024;

// floats per signal of ws.score: N scores, then the largest of each kGS of them
__host__ __device__ __forceinline__ size_t score_pitch(int N) { return static_cast<size_t>(N) + (N + kGS - 1) / kGS; }


struct SmallSmem {
  float* r;      // Mp: the residual
  float* P;      // Mp / 4 (rounded up to 32 lanes): per-slot partials of the ordered sums
  float* part;   // 8: per-warp sums; [8]: the result
  float* rs;     // 8 best scores and
  int* ri;       // 8 their atoms
  int* ctl;      // 4: candidates in the window, the pick
  float* sc;     // N (solo): the scores
  float* rows;   // RC x Mp: the support's first RC atom rows, or (solo) the whole dictionary
  GroupSmem gs;  // the append's fields: tri, w, z, f, sup, scal
};

__host__ __device__ __forceinline__ int slots4(int Mp) { return (Mp / 4 + 31) / 32 * 32; }

__host__ __device__ __forceinline__ size_t small_bytes(int Mp, int Smax, int nsc, int RC) {
  const size_t words = static_cast<size_t>(Mp) * (1 + RC) + slots4(Mp) + (tri_floats(Smax) + 3) / 4 * 4 +
                       (nsc + 3) / 4 * 4 + 16 + 8 + 8 + 4 + 4 + 4 * (static_cast<size_t>(Smax) + 4);
  return (words * 4 + 15) / 16 * 16;
}

__device__ __forceinline__ SmallSmem small_smem(unsigned char* base, int Mp, int Smax, int nsc, int RC) {
  SmallSmem s;
  s.r = reinterpret_cast<float*>(base);
  s.rows = s.r + Mp;
  s.P = s.rows + static_cast<size_t>(Mp) * RC;
  s.gs.tri = s.P + slots4(Mp);
  s.sc = s.gs.tri + (tri_floats(Smax) + 3) / 4 * 4;
  s.part = s.sc + (nsc + 3) / 4 * 4;
  s.rs = s.part + 16;
  s.ri = reinterpret_cast<int*>(s.rs + 8);
  s.ctl = s.ri + 8;
  s.gs.scal = s.ctl + 4;
  s.gs.w = reinterpret_cast<float*>(s.gs.scal + 4);
  s.gs.z = s.gs.w + Smax + 4;
  s.gs.f = s.gs.z + Smax + 4;
  s.gs.sup = reinterpret_cast<int*>(s.gs.f + Smax + 4);
  return s;
}

// rows of the support kept in shared memory: as many as `budget` bytes leave room for
int row_cache(int Mp, int Smax, int nsc, size_t budget) {
  const size_t base = small_bytes(Mp, Smax, nsc, 0);
  const size_t room = base < budget ? (budget - base) / (static_cast<size_t>(Mp) * 4) : 0;
  return room < static_cast<size_t>(Smax) ? static_cast<int>(room) : Smax;
}

// |<a, r>| / ||a|| as the batched BF16 rescoring forms it: the dot products of W0 warps' float4
// slots, each lane's slots in order, a butterfly per warp, the warps' sums in order. One warp.
__device__ __forceinline__ float rescore_dot(const float4* a, const float4* r, int M4, int W0, int V0, int lane) {
  float v = 0.f;
  for (int w = 0; w < W0; ++w) {
    float acc = 0.f;
#pragma unroll 8
    for (int t = 0; t < V0; ++t) {
      const int s = (t * W0 + w) * 32 + lane;
      if (s < M4) {
        const float4 x = __ldg(a + s);
        const float4 y = r[s];
        acc += dot4(x, y, V0);
      }
    }
    v += warp_sum_f(acc);
  }
  return v;
}

// <a, r> as the batched FP32 correlation forms it: one chain of FMAs over m = 0, 1, ... One thread.
__device__ __forceinline__ float chain_dot(const float4* a, const float4* r, int M4) {
  float acc = 0.f;
  for (int s0 = 0; s0 < M4; s0 += 16) {  // M4 is a multiple of 16
    float4 x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = __ldg(a + s0 + i);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float4 y = r[s0 + i];
      acc = fmaf(y.x, x[i].x, acc);
      acc = fmaf(y.y, x[i].y, acc);
      acc = fmaf(y.z, x[i].z, acc);
      acc = fmaf(y.w, x[i].w, acc);
    }
  }
  return acc;
}

// The ordered sum of the block's per-slot partials sm.P (see rescore_dot); every thread gets it.
// `part`: one of the two halves of sm.part (alternate them: no barrier follows the last read).
__device__ __forceinline__ float ordered_sum(const SmallSmem& sm, float* part, int M4, int W0, int V0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (warp < W0) {
    float acc = 0.f, p[8];  // V0 <= 8
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int s = (t * W0 + warp) * 32 + lane;
      p[t] = t < V0 && s < M4 ? sm.P[s] : 0.f;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (t < V0) acc += p[t];
    acc = warp_sum_f(acc);
    if (lane == 0) part[warp] = acc;
  }
  __syncthreads();
  float v = 0.f;
#pragma unroll
  for (int w = 0; w < kWarps; ++w)
    if (w < W0) v += part[w];
  return v;
}

// An atom whose norm is so far from 1 that FP32 products with it may overflow or lose bits below
// the normal range is always scored again: its score is a NaN, which passes the window's test.
// (A zero atom scores 0 everywhere.)
__device__ __forceinline__ float approx_score(float dot, float inv) {
  return inv == 0.f || (inv > 1e-15f && inv < 1e15f) ? fabsf(dot) * inv : __int_as_float(0x7fffffff);
}

// the larger of two scores, a NaN if either is one
__device__ __forceinline__ float max_keep_nan(float a, float b) { return a != a || a > b ? a : b; }

__device__ __forceinline__ void load_head(float (&head)[8], const float* gm, int NG) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int g = threadIdx.x + i * kT;
    head[i] = g < NG ? gm[g] : -2.f;
  }
}

// The pick of the signal whose residual is sm.r, from the scores sc[0..N) and, per GS of them, their
// largest gm[0..N/GS) (gm = sc for GS 1; a NaN where a group holds one): the block agrees on it
// (-1: no atom has a score).
// head: this thread's first 8 maxima (gm[tid + 256 i], -2 past the end), loaded ahead.
template <int GS>
__device__ __forceinline__ int pick_atom(const Ws& ws, const SmallSmem& sm, const float* sc, const float* gm,
                                         const float (&head)[8], float rnorm, int W0, int V0) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = ws.N, M4 = ws.Mp >> 2, NG = (N + GS - 1) / GS;
  float bs = -1.f;
  for (int g0 = tid; g0 < NG; g0 += 8 * kT) {
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = g0 == tid ? head[i] : g0 + i * kT < NG ? gm[g0 + i * kT] : -2.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      bs = fmaxf(bs, v[i]);  // a NaN is passed over
      if (GS > 1 && v[i] != v[i])
        for (int n = (g0 + i * kT) * GS; n < min(N, (g0 + i * kT) * GS + GS); ++n) bs = fmaxf(bs, sc[n]);
    }
  }
  bs = warp_max(bs);
  if (lane == 0) sm.rs[warp] = bs;
  if (tid == 0) sm.ctl[0] = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w) bs = fmaxf(bs, sm.rs[w]);
  // both orders of summation are within gam_32 ||a|| ||r|| of the exact product; the products with
  // 1/||a|| add two roundings each, 1% covers the rounding of the norms and of this bound
  const float eps = 1.01f * (2.f * ws.gam_32 + 4.f * 0x1p-24f);
  const bool ranged = rnorm > 1e-15f && rnorm < 1e15f;
  const float thr = ranged ? bs - 2.f * eps * rnorm : -2.f;
  int* list = reinterpret_cast<int*>(sm.P);  // the first kList atoms of the window
  auto window = [&](int g, float m) {
    if (!(m < thr))
      for (int n = g * GS; n < min(N, g * GS + GS); ++n)
        if (GS == 1 || !(sc[n] < thr)) {
          const int c = atomicAdd(sm.ctl, 1);
          if (c < kList) list[c] = n;
        }
  };
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (tid + i * kT < NG) window(tid + i * kT, head[i]);
  for (int g = tid + 8 * kT; g < NG; g += kT) window(g, gm[g]);
  __syncthreads();
  const int cnt = sm.ctl[0];
  if (cnt == 1) {  // alone in the window: the best, or an atom that has no score
    const int n = list[0];
    return sc[n] >= 0.f ? n : -1;
  }
  // score the window's atoms as the batched path does
  const float4* r4 = reinterpret_cast<const float4*>(sm.r);
  float cs = -1.f;
  int ci = 0x7fffffff;
  const float4* A4 = reinterpret_cast<const float4*>(ws.A32);
  auto take = [&](int n, float dot) {
    const float s = fabsf(dot) * __ldg(ws.inv_norm + n);
    if (better(s, n, cs, ci) && s >= 0.f) {  // false for a NaN
      cs = s;
      ci = n;
    }
  };
  const bool listed = cnt <= kList;  // else the whole row of scores is walked again
  const int end = listed ? cnt : N;
  if (ws.prec == OMP_PREC_FP32) {
    for (int i = tid; i < end; i += kT) {
      const int n = listed ? list[i] : i;
      if (listed || !(sc[n] < thr)) take(n, chain_dot(A4 + static_cast<size_t>(n) * M4, r4, M4));
    }
  } else {
    for (int i = warp; i < end; i += kWarps) {
      const int n = listed ? list[i] : i;
      if (listed || !(sc[n] < thr)) take(n, rescore_dot(A4 + static_cast<size_t>(n) * M4, r4, M4, W0, V0, lane));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float os = __shfl_xor_sync(0xffffffffu, cs, o);
    const int oi = __shfl_xor_sync(0xffffffffu, ci, o);
    if (better(os, oi, cs, ci)) {
      cs = os;
      ci = oi;
    }
  }
  if (lane == 0) {
    sm.rs[warp] = cs;
    sm.ri[warp] = ci;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w)
    if (better(sm.rs[w], sm.ri[w], cs, ci)) {
      cs = sm.rs[w];
      ci = sm.ri[w];
    }
  return ci < N ? ci : -1;
}

// One step (append, residual update, stop test) of signal b with kk atoms, the residual in sm.r and
// the support in sm.gs.sup. V: float4 slots per thread. Returns whether the signal goes on; *rn
// becomes its ||r||. The FP32 factor is in sm.gs.tri (Smax <= kTriMax) or in ws.F32. The first
// nrow rows of the support are in sm.rows (copies in flight included); a row past them goes there
// too if keep allows, for the next step. DICT: sm.rows is the whole dictionary.
template <int V, int GS, bool DICT>
__device__ __forceinline__ bool small_step(const Ws& ws, const SmallSmem& sm, const float* sc, const float* gm, const float (&head)[8], int nrow, int b, int kk, int S,
                                           float eps, int eps_rel, float ynorm, int W0, int V0, int keep, float* rn) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int M4 = ws.Mp >> 2;
  const GroupSmem& gs = sm.gs;
  const float rprev = *rn;
  const int ns = pick_atom<GS>(ws, sm, sc, gm, head, rprev, W0, V0);
  if (ns < 0) {
    if (tid == 0) {
      atomicOr(ws.err, OMP_DEVERR_BAD_STATE);
      ws.flag[b] = 0;
    }
    return false;
  }
  // the new atom's row arrives while the first warp appends
  float4 vn[V];
#pragma unroll
  for (int t = 0; t < V; ++t) {
    const int s = t * kT + tid;
    vn[t] = s < M4 ? __ldg(reinterpret_cast<const float4*>(ws.A32 + static_cast<size_t>(ns) * ws.Mp) + s)
                   : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (warp == 0) {
    const float* grow = ws.gram + static_cast<size_t>(ns) * ws.ldg;
    const double nrm2 = __ldg(ws.norm2 + ns);
    for (int i = lane; i < kk; i += 32) gs.w[i] = __ldg(grow + gs.sup[i]);
    __syncwarp();
    double* Fg = ws.F + static_cast<size_t>(b) * ws.Fstride;
    float* Ff = ws.F32 + static_cast<size_t>(b) * ws.Fstride;
    const int nb = (kk + 31) >> 5;
    float* tri = gs.tri;
    if (ws.Smax <= kTriMax) {
      if (nb <= 1) append_column<1, 4>(ws, gs, tri, tri, Fg, kk, ns, nrm2, lane);
      else append_column<2, 4>(ws, gs, tri, tri, Fg, kk, ns, nrm2, lane);
    } else {
      if (nb <= 1) append_column<1, 4>(ws, gs, Ff, Ff, Fg, kk, ns, nrm2, lane);
      else if (nb <= 2) append_column<2, 4>(ws, gs, Ff, Ff, Fg, kk, ns, nrm2, lane);
      else if (nb <= 4) append_column<4, 2>(ws, gs, Ff, Ff, Fg, kk, ns, nrm2, lane);
      else append_column<8>(ws, gs, Ff, Ff, Fg, kk, ns, nrm2, lane);
    }
  }
  cp_async_wait_all();  // the rows this thread copied
  __syncthreads();
  if (gs.scal[1]) {
    if (tid == 0) {
      ws.flag[b] = 0;
      ws.stop[b] = kStopDependent;
    }
    return false;
  }
  // q = A_S f: thread's slots tid + 256 t, the rows in order -- from shared memory, the rest (a
  // support longer than sm.rows) R rows in flight, the new one last
  float4 q[V];
#pragma unroll
  for (int t = 0; t < V; ++t) q[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add_row = [&](float f, int t, const float4& v) {
    q[t].x = fmaf(f, v.x, q[t].x);
    q[t].y = fmaf(f, v.y, q[t].y);
    q[t].z = fmaf(f, v.z, q[t].z);
    q[t].w = fmaf(f, v.w, q[t].w);
  };
#pragma unroll(V == 1 ? 4 : 1)
  for (int a = 0; a < (DICT ? kk : nrow); ++a) {
    const float f = gs.f[a];
    const float4* row = reinterpret_cast<const float4*>(sm.rows) + (DICT ? gs.sup[a] : a) * M4;
#pragma unroll
    for (int t = 0; t < V; ++t) {
      const int s = t * kT + tid;
      add_row(f, t, s < M4 ? row[s] : make_float4(0.f, 0.f, 0.f, 0.f));
    }
  }
  constexpr int R = V <= 2 ? 8 : V <= 4 ? 4 : 2;
  for (int a0 = DICT ? kk : nrow; a0 < kk; a0 += R) {
    float4 v[R][V];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int a = a0 + i;
      const float4* row = reinterpret_cast<const float4*>(ws.A32 + static_cast<size_t>(gs.sup[min(a, kk - 1)]) * ws.Mp);
#pragma unroll
      for (int t = 0; t < V; ++t) {
        const int s = t * kT + tid;
        v[i][t] = a < kk && s < M4 ? __ldg(row + s) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (a0 + i < kk) {
        const float f = gs.f[a0 + i];
#pragma unroll
        for (int t = 0; t < V; ++t) add_row(f, t, v[i][t]);
      }
    }
  }
  {
    const float f = gs.f[kk];
#pragma unroll
    for (int t = 0; t < V; ++t) {
      const int s = t * kT + tid;
      add_row(f, t, vn[t]);
      if (!DICT && kk < keep && s < M4) reinterpret_cast<float4*>(sm.rows + static_cast<size_t>(kk) * ws.Mp)[s] = vn[t];
    }
  }
  float4* r4 = reinterpret_cast<float4*>(sm.r);
  float4 r[V];
#pragma unroll
  for (int t = 0; t < V; ++t) {
    const int s = t * kT + tid;
    r[t] = s < M4 ? r4[s] : make_float4(0.f, 0.f, 0.f, 0.f);
    if (s < M4) sm.P[s] = dot4(q[t], r[t], V0);
  }
  const float bf = ordered_sum(sm, sm.part, M4, W0, V0);
#pragma unroll
  for (int t = 0; t < V; ++t) {
    const int s = t * kT + tid;
    r[t].x = fmaf(-bf, q[t].x, r[t].x);
    r[t].y = fmaf(-bf, q[t].y, r[t].y);
    r[t].z = fmaf(-bf, q[t].z, r[t].z);
    r[t].w = fmaf(-bf, q[t].w, r[t].w);
    if (s < M4) {
      r4[s] = r[t];
      sm.P[s] = slot_dot<false>(r[t], r[t]);
    }
  }
  const float rk = sqrtf(ordered_sum(sm, sm.part + 8, M4, W0, V0));
  *rn = rk;
  const float thr = eps_rel ? eps * ynorm : eps;
  const bool hit = rk <= thr, last = kk + 1 >= S;
  if (tid == 0) {
    const size_t o = static_cast<size_t>(b) * ws.Smax + kk;
    ws.bv[o] = static_cast<double>(bf);
    ws.sup[o] = ns;
    ws.drop[o] = rprev > 0.f ? (bf / rprev) * (bf / rprev) : 0.f;
    ws.niter[b] = kk + 1;
    ws.rnorm[b] = rk;
    if (hit || last) {
      ws.flag[b] = 0;
      ws.stop[b] = hit ? kStopEps : kStopIters;
    }
  }
  return !(hit || last);
}

// Scores of every atom for one residual in shared memory, LPA lanes per atom (16 when a row has 64
// elements), U atoms in flight per lane group; warp `first` of `stride` takes every stride-th group.
// With gm, the largest score of each U consecutive atoms too (LPA 32; a NaN if one is).
template <int LPA, int U, bool SH>
__device__ __forceinline__ void score_atoms(const Ws& ws, const float4* rows, const float4* r4, int first, int stride,
                                            float* sc, float* gm = nullptr) {
  const int lane = threadIdx.x & 31, sub = lane % LPA, grp = lane / LPA;
  constexpr int GP = 32 / LPA;  // atoms a warp takes side by side
  const int M4 = ws.Mp >> 2, N = ws.N;
  for (int n0 = first * GP * U; n0 < N; n0 += stride * GP * U) {
    float acc[U], inv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      acc[u] = 0.f;
      const int n = n0 + u * GP + grp;
      inv[u] = n < N ? __ldg(ws.inv_norm + n) : 0.f;
    }
#pragma unroll 4
    for (int s = sub; s < M4; s += LPA) {
      const float4 y = r4[s];
      float4 x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int n = min(n0 + u * GP + grp, N - 1);
        x[u] = SH ? rows[n * M4 + s] : __ldg(rows + static_cast<size_t>(n) * M4 + s);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        acc[u] = fmaf(x[u].w, y.w, fmaf(x[u].z, y.z, fmaf(x[u].y, y.y, fmaf(x[u].x, y.x, acc[u]))));
    }
    float best = -1.f;
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int o = LPA / 2; o > 0; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
      const int n = n0 + u * GP + grp;
      const float v = approx_score(acc[u], inv[u]);
      if (n < N) best = max_keep_nan(best, v);
      if (sub == 0 && n < N) sc[n] = v;
    }
    if (gm && lane == 0) gm[n0 / U] = best;
  }
}

// Every step of one signal per block.
// DICT: the dictionary fits in shared memory beside the rest; every step then reads it there.
template <int V, bool DICT>
__global__ void __launch_bounds__(kT, 2) solo_kernel(Ws ws, int S, float eps, int eps_rel, int W0, int V0, int RC) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int b = blockIdx.x, M4 = ws.Mp >> 2;
  if (!ws.flag[b]) return;  // y == 0 or non-finite
  SmallSmem sm = small_smem(smem, ws.Mp, ws.Smax, ws.N, RC);
  const float4* A4 = reinterpret_cast<const float4*>(ws.A32);
  float4* rows4 = reinterpret_cast<float4*>(sm.rows);
  const float4* r4 = reinterpret_cast<const float4*>(sm.r);
  if (DICT)
    for (int i = tid; i < ws.N * M4; i += kT) cp_async16(rows4 + i, A4 + i);
  const float4* rg = reinterpret_cast<const float4*>(ws.R32 + static_cast<size_t>(b) * ws.Mp);
  for (int s = tid; s < M4; s += kT) reinterpret_cast<float4*>(sm.r)[s] = rg[s];
  const float ynorm = ws.ynorm[b];
  float rn = ws.rnorm[b];
  bool go = true;
  cp_async_wait_all();
  for (int kk = 0; go; ++kk) {
    __syncthreads();  // the residual is complete, and every read of the last step's scores is done
    if (ws.Mp == 64)
      score_atoms<16, DICT ? 4 : 8, DICT>(ws, DICT ? rows4 : A4, r4, warp, kWarps, sm.sc);
    else
      score_atoms<32, 4, DICT>(ws, DICT ? rows4 : A4, r4, warp, kWarps, sm.sc);
    __syncthreads();
    float head[8];
    load_head(head, sm.sc, ws.N);
    go = small_step<V, 1, DICT>(ws, sm, sm.sc, sm.sc, head, min(kk, RC), b, kk, S, eps, eps_rel, ynorm, W0, V0, RC,
                                &rn);
  }
}

// Scores of every atom for the (up to kSmallMaxB) signals still going, written to ws.score (B x N).
// A warp takes atoms 8 apart over the grid; a row is read once for all signals.
__global__ void __launch_bounds__(kT) wide_score_kernel(Ws ws, int B) {
  extern __shared__ __align__(16) unsigned char smem[];
  float4* rs = reinterpret_cast<float4*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int M4 = ws.Mp >> 2, N = ws.N;
  const size_t NP = score_pitch(N);
  __shared__ int act[kSmallMaxB], na_s;  // the signals that go on
  if (tid == 0) {
    int n = 0;
    for (int b = 0; b < B; ++b)
      if (ws.flag[b]) act[n++] = b;
    na_s = n;
  }
  __syncthreads();
  const int na = na_s;
  if (na == 0) return;
  for (int i = 0; i < na; ++i)
    for (int s = tid; s < M4; s += kT)
      rs[static_cast<size_t>(i) * M4 + s] =
          reinterpret_cast<const float4*>(ws.R32 + static_cast<size_t>(act[i]) * ws.Mp)[s];
  __syncthreads();
  if (na == 1) {
    const int first = blockIdx.x * kWarps + warp, stride = gridDim.x * kWarps;
    score_atoms<32, kGS, false>(ws, reinterpret_cast<const float4*>(ws.A32), rs, first, stride, ws.score + static_cast<size_t>(act[0]) * NP, ws.score + static_cast<size_t>(act[0]) * NP + N);
    return;
  }
  constexpr int U = kGS;
  for (int n0 = (blockIdx.x * kWarps + warp) * U; n0 < N; n0 += gridDim.x * kWarps * U) {
    float acc[U][kSmallMaxB];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int i = 0; i < kSmallMaxB; ++i) acc[u][i] = 0.f;
    for (int s = lane; s < M4; s += 32) {
      float4 x[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        x[u] = n0 + u < N ? __ldg(reinterpret_cast<const float4*>(ws.A32 + static_cast<size_t>(n0 + u) * ws.Mp) + s)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < kSmallMaxB; ++i) {
        if (i < na) {
          const float4 y = rs[static_cast<size_t>(i) * M4 + s];
#pragma unroll
          for (int u = 0; u < U; ++u)
            acc[u][i] = fmaf(x[u].w, y.w, fmaf(x[u].z, y.z, fmaf(x[u].y, y.y, fmaf(x[u].x, y.x, acc[u][i]))));
        }
      }
    }
    float inv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) inv[u] = n0 + u < N ? __ldg(ws.inv_norm + n0 + u) : 0.f;
#pragma unroll
    for (int i = 0; i < kSmallMaxB; ++i) {
      if (i < na) {
        float* sc = ws.score + static_cast<size_t>(act[i]) * NP;
        float best = -1.f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float v = approx_score(warp_sum_f(acc[u][i]), inv[u]);
          if (n0 + u < N) best = max_keep_nan(best, v);
          if (lane == 0 && n0 + u < N) sc[n0 + u] = v;
        }
        if (lane == 0) sc[N + n0 / U] = best;
      }
    }
  }
}

// One step of each signal from the scores in ws.score
template <int V>
__global__ void __launch_bounds__(kT, 1) wide_step_kernel(Ws ws, int S, float eps, int eps_rel, int W0, int V0,
                                                          int RC) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x;
  const int b = blockIdx.x;
  const int flag = ws.flag[b], kk = ws.niter[b];
  float rn = ws.rnorm[b];
  const float ynorm = ws.ynorm[b];
  if (!flag) return;
  // the scores' maxima first: what follows queues behind them
  const float* sc = ws.score + static_cast<size_t>(b) * score_pitch(ws.N);
  float head[8];
  load_head(head, sc + ws.N, (ws.N + kGS - 1) / kGS);
  SmallSmem sm = small_smem(smem, ws.Mp, ws.Smax, 0, RC);
  const int M4 = ws.Mp >> 2;
  float4* rg = reinterpret_cast<float4*>(ws.R32 + static_cast<size_t>(b) * ws.Mp);
  for (int s = tid; s < M4; s += kT) cp_async16(reinterpret_cast<float4*>(sm.r) + s, rg + s);
  float* Ff = ws.F32 + static_cast<size_t>(b) * ws.Fstride;
  const bool staged = ws.Smax <= kTriMax;
  if (staged)
    for (int i = tid; i < (kk * (kk + 1) / 2 + 3) / 4; i += kT) cp_async16(sm.gs.tri + 4 * i, Ff + 4 * i);
  const int* sup = ws.sup + static_cast<size_t>(b) * ws.Smax;
  for (int i = tid; i < kk; i += kT) cp_async4(sm.gs.sup + i, sup + i);
  cp_async_commit();
  // the support's rows land while the block picks and appends
  const int nrow = min(kk, RC);
#pragma unroll 8
  for (int a = 0; a < nrow; ++a) {
    const float4* row = reinterpret_cast<const float4*>(ws.A32 + static_cast<size_t>(sup[a]) * ws.Mp);
#pragma unroll
    for (int t = 0; t < V; ++t) {
      const int s = t * kT + tid;
      if (s < M4) cp_async16(reinterpret_cast<float4*>(sm.rows + static_cast<size_t>(a) * ws.Mp) + s, row + s);
    }
  }
  cp_async_commit();
  cp_async_wait_one();  // all but the rows; pick_atom's barriers publish them
  const bool go = small_step<V, kGS, false>(ws, sm, sc, sc + ws.N, head, nrow, b, kk, S, eps, eps_rel, ynorm, W0, V0, 0,
                                     &rn);
  cp_async_wait_all();
  if (!go) return;
  for (int s = tid; s < M4; s += kT) rg[s] = reinterpret_cast<float4*>(sm.r)[s];
  if (staged)  // the new factor column
    for (int i = tid; i <= kk; i += kT) Ff[kk * (kk + 1) / 2 + i] = sm.gs.tri[kk * (kk + 1) / 2 + i];
}

int slots_per_thread(int Mp) {
  const int need = (Mp / 4 + kT - 1) / kT;
  int V = 1;
  while (V < need) V <<= 1;
  return V;
}

template <class F>
void by_slots(int V, F f) {
  if (V == 1) f(std::integral_constant<int, 1>{});
  else if (V == 2) f(std::integral_constant<int, 2>{});
  else if (V == 4) f(std::integral_constant<int, 4>{});
  else f(std::integral_constant<int, 8>{});
}

}  // namespace

// Which arrangement a solve takes: 0 batched, 1 solo, 2 wide. The quantised 8-bit path, fewer than
// 8 rescored candidates, recorded margins, the 24-bit gather and the hook that turns the score
// bound off stay batched: their picks depend on what the batched path keeps of its lists.
int small_form(const Ws& ws, int B, float eps) {
  if (ws.prec == OMP_PREC_FP8_E4M3 || ws.A24h || ws.margin) return 0;
  if (ws.prec == OMP_PREC_BF16 && (ws.topk != kMaxTopk || !(ws.rescore_eps > 0.f))) return 0;
  const bool fp32 = ws.prec == OMP_PREC_FP32;
  const int64_t elems = static_cast<int64_t>(ws.N) * ws.Mp;
  if (elems <= kSoloMaxElems && elems * B <= kSoloMaxTotal && small_bytes(ws.Mp, ws.Smax, ws.N, 0) <= kSmallMaxSmem) {
    // Two blocks fit on an SM, so a step takes rounds of 4 us and a time an atom: 20 ns and 20 for four
    // passes of a warp over its row (15 where a block has an SM to itself), 8 for each pass left over,
    // 9.5 in all for rows of 64. Against it stands the batched step. Measured, us a step solo / batched
    // FP32 / batched BF16: 64 x 128 300 signals 9.7 / 21 / 23, 900 19.4 / 22.0 / 24.0, 1200 24.4 / 22.6 / 23.6;
    // 64 x 256 600 signals 15.1 / 20.0 / 21.8, 900 21.2 / 20.5 / 22.4, 1500 34 / 21 / 23; 64 x 1024 300 17.1 /
    // 20.7 / 22.3, 310 29.8 / 20.8 / 22.6; 64 x 4096 16 41 / 19 / 21; 128 x 512 300 19.4 / 23.3 / 21.0, 310
    // 35 / 24 / 21; 128 x 2048 16 52 / 21 / 20; 256 x 512 100 21.9 / 26 / 21; 256 x 1024 16 36 / 24 / 19;
    // 400 x 512 10 30.6 / 26 / 21; 512 x 512 10 20.8 / 26 / 21; 1024 x 256 64 17.5 / 34 / 28.
    const int rounds = (B + 2 * ws.sms - 1) / (2 * ws.sms), M4 = ws.Mp / 4;
    const int left = (M4 % 128 + 31) / 32;
    const double atom = ws.Mp == 64 ? 9.5e-3 : 1e-3 * (20 + M4 / 128 * (B <= ws.sms ? 15 : 20) + 8 * left);
    const double batched = !fp32 ? 19.0 + ws.Mp / 170.0 : ws.Mp == 64 ? 19.5 : 22.0 + ws.Mp / 100.0;
    // (With a threshold a block ends with its signal, where every other form launches what is left of
    // the S steps: one signal over 256 x 512, BF16, 128 steps of which it takes some 16, 318 us a solve
    // for 412 by the wide form and 721 batched.)
    if (rounds * (4.0 + ws.N * atom) <= (eps > 0.f ? 1.3 : 1.0) * batched) return 1;
  }
  // Wide scores every atom for each signal on the CUDA cores and keeps the residuals in shared memory.
  // Measured, us a step wide / batched FP32 / batched BF16: 1024 x 8192 1 signal 13.6 / 32 / 28, 8 24.4 /
  // 36 / 28.5; 2048 x 8192 6 28.8 / 41 / 33, 8 33.6 / 44 / 32.8; 4096 x 3000 6 37 / 53 / 38, 8 44 / 58 / 39;
  // 4096 x 6000 3 34 to 43 / 53 / 40, 4 43 / 54 / 40, 6 51 / 57 / 41, 8 87 / 72 / 42; 700 x 30000 4 38 / 45 / 41,
  // 6 47 / 45 / 41, 8 55 / 45 / 41; 8192 x 600 3 43 / 81 / 57, 6 57 / 75 / 57; 8192 x 3000 1 50 to 59 / 70 / 56,
  // 2 67 / 73 / 57, 6 92 / 87 / 58.
  const int64_t work = fp32 ? kWideMaxWork : ws.Mp <= 4096 ? kWideMaxWork16 : kWideMaxWork16 / 4;
  if (B <= kSmallMaxB && elems <= kWideMaxElems && elems * B <= work &&
      static_cast<int64_t>(ws.Mp) * B <= (fp32 ? kWideMaxRows : kWideMaxRows / 2))
    return 2;
  return 0;
}

cudaError_t configure_small(const Ws& ws) {
  cudaError_t e = cudaSuccess;
  by_slots(slots_per_thread(ws.Mp), [&](auto v) {
    constexpr int V = decltype(v)::value;
    e = raise_smem_limit(reinterpret_cast<const void*>(solo_kernel<V, false>), kSmallMaxSmem);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void*>(solo_kernel<V, true>), kSmallMaxSmem);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void*>(wide_step_kernel<V>), kWideMaxSmem);
  });
  if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void*>(wide_score_kernel), kWideMaxRows * 4);
  return e;
}

size_t small_score_floats(int N, int Bmax) { return score_pitch(N) * (Bmax < kSmallMaxB ? Bmax : kSmallMaxB); }

void launch_solo(const Ws& ws, int B, int S, float eps, int eps_rel, cudaStream_t s) {
  const bool dict = small_bytes(ws.Mp, ws.Smax, ws.N, ws.N) <= kSmallMaxSmem;
  const int rc = dict ? ws.N : row_cache(ws.Mp, ws.Smax, ws.N, kSmallMaxSmem);
  const size_t bytes = small_bytes(ws.Mp, ws.Smax, ws.N, rc);
  by_slots(slots_per_thread(ws.Mp), [&](auto v) {
    constexpr int V = decltype(v)::value;
    (dict ? solo_kernel<V, true> : solo_kernel<V, false>)<<<B, kT, bytes, s>>>(ws, S, eps, eps_rel, ws.upd_w,
                                                                             update_slots(ws.Mp, ws.upd_w), rc);
  });
}

void launch_wide(const Ws& ws, int sms, int B, int S, float eps, int eps_rel, cudaStream_t s) {
  const int per = kWarps * kGS;
  const int blocks = (ws.N + per - 1) / per, grid = blocks < 2 * sms ? blocks : 2 * sms;
  wide_score_kernel<<<grid, kT, static_cast<size_t>(ws.Mp) * 4 * B, s>>>(ws, B);
  const int rc = row_cache(ws.Mp, ws.Smax, 0, kWideMaxSmem);
  by_slots(slots_per_thread(ws.Mp), [&](auto v) {
    constexpr int V = decltype(v)::value;
    wide_step_kernel<V><<<B, kT, small_bytes(ws.Mp, ws.Smax, 0, rc), s>>>(ws, S, eps, eps_rel, ws.upd_w,
                                                                         update_slots(ws.Mp, ws.upd_w), rc);
  });
}

}  // namespace ompk
