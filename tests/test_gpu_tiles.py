"""The FP32 tile kernels at the edges of their tiles, against FP64 on the same FP32 inputs.

A chain of M FMAs is within M 2^-24 ||a|| ||r|| of the exact product; the norm's reciprocal and the
product with it add three roundings, so a score is within (M + 4) 2^-24 ||r|| of the exact one and
the picked atom's exact score within twice that of the best."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_06434_gb300 import build
    build.build()
    from paper_2407_06434_gb300 import omp
    omp.load()
    return omp


def _problem(M, N, B, seed):
    rng = np.random.default_rng(seed)
    At = rng.standard_normal((N, M)).astype(np.float32) * rng.uniform(0.5, 2.0, (N, 1)).astype(np.float32)
    R = rng.standard_normal((B, M)).astype(np.float32)
    return At, R


# the last four take tiles 96, 64 and 128 atoms wide with ragged rows and columns
@pytest.mark.parametrize("M,N,B", [(1, 2, 1), (63, 64, 127), (64, 65, 128), (65, 97, 129),
                                   (100, 1207, 1200), (130, 8193, 1001), (40, 4097, 4999), (96, 129, 3)])
def test_fp32_correlation_tiles(lib, M, N, B):
    At, R = _problem(M, N, B, M + N)
    s = lib.OmpSolver(M, N, max_batch=B, max_iters=1, precision="fp32")
    idx = torch.empty((B, 1), dtype=torch.int32, device="cuda")
    sc = torch.empty((B, 1), device="cuda")
    lib.omp_correlate_topk(s.h, torch.from_numpy(At).cuda().t(), torch.from_numpy(R).cuda(), 1, idx, sc)
    idx, sc = idx.cpu().numpy()[:, 0], sc.cpu().numpy()[:, 0].astype(np.float64)
    A64, R64 = At.astype(np.float64), R.astype(np.float64)
    scores = np.abs(R64 @ (A64 / np.linalg.norm(A64, axis=1, keepdims=True)).T)
    tol = (M + 4) * 2.0 ** -24 * np.linalg.norm(R64, axis=1)
    own = scores[np.arange(B), idx]
    assert np.all(np.abs(sc - own) <= tol)
    assert np.all(own >= scores.max(axis=1) - 2 * tol)
    s.close()


# two steps from a signal in the span of two atoms recover it only through the Gram entry between
# them, on either side of the diagonal and in any tile
@pytest.mark.parametrize("N", [64, 65, 127, 129, 257, 1000, 2049])
def test_gram_entries_of_any_tile(lib, N):
    M = 80
    At, _ = _problem(M, N, 1, N)
    At /= np.linalg.norm(At, axis=1, keepdims=True)
    rng = np.random.default_rng(N)
    pairs = np.array([rng.choice(N, 2, replace=False) for _ in range(300)])
    Y = (3.0 * At[pairs[:, 0]] + 2.0 * At[pairs[:, 1]]).astype(np.float32)
    s = lib.OmpSolver(M, N, max_batch=300, max_iters=2, precision="fp32")
    X, sup = s.solve(torch.from_numpy(At).cuda().t(), torch.from_numpy(Y).cuda(), 2)
    X, sup = X.cpu().numpy(), sup.cpu().numpy()
    A64 = At.astype(np.float64)
    for b in range(300):
        ref, *_ = np.linalg.lstsq(A64[sup[b]].T, Y[b].astype(np.float64), rcond=None)
        cond = np.linalg.cond(A64[sup[b]])
        assert np.linalg.norm(X[b] - ref) <= 64 * 2.0 ** -24 * cond ** 2 * np.linalg.norm(ref)
    s.close()


def _planted(M, N, B, S, seed):
    rng = np.random.default_rng(seed)
    At = rng.standard_normal((N, M)).astype(np.float32)
    At *= (rng.uniform(0.5, 2.0, (N, 1)) / np.linalg.norm(At, axis=1, keepdims=True)).astype(np.float32)
    Y = 1e-3 * rng.standard_normal((B, M))
    for b in range(B):
        sup = rng.choice(N, S, replace=False)
        Y[b] += At[sup].T.astype(np.float64) @ rng.standard_normal(S)
    return torch.from_numpy(At).cuda().t(), torch.from_numpy(Y.astype(np.float32)).cuda()


# Few signals take kernels of their own, which pick the same atoms and round every sum alike: the
# device-side loop (use_graph 2) always runs the batched kernels, and the results are bit for bit
# the same. Sizes: one slot per lane and ragged ones, one block per signal at and above the small
# dictionary's limit, 1 to 8 signals over a large one, a factor too long to stage, an eps stop.
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("M,N,B,S,eps", [
    (64, 256, 16, 8, 0.0), (33, 40, 3, 5, 0.0), (128, 512, 100, 16, 0.0), (203, 700, 30, 20, 1e-2),
    (1024, 256, 40, 24, 0.0), (1024, 257, 8, 24, 0.0), (1024, 8192, 1, 32, 0.0), (700, 5000, 7, 24, 1e-2),
    (1500, 4001, 8, 30, 0.0), (4096, 3000, 2, 40, 0.0), (5000, 1201, 2, 100, 0.0), (8192, 600, 6, 16, 0.0)])
def test_few_signals_match_the_batched_kernels(lib, prec, M, N, B, S, eps):
    A, Y = _planted(M, N, B, S, M + 7 * N + B)
    if B > 2:
        Y[1] = 0.0                      # an empty signal
        Y[2] = Y[0]                     # and a repeated one
    out = []
    for graph in (1, 0, 2):
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=prec, use_graph=graph)
        out.append([t.cpu().numpy() for t in s.solve(A, Y, S, eps, diagnostics=True)])
        s.close()
    for got in out[:2]:
        for g, want in zip(got, out[2]):
            assert np.array_equal(g.view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_few_signals_ties_and_extreme_scales(lib, prec):
    """Duplicate atoms (the lowest index wins), a zero atom, atoms and signals far from unit norm."""
    A, Y = _planted(96, 300, 4, 6, 5)
    At = A.t().contiguous()
    At[200] = At[17]
    At[18] = At[17]
    At[5] = 0.0
    At[40] *= 1e18
    At[41] *= 1e-18
    Y[0] = 2.0 * At[17] + 0.5 * At[60]
    Y[1] *= 1e-17
    Y[3] = At[41] * 1e18 + At[40] * 1e-18
    out = []
    for graph in (1, 2):
        s = lib.OmpSolver(96, 300, max_batch=4, max_iters=6, precision=prec, use_graph=graph)
        out.append([t.cpu().numpy() for t in s.solve(At.t(), Y, 6, 0.0, diagnostics=True)])
        s.close()
    assert out[0][1][0, 0] == 17
    for g, want in zip(*out):
        assert np.array_equal(g.view(np.uint32), want.view(np.uint32))


def _solve_both(lib, monkeypatch, A, Y, S, eps, graph=1, **kw):
    """The FP32 solve with its filter and (OMP_RESCORE_ALWAYS=1 when the handle is created) without."""
    out = []
    for hook in ("0", "1"):
        monkeypatch.setenv("OMP_RESCORE_ALWAYS", hook)
        s = lib.OmpSolver(A.shape[0], A.shape[1], max_batch=Y.shape[0], max_iters=S, precision="fp32",
                          use_graph=graph, **kw)
        out.append([t.cpu().numpy() for t in s.solve(A, Y, S, eps, diagnostics=True)])
        s.close()
    return out


# The FP32 path scores in FP32 only the atoms that a bound on the BF16 scores leaves: the same bits
# as scoring every atom. Few and many column tiles, ragged rows, more steps than planted atoms (the
# noise floor, where many scores are close), an eps stop that retires signals at different steps.
@pytest.mark.parametrize("M,N,B,S,planted,eps,graph", [
    (64, 300, 700, 12, 12, 0.0, 1), (256, 1000, 300, 40, 20, 0.0, 1), (203, 1500, 129, 24, 24, 1e-2, 1),
    (1024, 4100, 257, 24, 16, 0.0, 1), (1024, 4100, 200, 20, 20, 1e-2, 2), (2100, 2500, 70, 16, 16, 0.0, 0),
    (640, 8000, 1100, 8, 4, 0.0, 1), (256, 9001, 200, 12, 12, 0.0, 1)])
def test_fp32_filter_is_exact(lib, monkeypatch, M, N, B, S, planted, eps, graph):
    A, Y = _planted(M, N, B, planted, M + N + B)
    Y[3] = 0.0
    got, want = _solve_both(lib, monkeypatch, A, Y, S, eps, graph)
    for g, w in zip(got, want):
        assert np.array_equal(g.view(np.uint32), w.view(np.uint32))


def test_fp32_filter_close_atoms_and_extreme_scales(lib, monkeypatch):
    """Clusters of more nearly equal atoms than a list holds, exact duplicates, signals and atoms far
    from unit norm, an atom of norm 0: the positions that the bound cannot decide."""
    rng = np.random.default_rng(11)
    A, Y = _planted(300, 2000, 400, 10, 12)
    At = A.t().contiguous()
    base = At[:20].repeat_interleave(40, 0)
    noise = torch.from_numpy(rng.standard_normal(base.shape).astype(np.float32)).cuda()
    At[1000:1800] = base + 1e-6 * noise          # 40 near copies of each of 20 atoms
    At[1900:1950] = At[7]                        # exact duplicates
    At[1960] = 0.0
    Y[:100] = At[torch.from_numpy(rng.integers(0, 20, 100)).cuda()] + 1e-3 * Y[:100]
    Y[100] *= 1e-20
    Y[101] *= 1e18
    for scale in (1.0, 1e17):
        At[1970] = At[1970] / At[1970].norm() * scale
        got, want = _solve_both(lib, monkeypatch, At.t(), Y, 10, 0.0)
        for g, w in zip(got, want):
            assert np.array_equal(g.view(np.uint32), w.view(np.uint32))


# The Gram-space solve with 1, 4 and 8 warps a signal (by atoms and batch), atom counts that leave
# the padded Gram rows 1 to 3 columns short, and more atoms than one pass of c holds, against the dense
# FP32 solve: the same picks wherever they agree so far, coefficients within the FP32 error of both.
@pytest.mark.parametrize("M,N,B,S", [(96, 1021, 4900, 8), (96, 1022, 700, 8), (96, 2047, 620, 8), (128, 2051, 640, 8),
                                     (128, 4099, 50, 8), (96, 63, 650, 6)])
def test_gram_solve_warps(lib, M, N, B, S):
    A, Y = _planted(M, N, B, S, M + N + B)
    s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision="fp32")
    X1, s1 = (t.cpu().numpy() for t in s.solve_gram(A, Y, S))
    X2, s2 = (t.cpu().numpy() for t in s.solve(A, Y, S))
    s.close()
    same = np.all(s1 == s2, axis=1)
    assert np.mean(same) > 0.98  # the rest are near-ties
    A64 = A.double().cpu().numpy()
    for b in np.flatnonzero(same)[::17]:
        cond = np.linalg.cond(A64[:, s1[b]])
        assert np.linalg.norm(X1[b] - X2[b]) <= 256 * 2.0 ** -24 * cond ** 2 * np.linalg.norm(X2[b])


# The K largest of a row by equal pieces of the row's range: rows of one value, of few values (a piece
# holds more keys than are listed), of ordinary logits, with infinities, with signed zeros; rows that
# do not fit in shared memory; K at both ends.
@pytest.mark.parametrize("N", [1, 37, 2048, 8192, 41000])
def test_topk_rows_distributions(lib, N):
    rng = np.random.default_rng(N)
    rows = [np.full(N, -3.25), rng.integers(-2, 3, N) * 0.5, rng.standard_normal(N) - 5.0,
            np.where(rng.random(N) < 0.3, np.inf, rng.standard_normal(N)), np.where(rng.random(N) < 0.5, 0.0, -0.0),
            -np.exp(20 * rng.random(N)), np.where(rng.random(N) < 0.9, -np.inf, rng.standard_normal(N)),
            rng.standard_normal(N) * 1e-40, 1.0 + rng.integers(0, 1500, N) * 2.0 ** -23]
    x = np.stack(rows).astype(np.float32)
    u = x.view(np.uint32).astype(np.int64)
    key = np.where(u >> 31, 0xffffffff - u, u | 0x80000000)  # the floats' order, -0 below +0
    for K in sorted({1, min(N, 256), N}):
        idx = torch.empty((len(rows), K), dtype=torch.int32, device="cuda")
        lib.omp_topk_rows(torch.from_numpy(x).cuda(), K, idx)
        want = np.sort(np.argsort(-key, axis=1, kind="stable")[:, :K], axis=1)
        assert np.array_equal(idx.cpu().numpy(), want)


# A dictionary that L2 does not hold has its gather in a launch of its own for 1024 signals and more:
# the same bits as the one-kernel step that smaller batches take. Ragged row lengths (the last piece
# short), every precision, the 24-bit gather, an eps stop that retires signals, margins recorded.
@pytest.mark.parametrize("prec,M,N,kw", [("fp8", 4000, 11000, {}), ("bf16", 3001, 14002, {}), ("fp32", 2050, 20500, {}),
                                         ("bf16", 2048, 21000, {"gather24": True}), ("bf16", 8192, 5200, {})])
def test_gather_apart_is_exact(lib, prec, M, N, kw):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N)
    B, S = 1100, 9
    At = torch.randn((N, M), generator=g, device="cuda")
    At /= At.norm(dim=1, keepdim=True)
    sup = torch.rand((B, N), generator=g, device="cuda").topk(6).indices
    coef = torch.randn((B, 6), generator=g, device="cuda")
    Y = 1e-3 * torch.randn((B, M), generator=g, device="cuda")
    for j in range(6):
        Y += coef[:, j, None] * At[sup[:, j]]
    Y[5] = 0.0
    for eps, margins in ((0.0, False), (0.3, False), (0.0, not kw)):
        out = []
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=prec, **kw)
        for n in (B, 550):
            parts = [s.solve(At.t(), Y[lo:lo + n].clone(), S, eps, diagnostics=True, margins=margins)
                     for lo in range(0, B, n)]
            out.append([torch.cat(p).cpu().numpy() for p in zip(*parts)])
        s.close()
        for got, want in zip(*out):
            assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


# The tensor-core lists against the FP32 tiles: ragged row and column tiles, lists of one column tile
# and of several, duplicate atoms at the edges of groups of 4 and 32 columns and of column tiles (the
# lowest index wins). The planted coefficients are far apart, so the picks are the same integers.
@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("M,N,B", [(128, 253, 1), (256, 300, 129), (256, 1021, 2000), (200, 4099, 700), (512, 1030, 5003),
                                   (256, 9001, 200)])
def test_tensor_core_lists_pick_as_fp32(lib, prec, M, N, B):
    S = 6
    rng = np.random.default_rng(M + N + B)
    At = rng.standard_normal((N, M)).astype(np.float32)
    At /= np.linalg.norm(At, axis=1, keepdims=True)
    for n in (3, 31, 127, 159, 251):
        At[n + 1] = At[n]
    sup = np.stack([rng.choice(N, S, replace=False) for _ in range(B)])
    coef = rng.permuted(np.tile(1.6 ** np.arange(S, dtype=np.float32), (B, 1)), axis=1)
    Y = np.einsum("bs,bsm->bm", coef * rng.choice([-1, 1], (B, S)), At[sup]).astype(np.float32)
    out = []
    for p in ("fp32", prec):
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=p, use_graph=2)
        out.append(s.solve(torch.from_numpy(At).cuda().t(), torch.from_numpy(Y).cuda(), 3)[1].cpu().numpy())
        s.close()
    assert np.array_equal(out[0][:, :3], out[1][:, :3])
    assert not np.isin(out[1][:, :3], (4, 32, 128, 160, 252)).any()
