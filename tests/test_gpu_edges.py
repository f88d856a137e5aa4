"""Values and sizes at the edges of what the kernels' shortcuts assume."""
import math

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


def _planted(M, N, B, S, seed, sigma=1e-3):
    rng = np.random.default_rng(seed)
    At = rng.standard_normal((N, M))
    At = (At / np.linalg.norm(At, axis=1, keepdims=True)).astype(np.float32)
    sup = np.stack([rng.choice(N, S, replace=False) for _ in range(B)])
    Y = np.einsum("bs,bsm->bm", rng.standard_normal((B, S)), At[sup].astype(np.float64))
    Y += sigma * rng.standard_normal((B, M))
    return torch.from_numpy(At).cuda(), torch.from_numpy(Y.astype(np.float32)).cuda(), sup


def _words(out):
    return [t.cpu().numpy().view(np.uint32) for t in out]


def _quantised(x, prec):
    """Rows as the correlation multiplies them, in FP64, and each row's scale."""
    if prec == "bf16":
        return x.bfloat16().double(), torch.ones(x.shape[0], dtype=torch.float64, device=x.device)
    amax = x.abs().amax(dim=1, keepdim=True)
    return (x * (448.0 / amax)).to(torch.float8_e4m3fn).double(), (amax[:, 0] / 448.0).double()


# omp_correlate_topk is one correlation of its own: what a solve left on the handle (its signals'
# residual norms, thresholds) does not enter its lists. A score is within the accumulation's
# Mp 2^-22 and four roundings of the product of the quantised rows, so the list's j-th score is within
# that of the j-th largest.
@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_topk_after_a_solve(lib, prec):
    M, N, B, S = 256, 2000, 200, 24
    At, Y, _ = _planted(M, N, B, 6, 3, sigma=0.0)
    s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=prec)
    s.solve(At.t(), Y, S)               # residuals far below the rows' norms that follow
    R = 30.0 * torch.from_numpy(np.random.default_rng(4).standard_normal((B, M)).astype(np.float32)).cuda()
    idx = torch.empty((B, 8), dtype=torch.int32, device="cuda")
    sc = torch.empty((B, 8), device="cuda")
    lib.omp_correlate_topk(s.h, At.t(), R, 8, idx, sc)
    s.close()
    qa, sa = _quantised(At, prec)
    qr, _ = _quantised(R, prec)
    scale = sa / torch.linalg.vector_norm(At.double(), dim=1)
    score = (qr @ qa.t()).abs() * scale
    tol = (M * 2.0 ** -22 + 4 * 2.0 ** -24) * torch.linalg.vector_norm(qr, dim=1, keepdim=True) * (
        torch.linalg.vector_norm(qa, dim=1) * scale).max()
    assert all(len(set(row)) == 8 and min(row) >= 0 for row in idx.tolist())
    own = score.gather(1, idx.long())
    assert bool(((sc.double() - own).abs() <= tol).all())
    assert bool(((sc.double() - score.topk(8, dim=1).values).abs() <= tol).all())


# An atom with a NaN or an infinity has no score: the solve goes as if it were zero, also at the steps
# whose thresholds leave a list nothing but that atom.
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("B", [1, 300])
def test_atoms_that_are_not_finite(lib, prec, B):
    M, N, S = 256, 2000, 12
    At, Y, sup = _planted(M, N, B, 6, 5)
    bad = [n for n in (0, 130, 700, 1300, 1999) if n not in set(sup.ravel())] or [2]
    out = []
    for v in (0.0, float("nan"), float("inf")):
        D = At.clone()
        D[bad] = 0.0
        D[bad, 7] = v
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=prec)
        out.append(_words(s.solve(D.t(), Y, S, diagnostics=True)))
        s.close()
    for got in out[1:]:
        for g, want in zip(got, out[0]):
            assert np.array_equal(g, want)


# Few signals over a large dictionary: an atom far from unit norm is scored again wherever it stands
# among the four atoms that share a recorded maximum.
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("B", [1, 4])
@pytest.mark.parametrize("scale", [1e18, 1e-18])
def test_few_signals_far_norms_at_any_place(lib, prec, B, scale):
    M, N, S = 512, 1027, 4
    At, _, _ = _planted(M, N, 1, 1, 6)
    atoms = [400, 405, 410, 415]                 # places 0, 1, 2, 3 of their fours
    Y = 3.0 * At[atoms] + At[[100, 200, 300, 500]]
    At[atoms] *= scale
    for lo in range(0, 4, B):
        out = []
        for graph in (1, 2):                     # the device-side loop runs the batched kernels
            s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=prec, use_graph=graph)
            out.append(_words(s.solve(At.t(), Y[lo:lo + B].clone(), S, diagnostics=True)))
            s.close()
        assert out[0][1][:, 0].tolist() == atoms[lo:lo + B]
        for g, want in zip(*out):
            assert np.array_equal(g, want)


def test_candidate_that_is_not_finite(lib):
    """A candidate atom with a NaN is passed over by the restricted steps."""
    M, N, B, S, K = 256, 1000, 50, 6, 40
    At, Y, sup = _planted(M, N, B, S, 7)
    rng = np.random.default_rng(8)
    bad = next(n for n in range(N) if n not in set(sup.ravel()))
    At[bad, 3] = float("nan")
    cand = np.stack([np.concatenate([r, rng.choice([n for n in range(N) if n != bad and n not in set(r)], K - S,
                                                   replace=False)]) for r in sup]).astype(np.int32)
    out = []
    for place in (bad, -1):                      # -1: no candidate
        c = cand.copy()
        c[:, -1] = place
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision="bf16")
        X = torch.empty((B, S), device="cuda")
        so = torch.empty((B, S), dtype=torch.int32, device="cuda")
        fb = torch.empty(B, dtype=torch.int32, device="cuda")
        lib.omp_solve_batch_candidates(s.h, At.t(), Y, S, 0.0, torch.from_numpy(c).cuda(),
                                       torch.zeros(S, device="cuda"), X, so, fallback_out=fb)
        out.append(_words((X, so, fb)))
        s.close()
    assert (out[1][2].view(np.int32) == -1).all()
    for g, want in zip(*out):
        assert np.array_equal(g, want)


def _near_copies(M, N, B, seed):
    """40 near copies of each of N / 40 atoms: FP32's filter decides almost no pick between them."""
    base, _, _ = _planted(M, (N + 39) // 40, 1, 1, seed)
    noise, _, _ = _planted(M, N, 1, 1, seed + 1)
    At = base.repeat_interleave(40, 0)[:N] + 1e-3 * noise
    At /= At.norm(dim=1, keepdim=True)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    sup = torch.rand((B, N), generator=g, device="cuda").topk(5).indices
    coef = torch.randn((B, 5), generator=g, device="cuda")
    Y = 1e-3 * torch.randn((B, M), generator=g, device="cuda")
    for j in range(5):
        Y += coef[:, j, None] * At[sup[:, j]]
    return At, Y


# Positions that the filter leaves to FP32 in numbers: more row tiles than one pass of the blocks, few
# and many column tiles, half of the positions only, steps that go without the filter and steps that try
# it again; the same words as with every atom scored in FP32.
@pytest.mark.parametrize("M,N,B,plain,graph", [(256, 2000, 2600, 0, 1), (300, 200, 4000, 0, 2), (256, 2000, 1500, 750, 0),
                                               (1030, 4100, 300, 0, 1)])
def test_fp32_overflow_is_exact(lib, monkeypatch, M, N, B, plain, graph):
    At, Y = _near_copies(M, N, B, M + N)
    if plain:  # signals that the filter decides: atoms of their own
        D, Yp, _ = _planted(M, N, plain, 5, 9)
        At = torch.cat([At[:N // 2], D[:N // 2]])
        Y[:plain] = D[:N // 2][torch.arange(plain, device="cuda") % (N // 2)] + 0.3 * Yp
    out = []
    for hook in ("0", "1"):
        monkeypatch.setenv("OMP_RESCORE_ALWAYS", hook)
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=10, precision="fp32", use_graph=graph)
        out.append(_words(s.solve(At.t(), Y, 10, diagnostics=True)))
        s.close()
    for g, want in zip(*out):
        assert np.array_equal(g, want)


def _solve_ms(s, At, Y, S):
    ts = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        s.solve(At.t(), Y, S)
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return min(ts)


def test_fp32_overflow_fills_the_gpu(lib, monkeypatch):
    """Where the filter decides nothing, a solve takes less than twice the time without it (one row of
    16 blocks took ten times)."""
    At, Y = _near_copies(256, 1024, 5000, 1)
    ms = []
    for hook in ("0", "1"):
        monkeypatch.setenv("OMP_RESCORE_ALWAYS", hook)
        s = lib.OmpSolver(256, 1024, max_batch=5000, max_iters=16, precision="fp32")
        ms.append(_solve_ms(s, At, Y, 16))
        s.close()
    assert ms[0] < 2.0 * ms[1], ms


# Each few-signal form gives way where the batched kernels are faster: more signals than its resident
# blocks take in a round or two, more atoms than a block scores quickly, more products than the tensor
# cores need long for. The device-side loop always runs the batched kernels (and takes a few us a step
# more), so a solve that chooses takes no longer.
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("M,N,B", [(64, 128, 3000), (64, 256, 1500), (64, 4096, 16), (128, 512, 360), (256, 1024, 60),
                                   (128, 2048, 16), (4096, 6000, 8)])
def test_few_signal_forms_give_way(lib, prec, M, N, B):
    At, Y, _ = _planted(M, N, B, 6, M + N)
    ms = []
    for graph in (1, 2):
        s = lib.OmpSolver(M, N, max_batch=B, max_iters=12, precision=prec, use_graph=graph)
        ms.append(_solve_ms(s, At, Y, 12))
        s.close()
    assert ms[0] < 1.1 * ms[1], ms


def _handle_bytes(lib, *args, **kw):
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s = lib.OmpSolver(*args, **kw)
    used = free - torch.cuda.mem_get_info()[0]
    s.close()
    return used


# Bytes a signal of a handle's workspaces: the residual and its two quantised copies, 32 candidate lists
# at most, the factor in FP64 and FP32, the traces, the staged signals and results.
@pytest.mark.parametrize("prec,M,N", [("bf16", 256, 1024), ("bf16", 64, 3000), ("fp8", 128, 256), ("fp32", 64, 100)])
def test_workspace_per_signal(lib, prec, M, N):
    S = 8
    B = 46000 if prec == "fp32" else 100000      # (46,000 signals of the FP32 size never use the filter)
    per = (_handle_bytes(lib, M, N, max_batch=B, max_iters=S, precision=prec) -
           _handle_bytes(lib, M, N, max_batch=B // 2, max_iters=S, precision=prec)) / (B - B // 2)
    tri = (S * (S + 1) // 2 + 3) // 4 * 4
    rows = 4 * M + {"fp32": 0, "bf16": 4 * M, "fp8": 2 * M}[prec] + 4 * M
    lists = 0 if prec == "fp32" else 32 * 64
    assert per <= rows + lists + 12 * tri + (8 + 4 * 5) * S + 120, per


# A handle whose workspaces do not fit does without those that only make solves faster, and gives the
# same words; one that does not fit without them either is refused.
@pytest.mark.parametrize("prec,M,N,B", [("fp32", 300, 700, 3000), ("bf16", 200, 9000, 16000), ("fp8", 3000, 15000, 1100)])
def test_workspaces_that_do_not_fit(lib, monkeypatch, prec, M, N, B):
    S = 6
    At, Y, _ = _planted(M, N, 200, S, M)
    Y = Y.repeat((B + 199) // 200, 1)[:B].contiguous()
    kw = dict(max_batch=B, max_iters=S, precision=prec)
    full = _handle_bytes(lib, M, N, **kw)
    out, used = [], []
    for limit in (None, full - (4 << 20)):       # (allocations come in pages of 2 MB)
        if limit:
            monkeypatch.setenv("OMP_FAULT_ALLOC_BYTES", str(limit))
        used.append(_handle_bytes(lib, M, N, **kw))
        s = lib.OmpSolver(M, N, **kw)
        out.append(_words(s.solve(At.t(), Y, S, diagnostics=True)))
        few = s.solve(At.t(), Y[:20].clone(), S)[1]
        assert torch.equal(few, torch.from_numpy(out[0][1][:20].astype(np.int32)).cuda())
        s.close()
    assert used[1] < used[0]
    for g, want in zip(*out):
        assert np.array_equal(g, want)
    monkeypatch.setenv("OMP_FAULT_ALLOC_BYTES", str(1 << 20))
    with pytest.raises(lib.OmpError):
        lib.OmpSolver(M, N, **kw)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_autotune_of_few_signals(lib, monkeypatch, tmp_path, prec):
    """Solves of few signals launch none of the kernels that the tuner times: it keeps the handle's
    shapes and records nothing, except where the device-side loop runs the batched kernels."""
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("OMP_AUTOTUNE_CACHE", str(cache))
    At, Y, _ = _planted(64, 256, 16, 6, 2)
    for graph in (1, 0, 2):
        s = lib.OmpSolver(64, 256, max_batch=16, max_iters=8, precision=prec, use_graph=graph)
        before = lib.omp_tuning(s.h)
        choice = lib.omp_autotune(s.h, At.t(), Y, 8, 0.0, repeats=1)
        assert choice == lib.omp_tuning(s.h)[0]
        if graph != 2:
            assert lib.omp_tuning(s.h) == before and not cache.exists()
        s.close()
    assert len(cache.read_text().splitlines()) == 1


def _near_midpoint(M, d, seed):
    """A signal whose norm lies d (relative, squared) from the midpoint of two neighbouring floats, and
    its norm rounded to the nearest."""
    rng = np.random.default_rng(seed)
    y = (rng.standard_normal(M) * np.exp(4 * rng.standard_normal(M))).astype(np.float32)
    y[-3:] = 0.0
    s = math.fsum(float(v) ** 2 for v in y)      # (the square of a float is a double)
    lo = np.float32(math.sqrt(s * 1.0001))
    hi = np.nextafter(lo, np.float32(np.inf))
    mid2 = ((float(lo) + float(hi)) / 2) ** 2
    for i, part in ((-3, 0.999), (-2, 0.999), (-1, 1.0)):
        rest = math.fsum([mid2, mid2 * d] + [-float(v) ** 2 for v in y])
        y[i] = np.float32(math.sqrt(max(rest, 0.0) * part))
    off = math.fsum([-mid2] + [float(v) ** 2 for v in y]) / mid2
    assert 0.5 * abs(d) < off * np.sign(d) < 2 * abs(d)
    return y, hi if d > 0 else lo


def test_signal_norms_keep_the_bits_of_fp64(lib):
    """||y|| is the float nearest to the norm as FP64 sums form it: to 2^-47 of the sum of squares, four
    times the rounding that 256 FP64 additions a lane and five across the warp showed (2^-48.8)."""
    M = 8192
    rows = [_near_midpoint(M, sign * 2.0 ** -46, seed) for seed in range(40) for sign in (1, -1)]
    Y = torch.from_numpy(np.stack([y for y, _ in rows])).cuda()
    s = lib.OmpSolver(M, 2, max_batch=len(rows), max_iters=1, precision="fp32")
    out = s.solve(torch.zeros(2, M, device="cuda").t(), Y, 1, diagnostics=True)
    s.close()
    assert not out[2].any()                      # no atom to pick: the residual is the signal
    assert np.array_equal(out[3].cpu().numpy(), np.array([n for _, n in rows]))


def test_training_loss_has_the_bits_of_log1p(lib):
    """One logit at a time, all others at -40 with label 0: the loss is log(1 + e^-|o|) of that logit to
    the error of FP32's own log1p and exp (those of torch on the same values)."""
    n = 64
    At = torch.eye(n, device="cuda")
    Y = torch.zeros(n, n, device="cuda")
    Y[0, 0] = 1.0
    Y[1:, 1] = 1.0
    s = lib.OmpSolver(n, n, max_batch=n, max_iters=1, precision="bf16")
    p = lib.Proposal(s.h, hidden=n, topk=8, train_batch=n)
    zero = [torch.zeros(k, device="cuda") for k in ((n, n), n, (n, n))]
    got, o = [], []
    loss = torch.zeros(1, device="cuda")
    for i, beta in enumerate(40.0 + np.random.default_rng(3).uniform(-12, 12, 1500).astype(np.float32)):
        b2 = torch.full((n,), -40.0, device="cuda")
        b2[1] = -200.0                           # the other rows' one feature
        logit = np.float32(beta) - np.float32(40.0)
        labels = torch.full((n, 1), -1, dtype=torch.int32, device="cuda")
        labels[0, 0] = 0 if logit > 0 else -1    # the label that leaves the logarithm alone
        p.set_weights(zero[0], zero[1], zero[2], b2, torch.full((1,), float(beta), device="cuda"))
        p.gradients(At.t(), Y, labels, loss_out=loss)
        got.append(float(loss) * n * n)          # (a power of two)
        o.append(float(logit))
    p.close()
    s.close()
    o = torch.tensor(o, device="cuda")
    exact = torch.log1p(torch.exp(-o.double().abs()))
    err = ((torch.tensor(got, device="cuda", dtype=torch.float64) - exact).abs() / exact).max()
    own = ((torch.log1p(torch.exp(-o.abs())).double() - exact).abs() / exact).max()
    assert err <= own * (1 + 1e-9), (float(err), float(own))


# The gather in a launch of its own from some step of a solve on (later for short rows, few signals and
# BF16), or for all steps of the device-side loop: the same words as the one-kernel steps that smaller
# batches take throughout.
@pytest.mark.parametrize("prec,M,N,B,S,kw", [
    ("fp8", 4000, 11000, 1100, 14, {}), ("fp8", 4000, 11000, 1100, 18, {"use_graph": 2}), ("bf16", 8192, 5200, 1100, 32, {}),
    ("fp32", 2050, 20500, 1100, 16, {}), ("bf16", 2048, 21000, 2100, 28, {"gather24": True}),
    ("fp8", 1000, 41000, 2100, 27, {}), ("fp32", 2048, 21000, 2100, 40, {"use_graph": 2})])
def test_gather_apart_from_a_step_on(lib, prec, M, N, B, S, kw):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N)
    At = torch.randn((N, M), generator=g, device="cuda")
    At /= At.norm(dim=1, keepdim=True)
    sup = torch.randint(0, N, (B, S), generator=g, device="cuda")
    coef = torch.randn((B, S), generator=g, device="cuda")
    coef[::3, S // 2:] = 0.0                     # these reach the threshold half way
    Y = 1e-4 * torch.randn((B, M), generator=g, device="cuda")
    for j in range(S):
        Y += coef[:, j, None] * At[sup[:, j]]
    Y[5] = 0.0
    out = []
    s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision=prec, **kw)
    for n in (B, 550):
        parts = [s.solve(At.t(), Y[lo:lo + n].clone(), S, 0.01, diagnostics=True) for lo in range(0, B, n)]
        out.append([torch.cat(p).cpu().numpy().view(np.uint32) for p in zip(*parts)])
    s.close()
    for got, want in zip(*out):
        assert np.array_equal(got, want)


def test_gather_apart_not_in_short_solves(lib):
    """1024 signals take a gather of its own where it pays; a short solve of them takes no longer than
    one of 1000, which never do (both fill eight row tiles): 2.4 % more signals, and as much again."""
    At, Y, _ = _planted(2048, 24576, 1024, 6, 1)
    ms = []
    for B in (1024, 1000):
        s = lib.OmpSolver(2048, 24576, max_batch=1024, max_iters=12, precision="bf16")
        ms.append(_solve_ms(s, At, Y[:B].contiguous(), 12))
        s.close()
    assert ms[0] < 1.05 * ms[1], ms


def test_candidates_without_the_filter(lib):
    """A small FP32 solve restricted to candidates runs its dense loop in three launches a step."""
    from torch.profiler import ProfilerActivity, profile
    M, N, B, S = 256, 1024, 20, 8
    At, Y, sup = _planted(M, N, B, S, 11)
    s = lib.OmpSolver(M, N, max_batch=B, max_iters=S, precision="fp32")
    X = torch.empty((B, S), device="cuda")
    so = torch.empty((B, S), dtype=torch.int32, device="cuda")
    cand = torch.from_numpy(np.ascontiguousarray(sup[:, :S // 2]).astype(np.int32)).cuda()
    tau = torch.full((S,), 1e-6, device="cuda")
    n = 0
    for _ in range(2):                           # (the profiler may miss the first)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            lib.omp_solve_batch_candidates(s.h, At.t(), Y, S, 0.0, cand, tau, X, so)
            torch.cuda.synchronize()
        n = max(n, sum(1 for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA
                       and "kernel" in e.name))
    s.close()
    assert n <= 3 * S + 5, n


def test_one_block_a_signal_ends_with_it(lib):
    """A signal that reaches its threshold after a few of many steps takes a fraction of the time of all
    the steps: its block ends, where the other forms still launch every step."""
    At, Y, _ = _planted(256, 512, 1, 4, 5)
    s = lib.OmpSolver(256, 512, max_batch=1, max_iters=128, precision="bf16")
    ms = []
    for eps in (0.05, 1e-30):
        for _ in range(3):
            s.solve(At.t(), Y, 128, eps)
        ts = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            n = s.solve(At.t(), Y, 128, eps, diagnostics=True)[2]
            b.record()
            torch.cuda.synchronize()
            ts.append(a.elapsed_time(b))
        ms.append((min(ts), int(n)))
    s.close()
    (t0, n0), (t1, n1) = ms
    assert n0 <= 8 and n1 > 64 and t0 < 0.2 * t1, ms
