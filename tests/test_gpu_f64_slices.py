"""The binary64 products as exact slices on the tensor cores, against exact rational sums of the same terms:
inside gamma_K S (the bound of a binary64 sum in any order, which the header promises) at every edge of the
tiles, and on the inputs that fixed point alone would get wrong."""

import math
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


def _product(spl, X, W, C=None):
    """X W^T through the correction (fp32 X), or fl32(X W^T - C) through the unmask (binary64 X; C = 0 if not given)."""
    M, K = X.shape
    N = W.shape[0]
    ws = spl.workspace(spl.spl_f64_workspace_bytes(M, K, N))
    # the slices' workspace: 12 bytes an output and K range, 8 a row
    assert ws.numel() >= 64 * 1024 + 12 * M * N + 8 * (M + N)
    if X.dtype == torch.float32:
        out = torch.full((M, N), float("nan"), device="cuda", dtype=torch.float64)
        spl.spl_precompute_noise_product_f64(out, X, W, workspace=ws)
    else:
        out = torch.full((M, N), float("nan"), device="cuda")
        if C is None:
            C = torch.zeros((M, N), device="cuda", dtype=torch.float64)
        spl.spl_masked_linear_unmask_f64(out, X, W, C, workspace=ws)
    assert spl.spl_get_device_status() == 0
    return out


def _sums(spl, X, W, exact):
    """The product's binary64 sums at the outputs of `exact` {(m, n): Fraction}.  Of a binary64 X the entry point
    returns fl32(sum - C): with C 1024 last places below the exact sum, sum - C is about 1024 of them and every bit
    of the sum is in the result."""
    if X.dtype == torch.float32:
        got = _product(spl, X, W).cpu()
        assert bool(torch.isfinite(got).all())
        return {o: Fraction(float(got[o])) for o in exact}
    C = torch.zeros((X.shape[0], W.shape[0]), dtype=torch.float64)
    for o, e in exact.items():
        C[o] = float(e) - 1024 * float(np.spacing(abs(float(e)))) if e else 0.0
    got = _product(spl, X, W, C.cuda()).cpu()
    assert bool(torch.isfinite(got).all())
    return {o: Fraction(float(got[o])) + Fraction(float(C[o])) for o in exact}


def _check(spl, X, W, samples):
    X, W = X.cuda(), W.cuda()
    K = X.shape[1]
    exact, S = {}, {}
    for m, n in samples:
        terms = [Fraction(a) * Fraction(b) for a, b in zip(X[m].tolist(), W[n].tolist())]
        exact[m, n], S[m, n] = sum(terms), float(sum(abs(t) for t in terms))
    for o, got in _sums(spl, X, W, exact).items():
        tol = K * U64 / (1 - K * U64) * S[o] + 4 * U64 * abs(float(exact[o])) + 2.0 ** -149  # the least fp32
        assert abs(float(got - exact[o])) <= tol, (o, float(got), float(exact[o]), tol)


def _sample(M, N, count=24):
    rng = np.random.default_rng(5)
    corners = [(0, 0), (M - 1, N - 1), (0, N - 1), (M - 1, 0)]
    return corners + [(int(rng.integers(M)), int(rng.integers(N))) for _ in range(count)]


# tokens at the tile widths and past them, weight rows at 128, K at a chunk, past one, over several K ranges
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("M,K,N", [(1, 8192, 1040), (16, 1024, 300), (17, 1152, 257), (32, 132 * 8, 129), (33, 4100, 128),
                                   (64, 640, 127), (65, 2052, 513), (130, 4096, 130), (256, 132, 129)])
def test_slices_match_exact_sums(spl, dtype, M, K, N):
    g = torch.Generator().manual_seed(M + K + N)
    X = torch.randn((M, K), generator=g, dtype=torch.float64) * 2.6e8
    W = torch.randn((N, K), generator=g) * 0.02
    _check(spl, X.to(dtype), W, _sample(M, N))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_slices_hold_the_largest_digit_sums(spl, dtype):
    """Digits of the largest magnitude and of one sign all along K, at every place of the weight: binary64 rows whose
    digits are 64 and six of -128, against fp32 rows whose entries are three digits of -127, placed by the row's one
    large entry (fp32 X: the same).  Three such pairs meet in an accumulator, as many as 24 bits of weight allow: 3 x
    128 x 127 x 128 of its 2^24.  All entries are whole in fixed point, so the error is the dropped products (below
    2^-57.6 of 2^(E_x + E_w) a term) and the result's rounding."""
    M, K, N = 40, 4096, 256
    low = [-float(0x7F7F7F) * 2.0 ** (8 * p - 53) for p in range(4)]  # beside an entry of 1: digits p, p + 1, p + 2
    W = torch.tensor(low, dtype=torch.float32).repeat(N // 4)[:, None].repeat(1, K)
    W[:, 0] = 1.0
    if dtype == torch.float64:
        X = torch.full((M, K), float(0x3F7F7F7F7F7F80) * 2.0 ** -53, dtype=dtype)  # E = 0
        X[1::2] *= -2.0 ** 40
    else:
        X = torch.tensor(low, dtype=dtype).repeat(M // 4)[:, None].repeat(1, K)
        X[:, 0] = 1.0
        X[4:8] *= -2.0 ** 40
    assert X.unique(dim=0).shape[0] <= 8
    exact = {}
    for m in range(8):
        for n in range(4):
            exact[m, n] = sum(Fraction(a) * Fraction(b) for a, b in zip(X[m].tolist(), W[n].tolist()))
    got = _sums(spl, X.cuda(), W.cuda(), exact)
    for (m, n), g in got.items():
        scale = 2.0 ** 40 if (m % 2 == 1 if dtype == torch.float64 else m >= 4) else 1.0
        tol = K * 2.0 ** -57.6 * scale + 2 * U64 * abs(float(exact[m, n]))
        assert abs(float(g - exact[m, n])) <= tol, (m, n, float(g), float(exact[m, n]))
    full = _product(spl, X.cuda(), W.cuda())  # every other row and column repeats these, bit for bit
    period = 2 if dtype == torch.float64 else 8
    for m in range(M):
        same = m % period if dtype == torch.float64 else (m if m < 8 else m % 4)
        assert torch.equal(full[m], full[same])
    assert torch.equal(full[:, 4:], full[:, :-4])


def test_slices_of_rows_that_fixed_point_loses(spl):
    """Large entries that meet zero weights, entries over 120 binades, rows of zeros, denormals: summed again in
    binary64 where the slices cannot hold the bound."""
    M, K, N = 24, 1024, 192
    g = torch.Generator().manual_seed(9)
    X = torch.randn((M, K), generator=g, dtype=torch.float64)
    W = torch.randn((N, K), generator=g) * 0.02
    X[:, 5] = 1e250
    W[:, 5] = 0.0
    X[3] = 0.0
    W[7] = 0.0
    X[4] = X[4].abs() * 5e-324 * 1000
    W[9, 1:] = 0.0
    X[6] = torch.ldexp(torch.randn(K, generator=g, dtype=torch.float64), torch.randint(-60, 60, (K,), generator=g))
    X[6, 5] = 1.0
    _check(spl, X, W, [(m, n) for m in (0, 3, 4, 23) for n in (0, 7, 9, 191)])
    got = _product(spl, X.cuda(), W.cuda())
    assert torch.equal(got[3], torch.zeros_like(got[3])) and torch.equal(got[:, 7], torch.zeros_like(got[:, 7]))


# one row (a task of one row), rows and columns past the tasks of 4, several blocks, K past the runs of 512; what is
# cleared by more of K, what only by all of it, what not at all
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("M,K,N", [(1, 8192, 1027), (5, 1028, 1029), (16, 516, 520), (33, 640, 257)])
@pytest.mark.parametrize("scale", [100.0, 1e3, 1e5, 1e30])
def test_slices_of_rows_with_one_large_entry(spl, dtype, M, K, N, scale):
    g = torch.Generator().manual_seed(M + K + N)
    X = torch.randn((M, K), generator=g, dtype=torch.float64)
    W = torch.randn((N, K), generator=g) * 0.02
    X[:, 7] *= scale
    if scale == 1e30:
        W[:, 7] = 0.0
    if M > 5:
        X[1::3, 7] = 0.0  # rows that the samples clear between the others
    _check(spl, X.to(dtype), W, _sample(M, N, 12))


def test_rows_with_one_large_entry_are_cleared_by_more_of_k(spl):
    """Rows that 128 samples of K do not clear cost little more than others (1.04 to 1.4 times): Down's shape, one entry
    1000 times the rest.  Summed again in binary64 they took 6 times as long for one row and 18 times for 16."""
    K, N = 8192, 3072
    for M in (1, 4, 16):
        g = torch.Generator(device="cuda").manual_seed(M)
        X = torch.randn((M, K), generator=g, device="cuda", dtype=torch.float64)
        X[:, 7] *= 1e3
        W = torch.randn((N, K), generator=g, device="cuda") * 0.02
        C, Y = torch.zeros((M, N), device="cuda", dtype=torch.float64), torch.empty((M, N), device="cuda")
        ws = spl.workspace(spl.spl_f64_workspace_bytes(M, K, N))

        def best(run):
            run()
            t = []
            for _ in range(10):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                run()
                b.record()
                b.synchronize()
                t.append(a.elapsed_time(b))
            return min(t)

        large = best(lambda: spl.spl_masked_linear_unmask_f64(Y, X, W, C, workspace=ws))
        X[:, 7] /= 1e3
        plain = best(lambda: spl.spl_masked_linear_unmask_f64(Y, X, W, C, workspace=ws))
        assert large <= 2.0 * plain, (M, large, plain)


def test_slices_pass_infinities_and_nans_on(spl):
    M, K, N = 44, 512, 200
    g = torch.Generator().manual_seed(11)
    X = torch.randn((M, K), generator=g, dtype=torch.float64).cuda()
    W = (torch.randn((N, K), generator=g) * 0.02).cuda()
    clean = _product(spl, X, W)
    X2, W2 = X.clone(), W.clone()
    X2[2, 7], X2[5, 9] = float("inf"), float("nan")
    W2[11, 100], W2[60, 7] = float("nan"), 0.0
    got = _product(spl, X2, W2)
    ref = (X2 @ W2.double().T).float()
    assert torch.equal(torch.isnan(got), torch.isnan(ref)) and torch.equal(torch.isinf(got), torch.isinf(ref))
    assert torch.equal(got[torch.isinf(ref)], ref[torch.isinf(ref)])
    keep = torch.ones((M, N), dtype=torch.bool, device="cuda")
    keep[2], keep[5], keep[:, 11], keep[:, 60] = False, False, False, False
    assert torch.equal(got[keep], clean[keep])


@pytest.mark.parametrize("top_x,top_w", [(24, 8), (23, 24), (1, 1), (12, 16)])
def test_slices_of_integers_are_exact(spl, top_x, top_w):
    """Slalom's products: integers below 2^24 whose sums stay below 2^53 lose nothing in the slices."""
    M, K, N = 37, 1028, 514
    g = torch.Generator(device="cuda").manual_seed(top_x)
    K_cut = K if top_x + top_w + 11 <= 53 else 60  # 60 terms of 2^47: the rest of the row is 0
    X = torch.randint(-2 ** top_x + 1, 2 ** top_x, (M, K), generator=g, device="cuda")
    W = torch.randint(-2 ** top_w + 1, 2 ** top_w, (N, K), generator=g, device="cuda")
    X[:, K_cut:] = 0
    X[:, 0] = 1 - 2 ** top_x
    got = _product(spl, X.float(), W.float()).cpu()
    want = (X.cpu() @ W.cpu().T).double()
    assert torch.equal(got, want)


@pytest.mark.parametrize("seed", [1, 2])
def test_slices_are_closer_than_a_binary64_sum(spl, seed):
    """No less precise than the FP64 pipe: over noise-like rows of the Down shape the error of the slices, in units
    of the result's standard deviation, stays below 2^-53 (a binary64 sum of 8192 terms is at 1.8e-16 there)."""
    M, K, N = 64, 8192, 256
    g = torch.Generator().manual_seed(seed)
    X = (torch.randn((M, K), generator=g) * 2.6e8).cuda()
    W = (torch.randn((N, K), generator=g) * 0.02).cuda()
    got = _product(spl, X, W)
    err = []
    for m, n in _sample(M, N, 60):
        exact = sum(Fraction(a) * Fraction(b) for a, b in zip(X[m].tolist(), W[n].tolist()))
        err.append(float(Fraction(float(got[m, n])) - exact))
    assert math.sqrt(np.mean(np.square(err))) <= U64 * 2.6e8 * 0.02 * math.sqrt(K)


def test_smaller_workspace_runs_on_the_fp64_pipe(spl):
    """A workspace below what the slices take, or none, is not refused where the FP64 pipe's kernel needs less."""
    M, K, N = 128, 512, 3072
    g = torch.Generator(device="cuda").manual_seed(9)
    X = torch.randn((M, K), generator=g, device="cuda")
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    full = _product(spl, X, W)
    out = torch.full((M, N), float("nan"), device="cuda", dtype=torch.float64)
    spl.spl_precompute_noise_product_f64(out, X, W, workspace=None)
    S = X.double().abs() @ W.double().abs().T
    assert bool(((out - full).abs() <= 2 * K * U64 / (1 - K * U64) * S).all())
