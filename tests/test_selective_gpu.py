"""GPU parity of pr_selective_metrics (coverage calibration, AUROC, AUARC;
Section 3.1 and Section 4.1) against the float64 oracle in oracle/selective.py.

Counts, the threshold and the AUROC numerator are integers or copied scores:
exact.  AUROC divides an exact integer by P N in double: 1e-12.  AUARC sums n
double terms C_k / k in a different order than numpy: the rounding is below
n * 2^-53 relative, 1e-9 here."""
import numpy as np
import pytest
import torch

from oracle import selective as sel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_28726_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.pr_ctx_create(0, 16, 4)
    yield c
    B.pr_ctx_destroy(c)


def make(n, seed, levels=0, nan_frac=0.0, neg_zero=False):
    """float32 scores (continuous, or `levels` values with many ties) and labels
    whose rate of correct answers rises with the score."""
    g = np.random.Generator(np.random.PCG64(seed))
    if levels:
        s = (np.floor(g.random(n) * levels) / levels).astype(np.float32)
    else:
        s = g.random(n).astype(np.float32)
    y = (g.random(n) < 0.2 + 0.6 * s).astype(np.uint8)
    if nan_frac:
        bad = g.random(n) < nan_frac
        s[bad] = np.where(g.random(bad.sum()) < 0.5, np.nan, np.inf).astype(np.float32)
    if neg_zero:
        s[::7] = np.float32(-0.0)
        s[3::7] = np.float32(0.0)
    return s, y


def run(B, ctx, s, y, q):
    ds = torch.from_numpy(s).cuda()
    dy = None if y is None else torch.from_numpy(y).cuda()
    return B.pr_selective_metrics(ctx, ds, q, labels=dy)


def check(g, s, y, q):
    o = sel.selective_metrics(s, y, q)
    assert g["n_finite"] == o["n_finite"]
    assert g["k"] == o["k"]
    assert g["n_ship"] == o["n_ship"]
    assert np.float32(g["tau"]) == np.float32(o["tau"])
    if y is None:
        assert np.isnan(g["auroc"]) and np.isnan(g["auarc"]) and g["n_pos"] == 0
        return
    assert g["n_pos"] == o["n_pos"]
    for name, tol in (("auroc", 1e-12), ("auarc", 1e-9), ("acc_shipped", 1e-12)):
        a, b = g[name], o[name]
        assert (np.isnan(a) and np.isnan(b)) or abs(a - b) <= tol, (name, a, b)


@pytest.mark.parametrize("n", [1, 2, 31, 2047, 2048, 2049, 4095, 4096, 4097, 12289, 100003])
def test_selective_matches_oracle_sizes(B, ctx, n):
    # bucket targets and ragged tails
    s, y = make(n, seed=n, levels=97, nan_frac=0.03)
    # q * n + 1/2 lands on an integer for some of these: the rounding of q itself
    # must be the oracle's (double)
    for q in (0.0, 0.05, 0.1, 0.3, 0.5, 0.7, 0.77, 0.9, 1.0):
        check(run(B, ctx, s, y, q), s, y, q)


@pytest.mark.parametrize("kind", ["continuous", "few_levels", "one_level", "signed_zero"])
def test_selective_tie_structures(B, ctx, kind):
    n = 30000
    if kind == "continuous":
        s, y = make(n, 1)
    elif kind == "few_levels":
        s, y = make(n, 2, levels=3)
    elif kind == "one_level":
        s, y = make(n, 3)
        s[:] = np.float32(0.625)
    else:
        s, y = make(n, 4, neg_zero=True)
    for q in (0.1, 0.5, 0.9):
        check(run(B, ctx, s, y, q), s, y, q)


@pytest.mark.parametrize("kind", ["logits", "clusters", "neighbours", "extremes", "ties_63_64",
                                  "long_ties", "one_bucket"])
@pytest.mark.parametrize("n", [900, 5000, 70000, 300007])
def test_selective_key_structures(B, ctx, n, kind):
    """Keys spread over both signs and many exponents, piled up in a few buckets,
    a few floats apart, at the ends of the float range; tie groups on both
    sides of the closed form, also at the very top ranks; buckets that are
    sorted and counted (with 32-bit counts: test_selective_large_pool)."""
    g = np.random.Generator(np.random.PCG64(n))
    if kind == "logits":
        s = g.normal(0.0, 2.0, n) ** 3
    elif kind == "clusters":
        s = g.choice([-3.0, 1e-30, 0.7, 0.70001, 1e20], n) * (1.0 + 1e-5 * g.random(n))
    elif kind == "neighbours":
        s = (np.float32(0.75).view(np.uint32) + g.integers(0, 3000, n)).astype(np.uint32)
        s = s.view(np.float32)
    elif kind == "extremes":
        s = g.choice(np.array([1e-45, -1e-45, 3.4028235e38, -3.4028235e38, 0.0, 1.1754944e-38],
                              np.float32), n)
    elif kind == "ties_63_64":
        s = np.repeat(np.arange(n // 60 + 1) / (n // 60 + 1), g.integers(62, 67, n // 60 + 1))[:n]
    elif kind == "long_ties":
        s = np.where(g.random(n) < 0.9, 1.0, g.random(n))
    else:
        s = 0.5 + 2.0 ** -24 * g.integers(0, 1 << 14, n) + 0.0
    s = s.astype(np.float32)
    y = (g.random(n) < 0.3 + 0.4 * (s > np.median(s))).astype(np.uint8)
    for q in (0.001, 0.4, 1.0):
        check(run(B, ctx, s, y, q), s, y, q)
    check(run(B, ctx, s, None, 0.4), s, None, 0.4)
    off = torch.from_numpy(np.concatenate([[0.5], s]).astype(np.float32)).cuda()[1:]  # no vector loads
    lab = torch.from_numpy(np.concatenate([[1], y]).astype(np.uint8)).cuda()[1:]
    check(B.pr_selective_metrics(ctx, off, 0.4, labels=lab), s, y, 0.4)


def test_selective_degenerate_pools(B, ctx):
    s, y = make(5000, 5)
    check(run(B, ctx, s, None, 0.4), s, None, 0.4)          # calibration only
    ones = np.ones_like(y)
    check(run(B, ctx, s, ones, 0.4), s, ones, 0.4)           # no incorrect answer: AUROC NaN
    bad = np.full(1000, np.nan, np.float32)
    g = run(B, ctx, bad, y[:1000], 0.5)
    assert g["n_finite"] == 0 and g["k"] == 0 and g["tau"] == np.inf and np.isnan(g["auarc"])
    g = B.pr_selective_metrics(ctx, torch.empty(0, device="cuda"), 0.5)
    assert g["n_finite"] == 0 and g["tau"] == np.inf
    with pytest.raises(B.PRError):
        run(B, ctx, s, y, 1.5)


def test_selective_is_deterministic(B, ctx):
    s, y = make(200000, 6, levels=1000)
    a = run(B, ctx, s, y, 0.3)
    b = run(B, ctx, s, y, 0.3)
    assert a == b


def test_selective_full_pool(B, ctx):
    """2^24 scores (the benchmark's pool), continuous with a few repeated values."""
    n = 1 << 24
    s, y = make(n, 7)
    s[::1000] = np.float32(0.5)
    check(run(B, ctx, s, y, 0.7), s, y, 0.7)



def test_selective_large_pool(B, ctx):
    """3.4e7 scores, more than 4,096 for each of 8,192 buckets: random bit patterns, whose
    buckets are resolved chunk by chunk; one bin with 5,000 equal scores among its others,
    a chunk that is counted; and one with 122,000 within 2^15 neighbouring keys, a bucket
    counted with 32-bit counts."""
    n = 34_000_000
    g = np.random.Generator(np.random.PCG64(11))
    s = g.integers(0, 2 ** 32, n, dtype=np.uint32).view(np.float32)
    s[~np.isfinite(s)] = 0.25
    at = g.permutation(n)[:127_000]
    one = np.float32(3.0).view(np.uint32)                       # a 2^20-key bin starts here
    s[at[:122_000]] = (one + (5 << 15) + g.integers(0, 2000, 122_000) ** 2 % (1 << 15)).astype(
        np.uint32).view(np.float32)
    s[at[122_000:]] = (np.float32(-7.0).view(np.uint32) + np.uint32(12345)).view(np.float32)
    y = (g.random(n) < np.where(s > 0, 0.7, 0.4)).astype(np.uint8)
    check(run(B, ctx, s, y, 0.3), s, y, 0.3)


@pytest.mark.parametrize("c", [2, 65, 300, 1000, 4000])
def test_selective_ties_below_incorrect_answers(B, ctx, c):
    """A tie group below 64 and below 1,024 times as many incorrect answers, where the
    expansion of its sum in 1 / rank leaves most: at most 2^-34 of the sum (stated in the
    kernel); 2^-33 with the roundings of the oracle's sum here."""
    for times in (64.5, 100, 1025, 1100, 2000):
        a = int(c * times)
        s = np.full(a + c, 0.75, np.float32)
        s[:a] = (np.float32(0.75).view(np.uint32) + np.arange(a, 0, -1, dtype=np.uint32)).view(
            np.float32)
        for p in sorted({1, c // 2, c - 1}):
            y = np.zeros(a + c, np.uint8)
            y[a:a + p] = 1
            k = np.arange(a + 1, a + c + 1, dtype=np.float64)
            want = float(np.sum((p / c) * np.arange(1, c + 1) / k) / (a + c))
            got = run(B, ctx, s, y, 0.5)["auarc"]
            assert abs(got - want) <= 2.0 ** -33 * want, (times, p, got, want)


@pytest.mark.parametrize("n", [500, 900, 20000, 150000, 1000000])
@pytest.mark.parametrize("kind", ["uniform", "bits", "logits"])
def test_selective_repeats_bit_for_bit(B, ctx, n, kind):
    """Pools whose buckets hold a few items, in whatever order these reach them."""
    g = np.random.Generator(np.random.PCG64(n))
    if kind == "bits":
        s = g.integers(0, 2 ** 32, n, dtype=np.uint32).view(np.float32)
        s[~np.isfinite(s)] = 0.25
    else:
        s = g.random(n).astype(np.float32) if kind == "uniform" else g.normal(0, 2, n).astype(np.float32) ** 3
    y = torch.from_numpy((g.random(n) < 0.6).astype(np.uint8)).cuda()
    s = torch.from_numpy(s).cuda()
    first = B.pr_selective_metrics(ctx, s, 0.4, labels=y)
    for _ in range(20):
        assert B.pr_selective_metrics(ctx, s, 0.4, labels=y) == first
