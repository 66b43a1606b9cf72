"""FP64 products: entry by entry as good as an FP64 sum, whatever path they take."""

import numpy as np
import pytest

from tests.test_gpu_f64_tc import _two_prod_dot

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2110_03607_gb300 as p

    p.load()
    return p


def _split(x):
    t = 134217729.0 * x
    h = t - (t - x)
    return h, x - h


def _error(got, terms):
    """|got - sum of x y over terms| without rounding the sum to 53 bits: exact products, summed as pairs."""
    hi, lo = -got, np.zeros_like(got)
    for x, y in terms:
        p = x * y
        (xh, xl), (yh, yl) = _split(x), _split(y)
        e = xl * yl - (((p - xh * yh) - xl * yh) - xh * yl)
        s = hi + p
        z = s - hi
        lo = lo + ((hi - (s - z)) + (p - z)) + e
        hi = s
    return np.abs(hi + lo)


def _graded(kind, m, n, k, rng):
    a, b = rng.standard_normal((m, k)), rng.standard_normal((n, k))
    x = np.linspace(0.0, 1.0, k)[None, :]
    if kind == "opposite":            # the largest of one row meets the smallest of the other
        return a * 2.0 ** (-80 * x), b * 2.0 ** (80 * x)
    if kind == "one_sided":
        return a * 2.0 ** (-80 * x), b
    if kind == "mixed_rows":          # some pairs of rows are aligned, some opposite, some far below
        s = rng.choice([-60.0, -12.0, 0.0, 12.0, 60.0], (m, 1))
        u = rng.choice([-60.0, 0.0, 60.0], (n, 1))
        return a * 2.0 ** (s * x) * 2.0 ** rng.integers(-200, 200, (m, 1)), b * 2.0 ** (u * x)
    if kind == "disjoint":            # supports that meet only in tiny elements
        h = k // 2
        a[:, h:] *= 1e-20
        b[:, :h] *= 1e-17
        return a, b
    # "integers": digits with structure, exact results
    return rng.integers(-2 ** 26, 2 ** 26, (m, k)).astype(float), rng.integers(-2 ** 20, 2 ** 20, (n, k)).astype(float)


@pytest.mark.parametrize("m,n,k", [(200, 700, 160), (129, 97, 2100), (33, 4096, 130)])
@pytest.mark.parametrize("kind", ["opposite", "one_sided", "mixed_rows", "disjoint", "integers"])
def test_every_entry_is_as_good_as_an_fp64_sum(pkg, kind, m, n, k):
    rng = np.random.default_rng(m + k)
    a, b = _graded(kind, m, n, k, rng)
    assert float(m) * n * k >= 2 ** 24   # the digits' range
    ref, scale = _two_prod_dot(a, b), np.abs(a) @ np.abs(b).T
    got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    # a sum of k products, each addition rounded: k 2^-53 sum |a b|
    assert np.max(np.abs(got - ref) / scale) <= k * 2.0 ** -53
    # and in the mean no worse than its rounding: sqrt(k) of them
    assert np.sqrt(np.mean((np.abs(got - ref) / scale) ** 2)) <= np.sqrt(k) * 2.0 ** -53


def test_small_entries_keep_their_digits(pkg):
    # rows (1, pi 1e-10) and (e 1e-10, 1), and (1, 1e-20) and (0, 1), among others
    rng = np.random.default_rng(1)
    a, b = rng.standard_normal((256, 300)), rng.standard_normal((256, 300))
    a[:2] = b[:2] = 0.0
    a[0, :2], b[0, :2] = (1.0, np.pi * 1e-10), (np.e * 1e-10, 1.0)
    a[1, :2], b[1, :2] = (1.0, 1e-20), (0.0, 1.0)
    got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    for i, j in ((0, 0), (0, 1), (1, 0), (1, 1)):
        want = a[i, 0] * b[j, 0] + a[i, 1] * b[j, 1]
        assert abs(got[i, j] - want) <= 2.0 ** -51 * abs(want)


def test_infinities_keep_their_signs(pkg):
    rng = np.random.default_rng(4)
    a, b = np.abs(rng.standard_normal((256, 300))), rng.standard_normal((256, 300))
    a[3, 5], a[4, 6], b[7, 0], b[8, 9] = np.inf, -np.inf, np.nan, np.inf
    a[5, 0], a[5, 1] = np.inf, -np.inf
    b[9, 5] = 0.0
    with np.errstate(all="ignore"):
        want = a @ b.T
    got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    for f in (np.isnan, np.isposinf, np.isneginf):
        np.testing.assert_array_equal(f(got), f(want))


def test_equal_rows_through_two_pointers(pkg):
    # one large element and many small ones: the squares of the small ones' middle digits are all positive
    rng = np.random.default_rng(8)
    a = 2.0 ** -10 * rng.uniform(0.5, 1.0, (64, 32768)) * rng.choice([-1.0, 1.0], (64, 32768))
    a[:, 0] = 1.0
    got = np.diag(pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, a.copy())).copy()
    assert np.max(_error(got, ((a[:, k], a[:, k]) for k in range(a.shape[1])))) <= 2.0 ** -52


def test_a_sum_is_not_short_of_an_accumulator(pkg):
    # random rows of one size: the products of digits that share a weight have a root mean square of
    # 2^12.4 sqrt(8 k) units of it; the result's own rounding is all that is allowed
    rng = np.random.default_rng(6)
    a, b = rng.uniform(-1, 1, (128, 2048)), rng.uniform(-1, 1, (96, 2048))
    got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    err = _error(got, ((a[:, k][:, None], b[:, k][None, :]) for k in range(a.shape[1])))
    assert np.all(err <= 2.0 ** -53 * np.abs(got) + 2.0 ** -56)


# one pass; several passes of B's rows with a ragged last one (K up to 2048 and above); A == B; A alone beyond
# the array (passes of its rows too, whole tiles or parts of one)
@pytest.mark.parametrize("m,n,k,same", [(200, 700, 160, False), (600, 1800, 1800, False), (300, 1900, 3000, False),
                                        (600, 600, 1024, True), (1700, 1700, 1700, True), (2600, 96, 2100, False),
                                        (31, 5000, 400, False), (72, 96, 32768, False), (48, 64, 120000, False)])
def test_caller_owned_memory_gives_the_same_bits(pkg, m, n, k, same):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    fall = torch.exp(-1.5 * torch.rand(k, generator=gen, device="cuda", dtype=torch.float64))
    a = torch.randn(m, k, generator=gen, device="cuda", dtype=torch.float64) * fall
    b = a if same else torch.randn(n, k, generator=gen, device="cuda", dtype=torch.float64) * fall
    c = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    pkg.hotrg_gemm_nt_noalloc(pkg.PREC_FP64, a, b, c, torch.cuda.current_stream().cuda_stream)
    ref = a @ b.T
    assert ((c - ref).abs() / (a.abs() @ b.abs().T)).max().item() <= 2 * k * 2.0 ** -53
    np.testing.assert_array_equal(c.cpu().numpy(), pkg.hotrg_gemm_nt(pkg.PREC_FP64, a.cpu().numpy(), b.cpu().numpy()))


def test_grams_in_several_passes_along_k(pkg):
    """400 rows of 160,000 terms: the digits do not fit the workspace at once."""
    import torch

    chi = 20
    gen = torch.Generator(device="cuda").manual_seed(2)
    t = torch.rand((chi,) * 6, generator=gen, device="cuda", dtype=torch.float64) - 0.3
    for k in range(6):
        shape = [1] * 6
        shape[k] = chi
        t *= torch.exp(-0.15 * torch.arange(chi, device="cuda", dtype=torch.float64)).reshape(shape)
    t /= torch.einsum("aabbcc->", t).item()
    g = pkg.Hotrg(3, 0.25, 0.01, tensor=t, chis=(chi,) * 3)
    try:
        n = pkg.shard_sizes(g.ctx, 0, chi)[0]
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        pkg.hotrg_shard_env(g.ctx, 0, chi, 0, 1, out=out)
        got = out.reshape(2, 4, chi * chi, chi * chi)
        held = torch.empty_like(t)
        pkg.hotrg_tensor(g.ctx, out=held)
        for j in (1, 2):
            for kind, (f, c) in enumerate(((2 * j, 1), (2 * j, 0), (2 * j + 1, 1), (2 * j + 1, 0))):
                x = held.permute([f, c] + [q for q in range(6) if q not in (f, c)]).reshape(chi * chi, -1)
                ref, scale = x @ x.T, x.abs() @ x.abs().T
                # the reference is a plain FP64 product with a rounding error of its own
                assert ((got[j - 1, kind] - ref).abs() / scale).max().item() <= 1e-13
    finally:
        g.close()
