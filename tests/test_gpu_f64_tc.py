"""FP64 products from exact digits on the tensor cores: against 64-bit products with the rounding bound
of the scheme, at the edges of tiles (128 x 64), slabs (32), chunks (128) and of the two ways to cut
rows (K = 2048)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2110_03607_gb300 as p

    p.load()
    return p


def _two_prod_dot(a, b):
    """sum_k a_k b_k to about 100 bits: exact products by splitting, summed as (hi, lo) pairs."""
    def split(x):
        t = 134217729.0 * x
        h = t - (t - x)
        return h, x - h

    hi = np.zeros((a.shape[0], b.shape[0]))
    lo = np.zeros_like(hi)
    for k in range(a.shape[1]):
        x, y = a[:, k][:, None], b[:, k][None, :]
        p = x * y
        (xh, xl), (yh, yl) = split(x), split(y)
        e = xl * yl - (((p - xh * yh) - xl * yh) - xh * yl)
        s = hi + p
        z = s - hi
        lo = lo + ((hi - (s - z)) + (p - z)) + e
        hi = s
    return hi + lo


def _bound(a, b, ref):
    # an element loses at most 2^-62 of 2^e < 2 max|row|; the products left out (a + b > 7: 7 of weight
    # 2^-64, then less) stay below 9 2^-62 of 2^e_i 2^e_j each; one rounding
    k = a.shape[1]
    big = 4.0 * np.abs(a).max(1)[:, None] * np.abs(b).max(1)[None, :]
    return 2.0 ** -53 * np.abs(ref) * (1 + 2.0 ** -40) + 12 * k * 2.0 ** -62 * big


@pytest.mark.parametrize("m,n,k", [(32, 4097, 160), (128, 64, 2048), (129, 65, 2049), (300, 16, 3500), (127, 1029, 129),
                                   (800, 700, 32), (1001, 517, 97), (40, 230, 2016)])
def test_products_within_one_rounding(pkg, m, n, k):
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    a = rng.standard_normal((m, k)) * 2.0 ** rng.integers(-300, 300, (m, 1))
    b = rng.standard_normal((n, k)) * 10.0 ** rng.uniform(-9, 0, (1, k))
    a[1] = 0.0
    b[2, : k // 2] = -b[2, : k // 2] * 1e-30
    ref = _two_prod_dot(a, b)
    got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    assert np.all(np.abs(got - ref) <= _bound(a, b, ref))
    assert np.all(got[1] == 0.0)


def test_largest_digits_do_not_overflow(pkg):
    # every digit at its extreme (-128, and 64 in front) in all 256 terms: the sums reach the bound of
    # the accumulators' exact range
    k = 256
    x = (64 * 256 ** 6 - sum(128 * 256 ** i for i in range(6))) / 2.0 ** 54
    a = np.full((192, k), x)
    b = np.full((512, k), x)
    ref = _two_prod_dot(a[:1], b[:1])[0, 0]
    got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    assert np.all(np.abs(got - ref) <= _bound(a, b, np.full_like(got, ref)))


def test_non_finite_and_tiny_rows(pkg):
    rng = np.random.default_rng(4)
    a, b = rng.standard_normal((256, 300)), rng.standard_normal((256, 300))
    a[3, 5], b[7, 0] = np.inf, np.nan
    a[9] *= 2.0 ** -1040          # subnormal row
    with np.errstate(all="ignore"):
        ref = a @ b.T
        got = pkg.hotrg_gemm_nt(pkg.PREC_FP64, a, b)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    rows = np.ones(256, bool)
    rows[[3, 9]] = False
    cols = np.ones(256, bool)
    cols[7] = False
    scale = np.abs(a[rows]) @ np.abs(b[cols]).T
    assert np.max(np.abs(got - ref)[rows][:, cols] / scale) <= 300 * 2.0 ** -53
    assert np.max(np.abs(got - ref)[9][cols]) <= 300 * 2.0 ** -1070


@pytest.mark.parametrize("chi,axis,field", [(12, 0, 0.0), (11, 1, 0.02), (13, 2, 0.0)])
def test_environment_grams(pkg, chi, axis, field):
    """Symmetric products in splits along K, whole and by parity blocks."""
    import torch

    rng = np.random.default_rng(chi)
    par = [(rng.permutation(chi) & 1).astype(int) for _ in range(3)]
    t = rng.standard_normal((chi,) * 6) * 2.0 ** (-0.5 * rng.integers(0, 24, (chi,) * 6))
    if field == 0.0:
        p = 0
        for k in range(3):
            for q in (0, 1):
                shape = [1] * 6
                shape[2 * k + q] = chi
                p = p ^ par[k].reshape(shape)
        t = np.where(p == 0, t, 0.0)
    t = t / np.einsum("aabbcc->", t)
    g = pkg.Hotrg(3, 0.25, field, tensor=t, chis=(chi,) * 3)
    if field == 0.0:
        pkg.hotrg_set_parity(g.ctx, [int(v) for x in par for v in x])
    n = pkg.shard_sizes(g.ctx, axis, chi)[0]
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    pkg.hotrg_shard_env(g.ctx, axis, chi, 0, 1, out=out)
    got = out.cpu().numpy().reshape(2, 4, chi * chi, chi * chi)
    to = [(axis + q) % 3 for q in range(3)]
    t = np.asarray(pkg.hotrg_tensor(g.ctx))   # as the context holds it: divided by its own trace
    ts = torch.tensor(t, device="cuda").permute([2 * v for v in to] + [2 * v + 1 for v in to])
    for j in (1, 2):
        for kind, (f, c) in enumerate(((j, 3), (j, 0), (3 + j, 3), (3 + j, 0))):
            x = ts.permute([f, c] + [q for q in range(6) if q not in (f, c)]).reshape(chi * chi, -1)
            # the reference in pieces of 32 along K, summed in pairs (s, r) without loss: a plain FP64 sum
            # of 14,641 like-signed terms has an error of its own
            s = torch.zeros(chi * chi, chi * chi, dtype=torch.float64, device="cuda")
            r = torch.zeros_like(s)
            for y in x.split(32, 1):
                p = y @ y.T
                u = s + p
                z = u - s
                r += (s - (u - z)) + (p - z)
                s = u
            ref, scale = (s + r).cpu().numpy(), (x.abs() @ x.abs().T).cpu().numpy()
            # what is left: the reference's rounding within pieces, ours once a split and in their sum
            assert np.max(np.abs(got[j - 1, kind] - ref) / scale.max()) <= 1e-14
            assert np.all(np.abs(got[j - 1, kind] - ref) <= 2.0 ** -44 * scale + 1e-300)
            assert np.array_equal(got[j - 1, kind], got[j - 1, kind].T)
    g.close()
