"""The eigen-solver and the selection through a step, against LAPACK on the same environments:
orders around the Jacobi limit, the leaf and tile edges, the largest order, unequal legs in one
batch, environments with degenerate, rank-deficient and exchange-symmetric structure."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2110_03607_gb300 as p

    p.load()
    return p


def _environment(t, axis, leg, prime):
    """A^(leg) (or A'^(leg)) with rows hat + check chi, from its definition (Sec. 3.2)."""
    d = t.ndim // 2
    chi_j, chi_c = t.shape[2 * leg], t.shape[2 * axis]
    s = []
    for cur in (2 * axis + 1, 2 * axis):
        free = 2 * leg + (1 if prime else 0)
        x = np.moveaxis(t, (free, cur), (0, 1)).reshape(chi_j * chi_c, -1)
        s.append((x @ x.T).reshape(chi_j, chi_c, chi_j, chi_c))
    a = np.einsum("frgs,hrks->hfkg", s[0], s[1], optimize=True)
    return a.reshape(chi_j * chi_j, chi_j * chi_j)


def _sum_of_products(chis, seed, terms, rate, skew):
    """sum_c prod_k f_k[c, x_k] f'_k[c, x_k']: the form of a block of spins, whose traces are positive
    (f' = f + skew x noise; skew = 0: symmetric under the reflections)."""
    rng = np.random.default_rng(seed)
    t = np.ones((terms, 1))
    for c in chis:
        fall = np.exp(-rate * np.arange(c))
        f = rng.standard_normal((terms, c)) * fall
        g = f + skew * rng.standard_normal((terms, c)) * fall
        t = (t[:, :, None, None] * f[:, None, :, None] * g[:, None, None, :]).reshape(terms, -1)
    return t.sum(0).reshape([c for c in chis for _ in range(2)])


def _product(chis, seed):
    """A tensor product of two equal tensors: every environment is a Kronecker square."""
    g = _sum_of_products([int(round(c ** 0.5)) for c in chis], seed, 12, 0.35, 0.0)
    n = g.ndim
    t = np.multiply.outer(g, g).transpose([v for k in range(n) for v in (k, n + k)])
    return t.reshape([c for c in chis for _ in range(2)])


CASES = {
    "jacobi_limit": ((4, 4, 4), 6, "flat"),         # n = 16
    "above_jacobi": ((3, 5, 5), 5, "flat"),        # n = 25, two leaves
    "unequal_legs": ((3, 2, 9), 7, "flat"),        # n = 4 and 81 in one batch
    "tile_edge": ((2, 6, 8), 8, "falling"),         # n = 36 and 64
    "odd": ((7, 13), 13, "falling"),                # n = 169
    "cluster16": ((3, 15), 15, "falling"),          # n = 225
    "large": ((2, 24), 24, "falling"),              # n = 576
    "beyond_shared": ((2, 28), 28, "falling"),      # n = 784: rows in global memory
    "largest": ((2, 32), 32, "falling"),            # n = 1024
    "exchange": ((6, 6, 6), 6, "reflect"),          # even and odd vectors
    "degenerate": ((4, 9), 9, "product"),
    "rank_deficient": ((2, 12), 12, "lowrank"),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_spectra_and_isometries_match_lapack(pkg, case):
    chis, chi, kind = CASES[case]
    if kind == "product":
        t = _product(chis, 5)
    else:
        terms, rate, skew = {"flat": (200, 0.0, 0.3), "falling": (200, 0.35, 0.3), "reflect": (200, 0.35, 0.0),
                             "lowrank": (3, 0.35, 0.3)}[kind]
        t = _sum_of_products(chis, 7, terms, rate, skew)
    t = t / np.einsum("".join(2 * chr(97 + k) for k in range(len(chis))) + "->", t)
    ctx = pkg.hotrg_init_tensor(len(chis), chis, t, 0.3)
    try:
        pkg.hotrg_set_precision(ctx, pkg.PREC_FP64)
        pkg.hotrg_step(ctx, 0, chi)
        for leg in range(1, len(chis)):
            u, prime = pkg.hotrg_isometry(ctx, leg)
            # both sides form A from FP64 sums over K elements (error of order sqrt(K) eps in A) and
            # decompose it backward stably (a few n eps): 1e-12 of lambda_1 covers n = 1024
            for side in (0, 1):
                want = np.linalg.eigvalsh(_environment(t, 0, leg, side))[::-1]
                # values in a group of near-ties (1e-12 lambda_1 apart) stand in the pivots' order
                lam = np.sort(pkg.hotrg_spectrum(ctx, leg, side))[::-1]
                np.testing.assert_allclose(lam, np.abs(want), rtol=0, atol=1e-12 * want[0])
            a = _environment(t, 0, leg, prime)
            lam = pkg.hotrg_spectrum(ctx, leg, int(prime))
            np.testing.assert_allclose(u.T @ u, np.eye(u.shape[1]), rtol=0, atol=1e-12)
            np.testing.assert_allclose(a @ u, u * lam[: u.shape[1]], rtol=0, atol=1e-12 * lam[0])
            piv = np.argmax(np.abs(u) >= (1 - 1e-6) * np.abs(u).max(0), axis=0)
            assert (u[piv, np.arange(u.shape[1])] > 0).all()
            assert pkg.hotrg_jacobi_sweeps(ctx, leg) >= 1
    finally:
        pkg.hotrg_free(ctx)
