"""The eigen-solver and the selection through a step, against LAPACK on the same environments:
orders around the Jacobi limit, the leaf and tile edges, the largest order, unequal legs in one
batch, environments with degenerate, rank-deficient and exchange-symmetric structure."""

import numpy as np
import pytest

from seeded_inputs import gaussian_tensor, reflection_symmetric_tensor

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


def _falling(t, rate=0.35):
    """The tensor with every leg falling off, as a coarse-grained one does."""
    for k in range(t.ndim):
        f = np.exp(-rate * np.arange(t.shape[k]))
        t = t * f.reshape([-1 if q == k else 1 for q in range(t.ndim)])
    return t


def _product(chis, seed):
    """A tensor product of two equal tensors: every environment is a Kronecker square."""
    h = [int(round(c ** 0.5)) for c in chis]
    g = _falling(reflection_symmetric_tensor(h, seed))
    t = np.multiply.outer(g, g)
    n = g.ndim
    t = t.transpose([v for k in range(n) for v in (k, n + k)])
    return t.reshape([c for c in chis for _ in range(2)])


CASES = {
    "jacobi_limit": ((4, 4, 4), 6, "gauss"),        # n = 16
    "above_jacobi": ((3, 5, 5), 5, "gauss"),        # n = 25, two leaves
    "unequal_legs": ((3, 2, 9), 7, "gauss"),        # n = 4 and 81 in one batch
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
    elif kind == "reflect":
        t = _falling(reflection_symmetric_tensor(chis, 3))
    else:
        t = gaussian_tensor(chis, 7)
        if kind == "lowrank":
            t = np.einsum("ab,cd->abcd", *(gaussian_tensor([c], 8 + c) for c in chis)) + 0.1 * _falling(t, 2.0)
        elif kind == "falling":
            t = _falling(t)
    tr = np.einsum("".join(2 * chr(97 + k) for k in range(len(chis))) + "->", t)
    t = t * np.sign(tr)
    t = t / abs(tr)
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
                lam = pkg.hotrg_spectrum(ctx, leg, side)
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
