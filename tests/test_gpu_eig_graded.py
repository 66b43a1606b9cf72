"""Kept eigenvectors of graded environments: their small angles against a reference in extended precision.

With a current bond of 1 the tensor is a matrix t and A' = G (x) G, G = t^T t.  For t = Q D, Q well conditioned and D
falling over many orders, G's entries determine its eigenvectors to a few eps / relative gap, whatever the
eigenvalues' ratio to lambda_1; a solver with a backward error of eps lambda_1 alone leaves eps lambda_1 / |lambda - mu|."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _left_vectors(w):
    """Orthogonalises the rows of w by one-sided Jacobi in extended precision: (vectors, norms), falling."""
    w = np.array(w, dtype=np.longdouble)
    n = w.shape[0]
    v = np.eye(n, dtype=np.longdouble)
    for _ in range(40):
        worst = 0.0
        for p in range(n):
            for q in range(p + 1, n):
                a, b, g = w[p] @ w[p], w[q] @ w[q], w[p] @ w[q]
                worst = max(worst, float(abs(g) / np.sqrt(a * b)))
                if g == 0:
                    continue
                z = (b - a) / (2 * g)
                t = (1 if z >= 0 else -1) / (abs(z) + np.sqrt(1 + z * z))
                c = 1 / np.sqrt(1 + t * t)
                s = c * t
                for m in (w, v):
                    m[p], m[q] = c * m[p] - s * m[q], s * m[p] + c * m[q]
        if worst < 1e-18:
            break
    norm = np.sqrt((w * w).sum(1))
    order = np.argsort(-norm)
    return v[order], norm[order]


CASES = {
    # diagonal exponents (powers of two of the singular values), kept
    "to_1e-9": ((0.0, 2.3, 5.2, 7.9, 11.6, 14.9), 24),
    "to_1e-12": ((0.0, 4.1, 8.9, 12.3, 17.8, 20.1), 19),
    "near_the_limit": ((0.0, 1.4, 11.7, 12.6, 13.9, 15.1), 20),      # angles about 2^-24 without the correction
    "long_tail": (tuple(2.07 * k + 0.17 * k * k for k in range(12)), 32),   # 144 rows, a tail of more than 96
    "above_jacobi": ((0.0, 3.3, 7.1, 11.9, 15.2), 17),               # 25 rows
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_kept_vectors_of_graded_environments(case):
    import paper_2110_03607_gb300 as pkg

    exps, keep = CASES[case]
    n = len(exps)
    rng = np.random.default_rng(n + keep)
    t = (np.eye(n) + 0.15 * rng.standard_normal((n, n))) * 2.0 ** -np.array(exps)
    t /= np.trace(t)
    vec, sing = _left_vectors(t.T)
    # eigenvalues and vectors of G (x) G: index hat + check n
    lam, ref = [], []
    for i in range(n):
        for j in range(i, n):
            x, y = np.outer(vec[j], vec[i]).ravel(), np.outer(vec[i], vec[j]).ravel()
            for sign in (1, -1) if i != j else (0,):
                lam.append(float((sing[i] * sing[j]) ** 2))
                ref.append(x if sign == 0 else (x + sign * y) / np.sqrt(np.longdouble(2)))
    order = np.argsort(-np.array(lam), kind="stable")
    lam, ref = np.array(lam)[order], np.array(ref)[order].astype(float)
    g = pkg.Hotrg(2, 0.3, 0.01, precision=pkg.PREC_FP64, tensor=t.reshape(1, 1, n, n), chis=(1, n))
    try:
        g.step(0, keep)
        u, prime = pkg.hotrg_isometry(g.ctx, 1)
        assert prime
    finally:
        g.close()
    gap = 1e300
    for i in range(keep):
        others = np.abs(lam / lam[i] - 1) > 1e-9
        if np.min(np.abs(lam[others] - lam[i])) <= 1e-12 * lam[0]:
            break   # from here on the selection orders ties by their pivots
        gap = min(gap, np.min(np.abs(lam[others] / lam[i] - 1)))
        # an even or an odd vector of its eigenvalue: what is left of it beside that one
        same = ref[~others]
        k = np.argmax(np.abs(same @ u[:, i]))
        left = u[:, i] - same[k] * (same[k] @ u[:, i])
        # G: n products an entry and the tensor's own rounding; its square; rotations stop at 4 n^2 eps; over the gap
        tol = (8 * n + 4 * n * n) * 2.0 ** -52 * 4 / gap
        assert np.linalg.norm(left) <= tol, (i, lam[i] / lam[0], np.linalg.norm(left), tol)
    assert lam[i] <= 1e-10 * lam[0]
