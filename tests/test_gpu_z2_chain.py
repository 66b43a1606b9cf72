"""The chain stages of the Z2 form that leave out the zero terms (d >= 3) against the dense form: odd and
even class sizes, a leg with one parity only, neighbours of a K list with different hat indices, new
bonds of 4 to 32."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2110_03607_gb300 as p

    p.load()
    return p


def _tensor(chis, parities, seed):
    """sum_c prod_k f_k[c, x_k] f'_k[c, x_k'] on even total parity, falling off along every leg."""
    rng = np.random.default_rng(seed)
    t = np.ones((60, 1))
    par = np.zeros(1, dtype=int)
    for c, p in zip(chis, parities):
        fall = np.exp(-0.2 * np.arange(c))
        f = rng.standard_normal((60, c)) * fall
        g = f + 0.3 * rng.standard_normal((60, c)) * fall
        t = (t[:, :, None, None] * f[:, None, :, None] * g[:, None, None, :]).reshape(60, -1)
        par = (par[:, None, None] ^ p[None, :, None] ^ p[None, None, :]).reshape(-1)
    t = np.where(par == 0, t.sum(0), 0.0).reshape([c for c in chis for _ in range(2)])
    return t / np.einsum("".join(2 * chr(97 + k) for k in range(len(chis))) + "->", t)


CASES = {
    "odd_classes": ((5, 6, 7), (2, 3, 3), 0, 7),
    "fours": ((4, 8, 8), (2, 4, 4), 0, 16),
    "one_parity": ((3, 4, 6), (1, 2, 0), 0, 6),
    "unbalanced": ((2, 8, 9), (1, 1, 8), 0, 9),
    "wide": ((2, 6, 7), (1, 3, 2), 0, 32),
    "new_24": ((2, 5, 9), (1, 2, 4), 0, 24),
    "axis_last": ((6, 5, 4), (3, 2, 2), 2, 6),
    "four_dims": ((2, 3, 4, 3), (1, 1, 2, 1), 1, 5),
    "four_dims_even": ((4, 2, 4, 4), (2, 1, 2, 2), 3, 8),
}


# against the dense form: FP32 sums in another order (2^-24 each, the chains' and the product's, in the
# 2-norm), and what the pieces leave out of an element (2^-16 with two BF16 pieces, 2^-22 with two of TF32)
@pytest.mark.parametrize("form,tol", [("PREC_BF16X6", 1e-6), ("PREC_TF32X3", 2e-6), ("PREC_BF16X3", 6e-5)])
@pytest.mark.parametrize("case", sorted(CASES))
def test_blocks_match_the_dense_form(pkg, case, form, tol):
    chis, odd, axis, chi = CASES[case]
    rng = np.random.default_rng(len(case))
    par = [rng.permutation(np.arange(c) < n).astype(int) for c, n in zip(chis, odd)]
    t = _tensor(chis, par, 17)
    out = []
    for blocks in (True, False):
        g = pkg.Hotrg(len(chis), 0.25, 0.0, precision=getattr(pkg, form), tensor=t, chis=chis, fp64_below=0.0,
                      z2=blocks)
        try:
            if blocks:
                pkg.hotrg_set_parity(g.ctx, [int(v) for p in par for v in p])
            g.step(axis, chi)
            if blocks:
                assert pkg.hotrg_bottleneck_flops(g.ctx)[2]
            out.append(np.asarray(pkg.hotrg_tensor(g.ctx)))
        finally:
            g.close()
    assert np.linalg.norm(out[0] - out[1]) <= tol * np.linalg.norm(out[1])
