"""The eigen-solver takes every matrix by its own order: what a leg's environment gives does not depend
on the other legs of the step."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _leg_tensor(chi_c, chi, seed):
    """Small integers with a trace of a power of two, so that environments are exact: symmetric in the leg up to a
    weak asymmetry, with nearly degenerate pairs of eigenvalues."""
    rng = np.random.default_rng(seed)
    t = rng.integers(-2, 3, (chi_c, chi_c, chi, chi))
    t = t + t.transpose(0, 1, 3, 2)
    t[0, 0, :, :] += 40 * np.eye(chi, dtype=t.dtype)
    t[0, 0, 0, 1] += 1
    tr = int(np.einsum("aabb->", t))
    t[1, 1, 0, 0] += 2 ** int(np.ceil(np.log2(tr))) - tr
    return t.astype(float)


@pytest.mark.parametrize("chi_c,chi,others", [(2, 4, (9,)), (2, 3, (5,)), (3, 4, (4, 6)), (2, 2, (4,)), (2, 3, (4, 3))])
def test_a_leg_does_not_depend_on_the_others(chi_c, chi, others):
    import paper_2110_03607_gb300 as pkg

    t = _leg_tensor(chi_c, chi, 11)
    got = []
    for extra in ((), others):
        # the other legs have one nonzero element, 1: they change no sum
        x = t
        for c in extra:
            one = np.zeros((c, c))
            one[0, 0] = 1.0
            x = np.multiply.outer(x, one)
        chis = (chi_c, chi) + extra
        g = pkg.Hotrg(len(chis), 0.3, 0.01, precision=pkg.PREC_FP64, tensor=x, chis=chis)
        try:
            g.step(0, chi)
            u, _ = pkg.hotrg_isometry(g.ctx, 1)
            got.append((u, pkg.hotrg_spectrum(g.ctx, 1, 0), pkg.hotrg_spectrum(g.ctx, 1, 1),
                        pkg.hotrg_jacobi_sweeps(g.ctx, 1)))
        finally:
            g.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
