"""The two tile widths of the CTA-pair GEMM (128 and 256 columns): exact products on both sides of the
choice, with partial tiles."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(256, 128, 64), (300, 129, 192), (1001, 1500, 128), (257, 127, 64),
                                   (2048, 2432, 64), (2048, 2433, 128)])
def test_pair_tiles_are_exact(m, n, k):
    import paper_2110_03607_gb300 as pkg

    rng = np.random.default_rng(m + n + k)
    # small integers times a power of two: exact in every piece format, every partial sum below 2^24
    a, b = [rng.integers(-8, 9, size=(r, k)).astype(np.float64) * 0.25 for r in (m, n)]
    for mode in (pkg.PREC_BF16X3, pkg.PREC_BF16X6, pkg.PREC_TF32, pkg.PREC_TF32X3):
        np.testing.assert_array_equal(pkg.hotrg_gemm_nt(mode, a, b), a @ b.T)
