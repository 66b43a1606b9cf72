"""Slices that share a pass of the contraction: the memory cap of hotrg_set_slice_budget, passes with a
remainder, and the same bits however the slices are grouped (by the cap, or over the ranks of a shard)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2110_03607_gb300 as p

    p.load()
    return p


def _tensor(chis, seed, odd=None):
    """A sum of products falling off along every leg; odd: entries of odd total parity are zero (the
    first half of each leg's indices is even)."""
    rng = np.random.default_rng(seed)
    t = np.ones((50, 1))
    par = np.zeros(1, dtype=int)
    for c in chis:
        f = rng.standard_normal((50, c)) * np.exp(-0.25 * np.arange(c))
        g = f + 0.3 * rng.standard_normal((50, c)) * np.exp(-0.25 * np.arange(c))
        t = (t[:, :, None, None] * f[:, None, :, None] * g[:, None, None, :]).reshape(50, -1)
        p = (np.arange(c) >= (c + 1) // 2).astype(int)
        par = (par[:, None, None] ^ p[None, :, None] ^ p[None, None, :]).reshape(-1)
    t = t.sum(0)
    if odd:
        t = np.where(par == 0, t, 0.0)
    t = t.reshape([c for c in chis for _ in range(2)])
    return t / np.einsum("".join(2 * chr(97 + k) for k in range(len(chis))) + "->", t)


def _context(pkg, chis, form, z2):
    g = pkg.Hotrg(len(chis), 0.25, 0.0 if z2 else 0.01, precision=getattr(pkg, form), tensor=_tensor(chis, 5, z2),
                  chis=chis, fp64_below=0.0)
    if z2:
        pkg.hotrg_set_parity(g.ctx, [int(i >= (c + 1) // 2) for c in chis for i in range(c)])
    return g


def test_operands_of_shared_passes_fit_the_cap(pkg):
    # a slice of this FP64 step has 38 MB of operands: several in a pass fit neither cap
    chis, held = (8, 8, 8), {}
    for cap in (1.0, 40e6, 90e6):
        g = _context(pkg, chis, "PREC_FP64", False)
        try:
            pkg.hotrg_set_slice_budget(g.ctx, cap)
            g.step(0, 8)
            held[cap] = pkg.hotrg_device_bytes(g.ctx)
        finally:
            g.close()
    # with one byte a pass holds the least it can: one n'_1 value of a slice
    for cap in (40e6, 90e6):
        assert held[cap] - held[1.0] <= cap


@pytest.mark.parametrize("chis,axis,chi,form,z2", [((7, 4, 5), 0, 5, "PREC_FP64", False),
                                                   ((7, 6, 6), 0, 6, "PREC_FP64", True),
                                                   ((11, 11), 1, 11, "PREC_FP64", False),
                                                   ((5, 4, 6), 2, 6, "PREC_BF16X6", False),
                                                   ((7, 4, 5), 0, 5, "PREC_BF16X3", True),
                                                   ((9, 8), 0, 8, "PREC_TF32X3", True)])
def test_same_bits_however_slices_are_grouped(pkg, chis, axis, chi, form, z2):
    def step(cap=None, ranks=None):
        g = _context(pkg, chis, form, z2)
        try:
            if cap is not None:
                pkg.hotrg_set_slice_budget(g.ctx, cap)
            if ranks is None:
                g.step(axis, chi)
            else:
                pkg.hotrg_shard_isometries(g.ctx, axis, chi, pkg.hotrg_shard_env(g.ctx, axis, chi, 0, 1))
                cuts = [chis[axis] * r // ranks for r in range(ranks + 1)]
                parts = [pkg.hotrg_shard_contract(g.ctx, axis, chi, lo, hi) for lo, hi in zip(cuts, cuts[1:])]
                pkg.hotrg_shard_finish(g.ctx, axis, chi, np.concatenate(parts))
            return np.asarray(pkg.hotrg_tensor(g.ctx)), g.free_energy()[0]
        finally:
            g.close()

    want = step()
    # caps from less than a unit to all slices: the passes in between hold 2, 3, .. slices and a remainder
    got = [step(cap=c) for c in np.geomspace(2e4, 4e7, 12)] + [step(ranks=2), step(ranks=chis[axis])]
    for t, lnz in got:
        np.testing.assert_array_equal(t, want[0])
        assert lnz == want[1]
