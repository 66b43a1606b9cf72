"""Batched steps whose chain stages need different amounts of shared memory from one kernel: the limit
belongs to the kernel, so a thread that sets its own size could take it from another's launch."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_threads_with_different_shared_memory_sizes():
    import torch

    import paper_2110_03607_gb300 as pkg

    rng = np.random.default_rng(3)
    chis, new = (2, 2, 20), [20, 19, 18, 17] * 2
    f = [rng.standard_normal((40, c)) * np.exp(-0.3 * np.arange(c)) for c in chis]
    t = np.einsum("zaA,zbB,zcC->aAbBcC", *[x[:, :, None] * x[:, None, :] for x in f])
    streams = [torch.cuda.Stream() for _ in new]
    runs = [pkg.Hotrg(3, 0.25, 0.01, precision=pkg.PREC_BF16X6, tensor=t, chis=chis, fp64_below=0.0) for _ in new]
    try:
        for g, s in zip(runs, streams):
            pkg.hotrg_set_stream(g.ctx, s.cuda_stream)
        for _ in range(40):
            for g in runs:
                pkg.hotrg_set_tensor(g.ctx, chis, t)
            assert pkg.hotrg_step_batch([g.ctx for g in runs], [0] * len(new), new, len(new)) == [0] * len(new)
    finally:
        for g in runs:
            g.close()
