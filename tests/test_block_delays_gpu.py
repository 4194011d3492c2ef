"""The delays a boundary's warp hands from one block of K steps to the next.

For even K the effective delays of step n + K go into the buffer that holds those of step n, which the same warp has just
read: the read must come first on every boundary.  A field of noise read at a delayed level differs at order one from the
same field read at another, so one wrong delay at one boundary stands far above the bar (1e-13 of the norm, as for blocks
against single steps elsewhere; here per cell, of the largest value)."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("k", [2, 4])
def test_every_boundary_takes_its_own_delays(k):
    from paper_1702_00496_gb300 import Solver, at_set_fusion
    spec = W.wl_1d(72 * 6000, 6000, 2, 8, 0, 801, (1, 2), scheme=W.ASYNC_STD)[0]
    u0 = np.random.default_rng(801).standard_normal(72 * 6000)
    runs = []
    for length in (1, k):
        s = Solver(spec, log_steps=50)
        assert at_set_fusion(s.h, length) == length
        s.reset(torch.as_tensor(u0, device="cuda"))
        s.step(50)
        s.sync()
        runs.append((s.field().clone(), s.delays().clone()))
        s.close()
    (u1, d1), (uk, dk) = runs
    assert torch.equal(d1, dk)
    assert float((u1 - uk).abs().max()) <= 1e-13 * float(u1.abs().max())
