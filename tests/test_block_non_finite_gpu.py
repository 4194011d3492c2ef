"""Infinities and NaN in blocks of K steps: tiles that hold one go through the chains of their cells, and after five steps (a
block of four and a step, or the like) the same cells are finite as in the oracle, with the same values."""
import os

import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

PROBLEMS = [
    ("o2", 4, lambda: W.wl_1d(72 * 24, 24, 2, 3, 0, 951, (1, 2))[0]),
    ("o4", 4, lambda: W.wl_1d(3 * 2072, 3, 4, 4, 0, 952, (1, 2))[0]),
    ("o4_k3", 3, lambda: W.wl_1d(128 * 16, 16, 4, 4, 0, 953, (1, 2))[0]),
    ("o6", 4, lambda: W.wl_1d(2 * 2500, 2, 6, 3, 0, 954, (1, 2), r_alpha=0.02)[0]),
    ("o4_unsplit", 4, lambda: W.wl_1d(4100, 1, 4, 4, 0, 955, (1, 2))[0]),
    ("o4_ragged", 4, lambda: W.wl_1d(205 * 5, 5, 4, 4, 0, 956, (1, 2))[0]),
    ("o4_wide_tiles", 4, lambda: W.wl_1d(655360, 4, 4, 4, 0, 957, (1, 2))[0]),
]


@pytest.mark.parametrize("steps", [4, 5, 9])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("name,K,make", PROBLEMS, ids=[p[0] for p in PROBLEMS])
def test_non_finite_values_in_blocks(name, K, make, value, steps):
    from paper_1702_00496_gb300 import Solver, at_set_fusion
    spec = make()
    cfg = oracle.Config(spec)
    u0 = oracle.initial(cfg) + 3.0
    u0[[5, u0.size // 2 + 333]] = value
    s = Solver(spec)
    assert at_set_fusion(s.h, 4) == K
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.step(steps)
    s.sync()
    u = s.field().cpu().numpy().copy()
    s.close()
    ref, _, _ = oracle.run(cfg, steps, threads=os.cpu_count() or 1, u0=u0)
    fine = np.isfinite(ref)  # (inf becomes NaN a step earlier in the oracle, which multiplies zero weights too)
    assert np.array_equal(fine, np.isfinite(u))
    assert 0 < (~fine).sum() < 4 * (spec["order"] // 2) * steps + 4 + 4 * spec["order"]
    assert np.abs(u[fine] - ref[fine]).max() <= 1e-12 * np.abs(ref[fine]).max()
