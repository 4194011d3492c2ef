"""The step kernels' fixed-point sums on fields that take each of their routes, against the FP64 oracle.

Smooth fields keep every value of a window near its largest (cross terms in FP32 in the blocks), noise does not (integer
cross terms), fields that fall by many binades within a few cells, exact zeros, infinities, NaN and values at the ends of
the exponent range go through the FP64 chain.  Bars: delays bit-exact, elementwise within 1e-12 of the max norm as in
the other parity tests; where the field falls steeply, elementwise within 256 ulp (5.7e-14) of the largest value in the
cell's domain of dependence (2 h + 1 roundings per step on each side, under 12 steps); non-finite cells in the same places."""
import os

import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

THREADS = os.cpu_count() or 1
STEPS = 11

PROBLEMS = [
    ("block_o2", lambda: W.wl_1d(72 * 24, 24, 2, 3, 0, 601, (1, 2))[0]),
    ("block_o4_tile_edge", lambda: W.wl_1d(3 * 2072, 3, 4, 4, 0, 602, (1, 2))[0]),
    ("block_o4_unsplit_small", lambda: W.wl_1d(64, 1, 4, 4, 0, 603, (1, 2))[0]),
    ("block_o6", lambda: W.wl_1d(2 * 2500, 2, 6, 3, 0, 604, (1, 2), r_alpha=0.02)[0]),
    ("single_o2", lambda: W.wl_1d(16 * 20, 20, 2, 3, 0, 605, (1, 2))[0]),
    ("single_o4", lambda: W.wl_1d(64 * 8, 8, 4, 3, 0, 606, (1, 2))[0]),
    ("single_o6", lambda: W.wl_1d(8 * 32, 32, 6, 3, 0, 607, (1, 2), r_alpha=0.01)[0]),
    ("ab2_o4", lambda: W.wl_1d(64 * 20, 20, 4, 3, 0, 608, (1, 2), r_alpha=0.02, tsteps=2)[0]),
    ("ab3_o6", lambda: W.wl_1d(64 * 20, 20, 6, 3, 0, 609, (1, 2), r_alpha=0.01, tsteps=3)[0]),
    ("burgers_ab2_o4", lambda: dict(W.wl_1d(64 * 20, 20, 4, 3, 0, 610, (1, 2), c=0.0, r_alpha=0.02, tsteps=2)[0], burgers=1)),
    ("burgers_euler_o2", lambda: dict(W.wl_1d(64 * 20, 20, 2, 3, 0, 611, (1, 2), c=0.0, r_alpha=0.02)[0], burgers=1)),
    # large shapes without aligned groups: a last group of 1, 2 or 3 points per PE, narrow PEs, one PE
    ("ragged_o2", lambda: W.wl_1d(197 * 1001, 1001, 2, 3, 0, 631, (1, 2))[0]),
    ("ragged_o4", lambda: W.wl_1d(250 * 800, 800, 4, 4, 0, 632, (1, 2))[0]),
    ("ragged_o4_narrow", lambda: W.wl_1d(5 * 40000, 40000, 4, 3, 0, 633, (1, 2))[0]),
    # blocks over PEs that are no multiple of four wide: the narrowest ones that take K = 4, a ring too short for K = 4,
    # tiles that end one cell into the next, a domain of odd length that wraps
    ("ragged_o2_blocks", lambda: W.wl_1d(73 * 2700, 2700, 2, 3, 0, 637, (1, 2))[0]),
    ("ragged_o4_blocks", lambda: W.wl_1d(145 * 1357, 1357, 4, 2, 0, 638, (1, 2), scheme=W.ASYNC_STD)[0]),
    ("ragged_o2_blocks_short_ring", lambda: W.wl_1d(257 * 801, 801, 2, 1, 0, 639, (1, 2))[0]),
    ("ragged_o6_blocks", lambda: W.wl_1d(305 * 651, 651, 6, 3, 0, 640, (1, 2), r_alpha=0.01)[0]),
    # and small ones, from one point more than what one launch takes point by point
    ("ragged_o4_blocks_smallest", lambda: W.wl_1d(205 * 5, 5, 4, 4, 0, 652, (1, 2))[0]),
    ("ragged_o2_blocks_unsplit", lambda: W.wl_1d(1027, 1, 2, 3, 0, 653, (1, 2))[0]),
    ("ragged_o6_blocks_odd", lambda: W.wl_1d(333 * 31, 31, 6, 3, 0, 654, (1, 2), r_alpha=0.01, scheme=W.ASYNC_STD)[0]),
    ("ragged_o6_ab3", lambda: W.wl_1d(19 * 10500, 10500, 6, 3, 0, 634, (1, 2), r_alpha=0.01, tsteps=3)[0]),
    ("ragged_o4_unsplit", lambda: W.wl_1d(200001, 1, 4, 3, 0, 635, (1, 2))[0]),
    ("ragged_burgers_ab2_o4", lambda: dict(W.wl_1d(131 * 1600, 1600, 4, 3, 0, 636, (1, 2), c=0.0, r_alpha=0.02, tsteps=2)[0], burgers=1)),
    ("3d_o2", lambda: W.wl_3d([24, 20, 18], [2, 2, 3], 2, 3, 0, 612, c=(0.3, 0.2, 0.1))[0]),
    ("3d_o4", lambda: W.wl_3d([72, 18, 20], [2, 1, 2], 4, 3, 0, 613, c=(0.3, 0.2, 0.1))[0]),
    ("3d_o4_ragged", lambda: W.wl_3d([39, 22, 14], [3, 2, 1], 4, 3, 0, 614, c=(0.3, 0.2, 0.1))[0]),
    ("3d_o6", lambda: W.wl_3d([40, 16, 24], [1, 2, 2], 6, 3, 0, 615, c=(0.3, 0.2, 0.1), dt=0.01 * W.dx_of(40) ** 2 / 0.05)[0]),
    ("3d_o4_ab2", lambda: W.wl_3d([24, 20, 16], [2, 2, 2], 4, 3, 0, 616, c=(0.3, 0.2, 0.1), tsteps=2)[0]),
    # large enough for the marched tiles: PEs of odd widths (partial tiles and groups, 8-byte stores), an unsplit axis
    # (the tile wraps around the domain), aligned ones (16-byte stores), chunks of a PE along z
    ("tiles_o2_ragged", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 2, 3, 0, 617, c=(0.3, 0.2, 0.1))[0]),
    ("tiles_o4_ragged", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 4, 3, 0, 618, c=(0.3, 0.2, 0.1))[0]),
    ("tiles_o6_ragged", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 6, 3, 0, 619, c=(0.3, 0.2, 0.1), dt=0.01 * W.dx_of(150) ** 2 / 0.05)[0]),
    ("tiles_o4_wrap", lambda: W.wl_3d([132, 128, 130], [1, 2, 1], 4, 4, 0, 620, c=(0.3, 0.2, 0.1), scheme=W.ASYNC_STD)[0]),
    ("tiles_o4_ab2", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 4, 3, 0, 621, c=(0.3, 0.2, 0.1), dt=0.02 * W.dx_of(150) ** 2 / 0.05, tsteps=2)[0]),
    ("tiles_o4_ab3_aligned", lambda: W.wl_3d([128, 128, 128], [2, 2, 2], 4, 3, 0, 622, c=(0.3, 0.2, 0.1), dt=0.01 * W.dx_of(128) ** 2 / 0.05, tsteps=3)[0]),
]


def _field(spec, kind):
    rng = np.random.default_rng([spec["seed"], len(kind)])
    u = oracle.initial(oracle.Config(spec)) + 3.0
    if kind == "smooth":
        return u
    noise = rng.standard_normal(u.shape)
    if kind == "noise":
        return noise
    if kind == "steep":  # falls by more than a binade from cell to cell along x, and is zero in places
        x = np.arange(u.shape[-1])
        v = u * np.exp(-((x % 64) - 20.0) ** 2 / 30.0)
        return np.where(x % 64 > 50, 0.0, v)
    if kind == "spikes":
        return np.where(rng.random(u.shape) < 0.02, 1e6 * noise, 1e-6 * noise)
    if kind == "small":
        return noise * 1e-250
    return {"tiny": noise * 1e-290, "large": noise * 1e280}[kind]


def _gpu(spec, u0, steps, single=False):
    from paper_1702_00496_gb300 import Solver, at_set_fusion
    s = Solver(spec, log_steps=steps)
    if single:
        at_set_fusion(s.h, 1)
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.step(steps)
    s.sync()
    u, d = s.field().cpu().numpy().copy(), s.delays().cpu().numpy().copy()
    s.close()
    return u, d


def _local_max(a, reach):
    """Largest |a| within `reach` cells along every axis (periodic)."""
    m = np.abs(a)
    for ax in range(a.ndim):
        if a.shape[ax] == 1:
            continue
        m = np.max([np.roll(m, s, ax) for s in range(-reach, reach + 1)], axis=0)
    return m


@pytest.mark.parametrize("kind", ["smooth", "noise", "steep", "spikes", "small", "tiny", "large"])
@pytest.mark.parametrize("name,make", PROBLEMS, ids=[p[0] for p in PROBLEMS])
def test_every_route_matches_the_oracle(name, make, kind):
    spec = make()
    u0 = _field(spec, kind)
    if spec.get("burgers") and kind in ("large", "spikes"):
        u0 = u0 * 1e-279 if kind == "large" else u0 * 1e-6  # u u_x stays finite and the step stable
    u, d = _gpu(spec, u0, STEPS)
    ref, dref, _ = oracle.run(oracle.Config(spec), STEPS, threads=THREADS, u0=u0)
    assert np.array_equal(d, dref)
    assert np.abs(u - ref).max() <= 1e-12 * np.abs(ref).max()
    if kind in ("steep", "spikes") and not spec.get("burgers"):
        # each cell against the values it can depend on (levels 0 .. STEPS of its neighbourhood: the initial field's)
        h = spec["order"] // 2
        local = np.maximum(_local_max(u0, h * STEPS), np.abs(ref))
        assert (np.abs(u - ref) <= 256 * 2.0 ** -52 * local).all()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("name,make", [p for p in PROBLEMS if not p[0].startswith(("block", "burgers"))],
                         ids=[p[0] for p in PROBLEMS if not p[0].startswith(("block", "burgers"))])
def test_non_finite_values_spread_as_in_the_oracle(name, make, value):
    spec = make()
    u0 = _field(spec, "smooth").copy()
    flat = u0.reshape(-1)
    flat[[5, flat.size // 2 + 3]] = value
    u, _ = _gpu(spec, u0, 3)
    ref, _, _ = oracle.run(oracle.Config(spec), 3, threads=THREADS, u0=u0)
    # the oracle multiplies each derivative's zero weights too (inf becomes NaN a cell or a step earlier there), so the
    # cells are compared by being finite or not
    fine = np.isfinite(ref)
    assert np.array_equal(fine, np.isfinite(u))
    assert np.abs(u[fine] - ref[fine]).max() <= 1e-12 * np.abs(ref[fine]).max()


SMALL = [
    ("n16_o2", lambda: W.wl_1d(16, 2, 2, 3, 0, 641, (1, 2))[0]),
    ("n256_o2_log", lambda: W.wl_1d(256, 8, 2, 3, 0, 642, (1, 2))[0]),
    ("n2048_o4_most_sides", lambda: W.wl_1d(2048, 512, 4, 4, 0, 643, (1, 2))[0]),
    ("n2048_o6_ab3", lambda: W.wl_1d(2048, 64, 6, 3, 0, 644, (1, 2), r_alpha=0.01, tsteps=3)[0]),
    ("n1288_o4_ab2_unsplit", lambda: W.wl_1d(1288, 1, 4, 3, 0, 645, (1, 2), r_alpha=0.02, tsteps=2)[0]),
    ("n640_o4_burgers", lambda: dict(W.wl_1d(640, 10, 4, 3, 0, 646, (1, 2), c=0.0, r_alpha=0.02, tsteps=2)[0], burgers=1)),
    ("n250_o4_points", lambda: W.wl_1d(250, 5, 4, 3, 0, 648, (1, 2))[0]),
    ("n1001_o6_ab3_points", lambda: W.wl_1d(1001, 7, 6, 3, 0, 649, (1, 2), r_alpha=0.01, tsteps=3)[0]),
    ("n102_burgers_points", lambda: dict(W.wl_1d(102, 6, 2, 3, 0, 650, (1, 2), c=0.0, r_alpha=0.02)[0], burgers=1)),
    ("n63_space_points", lambda: W.wl_1d(63, 9, 2, 3, 0, 651, (1, 2), scheme=W.AT_SPACE2)[0]),
    ("n640_space", lambda: W.wl_1d(640, 10, 2, 3, 0, 647, (1, 2), scheme=W.AT_SPACE2)[0]),
]


@pytest.mark.parametrize("callers_field", [False, True])
@pytest.mark.parametrize("name,make", SMALL, ids=[s[0] for s in SMALL])
def test_small_problems_in_one_launch_are_bitwise_single_steps(name, make, callers_field):
    """A call of several steps of a small problem runs in one launch, a call of one step is a launch of its own: the same
    bits and delays for any split of the steps, also where the multistep start-up falls into the launch."""
    from paper_1702_00496_gb300 import Solver, at_set_fusion
    spec = make()
    runs = []
    for split in ([1] * 37, [37], [2, 1, 34]):
        s = Solver(spec, log_steps=37)
        at_set_fusion(s.h, 1)
        if callers_field:
            s.reset(torch.as_tensor(_field(spec, "smooth"), device="cuda"))
        for m in split:
            s.step(m)
        s.sync()
        runs.append((s.field().clone(), s.delays().clone()))
        s.close()
    for u, d in runs[1:]:
        assert torch.equal(u, runs[0][0]) and torch.equal(d, runs[0][1])


ADJOINT_TILES = [
    ("o4_ragged", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 4, 3, 0, 661, c=(0.3, 0.2, 0.1))[0], False),
    ("o2_aligned_unsplit_y", lambda: W.wl_3d([128, 128, 128], [2, 1, 2], 2, 4, 0, 662, c=(0.3, 0.2, 0.1))[0], False),
    ("o6_std", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 6, 3, 0, 663, c=(0.3, 0.2, 0.1), scheme=W.ASYNC_STD,
                               dt=0.01 * W.dx_of(150) ** 2 / 0.05)[0], False),
    ("o4_ab2", lambda: W.wl_3d([128, 128, 128], [2, 2, 2], 4, 3, 0, 664, c=(0.3, 0.2, 0.1), tsteps=2,
                               dt=0.02 * W.dx_of(128) ** 2 / 0.05)[0], True),
]


@pytest.mark.parametrize("name,make,callers_field", ADJOINT_TILES, ids=[c[0] for c in ADJOINT_TILES])
def test_gradient_on_tiles_matches_the_cpu_adjoint(name, make, callers_field):
    """The transposed step over the marched tiles (its level-n part, the faces' older levels, the alpha sum) against the
    oracle's literal adjoint, with the bars of the other adjoint tests; and the initial field's gradient alone and other
    checkpoint intervals give the same bits."""
    from paper_1702_00496_gb300 import Solver
    spec = make()
    steps = 7
    cfg = oracle.Config(spec)
    u0 = oracle.initial(cfg) + (0.01 if callers_field else 0.0)
    rng = np.random.default_rng(7)
    target = 0.5 * u0 + 0.1 * rng.standard_normal(cfg.shape)
    grads = []
    for every, want_alpha in ((0, True), (steps, True), (2, False)):
        s = Solver(spec)
        s.reset(torch.as_tensor(u0, device="cuda"))
        s.adjoint_forward(steps, every)
        lam = s.field() - torch.as_tensor(target, device="cuda")
        g, ga = s.adjoint_backward(lam.clone(), want_alpha)
        grads.append((g.cpu().numpy(), ga))
        s.close()
    _, go, gao = oracle.adjoint(cfg, steps, target, u0=u0)
    g, ga = grads[0]
    assert np.linalg.norm(g - go) / np.linalg.norm(go) <= 1e-12
    assert ga == pytest.approx(gao, rel=1e-10)
    assert np.array_equal(grads[1][0], g) and grads[1][1] == ga and np.array_equal(grads[2][0], g)


@pytest.mark.parametrize("n,count", [(64, 153), (64, 640), (1028, 640), (2052, 153)])
def test_default_ensemble_shapes_give_the_same_members(n, count):
    """The CTA shapes that the members' number and size choose by default (256, 512, 1024 threads) against one of 1024:
    the fields bit for bit, the statistics up to the order of their sums (errors of 2^-53 per term, n terms)."""
    from paper_1702_00496_gb300 import Ensemble
    specs = [W.wl_1d(n, n // 4, 2, 3, 0, 700 + r, (1, 2))[0] for r in range(count)]
    a, b = Ensemble(specs, 9), Ensemble(specs, 9, threads=1024)
    for e in (a, b):
        e.run()
    for r in (0, 1, count // 2, count - 1):
        assert torch.equal(a.field(r), b.field(r)), r
    for x, y in zip(a.stats()[0], b.stats()[0]):
        assert x["rms"] == pytest.approx(y["rms"], rel=n * 2.0 ** -52, abs=0)
    a.close()
    b.close()
