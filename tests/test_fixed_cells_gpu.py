"""One launch of the fixed-point step kernels, every cell against its own stencil.

A norm does not see a cell that is small beside another one; here each cell is held to the largest value of its own
stencil.  As an FMA chain a sum of n taps may be off by n roundings of 2^-53 of that value times sum |w|, in fixed point by
7 + n of them (test_fixed_ring_host.py derives it), and the weights, a few roundings each, by up to n more
(both sides may contract them differently).  The reference applies the weights in extended precision.  The domains are
unsplit, so every point takes the central taps; the kernels and their routes are those of split ones."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CD1 = {2: [-1 / 2, 0.0, 1 / 2], 4: [1 / 12, -2 / 3, 0.0, 2 / 3, -1 / 12],
       6: [-1 / 60, 3 / 20, -3 / 4, 0.0, 3 / 4, -3 / 20, 1 / 60]}
CD2 = {2: [1.0, -2.0, 1.0], 4: [-1 / 12, 4 / 3, -5 / 2, 4 / 3, -1 / 12],
       6: [1 / 90, -3 / 20, 3 / 2, -49 / 18, 3 / 2, -3 / 20, 1 / 90]}


def _taps(spec):
    """dt f's merged taps per axis."""
    out = []
    for a in range(spec["dim"]):
        dx = 2.0 * np.pi / spec["n"][a]
        c1, c2 = np.array(CD1[spec["order"]]), np.array(CD2[spec["order"]])
        out.append((spec["dt"] * (-spec["c"][a] * c1 / dx + spec["alpha"] * c2 / (dx * dx))).astype(np.longdouble))
    return out


def _apply(u, taps, reverse=False):
    """(sum of w v, largest |v|) of dt f at every cell; u of shape (.., nx) in extended precision."""
    s, m = np.zeros_like(u), np.abs(u)
    for a, t in enumerate(taps):
        h = len(t) // 2
        for j in range(-h, h + 1):
            v = np.roll(u, j if reverse else -j, u.ndim - 1 - a)
            s += t[j + h] * v
            m = np.maximum(m, np.abs(v))
    return s, m


def _field(shape, kind, size, seed):
    rng = np.random.default_rng([seed, len(kind)])
    u = rng.uniform(0.5, 1.0, shape) * rng.choice([1.0, -1.0], shape)
    z = np.arange(shape[0]).reshape((-1,) + (1,) * (len(shape) - 1))
    if kind == "slab":  # two planes beside values of size 1, at every phase of a march
        u = np.where(z % 23 < 2, u * size, u)
    elif kind == "decay":  # falls and rises along z
        u = u * size ** (-0.25 * np.minimum(z % 41, 40 - z % 41))
    elif kind == "spikes":
        u = np.where(rng.random(shape) < 2e-4, u * size, u)
    return u


TILES = [
    ("o2", lambda: W.wl_3d([128, 96, 130], 1, 2, 3, 0, 901, c=(0.3, 0.2, 0.1))[0]),
    ("o4", lambda: W.wl_3d([128, 96, 130], 1, 4, 3, 0, 902, c=(0.3, 0.2, 0.1))[0]),
    ("o4_odd", lambda: W.wl_3d([125, 101, 127], 1, 4, 3, 0, 903, c=(0.3, 0.2, 0.1))[0]),
    ("o6", lambda: W.wl_3d([128, 96, 130], 1, 6, 3, 0, 904, c=(0.3, 0.2, 0.1), dt=0.01 * W.dx_of(130) ** 2 / 0.05)[0]),
    ("o4_ab2", lambda: W.wl_3d([128, 96, 130], 1, 4, 3, 0, 905, c=(0.3, 0.2, 0.1), tsteps=2)[0]),
]
FIELDS = [("slab", 1e4), ("slab", 1e8), ("slab", 1e16), ("slab", 1e20), ("decay", 4.0), ("decay", 1e4), ("decay", 1e8),
          ("spikes", 1e8)]


def _check(got, u, taps, n, reverse=False):
    f, m = _apply(u, taps, reverse)
    bar = (2 * n + 7) * np.longdouble(2.0) ** -53 * m * (1 + sum(np.abs(t).sum() for t in taps))
    off = np.abs(got.astype(np.longdouble) - (u + f))
    worst = np.unravel_index(np.argmax(off / bar), off.shape)
    assert (off <= bar).all(), (worst, got[worst], float((u + f)[worst]))


@pytest.mark.parametrize("kind,size", FIELDS, ids=[f"{k}_{s:g}" for k, s in FIELDS])
@pytest.mark.parametrize("name,make", TILES, ids=[t[0] for t in TILES])
def test_a_tiled_step_and_its_transpose_cell_by_cell(name, make, kind, size):
    from paper_1702_00496_gb300 import Solver
    spec = make()
    shape = tuple(spec["n"][::-1])
    u0, lam = _field(shape, kind, size, 1), _field(shape, kind, size, 2)
    s = Solver(spec)
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.step(1)
    s.sync()
    got = s.field().cpu().numpy().copy()
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.adjoint_forward(1, 1)
    g, _ = s.adjoint_backward(torch.as_tensor(lam, device="cuda"), False)
    g = g.cpu().numpy()
    s.close()
    n = 1 + 3 * spec["order"]
    _check(got, u0.astype(np.longdouble), _taps(spec), n)
    _check(g, lam.astype(np.longdouble), _taps(spec), n, reverse=True)


SPLIT = [
    ("o2_ragged", lambda: W.wl_3d([150, 126, 90], [3, 3, 2], 2, 3, 0, 911, c=(0.3, 0.2, 0.1))[0]),
    ("o4", lambda: W.wl_3d([128, 128, 128], [2, 2, 2], 4, 3, 0, 912, c=(0.3, 0.2, 0.1))[0]),
    ("o4_ab2", lambda: W.wl_3d([128, 128, 128], [2, 2, 2], 4, 3, 0, 913, c=(0.3, 0.2, 0.1), tsteps=2,
                               dt=0.02 * W.dx_of(128) ** 2 / 0.05)[0]),
]


@pytest.mark.parametrize("kind", ["half_zero", "ball", "pulse", "one_steep_tile"])
@pytest.mark.parametrize("name,make", SPLIT, ids=[s[0] for s in SPLIT])
def test_tiles_with_few_many_and_all_groups_listed_match_the_oracle(name, make, kind):
    """Groups that the tiles leave to the chains, in some planes of a tile, in most, in the rest of one: across faces with
    delays, in partial groups.  Bars as for the other routes: 1e-12 of the largest value, and 256 ulp of the largest value
    that a cell can depend on."""
    import os

    import oracle
    from paper_1702_00496_gb300 import Solver
    spec, steps = make(), 7
    cfg = oracle.Config(spec)
    rng = np.random.default_rng(spec["seed"])
    x = [(np.arange(n) / n - 0.5) for n in cfg.shape]
    r2 = x[0][:, None, None] ** 2 + x[1][None, :, None] ** 2 + x[2][None, None, :] ** 2
    noise = 1.0 + 0.1 * rng.standard_normal(cfg.shape)
    if kind == "half_zero":
        u0 = np.where(x[2][None, None, :] > 0.11, noise, 0.0)
    elif kind == "ball":
        u0 = np.where(r2 < 0.06, noise, 0.0)
    elif kind == "pulse":
        u0 = noise * np.exp(-r2 / 0.002)
    else:
        u0 = noise.copy()
        u0[10:40, 5:20, 3:30] *= 10.0 ** rng.uniform(-12, 0, (30, 15, 27))
    s = Solver(spec, log_steps=steps)
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.step(steps)
    s.sync()
    u, d = s.field().cpu().numpy().copy(), s.delays().cpu().numpy().copy()
    s.close()
    ref, dref, _ = oracle.run(oracle.Config(spec), steps, threads=os.cpu_count() or 1, u0=u0)
    assert np.array_equal(d, dref)
    assert np.abs(u - ref).max() <= 1e-12 * np.abs(ref).max()
    m = np.abs(u0)
    for ax in range(3):
        reach = spec["order"] // 2 * steps
        m = np.max([np.roll(m, k, ax) for k in range(-reach, reach + 1)], axis=0)
    assert (np.abs(u - ref) <= 256 * 2.0 ** -52 * np.maximum(m, np.abs(ref))).all()


@pytest.mark.parametrize("bits", [0, 12, 24, 36, 48])
@pytest.mark.parametrize("name,make", [t for t in TILES if t[0] != "o4_ab2"], ids=[t[0] for t in TILES if t[0] != "o4_ab2"])
def test_the_diffusivity_gradient_of_a_field_that_is_small_where_the_seed_is_not(name, make, bits):
    """dJ/dalpha of one step is the sum of lambda dt D2 U over the cells, and lambda here is nonzero only in a box where U is
    2^-bits of what it is elsewhere in the same tiles.  Each term is held to its own stencil as above, the sum of 512 terms
    to 512 roundings more."""
    from paper_1702_00496_gb300 import Solver
    spec = make()
    shape = tuple(spec["n"][::-1])
    rng = np.random.default_rng([spec["seed"], bits])
    u0 = rng.uniform(0.5, 1.0, shape)
    u0[40:60, 40:60, 40:60] *= 2.0 ** -bits
    lam = np.zeros(shape)
    lam[46:54, 46:54, 46:54] = rng.standard_normal((8, 8, 8))
    s = Solver(spec)
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.adjoint_forward(1, 1)
    _, ga = s.adjoint_backward(torch.as_tensor(lam, device="cuda"), True)
    s.close()
    q = [(spec["dt"] * np.array(CD2[spec["order"]]) / (2.0 * np.pi / n) ** 2).astype(np.longdouble) for n in spec["n"]]
    f, m = _apply(u0.astype(np.longdouble), q)
    n = 1 + 3 * spec["order"]
    bar = (2 * n + 7 + 512) * np.longdouble(2.0) ** -53 * (np.abs(lam) * m).sum() * sum(np.abs(t).sum() for t in q)
    assert abs(np.longdouble(ga) - (lam * f).sum()) <= bar


LINES = [
    ("block_o2", 8192, 2, 4, {}),
    ("block_o4", 8200, 4, 4, {}),
    ("block_o6", 8192, 6, 4, dict(r_alpha=0.02)),
    ("block_o4_k3", 8192, 4, 3, {}),
    ("block_o4_wide_tiles", 655364, 4, 4, {}),
    ("block_o4_odd", 8193, 4, 4, {}),
    ("block_o4_small_taps", 8192, 4, 4, dict(r_alpha=1e-6, c=0.0)),
    ("single_o2", 8192, 2, 1, {}),
    ("single_o4", 8192, 4, 1, {}),
    ("single_o6", 8192, 6, 1, dict(r_alpha=0.02)),
    ("single_o2_small_taps", 8192, 2, 1, dict(r_alpha=1e-6, c=0.0)),
    ("single_o4_ragged", 200001, 4, 1, {}),
    ("ab2_o4", 8192, 4, 1, dict(tsteps=2, r_alpha=0.02)),
    ("ab3_o6", 8192, 6, 1, dict(tsteps=3, r_alpha=0.01)),
    ("ab2_o2_ragged", 200001, 2, 1, dict(tsteps=2, r_alpha=0.02)),
]


@pytest.mark.parametrize("kind", ["ones", "noise", "spikes_1e6", "spikes_1e14", "steep", "half_zero", "waves"])
@pytest.mark.parametrize("name,n,order,K,kw", LINES, ids=[c[0] for c in LINES])
def test_a_1d_step_or_block_cell_by_cell(name, n, order, K, kw, kind):
    """Each cell of one step, or one block of K, to what the chain of its m taps may be off: 2^-53 of sum |w v| over its own
    stencil (Adams-Bashforth: and of its value) for each rounding, m more for the weights, and four for the fixed point."""
    from paper_1702_00496_gb300 import Solver, at_set_fusion
    spec = W.wl_1d(n, 1, order, 4, 0, 921, (1, 2), **kw)[0]
    rng = np.random.default_rng([921, len(name), len(kind)])
    u = rng.uniform(0.5, 1.0, n)
    x = np.arange(n)
    if kind == "ones":
        u = np.ones(n)
    elif kind == "noise":
        u = rng.standard_normal(n)
    elif kind.startswith("spikes"):
        u = np.where(rng.random(n) < 0.01, u * float(kind[7:]), u)
    elif kind == "steep":
        u = u * np.exp(-((x % 257) - 100.0) ** 2 / 200.0)
    elif kind == "half_zero":
        u = np.where(x > n // 3, u, 0.0)
    elif kind == "waves":
        u = np.sin(2 * np.pi * x / 97.0)
    s = Solver(spec)
    assert at_set_fusion(s.h, K) == K
    s.reset(torch.as_tensor(u, device="cuda"))
    s.step(K)
    s.sync()
    got = s.field().cpu().numpy().copy()
    s.close()
    f = _taps(spec)[0]
    one = f.copy()
    one[order // 2] += 1
    w = np.array([1], dtype=np.longdouble)
    for _ in range(K):
        w = np.convolve(w, one)
    v, h, m = u.astype(np.longdouble), len(w) // 2, len(w)
    want, size = np.zeros_like(v), np.zeros_like(v)
    for j in range(-h, h + 1):
        t = w[j + h] * np.roll(v, -j)
        want += t
        size += np.abs(t)
    if spec["tsteps"] > 1:  # dt f is added to the value
        size = np.abs(v) + sum(np.abs(f[j + order // 2] * np.roll(v, -j)) for j in range(-(order // 2), order // 2 + 1))
    bar = (2 * m + 4) * np.longdouble(2.0) ** -53 * size
    off = np.abs(got.astype(np.longdouble) - want)
    worst = int(np.argmax(off - bar))
    assert (off <= bar).all(), (worst, got[worst], float(want[worst]), float(off[worst] / bar[worst]) if bar[worst] else "")


@pytest.mark.parametrize("size", [1e-305, 1e-310, 1e-321])
@pytest.mark.parametrize("name,make", TILES, ids=[t[0] for t in TILES])
def test_a_tiled_step_and_its_transpose_of_denormal_numbers(name, make, size):
    """Fields whose largest value is denormal, or holds no bit of its upper word, are not zero.  As a chain each of the taps'
    roundings is at most half the smallest number there is, or 2^-53 of the values where those are larger."""
    from paper_1702_00496_gb300 import Solver
    spec = make()
    shape = tuple(spec["n"][::-1])
    u0 = _field(shape, "noise", 1.0, 3) * size
    s = Solver(spec)
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.step(1)
    s.sync()
    got = s.field().cpu().numpy().copy()
    s.reset(torch.as_tensor(u0, device="cuda"))
    s.adjoint_forward(1, 1)
    g, _ = s.adjoint_backward(torch.as_tensor(u0, device="cuda"), False)
    g = g.cpu().numpy()
    s.close()
    n, u = 1 + 3 * spec["order"], u0.astype(np.longdouble)
    for out, reverse in ((got, False), (g, True)):
        f, m = _apply(u, _taps(spec), reverse)
        bar = (n + 2) * np.longdouble(2.0) ** -1075 + (2 * n + 7) * np.longdouble(2.0) ** -53 * 2 * m
        assert (np.abs(out.astype(np.longdouble) - (u + f)) <= bar).all()
