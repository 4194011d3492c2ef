"""Fields and error statistics in runs of 16 points, by one, two or eight threads to a run: sizes on either side of every line,
last runs that are partial.  The field is the multi-sine sum (numpy in extended precision) to what the recurrences over ten
wavenumbers may be off (modes.cuh: kmax^2 / 2 ulp of the amplitudes' sum, and one per mode); an ensemble's member of the same
size has the same bits; the statistics are those of the field, summed in another order."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n", [4092, 4096, 4100, 4108, 65532, 65536, 65548, 524284, 524288, 1048580])
def test_field_and_statistics_of_every_split(n):
    from paper_1702_00496_gb300 import Ensemble, Solver
    spec = W.wl_1d(n, 4, 4, 3, 0, 961, range(1, 11))[0]
    s = Solver(spec)
    u = s.field().cpu().numpy().copy()
    x = np.arange(n).astype(np.longdouble) * (2 * np.longdouble("3.14159265358979323846264338327950288") / n)
    want = sum(np.longdouble(a) * np.sin(np.longdouble(int(k)) * x + np.longdouble(p))
               for a, p, k in zip(spec["amp"][0], spec["phase"][0], spec["kappa"][0]))
    assert np.abs(u - want).max() <= (10 * 10 / 2 + 10) * 2.0 ** -52 * spec["amp"].sum()
    if n < 100000 and n % 16 == 0:  # PEs of groups of four
        e = Ensemble([spec], 0)
        e.run()
        torch.cuda.synchronize()
        assert torch.equal(e.field(0), s.field())
        e.close()
    v = u + 1e-3 * np.random.default_rng(n).standard_normal(n)
    s.reset(torch.as_tensor(v, device="cuda"))
    st = s.error_stats()
    s.reset()
    again = s.field().cpu().numpy().copy()
    s.close()
    assert np.array_equal(again, u)
    d = v - u
    pos = np.arange(n) % (n // 4)
    edge = (pos < 2) | (pos >= n // 4 - 2)
    # n terms of one sign, each within 2^-53, added up in some order: n roundings at most
    for got, ref in ((st["rms"], np.sqrt((d * d).mean())), (st["mean_abs"], np.abs(d).mean()), (st["ua_rms"], np.sqrt((u * u).mean())),
                     (st["rms_I"], np.sqrt((d[~edge] ** 2).mean())), (st["rms_B"], np.sqrt((d[edge] ** 2).mean()))):
        assert got == pytest.approx(ref, rel=n * 2.0 ** -52)
    assert st["max_abs"] == np.abs(d).max()
    assert (st["n_I"], st["n_B"]) == (int((~edge).sum()), int(edge.sum()))
