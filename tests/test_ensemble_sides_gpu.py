"""What an ensemble leaves in the caller's memory, and members with as many PE sides as its shared memory takes: the delays of all sides, two buffers of a byte each,
lie beside the member's parameters.  The fields are those of single steps of the same problem, bit for bit."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _spec(P):
    return W.wl_1d(4 * P, P, 2, 3, 0, 931, (1, 2))[0]


@pytest.mark.parametrize("threads", [0, 256])
@pytest.mark.parametrize("P", [9600, 9984, 10000, 10496, 12288])
def test_members_with_many_sides_run(P, threads):
    from paper_1702_00496_gb300 import Ensemble, Solver, at_set_fusion
    e = Ensemble([_spec(P)], 20, log=True, threads=threads)
    e.ring.fill_(float("nan"))
    e.run()
    s = Solver(_spec(P), log_steps=20)
    at_set_fusion(s.h, 1)
    s.step(20)
    s.sync()
    torch.cuda.synchronize()
    assert torch.equal(e.field(0), s.field()) and torch.equal(e.delays(0), s.delays())
    assert e.stats()[0][0]["rms"] == pytest.approx(s.error_stats()["rms"], rel=1e-9)
    e.close()
    s.close()


def test_more_sides_than_that_are_refused():
    from paper_1702_00496_gb300 import Ensemble
    with pytest.raises(Exception, match="too many PE sides"):
        Ensemble([_spec(12292)], 20)


@pytest.mark.parametrize("n", [64, 4096, 6000])
def test_the_ring_keeps_every_level_that_a_single_run_keeps(n):
    """Level m lies in slot m mod (L + T) after the run too, the oldest one included: as after single steps, bit for bit."""
    from paper_1702_00496_gb300 import Ensemble, Solver, at_set_fusion
    specs = [W.wl_1d(n, n // 8, 2, 3, 0, 941 + r, (1, 2))[0] for r in range(2)]
    e = Ensemble(specs, 17)
    e.run()
    torch.cuda.synchronize()
    at = 0
    for spec in specs:
        s = Solver(spec)
        at_set_fusion(s.h, 1)
        s.step(17)
        s.sync()
        assert torch.equal(e.ring[at:at + s.ring.numel()], s.ring)
        at += s.ring.numel()
        s.close()
    e.close()
