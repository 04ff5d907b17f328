"""The batch autotuner times what the tile variant decides."""
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_times_are_those_of_the_variants_own_step():
    """Large members, whose steps before a call's last one run on regions at
    less than half the time of a tile kernel's step.  The autotuner's figure of
    a variant is the time of reduced steps with it (calls of one step add the
    final sums and a copy of the member table)."""
    import torch
    from paper_1912_09327_gb300 import binding as b
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        doms = [b.Domain.from_problem(wl.cavity(1500, 0.1), stream=s)
                for _ in range(3)]
        batch = b.Batch(3, 3 * b.lbm_tile_count(1500, 1500), stream=s)
        for d in doms:
            batch.add(d)
        chosen, ms = batch.autotune(20)
        assert doms[0].step_count() == 22 * b.lbm_variant_count()
        assert ms[chosen] == min(ms)
        for v in range(b.lbm_variant_count()):
            batch.set_variant(v)
            batch.step(1)
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record(s)
            for _ in range(20):
                batch.step(1)
            t1.record(s)
            t1.synchronize()
            assert 0.6 < ms[v] / (t0.elapsed_time(t1) / 20) < 1.2
        batch.close()


def test_members_without_regions():
    """A side below 8 keeps the batch off the regions; the autotuner's steps
    are then one call's, and the members advance alike."""
    from paper_1912_09327_gb300 import binding as b
    doms = [b.Domain.from_problem(wl.random_problem(nx, ny, seed=3))
            for nx, ny in ((7, 40), (120, 64))]
    batch = b.Batch(2, sum(b.lbm_tile_count(d.nx, d.ny) for d in doms))
    for d in doms:
        batch.add(d)
    _, ms = batch.autotune(4)
    assert min(ms) > 0
    for d in doms:
        assert d.step_count() == 6 * b.lbm_variant_count()
    batch.close()
