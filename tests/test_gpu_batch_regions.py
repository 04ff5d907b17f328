"""The multi-step region launches of a batch (lbm_resident.cuh): members of
every kind in one list, against each member stepped one launch per step."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1912_09327_gb300 import binding
    return binding


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("extra", [None, (7, 40)])
def test_mixed_members_equal_alone(b, storage, extra):
    """Members of different sizes, periodicities, step counts and rounding
    modes; with a member too narrow for the regions the whole batch takes one
    launch per step.  Bit-equal states either way (same arithmetic), over
    calls that alternate the copies."""
    shapes = [(8, 8), (64, 64), (61, 65), (130, 57), (333, 41), (70, 300)]
    shapes += [extra] if extra else []
    doms, want = [], []
    for i, (nx, ny) in enumerate(shapes):
        p = wl.random_problem(nx, ny, seed=5 * i, amp=0.02,
                              p_solid=0.1 * (i % 3),
                              periodic=(i % 2 == 0, i % 3 == 0))
        pair = []
        for _ in range(2):
            d = b.Domain(nx, ny, p.periodic, p.force, storage=storage,
                         rounding=("nearest", "stochastic")[i % 2])
            d.set_geometry(p.mask)
            d.set_moments(p.rho, p.jx, p.jy)
            d.set_step_count(3 * i)
            pair.append(d)
        doms.append(pair[0])
        want.append(pair[1])
    tiles = sum(b.lbm_tile_count(*s) for s in shapes)
    batch = b.Batch(len(doms), tiles)
    for d in doms:
        batch.add(d)
    for n in (3, 30, 1, 12):
        batch.step(n)
        for d in want:
            d.set_variant(3)
            d.step(n)
    bits = np.uint32 if storage == "f32" else np.uint16
    for d, e in zip(doms, want):
        for x, y in zip(d.get_state(), e.get_state()):
            assert np.array_equal(x.view(bits), y.view(bits))
        assert d.step_count() == e.step_count()
    batch.close()
    for d in doms + want:
        d.close()
