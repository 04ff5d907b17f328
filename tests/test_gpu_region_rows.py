"""The region launches with 4 and 8 rows per warp, which mid-sized and large
domains take: bit for bit the states of one launch per step (a tile variant
set by hand), in every format and rounding mode, with walls in a part of the
domain (blocks with walls and blocks without run different copies of the
code).  The tiling is asserted, so that the cover does not rest on the cost
model."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SIZES = [(1027, 1300), (1333, 1101)]
PLACES = [((False, False), (1e-4, -5e-5)), ((True, True), (0.0, 0.0)),
          ((True, False), (0.0, 0.0)), ((False, True), (1e-4, -5e-5))]
CALLS = (3, 31, 6)


def rows(nx, ny, periodic, run, reach=1):
    from . import regions
    return regions.choose([regions.shape(nx, ny, periodic, reach=reach)],
                          run).rows


def half_walled(p):
    """Node types of the left part only; a fluid at the same state elsewhere."""
    p.mask[:, p.mask.shape[1] // 3:] = wl.FLUID
    return p


def advance(p, variant, calls, **kw):
    from paper_1912_09327_gb300 import binding as b
    d = b.Domain.from_problem(p, **kw)
    d.set_variant(variant)
    for n in calls:
        d.step(n)
    out = d.get_state(), d.residual(), d.step_count()
    d.close()
    return out


def assert_same(got, want):
    for x, y in zip(got, want):
        bits = np.uint32 if x.dtype.itemsize == 4 else np.uint16
        assert np.array_equal(x.view(bits), y.view(bits))


@pytest.mark.parametrize("storage,rounding", [
    ("f32", "nearest"), ("f32", "stochastic"), ("f16", "stochastic"),
    ("f16", "nearest"), ("bf16", "stochastic")])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("periodic,force", PLACES)
def test_eight_rows(nx, ny, storage, rounding, periodic, force):
    for run in (2, 5, 30):
        assert rows(nx, ny, periodic, run) == 8
    p = half_walled(wl.random_problem(nx, ny, seed=nx + ny, amp=0.02,
                                      p_solid=0.05, periodic=periodic,
                                      force=force))
    got, want = (advance(p, v, CALLS, storage=storage, rounding=rounding)
                 for v in (-1, 3))
    assert_same(got[0], want[0])
    assert got[2] == want[2] == sum(CALLS)


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("periodic,force", PLACES)
def test_eight_rows_multiphase(nx, ny, periodic, force):
    for run in (5, 30):
        assert rows(nx, ny, periodic, run, reach=2) == 8
    p = half_walled(wl.multiphase_random(nx, ny, seed=nx + ny, p_solid=0.05,
                                         periodic=periodic, force=force))
    assert_same(*(advance(p, v, CALLS)[0] for v in (-1, 3)))


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("periodic,force", PLACES[:2])
def test_eight_rows_reduced(nx, ny, storage, periodic, force):
    """One reduced step.  Both kernels add a lane's terms in FP32 (at most 64
    rows x 4 columns, the mass compensated): the positive sums agree to 256 *
    2^-24 = 1.5e-5, the mass to 2^-24 of the lanes' |rho - 1| <= 0.1 sums."""
    assert rows(nx, ny, periodic, 1) == 8
    p = half_walled(wl.random_problem(nx, ny, seed=nx * 3, amp=0.02,
                                      p_solid=0.05, periodic=periodic,
                                      force=force))
    got, want = (advance(p, v, (1,), storage=storage) for v in (-1, 3))
    assert_same(got[0], want[0])
    assert got[1][0] == pytest.approx(want[1][0], rel=1.5e-5)
    assert abs(got[1][1] - want[1][1]) <= 6e-8 * 0.1 * nx * ny


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("kind,shapes", [
    (4, [(500, 500), (300, 200)]),
    (8, [(700, 640), (520, 333), (9, 400)])])
def test_batch_rows(kind, shapes, storage):
    """Batches whose members share regions of 4 and of 8 rows per warp, of
    both rounding modes, against each member alone."""
    from paper_1912_09327_gb300 import binding as b
    from . import regions
    places = [((i % 2 == 0, i % 3 == 0), PLACES[i % 2][1])
              for i in range(len(shapes))]
    doms = [regions.shape(*s, per) for s, (per, _) in zip(shapes, places)]
    assert regions.choose(doms, 8).rows == kind
    batch = b.Batch(len(shapes), sum(b.lbm_tile_count(*s) for s in shapes))
    got, want = [], []
    for i, ((nx, ny), (per, force)) in enumerate(zip(shapes, places)):
        p = half_walled(wl.random_problem(nx, ny, seed=i, amp=0.02,
                                          p_solid=0.05, periodic=per,
                                          force=force))
        kw = dict(storage=storage, rounding=("nearest", "stochastic")[i % 2])
        got.append(b.Domain.from_problem(p, **kw))
        want.append(advance(p, 3, CALLS, **kw)[0])
        batch.add(got[-1])
    for n in CALLS:
        batch.step(n)
    for d, w in zip(got, want):
        assert_same(d.get_state(), w)
    batch.close()
