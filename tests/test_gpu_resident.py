"""lbm_step's inner steps on register-resident regions (lbm_resident.cuh):
several steps per launch give, bit for bit, the state of one launch per step."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# widths around the 64-column regions' edges (one region up to 61 columns
# walled, 64 less the halo periodic), heights around the regions' rows
SIZES = [(8, 8), (9, 64), (60, 17), (61, 33), (62, 32), (63, 65), (65, 130),
         (117, 57), (118, 259), (301, 143), (520, 9), (1027, 300)]


@pytest.fixture(scope="module")
def b():
    from paper_1912_09327_gb300 import binding
    return binding


def run(b, p, storage, rounding, calls, variant):
    ny, nx = p.mask.shape
    d = b.Domain(nx, ny, p.periodic, p.force, storage=storage,
                 rounding=rounding)
    d.set_geometry(p.mask)
    d.set_moments(p.rho, p.jx, p.jy)
    d.set_variant(variant)
    for n in calls:
        d.step(n)
    out = d.get_state(), d.residual()[1], d.step_count()
    d.close()
    return out


@pytest.mark.parametrize("storage,rounding", [
    ("f32", "nearest"), ("f32", "stochastic"), ("f16", "stochastic"),
    ("f16", "nearest"), ("bf16", "stochastic")])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_equals_one_launch_per_step(b, nx, ny, storage, rounding):
    """Random walls, fixed nodes and force (none: its sums are left out of the
    kernel), every periodicity, calls of
    several lengths, against a caller-chosen tile variant, which takes one
    launch per step.  Both round each node's arithmetic alike, so the states
    are equal bit for bit; the masses are sums of |rho - 1| < 0.1 terms
    grouped by tile (FP32 per lane)."""
    for k, per in enumerate([(False, False), (True, False), (False, True),
                             (True, True)]):
        p = wl.random_problem(nx, ny, seed=31 * nx + ny + k, amp=0.02,
                              p_solid=0.15 if k % 2 else 0.02, periodic=per,
                              force=(1e-4, -5e-5) if k < 2 else (0.0, 0.0))
        calls = (3, 31, 4 + k)
        got = run(b, p, storage, rounding, calls, -1)
        want = run(b, p, storage, rounding, calls, 3)
        bits = np.uint32 if storage == "f32" else np.uint16
        for x, y in zip(got[0], want[0]):
            assert np.array_equal(x.view(bits), y.view(bits)), per
        assert got[2] == want[2] == sum(calls)
        assert abs(got[1] - want[1]) <= 1.5e-5 * 0.1 * nx * ny


@pytest.mark.parametrize("nx,ny", SIZES)
def test_multiphase_equals_one_launch_per_step(b, nx, ny):
    """The multiphase step, whose rim goes stale by two nodes a step: random
    densities with walls and fixed nodes in every periodicity, bit for bit."""
    for k, per in enumerate([(False, False), (True, False), (False, True),
                             (True, True)]):
        p = wl.multiphase_random(nx, ny, seed=7 * nx + ny + k, periodic=per,
                                 force=(1e-4, -5e-5) if k < 2 else (0.0, 0.0))
        got = []
        for variant in (-1, 3):
            d = b.Domain.from_problem(p)
            d.set_variant(variant)
            for n in (3, 12, 4 + k):
                d.step(n)
            got.append(d.get_state())
            d.close()
        for x, y in zip(*got):
            assert np.array_equal(x.view(np.uint32), y.view(np.uint32)), per


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_reduced_step_sums(b, nx, ny, storage):
    """The residual and the mass of a reduced step on regions against the
    single-step kernel's, from the same state (which ends equal bit for bit).
    Both add a lane's terms in FP32 (at most 64 rows x 4 columns, the mass
    compensated): the positive sums agree to 256 * 2^-24 = 1.5e-5, the mass to
    2^-24 of the lanes' |rho - 1| <= 0.1 sums."""
    for k, per in enumerate([(False, False), (True, True)]):
        p = wl.random_problem(nx, ny, seed=nx + 3 * ny + k, amp=0.02,
                              p_solid=0.15 * k, periodic=per)
        got = []
        for variant in (-1, 3):
            d = b.Domain(nx, ny, p.periodic, p.force, storage=storage)
            d.set_geometry(p.mask)
            d.set_moments(p.rho, p.jx, p.jy)
            d.set_variant(variant)
            d.step(1)
            got.append((d.get_state(), d.residual()))
            d.close()
        bits = np.uint32 if storage == "f32" else np.uint16
        for x, y in zip(got[0][0], got[1][0]):
            assert np.array_equal(x.view(bits), y.view(bits)), per
        (r0, m0), (r1, m1) = got[0][1], got[1][1]
        assert r0 == pytest.approx(r1, rel=1.5e-5)
        assert abs(m0 - m1) <= 6e-8 * 0.1 * nx * ny


def test_captured_calls_replay(b):
    """A caller's graph of an even number of steps leaves the state in the
    copy it found it in, so that replays go on from one another."""
    import torch
    p = wl.random_problem(333, 170, seed=41, amp=0.02, periodic=(True, False))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        d, e = (b.Domain.from_problem(p, stream=s) for _ in range(2))
        e.step(3 * 22)
        d.step(22)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            d.step(22)
        g.replay()
        g.replay()
        got, want = d.get_state(), e.get_state()
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
    d.close()
    e.close()
