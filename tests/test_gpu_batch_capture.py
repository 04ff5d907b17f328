"""A caller's CUDA graph of a batch call, replayed between other calls: an even
number of steps leaves every member's state in the copy it was in."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(200, 150), (333, 91), (700, 640)]


def make(b, stream, storage, rounding):
    doms = []
    for i, (nx, ny) in enumerate(SHAPES):
        p = wl.random_problem(nx, ny, seed=i, amp=0.02, p_solid=0.05,
                              periodic=(i % 2 == 0, True))
        d = b.Domain(nx, ny, p.periodic, p.force, stream=stream,
                     storage=storage, rounding=rounding)
        d.set_geometry(p.mask)
        d.set_moments(p.rho, p.jx, p.jy)
        doms.append(d)
    batch = b.Batch(len(doms), sum(b.lbm_tile_count(*s) for s in SHAPES),
                    stream=stream)
    for d in doms:
        batch.add(d)
    return batch, doms


def states(doms):
    return [np.asarray(x).view(np.uint16) for d in doms for x in d.get_state()]


@pytest.mark.parametrize("storage,rounding", [
    ("f32", "nearest"), ("bf16", "stochastic"), ("f32", "stochastic")])
def test_replays_equal_calls(storage, rounding):
    """Each replay goes on with the random bits of the steps it takes, as a
    call does (members' step counts are the host's and are not compared)."""
    import torch
    from paper_1912_09327_gb300 import binding as b
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        got, doms = make(b, s, storage, rounding)
        want, other = make(b, s, storage, rounding)
        got.step(8)  # uploads, outside the capture
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
            got.step(8)
        for _ in range(3):
            g.replay()
        for _ in range(4):
            want.step(8)
        for x, y in zip(states(doms), states(other)):
            assert np.array_equal(x, y)
        got.close()
        want.close()


@pytest.mark.parametrize("between", [2, 4, 30])
def test_replays_between_calls_of_other_lengths(between):
    """A replay finds the members' regions as the captured call left them,
    whatever (even) lengths the calls since then had (an odd call leaves the
    member table naming the other copies)."""
    import torch
    from paper_1912_09327_gb300 import binding as b
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        got, doms = make(b, s, "f32", "nearest")
        want, other = make(b, s, "f32", "nearest")
        got.step(8)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
            got.step(8)
        g.replay()
        for _ in range(2):
            got.step(between)
        g.replay()
        want.step(24 + 2 * between)
        for x, y in zip(states(doms), states(other)):
            assert np.array_equal(x, y)
        got.close()
        want.close()


@pytest.mark.parametrize("first", [0, 1])
def test_lists_of_a_capture_that_never_ran(first):
    """Work lists that a capture only recorded are uploaded by the next call
    (the members' block tiles with no call before the capture, their regions
    with none of three steps or more), and a replay after it finds them too."""
    import torch
    from paper_1912_09327_gb300 import binding as b
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        got, doms = make(b, s, "f32", "stochastic")
        want, other = make(b, s, "f32", "stochastic")
        if first:
            got.step(2)
            want.step(2)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
            got.step(8)
        got.step(8)
        want.step(8)
        for x, y in zip(states(doms), states(other)):
            assert np.array_equal(x, y)
        got.close()
        want.close()
