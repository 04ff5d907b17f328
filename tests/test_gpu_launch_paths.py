"""One launch per step with captured graphs: the path of a tile variant set by
hand and of domains that the regions do not serve (a side below 8 nodes)."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1912_09327_gb300 import binding
    return binding


def same(got, want):
    return all(np.array_equal(x.view(np.uint32), y.view(np.uint32))
               for x, y in zip(got, want))


def test_single_domain_graphs_equal_direct_launches(b):
    """A variant set by hand, on a capturable stream (runs of 16 steps from a
    graph) and on the default stream (every step launched): odd call lengths
    (graphs for both starting copies), then another variant (captured again)
    and another wait limit (captured again)."""
    import torch
    p = wl.random_problem(333, 170, seed=41, amp=0.02, periodic=(True, False))
    runs = []
    for stream in (None, torch.cuda.Stream()):
        d = b.Domain.from_problem(p, stream=stream)
        d.set_variant(1)
        d.step(37)
        d.step(50)
        first = d.get_state()
        d.set_variant(2)
        d.step(40)
        d.set_copy_wait_ns(10**9 - 1)
        d.step(41)
        runs.append((first, d.get_state(), d.residual(), d.step_count()))
        d.close()
    assert same(runs[0][0], runs[1][0])
    assert same(runs[0][1], runs[1][1])
    assert runs[0][2:] == runs[1][2:]


def test_wait_limit_reaches_captured_graphs(b):
    """Graphs captured under the default limit are captured again after the
    limit changes: with 0 every staged row is given up at once (the flag),
    and with the default again nothing is."""
    import torch
    p = wl.random_problem(200, 120, seed=5, amp=0.02)
    d = b.Domain.from_problem(p, stream=torch.cuda.Stream())
    d.set_variant(1)
    d.step(40)
    d.residual()
    d.set_copy_wait_ns(0)
    d.step(40)
    with pytest.raises(b.LbmError) as e:
        d.residual()
    assert e.value.status == b.LBM_E_CUDA
    d.set_copy_wait_ns(10**9)
    d.set_moments(p.rho, p.jx, p.jy)
    d.step(40)
    d.residual()
    got = d.get_state()
    d.close()
    r = b.Domain.from_problem(p)
    r.step(40)
    assert same(got, r.get_state())
    r.close()


@pytest.mark.parametrize("variant", range(5))
@pytest.mark.parametrize("storage,rounding", [("f32", "nearest"),
                                              ("f32", "stochastic")])
def test_batch_graphs_equal_alone(b, variant, storage, rounding):
    """A member of six columns keeps its batch off the regions: every step
    goes through the batched tile kernel of the variant, runs of 16 from a
    graph, with large clean members among them and a change of membership."""
    import torch
    s = torch.cuda.Stream()
    probs = [wl.random_problem(6, 40, seed=1), wl.cavity(600, 0.1, ny=420),
             wl.random_problem(300, 170, seed=5, periodic=(True, False)),
             wl.channel(700, 300, 0.01)]
    with torch.cuda.stream(s):
        doms = [b.Domain.from_problem(p, stream=s, storage=storage,
                                      rounding=rounding) for p in probs]
        batch = b.Batch(len(doms), 100000, stream=s)
        slots = [batch.add(d) for d in doms]
        batch.set_variant(variant)
        batch.step(37)
        batch.step(20)
        batch.remove(slots[2])
        batch.step(35)
        for i, (d, p) in enumerate(zip(doms, probs)):
            r = b.Domain.from_problem(p, stream=s, storage=storage,
                                      rounding=rounding)
            r.step(57 if i == 2 else 92)
            assert same(d.get_state(), r.get_state()), i
            assert d.step_count() == r.step_count()
            r.close()
        batch.close()
