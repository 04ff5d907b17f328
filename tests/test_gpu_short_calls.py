"""Calls of two and three steps on a large clean domain."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [2, 3])
def test_large_clean_domain_takes_the_faster_kernel(steps):
    """One step per launch moves the same bytes by either kernel: a call is
    not slower than with the clean-tile variant set by hand (regions took 5 and
    9 % longer; the best of several runs differs by about 1 %)."""
    import torch
    from paper_1912_09327_gb300 import binding as b
    n = 16384
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        d = b.Domain(n, n, (True, True), stream=s)
        d.set_geometry(np.zeros((n, n), np.uint8))
        best = {}
        for _ in range(5):
            for variant in (4, -1):
                d.set_variant(variant)
                t0, t1 = (torch.cuda.Event(enable_timing=True)
                          for _ in range(2))
                d.step(steps)
                t0.record(s)
                for _ in range(4):
                    d.step(steps)
                t1.record(s)
                t1.synchronize()
                ms = t0.elapsed_time(t1)
                best[variant] = min(ms, best.get(variant, ms))
        d.close()
    torch.cuda.empty_cache()
    assert best[-1] < 1.03 * best[4]
