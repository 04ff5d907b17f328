"""lbm_step_noalloc on fields whose rows are far apart (a caller's layout):
wider rows than the region launches serve, through the single-step kernel."""
import numpy as np
import pytest

from paper_1912_09327_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pitch", [1 << 23, (1 << 23) + 32, 1 << 24])
def test_wide_pitch_equals_a_context(pitch):
    """Bit for bit at fluid and fixed nodes; the flag stays down."""
    import torch
    from paper_1912_09327_gb300 import binding as b
    nx, ny = 203, 41
    p = wl.random_problem(nx, ny, seed=77, amp=0.02, periodic=(True, False),
                          force=(1e-4, -5e-5))
    d = b.Domain.from_problem(p)
    d.step(1)
    want, (_, mass) = d.get_state(), d.residual()
    init = [(p.rho - 1.0).astype(np.float32), p.jx.astype(np.float32),
            p.jy.astype(np.float32)]
    # the three input fields side by side in one row; one buffer per output
    f = torch.empty((ny, pitch), dtype=torch.float32, device="cuda")
    src = [f[:, 1024 * k: 1024 * k + nx] for k in range(3)]
    for t, a in zip(src, init):
        t.copy_(torch.from_numpy(a))
    dst = [torch.empty((ny, pitch), dtype=torch.float32, device="cuda")
           for _ in range(3)]
    m = torch.empty(ny * pitch + 256, dtype=torch.uint8, device="cuda")
    m[: ny * pitch].view(ny, pitch)[:, :nx].copy_(torch.from_numpy(p.mask))
    sums = torch.zeros(3, dtype=torch.float64, device="cuda")
    flag = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    b.lbm_step_noalloc(*[t.data_ptr() for t in src],
                       *[t.data_ptr() for t in dst], m.data_ptr(), nx, ny,
                       pitch, p.periodic, p.force, sums.data_ptr(),
                       flag.data_ptr(),
                       torch.cuda.current_stream().cuda_stream)
    keep = p.mask != wl.SOLID
    for t, ref in zip(dst, want):
        got = t[:, :nx].cpu().numpy()
        assert np.array_equal(got[keep].view(np.uint32),
                              ref[keep].view(np.uint32))
    assert int(flag.item()) == 0
    # the masses are sums of |rho - 1| < 0.1 terms grouped by tile
    got = int((p.mask == wl.FLUID).sum()) + float(sums[2].item())
    assert abs(got - mass) <= 6e-8 * 0.1 * nx * ny
    d.close()
    del f, src, dst, m
    torch.cuda.empty_cache()
