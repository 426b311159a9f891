"""GPU tests of the launch rules: every kernel a call can be routed to, at the
edges where the rule or the kernel's tiling changes, against the other route
or the oracle."""
import numpy as np
import pytest
import torch

from paper_2603_09668_gb300 import binding as B

pytestmark = pytest.mark.gpu


# HOME-LBM: a call of several steps on populations against the same steps one
# call at a time. Above 2^20 cells one step runs the tile kernel, below it the
# population kernels too, so both routes and both parities of the last step
# meet. The two round alike except for contraction: 5e-7 of the largest moment
# per step (a few float32 roundings of sums of order one).
@pytest.mark.parametrize("shape,bc_x", [((131, 103, 79), 1), ((130, 97, 85), 0), ((33, 7, 5), 1),
                                        ((2, 2, 2), 0)])
@pytest.mark.parametrize("steps", [1, 2, 3, 4, 5])
def test_home_steps_on_populations(shape, bc_x, steps):
    nx, ny, nz = shape
    g = torch.Generator(device="cuda").manual_seed(5)
    lbm = B.LBM(shape, 0.6, u_inlet=(0.05, 0.01, -0.02), force=(1e-5, 0.0, -2e-5), bc_x=bc_x)
    a = lbm.moments()
    lbm.home_init(a, 1.0, (0.04, 0.0, 0.01))
    a[:4] += 5e-3 * torch.randn(a[:4].shape, generator=g, device="cuda")
    solid = (torch.rand((nz, ny, nx), generator=g, device="cuda") < 0.1).to(torch.uint8)
    b, start = a.clone(), a.clone()
    lbm.home_step(a, solid, steps)
    for _ in range(steps):
        lbm.home_step(b, solid, 1)
    assert torch.isfinite(a).all()
    assert (a - b).abs().max().item() <= 5e-7 * steps
    keep = solid.bool().expand(10, nz, ny, nx)
    assert torch.equal(a[keep], start[keep])
    lbm.close()
