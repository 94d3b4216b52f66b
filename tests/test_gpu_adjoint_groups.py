"""The trace adjoint's fixed-point sums do not depend on how lanes that add to one vertex are
grouped: ray counts on either side of where the groups that add as one change (8,192 and 40,000
rays), with the rays in grid order (large groups) and shuffled (small ones), give the same bits."""
import numpy as np
import pytest
import torch

from sbr_inputs import ground_plane, icosphere, merge_meshes, radar_single_tx, ray_grid_for_sphere
from tests.test_gpu_adjoint_order import gradient

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8192, 8193, 40000, 40001])
def test_ray_order_leaves_the_gradient_unchanged(sbr, n):
    mesh = merge_meshes(icosphere(2, 0.2, (0.0, 0.0, 1.0)), ground_plane(-0.2, 0.0, 1.0))
    v, f = torch.from_numpy(mesh[0]).cuda(), torch.from_numpy(mesh[1]).cuda()
    radar = radar_single_tx(256, 1)
    grid = ray_grid_for_sphere((0.0, -0.1, 1.0), 0.3, 201)
    gcube = torch.randn(4, 1, 256, 2, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    ids = np.arange(n, dtype=np.int32)
    a = gradient(sbr, v, f, radar, grid, torch.from_numpy(ids).cuda(), gcube, True)
    b = gradient(sbr, v, f, radar, grid, torch.from_numpy(np.random.default_rng(n).permutation(ids)).cuda(), gcube, True)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert bool(a[0].abs().sum() > 0)
