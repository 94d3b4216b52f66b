"""The trace adjoint's fixed-point sums do not depend on which rays share a warp: the same rays
in another order (large shared triangles and single-ray ones mixed) give the same bits."""
import numpy as np
import pytest
import torch

from sbr_inputs import ground_plane, icosphere, merge_meshes, radar_single_tx, ray_grid_for_sphere

pytestmark = pytest.mark.gpu


def gradient(sbr, v, f, radar, grid, ids, gcube, materials):
    scene = sbr.Scene(v, f)
    if materials:
        scene.set_materials([4.0 - 0.5j, 9.0 - 2.0j],
                            torch.from_numpy((np.arange(f.shape[0]) % 2).astype(np.int32)).cuda())
    paths = sbr.trace(scene, radar, grid, 3, ids)
    glen, gamp, gph = sbr.synthesize_bwd(paths, radar, gcube, phase=True)
    geps = torch.zeros(2, 2, device="cuda")
    g = sbr.trace_bwd(scene, v, radar, grid, paths, glen, gamp, ids, gphase=gph, geps=geps if materials else None)
    return g, geps


@pytest.mark.parametrize("n,materials", [(1, False), (33, False), (700, True), (4096, False)])
def test_ray_order_leaves_the_gradient_unchanged(sbr, n, materials):
    mesh = merge_meshes(icosphere(3, 0.2, (0.0, 0.0, 1.0)), ground_plane(-0.2, 0.0, 1.0))
    v, f = torch.from_numpy(mesh[0]).cuda(), torch.from_numpy(mesh[1]).cuda()
    radar = radar_single_tx(256, 1)
    grid = ray_grid_for_sphere((0.0, -0.1, 1.0), 0.3, 64)
    gcube = torch.randn(4, 1, 256, 2, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    rng = np.random.default_rng(n)
    ids = np.sort(rng.choice(4096, n, replace=False)).astype(np.int32)
    a = gradient(sbr, v, f, radar, grid, torch.from_numpy(ids).cuda(), gcube, materials)
    b = gradient(sbr, v, f, radar, grid, torch.from_numpy(rng.permutation(ids)).cuda(), gcube, materials)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert bool(a[0].abs().sum() > 0) or n == 1
