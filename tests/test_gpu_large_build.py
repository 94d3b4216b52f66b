"""The build of meshes above 65,536 triangles (separate launches) against the fused build of the part
that the rays can reach: the same hits, also after a refit to other positions and back."""
import numpy as np
import pytest
import torch

from sbr_inputs import merge_meshes, radar_single_tx, ray_grid_for_sphere, superquadric

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("total", [65537, 67584, 67585, 69632, 100001, 150000])
def test_large_build(sbr, total):
    v, f, _ = superquadric(8, 100, 100, center=(0.0, 0.0, 1.0))
    w, g, _ = superquadric(3, 270, 270, center=(0.0, 0.0, 40.0))  # behind it
    keep = np.random.default_rng(total).permutation(len(g))[:total - len(f)]
    both = merge_meshes((v, f), (w, g[np.sort(keep)]))
    assert len(both[1]) == total
    radar = radar_single_tx(256, 1)
    grid = ray_grid_for_sphere((0.0, 0.0, 1.0), 0.15, 100)
    part = sbr.Scene(torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda())
    verts = torch.from_numpy(both[0]).cuda()
    scene = sbr.Scene(verts, torch.from_numpy(both[1]).cuda())
    want = sbr.trace(part, radar, grid, 1)
    hit = want.hits()[0] >= 0  # the others are the same object's

    def check():
        got = sbr.trace(scene, radar, grid, 1)
        scene.check()
        assert torch.equal(got.hits()[0][hit], want.hits()[0][hit])
        assert torch.equal(got.hit_pos()[hit], want.hit_pos()[hit])

    assert bool(hit.any())
    check()
    scene.refit(verts * 1.5)
    scene.refit(verts)
    check()
    scene.update(verts)
    check()
