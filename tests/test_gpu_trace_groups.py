"""The few-ray trace (a group of lanes per ray) against the many-ray one (a thread per ray): the
same rays as a list and in a full grid hit the same triangles at the same points, bit for bit."""
import numpy as np
import pytest
import torch

from sbr_inputs import (icosphere, merge_meshes, ground_plane, jittered, radar_single_tx, ray_grid_for_sphere,
                        superquadric)

pytestmark = pytest.mark.gpu


def mesh(kind):
    if kind == "one":
        return (np.array([[-0.1, -0.1, 1.0], [0.1, -0.1, 1.0], [0.0, 0.1, 1.0]], np.float32),
                np.array([[0, 1, 2]], np.int32))
    if kind == "plane":
        return ground_plane(-0.1, 0.0, 1.0)
    if kind == "ico":
        return icosphere(4, 0.2, (0.0, 0.0, 1.0))
    v, f, _ = superquadric(5, 90, 90, center=(0.0, 0.0, 1.0))
    return merge_meshes((v, f), ground_plane(-0.2, 0.0, 1.0))


@pytest.mark.parametrize("kind,n", [("one", 9), ("plane", 4097), ("ico", 1), ("ico", 33), ("ico", 4096), ("quadric", 7),
                                    ("quadric", 1023), ("quadric", 32768)])
def test_few_rays_match_many(sbr, kind, n):
    v, f = (torch.from_numpy(x).cuda() for x in mesh(kind))
    radar = radar_single_tx(256, 1)
    grid = jittered(ray_grid_for_sphere((0.0, 0.0, 1.0), 0.35, 200), 3)
    scene = sbr.Scene(v, f)
    full = sbr.trace(scene, radar, grid, 4)
    ids = np.random.default_rng(n).permutation(grid.n_rays)[:n].astype(np.int32)
    few = sbr.trace(scene, radar, grid, 4, torch.from_numpy(ids).cuda())
    at = torch.from_numpy(ids.astype(np.int64)).cuda()
    assert torch.equal(few.hits()[0], full.hits()[0][at])
    assert torch.equal(few.hit_pos(), full.hit_pos()[at])
    assert torch.equal(few.ray_weight(), full.ray_weight()[at])
    assert few.count() == int((few.hits()[0] >= 0).sum())


@pytest.mark.parametrize("n", [1, 2, 3, 31, 33, 500, 512, 513, 1023, 1024])
def test_one_tile_build(sbr, n):
    """A mesh of at most 1024 triangles (one sort in one CTA) against the same triangles with others
    behind the radar added (several tiles): the same hits."""
    v, f, _ = superquadric(8, 24, 24, center=(0.0, 0.0, 1.0))
    f = f[np.random.default_rng(n).permutation(len(f))[:n]]
    w, g = icosphere(3, 0.2, (0.0, 0.0, -1.0))
    both = merge_meshes((v, f), (w, g))
    radar = radar_single_tx(256, 1)
    grid = ray_grid_for_sphere((0.0, 0.0, 1.0), 0.5, 100)
    out = []
    for mesh_v, mesh_f in ((v, f), both):
        scene = sbr.Scene(torch.from_numpy(mesh_v).cuda(), torch.from_numpy(mesh_f).cuda())
        out.append(sbr.trace(scene, radar, grid, 3))
        scene.check()
    hit = out[0].hits()[0]
    same = (hit == out[1].hits()[0]).all(1)  # a ray reflected back may meet the others
    assert bool((same | (out[1].hits()[0] >= n).any(1)).all())
    assert n < 500 or bool((hit >= 0).any())
