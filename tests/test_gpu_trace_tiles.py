"""A full grid (in order up to one wave of CTAs, then in tiles of 32 x 32 and above 400,000 rays of 16 x
16 rays from the border inwards) against the same rays as a list (taken in its order): the same
records, bit for bit, and every ray traced once."""
import pytest
import torch

from sbr_inputs import ground_plane, jittered, merge_meshes, radar_single_tx, ray_grid_for_sphere, superquadric

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,jitter", [(182, False), (369, True), (370, False), (383, True), (384, False), (385, True),
                                      (632, False), (633, True), (640, False), (641, True)])
def test_tiles_match_list(sbr, G, jitter):
    v, f, _ = superquadric(5, 60, 60, center=(0.0, 0.0, 1.0))
    v, f = (torch.from_numpy(x).cuda() for x in merge_meshes((v, f), ground_plane(-0.2, 0.0, 1.0)))
    radar = radar_single_tx(256, 1)
    grid = ray_grid_for_sphere((0.0, 0.0, 1.0), 0.35, G)
    if jitter:
        grid = jittered(grid, G)
    scene = sbr.Scene(v, f)
    ids = torch.arange(G * G, dtype=torch.int32, device="cuda")
    a, b = (sbr.PathBuffers(G * G, 3, radar.n_virt) for _ in range(2))
    for p in (a, b):
        p.mem.fill_(0xAA)
    sbr.trace(scene, radar, grid, 3, out=a)
    sbr.trace(scene, radar, grid, 3, ids, out=b)
    assert torch.equal(a.hits()[0], b.hits()[0]) and torch.equal(a.hits()[1], b.hits()[1])
    assert torch.equal(a.hit_pos(), b.hit_pos()) and torch.equal(a.ray_weight(), b.ray_weight())
    P = a.count()
    assert P == b.count() == int((a.hits()[0] >= 0).sum()) and torch.equal(a.prep()[:, :P], b.prep()[:, :P])
    assert sbr.sim.trace_counts(scene, radar, grid, 3, a) == sbr.sim.trace_counts(scene, radar, grid, 3, b, ids)
