"""The point selection of any map size in one CTA: the points of a call with few kept equal the
first points of a call that keeps every detection (on a map above 65,536 cells the multi-kernel
sort), for a few, some hundreds and tens of thousands of detections."""
import dataclasses

import numpy as np
import pytest
import torch

from sbr_inputs import CfarParams, radar_single_tx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,theta,noise,floor,k_max", [
    (4096, 64, 0.0, 1e-4, 2000),    # a few tones
    (4096, 64, 1.0, 0.0, 2000),     # noise: thousands of detections, radix selection
    (4096, 64, 1.0, 0.0, 7),
    (4096, 64, 0.02, 1e-4, 4096),
    (2048, 256, 1.0, 0.0, 4096),    # 524,288 cells
    (256, 64, 1.0, 0.0, 100),       # 16,384 cells
])
def test_selection_matches_full_sort(sbr, ns, theta, noise, floor, k_max):
    radar = radar_single_tx(ns, 1)
    rng = np.random.default_rng(ns + theta + k_max)
    n = np.arange(ns)
    cube = sum(a * np.exp(2j * np.pi * (f * n + p))[None] * np.ones((4, 1))
               for f, a, p in zip(rng.uniform(0.05, 0.45, 5), rng.uniform(0.2, 1, 5), rng.uniform(0, 1, 5)))
    cube = cube + noise * (rng.standard_normal((4, ns)) + 1j * rng.standard_normal((4, ns)))
    c = torch.from_numpy(np.stack([cube.real, cube.imag], -1)[:, None].astype(np.float32)).cuda().contiguous()
    cfg = dataclasses.replace(CfarParams(), n_theta=theta, k_max=k_max, floor_rel=floor, w_min=0.0 if noise == 1.0 else 0.01)
    few, st = sbr.pointcloud(c, radar, cfg)
    every, st_all = sbr.pointcloud(c, radar, dataclasses.replace(cfg, k_max=ns * theta // 2))
    m = st.n_points()
    assert m == min(k_max, st_all.n_points()) and m > 0
    assert torch.equal(few[:m], every[:m]) and not few[m:].any()
    assert torch.equal(st.peak_cells()[:m], st_all.peak_cells()[:m])
    if noise == 1.0:
        assert st_all.n_points() > min(k_max, 256)
