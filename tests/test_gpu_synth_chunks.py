"""sbr_synthesize on given records: CTAs that walk several chunks of 1,024 records, and grid positions
at the borders of the blocks of 512 cells, against FP64 (tolerances: tests/test_gpu_synth_records.py)."""
import numpy as np
import pytest
import torch

from sbr_inputs import C_LIGHT, radar_single_tx
from tests.test_gpu_synth_records import TOL, bind, bind64, direct, rel, records

pytestmark = pytest.mark.gpu

SMS = 152  # 4 antennas, three CTAs per SM: 114 CTAs per antenna


def edges(rng, ns, V, P):
    """Grid positions u at every border of 512 cells and one cell before it: on the cell, just
    past it, at its middle and just below the next."""
    M = 2 * ns
    border = np.arange(0, M, min(512, M))
    cell = rng.choice(np.concatenate([border, border - 1]), (V, P))
    return (cell + rng.choice([0.0, 2.0 ** -11, 0.5, 1 - 2.0 ** -11], (V, P))) % M


def moving(sbr, ns, nc, delta, phi, A, rate):
    radar = radar_single_tx(ns, nc)
    P = delta.shape[1]
    paths, phi, delta, A = bind(sbr, radar, P + 2, delta, phi, A, rate)
    cube = sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | sbr.SYNTH_MOVING)
    assert torch.equal(cube, sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | sbr.SYNTH_MOVING))
    per = radar.chirp_rep / C_LIGHT
    rate = rate.astype(np.float64)
    ref = torch.stack([direct(phi + rate * (c * per * radar.f0), delta + rate * (c * per * radar.bandwidth / ns), A, ns)
                       for c in range(nc)], 1)
    assert rel(cube, ref) <= 2 * TOL


@pytest.mark.parametrize("ns,nc", [(256, 4), (512, 4), (32, 16)])
def test_moving_several_chunks(sbr, ns, nc):
    """Chirps in tiles, three chunks per CTA (the last of a single record or two), their largest
    amplitudes a decade apart."""
    P = (SMS * 3 // 4) * 2 * 1024 + 114 + 57
    delta, phi, A = records(ns, 4, P, ns)
    A *= 10.0 ** (np.arange(P) // 1024 % 3 - 1)
    rate = np.random.default_rng(ns).uniform(-8.0, 8.0, delta.shape).astype(np.float32)
    rate[:, ::7] = 0.0
    moving(sbr, ns, nc, delta, phi, A, rate)


@pytest.mark.parametrize("ns,nc", [(256, 8), (512, 8), (512, 2)])
def test_moving_block_borders(sbr, ns, nc):
    """Cells at the borders, where chirps step over them in both directions."""
    P = 17001
    rng = np.random.default_rng(ns + nc)
    _, phi, A = records(nc, 4, P, ns)
    delta = (edges(rng, ns, 4, P) / (2 * ns) + 0.5) % 1.0 - 0.5
    moving(sbr, ns, nc, delta, phi, A, rng.choice([-2000.0, -8.0, 0.0, 8.0, 2000.0], delta.shape).astype(np.float32))


@pytest.mark.parametrize("ns,P", [(512, 17001), (1024, 9001), (2048, 30001), (4096, 240001)])
def test_split_block_borders(sbr, ns, P):
    radar = radar_single_tx(ns, 1)
    rng = np.random.default_rng(P)
    _, phi, A = records(P, 4, P, ns)
    paths, phi, delta, A = bind(sbr, radar, P + 7, (edges(rng, ns, 4, P) / (2 * ns) + 0.5) % 1.0 - 0.5, phi, A)
    cube = sbr.synthesize(paths, radar)
    assert torch.equal(cube, sbr.synthesize(paths, radar))
    assert rel(cube[:, 0], direct(phi, delta, A, ns)) <= TOL


@pytest.mark.parametrize("ns,P,nc", [(32, 3001, 1), (256, 20001, 1), (1024, 9001, 2), (4096, 40001, 1)])
def test_fp64_borders(sbr, ns, P, nc):
    """Path lengths that put the FP64 grid position at cell and block borders and just beside them."""
    radar = radar_single_tx(ns, nc)
    rng = np.random.default_rng(P)
    u = edges(rng, ns, 4, P) + rng.choice([-1e-9, 0.0, 1e-9], (4, P)) + 2 * ns
    L = u * C_LIGHT / (2 * radar.bandwidth)  # u = 2 N_s B L / (c N_s)
    rate = rng.uniform(-30.0, 30.0, (4, P)).astype(np.float32) if nc > 1 else None
    paths, L, A = bind64(sbr, radar, P + 3, L, rng.uniform(0.1, 1.0, (4, P)), rate)
    cube = sbr.synthesize(paths, radar, sbr.PHASE_FP64 | (sbr.SYNTH_MOVING if nc > 1 else 0))
    for c in range(nc):
        Lc = L + (c * radar.chirp_rep * rate if nc > 1 else 0.0)
        phi, delta = radar.f0 / C_LIGHT * Lc, radar.bandwidth / (C_LIGHT * ns) * Lc
        assert rel(cube[:, c], direct(phi - np.round(phi), delta - np.round(delta), A, ns)) <= TOL
