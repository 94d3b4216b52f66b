"""sbr_synthesize on records of very unequal, cancelling and very small amplitudes against FP64.

The spreading rounds a class of records on one scale: the class's rms amplitude is an eighth of
its largest or more, a term's rounding (2^-24 of the largest at worst, 16 terms a record, their
kernel's squares 1.9 in sum) is then 4e-7 of the class's samples, whatever the other records are;
with the other contributions (1.7e-7, tests/test_gpu_synth_records.py) 4.4e-7.  The tolerance is
about twice that, and twice again for chirps whose shifts are rounded once more."""

import math

import numpy as np
import pytest
import torch

from sbr_inputs import C_LIGHT, radar_single_tx
from tests.test_gpu_synth_records import bind, bind64, direct, rel

pytestmark = pytest.mark.gpu

TOL = 1e-6


def amplitudes(rng, kind, V, P):
    A = rng.uniform(0.5, 1.0, (V, P)) * rng.choice([1.0, -1.0], (V, P))
    if kind == "strong":      # one record in 1,024 a hundred times the others
        A[:, ::1024] *= 100.0
    elif kind == "decades":   # six decades, evenly
        A = np.sign(A) * 10.0 ** rng.uniform(-6.0, 0.0, (V, P))
    elif kind == "few":       # a few of strength, the others 1e-2 to 1e-5 of it, some none at all
        A = np.sign(A) * 10.0 ** rng.uniform(-5.0, -2.0, (V, P))
        A[:, 5::1024], A[:, 3::7] = 1.0, 0.0
    elif kind == "cancel":    # pairs a thousand times the others, equal and opposite
        A[:, 0::1024] *= 1000.0
        A[:, 1::1024] = -A[:, 0::1024][:, :A[:, 1::1024].shape[1]]
    elif kind.startswith("1e"):
        A *= float(kind)
    return A


def pairs(kind, *arrays):
    for x in arrays:
        if kind == "cancel":
            x[:, 1::1024] = x[:, 0::1024][:, :x[:, 1::1024].shape[1]]


KINDS = ["strong", "decades", "few", "cancel", "1e-25", "1e-33", "1e30"]


def reference(phi, delta, A, ns):
    top = np.abs(A).max()
    return direct(phi, delta, A / top, ns) * top


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("ns,P", [(64, 200000), (256, 40001), (4096, 9000)])
def test_split(sbr, ns, P, kind):
    rng = np.random.default_rng(P)
    delta, phi = rng.uniform(-0.5, 0.5, (4, P)), rng.uniform(-0.5, 0.5, (4, P))
    pairs(kind, delta, phi)
    paths, phi, delta, A = bind(sbr, radar_single_tx(ns, 1), P + 3, delta, phi, amplitudes(rng, kind, 4, P))
    cube = sbr.synthesize(paths, radar_single_tx(ns, 1))
    assert torch.equal(cube, sbr.synthesize(paths, radar_single_tx(ns, 1)))
    assert rel(cube[:, 0], reference(phi, delta, A, ns)) <= TOL


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("ns,P", [(256, 3000), (1024, 9001)])
def test_fp64(sbr, ns, P, kind):
    radar = radar_single_tx(ns, 1)
    rng = np.random.default_rng(P)
    L = rng.uniform(0.1, 0.999, (4, P)) * ns * C_LIGHT / radar.bandwidth
    pairs(kind, L)
    paths, L, A = bind64(sbr, radar, P + 3, L, amplitudes(rng, kind, 4, P))
    cube = sbr.synthesize(paths, radar, sbr.PHASE_FP64)
    phi, delta = radar.f0 / C_LIGHT * L, radar.bandwidth / (C_LIGHT * ns) * L
    assert rel(cube[:, 0], reference(phi - np.round(phi), delta - np.round(delta), A, ns)) <= TOL


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("ns,nc,P", [(256, 4, 30000), (512, 4, 17000), (128, 2, 30000)])
def test_moving(sbr, ns, nc, P, kind):
    """Chirps in tiles (a grid in one block and in two) and in a group."""
    radar = radar_single_tx(ns, nc)
    rng = np.random.default_rng(P)
    delta, phi = rng.uniform(-0.5, 0.5, (4, P)), rng.uniform(-0.5, 0.5, (4, P))
    rate = rng.uniform(-8.0, 8.0, (4, P)).astype(np.float32)
    pairs(kind, delta, phi, rate)
    paths, phi, delta, A = bind(sbr, radar, P + 3, delta, phi, amplitudes(rng, kind, 4, P), rate)
    cube = sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | sbr.SYNTH_MOVING)
    assert torch.equal(cube, sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | sbr.SYNTH_MOVING))
    per = radar.chirp_rep / C_LIGHT
    ref = torch.stack([reference(phi + rate * (c * per * radar.f0), delta + rate * (c * per * radar.bandwidth / ns), A, ns)
                       for c in range(nc)], 1)
    assert rel(cube, ref) <= 2 * TOL


@pytest.mark.parametrize("what", ["inf", "nan", "phase", "rate"])
@pytest.mark.parametrize("ns,nc,P,mode", [(256, 1, 20000, "split"), (4096, 1, 5000, "split"), (256, 1, 3000, "fp64"),
                                          (256, 4, 17000, "moving"), (512, 4, 17000, "moving"), (128, 2, 3000, "moving")])
def test_not_finite(sbr, ns, nc, P, mode, what):
    """A record that is not finite makes its antenna's samples NaN, and no others, among amplitudes
    that need several classes."""
    radar = radar_single_tx(ns, nc)
    rng = np.random.default_rng(P)
    A = amplitudes(rng, "decades", 4, P)
    rate = rng.uniform(-8.0, 8.0, (4, P)).astype(np.float32)
    delta, phi = rng.uniform(-0.5, 0.5, (4, P)), rng.uniform(-0.5, 0.5, (4, P))
    L = rng.uniform(0.1, 0.999, (4, P)) * ns * C_LIGHT / radar.bandwidth
    if what == "rate" and mode != "moving":
        pytest.skip("no rates")
    {"inf": A, "nan": A, "phase": L if mode == "fp64" else phi, "rate": rate}[what][2, 1030] = \
        np.nan if what == "nan" else np.inf
    if mode == "fp64":
        paths = bind64(sbr, radar, P + 3, np.where(np.isfinite(L), L, 1.0), A)[0]
        if what == "phase":
            paths.phase_ofs()[:P].zero_()
            raw = paths.mem[paths.s.path_len - paths.mem.data_ptr():][:8 * 4 * (P + 3)].view(torch.float32)
            raw.view(4, P + 3, 2)[2, 1030, 0] = math.inf
        cube = sbr.synthesize(paths, radar, sbr.PHASE_FP64)
    else:
        paths = bind(sbr, radar, P + 3, delta, phi, A, rate)[0]
        cube = sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | (sbr.SYNTH_MOVING if mode == "moving" else 0))
    assert torch.isnan(cube[2]).all() and torch.isfinite(cube[[0, 1, 3]]).all()
