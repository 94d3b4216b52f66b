"""sbr_synthesize on given path records against the same sum in FP64 (Eq. 8).

The records are seeded and written into the path buffers directly, so the comparison holds the
synthesis alone: sample counts over the whole range, record counts around the kernels' chunks
(256 threads, 1024 records), cells at the ends of the spreading grid and of its blocks.

Tolerance of the non-uniform FFT, relative L2 over the cube, rms contributions: carrier phase
rounded to 2^-25 cycles 1.1e-7, kernel polynomials and products 6e-8, aliasing 7e-8, terms
rounded to 2^-23 of twice the largest amplitude 2.6e-7 (amplitudes uniform in [0.1, 1]),
transform 1e-7: 3.3e-7 together; three times that is 1e-6."""
import math

import numpy as np
import pytest
import torch

from sbr_inputs import C_LIGHT, radar_mimo_3x4, radar_single_tx

pytestmark = pytest.mark.gpu

TOL = 1e-6


def bind64(sbr, radar, cap, L, A, rate=None):
    """Path buffers holding path lengths (float-float pairs) and strengths, for the FP64 phase."""
    P = L.shape[1]
    paths = sbr.PathBuffers(cap, 1, radar.n_virt)
    paths.prep()[:, :P, 3] = torch.from_numpy(A.astype(np.float32)).cuda()
    paths.phase_ofs().zero_()
    hi = L.astype(np.float32)
    at = paths.s.path_len - paths.mem.data_ptr()
    raw = paths.mem[at:at + 8 * radar.n_virt * cap].view(torch.float32).view(radar.n_virt, cap, 2)
    raw[:, :P] = torch.from_numpy(np.stack([hi, (L - hi).astype(np.float32)], -1)).cuda()
    if rate is not None:
        paths.path_rate()[:, :P] = torch.from_numpy(rate.astype(np.float32)).cuda()
    paths.count_tensor().fill_(P)
    return paths, paths.path_len().cpu().numpy()[:, :P], A.astype(np.float32).astype(np.float64)


def bind(sbr, radar, cap, delta, phi, A, rate=None):
    """Path buffers of ``cap`` slots per antenna holding the records (phi, delta in cycles, FP64)."""
    P = delta.shape[1]
    paths = sbr.PathBuffers(cap, 1, radar.n_virt)
    dhi = np.round(delta * 4096) / 4096
    rec = np.stack([phi, dhi, delta - dhi, A], -1).astype(np.float32)
    paths.prep()[:, :P] = torch.from_numpy(rec).cuda()
    if rate is not None:
        paths.path_rate()[:, :P] = torch.from_numpy(rate.astype(np.float32)).cuda()
    paths.count_tensor().fill_(P)
    rec = rec.astype(np.float64)
    return paths, rec[..., 0], rec[..., 1] + rec[..., 2], rec[..., 3]


def direct(phi, delta, A, ns):
    n = torch.arange(ns, dtype=torch.float64, device="cuda")
    out = []
    for p, d, a in zip(*(torch.from_numpy(x).cuda() for x in (phi, delta, A))):
        acc = torch.zeros(ns, dtype=torch.complex128, device="cuda")
        for s in range(0, len(p), 4096):
            x = p[s:s + 4096, None] + d[s:s + 4096, None] * n
            x = 2 * math.pi * (x - x.round())
            acc += (a[s:s + 4096, None] * torch.complex(x.cos(), x.sin())).sum(0)
        out.append(acc)
    return torch.stack(out)


def rel(cube, ref):
    got = torch.view_as_complex(cube.double().contiguous())
    return float((got - ref).norm() / ref.norm())


def records(seed, V, P, ns, where="all"):
    rng = np.random.default_rng(seed)
    delta = rng.uniform(-0.5, 0.5, (V, P))
    if where == "edges":  # cells at both ends of the grid and of its 1024-cell blocks, exact cell borders among them
        M = 2 * ns
        edge = np.concatenate([[0, M - 1, M // 2, M // 2 - 1], np.arange(1024, M, 1024), np.arange(1024, M, 1024) - 1])
        cell = rng.choice(edge, (V, P)) + rng.choice([0.0, 0.25, 1 - 2.0 ** -12], (V, P))
        delta = (cell / M + 0.5) % 1.0 - 0.5
    if where == "one":
        delta = np.full((V, P), 0.1234567)
    return delta, rng.uniform(-0.5, 0.5, (V, P)), rng.uniform(0.1, 1.0, (V, P)) * rng.choice([1, -1], (V, P))


@pytest.mark.parametrize("ns,P,where", [
    (32, 20000, "all"), (64, 16385, "edges"), (128, 17001, "all"), (256, 16384, "all"), (256, 16415, "edges"),
    (256, 150000, "one"), (256, 3 * 152 * 1024 + 1, "all"), (512, 20011, "edges"), (512, 16384, "all"),
    (1024, 2048, "edges"), (1024, 2047, "all"), (2048, 10007, "edges"), (4096, 2049, "all"), (4096, 70001, "edges"),
    (4096, 30000, "one")])
def test_split_records(sbr, ns, P, where):
    radar = radar_single_tx(ns, 1)
    delta, phi, A = records(ns + P, 4, P, ns, where)
    paths, phi, delta, A = bind(sbr, radar, P + 7, delta, phi, A)
    cube = sbr.synthesize(paths, radar)
    again = sbr.synthesize(paths, radar)
    assert torch.equal(cube, again)
    assert rel(cube[:, 0], direct(phi, delta, A, ns)) <= TOL


@pytest.mark.parametrize("nc,ns", [(1, 256), (4, 32), (16, 256), (128, 64), (8, 2048)])
def test_chirps_and_cube_alignment(sbr, nc, ns):
    """Every chirp of a static scene equal, in a cube that starts 8 bytes past a 16-byte boundary
    and in an aligned one."""
    radar = radar_single_tx(ns, nc)
    delta, phi, A = records(nc + ns, 4, 17000, ns)
    paths, phi, delta, A = bind(sbr, radar, 17000, delta, phi, A)
    n = 4 * nc * ns * 2
    buf = torch.full((n + 4,), 7.0, device="cuda")
    sbr.synthesize(paths, radar, out=buf[2:n + 2].view(4, nc, ns, 2))
    cube = sbr.synthesize(paths, radar)
    host = buf.cpu()
    assert torch.equal(host[2:n + 2].view(4, nc, ns, 2), cube.cpu()) and bool((cube == cube[:, :1]).all())
    assert bool((host[:2] == 7).all()) and bool((host[n + 2:] == 7).all())
    assert rel(cube[:, 0], direct(phi, delta, A, ns)) <= TOL


def test_split_records_not_finite(sbr):
    """A record that is not finite makes its antenna's samples NaN, and no others."""
    radar = radar_single_tx(256, 1)
    delta, phi, A = records(3, 4, 20000, 256)
    A[2, 17] = np.inf
    paths, _, _, _ = bind(sbr, radar, 20000, delta, phi, A)
    cube = sbr.synthesize(paths, radar)
    assert torch.isnan(cube[2]).all() and torch.isfinite(cube[[0, 1, 3]]).all()


@pytest.mark.parametrize("ns,nc,P", [(256, 16, 7001), (32, 2, 1025), (64, 128, 300), (128, 64, 2049), (512, 4, 5000),
                                     (32, 16, 5460), (64, 32, 5459), (128, 64, 6145), (512, 4, 5460), (512, 16, 7001)])
def test_moving_records(sbr, ns, nc, P):
    """Every chirp from its own delays: chirps in tiles (from 65,536 record slots) and in groups."""
    radar = radar_mimo_3x4(ns, nc)
    delta, phi, A = records(9 + ns, 12, P, ns)
    rate = np.random.default_rng(4).uniform(-8.0, 8.0, delta.shape).astype(np.float32)
    rate[:, ::5] = 0.0
    paths, phi, delta, A = bind(sbr, radar, P + 2, delta, phi, A, rate)
    cube = sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | sbr.SYNTH_MOVING)
    assert torch.equal(cube, sbr.synthesize(paths, radar, sbr.PHASE_SPLIT | sbr.SYNTH_MOVING))
    per = radar.chirp_rep / C_LIGHT
    ref = torch.stack([direct(phi + rate * (c * per * radar.f0), delta + rate * (c * per * radar.bandwidth / ns), A, ns)
                       for c in range(nc)], 1)
    # the chirp's phase shift (up to 10 cycles here), delta shift and turns are each rounded once more in FP32
    assert rel(cube, ref) <= 2 * TOL


@pytest.mark.parametrize("ns,P,moving", [(32, 1, False), (64, 1023, False), (256, 1025, True), (1024, 1024, False),
                                         (2048, 3001, True), (4096, 20000, False)])
def test_fp64_records(sbr, ns, P, moving):
    """The FP64 phase over delays of the whole unambiguous range, static and moving (4 chirps)."""
    radar = radar_single_tx(ns, 4 if moving else 1)
    rng = np.random.default_rng(ns)
    L = rng.uniform(0.1, 0.999, (4, P)) * ns * C_LIGHT / radar.bandwidth
    A = rng.uniform(0.1, 1.0, (4, P))
    rate = rng.uniform(-30.0, 30.0, (4, P)).astype(np.float32) if moving else None
    paths, L, A = bind64(sbr, radar, P + 3, L, A, rate)
    cube = sbr.synthesize(paths, radar, sbr.PHASE_FP64 | (sbr.SYNTH_MOVING if moving else 0))
    for c in range(radar.n_chirps):
        Lc = L + (c * radar.chirp_rep * rate if moving else 0.0)
        phi, delta = radar.f0 / C_LIGHT * Lc, radar.bandwidth / (C_LIGHT * ns) * Lc
        assert rel(cube[:, c], direct(phi - np.round(phi), delta - np.round(delta), A, ns)) <= TOL


@pytest.mark.parametrize("ns,nc,P,where", [
    (32, 8, 1, "all"), (64, 1, 50001, "edges"), (256, 1, 12288, "all"), (256, 1, 12289, "edges"), (256, 128, 255, "all"),
    (512, 4, 6200, "one"), (1024, 1, 257, "edges"), (2048, 16, 513, "all"), (4096, 1, 4099, "edges")])
def test_adjoint_records(sbr, ns, nc, P, where):
    """sbr_synthesize_bwd (dL/dlength, dL/dA, dL/dphase) on given records against FP64 sums."""
    radar = radar_single_tx(ns, nc)
    delta, phi, A = records(ns + P, 4, P, ns, where)
    paths, phi, delta, A = bind(sbr, radar, P + 5, delta, phi, A)
    gen = torch.Generator(device="cuda").manual_seed(P)
    gcube = torch.randn(4, nc, ns, 2, generator=gen, device="cuda")
    got = sbr.synthesize_bwd(paths, radar, gcube, phase=True)
    g = torch.view_as_complex(gcube.double()).sum(1)
    n = torch.arange(ns, dtype=torch.float64, device="cuda")
    k0, k1 = radar.f0 / C_LIGHT, radar.bandwidth / (C_LIGHT * ns)
    ref = torch.empty(3, 4, P, dtype=torch.float64, device="cuda")
    for v in range(4):
        p, d, a = (torch.from_numpy(x[v]).cuda() for x in (phi, delta, A))
        for s in range(0, P, 4096):
            x = p[s:s + 4096, None] + d[s:s + 4096, None] * n
            e = torch.polar(torch.ones_like(x), 2 * math.pi * (x - x.round()))
            z0, z1 = (e * g[v].conj()).sum(1), (e * (g[v].conj() * n)).sum(1)
            ref[0, v, s:s + 4096] = -2 * math.pi * a[s:s + 4096] * (k0 * z0.imag + k1 * z1.imag)
            ref[1, v, s:s + 4096] = z0.real
            ref[2, v, s:s + 4096] = -2 * math.pi * a[s:s + 4096] * z0.imag
    for x, y in zip(got, ref):
        assert float((x[:, :P].double() - y).norm() / y.norm()) <= TOL
