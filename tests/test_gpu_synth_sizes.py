"""sbr_synthesize with several sample counts in one process, in any order."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SIZES = """
import sys
import torch
import paper_2311_13182_gb300 as sbr
from sbr_inputs import radar_single_tx

def cube(ns):
    paths = sbr.PathBuffers(4099, 1, 4)
    gen = torch.Generator(device="cuda").manual_seed(ns)
    paths.prep().copy_(torch.rand(4, 4099, 4, generator=gen, device="cuda"))
    paths.prep()[..., 1] = torch.round(paths.prep()[..., 1] * 4096) / 4096
    paths.prep()[..., 2] *= 2.0 ** -14
    paths.count_tensor().fill_(4099)
    return sbr.synthesize(paths, radar_single_tx(ns, 1))

first = {}
for ns in map(int, sys.argv[1:]):
    got = cube(ns)
    assert torch.equal(first.setdefault(ns, got), got) and float(got.norm()) > 0, ns
torch.cuda.synchronize()
"""


@pytest.mark.parametrize("sizes", [(4096, 2048, 4096, 1024, 2048, 4096), (1024, 4096, 32, 2048, 512, 4096, 256, 64, 512, 128, 256)])
def test_sample_counts_in_any_order(sizes):
    """Each size gives the same cube whatever sizes the process (a fresh one: the kernels' limits are
    set once in it) has asked for before, the longest again after shorter ones."""
    r = subprocess.run([sys.executable, "-c", SIZES, *map(str, sizes)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode == 0, r.stderr[-2000:]


def test_refused_sample_count_leaves_the_next_call_alone(sbr):
    """A sample count that is refused raises its own error, and no later call inherits one."""
    import torch
    from sbr_inputs import radar_single_tx
    paths = sbr.PathBuffers(3000, 1, 4)
    paths.mem.zero_()
    for ns in (16384, 16, 100):
        assert sbr.synth_ws_bytes(radar_single_tx(ns, 1), paths.cap) == 0
        with pytest.raises(Exception, match="n_samples"):
            sbr.synthesize(paths, radar_single_tx(ns, 1))
        assert float(sbr.synthesize(paths, radar_single_tx(1024, 1)).abs().max()) == 0.0
    torch.cuda.synchronize()


@pytest.mark.parametrize("ns,nc,P,fp64", [(256, 128, 20000, False), (256, 4, 600, False), (512, 16, 6000, False),
                                          (2048, 8, 700, True)])
def test_workspace_for_one_chirp_serves_many(sbr, ns, nc, P, fp64):
    """A buffer sized for one chirp is taken for any number: static (and its adjoint), the same
    result; moving, chirps one by one, within rounding of what the full buffer gives."""
    import ctypes

    import torch
    from paper_2311_13182_gb300 import _lib, sim
    from sbr_inputs import radar_mimo_3x4
    one, radar = radar_mimo_3x4(ns, 1), radar_mimo_3x4(ns, nc)
    paths = sbr.PathBuffers(P, 1, 12)
    gen = torch.Generator(device="cuda").manual_seed(P)
    paths.mem.zero_()
    paths.prep().copy_(torch.rand(12, P, 4, generator=gen, device="cuda"))
    paths.prep()[..., 1] = torch.round(paths.prep()[..., 1] * 4096) / 4096
    paths.prep()[..., 2] *= 2.0 ** -14
    paths.path_rate().copy_(torch.rand(12, P, generator=gen, device="cuda") * 16 - 8)
    paths.count_tensor().fill_(P)
    small, full = sbr.synth_ws_bytes(one, P), sbr.synth_ws_bytes(radar, P)
    assert small <= full
    mode = sbr.PHASE_FP64 if fp64 else sbr.PHASE_SPLIT

    def run(mode, nbytes):
        guard = torch.full((nbytes + 4096,), 7, dtype=torch.uint8, device="cuda")
        out = torch.empty((12, radar.n_chirps, ns, 2), device="cuda")
        r = sim.radar_struct(radar)
        _lib.call("sbr_synthesize", ctypes.byref(paths.s), ctypes.byref(r), mode, ctypes.c_void_p(out.data_ptr()),
                  ctypes.c_void_p(guard.data_ptr()), nbytes, sim._stream())
        assert bool((guard[nbytes:] == 7).all())
        return out

    assert torch.equal(run(mode, small), run(mode, full))
    a, b = run(mode | sbr.SYNTH_MOVING, small), run(mode | sbr.SYNTH_MOVING, full)
    assert float((a.double() - b.double()).norm() / b.double().norm()) <= 4e-6  # each within 2e-6 of the FP64 sum
    g = torch.rand(a.shape, generator=gen, device="cuda")
    ws = torch.empty(small, dtype=torch.uint8, device="cuda")
    for x, y in zip(sbr.synthesize_bwd(paths, radar, g, ws=ws), sbr.synthesize_bwd(paths, radar, g)):
        assert torch.equal(x[:, :P], y[:, :P])
