"""CPU checks of the synthesis workspace's size query."""
import ctypes

import pytest


def radar(n_samples, n_chirps=1):
    from paper_2311_13182_gb300 import _lib
    r = _lib.RadarCfg()
    r.n_tx, r.n_rx, r.n_samples, r.n_chirps = 3, 4, n_samples, n_chirps
    r.f0, r.bandwidth, r.chirp_time, r.chirp_rep = 77e9, 4e9, 4e-5, 4e-5
    return r


def size(n_samples, cap, n_chirps=1):
    from paper_2311_13182_gb300 import _lib, build
    build.build()
    return _lib.load().sbr_synth_ws_bytes(ctypes.byref(radar(n_samples, n_chirps)), cap)


@pytest.mark.parametrize("n_samples", [-4096, 0, 1, 16, 33, 100, 4095, 8192, 32768, 65536, (1 << 30) + 1, (1 << 31) - 1])
def test_unsupported_sample_counts_have_no_workspace(n_samples):
    """Sample counts that no synthesis takes are answered at once, without asking the device."""
    from paper_2311_13182_gb300 import _lib
    assert size(n_samples, 1000) == 0
    if n_samples > 0:
        assert "n_samples" in _lib.last_error()


@pytest.mark.parametrize("n_samples", [32, 256, 512, 1024, 4096])
def test_workspace_grows_with_the_paths(n_samples):
    sizes = [size(n_samples, cap) for cap in (1, 1000, 100000, 1000000)]
    assert sizes[0] > 0 and sizes == sorted(sizes)


@pytest.mark.parametrize("n_samples", [256, 512, 4096])
def test_workspace_of_a_static_scene_does_not_grow_with_the_chirps(n_samples):
    """What a mode uses: one chirp's room without motion, more with it."""
    from types import SimpleNamespace

    import numpy as np
    from paper_2311_13182_gb300 import _lib, build, sim
    build.build()
    def rad(n_chirps):
        return SimpleNamespace(f0=77e9, bandwidth=4e9, chirp_time=4e-5, chirp_rep=4e-5, n_samples=n_samples,
                               n_chirps=n_chirps, n_tx=3, n_rx=4, tx=np.zeros((3, 3)), rx=np.zeros((4, 3)))
    one = sim.synth_ws_bytes(rad(1), 100000)
    assert sim.synth_ws_bytes(rad(128), 100000, 0) == one == size(n_samples, 100000)
    assert sim.synth_ws_bytes(rad(128), 100000) == size(n_samples, 100000, 128)
    assert sim.synth_ws_bytes(rad(128), 100000, _lib.SYNTH_MOVING) == size(n_samples, 100000, 128) >= one
