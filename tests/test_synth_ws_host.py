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
