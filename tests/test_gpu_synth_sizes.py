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
