"""Antenna positions as sbr_radar_cfg takes them from a radar's tx and rx."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

TX = [[0.0, 0.0, 0.0], [0.0078, 0.001, 0.0], [0.0156, 0.0, -0.002]]
RX = [[0.00195 * k, 0.0, 0.0] for k in range(4)]


def filled(tx, rx):
    from paper_2311_13182_gb300 import sim
    r = sim.radar_struct(SimpleNamespace(f0=77e9, bandwidth=4e9, chirp_time=4e-5, chirp_rep=4e-5, n_samples=256,
                                         n_chirps=1, n_tx=3, n_rx=4, tx=tx, rx=rx))
    return [list(r.tx[t]) for t in range(3)], [list(r.rx[t]) for t in range(4)]


FORMS = dict(array=np.array, columns=lambda x: np.asfortranarray(np.array(x)), lists=lambda x: x, tuples=tuple,
             tensor=lambda x: torch.tensor(x, dtype=torch.float64),
             gradient=lambda x: torch.tensor(x, dtype=torch.float64, requires_grad=True),
             tensors=lambda x: [torch.tensor(p, dtype=torch.float64, requires_grad=True) for p in x],
             ragged=lambda x: [p + [9.0] * i for i, p in enumerate(x)], objects=lambda x: np.array(x, dtype=object),
             more=lambda x: np.array(x + [[7.0, 7.0, 7.0]]))


@pytest.mark.parametrize("form", sorted(FORMS))
def test_positions_from(form):
    assert filled(FORMS[form](TX), FORMS[form](RX)) == (TX, RX)


def test_single_precision_and_whole_numbers():
    assert filled(np.array(TX, dtype=np.float32), np.zeros((4, 3), dtype=np.int64))[0] == \
        np.array(TX, dtype=np.float32).astype(np.float64).tolist()


def test_too_few_positions():
    with pytest.raises(IndexError):
        filled(np.array(TX[:2]), np.array(RX))
    with pytest.raises(IndexError):
        filled(TX, RX[:3])


@pytest.mark.gpu
def test_positions_on_the_device():
    assert filled(torch.tensor(TX, dtype=torch.float64).cuda(), torch.tensor(RX, dtype=torch.float64).cuda()) == (TX, RX)
