"""Equalizer tap adjoints beside the chain and on it (GPU): captured steps against passes on one stream, bit for bit, on every
side of the rule (subgroup equalizers before few and before many track blocks, with and without a scan between)."""
import numpy as np
import pytest

import workloads as W
from tests.cases import make_case, gpu_console

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("types,tracks,samples", [("e", 3, 6146), ("eg", 4, 88200), ("eg", 12, 88200), ("ecg", 12, 88200),
                                                  ("er", 2, 30011)])
def test_captured_equalizer_adjoints_against_one_stream(types, tracks, samples):
    case = make_case([W.SongLayout(tracks, 2, [k % 2 for k in range(tracks)], samples)], types=types, seed=26, n_fft=(512, 2048))
    con = gpu_console(case)
    out = []
    for serial in (False, True):
        con.set_profiling(serial)
        con.reset_optimizer()
        con.set_params(case.params)
        losses = [con.train_step().cpu().numpy().copy() for _ in range(3)]
        out.append(losses + [con.get_grads().cpu().numpy(), con.get_params().cpu().numpy()])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
