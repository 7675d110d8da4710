"""A song's results do not depend on the songs it shares a console with (GPU), at transforms so small that the block size
of the four-step passes used to follow the largest song of the launch."""
import numpy as np
import pytest

import workloads as W
from tests.cases import make_case, gpu_console

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("retain", [1, -1])
@pytest.mark.parametrize("fs,samples,log_n,log_n1", [(4000, 4201, 12, 6), (8000, 30011, 14, 7)])
def test_small_transforms_alone_and_in_a_batch(fs, samples, log_n, log_n1, retain):
    """Songs of 1 s at 4 kHz and 3.8 s at 8 kHz: reverb and delay transforms of 3 2^12 points (column tiles of 512 elements)
    and 3 2^14 (1,024), alone and beside a song whose tiles have 4,096.  The same bits: energies, dL/dw and with them
    every gradient come from sums of a fixed order."""
    lays = [W.SongLayout(2, 1, [0, -1], samples), W.SongLayout(1, 0, [-1], 400003)]
    batch = make_case(lays, types="dr", seed=31, n_fft=(256, 1024), fs=fs)
    sel = [p for p in batch.oracle.procs if p.song == 0]
    q0 = batch.oracle.n_proc_params
    idx = np.concatenate([np.arange(p.offset, p.offset + p.count) for p in sel] +
                         [q0 + np.array([p.index for p in sel])])
    alone = make_case(lays[:1], types="dr", seed=31, n_fft=(256, 1024), fs=fs)
    alone.sources, alone.targets = batch.sources[:1], batch.targets[:1]
    alone.noise = batch.noise[[p.rev for p in sel if p.type == "r"]]
    out = []
    for case, params, pick in ((batch, batch.params, idx), (alone, batch.params[idx], slice(None))):
        con = gpu_console(case, retain_spectra=retain)
        assert tuple(con.fft_sizes()[0]) == (3, log_n, log_n1)
        con.set_params(params)
        losses, mix = con.forward_loss(with_mix=True)
        con.backward()
        out.append((mix[0].cpu().numpy(), losses[0].cpu().numpy(), con.get_grads().cpu().numpy()[pick]))
        con.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
