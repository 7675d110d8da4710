"""The kernels' and launch paths' edges: equalizer block boundaries, band layouts of the loss, imager + gain/pan pairs,
forwards that keep nothing for a backward, and passes on one stream against passes with side streams (GPU).

Against the FP64 oracle the bounds are test_gpu_parity.check's; between two routes of the library results are equal bit
for bit where the same sums run in the same order."""
import numpy as np
import pytest

import workloads as W
from tests.cases import make_case, gpu_console
from tests.test_gpu_parity import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("samples", [700, 6145, 6146, 6147, 12293, 18439])
def test_equalizer_at_its_block_edges(samples):
    """Overlap-save blocks of 6146 samples: less than one, one, one sample more, and odd last blocks.  The equalizer's y,
    du and dL/dh against 64-bit convolutions of what the console itself holds (taps, dL/dy, L_g's coefficients), so nothing
    but its own transforms is in the error: worst-case rounding of three radix-2 transforms of 8192 points,
    15 log2(N) 2^-24 = 1.2e-5 of the summed term magnitudes."""
    tol = 15 * 13 * 2.0 ** -24
    case = make_case([W.SongLayout(2, 0, [-1, -1], samples)], types="eg", seed=21, n_fft=(256, 512))
    con = gpu_console(case)
    con.set_params(case.params)
    con.forward_loss()
    con.backward()
    q = case.params[case.oracle.n_proc_params:].astype(np.float64)
    for p in case.oracle.procs:
        if p.type != "e":
            continue
        def read(what, cols):
            return con.debug_read(p.index, what, (2, cols)).astype(np.float64)
        u = np.repeat(np.asarray(case.sources[0][p.index // 2], np.float64)[None], 2, 0)
        h, dh, y, du, dy = read(1, 2047)[0], read(2, 2047), read(0, samples), read(3, samples), read(5, samples)
        c1, c2 = con.debug_read(p.index, 4, (1, 16))[0, 2:4].astype(np.float64)
        w = 1.0 / (1.0 + np.exp(-q[p.index]))

        def conv(x, f):
            return np.stack([np.convolve(x[c], f)[1023:1023 + samples] for c in range(2)])
        yb = conv(u, h)
        big = conv(np.abs(u), np.abs(h)) + np.abs(u)
        assert np.linalg.norm(y - (w * yb + (1 - w) * u)) <= tol * np.linalg.norm(big)
        g = w * dy + c1 * yb.sum(0)
        want = (1 - w) * dy + conv(g, h[::-1]) + c2 * u.sum(0)
        big = np.abs(dy) + conv(np.abs(w * dy) + np.abs(c1) * np.abs(u).sum(0) * np.abs(h).sum(), np.abs(h)) + np.abs(c2) * np.abs(u).sum(0)
        assert np.linalg.norm(du - want) <= tol * np.linalg.norm(big)

        def corr(a, b):   # sum_n a[n] b[n - j], j = -1023..1023
            return sum(np.convolve(np.pad(a[c], 1023), b[c][::-1])[samples - 1:samples + 2046] for c in range(2))
        big = corr(np.abs(w * dy) + np.abs(c1) * np.abs(yb).sum(0), np.abs(u))
        assert np.linalg.norm(dh[0] - corr(g, u)) <= tol * np.linalg.norm(big) and not dh[1].any()


@pytest.mark.parametrize("n_fft,n_mels", [((64, 256, 512), 5), ((512, 2048, 8192), 96), ((512, 2048, 8192), 24),
                                          ((256, 1024), 0)])
def test_loss_band_layouts(n_fft, n_mels):
    """Narrow and wide Mel bands, fewer than eight bands, linear bins."""
    check(make_case([W.SongLayout(2, 1, [0, -1], 20011)], types="gs", seed=22, n_fft=n_fft, n_mels=n_mels))


@pytest.mark.parametrize("drop", ["", "s", "g"])
def test_imager_and_gain_in_one_pass(drop):
    """Imagers followed by a gain/pan run as pairs; with every second one of a type pruned, pairs and single nodes stand side
    by side.  The pruned console equals the same console with the processors masked, and the adjoint between
    the two nodes of a pair, which is not stored, is read back as the gain/pan's dL/dy times its gains."""
    case = make_case([W.SongLayout(3, 1, [0, 0, -1], 9001)], types="sg", seed=23)
    keep = np.ones(len(case.ptypes), np.uint8)
    for k, i in enumerate(i for i, t in enumerate(case.ptypes) if t == drop):
        keep[i] = k % 2
    if not drop:
        check(case)
    con, masked = gpu_console(case), gpu_console(case)
    masked.set_params(case.params)
    want, wmix = masked.forward_loss(mask=keep, with_mix=True)
    if drop:
        con.prune(keep)
    con.set_params(case.params)
    losses, mix = con.forward_loss(with_mix=True)
    con.backward()
    assert np.array_equal(mix[0].cpu().numpy(), wmix[0].cpu().numpy())
    assert np.array_equal(losses.cpu().numpy()[0, :4], want.cpu().numpy()[0, :4])
    q = case.params[case.oracle.n_proc_params:].astype(np.float64)
    for p in case.oracle.procs:
        if p.type != "g" or not (keep[p.index] and keep[p.index - 1]):
            continue
        dy, du = con.debug_read(p.index, 5, (2, 9001)), con.debug_read(p.index, 3, (2, 9001))
        w = 1.0 / (1.0 + np.exp(-q[p.index]))
        k = (1.0 - w) + w * np.exp(case.params[p.offset:p.offset + 2].astype(np.float64))
        assert np.abs(du - k[:, None] * dy).max() <= 1e-6 * np.abs(du).max()
        assert np.array_equal(du, con.debug_read(p.index - 1, 5, (2, 9001)))


@pytest.mark.parametrize("retain", [1, -1])
def test_masked_forward_keeps_nothing_and_gives_the_same(retain):
    case = make_case([W.SongLayout(2, 1, [0, -1], 30011)], seed=24)
    con = gpu_console(case, retain_spectra=retain)
    con.set_params(case.params)
    a, ma = con.forward_loss(mask=np.ones(len(case.ptypes), np.uint8), with_mix=True)
    with pytest.raises(Exception):
        con.backward()
    b, mb = con.forward_loss(with_mix=True)
    con.backward()
    assert np.array_equal(ma[0].cpu().numpy(), mb[0].cpu().numpy())
    assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())


@pytest.mark.parametrize("retain", [1, -1])
def test_side_streams_against_one_stream(retain):
    """Per-launch timing keeps every kernel on the console's stream, one after the other: losses and gradients of eager
    passes and of captured steps are the same bits.  Songs of 0.4 and 6 s give the four-step passes several sizes."""
    lays = [W.SongLayout(2, 1, [0, -1], 17001), W.SongLayout(4, 2, [0, 1, 0, 1], 264001)]
    case = make_case(lays, seed=25)
    con = gpu_console(case, retain_spectra=retain)
    out = []
    for serial in (False, True):
        con.set_profiling(serial)
        con.set_params(case.params)
        for _ in range(2):
            losses = con.forward_loss()
            con.backward()
        out.append([losses.cpu().numpy(), con.get_grads().cpu().numpy()])
        con.reset_optimizer()
        con.set_params(case.params)
        for _ in range(3):
            con.train_step()
        out[-1] += [con.get_params().cpu().numpy()]
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("drop", ["", "s", "g"])
def test_gradients_of_pairs_beside_single_nodes(drop):
    """The console of the test before, pairs and single nodes side by side: gradients against the FP64 oracle under the same
    mask (a masked processor's gradients are zero, as a pruned one's read), and the adjoint that every imager writes against
    its closed form from the adjoint that it reads, within 16 roundings of the summed magnitudes."""
    import torch
    from tests.cases import grad_groups, rel_l2
    case = make_case([W.SongLayout(3, 1, [0, 0, -1], 9001)], types="sg", seed=23)
    keep = np.ones(len(case.ptypes), np.uint8)
    for k, i in enumerate(i for i, t in enumerate(case.ptypes) if t == drop):
        keep[i] = k % 2
    x = torch.tensor(np.asarray(case.params, np.float64), requires_grad=True)
    sum(r["total"] for r in case.oracle.forward(x, mask=keep, alpha_p=1e-3)).backward()
    con = gpu_console(case)
    if drop:
        con.prune(keep)
    con.set_alpha_p(1e-3)
    con.set_params(case.params)
    con.forward_loss()
    con.backward()
    got = con.get_grads().cpu().numpy()
    for name, idx in grad_groups(case).items():
        assert rel_l2(got[idx], x.grad.numpy()[idx]) <= 1e-3, name
    q = case.params[case.oracle.n_proc_params:].astype(np.float64)
    for p in case.oracle.procs:
        if p.type != "s" or not keep[p.index]:
            continue
        g, du = con.debug_read(p.index, 5, (2, 9001)).astype(np.float64), con.debug_read(p.index, 3, (2, 9001))
        w, e = 1.0 / (1.0 + np.exp(-q[p.index])), np.exp(np.float64(case.params[p.offset]))
        mid, side = 0.5 * w * (g[0] + g[1]), 0.5 * w * e * (g[0] - g[1])
        want = np.stack([(1 - w) * g[0] + mid + side, (1 - w) * g[1] + mid - side])
        big = (1 - w) * np.abs(g) + 0.5 * w * (1 + e) * np.abs(g).sum(0)
        assert (np.abs(du - want) <= 16 * 2.0 ** -24 * big).all(), p.index
