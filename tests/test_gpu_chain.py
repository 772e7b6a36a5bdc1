"""The selection of larger pushes: tiles of frames linked by their gap maps.
Pushes around the tile sizes and around the number of tiles that a tile looks
back on, the rows of all lags staged at once and of some at a time, one and several mask words,
ring and state carried from push to push, and batches of unequal lengths,
against the oracle's single pass."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from tests.gpu_helpers import assert_parity, oracle_run, run_stream

pytestmark = pytest.mark.gpu

W, H = 32, 8


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _frames(T, seed=41, mean=9):
    return synth.generate(synth.medium(seed=seed).with_(width=W, height=H, frames=T, mean_scene_len=mean))


# 8 frames per tile up to 1216 on 152 SMs, 16 up to 2432, 32 beyond; a tile looks back on 128
PUSHES = [[65], [66, 72, 1], [1033, 1024], [1216, 1217], [2432, 70], [2433, 5000], [3, 9001]]


@pytest.mark.parametrize("bins,l_max,tau", [(32, 30, 0.15), (32, 1, 0.30), (7, 33, 0.20), (256, 60, 0.50), (32, 256, 0.35),
                                            (256, 256, 0.60), (256, 161, 0.50), (255, 250, 0.55),
                                            (4, 64, 2.0), (32, 30, 0.0)])
@pytest.mark.parametrize("sizes", PUSHES)
def test_pushes_match_the_oracle(sizes, bins, l_max, tau):
    from paper_2609_03675_gb300 import NGFF
    fr = _frames(sum(sizes))
    want = oracle_run(fr, O.Params(W, H, bins=bins, l_max=l_max, tau=tau))
    dev = torch.from_numpy(fr).cuda()
    f = NGFF(W, H, bins=bins, l_max=l_max, tau=tau, max_frames_per_push=max(sizes))
    assert_parity(run_stream(f, dev, sizes), want, tau, "with histograms")
    f.reset()
    got = [f.push(part) for part in torch.split(dev, sizes)]  # rows cleared by the selection itself
    torch.cuda.synchronize()
    f.status()
    assert np.array_equal(torch.cat([k for _, k in got]).cpu().numpy(), want[2])
    assert torch.equal(f.candidates().cpu(), torch.from_numpy(O.load().candidates(want[2], 4).astype(np.int32)))


@pytest.mark.parametrize("bins,l_max", [(32, 30), (256, 256)])
def test_batches_of_unequal_lengths(bins, l_max):
    from paper_2609_03675_gb300 import NGFF
    calls = [(0, 1, 65, 700), (9, 70, 0, 8), (130, 64, 3, 1500)]
    fr = [_frames(sum(c[s] for c in calls) or 1, seed=50 + s) for s in range(4)]
    tau = 0.2
    f = NGFF(W, H, bins=bins, l_max=l_max, tau=tau, max_streams=4)
    dev = [torch.from_numpy(x).cuda() for x in fr]
    outs = [(torch.empty(len(x), dtype=torch.float32, device="cuda"), torch.empty(len(x), dtype=torch.uint8, device="cuda"))
            for x in fr]
    at = [0] * 4
    for c in calls:
        items = []
        for s in range(4):
            a, b = at[s], at[s] + c[s]
            items.append((s, dev[s][a:b], outs[s][0][a:b], outs[s][1][a:b]))
            at[s] = b
        f.push_batch(items)
    torch.cuda.synchronize()
    f.status()
    for s in range(4):
        _, so, ko = oracle_run(fr[s], O.Params(W, H, bins=bins, l_max=l_max, tau=tau))
        assert np.array_equal(outs[s][1].cpu().numpy(), ko), s
        assert np.all(np.abs(outs[s][0].cpu().numpy().astype(np.float64) - so) <= 1e-6 * so), s


@pytest.mark.parametrize("bins,l_max", [(256, 30), (256, 64), (255, 30), (128, 33)])
@pytest.mark.parametrize("scd", [False, True])
def test_small_pushes_of_wide_rows(bins, l_max, scd):
    """Pushes of up to 64 frames whose rows with the walk's tables are a little
    under, at and over 48 KiB (15, 16 and 17 frames at 256 words, L_max = 30)."""
    from oracle import scd_oracle as SC
    from paper_2609_03675_gb300 import NGFF, _abi
    sizes = [3, 15, 16, 17, 1, 33, 64, 63]
    fr = _frames(sum(sizes), seed=61)
    p = O.Params(W, H, bins=bins, l_max=l_max, tau=0.5)
    kw = dict(bins=bins, l_max=l_max, tau=0.5)
    if scd:
        _, so, ko = SC.run(fr, p, 0.6, 0.2)
        kw.update(signal=_abi.SIGNAL_SCD, scd_cut=0.6, scd_gradual=0.2)
    else:
        _, so, ko = oracle_run(fr, p)
    f = NGFF(W, H, **kw)
    got = [f.push(part) for part in torch.split(torch.from_numpy(fr).cuda(), sizes)]
    torch.cuda.synchronize()
    f.status()
    assert np.array_equal(torch.cat([k for _, k in got]).cpu().numpy(), ko)
    assert np.all(np.abs(torch.cat([s for s, _ in got]).cpu().numpy().astype(np.float64) - so) <= 1e-6 * so)


# Few distances per frame, or several streams: the window and scan kernels on
# one side of a line, tiles on the other (500 and 8 x 152 frames of one stream,
# 800, 3000 and 9000 of several, none of them short).
@pytest.mark.parametrize("bins,l_max,calls", [
    (32, 1, [(499,), (500,), (1216,), (1217,)]), (64, 1, [(500,)]), (65, 1, [(500,)]), (2, 32, [(1216,), (1217,)]),
    (32, 30, [(66, 733), (67, 733), (300, 8700), (301, 8700)]), (32, 1, [(66, 433), (67, 433), (700, 9000)]),
    (256, 2, [(99, 2900), (100, 2900), (65, 735)]), (32, 33, [(400, 500)]),
    (64, 30, [(200, 5000), (3, 5000)])])  # and a later stream of more tiles than one looks back on
def test_pushes_around_the_choice_of_kernel(bins, l_max, calls):
    from paper_2609_03675_gb300 import NGFF
    S, tau = len(calls[0]), 0.25
    T = [sum(c[s] for c in calls) for s in range(S)]
    fr = [_frames(T[s], seed=90 + s) for s in range(S)]
    dev = [torch.from_numpy(x).cuda() for x in fr]
    outs = [(torch.empty(t, dtype=torch.float32, device="cuda"), torch.empty(t, dtype=torch.uint8, device="cuda")) for t in T]
    f = NGFF(W, H, bins=bins, l_max=l_max, tau=tau, max_streams=S, max_frames_per_push=10000)
    at = [0] * S
    for c in calls:
        items = []
        for s in range(S):
            a, b = at[s], at[s] + c[s]
            items.append((s, dev[s][a:b], outs[s][0][a:b], outs[s][1][a:b]))
            at[s] = b
        f.push_batch(items)
    torch.cuda.synchronize()
    f.status()
    for s in range(S):
        _, so, ko = oracle_run(fr[s], O.Params(W, H, bins=bins, l_max=l_max, tau=tau))
        assert np.array_equal(outs[s][1].cpu().numpy(), ko), s
        assert np.all(np.abs(outs[s][0].cpu().numpy().astype(np.float64) - so) <= 1e-6 * so), s


def test_streams_of_a_batch_are_decided_side_by_side():
    """A batched call of four streams runs one CTA per stream, on an SM each:
    it takes little longer than the same call for one of them, not twice as
    long (as when all four were placed on the first SM that came free)."""
    from paper_2609_03675_gb300 import NGFF
    n, us = 64, []
    for S in (1, 4):
        f = NGFF(64, 48, l_max=64, tau=0.15, max_streams=S)
        fr = torch.randint(0, 256, (S, n, 48, 64, 3), dtype=torch.uint8, device="cuda")
        out = [(torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")) for _ in range(S)]
        batch = f.make_batch([(s, fr[s], *out[s]) for s in range(S)])
        f.push_batch_raw(*batch)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(50):
                f.push_batch_raw(*batch)
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        f.status()
        us.append(sorted(times)[4] * 20)
    assert us[1] < 1.6 * us[0], us
