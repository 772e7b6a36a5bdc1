"""L_max = 0 (no forced retention; Eq. 5's second term off): the rule walked in
frame order by one CTA per stream, or, in larger pushes, followed along links
between reference frames, against the oracles (C for the histogram, Python for
the other signals) read the same way."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from oracle import scd_oracle as SC
from oracle import signals_oracle as SO

from tests.gpu_helpers import SCORE_RTOL, assert_parity, run_stream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _frames(w, h, T, seed, mean=9):
    return synth.generate(synth.medium(seed=seed).with_(width=w, height=h, frames=T, mean_scene_len=mean))


@pytest.mark.parametrize("bins,tau", [(32, 0.05), (32, 0.3), (7, 0.08), (256, 0.1), (1, 0.0), (32, 1.5)])
def test_histogram_rule_without_gap(bins, tau):
    from paper_2609_03675_gb300 import NGFF
    w, h, T = 64, 48, 700
    fr = _frames(w, h, T, seed=700 + bins)
    p = O.Params(w, h, bins=bins, tau=tau, l_max=0)
    want = O.load().run(fr, p)
    assert not (want[2] == O.KEEP_GAP).any()
    dev = torch.from_numpy(fr).cuda()
    for chunks in ([T], [1, 2, 63, 64, 65, 505], [1] * 40 + [T - 40]):
        f = NGFF(w, h, bins=bins, tau=tau, l_max=0, max_frames_per_push=1024)
        assert_parity(run_stream(f, dev, chunks), want, tau, f"bins {bins} chunks {chunks[:3]}")


def test_long_stream_many_tiles_and_host_frames():
    from paper_2609_03675_gb300 import NGFF
    w, h, T = 32, 24, 9000  # several 256-row shared-memory tiles per push
    fr = _frames(w, h, T, seed=711, mean=40)
    p = O.Params(w, h, tau=0.04, l_max=0)
    _, so, ko = O.load().run(fr, p)
    f = NGFF(w, h, tau=0.04, l_max=0, max_frames_per_push=T)
    s, k = f.push(torch.from_numpy(fr).pin_memory())  # host frames and outputs
    torch.cuda.synchronize()
    f.status()
    assert np.array_equal(k.numpy(), ko)
    assert (np.abs(s.numpy().astype(np.float64) - so) <= SCORE_RTOL * so).all()
    assert (ko != 0).sum() > 50 and (ko == 0).sum() > 50


@pytest.mark.parametrize("kind", [SO.LOWRES, SO.DHASH])
def test_spatial_signals_without_gap(kind):
    from paper_2609_03675_gb300 import NGFF
    w, h, T = 64, 48, 300
    fr = _frames(w, h, T, seed=720 + kind)
    tau = 0.03 if kind == SO.LOWRES else 0.1
    _, so, ko = SO.run(fr, O.Params(w, h, tau=tau, l_max=0), kind)
    f = NGFF(w, h, tau=tau, l_max=0, signal=kind)
    _, sg, kg = run_stream(f, torch.from_numpy(fr).cuda(), [100, 1, 199])
    assert np.array_equal(kg, ko)
    assert (np.abs(sg.astype(np.float64) - so) <= SCORE_RTOL * so).all()


def test_scene_change_signal_without_gap_and_state():
    from paper_2609_03675_gb300 import NGFF, NGFFError, _abi
    w, h, T = 64, 48, 400
    fr = _frames(w, h, T, seed=731, mean=15)
    p = O.Params(w, h, tau=0.35, l_max=0)
    hist = np.stack([O.load().histogram(x, p) for x in fr])
    sd = np.array([SC.l1(hist[t], hist[t - 1]) for t in range(1, T)]) / (2 * w * h)
    t_grad, t_cut = float(np.quantile(sd, 0.5)), float(np.quantile(sd, 0.97))
    so, ko = SC.select(hist, p, t_cut, t_grad)
    assert (ko == SC.KEEP_SCENE).any()
    dev = torch.from_numpy(fr).cuda()
    kw = dict(tau=0.35, l_max=0, signal=_abi.SIGNAL_SCD, scd_cut=t_cut, scd_gradual=t_grad)
    a = NGFF(w, h, **kw)
    s1, k1 = a.push(dev[:173])
    state = a.state_save()
    b = NGFF(w, h, **kw)
    b.state_load(state)
    s2, k2 = b.push(dev[173:])
    torch.cuda.synchronize()
    b.status()
    assert np.array_equal(torch.cat([k1, k2]).cpu().numpy(), ko)
    assert (np.abs(torch.cat([s1, s2]).cpu().numpy().astype(np.float64) - so) <= SCORE_RTOL * so).all()
    with pytest.raises(NGFFError) as e:
        NGFF(w, h, tau=0.35, l_max=0).shard_prepare(dev[:10], n_halo=0, t0=0)
    assert e.value.code == _abi.EINVAL


def test_batch_of_streams_without_gap():
    from paper_2609_03675_gb300 import NGFF
    w, h, S, T = 48, 32, 6, 120
    frs = [_frames(w, h, T, seed=740 + s, mean=6) for s in range(S)]
    f = NGFF(w, h, tau=0.06, l_max=0, max_streams=S)
    dev = [torch.from_numpy(x).cuda() for x in frs]
    outs = {s: [] for s in range(S)}
    for a, b in ((0, 50), (50, 51), (51, 120)):
        items = []
        for s in range(S):
            sc = torch.empty(b - a, dtype=torch.float32, device="cuda")
            kp = torch.empty(b - a, dtype=torch.uint8, device="cuda")
            items.append((s, dev[s][a:b], sc, kp))
            outs[s].append((sc, kp))
        f.push_batch(items)
    torch.cuda.synchronize()
    f.status()
    for s in range(S):
        _, so, ko = O.load().run(frs[s], O.Params(w, h, tau=0.06, l_max=0))
        assert np.array_equal(torch.cat([k for _, k in outs[s]]).cpu().numpy(), ko), f"stream {s}"


# Pushes on both sides of the single-kernel limit (384 frames, fewer with wide
# rows) and of its ways to share out the pairs (16 frames), of the links'
# tiles and staged rows (fewer with wide rows), and of the chain's passes of
# 4096 frames; a still stream, whose links run past the staged rows, between
# scenes; every frame kept.
@pytest.mark.parametrize("bins,tau,still", [(32, 0.06, 0), (32, 0.06, 700), (256, 0.2, 300), (6, 0.1, 150), (32, 0.0, 0),
                                            (64, 0.9, 0)])
@pytest.mark.parametrize("scd", [False, True])
@pytest.mark.parametrize("chunks", [[1, 16, 17, 7, 33, 2], [192, 193, 129, 64], [4096, 5], [3, 4097, 400],
                                    [257, 1300, 66], [384, 385, 380]])
def test_links_and_chain(chunks, bins, tau, still, scd):
    from paper_2609_03675_gb300 import NGFF, _abi
    w, h, T = 32, 8, sum(chunks)
    fr = _frames(w, h, T, seed=760 + bins + T, mean=7)
    for a in range(100, T, 2 * still) if still else ():
        fr[a:a + still] = fr[a]
    p = O.Params(w, h, bins=bins, tau=tau, l_max=0)
    kw = dict(bins=bins, tau=tau, l_max=0, max_frames_per_push=max(chunks))
    if scd:
        hist = np.stack([O.load().histogram(x, p) for x in fr])
        sd = np.array([SC.l1(hist[t], hist[t - 1]) for t in range(1, T)]) / (2 * w * h)
        sd = sd[sd > 0]
        t_grad, t_cut = float(np.quantile(sd, 0.6)), float(np.quantile(sd, 0.97))
        so, ko = SC.select(hist, p, t_cut, t_grad)
        kw.update(signal=_abi.SIGNAL_SCD, scd_cut=t_cut, scd_gradual=t_grad)
    else:
        _, so, ko = O.load().run(fr, p)
    f = NGFF(w, h, **kw)
    got = [f.push(part) for part in torch.split(torch.from_numpy(fr).cuda(), chunks)]
    torch.cuda.synchronize()
    f.status()
    kg = torch.cat([k for _, k in got]).cpu().numpy()
    assert np.array_equal(kg, ko), np.flatnonzero(kg != ko)[:10]
    assert (np.abs(torch.cat([s for s, _ in got]).cpu().numpy().astype(np.float64) - so) <= SCORE_RTOL * so).all()
    assert torch.equal(f.candidates().cpu(), torch.from_numpy(O.load().candidates(ko, 4).astype(np.int32)))


def test_batch_of_unequal_lengths_without_gap():
    from paper_2609_03675_gb300 import NGFF
    calls = [(0, 1, 65, 700), (9, 70, 0, 8), (512, 64, 3, 2), (1, 513, 3, 2)]  # of four streams, 512 frames each are walked
    frs = [_frames(32, 8, sum(c[s] for c in calls), seed=790 + s, mean=6) for s in range(4)]
    f = NGFF(32, 8, tau=0.06, l_max=0, max_streams=4)
    dev = [torch.from_numpy(x).cuda() for x in frs]
    outs = [(torch.empty(len(x), dtype=torch.float32, device="cuda"), torch.empty(len(x), dtype=torch.uint8, device="cuda"))
            for x in frs]
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
        _, so, ko = O.load().run(frs[s], O.Params(32, 8, tau=0.06, l_max=0))
        assert np.array_equal(outs[s][1].cpu().numpy(), ko), s
        assert (np.abs(outs[s][0].cpu().numpy().astype(np.float64) - so) <= SCORE_RTOL * so).all(), s


@pytest.mark.parametrize("bins,tau,apart", [(256, 3.0, 80), (256, 0.3, 80), (32, 3.0, 700), (32, 0.3, 700), (6, 3.0, 300),
                                            (256, 3.0, 5000)])
@pytest.mark.parametrize("chunks", [[9000], [4096, 4904], [300, 4200, 4500]])
def test_scenes_far_apart(chunks, bins, tau, apart):
    """Stills whose scenes lie further apart than the rows that are staged with
    a reference, so that nearly every link is scanned for: up to a scene
    change (no novelty at tau = 3), to a novelty keep, and on over the chain's
    passes of 4096 frames and from push to push."""
    from paper_2609_03675_gb300 import NGFF, _abi
    w, h, T = 32, 8, sum(chunks)
    fr = _frames(w, h, T, seed=820 + bins, mean=apart)
    for a in range(0, T, apart):
        fr[a:a + apart] = fr[a]
    fr[5::apart // 3, 0, 0] ^= 1  # a few small differences within the scenes
    p = O.Params(w, h, bins=bins, tau=tau, l_max=0)
    hist = np.stack([O.load().histogram(x, p) for x in fr])
    so, ko = SC.select(hist, p, 0.2, 0.1)
    assert (ko != 0).sum() > T // apart // 3
    f = NGFF(w, h, bins=bins, tau=tau, l_max=0, max_frames_per_push=max(chunks), signal=_abi.SIGNAL_SCD, scd_cut=0.2,
             scd_gradual=0.1)
    got = [f.push(part) for part in torch.split(torch.from_numpy(fr).cuda(), chunks)]
    torch.cuda.synchronize()
    f.status()
    kg = torch.cat([k for _, k in got]).cpu().numpy()
    assert np.array_equal(kg, ko), np.flatnonzero(kg != ko)[:10]
    assert (np.abs(torch.cat([s for s, _ in got]).cpu().numpy().astype(np.float64) - so) <= SCORE_RTOL * so).all()


def test_scan_time_grows_with_the_frames():
    """No frame is scanned for more than one reference: four times the frames
    with the same distance between scenes take about four times as long, not
    sixteen (as when every reference's scan ran to the end of the push)."""
    from paper_2609_03675_gb300 import NGFF, _abi
    w, h, apart, us = 32, 8, 80, []
    for T in (4096, 16384):
        f = NGFF(w, h, bins=256, tau=3.0, l_max=0, max_frames_per_push=T, signal=_abi.SIGNAL_SCD)
        still = torch.randint(0, 256, (T // apart + 1, h, w, 3), dtype=torch.uint8, device="cuda")
        fr = still.repeat_interleave(apart, dim=0)[:T].contiguous()
        out = dict(scores=torch.empty(T, device="cuda"), keep=torch.empty(T, dtype=torch.uint8, device="cuda"))
        times = []
        for _ in range(9):
            f.reset()
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            f.push(fr, **out)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        f.status()
        assert int((out["keep"] != 0).sum()) == (T + apart - 1) // apart
        us.append(sorted(times)[4])
    assert us[1] < 8 * us[0], us
