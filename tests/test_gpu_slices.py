"""The generic histogram kernel's slices: launches on both sides of each size at
which the slices change, bin counts on both sides of 64 and 128, frames that
K1 would take and frames that it would not, against the oracle's histograms."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (width, height), pushes in 16-pixel groups: a group short of, at and past a
# slice; 480,000 and 4,000,000 groups; five CTAs of 2048 groups per SM and one
# resident wave and an eighth of 152 SMs (760 and 1368 CTAs)
@pytest.mark.parametrize("bins", [32, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("w,h,frames", [(16, 255, 3), (16, 256, 3), (16, 257, 3), (48, 1025, 40), (160, 160, 300),
                                        (160, 161, 299), (333, 251, 400), (640, 360, 95), (640, 360, 96), (641, 359, 171),
                                        (640, 360, 172), (640, 360, 285)])
def test_histograms_across_the_slice_sizes(w, h, frames, bins):
    from paper_2609_03675_gb300 import NGFF
    rng = np.random.default_rng(w * h + bins)
    base = rng.integers(0, 256, (7, h, w, 3), dtype=np.uint8)
    base[5], base[6] = 255, 0
    want = np.stack([O.load().histogram(x, O.Params(w, h, bins=bins)) for x in base])
    pick = rng.integers(0, 7, frames)
    dev = torch.from_numpy(base).cuda()[torch.from_numpy(pick).cuda()]
    f = NGFF(w, h, bins=bins)
    for _ in range(2):  # the second finds the rows as the first left them
        _, _, hist = f.push(dev, return_hist=True)
        assert np.array_equal(hist.cpu().numpy().view(np.uint32), want[pick])
    f.status()


@pytest.mark.parametrize("bins", [16, 64, 65, 128])
@pytest.mark.parametrize("w,h,frames", [(640, 360, 69), (640, 360, 70), (3840, 2160, 2), (640, 360, 121), (640, 360, 122),
                                        (160, 160, 626)])
def test_histograms_around_the_even_shares(w, h, frames, bins):
    """1,000,000 groups, from which launches of fewer than five long slices per
    SM run in even shares, and 1,750,000, from which others do; frames too small
    for shares; 64 bins, up to which they are used."""
    test_histograms_across_the_slice_sizes(w, h, frames, bins)


def test_more_rows_than_a_grid_dimension():
    from paper_2609_03675_gb300 import NGFF
    w, h, T = 16, 2, 70001
    rng = np.random.default_rng(5)
    fr = rng.integers(0, 256, (T, h, w, 3), dtype=np.uint8)
    fr[1::2] = fr[0]
    _, so, ko = O.load().run(fr, O.Params(w, h, tau=0.4))
    f = NGFF(w, h, tau=0.4, max_frames_per_push=T)
    s, k = f.push(torch.from_numpy(fr).cuda())
    torch.cuda.synchronize()
    f.status()
    assert np.array_equal(k.cpu().numpy(), ko)
    assert np.all(np.abs(s.cpu().numpy().astype(np.float64) - so) <= 1e-6 * so)


@pytest.mark.parametrize("w,h,counts", [(640, 360, [1, 0, 30, 8, 91]), (640, 360, [18] * 9), (224, 224, [97, 500, 13]),
                                        (1920, 1080, [2, 7, 6])])
@pytest.mark.parametrize("bins", [32, 48, 128])
def test_even_shares_over_segments(w, h, counts, bins):
    """Batched calls of about one resident wave: shares that end inside frames
    and pass from one stream's frames to the next stream's, in other memory."""
    from paper_2609_03675_gb300 import NGFF
    rng = np.random.default_rng(sum(counts) + bins)
    base = rng.integers(0, 256, (5, h, w, 3), dtype=np.uint8)
    base[4] = 255
    p = O.Params(w, h, bins=bins, tau=0.02)
    f = NGFF(w, h, bins=bins, tau=0.02, max_streams=len(counts))
    src = torch.from_numpy(base).cuda()
    items, picks = [], []
    for s, n in enumerate(counts):
        pick = rng.integers(0, 5, n)
        picks.append(pick)
        items.append((s, src[torch.from_numpy(pick).cuda()], torch.empty(n, device="cuda"),
                      torch.empty(n, dtype=torch.uint8, device="cuda")))
    f.push_batch(items)
    torch.cuda.synchronize()
    f.status()
    for (s, _, sc, kp), pick in zip(items, picks):
        if len(pick):
            _, so, ko = O.load().run(base[pick], p)
            assert np.array_equal(kp.cpu().numpy(), ko), s
            assert np.all(np.abs(sc.cpu().numpy().astype(np.float64) - so) <= 1e-6 * so), s
