"""The detector's clipped statistics keep FP64 precision: a difference image on a
pedestal of a million times its scatter, where the first pass's variance is what
is left of two numbers 4e12 times larger, and the clipping rule hands its error
on to the next passes.

sigma_D is read from the SNR map: the ratio of the oracle's map to the GPU's,
both of the same filter sums, whose FP32 roundings (fourteen, 2^-25 each) move
the median ratio by less than 5e-7; 2e-6 is allowed.  FP64 sums are off by 3e-7
here.  The sums themselves are read from the workspace and held to FP64 accuracy:
the block partials of the last pass against exact sums, where a thread's sums
are rounded to FP64 once and added in FP64 thirteen times (2^-53 each, of sums
that keep their sign: 2^-50 is allowed; pairs of floats are off by 5e-15)."""
import math

import numpy as np
import pytest

from oracle import detect_oracle as DO

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,pedestal", [(4096, 2048, 4.0e6), (4096, 2048, -4.0e6), (1024, 1024, 4.0e6),
                                          (1024, 1024, 3.0), (1024, 1024, 0.0)])
def test_sigma_on_a_pedestal(H, W, pedestal):
    from paper_2603_08593_gb300 import Detector
    rng = np.random.default_rng(H + int(abs(pedestal)))
    D = (rng.normal(0.0, 2.0, (H, W)) + pedestal).astype(np.float32)
    D.ravel()[rng.integers(0, H * W, H * W // 350)] += np.float32(9.0)       # a tail for the clipping passes
    sigma = DO.clipped_sigma(D.astype(np.float64))[1]
    want = DO.matched_snr(D.astype(np.float64), None, 1.0, sigma)
    det = Detector(H, W, batch=1, max_cand=16)
    t = torch.from_numpy(D)[None].cuda()
    det(t, t, t, None, psf_sigma=1.0, thresh=1e30)
    torch.cuda.synchronize()
    got = det.snr_map[0].cpu().numpy().astype(np.float64)
    big = np.abs(want) > 0.5 * np.abs(want[100:-100, 100:-100]).max()   # away from the borders' partial sums, or noise peaks
    assert abs(np.median(got[big] / want[big]) - 1.0) <= 2e-6


@pytest.mark.parametrize("H,W,mean", [(4096, 2048, 0.3), (1500, 1301, -25.0), (2048, 2048, 2000.0)])
def test_last_pass_sums_are_fp64_accurate(H, W, mean):
    from paper_2603_08593_gb300 import Detector
    rng = np.random.default_rng(H + W)
    D = rng.normal(mean, 10.0, (H, W)).astype(np.float32)
    det = Detector(H, W, batch=1, max_cand=16)
    t = torch.from_numpy(D)[None].cuda()
    det(t, t, t, None, psf_sigma=1.0, thresh=1e30)
    torch.cuda.synchronize()
    ws = det.ws_view.cpu().numpy()

    def align(n):
        return (n + 255) // 256 * 256
    # the SNR map, four sets of mask words, then [608][3] block sums and the interval they are of
    off = align(4 * H * W) + 4 * align(4 * H * ((W + 31) // 32))
    groups = ((W + 31) // 32 + 7) // 8
    part = ws[off:off + 608 * 24].view(np.float64).reshape(608, 3)[:min(608, H, (H * groups + 7) // 8)]
    shift, lo, hi = ws[off + align(608 * 24):][:12].view(np.float32).astype(np.float64)
    x = D[15:-15, 15:-15].astype(np.float64).ravel()
    x = x[(x >= lo) & (x <= hi)]
    d = x - shift                                      # exact: both are floats of neighbouring magnitude
    # squares as exact pairs of doubles
    hi_ = d.astype(np.float32).astype(np.float64)
    lo_ = d - hi_
    s2 = math.fsum(np.concatenate([hi_ * hi_, 2.0 * hi_ * lo_, lo_ * lo_]))
    n, g1, g2 = (math.fsum(part[:, k]) for k in range(3))
    assert n == x.size
    assert abs(g2 - s2) <= 2.0 ** -50 * s2
    assert abs(g1 - math.fsum(d)) <= 2.0 ** -50 * math.fsum(np.abs(d))
