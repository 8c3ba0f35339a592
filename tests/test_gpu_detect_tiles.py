"""The detector's tile kernel at its edges against the oracle: image sizes
around the 64 x 32 tile and the 32-pixel mask words, every filter radius class,
guard bands, and pixel values whose squares leave the range of a float.

Tolerance: the SNR map is an FP32 sum of (2 r + 1)^2 products against FP64,
1e-5 of its largest value; candidate lists agree except where the oracle's SNR
lies within that of the threshold or of a neighbour."""
import numpy as np
import pytest

from oracle import detect_oracle as DO

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,sigma,guard,scale", [
    (31, 31, 0.3, 0, 1.0), (32, 64, 1.0, 3, 1.0), (33, 65, 1.4, 0, 1.0), (63, 127, 2.0, 15, 1.0),
    (64, 129, 3.0, 5, 1.0), (95, 96, 5.0, 1, 1.0), (161, 193, 0.76, 5, 1.0), (70, 200, 1.0, 5, 1e-17),
    (70, 200, 1.0, 5, 1e19),
])
def test_detector_at_tile_edges(H, W, sigma, guard, scale):
    from paper_2603_08593_gb300 import Detector
    rng = np.random.default_rng(H * 1000 + W)
    D = rng.normal(0.3, 10.0, (H, W))
    yy, xx = np.mgrid[:H, :W]
    for _ in range(max(2, H * W // 900)):
        y, x = rng.uniform(0, H), rng.uniform(0, W)
        D += rng.uniform(60, 600) * np.exp(-((yy - y) ** 2 + (xx - x) ** 2) / (2 * max(sigma, 0.7) ** 2))
    D = (D * scale).astype(np.float32)
    D[rng.integers(0, H, 2), rng.integers(0, W, 2)] = [np.nan, np.inf]
    bad = (rng.random((H, W)) < 0.01).astype(np.uint8)
    S, R = (rng.normal(0, 1, (H, W)).astype(np.float32) for _ in range(2))
    o = DO.detect(D.astype(np.float64), S, R, bad, sigma, 4.0, guard=guard)
    det = Detector(H, W, batch=1, max_cand=512)
    t = lambda a: torch.from_numpy(a)[None].cuda()  # noqa: E731
    xy, snr, count, _ = det(t(D), t(S), t(R), t(bad), psf_sigma=sigma, thresh=4.0, guard=guard)
    torch.cuda.synchronize()
    if not o["sigma_D"] > 0:     # one interior pixel: no scatter, no candidate
        assert int(count[0]) == 0
        return
    m = det.snr_map[0].cpu().numpy().astype(np.float64)
    tol = 1e-5 * np.abs(o["snr_map"]).max()
    assert np.abs(m - o["snr_map"]).max() <= tol
    n = int(count[0])
    got = {tuple(p) for p in xy[0, :n].cpu().numpy().tolist()}
    want = set(zip(o["x"].tolist(), o["y"].tolist()))
    for x, y in got ^ want:
        box = o["snr_map"][max(0, y - 2):y + 3, max(0, x - 2):x + 3]
        v = o["snr_map"][y, x]
        near = np.sort(np.abs(box - v).ravel())[1] <= 2 * tol
        assert abs(v - 4.0) <= 2 * tol or near, (x, y, v)
    order = xy[0, :n].cpu().numpy()
    assert np.all(np.diff(order[:, 1].astype(np.int64) * W + order[:, 0]) > 0)
    assert np.array_equal(snr[0, :n].cpu().numpy(), m.astype(np.float32)[order[:, 1], order[:, 0]])
