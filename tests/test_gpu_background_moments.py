"""Background block of A and b_B of the default mixed plan: moments of the fit
mask and of S over it.

They are plain sums of monomials, with FP64 sums over the rows and FP64 powers
of yt, so what is left is the FP32 rounding of the powers of xt and of a row's
sums over short groups: 2^-24 of the terms' size (of sqrt(A_qq A_q'q') for A,
of sqrt(A_qq) ||S'|| for b), which is the tolerance.  The reference is plain
FP64 on the CPU, from the eroded mask."""
import numpy as np
import pytest

from synth import small_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2.0 ** -24


@pytest.mark.parametrize("shape,L,DK,DB,sky", [((1024, 1024), 11, 2, 2, 1000.0), ((700, 1500), 5, 2, 2, 0.0),
                                               ((2048, 200), 7, 1, 2, 0.0), ((1000, 1000), 3, 1, 2, 0.0),
                                               ((33, 2048), 1, 0, 1, 1000.0), ((40, 16), 11, 0, 2, 1000.0)])
def test_background_moments_in_fp64_over_rows(shape, L, DK, DB, sky):
    from paper_2603_08593_gb300 import Plan
    H, W = shape
    d = small_pair(H, W, seed=6400 + H, mask_fraction=0.03)
    w = (L - 1) // 2
    good = (d["bad"] == 0) & np.isfinite(d["R"]) & np.isfinite(d["S"])
    M = np.zeros((H, W), bool)
    win = np.lib.stride_tricks.sliding_window_view(good, (L, L)).all(axis=(2, 3))
    M[w:H - w, w:W - w] = win
    xt, yt = (2.0 * np.arange(n) / (n - 1) - 1.0 for n in (W, H))
    ab = [(g - b, b) for g in range(DB + 1) for b in range(g + 1)]
    psi = np.stack([np.outer(yt ** b, xt ** a)[M] for a, b in ab])
    v = d["S"].astype(np.float64)[M] - sky
    A64, b64 = psi @ psi.T, psi @ v
    dev = [torch.from_numpy(np.ascontiguousarray(d[k]))[None].cuda() for k in ("R", "S", "bad")]
    sk = torch.full((1, 2), sky, dtype=torch.float64, device="cuda")
    A, b = Plan(H, W, L, DK, DB, batch=1, prec="mixed").build_normal(*dev, sk)
    torch.cuda.synchronize()
    n = len(ab)
    A, b = A[0, -n:, -n:].cpu().numpy(), b[0, -n:].cpu().numpy()
    size = np.sqrt(np.diag(A64))
    assert (np.abs(A - A64) / np.outer(size, size)).max() <= TOL
    assert (np.abs(b - b64) / (size * np.sqrt(v @ v))).max() <= TOL
