"""The two assemblies of the normal equations against each other: image-space
tap and mask-edge sums (the default) and row spectra (a set ccd_group), over
kernel sizes, degrees, odd shapes, mask forms and batches.

Tolerances: each side is held to the oracle at 1e-11 (FP64) and 2e-5 (mixed)
of max|A| and max|b| elsewhere, so the two differ by at most twice that."""
import numpy as np
import pytest

from synth import small_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda"


def _mask(kind, H, W, L, rng):
    bad = np.zeros((H, W), np.uint8)
    if kind == "specks":            # isolated bad pixels: as many mask edges as an erosion by L x L allows
        bad[L // 2::2 * L + 1, L // 2::2 * L + 1] = 1
    elif kind == "lines":           # bad rows and columns, also at the borders
        bad[:, rng.integers(0, W, 2)] = 1
        bad[rng.integers(0, H, 1), :] = 1
        bad[:, 0] = bad[0, :] = 1
    elif kind == "random":
        bad[rng.random((H, W)) < 0.004] = 1
    elif kind == "all":
        bad[:] = 1
    return bad


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,L,DK,DB,mask", [
    ((17, 16), 1, 0, 0, "random"), ((61, 45), 1, 2, 0, "random"), ((33, 129), 3, 1, 2, "specks"),
    ((64, 64), 3, 2, 1, "none"), ((70, 259), 5, 2, 2, "lines"), ((31, 33), 5, 0, 2, "none"),
    ((7, 16), 7, 0, 0, "none"), ((95, 127), 7, 0, 1, "specks"), ((131, 97), 7, 1, 0, "lines"),
    ((96, 385), 9, 2, 0, "specks"), ((64, 2048), 9, 1, 2, "random"), ((12, 16), 11, 1, 1, "none"),
    ((257, 200), 11, 2, 2, "specks"), ((160, 130), 11, 2, 1, "lines"), ((90, 120), 11, 0, 2, "all"),
])
def test_image_space_sums_match_spectra(prec, shape, L, DK, DB, mask):
    from paper_2603_08593_gb300 import Plan
    H, W = shape
    rng = np.random.default_rng(H * W + L)
    B = 2 if H * W < 20000 else 1
    imgs = [small_pair(H, W, seed=7000 + H + i) for i in range(B)]
    bad = np.stack([_mask(mask, H, W, L, rng) for _ in range(B)])
    R, S = (torch.from_numpy(np.stack([d[k] for d in imgs])).to(DEV) for k in "RS")
    bad = torch.from_numpy(bad).to(DEV)
    sky = torch.tensor([[1000.0, 1001.0]] * B, dtype=torch.float64, device=DEV)
    got = []
    for group in (0, B):
        p = Plan(H, W, L, DK, DB, batch=B, prec=prec, ccd_group=group)
        got.append(p.build_normal(R, S, bad, sky))
    torch.cuda.synchronize()
    tol = 4e-5 if prec == "mixed" else 2e-11
    for x, y in zip(*got):
        assert bool(torch.isfinite(x).all())
        assert float((x - y).abs().max()) <= tol * float(y.abs().max())
        if mask == "all":
            assert float(x.abs().max()) == 0.0

