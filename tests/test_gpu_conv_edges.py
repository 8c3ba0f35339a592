"""The convolution kernel where its loads and boxes change: kernels of one and
three pixels (L = 1 runs in a box of three), images of several tiles each way
with every pair summed over the image, and images that do not start on a
16-byte boundary although their rows are whole groups of four.

Fits are held to the oracle at the mixed path's stated errors.  Loading four
pixels at once or one by one changes no arithmetic: the results are the same
bits."""
import numpy as np
import pytest

from oracle import sfft_oracle as O
from synth import SIGMA_SKY, small_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda"


def _fit(d, ref, L, DK, DB, prec, refine, **kw):
    from paper_2603_08593_gb300 import Plan
    H, W = d["R"].shape
    p = Plan(H, W, L, DK, DB, batch=1, prec=prec, **kw)
    sky = torch.tensor([[ref["prep"]["s_R"], ref["prep"]["s_S"]]], dtype=torch.float64, device=DEV)
    o = p.subtract(*(torch.from_numpy(np.ascontiguousarray(d[k]))[None].to(DEV) for k in ("R", "S", "bad")), sky,
                   refine=refine)
    torch.cuda.synchronize()
    assert int(o["info"][0]) == 0
    return o["theta"][0].cpu().numpy(), o["D"][0].cpu().numpy()


@pytest.mark.parametrize("shape,L,DK,DB", [((61, 45), 1, 2, 2), ((33, 16), 1, 0, 0), ((300, 700), 1, 2, 1),
                                           ((300, 701), 3, 2, 2), ((257, 515), 5, 2, 2)])
@pytest.mark.parametrize("spectral", [False, True])
def test_small_kernels_match_oracle(shape, L, DK, DB, spectral):
    d = small_pair(*shape, seed=6500 + shape[1] + L, mask_fraction=0.03)
    ref = O.fit(d["R"], d["S"], d["bad"], L, DK, DB)
    kw = dict(d_batch=4 * L * L) if spectral else {}
    for refine in (0, 1):
        th, D = _fit(d, ref, L, DK, DB, "mixed", refine, **kw)
        assert O.kernel_coef_rel_err(th, ref["theta_orig"], L, DK, DB) <= 1e-5
        assert np.abs(D - ref["D"]).max() <= 1e-3 * SIGMA_SKY
    th, D = _fit(d, ref, L, DK, DB, "fp64", 1, **kw)
    assert np.abs(th - ref["theta_orig"]).max() <= 1e-8 * np.abs(ref["theta_orig"]).max()
    assert np.all(np.abs(D - ref["D"]) <= 2.0 ** -24 * np.abs(ref["D"]) + 1e-7 * SIGMA_SKY)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,L,DK", [((70, 132), 7, 2), ((40, 300), 1, 1), ((130, 256), 11, 2)])
def test_images_off_a_16_byte_boundary(prec, shape, L, DK):
    from paper_2603_08593_gb300 import Plan
    H, W = shape
    d = small_pair(H, W, seed=6600 + W, mask_fraction=0.02)
    sky = torch.tensor([[1000.0, 1001.0]], dtype=torch.float64, device=DEV)
    p = Plan(H, W, L, DK, 1, batch=1, prec=prec)
    out = []
    for off in (0, 1, 3):
        def at(a):
            buf = torch.zeros(H * W + 4, dtype=torch.from_numpy(a).dtype, device=DEV)
            v = buf[off:off + H * W].view(1, H, W)
            v.copy_(torch.from_numpy(a)[None])
            return v
        R, S, bad, D, D2 = (at(x) for x in (d["R"], d["S"], d["bad"], np.zeros((H, W), np.float32),
                                            np.zeros((H, W), np.float32)))
        assert R.data_ptr() % 16 == 4 * off
        o = p.subtract(R, S, bad, sky, refine=1, out={"D": D})
        p.apply(R, S, o["theta"], sky, D=D2)
        torch.cuda.synchronize()
        assert int(o["info"][0]) == 0
        out.append([o["A"].clone(), o["theta"].clone(), D.clone(), D2.clone()])
    for other in out[1:]:
        for x, y in zip(out[0], other):
            assert torch.equal(x, y)
