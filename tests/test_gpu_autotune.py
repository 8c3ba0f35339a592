"""Plan-time tuning: the tiles that it reports reach a plan of the spectral
assembly that is given them, and give the same normal equations.

A plan-time tuning of which every candidate fails (the only candidate's first
device allocation is made to fail): an image-space plan, which runs without
the tuned tiles, is made and gives the fit; a plan of the spectral assembly is
refused and leaves nothing behind."""
import ctypes

import numpy as np
import pytest

from oracle import sfft_oracle as O
from synth import small_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# L = 1 has one difference, FP64 one choice of lag parts, fewer than 256 rows one band: a single candidate
H, W = 61, 67


def test_image_space_plan_survives_failed_tuning(monkeypatch):
    from paper_2603_08593_gb300 import Plan
    d = small_pair(H, W, seed=6300)
    ref = O.fit(d["R"], d["S"], d["bad"], 1, 0, 0)
    monkeypatch.setenv("SFFT_FAIL_ALLOC", "1")
    p = Plan(H, W, 1, 0, 0, batch=1, prec="fp64", autotune=1)
    monkeypatch.delenv("SFFT_FAIL_ALLOC")
    sky = torch.tensor([[ref["prep"]["s_R"], ref["prep"]["s_S"]]], dtype=torch.float64, device="cuda")
    o = p.subtract(*(torch.from_numpy(d[k])[None].cuda() for k in ("R", "S", "bad")), sky, refine=1)
    torch.cuda.synchronize()
    assert int(o["info"][0]) == 0
    th = o["theta"][0].cpu().numpy()
    assert np.abs(th - ref["theta_orig"]).max() <= 1e-8 * np.abs(ref["theta_orig"]).max()


def test_spectral_plan_still_reports_failed_tuning(monkeypatch):
    from paper_2603_08593_gb300 import binding
    lib = binding.load()
    before = lib.sfft_debug_live_allocations()
    desc = binding.Desc(H, W + 1, 1, 0, 0, 1, binding.PREC["fp64"], 1, 1, 0, 0, 0)
    h = ctypes.c_void_p()
    monkeypatch.setenv("SFFT_FAIL_ALLOC", "1")
    assert lib.sfft_plan(ctypes.byref(desc), None, ctypes.byref(h)) == binding.SFFT_ERR_CUDA
    assert h.value is None and lib.sfft_debug_live_allocations() == before


def test_tuned_tiles_run_in_a_spectral_plan():
    """The two assemblies of one pair, each within the stated 2e-5 of max|A|."""
    from paper_2603_08593_gb300 import Plan
    L, DK, DB = 5, 1, 1
    d = small_pair(300, 210, seed=6301, mask_fraction=0.02)
    dev = [torch.from_numpy(d[k])[None].cuda() for k in ("R", "S", "bad")]
    sky = torch.tensor([[1000.0, 1001.0]], dtype=torch.float64, device="cuda")
    pt = Plan(300, 210, L, DK, DB, batch=1, prec="mixed", autotune=1)
    ps = Plan(300, 210, L, DK, DB, batch=1, prec="mixed", d_batch=pt.tiles[0], rows_per_cta=pt.tiles[1],
              lag_parts=pt.tiles[2])
    assert ps.tiles == pt.tiles
    ps.profile()
    (A, b), (As, bs) = pt.build_normal(*dev, sky), ps.build_normal(*dev, sky)
    torch.cuda.synchronize()
    prof = ps.profile_read()
    assert prof["fft_prod"][1] > 0 and prof["fft_weights"][1] > 0      # it did form spectra
    assert float((A - As).abs().max()) <= 4e-5 * float(As.abs().max())
    assert float((b - bs).abs().max()) <= 4e-5 * float(bs.abs().max())
