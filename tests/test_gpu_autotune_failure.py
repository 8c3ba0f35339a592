"""A plan-time tuning of which every candidate fails (the only candidate's first
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
