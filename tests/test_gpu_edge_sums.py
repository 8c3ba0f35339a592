"""Mask-edge sums of the default mixed plan where the edge lists are long: many
thousand points per partial sum, in batches whose slots are few.

The reference is the FP64 plan of the same images, itself held to the oracle
at 1e-11; the tolerance is the mixed path's stated 2e-5 of max|A| and max|b|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda"
TOL = 2e-5


def _compare(R, S, bad, sky, L, DK, DB):
    from paper_2603_08593_gb300 import Plan
    B, H, W = R.shape
    A, b = Plan(H, W, L, DK, DB, batch=B, prec="mixed").build_normal(R, S, bad, sky)
    ref = Plan(H, W, L, DK, DB, batch=1, prec="fp64")
    for i in range(B):
        A64, b64 = ref.build_normal(*(t[i:i + 1].contiguous() for t in (R, S, bad, sky)))
        torch.cuda.synchronize()
        for x, y in ((A[i], A64[0]), (b[i], b64[0])):
            assert float((x - y).abs().max()) <= TOL * float(y.abs().max()), i


def test_equal_products_over_long_lists():
    """Bright rows of one value per CCD, in step with a mask of every twelfth
    row: for some offsets every rising edge adds the same product and every
    falling edge nothing, 10^4 of them per slot.  Added one after another in
    FP32 they lose up to 1e-4 of the sum."""
    B, H, W, L = 8, 1024, 2048, 11
    g = torch.Generator(device=DEV)
    g.manual_seed(12)
    value = torch.rand(B, 1, 1, generator=g, device=DEV) * 200.0 + 900.0
    R = torch.randn(B, H, W, generator=g, device=DEV)
    R[:, 3::12, :] = value
    S = torch.randn(B, H, W, generator=g, device=DEV)
    bad = torch.zeros(B, H, W, dtype=torch.uint8, device=DEV)
    bad[:, 6::12, :] = 1
    _compare(R, S, bad, torch.zeros(B, 2, dtype=torch.float64, device=DEV), L, 2, 2)


@pytest.mark.parametrize("L,DK,DB,period,kind", [(11, 2, 2, 12, "specks"), (11, 1, 2, 13, "rows"),
                                                 (9, 2, 0, 10, "specks"), (7, 2, 2, 8, "specks"), (7, 0, 1, 9, "rows"),
                                                 (11, 2, 2, 12, "columns")])
def test_dense_edges_in_a_batch(L, DK, DB, period, kind):
    """As many edges as an erosion by L x L allows, of sky noise with stars, for
    a batch of five (gy = 16 slots at least, 64 for the x edges)."""
    B, H, W = 5, 700, 1500
    g = torch.Generator(device=DEV)
    g.manual_seed(period + L)
    R, S = (1000.0 + 32.0 * torch.randn(B, H, W, generator=g, device=DEV) for _ in range(2))
    star = torch.rand(B, H, W, generator=g, device=DEV) > 0.995
    R, S = R + 4000.0 * star, S + 4000.0 * star
    bad = torch.zeros(B, H, W, dtype=torch.uint8, device=DEV)
    if kind == "specks":
        bad[:, L // 2::period, L // 2::period] = 1
    elif kind == "rows":
        bad[:, L // 2::period, :] = 1
    else:
        bad[:, :, L // 2::period] = 1
    sky = torch.tensor([[1000.0, 1001.0]] * B, dtype=torch.float64, device=DEV)
    _compare(R, S, bad, sky, L, DK, DB)


@pytest.mark.parametrize("shape,L,DK,period,kind", [((2048, 2048), 11, 2, 12, "specks"), ((2048, 2048), 11, 2, 12, "rows"),
                                                    ((2048, 2048), 7, 2, 8, "specks")])
def test_densest_masks_cost_no_more_than_spectra(shape, L, DK, period, kind):
    """The masks with the most edges: the default assembly against the spectral
    one, whose time does not depend on the mask (a set d_batch of every
    difference).  A tenth is allowed for the clock."""
    from paper_2603_08593_gb300 import Plan
    H, W = shape
    g = torch.Generator(device=DEV)
    g.manual_seed(period)
    R, S = (1000.0 + 32.0 * torch.randn(1, H, W, generator=g, device=DEV) for _ in range(2))
    bad = torch.zeros(1, H, W, dtype=torch.uint8, device=DEV)
    if kind == "specks":
        bad[:, L // 2::period, L // 2::period] = 1
    else:
        bad[:, L // 2::period, :] = 1
    ms = []
    for d_batch in (0, 4 * L * L):
        p = Plan(H, W, L, DK, DK, batch=1, prec="mixed", d_batch=d_batch)
        A, b = p.build_normal(R, S, bad)
        ev = []
        for _ in range(7):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            p.build_normal(R, S, bad, A=A, b=b)
            e[1].record()
            ev.append(e)
        torch.cuda.synchronize()
        ms.append(sorted(x.elapsed_time(y) for x, y in ev)[3])
    assert ms[0] <= 1.1 * ms[1], ms
