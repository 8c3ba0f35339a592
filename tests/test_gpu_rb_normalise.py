"""Median and MAD of the stamp normalisation where the selection takes each of
its ways: a first probe that lands, probes that never land (two levels far
apart, where a result one rank off moves every pixel), ties, outliers that
spoil the first probe, values about zero, tiny and huge values, and non-finite
sums.  The bar is the one of the classifier's logits against the oracle with
BF16 operands: 1e-2 of the logits' RMS + 1e-4.
"""
import numpy as np
import pytest

from oracle import cnn_oracle as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _levels(rng, n, n_low):
    v = np.where(np.arange(961) < n_low, rng.random((n, 961)), 1000 + rng.random((n, 961)))
    return rng.permuted(v, axis=-1)


FORMS = {
    "noise": lambda rng, n: rng.normal(0, 1, (n, 961)),
    "sky": lambda rng, n: rng.normal(1000, 30, (n, 961)),
    "sorted": lambda rng, n: np.sort(rng.normal(-5, 2, (n, 961)), axis=-1),
    "median_below_gap": lambda rng, n: _levels(rng, n, 481),
    "median_above_gap": lambda rng, n: _levels(rng, n, 480),
    "ties": lambda rng, n: rng.integers(-2, 4, (n, 961)).astype(float),
    "one_value_but_one": lambda rng, n: np.where(np.arange(961) == 500, 7.0, np.full((n, 961), 3.0)),
    "outliers": lambda rng, n: rng.normal(0, 1, (n, 961)) * np.where(rng.random((n, 961)) < 0.2, 1e6, 1.0),
    "exponential": lambda rng, n: np.exp(rng.normal(0, 6, (n, 961))),
    "tiny": lambda rng, n: rng.normal(0, 1e-30, (n, 961)),
    "overflowing_mean": lambda rng, n: 3e38 - 1e37 * rng.random((n, 961)),
}


@pytest.mark.parametrize("form", FORMS)
def test_median_and_mad(form):
    from paper_2603_08593_gb300 import RBModel
    rng = np.random.default_rng(31)
    n = 8
    st = FORMS[form](rng, 3 * n).reshape(n, 3, 31, 31).astype(np.float32)
    p = C.init_params(4)
    m = RBModel(max_batch=n, seed=0)
    m.set_weights(C.flatten(p).astype(np.float32))
    z = m.logits(torch.from_numpy(st).cuda()).cpu().numpy().astype(np.float64)
    zb = C.forward_bf16(p, C.normalise(st.astype(np.float64)))
    rms = max(np.sqrt(np.mean(zb ** 2)), 1e-3)
    assert np.max(np.abs(z - zb)) <= 1e-2 * rms + 1e-4, (np.max(np.abs(z - zb)), rms)
