"""The rotation-invariant inference stack at the edges of its persistent grid:
fewer images than CTAs, one image more than a round, several rounds.  Every
stamp's logit is that of the oracle's BF16 operand model (the bar of the other
classifier tests) and does not depend on the batch it came in: a stamp's
products and sums are the same whichever CTA and round takes it, so the values
are equal bit for bit."""
import numpy as np
import pytest

from oracle import cnn_oracle as C
from synth.stamps import make_stamps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 37, 38, 39, 153])
def test_stack_is_independent_of_the_batch(n):
    from paper_2603_08593_gb300 import RIModel
    stamps = make_stamps(n, seed=900 + n)["stamps"]
    st = torch.from_numpy(np.ascontiguousarray(stamps, dtype=np.float32)).cuda()
    p = C.init_params_ri(3)
    m = RIModel(max_batch=160, seed=0)
    m.set_weights(C.flatten_ri(p).astype(np.float32))
    whole = m.logits(st).cpu().numpy()
    parts = np.concatenate([m.logits(st[i:i + 7].contiguous()).cpu().numpy() for i in range(0, n, 7)])
    assert np.array_equal(whole, parts)
    few = list(range(0, n, max(1, n // 5)))[:5]
    zb = C.forward_ri_bf16(p, C.normalise(stamps[few].astype(np.float64)))
    assert np.abs(whole[few] - zb).max() <= 1e-2 * max(1.0, np.sqrt(np.mean(zb ** 2)))
