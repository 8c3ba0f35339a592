"""Readers of one model on several host threads: each gets its own vector.

The getters share a device buffer of the model in which a vector is put into
the C ABI's order, so a reader that is overtaken between its gather and its
copy would return another reader's values.  Weights, gradients and the
optimiser state are read at the same time, many times over, and each result is
compared bit for bit with the one read alone."""
import threading

import numpy as np
import pytest

from synth.stamps import make_stamps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["RBModel", "RIModel"])
def test_concurrent_readers_get_their_own_vectors(kind):
    import paper_2603_08593_gb300 as P
    m = getattr(P, kind)(max_batch=32, seed=3)
    d = make_stamps(32, seed=77)
    st = torch.from_numpy(np.ascontiguousarray(d["stamps"], dtype=np.float32)).cuda()
    y = torch.from_numpy((np.arange(32) % 2).astype(np.float32)).cuda()
    m.train_step(st, y, 1e-3)
    m.backward(st, y)
    torch.cuda.synchronize()
    want = {"w": m.get_weights(), "g": m.get_grads(), "s": m.get_state()[0]}
    assert np.array_equal(want["s"][:want["w"].size], want["w"])
    assert not np.array_equal(want["w"], want["g"])
    read = {"w": m.get_weights, "g": m.get_grads, "s": lambda: m.get_state()[0]}
    wrong, start = [], threading.Barrier(3)

    def reader(k):
        start.wait()
        for i in range(150):
            if not np.array_equal(read[k](), want[k]):
                wrong.append((k, i))

    ts = [threading.Thread(target=reader, args=(k,)) for k in read]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong, (len(wrong), wrong[:5])
