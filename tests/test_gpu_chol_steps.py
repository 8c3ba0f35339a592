"""The FP32 factorisation with a block step in one phase (few trailing tiles) and
in two (many CCDs): the arithmetic is the same, so the solutions are equal bit
for bit; and one residual step against the FP64 system leaves at most
(8 N 2^-24 kappa)^2 of the solution, kappa < 4 for these matrices.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# N = 246 and 300 with a ragged last block, 732; the first steps of these
# batches have more tiles than three CTAs per SM (two phases), the later ones
# fewer (one phase); the last batch keeps two phases to its last step but one
@pytest.mark.parametrize("L,DK,DB,batch", [(9, 1, 1, 20), (7, 2, 2, 24), (11, 2, 2, 3), (9, 1, 1, 200)])
def test_one_and_two_phase_steps_agree(L, DK, DB, batch):
    from paper_2603_08593_gb300 import Plan
    many = Plan(64, 64, L, DK, DB, batch=batch)
    one = Plan(64, 64, L, DK, DB)
    N = many.N
    assert N > 160               # past the single-CTA solver
    many.ws_view.zero_()         # sky constants 0: theta as solved
    one.ws_view.zero_()
    rng = np.random.default_rng(N)
    g = rng.normal(size=(N, 4 * N)) / np.sqrt(4 * N)
    base = g @ g.T + np.eye(N)   # eigenvalues in 1 + [0.25, 2.25]
    scale = 10.0 ** rng.uniform(-3, 3, (batch, N))
    A = base[None] * scale[:, :, None] * scale[:, None, :]
    b = rng.normal(size=(batch, N)) * scale
    dA, db = torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda()
    th, info = many.solve(dA, db, refine=0)
    assert not info.any()
    for c in {0, batch // 2, batch - 1}:
        t1, i1 = one.solve(dA[c:c + 1].contiguous(), db[c:c + 1].contiguous(), refine=0)
        assert not i1.any()
        assert torch.equal(t1[0], th[c])
        r = (A[c] @ th[c].cpu().numpy() - b[c]) / scale[c]
        assert np.linalg.norm(r) <= (8 * N * 2.0 ** -24 * 4) ** 2 * np.linalg.norm(b[c] / scale[c])
