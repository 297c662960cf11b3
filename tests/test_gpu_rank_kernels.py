"""Every tile size of the ranking's scoring kernel.  A tile of 8 q candidates
occupies an SM, and the call takes the q whose rounds of tiles over the SMs cost
least, a tile costing q + 2: one round of q, an SM short of none, is always
cheaper than two or more of a smaller q, so 8 q SMs - 1 candidates (a ragged
last tile) select q on any GPU, and so does one candidate more than the next
smaller q covers in a round.

The scores agree with the float64 network to 1e-5: 256-term float32 sums of
terms of order 1/16 through tanh and softplus of slope at most 1, 2 x 256 x 6e-8
x 256 x (1/16)^2 = 3e-5 if every rounding were aligned, a square root of the
terms' number less where they are not (2e-6)."""
import numpy as np
import pytest

import oracle
from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu

Q = (2, 4, 8, 12, 14, 16)


@pytest.mark.parametrize("n_in", [3, 6])
@pytest.mark.parametrize("q", Q)
@pytest.mark.parametrize("edge", ["first", "last"])
def test_scores_and_selection_of_every_tile_size(n_in, q, edge):
    import torch
    import paper_2602_19699_gb300 as P
    P.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    C = 8 * q * sms - 1 if edge == "last" else (8 * Q[Q.index(q) - 1] * sms + 1 if q > 2 else 1)
    rng = np.random.default_rng(q)
    X = rng.normal(size=(C, n_in))
    w = W.std_critic_weights(n_in, seed=5)
    r = P.Ranker(n_in, w)
    N = max(1, C // 10)
    idx, sc = r.rank(X, N, want_scores=True)
    np.testing.assert_allclose(sc, oracle.std_critic(w, X), rtol=1e-5)
    np.testing.assert_array_equal(idx, np.sort(np.argsort(-sc, kind="stable")[:N]))
    r.close()
