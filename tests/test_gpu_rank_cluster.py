"""GPU edge sizes of the clustered top-r selection: lengths around its lower limit and
around multiples of the cluster's 8 chunks, the longest keys' smem case aside; batches on
both sides of its one-CTA-per-SM rule; selections of 0, 1, T - 1 and T tokens; all keys
equal, ties that straddle the chunks, NaN, infinities and signed zeros.  Flags and slots
are compared with the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2608_28911_gb300 import synthetic

pytestmark = pytest.mark.gpu


def _check(s, n_high):
    import torch
    from paper_2608_28911_gb300 import semkv
    d = torch.device("cuda:0")
    h = torch.full(s.shape, 7, dtype=torch.uint8, device=d)
    slot = torch.full(s.shape, -1, dtype=torch.int32, device=d)
    semkv.semkv_rank_assign(torch.from_numpy(s).to(d), n_high, h, slot)
    torch.cuda.synchronize()
    want_h, want_slot = oracle.rank_assign(s, n_high)[:2]
    assert np.array_equal(h.cpu().numpy(), want_h)
    assert np.array_equal(slot.cpu().numpy().astype(np.int64), np.asarray(want_slot, np.int64))


@pytest.mark.parametrize("B,T,n_high", [
    (1, 8191, 2000), (1, 8192, 1), (2, 8193, 8192), (12, 8200, 2132), (13, 8200, 2132),
    (1, 20011, 0), (1, 20011, 20011), (3, 32777, 8522), (1, 131073, 131072),
])
def test_cluster_selection_edges(B, T, n_high):
    _check(synthetic.scores_zipf(40 + T % 97, B, T), n_high)


@pytest.mark.parametrize("kind", ["equal", "straddle", "special", "normal"])
def test_cluster_selection_values(kind):
    T = 9001
    rng = np.random.default_rng(8)
    if kind == "equal":
        s = np.full((2, T), 3.0, np.float32)
    elif kind == "straddle":
        s = np.where(rng.random((2, T)) < 0.7, 2.0, rng.integers(0, 5, (2, T))).astype(np.float32)
    elif kind == "special":
        s = rng.choice(np.array([np.nan, np.inf, -np.inf, 0.0, -0.0, 1.0, -1.0], np.float32), (2, T))
    else:
        s = rng.normal(30, 3, (2, T)).astype(np.float32)
    for n_high in (1, 2340, T - 1):
        _check(s, n_high)
