"""Lifetime weights (Eq. calibration_lifetime): the early stop and the host threads
leave every value what the plain sum gives."""
import math

import numpy as np
import pytest

from paper_2609_38169_gb300 import api as A


@pytest.mark.parametrize("ell,H", [(0.0, 2048), (-1e-18, 64), (-1e-4, 2048), (math.log(0.9), 2048),
                                   (-5.0, 3), (-800.0, 2048), (0.01, 100)])
def test_lifetime_weight_is_the_whole_sum(ell, H):
    """Stopping once a term no longer changes the sum gives every term's sum, bit for bit."""
    total = 0.0
    for j in range(H):
        total += math.exp(2.0 * j * ell)
    assert A.stepq_lifetime_weight(ell, H) == total


def test_pivots_of_many_units_match_their_single_lifetimes():
    """Unit counts that spread the lifetimes over host threads (a remainder included)."""
    cfg = A.Config(n_layers=3, n_key_heads=7, n_value_heads=7, gate_kind=A.GATE_CHANNEL, n_pivots=40)
    g = np.random.default_rng(3)
    n = A.stepq_num_units(cfg)
    ell, dist = np.log(g.uniform(0.8, 0.999, n)), g.lognormal(size=(n, 4))
    risk = np.array([A.stepq_lifetime_weight(e, cfg.horizon) for e in ell]) * (dist[:, 1] - dist[:, 3])
    want = np.zeros(n, np.uint8)
    want[np.argsort(-risk, kind="stable")[:40]] = 1
    np.testing.assert_array_equal(A.stepq_select_pivots(cfg, ell, dist), want)
