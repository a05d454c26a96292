"""The rows that a sweep's resampling takes, against the oracle's ancestors: up to 64 blocks of 256
particles every warp searches its ancestor by itself (k_resample_gather), above that one search kernel
does; and a step's first move takes the rows from where the gather left them."""
import numpy as np
import pytest

import oracle
from paper_1106_0322_gb300 import synth

pytestmark = pytest.mark.gpu

NU, C, SEED = 1.0, 0.05, 31


@pytest.fixture(scope="module")
def spa():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1106_0322_gb300 as mod

    return mod


def _ancestors(spa, region, N, p):
    """The prior draws of a sweep at scale C, and their ancestors under the likelihood's weights with the
    sweep's uniform (the first word of Philox block (0, 0, 0, tag 4), 24 bits)."""
    B = spa.prior_sample(SEED, NU, C, N, p)
    ll = region.loglik(B)
    lse, _ = spa.lse_ess(ll)
    u = (int(oracle.philox4x32_10([0, 0, 0, 4 << 16], [SEED, 0])[0]) >> 8) / 2.0 ** 24
    return B, oracle.resample_systematic(np.exp(ll - lse), u)


def _check(mean, B, anc):
    """The mean of N rows with weights 1/N: FP32 weights and products, compensated sums, so 4e-7 of the
    mean of |beta_j|. One row another changes it by about |beta_j| / N, 6e-5 at the largest N."""
    rows = B[anc].astype(np.float64)
    assert np.all(np.abs(mean - rows.mean(0)) <= 4e-7 * np.abs(rows).mean(0) + 1e-12)


SIZES = [1, 31, 255, 256, 257, 8191, 16384, 16385, 20000]


@pytest.mark.parametrize("p", [7, 8])
@pytest.mark.parametrize("N", SIZES)
def test_gathered_rows_are_the_oracles_ancestors(spa, N, p):
    reg = synth.make_region(60, p, 0.5, (0.5,), seed=2300)
    with spa.Region(reg.G, reg.y, NU, config=spa.make_config(move="rw", init="resample_move")) as r:
        B, anc = _ancestors(spa, r, N, p)
        assert N < 200 or len(np.unique(anc)) > N // 20  # (weights that tell the rows apart)
        out = r.run([C], N, 0, SEED)
    _check(out["mean"][0], B, anc)


# A first move none of whose proposals is accepted (steps 10^6 times as long) leaves the resampled rows.
@pytest.mark.parametrize("move,long", [("rw", {"rw_scale": 2.38e6}), ("mala", {"mala_h": 1.65e6})])
@pytest.mark.parametrize("p", [7, 8])
@pytest.mark.parametrize("N", SIZES)
def test_rows_taken_by_the_first_move_are_the_oracles_ancestors(spa, N, p, move, long):
    reg = synth.make_region(60, p, 0.5, (0.5,), seed=2300)
    with spa.Region(reg.G, reg.y, NU, config=spa.make_config(move=move, ess_frac=1.0, **long)) as r:
        B, anc = _ancestors(spa, r, N, p)
        out = r.run([C], N, 1, SEED)
    assert out["accept_rate"][0] == 0.0
    if N == 1:
        anc = np.zeros(1, np.int64)  # (one particle: its ESS is 1, nothing to resample)
    else:
        assert out["resampled"][0] == 1
    _check(out["mean"][0], B, anc)
