"""Kernel variants chosen by size, at the edges of their ranges, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1106_0322_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spa():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1106_0322_gb300 as mod

    return mod


# The single-coordinate cycle keeps eta in registers for n <= 2048 (4 to 64 individuals per
# lane, in steps of 4) and in shared memory above; updates go 32 at a time.
@pytest.mark.parametrize("n,p,N", [(31, 1, 3), (33, 5, 64), (128, 32, 65), (129, 33, 64), (500, 20, 33), (1536, 6, 64),
                                   (1537, 6, 64), (2048, 7, 64), (2049, 7, 64)])
def test_site_register_and_shared_kernels_at_their_edges(spa, n, p, N):
    """With one seed both sides draw the same Philox blocks, so the first step's updates take
    the same decisions except where a log ratio lies within the kernels' rounding (about 1e-5)
    of log U. A flipped update moves one of N p acceptances, and one particle's coordinate by
    about one proposal step (0.5 sd) with its weight of order 1/N; up to two flips are allowed."""
    reg = synth.make_region(n, p, 0.9, (0.5,), seed=1200 + n)
    sched = synth.geometric_schedule(2, -3.0, -2.0)
    with spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(move="site", init="resample_move")) as r:
        g = r.run(sched, N, 1, 11)
    o = oracle.run(reg.G, reg.y, 1.0, sched, N, 1, seed=11,
                   cfg=oracle.make_config(move="site", init="mcmc"))
    assert abs(g["accept_rate"][0] - o["accept_rate"][0]) <= 2.0 / (N * p) + 1e-12
    assert np.max(np.abs(g["mean"][0] - o["mean"][0])) <= 2 * 2.0 / N + 1e-4


# A MALA sweep evaluates likelihood and gradient in one kernel when p <= 255; a batch's regions
# run the residual pass and the adjoint as two kernels. Edges: k-blocks (p + 1 mod 64, narrow last
# ones), marker tiles (16, 128, 208, 255), 32-, 64- and 128-individual tiles, K-splits 1 to 8.
@pytest.mark.parametrize("n,p,N", [(31, 1, 5), (63, 15, 130), (64, 16, 300), (65, 31, 1100), (127, 32, 700),
                                   (128, 63, 900), (129, 64, 2600), (191, 95, 3000), (257, 127, 520), (640, 128, 5000),
                                   (700, 129, 1000), (900, 191, 390), (1000, 207, 2100), (1100, 208, 260),
                                   (600, 223, 640), (513, 224, 770), (2111, 255, 1500), (96, 40, 20000)])
def test_gradient_kernel_gives_the_two_kernels_bits(spa, n, p, N):
    reg = synth.make_region(n, p, 0.9, (0.4, -0.3), seed=1300 + n)
    sched = synth.geometric_schedule(3, -4.0, -1.0)
    with spa.Region(reg.G, reg.y, 2.0, config=spa.make_config(move="mala")) as r:
        one = r.run(sched, N, 2, 5)
        b = spa.Batch([r], [sched], [N], [2], [5])
        (two,) = b.run()
        b.close()
        for k in one:
            assert np.array_equal(one[k], two[k]), k


# One EM solve keeps the genotypes in registers for n <= 512 and p <= 64, a warp's markers (16
# warps) in groups of 1, 2 or 4; larger problems read them in both products.
@pytest.mark.parametrize("n,p", [(40, 1), (97, 15), (511, 16), (512, 17), (300, 32), (512, 33), (512, 64), (513, 33),
                                 (512, 65)])
def test_map_register_and_general_kernels_at_their_edges(spa, n, p):
    """The double-exponential mode is unique, so the oracle's is the same point; the tolerances are
    those of the FP32 inner solves (a last step below 1e-7 at a contraction no worse than 1e-4)."""
    reg = synth.make_region(n, p, 0.5, (0.5,), seed=1400 + n)
    start = np.random.default_rng(n + p).normal(0, 0.1, (1, p)).astype(np.float32)
    with spa.Region(reg.G, reg.y, np.inf) as r:
        g, glp = r.map(start, 0.05, max_em=100, tol=1e-6)
    o, olp = oracle.map_em(reg.G, reg.y, np.inf, 0.05, start[0].astype(np.float64), max_em=100, tol=1e-10)
    assert np.max(np.abs(g[0] - o)) < 2e-3 * max(1.0, np.max(np.abs(o)))
    assert abs(glp[0] - olp) < 1e-4 * abs(olp) + 1e-3


# The plain FP32 products run in tiles of 32 x 64, 64 x 64 or 128 x 128 (particles by individuals,
# then particles by markers), 16 of the summed dimension at a time.
@pytest.mark.parametrize("n,p,N", [(31, 1, 3), (64, 16, 32), (65, 17, 33), (129, 15, 64), (641, 33, 1030),
                                   (1000, 100, 4096), (999, 101, 4095), (300, 500, 8191)])
def test_plain_fp32_tiles_at_their_edges(spa, n, p, N):
    """FP32 sums of at most 1000 terms: 1e-5 of the log-likelihood, 1e-5 of sum_i |x_ij| for the
    gradient (FP32 rounding 6e-8 a term, and r's error of a quarter of eta's)."""
    reg = synth.make_region(n, p, 0.9, (0.4,), seed=1500 + n)
    B = synth.random_particles(N, p, 0.05, seed=p)
    with spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(precision="fp32")) as r:
        l = r.loglik(B)
        ll, g = r.grad(B, 0.0)
    o_ll, o_g = oracle.loglik_grad(reg.G, reg.y, B.astype(np.float64))
    assert np.all(np.abs(l - o_ll) <= 1e-5 * np.abs(o_ll))
    assert np.all(np.abs(ll - o_ll) <= 1e-5 * np.abs(o_ll))
    scale = np.abs((reg.G - reg.G.mean(0)) / reg.G.std(0)).sum(0)
    assert np.all(np.abs(g - o_g) <= 1e-5 * scale[None, :])


# The summaries kernel is compiled for up to 4 quantile levels and 2 thresholds, and for 8 and 8;
# 512 threads read 4 (then 8) values each at a time.
@pytest.mark.parametrize("N", [1, 31, 511, 513, 2048, 2051, 4096, 5003])
def test_summary_kernels_give_the_same_values(spa, N):
    reg = synth.make_region(150, 6, 0.9, (0.5,), seed=1600)
    sched = synth.geometric_schedule(3, -4.0, -1.0)
    few, many = dict(quantiles=(0.05, 0.5, 0.95), deltas=(0.05, 0.1)), dict(
        quantiles=(0.01, 0.05, 0.25, 0.5, 0.75, 0.95, 0.99, 0.999), deltas=(0.01, 0.05, 0.1, 0.2))
    out = []
    for cfg in (few, many):
        with spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(move="rw", **cfg)) as r:
            out.append(r.run(sched, N, 1, 4))
    assert np.array_equal(out[0]["mean"], out[1]["mean"])
    assert np.array_equal(out[0]["quantile"], out[1]["quantile"][:, :, [1, 3, 5]])
    assert np.array_equal(out[0]["conc"], out[1]["conc"][:, :, 1:3])
    q = out[1]["quantile"]
    assert np.all(np.diff(q, axis=2) >= 0.0)


# Running sums of the weights: 32 at a time by a scan over integers where the sum keeps its
# exponent, FP64 additions elsewhere; ties, subnormals, jumps of scale, block and group edges.
@pytest.mark.parametrize("kind", ["equal", "thirds", "powers", "ties", "lognormal", "subnormal", "last", "zeros"])
@pytest.mark.parametrize("N", [1, 31, 33, 256, 257, 8191, 16384, 16385, 70001])
def test_resampling_sums_are_the_additions_in_order(spa, kind, N):
    rng = np.random.default_rng(N)
    W = {"equal": lambda: np.full(N, 1.0 / N), "thirds": lambda: np.full(N, 1.0 / 3.0),
         "powers": lambda: 2.0 ** -rng.integers(0, 60, N),
         "ties": lambda: 2.0 ** -rng.integers(0, 56, N) * (1.0 + 2.0 ** -52 * rng.integers(0, 4, N)),
         "lognormal": lambda: np.exp(rng.normal(0.0, 8.0, N)),
         "subnormal": lambda: rng.integers(0, 1 << 20, N) * 5e-324,
         "last": lambda: np.where(np.arange(N) == N - 1, 1.0, 1e-300),
         "zeros": lambda: rng.random(N) * (rng.random(N) < 0.02) + np.where(np.arange(N) == 0, 1e-3, 0.0)}[kind]()
    if kind not in ("subnormal", "thirds"):
        W = W / W.sum()
    for u in (0.0, 0.37, 0.999):
        assert np.array_equal(spa.resample_systematic(W, u), oracle.resample_systematic(W, u))


# The kernel that tests a MALA proposal forms its gradient from the contraction's K-split partials
# for p % 4 == 0 (groups of 4) and p <= 128 (4 coordinates 32 apart); other p take the finish kernel.
@pytest.mark.parametrize("n,p", [(40, 1), (100, 3), (129, 4), (300, 31), (400, 33), (800, 97), (1500, 127), (2100, 128),
                                 (700, 129), (600, 132), (900, 252), (500, 256), (500, 260)])
def test_mala_gradient_formed_where_it_is_tested(spa, n, p):
    """One seed, so the same proposals on both sides: the first step's decisions differ where a log
    ratio lies within the split product's rounding of log U (a few 1e-3 at most): about 0.3 of 256
    proposals are expected to, 4 are allowed, each moving a particle's coordinates by less than 1."""
    N, M = 128, 2
    reg = synth.make_region(n, p, 0.9, (0.5,), seed=1700 + n)
    sched = synth.geometric_schedule(2, -3.0, -2.0)
    with spa.Region(reg.G, reg.y, 2.0, config=spa.make_config(move="mala", init="resample_move")) as r:
        g = r.run(sched, N, M, 9)
    o = oracle.run(reg.G, reg.y, 2.0, sched, N, M, seed=9, cfg=oracle.make_config(move="mala", init="mcmc"))
    assert abs(g["accept_rate"][0] - o["accept_rate"][0]) <= 4.0 / (N * M) + 1e-12
    assert np.max(np.abs(g["mean"][0] - o["mean"][0])) <= 4.0 / N + 1e-4


# A batch's likelihood launches are sized by the regions' shares of the work (down to one CTA for a
# small region beside large ones, all SMs for a large one); alone each takes all SMs.
@pytest.mark.parametrize("move", ["rw", "mala"])
def test_uneven_batch_shares_give_the_single_runs(spa, move):
    shapes = [(31, 1, 5, 2), (4000, 200, 9000, 2), (513, 255, 770, 0), (900, 300, 2000, 3), (129, 64, 2600, 1)]
    sched = synth.geometric_schedule(3, -4.0, -1.0)
    regs = [synth.make_region(n, p, 0.9, (0.4, -0.3), seed=1800 + n) for n, p, _, _ in shapes]
    rs = [spa.Region(g.G, g.y, 2.0, config=spa.make_config(move=move)) for g in regs]
    alone = [r.run(sched, s[2], s[3], 5 + k) for k, (r, s) in enumerate(zip(rs, shapes))]
    b = spa.Batch(rs, [sched] * 5, [s[2] for s in shapes], [s[3] for s in shapes], [5 + k for k in range(5)])
    together = b.run()
    b.close()
    for one, two in zip(alone, together):
        for k in one:
            assert np.array_equal(one[k], two[k]), k
    for r in rs:
        r.close()


# The reverse move's gradient sum is one multiply-add in every form of the MALA kernels: for p <= 255
# a region alone takes the fused gradient kernel and, beside another, the two kernels, and p decides
# whether the gradient is formed where it is tested. A rounding more in one form shows only in
# about one of 10^7 decisions, so the sweeps are long enough to meet one.
@pytest.mark.parametrize("n,p", [(2714, 226), (1500, 190), (1200, 77)])
def test_mala_decisions_do_not_depend_on_the_launches(spa, n, p):
    reg = synth.make_region(n, p, 0.86, (0.3, 0.5, -0.4), seed=1803)
    sched = synth.geometric_schedule(10)
    with spa.Region(reg.G, reg.y, 16.0, config=spa.make_config(move="mala")) as r:
        for seed in (100, 101):
            one = r.run(sched, 16384, 12, seed)
            b = spa.Batch([r], [sched], [16384], [12], [seed])
            (two,) = b.run()
            b.close()
            for k in one:
                assert np.array_equal(one[k], two[k]), k


@pytest.mark.parametrize("n,p,N", [(31, 1, 4096), (33, 2, 3001)])
def test_site_kernel_of_the_smallest_regions_takes_the_oracles_decisions(spa, n, p, N):
    """As above at sizes where a handful of flips cannot hide a wrong decision: of about 5000
    decisions fewer than one is expected to lie within 1e-5 of its log U, two may flip."""
    reg = synth.make_region(n, p, 0.9, (0.5,), seed=1200 + n)
    sched = synth.geometric_schedule(2, -3.0, -2.0)
    with spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(move="site", init="resample_move")) as r:
        g = r.run(sched, N, 1, 11)
    o = oracle.run(reg.G, reg.y, 1.0, sched, N, 1, seed=11,
                   cfg=oracle.make_config(move="site", init="mcmc"))
    assert abs(g["accept_rate"][0] - o["accept_rate"][0]) <= 2.0 / (N * p) + 1e-12
    assert np.max(np.abs(g["mean"][0] - o["mean"][0])) <= 2 * 2.0 / N + 1e-4
