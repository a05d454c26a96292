"""The device entry points and the caller's memory and streams: particles read where they lie or
copied first, and work of the context that another stream has to wait for."""
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


# Read in place: an aligned base, and outputs elsewhere. Copied first: a base off by one float where
# rows are read 16 bytes at a time (p % 4 == 0), and an output inside the particles' memory.
@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
@pytest.mark.parametrize("n,p,N", [(300, 20, 130), (300, 21, 130), (129, 64, 1)])
def test_particles_copied_first_give_the_values_of_those_read_in_place(spa, precision, n, p, N):
    import torch

    reg = synth.make_region(n, p, 0.9, (0.4,), seed=1900 + n + p)
    B = torch.from_numpy(synth.random_particles(N, p, 0.1, seed=p)).cuda()
    st = torch.cuda.Stream()
    with spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(precision=precision)) as r:

        def evaluate(b, ll, g):
            out = torch.full((N,), float("nan"), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            r.loglik_device(b, out, st.cuda_stream)
            r.grad_device(b, 0.7, ll, g, st.cuda_stream)
            return out.cpu().numpy(), ll.cpu().numpy(), g.cpu().numpy()

        ll, g = torch.empty(N, dtype=torch.float64, device="cuda"), torch.empty((N, p), device="cuda")
        want = evaluate(B, ll, g)
        assert np.allclose(want[0], oracle.loglik(reg.G, reg.y, B.cpu().numpy().astype(np.float64)), rtol=1e-3)
        off = torch.empty(N * p + 1, device="cuda")[1:].view(N, p)
        assert off.data_ptr() % 16 == 4
        off.copy_(B)
        for a, b in zip(want, evaluate(off, ll, g)):
            assert np.array_equal(a, b)
        # the gradient written over the particles it is of
        over = B.clone()
        for a, b in zip(want[1:], evaluate(over, ll, over)[1:]):
            assert np.array_equal(a, b)
        # the log-likelihood written into their first rows
        room = torch.empty(max(N * p, 2 * N), device="cuda")
        room[: N * p] = B.view(-1)
        torch.cuda.synchronize()
        r.loglik_device(room[: N * p].view(N, p), room.view(torch.float64)[:N], st.cuda_stream)
        assert np.array_equal(room.view(torch.float64)[:N].cpu().numpy(), want[0])


def test_a_call_on_another_stream_waits_for_a_sweep_left_running(spa):
    """A sweep is left running on the context's own stream; a call on a configured stream ends in
    between and waits for that one only; then a caller's stream uses the same workspace."""
    import torch

    n, p, N, T, M = 1500, 100, 4096, 60, 5
    reg = synth.make_region(n, p, 0.9, (0.4,), seed=2000)
    sched = synth.geometric_schedule(T)
    sched_d = torch.from_numpy(sched).cuda()
    B = torch.from_numpy(synth.random_particles(N, p, 0.1, seed=3)).cuda()
    ll = torch.empty(N, dtype=torch.float64, device="cuda")
    ess = torch.empty(T, dtype=torch.float64, device="cuda")
    conf, user = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with spa.Region(reg.G, reg.y, 1.0) as r:
        want = r.run(sched, N, M, 7)
        r.loglik_device(B, ll, user.cuda_stream)
        alone = ll.cpu().numpy()
        own_cfg, conf_cfg = r.config(), r.config()
        conf_cfg.stream = conf.cuda_stream
        for between in (False, True):
            ll.fill_(float("nan"))
            torch.cuda.synchronize()
            r.run_device(sched_d, N, M, 7, {"ess": ess})
            if between:
                r.set_config(conf_cfg)
                r.sync()
                r.set_config(own_cfg)
            r.loglik_device(B, ll, user.cuda_stream)
            assert np.array_equal(ll.cpu().numpy(), alone)
            r.sync()
            assert np.array_equal(ess.cpu().numpy(), want["ess"])


def test_a_changed_stream_waits_for_a_sweep_left_on_the_one_before(spa):
    """Own stream to a configured one, from that to another, and back to the own one, each with a
    sweep left running on the stream before; the sweeps share the workspace and the captured graph's
    buffers."""
    import torch

    n, p, N, T, M = 1500, 100, 4096, 60, 5
    reg = synth.make_region(n, p, 0.9, (0.4,), seed=2100)
    sched = synth.geometric_schedule(T)
    sched_d = torch.from_numpy(sched).cuda()
    streams = [0, torch.cuda.Stream().cuda_stream, torch.cuda.Stream().cuda_stream, 0]
    ess = [torch.empty(T, dtype=torch.float64, device="cuda") for _ in streams]
    torch.cuda.synchronize()
    with spa.Region(reg.G, reg.y, 1.0) as r:
        want = [r.run(sched, N, M, 20 + k)["ess"] for k in range(len(streams))]
        for k, s in enumerate(streams):
            cfg = r.config()
            cfg.stream = s or None
            r.set_config(cfg)
            r.run_device(sched_d, N, M, 20 + k, {"ess": ess[k]})
        r.sync()
    torch.cuda.synchronize()
    for k in range(len(streams)):
        assert np.array_equal(ess[k].cpu().numpy(), want[k])


# Work queued on torch's default stream just before the call: 20 ms of it, then the update of the
# particles that the call is to see.
@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
def test_calls_without_a_stream_see_what_the_default_stream_has_queued(spa, precision):
    import torch

    n, p, N = 500, 40, 2000
    reg = synth.make_region(n, p, 0.9, (0.4,), seed=2200)
    old, new = (torch.from_numpy(synth.random_particles(N, p, 0.1, seed=s)).cuda() for s in (1, 2))
    ll, g = torch.empty(N, dtype=torch.float64, device="cuda"), torch.empty((N, p), device="cuda")

    def queue(B):
        torch.cuda.synchronize()
        torch.cuda._sleep(40_000_000)
        B.copy_(new)

    with spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(precision=precision)) as r:
        want_ll, want_g = r.grad(new.cpu().numpy())
        want = r.loglik(new.cpu().numpy())
        B = old.clone()
        queue(B)
        r.loglik_device(B, ll)
        assert np.array_equal(ll.cpu().numpy(), want)
        B.copy_(old)
        queue(B)
        r.grad_device(B, 0.0, ll, g)
        assert np.array_equal(ll.cpu().numpy(), want_ll) and np.array_equal(g.cpu().numpy(), want_g)
        B = old.clone().requires_grad_(True)
        with torch.no_grad():
            queue(B)
        out = spa.loglik_autograd(B, r)
        torch.cuda._sleep(40_000_000)
        (grad,) = torch.autograd.grad(out, B, torch.full_like(out, 2.0))
        assert np.array_equal(out.detach().cpu().numpy(), want)
        assert np.array_equal(grad.cpu().numpy(), 2.0 * want_g)
        # a block of the output's memory that the default stream still reads when the call writes it
        keep = torch.empty((N, p), device="cuda")
        g.fill_(7.0)
        torch.cuda.synchronize()
        torch.cuda._sleep(40_000_000)
        keep.copy_(g)
        r.grad_device(new, 0.0, ll, g)
        assert bool((keep == 7.0).all()) and np.array_equal(g.cpu().numpy(), want_g)
        # a schedule that the default stream is still to write
        sched = synth.geometric_schedule(5)
        want_ess = r.run(sched, N, 1, 3)["ess"]
        later, ess = torch.from_numpy(sched).cuda(), torch.empty(5, dtype=torch.float64, device="cuda")
        sched_d = torch.full((5,), 0.5, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(40_000_000)
        sched_d.copy_(later)
        r.run_device(sched_d, N, 1, 3, {"ess": ess})
        r.sync()
        assert np.array_equal(ess.cpu().numpy(), want_ess)
