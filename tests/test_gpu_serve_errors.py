"""Serving when a launch of the engine fails (injected on the host, nothing is
done to the device): no request of it is reported OK, the engine refuses work
until it is started again, and then gives the direct call's results.  And the
engine stopped with requests unfinished: each of them is done or untouched."""
import time

import pytest

from paper_2206_02937_gb300 import workloads as wl
from tests.test_gpu_serve import _ctx
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def disarm():
    yield
    import paper_2206_02937_gb300 as cg
    cg.compton_debug_inject(0, 0)


def _pairs(torch, n, seed):
    u, k = wl.c3(n, seed=seed)
    return torch.from_numpy(u).cuda(), torch.from_numpy(k).cuda()


def _direct(cg, torch, ctx, u, k, dens, seed, mode):
    ud, kd = u.clone(), k.clone()
    cg.compton_scatter_pairs(ctx, ud, kd, torch.full((u.shape[1],), dens, device="cuda"), seed, 2, mode)
    torch.cuda.synchronize()
    return ud, kd


def _end(cg, ctx, ticket):
    """The request's end: 0, or the status of the error that poll raised."""
    t0 = time.time()
    while True:
        try:
            r = cg.compton_poll(ctx, ticket)
        except cg.ComptonError as e:
            return e.status
        if r is not None:
            assert r["status"] == cg.COMPTON_OK
            return 0
        assert time.time() - t0 < 30, "the request did not end"
        time.sleep(0.001)


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_a_failed_launch_ends_its_requests_with_the_error(mode):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    n, dens = 30011, 30.0
    u, k = _pairs(torch, n, 5)
    ctx = _ctx(cg)
    failures = 0
    try:
        ref = _direct(cg, torch, ctx, u, k, dens, 8, mode)
        for skip in range(40):
            cg.compton_serve_start(ctx, 1 << 26, 16)
            uo, ko = torch.empty_like(u), torch.empty_like(k)
            torch.cuda.synchronize()
            cg.compton_debug_inject(skip, 1)
            st = _end(cg, ctx, cg.compton_submit(ctx, u, k, uo, ko, dens, 8, 2, mode))
            pending = cg.compton_debug_inject(0, 0)
            if pending:  # every checked call of the request has been failed once
                assert st == 0 and torch.equal(uo, ref[0]) and torch.equal(ko, ref[1])
            else:
                failures += 1
                assert st == cg.COMPTON_ECUDA, skip
                assert cg.compton_serve_info(ctx)["in_use"] == 0
                with pytest.raises(cg.ComptonError) as e:
                    cg.compton_submit(ctx, u, k, uo, ko, dens, 8, 2, mode)
                assert e.value.status == cg.COMPTON_ECUDA
            cg.compton_serve_stop(ctx)
            if pending:
                break
        assert pending and failures >= (4 if mode == 0 else 6)
    finally:
        cg.compton_destroy(ctx)


def test_the_other_requests_end_too():
    """Requests beside and behind the failed launch (a pool that admits few at a
    time) end as well: right, or with the error."""
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    ctx = _ctx(cg)
    try:
        cg.compton_serve_start(ctx, 4 * 32 * 60000, 16)
        jobs = []
        for i in range(24):
            u, k = _pairs(torch, 50021, 20 + i)
            mode = (0, 2, 1, 3)[i % 4]
            jobs.append((u, k, torch.empty_like(u), torch.empty_like(k), mode,
                         _direct(cg, torch, ctx, u, k, 30.0, 40 + i, mode)))
        cg.compton_debug_inject(12, 1)
        tickets = []
        for i, (u, k, uo, ko, mode, _) in enumerate(jobs):
            try:
                tickets.append(cg.compton_submit(ctx, u, k, uo, ko, 30.0, 40 + i, 2, mode))
            except cg.ComptonError as e:
                assert e.status == cg.COMPTON_ECUDA
                tickets.append(None)
        ends = [cg.COMPTON_ECUDA if t is None else _end(cg, ctx, t) for t in tickets]
        assert cg.compton_debug_inject(0, 0) == 0
        assert cg.COMPTON_ECUDA in ends and set(ends) <= {0, cg.COMPTON_ECUDA}
        torch.cuda.synchronize()
        for st, (u, k, uo, ko, mode, ref) in zip(ends, jobs):
            if st == 0:
                assert torch.equal(uo, ref[0]) and torch.equal(ko, ref[1])
        assert cg.compton_serve_info(ctx)["in_use"] == 0
    finally:
        cg.compton_destroy(ctx)


@pytest.mark.parametrize("pause", [0.0, 2e-4, 5e-4, 1e-3, 2e-3])
def test_stop_leaves_in_place_requests_done_or_untouched(pause):
    """Requests of several launches each (every pair a candidate, more of them
    than a launch's list holds), in place; more than the pool admits at once."""
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    n, dens = 700001, 200.0
    ctx = _ctx(cg, n)
    try:
        jobs = []
        for i in range(5):
            u, k = _pairs(torch, n if i < 3 else 60013, 90 + i)
            mode = (2, 3, 1, 0, 2)[i]
            jobs.append((u, k, u.clone(), k.clone(), mode, _direct(cg, torch, ctx, u, k, dens, 60 + i, mode)))
        cg.compton_serve_start(ctx, 3 * 32 * 720000, 16)
        for i, (u, k, _, _, mode, _) in enumerate(jobs):
            cg.compton_submit(ctx, u, k, u, k, dens, 60 + i, 2, mode)
        time.sleep(pause)
        cg.compton_serve_stop(ctx)
        torch.cuda.synchronize()
        for i, (u, k, u0, k0, _, (ur, kr)) in enumerate(jobs):
            done = torch.equal(u, ur) and torch.equal(k, kr)
            assert done or (torch.equal(u, u0) and torch.equal(k, k0)), i
    finally:
        cg.compton_destroy(ctx)
