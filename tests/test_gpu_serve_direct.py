"""The serving kernels on the caller's own arrays: every mode at the edges of
the 1024-pair tiles, outputs apart from the inputs, on them, and overlapping
them otherwise (staged); and more surrogate candidates than a launch's list
holds (2^18), whose tiles are launched again.  Everything equals the direct
compton_scatter_pairs call bit for bit, the collision counts too."""
import numpy as np
import pytest

from paper_2206_02937_gb300 import workloads as wl
from tests.test_gpu_serve import _ctx, _wait
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

MODES = {"plain": 0, "fp32": 1, "bf16": 2, "fp8": 3}


def _direct(cg, torch, ctx, u, k, dens, seed, step, mode):
    n = u.shape[1]
    ud, kd = u.clone(), k.clone()
    nd = dens if torch.is_tensor(dens) else torch.full((n,), float(dens), device="cuda")
    flag = torch.zeros(n, dtype=torch.uint8, device="cuda")
    cg.compton_scatter_pairs(ctx, ud, kd, nd, seed, step, mode, None, flag)
    torch.cuda.synchronize()
    return ud, kd, int(flag.sum())


def _pairs(torch, n, seed):
    u, k = wl.c3(n, seed=seed)
    return torch.from_numpy(u).cuda(), torch.from_numpy(k).cuda()


@pytest.mark.parametrize("mode", sorted(MODES))
def test_tile_edges_and_aliasing(mode):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    ctx = _ctx(cg)
    try:
        cg.compton_mlp_calibrate(ctx, *_pairs(torch, 4096, 1))
        cg.compton_serve_start(ctx, 1 << 28, 64)
        jobs = []
        for i, n in enumerate((1, 255, 1023, 1024, 1025, 4999, 30011)):
            for form in ("apart", "inplace", "shifted", "crossed"):
                u, k = _pairs(torch, n, 50 + i)
                dens = torch.rand(n, device="cuda") * 40 if i % 2 else 25.0
                ref = _direct(cg, torch, ctx, u, k, dens, 9 + i, 4, MODES[mode])
                if form == "apart":
                    ui, ki, uo, ko = u, k, torch.empty_like(u), torch.empty_like(k)
                elif form == "inplace":
                    ui, ki, uo, ko = u, k, u, k
                elif form == "shifted":  # each output row one element past its input row
                    ub, kb = torch.zeros(3, n + 1, device="cuda"), torch.zeros(3, n + 1, device="cuda")
                    ub[:, :n], kb[:, :n] = u, k
                    ui, ki, uo, ko = ub[:, :n], kb[:, :n], ub[:, 1:], kb[:, 1:]
                else:  # the outputs of the electrons on the inputs of the photons
                    ui, ki, uo, ko = u, k, k, u
                t = cg.compton_submit(ctx, ui, ki, uo, ko, dens, 9 + i, 4, MODES[mode])
                jobs.append((t, uo, ko, ref, (n, form), (ui, ki, dens)))
        res = _wait(cg, ctx, [j[0] for j in jobs])
        torch.cuda.synchronize()
        for t, uo, ko, (ur, kr, hits), what, _ in jobs:
            assert torch.equal(uo, ur) and torch.equal(ko, kr), what
            assert res[t]["scatters"] == hits, what
        assert cg.compton_serve_info(ctx)["in_use"] == 0
        assert cg.compton_check(ctx) == cg.COMPTON_OK
    finally:
        cg.compton_destroy(ctx)


@pytest.mark.parametrize("per_pair", [False, True])
def test_more_candidates_than_the_list_holds(per_pair):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    ctx = _ctx(cg, 700000)
    try:
        cg.compton_serve_start(ctx, 1 << 28, 64)
        jobs = []
        for i, (n, mode) in enumerate(((600001, 2), (150000, 1), (400003, 2), (5000, 0), (300000, 3))):
            u, k = _pairs(torch, n, 70 + i)
            # every pair a candidate; per-pair densities hide that from the host's estimate
            dens = torch.full((n,), 200.0, device="cuda") if per_pair else 200.0
            ref = _direct(cg, torch, ctx, u, k, dens, 3 + i, 1, mode)
            uo, ko = torch.empty_like(u), torch.empty_like(k)
            jobs.append((cg.compton_submit(ctx, u, k, uo, ko, dens, 3 + i, 1, mode), uo, ko, ref, u, k, dens))
        res = _wait(cg, ctx, [j[0] for j in jobs])
        torch.cuda.synchronize()
        for t, uo, ko, (ur, kr, hits), *_ in jobs:
            assert torch.equal(uo, ur) and torch.equal(ko, kr)
            assert res[t]["scatters"] == hits
        st = cg.compton_get_stats(ctx, reset=True)
        # each pair tested once by the direct calls and once here
        assert st["pairs_tested"] == 2 * sum(j[1].shape[1] for j in jobs)
    finally:
        cg.compton_destroy(ctx)


@pytest.mark.parametrize("n,launches", [(1000003, 2), (5000003, 6)])
def test_dense_densities_per_pair_take_few_launches(n, launches):
    """Every pair a candidate, which the host cannot know: the list follows the
    pool (2^21 candidates here), and what a launch turns away is taken in full
    lists once its candidates are counted (three full lists for 5 million, two
    launches before the count)."""
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    ctx = _ctx(cg, n)
    try:
        u, k = _pairs(torch, n, 31)
        dens = torch.full((n,), 200.0, device="cuda")
        ref = _direct(cg, torch, ctx, u, k, dens, 6, 1, 2)
        cg.compton_serve_start(ctx, 1 << 28, 8)
        cg.compton_kernel_timing(ctx, True)
        uo, ko = torch.empty_like(u), torch.empty_like(k)
        t = cg.compton_submit(ctx, u, k, uo, ko, dens, 6, 1, 2)
        res = _wait(cg, ctx, [t])
        torch.cuda.synchronize()
        assert torch.equal(uo, ref[0]) and torch.equal(ko, ref[1]) and res[t]["scatters"] == ref[2]
        assert cg.compton_kernel_times(ctx)["k_mlp"]["launches"] <= launches
    finally:
        cg.compton_destroy(ctx)


def test_more_candidates_than_a_small_pools_list_holds():
    # 2^18 candidates a launch; requests of mixed modes, scalar and per-pair densities
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    ctx = _ctx(cg, 400003)
    try:
        cg.compton_serve_start(ctx, 1 << 24, 64)
        jobs = []
        for i, (n, mode) in enumerate(((400003, 2), (150000, 1), (300001, 3), (5000, 0), (400003, 1), (200001, 2))):
            u, k = _pairs(torch, n, 80 + i)
            dens = torch.rand(n, device="cuda") * 200 if i % 2 == 0 else 200.0
            ref = _direct(cg, torch, ctx, u, k, dens, 3 + i, 1, mode)
            uo, ko = torch.empty_like(u), torch.empty_like(k)
            jobs.append((cg.compton_submit(ctx, u, k, uo, ko, dens, 3 + i, 1, mode), uo, ko, ref, u, k, dens))
        res = _wait(cg, ctx, [j[0] for j in jobs])
        torch.cuda.synchronize()
        for t, uo, ko, (ur, kr, hits), *_ in jobs:
            assert torch.equal(uo, ur) and torch.equal(ko, kr)
            assert res[t]["scatters"] == hits
        assert cg.compton_get_stats(ctx, reset=True)["pairs_tested"] == 2 * sum(j[1].shape[1] for j in jobs)
        assert cg.compton_serve_info(ctx)["in_use"] == 0
    finally:
        cg.compton_destroy(ctx)
