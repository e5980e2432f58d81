"""Calls whose launches are chained (each kernel's blocks placed while the one
before drains): captured in a CUDA graph and replayed on other inputs, on a side
stream behind an event, and one call after another without a wait, against the
same calls with a synchronisation after each.  Steps of one and of several
sort blocks per SM, networks, collisions in the probability kernel or behind it."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2206_02937_gb300 import workloads as wl
from tests.gpu_util import species_np, to_species, torch_cuda

pytestmark = pytest.mark.gpu

KEYS = ("ux", "uy", "uz", "cell", "id")
SIZES = {"small": (8, 8, 32), "middle": (40, 40, 40), "large": (128, 96, 48)}
MODES = ("plain", "fp32", "bf16", "fp8", "pnet", "ntc")


def _context(cg, w):
    ctx = cg.compton_init(w.n_cells, max(w.n_e, w.n_g), w.w_over_v, w.dt, w.seed, max_train_batch=20000)
    cg.compton_mlp_set_params(ctx, omlp.init_params(3).astype(np.float32))
    cg.compton_pnet_set_params(ctx, np.random.default_rng(4).uniform(-0.5, 0.5, cg.PNET_PARAMS).astype(np.float32))
    return ctx


def _inputs(torch, w, order):
    """The workload's species in cell order (0), a tenth moved (1) or in no order (2)."""
    rng = np.random.default_rng(order)
    out = []
    for d in (w.e, w.g):
        d = {k: v.copy() for k, v in d.items()}
        if order == 1:
            at = rng.random(d["cell"].size) < 0.1
            d["cell"][at] = (d["cell"][at] + 1) % w.n_cells
        elif order == 2:
            p = rng.permutation(d["cell"].size)
            d = {k: np.ascontiguousarray(v[p]) for k, v in d.items()}
        out.append(to_species(torch, d))
    return out


def _step(cg, ctx, e, g, eo, go, mode):
    pairs = cg.compton_bin_pairs(ctx, e, g, eo, go, 3)
    if mode == "ntc":
        cg.compton_scatter_step_ntc(ctx, eo, go, pairs, 3)
    else:
        cg.compton_scatter_step(ctx, eo, go, pairs, dict(plain=0, fp32=1, bf16=2, fp8=3, pnet=4)[mode], 3)


def _reference(cg, torch, ctx, w, mode):
    """Each input order's result with a synchronisation between the calls."""
    ref = []
    for order in range(3):
        e, g = _inputs(torch, w, order)
        eo, go = cg.Species.empty_like(e), cg.Species.empty_like(g)
        torch.cuda.synchronize()
        _step(cg, ctx, e, g, eo, go, mode)
        torch.cuda.synchronize()
        ref.append((species_np(eo), species_np(go)))
    return ref


def _equal(got, ref):
    return all(np.array_equal(a[k].view(np.uint32), b[k].view(np.uint32)) for a, b in zip(got, ref) for k in KEYS)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("size", sorted(SIZES))
def test_graph_side_stream_and_back_to_back(size, mode):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    w = wl.c2(*SIZES[size], seed=21)
    ctx = _context(cg, w)
    try:
        ref = _reference(cg, torch, ctx, w, mode)
        inputs = [_inputs(torch, w, order) for order in range(3)]
        e, g = (cg.Species.empty_like(s) for s in inputs[0])
        eo, go = cg.Species.empty_like(e), cg.Species.empty_like(g)

        def load(order):
            for s, t in zip((e, g), inputs[order]):
                for k in KEYS:
                    getattr(s, k).copy_(getattr(t, k))

        # captured once, replayed on the three orders
        graph = torch.cuda.CUDAGraph()
        load(0)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            _step(cg, ctx, e, g, eo, go, mode)
        for order in (2, 0, 1, 2):
            load(order)
            graph.replay()
            torch.cuda.synchronize()
            assert _equal((species_np(eo), species_np(go)), ref[order]), ("graph", order)

        # on a side stream, behind the copies of another one by an event
        side, feed = torch.cuda.Stream(), torch.cuda.Stream()
        busy = torch.randn(2048, 2048, device="cuda")
        torch.cuda.synchronize()
        for order in (1, 2, 0):
            done = torch.cuda.Event()
            with torch.cuda.stream(feed):
                for _ in range(4):
                    busy = (busy @ busy).clamp_(-1.0, 1.0)
                load(order)
                done.record(feed)
            with torch.cuda.stream(side):
                side.wait_event(done)
                _step(cg, ctx, e, g, eo, go, mode)
            feed.wait_stream(side)
            side.synchronize()
            assert _equal((species_np(eo), species_np(go)), ref[order]), ("side stream", order)
        torch.cuda.synchronize()

        # one after another on one stream, nothing waited for
        outs = []
        for order in (0, 1, 2, 2, 1, 0):
            o = [cg.Species.empty_like(s) for s in inputs[order]]
            _step(cg, ctx, *inputs[order], *o, mode)
            outs.append((order, o))
        torch.cuda.synchronize()
        for order, o in outs:
            assert _equal([species_np(s) for s in o], ref[order]), ("back to back", order)
        assert cg.compton_check(ctx) == cg.COMPTON_OK
    finally:
        cg.compton_destroy(ctx)


@pytest.mark.parametrize("kind", ["fp32", "bf16", "pnet"])
def test_training_and_inference_back_to_back(kind):
    """Training steps with the updated network run after each: with and without
    a synchronisation between the calls.  The gradient's atomics add up in any
    order: 1e-7 of a gradient, or a parameter whose gradient cancels to that and
    moves the other way by Adam's 1e-3 (r by less than 1e-4 each); a step that
    was not waited for shows as a whole step's move of r, above 1e-3."""
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    n = 20000
    w = wl.c1()
    u, k = (torch.from_numpy(a).cuda() for a in wl.c3(n, seed=6))
    y = torch.empty(n, device="cuda")
    results = []
    for wait in (True, False):
        ctx = _context(cg, w)
        try:
            cg.compton_kn_ratio(ctx, u, k, y)
            cg.compton_mlp_set_train_precision(ctx, cg.MODE_MLP_BF16 if kind == "bf16" else cg.MODE_MLP_FP32)
            torch.cuda.synchronize()
            outs = []
            for _ in range(6):
                r = torch.empty(n, device="cuda")
                if kind == "pnet":
                    cg.compton_pnet_train_step(ctx, u, k, y, None, 0.02, 0.02, 0.1, 1e-3, want_loss=False)
                    cg.compton_pnet_infer(ctx, u, k, 0.02, 0.02, 0.1, r)
                else:
                    cg.compton_mlp_train_step(ctx, u, k, y, None, 1e-3, want_loss=False)
                    cg.compton_mlp_infer(ctx, u, k, cg.MODE_MLP_FP32, r)
                if wait:
                    torch.cuda.synchronize()
                outs.append(r)
            torch.cuda.synchronize()
            results.append([r.cpu().numpy() for r in outs])
        finally:
            cg.compton_destroy(ctx)
    for a, b in zip(*results):
        assert np.abs(a - b).max() <= 2e-4
    for a, b in zip(results[0], results[0][1:]):
        assert np.abs(a - b).max() > 1e-3
