"""The binning's general path (more than 4096 cells or 16384 particles: smaller
calls are binned by one CTA, which always places indices) on its three sources,
input in cell order, through k_place's indices and through its records: against
the order by (cell, key, id) formed in numpy.  Cells at the edges of a sort
tile's capacity, weights, equal ids; and input of few descents whose particles
lie apart all the same (particle i in cell i mod C, short runs of equal cells),
below and above the size from which the histogram looks for it."""
import numpy as np
import pytest

from tests.gpu_util import torch_cuda
from tests.test_gpu_sort_sources import COUNTS, SEED, STEP, _philox0, _species

pytestmark = pytest.mark.gpu

KEYS = ("ux", "uy", "uz", "cell", "id", "w")


def _input(rng, sizes, order):
    if order not in ("robin", "clump"):
        return _species(rng, sizes, order)
    d = _species(rng, sizes, "cells")
    cell = d["cell"]
    if order == "robin":  # every cell's first particle, every cell's second, ...
        first = np.concatenate([[0], np.cumsum(sizes)[:-1]])
        cell = cell[np.argsort(np.arange(cell.size) - first[cell], kind="stable")]
    else:  # runs of three in no order
        m = cell.size // 3
        cell = np.concatenate([cell[:3 * m].reshape(m, 3)[rng.permutation(m)].reshape(-1), cell[3 * m:]])
    d["cell"] = np.ascontiguousarray(cell)
    return d


def _device(torch, d, weighted):
    return _blank(torch, d, weighted, [torch.from_numpy(d[k].view(np.int32) if k == "id" else d[k]).cuda() for k in KEYS])


def _blank(torch, d, weighted, arrays=None):
    import paper_2206_02937_gb300 as cg
    if arrays is None:
        arrays = [torch.zeros(d["cell"].size, dtype=torch.int32 if k in ("cell", "id") else torch.float32, device="cuda")
                  for k in KEYS]
    return cg.Species(*arrays[:5 + weighted])


def _check_order(sizes, e, g, weighted):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    ctx = cg.compton_init(sizes.shape[0], max(1, e["cell"].size), 1.0, 0.05, SEED)
    try:
        eo, go = _blank(torch, e, weighted), _blank(torch, g, weighted)
        cg.compton_bin_pairs(ctx, _device(torch, e, weighted), _device(torch, g, weighted), eo, go, STEP)
        assert cg.compton_check(ctx) == cg.COMPTON_OK
    finally:
        cg.compton_destroy(ctx)
    for d, o, stream in ((e, eo, 1), (g, go, 2)):
        by_id = np.argsort(d["id"], kind="stable")
        key = (d["cell"].astype(np.uint64) << np.uint64(32)) | _philox0(d["id"], stream)
        perm = by_id[np.argsort(key[by_id], kind="stable")]
        for k in KEYS[:5 + weighted]:
            assert np.array_equal(getattr(o, k).cpu().numpy().view(np.uint32), d[k][perm].view(np.uint32)), k


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("order", ["cells", "moved", "runs", "none", "robin", "clump"])
@pytest.mark.parametrize("counts", sorted(COUNTS))
def test_every_source_matches_the_defined_order(counts, order, weighted):
    rng = np.random.default_rng(len(counts) * 100 + len(order) * 10 + weighted)
    sizes = np.concatenate([COUNTS[counts](rng), np.zeros(4097, np.int64)])
    _check_order(sizes, _input(rng, sizes, order), _input(rng, rng.permutation(sizes), order), weighted)


@pytest.mark.parametrize("order", ["cells", "moved", "runs", "none", "robin", "clump"])
def test_large_input(order):
    rng = np.random.default_rng(len(order))
    sizes = rng.poisson(64, 66500)  # above 2^22 particles
    assert sizes.sum() > 1 << 22
    _check_order(sizes, _input(rng, sizes, order), _input(rng, rng.permutation(sizes), order), False)


@pytest.mark.parametrize("order", ["cells", "moved", "none", "robin"])
def test_equal_ids_still_give_a_permutation(order):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    rng = np.random.default_rng(5)
    sizes = np.concatenate([rng.integers(10, 60, 80), np.zeros(4097, np.int64)])
    d = _input(rng, sizes, order)
    n = d["cell"].size
    d["id"][:] = 7
    d["id"][::5] = np.arange(0, n, 5)
    d["ux"] = np.arange(n, dtype=np.float32)
    ctx = cg.compton_init(sizes.size, n, 1.0, 0.05, SEED)
    try:
        outs = [_blank(torch, d, False) for _ in range(2)]
        cg.compton_bin_pairs(ctx, _device(torch, d, False), _device(torch, d, False), *outs, STEP)
        assert cg.compton_check(ctx) == cg.COMPTON_OK
        for o in outs:
            src = o.ux.cpu().numpy().astype(np.int64)
            assert np.array_equal(np.sort(src), np.arange(n))
            assert np.array_equal(o.cell.cpu().numpy(), np.sort(d["cell"]))
            for k in ("uy", "uz", "cell"):
                assert np.array_equal(getattr(o, k).cpu().numpy(), d[k][src])
            assert np.array_equal(o.id.cpu().numpy().view(np.uint32), d["id"][src])
    finally:
        cg.compton_destroy(ctx)
