"""The one-launch binning of small calls (at most 4096 cells and 16384 particles
of both species together) at its limits and one past them: offsets, pairs and
the sorted copies as the general path's definition gives them, in order and
not, with bad cell indices, one species empty, and twice in a row on one
context; and the whole step against the oracle on both sides of the line."""
import numpy as np
import pytest

import oracle
from paper_2206_02937_gb300 import workloads as wl
from tests.gpu_util import _dev_array, torch_cuda
from tests.test_gpu_parity import _random_workload, compare_with_oracle
from tests.test_gpu_sort_sources import SEED, STEP, _philox0, _species

pytestmark = pytest.mark.gpu
KEYS = ("ux", "uy", "uz", "cell", "id")


def _dev(cg, torch, d):
    return cg.Species(*(torch.from_numpy(np.ascontiguousarray(d[k].view(np.int32) if k == "id" else d[k])).cuda()
                        for k in KEYS))


@pytest.mark.parametrize("order", ["cells", "moved", "none"])
@pytest.mark.parametrize("cells,n", [(1, 1), (1, 600), (3, 3), (64, 4096), (4096, 8192), (4097, 8192), (4096, 8193),
                                     (4095, 8191), (1025, 31), (100, 8192)])
def test_offsets_and_order(cells, n, order):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    rng = np.random.default_rng(cells + n)
    sizes = np.bincount(rng.integers(0, cells, n), minlength=cells)
    e, g = _species(rng, sizes, order), _species(rng, rng.permutation(sizes), order)
    if order == "none" and n > 50:
        e["cell"][[3, 17, n - 1]] = (-1, cells, 1 << 30)  # left out of every cell, and reported
    ctx = cg.compton_init(cells, n, 1.0, 0.05, SEED)
    try:
        for _ in range(2):
            ein, gin = _dev(cg, torch, e), _dev(cg, torch, g)
            eo, go = cg.Species.empty_like(ein), cg.Species.empty_like(gin)
            pairs = cg.compton_bin_pairs(ctx, ein, gin, eo, go, STEP)
            bad = (e["cell"] < 0) | (e["cell"] >= cells)
            assert cg.compton_check(ctx) == (cg.COMPTON_ERANGE if bad.any() else cg.COMPTON_OK)
            counts = []
            for d, o, stream, off in ((e, eo, 1, pairs.off_e_dev), (g, go, 2, pairs.off_g_dev)):
                ok = (d["cell"] >= 0) & (d["cell"] < cells)
                perm = np.lexsort((d["id"], _philox0(d["id"], stream), d["cell"]))
                perm = perm[ok[perm]]
                count = np.bincount(d["cell"][ok], minlength=cells)
                counts.append(count)
                assert np.array_equal(_dev_array(torch, off, cells + 1), np.concatenate([[0], np.cumsum(count)]))
                for k in KEYS:
                    got = getattr(o, k).cpu().numpy()[:perm.shape[0]]
                    assert np.array_equal(got.view(np.uint32), d[k][perm].view(np.uint32)), k
            n_pairs = _dev_array(torch, pairs.n_pairs_dev, 2).view(np.int64)[0]
            assert n_pairs == np.minimum(*counts).sum()
    finally:
        cg.compton_destroy(ctx)


@pytest.mark.parametrize("cells,ppc", [(128, 64), (129, 64), (512, 64), (520, 64), (4096, 2), (40, 200)])
def test_step_on_both_sides_of_the_lines(cells, ppc):
    # 8192 + 8192 particles (one-launch binning), 32768 pairs (collisions in the probability kernel)
    compare_with_oracle(wl.c2(cells, 1, ppc, seed=31))


def test_one_species_empty():
    w = _random_workload(41, n_cells=50, ppc_e=20, ppc_g=20)
    w.g = {k: v[:0] for k, v in w.g.items()}
    compare_with_oracle(w)


@pytest.mark.parametrize("cells", [65, 4096, 6000])
@pytest.mark.parametrize("n_e", [1, 10, 200, 3000])
def test_few_pairs_among_many_cells(n_e, cells):
    """Pairs whose cells lie far apart, more cells than a warp's window holds
    between two of them (the cell of a pair is then found by bisection)."""
    from paper_2206_02937_gb300 import workloads as wl
    from tests.test_gpu_parity import compare_with_oracle
    rng = wl.rng_for(cells + n_e)
    n_g = 12000
    ce, cg = rng.integers(0, cells, n_e), rng.integers(0, cells, n_g)
    ce[0] = cells - 1
    u = 3.0 * wl.isotropic(rng, n_e)
    k = 10 ** rng.uniform(-4, 0, n_g) * wl.isotropic(rng, n_g)
    compare_with_oracle(wl.Workload("few pairs", cells, 0.1, 1.0, 17, 1, wl._species(u, ce), wl._species(k, cg)), step=4)
