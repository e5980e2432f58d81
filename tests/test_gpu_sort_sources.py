"""The binning's three sources (input in cell order read in place, nearly in
order through placed indices, in no order through placed records) against the
order by (cell, key, id) formed in numpy: every output array equal, at cell
sizes around a sort tile's capacity (640 slots), with and without weights, and
with arrays that start off a 16-byte boundary."""
import numpy as np
import pytest

from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

SEED, STEP = 0x1234567890ABCDEF, (7 << 32) | 11


def _philox0(ident, stream):
    """Word 0 of Philox4x32-10 at counter (id, step lo, stream, step hi)."""
    m = np.uint64(0xFFFFFFFF)
    c = [ident.astype(np.uint64)] + [np.full(ident.shape, v, np.uint64) for v in (STEP & 0xFFFFFFFF, stream, STEP >> 32)]
    k0, k1 = SEED & 0xFFFFFFFF, SEED >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[0]


def _species(rng, counts, order):
    n, cells = int(counts.sum()), counts.shape[0]
    cell = np.repeat(np.arange(cells), counts).astype(np.int32)
    if order == "moved":
        hop = rng.integers(-1, 2, n) * (rng.random(n) < 0.15)
        cell = ((cell + hop) % cells).astype(np.int32)
    elif order == "runs":  # three ordered runs one after another
        cell = np.concatenate([cell[k::3] for k in range(3)])
    elif order == "none":
        cell = cell[rng.permutation(n)]
    return dict(ux=rng.standard_normal(n).astype(np.float32), uy=rng.standard_normal(n).astype(np.float32),
                uz=rng.standard_normal(n).astype(np.float32), cell=cell,
                id=rng.permutation(np.uint32(3) * np.arange(n, dtype=np.uint32)),
                w=rng.uniform(0.5, 2.0, n).astype(np.float32))


COUNTS = {
    "ragged": lambda rng: rng.poisson(21, 301),
    "sparse": lambda rng: rng.poisson(0.4, 4001),
    "cells16": lambda rng: np.full(700, 16),
    "wide": lambda rng: rng.integers(0, 330, 97),
    "capacity": lambda rng: np.array([636, 637, 638, 639, 640, 641, 642, 643, 0, 1, 2, 3, 640, 5, 636, 900, 1, 640]),
    "one_cell": lambda rng: np.array([1500]),
    "one": lambda rng: np.array([0, 1, 0]),
}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("order", ["cells", "moved", "runs", "none"])
@pytest.mark.parametrize("counts", sorted(COUNTS))
def test_sorted_copies_match_the_defined_order(counts, order, weighted):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    rng = np.random.default_rng(len(counts) * 100 + len(order) * 10 + weighted)
    sizes = COUNTS[counts](rng)
    e, g = _species(rng, sizes, order), _species(rng, rng.permutation(sizes), order)
    keys = ("ux", "uy", "uz", "cell", "id", "w")

    def device(d, shift):
        def t(a):
            base = torch.zeros(a.shape[0] + shift, dtype=torch.from_numpy(a).dtype, device="cuda")
            base[shift:] = torch.from_numpy(a).cuda()
            return base[shift:]
        return cg.Species(*(t(d[k].view(np.int32) if k == "id" else d[k]) for k in keys[:5 + weighted]))

    ctx = cg.compton_init(sizes.shape[0], max(1, e["cell"].shape[0]), 1.0, 0.05, SEED)
    try:
        for shift_in, shift_out in ((0, 0), (1, 0), (0, 3)):
            ein, gin = device(e, shift_in), device(g, shift_in)
            blank = [{k: np.zeros_like(d[k]) for k in keys} for d in (e, g)]
            eo, go = device(blank[0], shift_out), device(blank[1], shift_out)
            cg.compton_bin_pairs(ctx, ein, gin, eo, go, STEP)
            assert cg.compton_check(ctx) == cg.COMPTON_OK
            for d, o, stream in ((e, eo, 1), (g, go, 2)):
                perm = np.lexsort((d["id"], _philox0(d["id"], stream), d["cell"]))
                for k in keys[:5 + weighted]:
                    got = getattr(o, k).cpu().numpy()
                    assert np.array_equal(got.view(np.uint32), d[k][perm].view(np.uint32)), (k, shift_in, shift_out)
    finally:
        cg.compton_destroy(ctx)


@pytest.mark.parametrize("order", ["cells", "moved", "none"])
def test_equal_ids_still_give_a_permutation(order):
    """Equal ids (invalid input) draw equal keys: more than a bucket's counters
    hold; every particle still comes out once, in its cell."""
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    rng = np.random.default_rng(5)
    d = _species(rng, rng.integers(10, 60, 80), order)
    n = d["cell"].shape[0]
    d["id"][:] = 7
    d["id"][::5] = np.arange(0, n, 5)
    d["ux"] = np.arange(n, dtype=np.float32)
    sp = lambda: cg.Species(*(torch.from_numpy(np.ascontiguousarray(d[k].view(np.int32) if k == "id" else d[k])).cuda()
                              for k in ("ux", "uy", "uz", "cell", "id")))
    ctx = cg.compton_init(80, n, 1.0, 0.05, SEED)
    try:
        e, g = sp(), sp()
        eo, go = cg.Species.empty_like(e), cg.Species.empty_like(g)
        cg.compton_bin_pairs(ctx, e, g, eo, go, STEP)
        assert cg.compton_check(ctx) == cg.COMPTON_OK
        for o in (eo, go):
            src = o.ux.cpu().numpy().astype(np.int64)
            assert np.array_equal(np.sort(src), np.arange(n))
            assert np.array_equal(o.cell.cpu().numpy(), np.sort(d["cell"]))
            for k in ("uy", "uz", "cell"):
                assert np.array_equal(getattr(o, k).cpu().numpy(), d[k][src])
            assert np.array_equal(o.id.cpu().numpy().view(np.uint32), d["id"][src])
    finally:
        cg.compton_destroy(ctx)
