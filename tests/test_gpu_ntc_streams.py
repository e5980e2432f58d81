"""The No-Time-Counter kernel's candidate streams: cells whose candidates fill a
warp's 32 exactly (16 particles: four candidates a cell, eight cells a run),
one short and one over, cells of one particle each, listed cells of more than
64 candidates, cells whose candidates all share two particles, and queues that
wrap - each against the in-order oracle."""
import numpy as np
import pytest

from paper_2206_02937_gb300 import workloads as wl
from tests.test_gpu_ntc import _compare

pytestmark = pytest.mark.gpu


def _workload(sizes, w_over_v, dt, seed):
    rng = wl.rng_for(seed)
    cell = np.repeat(np.arange(len(sizes)), sizes)
    n = cell.shape[0]
    u = wl.maxwell_juttner_u(rng, n, 1.0) * wl.isotropic(rng, n)
    k = wl.planck_eps(rng, n, 1e-2) * wl.isotropic(rng, n)
    return wl.Workload("streams", len(sizes), w_over_v, dt, seed, 1, wl._species(u, cell), wl._species(k, cell))


@pytest.mark.parametrize("cells", [1, 7, 8, 9, 64, 65, 4096])
@pytest.mark.parametrize("n", [1, 2, 16, 130])
def test_equal_cells(cells, n):
    if n * cells > 100000:
        pytest.skip("covered by the smaller cells")
    # E = n^2 / 64: exactly four candidates a cell at n = 16, 264 at n = 130
    st, _ = _compare(_workload([n] * cells, 1.0 / 64.0, 0.5, 100 + n), step=5)
    if n == 16:
        assert st["pairs_tested"] == 4 * cells


def test_ragged_and_empty_cells():
    rng = np.random.default_rng(3)
    _compare(_workload(list(rng.integers(0, 90, 700)), 1.0 / 64.0, 0.3, 200), step=1 << 33)


def test_candidates_that_all_share_two_particles():
    # two electrons and two photons a cell, dozens of candidates: most are held back
    _compare(_workload([2] * 40, 2.0, 4.0, 300), step=2)


@pytest.mark.parametrize("cells", [1, 31, 32, 33, 1000, 4097])
def test_runs_of_32_cells(cells):
    # less than a candidate a cell in the mean, some cells empty, one listed
    rng = np.random.default_rng(cells)
    sizes = rng.poisson(4, cells)
    if cells > 1:
        sizes[cells // 2] = 130
    w = _workload(list(sizes), 1.0 / 64.0, 0.25, 400 + cells)
    assert (sizes.sum() / cells) ** 2 / 128.0 < 1.0
    _compare(w, step=7)


def test_runs_of_32_cells_among_many_cells():
    # above a run of 32 for every resident warp, 1.6 candidates a cell
    sizes = np.random.default_rng(9).integers(1, 4, 150001)
    _compare(_workload(list(sizes), 0.4, 0.5, 500), step=8)
