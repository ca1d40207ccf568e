"""Cells beyond what one warp sorts (128 particles) and beyond the block sort's
2,048: alone, several to a block's turn and among small ones, the storage order
is the stable one and forces and steps do not depend on the cells, bit for bit;
and large cells are sorted side by side, not one after the other."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def lipids(n):
    mem = M.vesicle(n, 7, f=1, chain_beads=5, n_centroids=10)
    k = np.flatnonzero(mem.type == 0)
    return [mem.pos[k], mem.vel[k], mem.ori[k], mem.angvel[k], mem.type[k], np.arange(n, dtype=np.uint32)]


def system(n, K, centroids=None, **kw):
    rows = lipids(n)
    g = G.System(G.make_params(kT=0.2, n_centroids=K, n_lloyd_init=0 if centroids is not None else 3, seed=3, **kw))
    g.set_particles(*rows)
    g.init_cells(None if centroids is None else rows[0][centroids])
    return g


def run(n, K, centroids=None):
    with system(n, K, centroids) as g:
        before = g.cells()
        place = np.empty(n, np.int64)
        place[before["slot_ids"]] = np.arange(n)
        g.integrate(1)
        c = g.cells()
        for cells, key in ((before, np.arange(n)), (c, place)):
            cell = cells["cell_of_id"]
            assert np.array_equal(cells["slot_ids"], np.lexsort((key, cell)))
        s = g.state()
        return [s[k] for k in ("pos", "vel", "ori", "angvel")], np.diff(before["start"])


@pytest.mark.parametrize("n, K", [(129, 1), (1000, 1), (2047, 1), (2048, 1), (2049, 1), (4095, 1), (4096, 1), (4097, 1),
                                  (6200, 1), (6200, 2), (6200, 9)])
def test_few_cells(n, K):
    got, sizes = run(n, K)
    assert sizes.max() >= n // K
    want, _ = run(n, max(n // 60, 2))
    for x, y in zip(got, want):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n, K, large", [(700, 7, 128), (6200, 62, 2048)])
def test_large_cell_among_small_ones(n, K, large):
    # all centroids but one near a pole, the last one's cell beyond the equator
    # (a row of neighbours holds 64 cells)
    up = np.argsort(-lipids(n)[0][:, 2], kind="stable")
    got, sizes = run(n, K, np.concatenate([up[:K - 1], up[-1:]]))
    assert sizes.max() > large and n <= 100 * K      # (still one launch builds the cells)
    want, _ = run(n, n // 60)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)


def rebuild_ms(n, K):
    with system(n, K) as g:
        g.integrate(2)
        best = np.inf
        for _ in range(15):
            g.set_timing(True)
            g.integrate(2)
            t = g.kernel_times()["rebuild"]
            best = min(best, t["ms"] / t["launches"])
        return best


def test_large_cells_side_by_side():
    # eight cells' sorts fill 8 of 152 SMs: a rebuild takes about as long as
    # with one of them (one after the other it takes well over twice as long)
    assert rebuild_ms(8 * 1300, 8) < 1.7 * rebuild_ms(1300, 1)
