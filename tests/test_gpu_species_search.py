"""The neighbour search in its species-pair form (band-3, glycophorin) with wide
cells, whose distance tests round most, and with a skin that the steps use up:
the trajectory is that of small cells rebuilt every step, bit for bit, with
FP32 and with FP64 pair terms."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")

EPS = [[0.0, 1.2, 0.9], [1.2, 1.4, 1.1], [0.9, 1.1, 0.0]]
RC = [[0.0, 2.8, 0.0], [2.8, 2.9, 2.7], [0.0, 2.7, 0.0]]


def run(mem, K, steps, **kw):
    with G.System(G.make_params(kT=mem.kT, n_centroids=K, n_lloyd_init=3, seed=4, eps_mem=EPS, rc_mem=RC, **kw)) as g:
        g.load_membrane(mem)
        g.init_cells()
        g.integrate(steps)
        s = g.state()
        return [s[k] for k in ("pos", "vel", "ori", "angvel")], np.diff(g.cells()["start"]).max()


@pytest.mark.parametrize("precision", [G.F32_FORCE_F64_STATE, G.F64_ALL])
@pytest.mark.parametrize("lipids, K, skin", [(9000, 2, 0.0), (9000, 2, 0.2), (9000, 12, 0.3), (9000, 40, 0.05)])
def test_wide_cells(precision, lipids, K, skin):
    mem = M.with_membrane_proteins(M.vesicle(lipids, 3, kT=0.3, f=3, chain_beads=6), seed=4)
    kw = {"rebuild_every": 50, "skin": skin} if skin else {}
    got, largest = run(mem, K, 20, precision=precision, **kw)
    assert largest >= len(mem.type) // K
    want, _ = run(mem, len(mem.type) // 60, 20, precision=precision)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
