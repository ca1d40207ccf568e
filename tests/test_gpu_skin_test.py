"""Cells rebuilt when a particle has moved beyond the skin: with a skin that a
few steps use up the trajectory is the every-step rebuild's bit for bit (a
missed rebuild would lose pairs); the same with the phases timed one by one
and with the fused step."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def run(n, timing=False, fusion=False, **kw):
    mem = M.vesicle(n, 13, kT=0.3, f=2, chain_beads=5, n_centroids=max(n // 60, 10))
    with G.System(G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=4,
                                **kw)) as g:
        g.load_membrane(mem)
        g.init_cells()
        g.set_timing(timing)
        g.set_step_fusion(fusion)
        for steps in (1, 17, 2, 20):
            g.integrate(steps)
        return g.state()


@pytest.mark.parametrize("n", [700, 12800])
@pytest.mark.parametrize("skin, every", [(0.02, 100), (0.02, 3)])
def test_skin_equals_every_step(n, skin, every):
    want = run(n)
    for mode in ({}, {"timing": True}, {"fusion": True}):
        got = run(n, rebuild_every=every, skin=skin, **mode)
        for k in ("pos", "vel", "ori", "angvel"):
            assert np.array_equal(got[k], want[k]), (mode, k)


def test_wide_skin_beyond_the_lists():
    """A skin that sends about one listed pair in ten beyond the lists' 32
    entries: the overflow list holds them, also those that the search lists
    within its margin only."""
    mem = M.biconcave(n_lipids=446_378, n_junctions=4_125, n_centroids=8_192, seed=2, name="rbc-500k")
    out = []
    for kw in ({}, {"rebuild_every": 20, "skin": 0.35}):
        with G.System(G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=4,
                                    **kw)) as g:
            g.load_membrane(mem)
            g.init_cells()
            g.integrate(3)
            out.append(g.state())
    for k in ("pos", "vel", "ori", "angvel"):
        assert np.array_equal(out[0][k], out[1][k]), k
