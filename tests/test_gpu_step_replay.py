"""Steps replayed as CUDA graphs against the same launches made one by one
(timing on), bit for bit: however the steps are cut into calls, on either
state buffer, with the cells read in between, and after a change that makes
the captured step stale (the volume constraint)."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def system(precision):
    mem = M.vesicle(3000, 5, f=2, chain_beads=5, n_centroids=50)
    g = G.System(G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=3,
                               precision=precision))
    g.load_membrane(mem)
    g.init_cells()
    return g


def everything(g):
    s, c = g.state(), g.cells()
    return [s[k] for k in ("pos", "vel", "ori", "angvel")] + [np.array(s["step"])] + [c[k] for k in sorted(c)]


@pytest.mark.parametrize("precision", [G.F32_FORCE_F64_STATE, G.F64_ALL, G.F32_FORCE_F32_STEP])
@pytest.mark.parametrize("cuts", [[24], [1] * 24, [3, 1, 9, 2, 9]])
def test_replay_equals_launches(precision, cuts):
    with system(precision) as a, system(precision) as b:
        b.set_timing(True)
        for n in cuts:
            a.integrate(n)
            b.integrate(n)
            for x, y in zip(everything(a), everything(b)):
                assert np.array_equal(x, y)


def test_replay_after_a_change():
    with system(G.F32_FORCE_F64_STATE) as a, system(G.F32_FORCE_F64_STATE) as b:
        b.set_timing(True)
        for g in (a, b):
            g.integrate(12)
            g.set_volume_constraint(1e-4, 0.98 * g.volume(1.09), 1.09)
            g.integrate(12)
            g.set_volume_constraint(0.0, 0.0, 1.09)
            g.quench(9, 0.005)
            g.quench(9, 0.003)
            g.integrate(11)
        for x, y in zip(everything(a), everything(b)):
            assert np.array_equal(x, y)
