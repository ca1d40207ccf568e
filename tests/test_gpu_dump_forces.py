"""Reading the pair list leaves the forces as they are, with the volume
constraint's pressure in them, and so the steps that follow."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


@pytest.mark.parametrize("precision", [G.F32_FORCE_F64_STATE, G.F64_ALL, G.F32_FORCE_F32_STEP])
@pytest.mark.parametrize("constraint", [False, True])
def test_dump_keeps_forces(precision, constraint):
    mem = M.vesicle(1279, 7, f=1, chain_beads=4, n_centroids=20)
    out = []
    for dump in (False, True):
        with G.System(G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=3,
                                    precision=precision)) as g:
            g.load_membrane(mem)
            g.init_cells()
            if constraint:
                # 2 % off the target volume: a pressure well above the
                # forces' resolution
                g.set_volume_constraint(1e-3, 0.98 * g.volume(1.09), 1.09)
            for call in (g.compute_forces, lambda: g.integrate(2)):
                call()
                before = g.forces()
                if dump:
                    assert len(g.pairs()) > 0
                for x, y in zip(before, g.forces()):
                    assert np.array_equal(x, y)
            g.integrate(1)
            s = g.state()
            out.append([*g.forces(), *(s[k] for k in ("pos", "vel", "ori", "angvel"))])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
