"""The rotational update on the GPU where the fixed-point code hands lipids
to the FP64 code: fast rotations, constants outside its range.  Against the FP64 oracle with FP64 forces; the state is
rounded onto the 2^-40 grid ten times a step and the force sums onto 2^-32,
so after two steps the RMS distance stays well below 1e-9 dt-scaled units."""
import numpy as np
import pytest

import oracle
from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


@pytest.mark.parametrize("dt, spin", [(0.01, 1.0), (0.01, 12.0), (0.01, 60.0), (1e-8, 1.0)])
def test_rotation_matches_oracle(dt, spin):
    mem = M.flat_patch_2304()
    mem.angvel = mem.angvel * spin
    p = G.make_params(kT=mem.kT, dt=dt, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=0,
                      precision=G.F64_ALL)
    o = oracle.OracleSystem(oracle.model(box=mem.box, periodic=mem.periodic),
                            oracle.run(kT=mem.kT, dt=dt, n_centroids=mem.n_centroids, seed=0))
    with G.System(p) as g:
        g.load_membrane(mem)
        g.init_cells()
        g.integrate(2)
        sg = g.state()
    o.load(mem)
    o.init_cells()
    o.integrate(2)
    so = o.state()
    for k in ("pos", "ori", "angvel", "vel"):
        assert np.sqrt(((sg[k] - so[k]) ** 2).sum(1).mean()) <= 1e-9, k
