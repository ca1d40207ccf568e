"""Two systems on one caller's stream, stepped by a thread each while their
step graphs are captured again and again: each as alone, bit for bit."""
import threading

import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_1701_02059_gb300")


def steps(mem, seed, stream):
    with G.System(G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=seed),
                  stream=stream) as g:
        g.load_membrane(mem)
        g.init_cells()
        v0 = g.volume(1.09)
        for k in range(6):
            # (a change of the constraint drops the captured steps)
            g.set_volume_constraint(1e-4, v0 * (1.0 - 1e-4 * k), 1.09)
            g.integrate(12)
        return g.state()


def test_two_threads():
    mems = [M.vesicle(n, 5, f=2, chain_beads=5, n_centroids=n // 60) for n in (3000, 1300)]
    want = [steps(m, k, None) for k, m in enumerate(mems)]
    stream = torch.cuda.Stream()
    got, err = [None, None], []

    def work(k):
        try:
            got[k] = steps(mems[k], k, stream.cuda_stream)
        except Exception as e:      # (an assertion in a thread would be lost)
            err.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not err and not any(t.is_alive() for t in threads)
    for a, b in zip(got, want):
        for k in ("pos", "vel", "ori", "angvel"):
            assert np.array_equal(a[k], b[k]), k
