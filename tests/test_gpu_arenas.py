"""States and tapes reuse each other's device memory: what one leaves behind
must not show in the next, whatever the order, the sizes and the threads."""
import threading

import numpy as np
import pytest

from paper_1807_00672_gb300 import inputs, swe

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


def rollout(mesh, c, steps, K):
    st = swe.State(mesh, c.h, c.hu, c.hv, c.z, c.n)
    tape = swe.Tape(st, steps, K, [0, 7])
    g = tape.grad(g_h=np.linspace(0.5, 1.5, mesh.T), g_gauge=np.ones((steps, 2)))
    out = [*st.fields(), tape.gauge_h, *(g[k] for k in ("h", "hu", "hv", "z", "n"))]
    tape.close()
    st.close()
    return out


def test_reused_memory_does_not_show():
    ensure_built()
    cases = [inputs.random_flow_case(nx=nx, ny=ny, seed=nx) for nx, ny in ((40, 31), (33, 29), (12, 9))]
    jobs = [(c, prec, steps, K) for c in cases for prec in ("f64", "f32")
            for steps, K in ((6, 2), (7, 7))]
    fresh = []
    for c, prec, steps, K in jobs:  # one mesh at a time: nothing is kept from the job before
        mesh = swe.Mesh(c.mesh.xy, c.mesh.tri, precision=prec)
        fresh.append(rollout(mesh, c, steps, K))
        mesh.close()
    bad = cases[0]
    meshes = {(i, p): swe.Mesh(c.mesh.xy, c.mesh.tri, precision=p)
              for i, c in enumerate(cases) for p in ("f64", "f32")}

    def poison():  # a state full of NaN leaves its memory behind
        for p in ("f64", "f32"):
            with pytest.raises(swe.SweError):
                swe.State(meshes[0, p], bad.h * np.nan, bad.hu, bad.hv, bad.z, bad.n)

    def worker(order, errors):
        try:
            for j in order:
                c, prec, steps, K = jobs[j]
                i = next(k for k, x in enumerate(cases) if x is c)
                mesh = meshes[i, prec] if errors is None else swe.Mesh(c.mesh.xy, c.mesh.tri, precision=prec)
                for a, b in zip(rollout(mesh, c, steps, K), fresh[j]):
                    assert np.array_equal(a, b), jobs[j][1:]
        except Exception as e:  # noqa: BLE001
            if errors is None:
                raise
            errors.append(e)

    order = np.random.default_rng(1).permutation(len(jobs))
    for _ in range(2):
        poison()
        worker(order, None)
    errors = []  # threads with meshes (and streams) of their own
    threads = [threading.Thread(target=worker, args=(np.roll(order, 3 * t), errors)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
