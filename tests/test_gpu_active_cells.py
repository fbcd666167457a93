"""The active-cell mask (the corners of every node, reset every 128 steps): an
object that crosses a cell every few steps, through the periodic faces and
across several resets, against the FP64 oracle.  A cell that a reset forgot
would keep an old spread force (found again when the second object, on the same
track, comes by), one that was not marked in time would miss a force or give a
stale velocity.  Bars as stated for the method: velocity 1e-5 relative L2, nodes
1e-6 lu."""
import numpy as np
import pytest

import oracle
from paper_1312_3426_gb300 import lbib
from workloads import mesh, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


@pytest.mark.parametrize("speed", [(0.3, 0.0, 0.0), (-0.21, 0.02, 0.37)])
@pytest.mark.parametrize("batched", [False, True])
def test_fast_objects_across_mask_resets(speed, batched):
    nodes, tris = mesh.icosphere(2)
    sc = scenes.Scene("fast", 40, 24, 32, friction=0.01)
    sc.templates.append(scenes.Template(nodes, tris, (4.0, 4.0, 4.0), **scenes.PAPER_MODULI))
    for x in (10.3, 30.7):
        sc.objects.append(scenes.Obj(0, (x, 11.9, 16.2), mass=20.0))
    o, g = oracle.Oracle.from_scene(sc), lbib.Sim.from_scene(sc)
    for k in range(2):
        v = np.tile(speed, (len(nodes), 1))
        o.object_set_velocities(k, v)
        g.object_set_velocities(k, v)
    x0 = o.read_nodes(0)[0]
    o.step(300)
    if batched:
        lbib.lbib_batch_step([g.h], 300)
    else:
        g.step(300)
    u, uo = g.velocity()[:, :, 1:-1].astype(np.float64), o.velocity()[:, :, 1:-1]
    assert np.abs(o.read_nodes(0)[0] - x0).max() > 20  # cells crossed
    assert np.linalg.norm(u - uo) <= 1e-5 * np.linalg.norm(uo)
    for k in range(2):
        assert np.abs(g.read_nodes(k)[0] - o.read_nodes(k)[0]).max() <= 1e-6
    g.close()
