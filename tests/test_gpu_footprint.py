"""lbib_footprint_bytes covers what a simulation holds after its first step, also
where the membrane launch keeps its edge scalars in memory (two blocks per object),
with objects of 4098, 162 and 42 nodes side by side; and each object has its own
place there: equal to the launch that keeps them in shared memory, up to the
order of the sums and atomics (nodes 1e-6 lu, as the other equalities of launch shapes)."""
import numpy as np
import pytest

from paper_1312_3426_gb300 import lbib
from workloads import mesh, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


def _run(cluster, batched):
    sc = scenes.Scene("mixed", 60, 40, 40)
    for m, r in ((mesh.octasphere(5), 7.0), (mesh.icosphere(1), 2.0), (mesh.icosphere(2), 3.0)):
        sc.templates.append(scenes.Template(m[0], m[1], (r,) * 3, **scenes.PAPER_MODULI))
    sc.objects.append(scenes.Obj(0, (50.0, 20.0, 20.0)))
    for k in range(30):
        sc.objects.append(scenes.Obj(1 + k % 2, (5.0 + 9.0 * (k % 4), 8.0 + 10.0 * (k // 4 % 3), 6.0 + 12.0 * (k // 12)), mass=4.0))
    g = lbib.Sim.from_scene(sc)
    lbib.lbib_set_tuning(g.h, lbib.LBIB_TUNE_IB_CLUSTER, cluster)
    for oid in (0, 1, 2, 30):
        x, _ = g.read_nodes(oid)
        g.object_set_nodes(oid, x.mean(0) + (x - x.mean(0)) * np.array([1.03, 1.0 / 1.03, 1.0]))
    start, _ = g.read_nodes()
    if batched:
        lbib.lbib_batch_step([g.h], 20)
    else:
        g.step(20)
    g.sync()
    params = lbib.fluid_params(sc.nx, sc.ny, sc.nz, sc.walls, sc.tau, sc.rho0, sc.body_force, sc.friction)
    said = lbib.lbib_footprint_bytes(params, sc.n_nodes, sum(len(t.tris) for t in sc.templates))
    held, nodes = int(g.info()[5]), g.read_nodes()[0]
    g.close()
    return held, said, nodes, np.abs(nodes - start).max()


@pytest.mark.parametrize("batched", [False, True])
def test_footprint_covers_the_edge_scalars(batched):
    shared = _run(1, False)
    held, said, nodes, moved = _run(2, batched)
    assert shared[0] <= said and held <= said
    assert held > shared[0]  # the scalars are in memory
    assert moved > 0.01 and np.abs(nodes - shared[2]).max() <= 1e-6
