"""A batched call whose membrane forces are stale (nodes replaced since the last
call) after a graph was captured, with two size classes of objects launched on
two streams: the first membrane launch of the call waits for work of this call,
not for an event of the captured graph.  Compared with the same simulations
stepped alone (equal up to the order of the spreading's FP32 atomics, as the
other batch tests: nodes 1e-6 lu)."""
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


def _scene(level, radius):
    nodes, tris = mesh.icosphere(level)
    sc = scenes.Scene(f"l{level}", 32, 24, 24)
    sc.templates.append(scenes.Template(nodes, tris, (radius,) * 3, **scenes.PAPER_MODULI))
    sc.objects.append(scenes.Obj(0, (10.2, 12.1, 11.9)))
    return sc


@pytest.mark.parametrize("group", [0, 2])  # 0: the step's own choice
def test_nodes_replaced_between_batched_calls(group):
    scs = [_scene(3, 4.0), _scene(2, 3.0), _scene(2, 4.0)]  # 642 nodes, 162 nodes: two classes
    batch, alone = ([lbib.Sim.from_scene(s) for s in scs] for _ in range(2))
    if group:
        lbib.lbib_set_tuning(batch[0].h, lbib.LBIB_TUNE_MEMBRANE_GROUP, group)
    for rep in range(3):
        for b, a in zip(batch, alone):
            x = a.read_nodes(0)[0] + np.array([0.3, 0.0, -0.2])
            x[:, 1] = (x[:, 1] - 12.0) * 1.01 + 12.0
            for g in (a, b):
                g.object_set_nodes(0, x)
        lbib.lbib_batch_step([b.h for b in batch], 20)  # a captured chunk of 16 and 4 more
        for a in alone:
            a.step(20)
        for b, a in zip(batch, alone):
            assert np.abs(b.read_nodes(0)[0] - a.read_nodes(0)[0]).max() <= 1e-6, rep
    for g in batch + alone:
        g.close()
