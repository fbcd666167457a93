"""A batch in which the largest template has no object: the sizes of a launch
follow the objects, so it equals the simulations stepped alone (up to the order
of the spreading's FP32 atomics: nodes 1e-6 lu)."""
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


def _scene(templates, radius):
    sc = scenes.Scene("unused", 32, 24, 24)
    for nodes, tris in templates:
        sc.templates.append(scenes.Template(nodes, tris, (radius,) * 3, **scenes.PAPER_MODULI))
    sc.objects += [scenes.Obj(len(templates) - 1, (8.2, 12.1, 11.9)), scenes.Obj(len(templates) - 1, (24.2, 11.7, 12.3))]
    return sc


# 2562, 4098 (more than one block's shared memory) and 4 nodes nobody uses, beside objects of 162 and 642
@pytest.mark.parametrize("unused", [mesh.icosphere(4), mesh.octasphere(5), mesh.tetrahedron()],
                         ids=["level4", "4098", "tetrahedron"])
@pytest.mark.parametrize("other", [2, 3])
def test_batch_with_an_unused_template_equals_individual_steps(unused, other):
    small = mesh.icosphere(2)
    scs = [_scene([unused, small], 3.0), _scene([mesh.icosphere(other)], 3.5)]
    batch, alone = ([lbib.Sim.from_scene(s) for s in scs] for _ in range(2))
    for b, a in zip(batch, alone):
        for k in range(2):
            x = a.read_nodes(k)[0]
            x[:, 1] = (x[:, 1] - x[:, 1].mean()) * 1.02 + x[:, 1].mean()
            for g in (a, b):
                g.object_set_nodes(k, x)
    for n in (20, 3):  # a captured chunk of 16 and 4 more; no chunk
        lbib.lbib_batch_step([b.h for b in batch], n)
        for a in alone:
            a.step(n)
    for b, a in zip(batch, alone):
        b.sync()
        assert np.abs(b.read_nodes()[0] - a.read_nodes()[0]).max() <= 1e-6
    for g in batch + alone:
        g.close()
