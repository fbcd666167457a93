"""Repulsion between objects when the steps of one call run in one launch
(csrc/steps.cu): against one step per call, which finds the pairs and their
forces in kernels of their own.  Bodies in touch inside the box and through
its periodic sides, the later or the earlier of a pair at the image, bodies of
different sizes, none in touch, and walls.  Both sides sum in FP32 in their own
order: 1e-6 lu, as the other equalities of this kind."""
import numpy as np
import pytest

from paper_1312_3426_gb300 import lbib
from workloads import mesh, scenes

pytestmark = pytest.mark.gpu

NEAR = {
    "inside": [(12.0, 12.0, 12.0), (18.1, 12.4, 12.2)],
    "through x": [(3.0, 12.0, 12.0), (37.0, 12.3, 12.1)],
    "through z, earlier at the image": [(20.0, 12.0, 20.9), (20.2, 12.0, 3.0)],
    "three, two sizes": [(12.0, 12.0, 12.0), (18.1, 12.4, 12.2), (15.0, 12.2, 17.9)],
    "apart": [(8.0, 12.0, 8.0), (28.0, 12.0, 16.0)],
    "at the wall": [(12.0, 4.3, 12.0), (18.1, 4.3, 12.2)],
}


@pytest.mark.parametrize("where", list(NEAR))
def test_one_launch_equals_single_steps(where):
    sc = scenes.Scene("near", 40, 24, 24, walls=True, tau=0.9, body_force=(2e-5, 0.0, 0.0))
    for level in (2, 3):
        n, t = mesh.icosphere(level)
        sc.templates.append(scenes.Template(n, t, (3.0, 3.0, 3.0), **scenes.PAPER_MODULI))
    sc.objects += [scenes.Obj(i % 2, c, (0.3, 0.2, 0.1)) for i, c in enumerate(NEAR[where])]
    runs = []
    for single, rep in ((False, True), (True, True), (False, False)):
        g = lbib.Sim.from_scene(sc)
        if rep:
            lbib.lbib_set_repulsion(g.h, (5e-4, 1.5, 0.6), (1e-4, 1.2, 0.5))
        X = []
        for n in (40, 130):
            for _ in range(n if single else 1):
                g.step(1 if single else n)
            X.append(g.read_nodes()[0])
        runs.append(X)
        g.close()
    for a, b in zip(runs[0], runs[1]):
        assert np.abs(a - b).max() <= 1e-6
    moved = np.abs(runs[0][0] - runs[2][0]).max()
    assert moved > 1e-4 if where != "apart" else moved <= 1e-6
