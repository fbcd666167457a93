"""The membrane kernel's node walks where they can go wrong, in a channel
against the FP64 oracle over the launch shapes (the step's own choice, blocks
of a cluster with the edge scalars in global memory, several objects per
block): a body with a node in which two fans of triangles meet, and one with
two nodes of valence 70.

Bars as stated for the method: velocity 1e-5 relative L2, nodes 1e-6 lu;
1e-5 lu for the valence-70 body, whose triangles are 11 times longer than
wide (a height is the small difference of two long sides).  Node mass 10, as
for the other bodies of few large triangles."""
import numpy as np
import pytest

import oracle
from paper_1312_3426_gb300 import lbib
from test_ring_walks_cpu import bipyramid, pinched
from workloads import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


@pytest.mark.parametrize("threads,cluster,group", [(0, 1, 1), (32, 2, 1), (32, 1, 2)])
@pytest.mark.parametrize("mesh,radius,bar", [(pinched, 4.0, 1e-6), (lambda: bipyramid(70), 8.0, 1e-5)],
                         ids=["two_fans", "valence70"])
def test_walks_match_oracle(mesh, radius, bar, threads, cluster, group):
    nodes, tris = mesh()
    sc = scenes.Scene("walks", 64, 32, 40)
    sc.templates.append(scenes.Template(nodes, tris, (radius,) * 3, **scenes.PAPER_MODULI))
    for x in (15.2, 46.1):
        sc.objects.append(scenes.Obj(0, (x, 15.9, 20.4), (0.3, 0.9, -0.2), 10.0))
    o, g = oracle.Oracle.from_scene(sc), lbib.Sim.from_scene(sc)
    if threads:
        lbib.lbib_set_tuning(g.h, lbib.LBIB_TUNE_MEMBRANE_THREADS, threads)
    lbib.lbib_set_tuning(g.h, lbib.LBIB_TUNE_IB_CLUSTER, cluster)
    if group > 1:
        lbib.lbib_set_tuning(g.h, lbib.LBIB_TUNE_MEMBRANE_GROUP, group)
    o.step(100)
    g.step(100)
    u, uo = g.velocity()[:, :, 1:-1].astype(np.float64), o.velocity()[:, :, 1:-1]
    assert np.linalg.norm(u - uo) <= 1e-5 * np.linalg.norm(uo)
    for k in range(2):
        assert np.abs(g.read_nodes(k)[0] - o.read_nodes(k)[0]).max() <= bar
    g.close()
