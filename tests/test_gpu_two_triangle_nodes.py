"""Nodes with only two triangles: a doubled triangle (front and back) that hangs
from one node of a closed mesh.  Such a mesh is accepted, and the walk around its
free nodes has three records, fewer than any other.  Every modulus but bending
(the rest angle of a folded edge is a full turn, where the angle is not
continuous), each alone and all together, against the oracle: the method's bar of
1e-6 lu for the node positions."""
import numpy as np
import pytest

import oracle
from paper_1312_3426_gb300 import lbib
from workloads import mesh, scenes

pytestmark = pytest.mark.gpu

MODULI = dict(ks=0.1, kal=0.1, kag=0.4, kv=1.0)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


def _hanging(nodes, tris, flaps):
    """`flaps` doubled triangles, each with two nodes of its own, on the first
    nodes, in planes of constant z (their folded rest angles are then exact)."""
    x, t = [nodes], [tris]
    n = len(nodes)
    for k in range(flaps):
        out = np.copysign(0.5, nodes[k])
        x.append(nodes[k] + np.array([[out[0], 0.0, 0.0], [0.0, out[1], 0.0]]))
        t.append(np.array([[k, n, n + 1], [k, n + 1, n]], np.int32))
        n += 2
    return np.concatenate(x), np.concatenate(t).astype(np.int32)


@pytest.mark.parametrize("base,flaps", [(mesh.tetrahedron(), 1), (mesh.icosphere(2), 40)], ids=["tetrahedron", "icosphere2"])
@pytest.mark.parametrize("moduli", [("ks",), ("kal",), ("kag",), ("kv",), ("ks", "kal", "kag", "kv")],
                         ids=lambda m: "+".join(m))
@pytest.mark.parametrize("calls", [(1,) * 40, (40,)], ids=["single", "many"])  # separate launches, many steps in one
def test_forces_of_hanging_triangles(base, flaps, moduli, calls):
    nodes, tris = _hanging(*base, flaps)
    radius = 2.0 if len(base[0]) == 4 else 4.0
    sc = scenes.Scene("hanging", 40, 24, 24)
    sc.templates.append(scenes.Template(nodes, tris, (radius,) * 3, **{k: MODULI[k] for k in moduli}))
    sc.objects.append(scenes.Obj(0, (20.1, 12.2, 11.8), mass=10.0))
    o, g = oracle.Oracle.from_scene(sc), lbib.Sim.from_scene(sc)
    x, _ = o.read_nodes(0)
    c = x.mean(0)
    x = c + (x - c) * np.array([1.05, 1.0 / 1.05, 1.02])
    for s in (o, g):
        s.object_set_nodes(0, x)
    o.step(sum(calls))
    for n in calls:
        g.step(n)
    xo, xg = o.read_nodes(0)[0], g.read_nodes(0)[0]
    g.close()
    assert np.abs(xo - x)[len(base[0]):].max() > 1e-4  # the hanging nodes moved
    assert np.abs(xg - xo).max() <= 1e-6
