"""Node states between host and device: read-outs and replaced nodes, on both
sides of the size from which the conversion runs on the device, give back what
was set, to the 48 bits of the device's FP32 pairs."""
import numpy as np
import pytest

from paper_1312_3426_gb300 import lbib
from workloads import mesh

pytestmark = pytest.mark.gpu

REL = 2.0 ** -46  # hi + lo of a value below 256: 24 + 23 bits and the rounding of lo


def channel(level, objects, posts=False):
    g = lbib.Sim(64, 48, 48, tau=1.0, friction=0.05)
    if posts:
        solid = np.zeros((48, 48, 64), np.uint8)
        solid[20:24, :, 30:34] = 1
        lbib.lbib_set_solid(g.h, solid)
    xyz, tri = mesh.icosphere(level)
    t = g.template_create(xyz, tri, stretch=(4.0, 4.0, 4.0), ks=0.1, kb=0.03, kal=0.1, kag=0.4, kv=1.0)
    for k in range(objects):
        g.object_add(t, (10.0 + 14.0 * (k % 4), 12.0 + 12.0 * (k // 4 % 3), 10.0 + 14.0 * (k // 12)))
    g.fluid_init()
    return g, len(xyz)


# 162 nodes a body: 4050 and 4212 nodes lie on the two sides of 4096
@pytest.mark.parametrize("level,objects,posts", [(2, 1, False), (2, 25, False), (2, 26, False), (3, 7, False),
                                                 (2, 26, True)])
def test_replaced_nodes_and_read_outs(level, objects, posts):
    g, n = channel(level, objects, posts)
    rng = np.random.default_rng(level + objects)
    g.step(3)
    X0, V0 = g.read_nodes()
    # some positions, some velocities, one of both: the others stay the device's
    X, V = X0.copy(), V0.copy()
    for o in range(objects):
        s = slice(o * n, (o + 1) * n)
        if o % 3 != 1:
            X[s] += rng.uniform(-1e-3, 1e-3, (n, 3))
            g.object_set_nodes(o, X[s])
        if o % 3 != 0:
            V[s] = rng.uniform(-1e-3, 1e-3, (n, 3))
            g.object_set_velocities(o, V[s])
    g.objects_analyze()  # uploads
    g.step(0)
    X1, V1 = g.read_nodes()
    assert np.array_equal(X1, X) and np.array_equal(V1, V)  # the mirror
    for o in range(objects):
        s = slice(o * n, (o + 1) * n)
        a, b = lbib.lbib_read_nodes(g.h, o, n)
        assert np.array_equal(a, X[s]) and np.array_equal(b, V[s])
    g.step(2)
    A, W = g.read_nodes()
    B, U = g.read_nodes()
    assert np.array_equal(A, B) and np.array_equal(W, U)
    for o in range(objects):
        a, b = lbib.lbib_read_nodes(g.h, o, n)
        s = slice(o * n, (o + 1) * n)
        assert np.array_equal(a, A[s]) and np.array_equal(b, W[s])
    # every object replaced: nothing of the device's state is left, and an
    # upload followed by a step of an equal new simulation gives its nodes
    for o in range(objects):
        s = slice(o * n, (o + 1) * n)
        g.object_set_nodes(o, X[s])
        g.object_set_velocities(o, V[s])
    g.fluid_init()
    g.step(1)
    h, _ = channel(level, objects, posts)
    for o in range(objects):
        s = slice(o * n, (o + 1) * n)
        h.object_set_nodes(o, X[s])
        h.object_set_velocities(o, V[s])
    h.step(1)
    (a, b), (c, d) = g.read_nodes(), h.read_nodes()
    assert np.abs(a - c).max() <= 256 * REL and np.abs(b - d).max() <= 256 * REL


def test_read_outs_between_steps_change_nothing():
    """Read-outs pass through the population buffer the next step overwrites."""
    got = []
    for read in (False, True):
        g = lbib.Sim(62, 40, 38, tau=0.8, body_force=(1e-5, 0, 0))
        g.fluid_init()
        for k in range(7):
            g.step(1 + k % 3)
            if read:
                u = g.velocity()
                assert np.isfinite(u).all() and not u[:, :, [0, -1]].any()
                g.density(), g.mass()
        got.append((g.populations(), g.velocity()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
