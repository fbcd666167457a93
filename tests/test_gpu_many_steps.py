"""Small simulations run the steps of one call in one launch (csrc/steps.cu):
against the same simulation stepped one step per call, which launches each
kernel on its own.  Without objects the populations are bit-identical; with
them the spreading's FP32 atomics are summed in another order (nodes 1e-6 lu, as
the other equalities of this kind; 1e-3 for 16-bit storage, whose stochastic
rounding turns a last-place difference into one of a 16-bit number, the bar of
the 16-bit parity tests).  Boxes below and above one block's tile, odd and even
widths, all storage types, with and without walls, obstacles and an inlet, and
several runs between mask resets."""
import numpy as np
import pytest

from paper_1312_3426_gb300 import lbib
from workloads import geometry, mesh, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


def _scene(nx, ny, nz, walls, objects, obstacles):
    sc = scenes.Scene("many", nx, ny, nz, walls=walls, tau=0.9, body_force=(2e-5, 1e-6, -1e-6))
    if obstacles:
        sc.solid = geometry.staggered_rhomboids(nx, ny, nz, count=2, seed=5)
        sc.inlet = ((0, 1, 1, ny - 1, 0, nz), (0.01, 0.0, 0.0))
    if objects:
        for level, r in ((2, 3.0), (3, 4.0)):
            n, t = mesh.biconcave(level)
            sc.templates.append(scenes.Template(n, t, (r, r, r), **scenes.PAPER_MODULI))
        sc.objects += [scenes.Obj(0, (nx / 4, ny / 2, nz / 4), (0.3, 0.2, 0.1)),
                       scenes.Obj(1, (3 * nx / 4, ny / 2, 3 * nz / 4), (0.1, 0.9, 0.4))]
    return sc


def _pair(sc, prec):
    return [lbib.Sim.from_scene(sc, precision=prec, pop_scale_log2=0 if prec == "f32" else 12) for _ in range(2)]


@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("box,walls,obstacles", [((1, 3, 1), True, False), ((6, 5, 7), False, False),
                                                 ((37, 19, 29), True, False), ((40, 20, 20), False, False),
                                                 ((38, 20, 30), True, True), ((100, 50, 61), True, False)])
def test_fluid_alone_is_bit_identical(box, walls, obstacles, prec):
    many, single = _pair(_scene(*box, walls, False, obstacles), prec)
    for n in (2, 131, 1, 7):
        many.step(n)
        for _ in range(n):
            single.step(1)
        assert np.array_equal(many.populations(), single.populations()), n
    many.close()
    single.close()


@pytest.mark.parametrize("prec,bar", [("f32", 1e-6), ("f16s", 1e-3), ("bf16s", 1e-3)])
@pytest.mark.parametrize("box,walls,obstacles", [((40, 20, 24), True, False), ((37, 20, 29), False, False),
                                                 ((60, 20, 30), True, True), ((100, 50, 60), True, False)])
def test_with_objects_equals_single_steps(box, walls, obstacles, prec, bar):
    many, single = _pair(_scene(*box, walls, True, obstacles), prec)
    for n in (3, 140, 20):
        many.step(n)
        for _ in range(n):
            single.step(1)
        for k in range(2):
            assert np.abs(many.read_nodes(k)[0] - single.read_nodes(k)[0]).max() <= bar, n
    many.close()
    single.close()
