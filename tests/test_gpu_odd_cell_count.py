"""An odd number of cells: the two-cells kernel's last thread has one cell and a
place of padding, which holds whatever was last stored there (node read-outs pass
through the population buffers, and the one-cell kernels do not write it).  The
padding takes no part: a healthy run stays healthy and equals one that was never
read in between, through many steps in one launch, batched and single steps."""
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


def _scene():
    nodes, tris = mesh.icosphere(4)  # two of them: enough nodes for the transfer on the device
    sc = scenes.Scene("odd", 23, 21, 23, body_force=(2e-5, 1e-5, -1e-5))
    sc.templates.append(scenes.Template(nodes, tris, (6.0,) * 3, **scenes.PAPER_MODULI))
    sc.objects += [scenes.Obj(0, (6.1, 10.3, 6.2)), scenes.Obj(0, (17.2, 10.6, 17.4))]
    return sc


# bound: the order of the spreading's FP32 atomics, and in 16 bits the roundings that fall the other way for it
@pytest.mark.parametrize("prec,scale,bound", [("f32", 0, 1e-4), ("f16s", 12, 1e-2)])
def test_padding_takes_no_part(prec, scale, bound):
    sc = _scene()
    read, quiet = (lbib.Sim.from_scene(sc, precision=prec, pop_scale_log2=scale) for _ in range(2))
    assert read.info()[3] % 2 == 1 and read.info()[2] >= 4096
    for how, n in [("many", 2), ("single", 1), ("many", 3), ("single", 1), ("batch", 2), ("single", 1), ("batch", 17),
                   ("single", 2)]:
        for g in (read, quiet):
            if how == "batch":
                lbib.lbib_batch_step([g.h], n)
            elif how == "many":
                g.step(n)
            else:
                for _ in range(n):
                    g.step(1)
        read.sync()
        read.read_nodes()
    ur, uq = read.velocity(), quiet.velocity()
    assert np.abs(ur - uq).max() <= bound * np.abs(uq).max()
    assert np.abs(read.read_nodes()[0] - quiet.read_nodes()[0]).max() <= 1e-6
    for g in (read, quiet):
        g.close()
