"""Two cells per thread at odd widths (pairs that lie in two rows, a last cell
alone, rows of one cell) against the one-cell kernel
(LBIB_TUNE_FLUID_KERNEL = 3): the same arithmetic and rounding bits, so exactly the
same populations, alone, in one launch and batched.  FP32 has no such switch; its
one-cell kernel runs the steps of a small box in one launch, its two-cells
kernel single steps."""
import numpy as np
import pytest

from paper_1312_3426_gb300 import lbib

pytestmark = pytest.mark.gpu

BOXES = [(1, 3, 1, True), (1, 4, 3, False), (3, 5, 3, True), (5, 4, 7, False), (37, 19, 29, True), (101, 37, 53, True),
         (63, 6, 8, False), (255, 9, 5, True)]


def make(box, prec, kernel):
    nx, ny, nz, walls = box
    g = lbib.Sim(nx, ny, nz, walls=walls, tau=0.8, body_force=(2e-5, 1e-6, -3e-6), precision=prec,
                 pop_scale_log2=0 if prec == "f32" else 12)
    lbib.lbib_set_tuning(g.h, lbib.LBIB_TUNE_FLUID_KERNEL, kernel)
    g.fluid_init()
    rng = np.random.default_rng(nx)
    g.set_populations(rng.uniform(-1e-3, 1e-3, g.populations().shape))
    return g


@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("box", BOXES)
def test_equals_the_one_cell_kernel(box, prec):
    one, single, many, batched = (make(box, prec, k) for k in (3, 1, 1, 1))
    for n in (1, 2, 20):
        one.step(n)
        for _ in range(n):
            single.step(1)
        many.step(n)
        lbib.lbib_batch_step([batched.h], n)
        want = one.populations()
        for g in (single, many, batched):
            assert np.array_equal(g.populations(), want), n
