"""Fewer membrane blocks than objects beside a long fluid update (the default
there) against one block per object: every object is updated, in a launch whose
last round is nearly empty and in one where it is full.  The sums of an object
do not depend on the block; the spreading's FP32 atomics do (nodes 1e-6 lu, as
the other equalities of this kind)."""
import numpy as np
import pytest

from paper_1312_3426_gb300 import lbib
from workloads import mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("objects", [153, 304, 320])
def test_shared_blocks_equal_one_block_per_object(objects):
    n, t = mesh.icosphere(2)
    got = []
    for clusters in (0, 65535):
        g = lbib.Sim(200, 162, 180, tau=0.9, body_force=(2e-5, 0, 0))
        lbib.lbib_set_tuning(g.h, lbib.LBIB_TUNE_MEMBRANE_CLUSTERS, clusters)
        tid = g.template_create(n, t, stretch=(4.0, 4.2, 3.9), ks=0.1, kb=0.03, kal=0.1, kag=0.4, kv=1.0)
        rng = np.random.default_rng(objects)
        for k in range(objects):
            where = np.array([10.0 + 12 * (k % 15), 10.0 + 12 * (k // 15 % 11), 10.0 + 12 * (k // 165)])
            g.object_add(tid, where + rng.uniform(-0.4, 0.4, 3), rotate=rng.uniform(0, 6, 3))
            assert g.n_nodes[tid] == len(n)
        g.fluid_init()
        X = np.concatenate([lbib.lbib_read_nodes(g.h, k, len(n))[0] * (1 + 1e-3) for k in range(objects)])
        for k in range(objects):  # away from rest
            g.object_set_nodes(k, X[k * len(n):(k + 1) * len(n)])
        g.step(6)
        got.append(g.read_nodes())
        g.close()
    assert np.abs(got[0][0] - X).max(axis=1).reshape(objects, -1).max(axis=1).min() > 0  # every object moved
    assert np.abs(got[0][0] - got[1][0]).max() <= 1e-6
