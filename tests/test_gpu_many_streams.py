"""Simulations on streams of their own: a launch of many steps, whose blocks hold
their SMs while they wait, takes no more than half of the device then (seen by the
profiler), and simulations that run at once equal the same ones alone (up to the
order of the spreading's FP32 atomics: nodes 1e-6 lu, velocities 1e-5)."""
import json

import numpy as np
import pytest
import torch

from paper_1312_3426_gb300 import lbib
from workloads import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


@pytest.fixture
def one_launch(tmp_path):
    from torch.profiler import ProfilerActivity, profile

    def names(work):
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            work()
            torch.cuda.synchronize()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        with open(tmp_path / "trace.json") as f:
            return [e["name"] for e in json.load(f)["traceEvents"] if e.get("cat") == "kernel"]

    for _ in range(2):  # the first trace of a process may be empty
        seen = names(lambda: torch.zeros(64, device="cuda").add_(1))
    if not seen:
        pytest.skip("no kernel tracing on this machine")

    def check(g):
        found = names(lambda: g.step(4))
        assert found
        return any("k_steps" in n for n in found)

    return check


def test_one_launch_leaves_room_for_other_streams(one_launch):
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    free = scenes.Scene("free", 64, 64, 64)  # more than half of the SMs
    g = lbib.Sim.from_scene(free, stream=a.cuda_stream)
    assert one_launch(g)
    same = lbib.Sim.from_scene(free, stream=a.cuda_stream)
    assert one_launch(g) and one_launch(same)
    beside = lbib.Sim.from_scene(scenes.channel_sphere(), stream=b.cuda_stream)
    assert not one_launch(g) and not one_launch(same)
    assert one_launch(beside)  # 20 blocks
    beside.close()
    assert one_launch(g)
    g.close()
    same.close()


@pytest.mark.parametrize("box,prec,one", [((48, 40, 40), "f16s", False), ((48, 48, 48), "f16s", True),
                                          ((41, 40, 39), "bf16s", True), ((40, 40, 40), "f32", True)])
def test_small_channels_without_objects(one_launch, box, prec, one):
    """Where a launch of many steps starts to be faster (figures at steps_fit)."""
    g = lbib.Sim(*box, body_force=(1e-5, 0, 0), precision=prec, pop_scale_log2=0 if prec == "f32" else 12)
    g.fluid_init()
    assert one_launch(g) == one
    g.close()


def test_simulations_at_once_equal_alone():
    scs = [scenes.channel_sphere(), scenes.Scene("free", 64, 64, 64, body_force=(2e-5, 0.0, 1e-5)),
           scenes.channel_sphere(), scenes.Scene("odd", 41, 30, 37, body_force=(1e-5, 0.0, 2e-5))]
    alone = []
    for sc in scs:
        g = lbib.Sim.from_scene(sc)
        g.step(300)
        alone.append((g.velocity(), g.read_nodes()[0] if sc.objects else np.zeros((1, 3))))
        g.close()
    streams = [torch.cuda.Stream() for _ in scs]
    sims = [lbib.Sim.from_scene(sc, stream=st.cuda_stream) for sc, st in zip(scs, streams)]
    for _ in range(3):
        for g in sims:
            g.step(100)
    for g, sc, (u, x) in zip(sims, scs, alone):
        g.sync()
        assert np.abs(g.velocity() - u).max() <= 1e-5 * np.abs(u).max()
        if sc.objects:
            assert np.abs(g.read_nodes()[0] - x).max() <= 1e-6
    for g in sims:
        g.close()
