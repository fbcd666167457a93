"""The launch knobs mean what they say: a default knob reports what runs, and every
value that is set is the block size of the kernel (as the profiler sees it)."""
import json

import pytest
import torch

from paper_1312_3426_gb300 import lbib
from workloads import mesh, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_3426_gb300 import build
    build.build()
    lbib.load()


@pytest.fixture
def launched(tmp_path):
    from torch.profiler import ProfilerActivity, profile

    def kernels(work):
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            work()
            torch.cuda.synchronize()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        with open(tmp_path / "trace.json") as f:
            events = [e for e in json.load(f)["traceEvents"] if e.get("cat") == "kernel"]
        return {name: e["args"]["block"][0] for name in ("k_nodes", "k_membrane", "k_batch_nodes", "k_batch_membrane")
                for e in events if f"{name}<" in e["name"]}

    kernels(lambda: torch.zeros(1, device="cuda"))  # the first trace of a process may be empty
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        torch.zeros(64, device="cuda").add_(1)
        torch.cuda.synchronize()
    if not p.events():
        pytest.skip("no kernel tracing on this machine")
    return kernels


def test_every_value_of_a_knob_is_what_runs(launched):
    n, t = mesh.biconcave(3)
    g = lbib.Sim(64, 48, 48, body_force=(1e-5, 0, 0))
    g.template_create(n, t, (8.0,) * 3, **scenes.PAPER_MODULI)
    for k in range(2):
        g.object_add(0, (16.0 + 30 * k, 24.0, 24.0))
    g.fluid_init()
    single = lambda: (g.step(1), g.step(1))  # noqa: E731
    batch = lambda: lbib.lbib_batch_step([g.h], 2)  # noqa: E731
    get = lambda key: lbib.lbib_get_tuning(g.h, key)  # noqa: E731
    node, threads = lbib.LBIB_TUNE_NODE_THREADS, lbib.LBIB_TUNE_MEMBRANE_THREADS
    single()  # the membrane forces of the first positions are a launch of their own

    assert get(node) == 64 and get(threads) == 0
    by_rule = launched(single)
    assert by_rule["k_nodes"] == 2 * 64 and by_rule["k_membrane"] >= 512  # two objects: the step waits for them
    for value in (32, 64, 128, 256):
        lbib.lbib_set_tuning(g.h, node, value)
        assert get(node) == value
        assert launched(single)["k_nodes"] == launched(batch)["k_batch_nodes"] == 2 * value
    lbib.lbib_set_tuning(g.h, node, 64)
    for value in (96, 192, 256):
        lbib.lbib_set_tuning(g.h, threads, value)
        assert get(threads) == value
        assert launched(single)["k_membrane"] == launched(batch)["k_batch_membrane"] == value
    lbib.lbib_set_tuning(g.h, threads, 0)
    assert get(threads) == 0 and launched(single) == by_rule
    for bad in (-1, 16, 100, 288):
        with pytest.raises(lbib.LbibError):
            lbib.lbib_set_tuning(g.h, threads, bad)
    g.close()
