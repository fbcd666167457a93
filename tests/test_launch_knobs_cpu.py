"""The autotuner keeps the library's own rule for the membrane threads where no
fixed number of threads was faster."""
import pytest

from paper_1312_3426_gb300 import lbib, tune


class FakeSim:
    def __init__(self):
        self.h, self.knobs = self, {}

    def info(self):
        return [1, 3, 3 * 642, 64 * 46 * 48, 0, 0, lbib.LBIB_POP_F32, 1]


@pytest.mark.parametrize("fixed,threads", [(2.0, 0), (0.5, 128)])
def test_the_rule_stays_unless_a_fixed_number_is_faster(monkeypatch, fixed, threads):
    key_of = {key: name for name, key in tune.KNOBS}
    monkeypatch.setattr(lbib, "lbib_set_tuning", lambda h, key, value: h.knobs.update({key_of[key]: value}))

    def cost(sims, steps, batched):
        k = sims[0].knobs
        return (1.0 if k["membrane_threads"] == 0 else fixed + abs(k["membrane_threads"] - 128)) + \
            abs(k["node_threads"] - 32) + k["cluster"] + k["membrane_group"] + k["early_launch"] + 1 - k["overlap"]

    monkeypatch.setattr(tune, "_time", cost)
    monkeypatch.setattr(tune, "_CACHE", {})
    sim = FakeSim()
    choice, _ = tune.autotune([sim], steps=8, batched=False)
    want = dict(tune.DEFAULT, membrane_threads=threads)
    assert choice == want and sim.knobs == want
