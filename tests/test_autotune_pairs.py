"""Host logic of the launch-shape cache with pairs of steps: a hit leaves an object as
the autotuner left the one that was timed, and entries of library versions that knew
no pairs are not taken."""
import json
from types import SimpleNamespace

import pytest

from paper_1806_09403_gb300 import autotune as T
from paper_1806_09403_gb300 import btdf as B


class Fake:
    def __init__(self, pairs):
        self.cfg = SimpleNamespace(nx=1600, ny=800, storage=0, layout=1, delta=3, nf=1)
        self.cases = [SimpleNamespace(nx=64, ny=32)]
        self.storage = 0
        self.marker_count = 126
        self.pairs_win = pairs
        self.tuned_pairs = False
        self.timed = 0
        self.state = ("automatic", None)   # the last calls' variant and pairs

    def autotune(self, steps, flush_l2):
        self.timed += 1
        self.tuned_pairs = self.pairs_win
        self.state = (2, self.pairs_win)
        return 2, {1: 0.030, 2: 0.025}

    def tune(self, variant, grid=0):
        self.state = (variant, False)

    def tune_pairs(self, on=True):
        self.state = (self.state[0], bool(on))


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("tune", [T.tune_lattice, T.tune_batch])
def test_a_hit_restores_the_tuned_state(tmp_path, tune, pairs):
    path = str(tmp_path / "tune.json")
    a, b = Fake(pairs), Fake(pairs)
    first = tune(a, T.TuneCache(path), device="GB300")
    again = tune(b, T.TuneCache(path), device="GB300")
    assert a.timed == 1 and b.timed == 0 and again["cached"]
    assert b.state == a.state == (2, pairs)
    assert first["pairs"] == again["pairs"] == pairs


def test_entries_from_before_pairs_are_timed_again(tmp_path):
    path = tmp_path / "tune.json"
    a = Fake(True)
    key = T.lattice_key(a, "GB300")
    old = key.replace(f"lib={B.btdf_version()}", "lib=1")
    path.write_text(json.dumps({old: {"variant": 3, "ms_per_step": {"3": 0.02}}}))
    T.tune_lattice(a, T.TuneCache(str(path)), device="GB300")
    assert a.timed == 1 and a.state == (2, True)
