"""What the autotuner compares, on times made up for each kernel: the whole
grouping stage of either mode, and the record sort only where records are
sorted."""
import numpy as np
import pytest

from paper_2403_09010_gb300 import autotune, native, xtn

torch = pytest.importorskip("torch")

G, R, P, H = (native.XTN_TUNE_GROUPING, native.XTN_TUNE_SORT_RECORDS, native.XTN_TUNE_SORT_PAIRS,
              native.XTN_TUNE_RECORD_HISTOGRAM)


class Machine:
    """Stands in for the library: knobs, plans, and a profile by their state."""

    def __init__(self, kept_ms):
        self.knobs = {G: 0, R: 22, P: 21, H: 0}
        self.kept_ms = kept_ms
        self.records_tried = []
        self.last = {}

    def plan(self, offsets, d, rep_offsets=None):
        machine = self

        class Plan:
            def run(self, seqs):
                k = machine.knobs
                machine.records_tried.append((k[G], k[R], k[H]))
                ms = {"k_onesweep_pairs": 1.0 + abs(k[P] - 3), "k_verify_candidates": 9.0,
                      "k_expand": 2.0}
                if k[G] == 0:
                    ms.update({"k_bucket_filter": 1.0, "k_group_kept": machine.kept_ms,
                               "k_onesweep_records": 0.01, "k_group_flags": 0.01,
                               "k_emit_pairs": 0.01})
                else:
                    ms.update({"k_onesweep_records": 3.0 + abs(k[R] - 2) + k[H],
                               "k_group_flags": 0.5, "k_emit_pairs": 0.5})
                for name, t in ms.items():
                    n, total, b = machine.last.get(name, (0, 0.0, 0.0))
                    machine.last[name] = (n + 1, total + t, b)

            def stats(self):
                return {"candidates": 1_000_000}

            def free(self):
                pass
        return Plan()

    def report(self):
        out, self.last = self.last, {}
        return out


@pytest.mark.parametrize("kept_ms,mode", [(0.5, 0), (40.0, 1)])
def test_grouping_and_record_sort(monkeypatch, kept_ms, mode):
    m = Machine(kept_ms)
    monkeypatch.setattr(xtn, "Plan", m.plan)
    monkeypatch.setattr(xtn, "tune_set", m.knobs.__setitem__)
    monkeypatch.setattr(xtn, "tune_get", m.knobs.__getitem__)
    monkeypatch.setattr(xtn, "tune_count", lambda knob: 2 if knob == H else 5)
    monkeypatch.setattr(xtn, "profile_enable", lambda on=True: None)
    monkeypatch.setattr(xtn, "profile_report", m.report)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    r = autotune.tune(None, np.zeros(3, np.int64), 2, use_cache=False)
    assert r["grouping"] == mode and r["pairs_cfg"] == 3
    assert r["pair_capacity"] == 1_250_000
    assert m.knobs == {G: 0, R: 22, P: 21, H: 0}
    if mode == 0:  # nothing is sorted: nothing to choose from
        assert (r["records_cfg"], r["record_hist"]) == (22, 0)
        assert "records" not in r["sort_ms"]
        assert all((c, h) == (22, 0) for g, c, h in m.records_tried if g == 0)
    else:
        assert (r["records_cfg"], r["record_hist"]) == (2, 0)
        assert r["sort_ms"]["records"] == 3.0
