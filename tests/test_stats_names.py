"""The names under which native.lw_get_stats reports the kernel's timers, against
the counters that include/lw.h describes (CPU, a fake library)."""
from paper_1709_06816_gb300 import native


class _Fake:
    def __init__(self, counters):
        self.counters = counters

    def lw_get_stats(self, ctx, array, count):
        for q in range(count):
            array[q] = self.counters.get(q, 0)
        return 0


def _stats(monkeypatch, counters):
    monkeypatch.setattr(native, "load", lambda *a: _Fake(counters))
    return native.lw_get_stats(0)


def test_every_timer_has_the_name_of_what_it_times(monkeypatch):
    # counter -> (table, name): lw_get_stats in include/lw.h
    phases = {8: "barrier", 9: "merges", 10: "to_new_cells", 11: "gather_wait", 13: "apply"}
    parts = {16: "lists", 17: "selection", 18: "member_cells", 19: "merges", 20: "new_cells", 21: "records",
             22: "caches", 23: "rescans", 25: "refill_scans"}
    counters = {q: 3 * (q + 1) * 10**6 for q in list(phases) + list(parts)}
    counters[3] = 3  # CTAs
    st = _stats(monkeypatch, counters)
    assert st["phase_ms"] == {name: q + 1 for q, name in phases.items()}
    assert st["subphase_ms"] == {name: q + 1 for q, name in parts.items()}


def test_no_timers_without_the_option(monkeypatch):
    st = _stats(monkeypatch, {0: 7, 3: 2, 14: 5})
    assert st["rounds"] == 7 and st["rescans"] == 5
    assert "phase_ms" not in st and "subphase_ms" not in st
