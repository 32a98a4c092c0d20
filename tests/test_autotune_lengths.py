"""Cached schedules belong to a transform length (no GPU)."""

import json

from paper_1602_04691_gb300 import autotune as AT


class FakePlan:
    def __init__(self, n, transform_length):
        self.n, self.transform_length = n, transform_length
        self.applied = []

    def set_schedule(self, s):
        self.applied.append(dict(s))

    def autotune_now(self, nrhs, reps):
        s = {f: 0 for f in AT._FIELDS}
        return dict(s, zconv_variant=self.transform_length % 3), 1.0


def test_plans_of_one_n_and_several_lengths_do_not_share_an_entry(tmp_path):
    path = str(tmp_path / "c.json")
    runs = [AT.tune(FakePlan(200, M), 1, "G", path=path) for M in (400, 512, 1024)]
    assert len({r["key"] for r in runs}) == 3 and not any(r["cached"] for r in runs)
    for M, r in zip((400, 512, 1024), runs):
        p = FakePlan(200, M)
        again = AT.tune(p, 1, "G", path=path)
        assert again["cached"] and p.applied == [r["schedule"]]


def test_entries_without_a_length_are_not_applied(tmp_path):
    """Written when the kernels behind the fields were others."""
    path = tmp_path / "old.json"
    old = dict({f: 0 for f in AT._FIELDS}, ctas_per_sm=1)
    path.write_text(json.dumps({AT.cache_key("G", 300, 1): {"schedule": old, "ms": 1.0}}))
    p = FakePlan(300, 800)
    assert not AT.tune(p, 1, "G", path=str(path))["cached"] and p.applied == []
