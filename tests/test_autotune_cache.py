"""The autotuner's cache holds for the kernels that it was timed with."""
import json

from paper_2509_05216_gb300 import autotune, build


class Ctx:
    def gs_set_option(self, opt, value):
        pass


def test_choices_of_other_kernels_are_searched_again(tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("GS_AUTOTUNE_CACHE", str(path))
    searched = []
    monkeypatch.setattr(autotune, "time_step", lambda step, reps=3: searched.append(1) or float(len(searched)))
    cands = {1: [8, 2]}
    # a file written before the entries named their kernels, and an unrelated key
    path.write_text(json.dumps({"k": {"options": {"1": 2}, "ms": {"1=2": 1.0}}, "other": {"options": {}, "ms": {}}}))
    assert autotune.report("k") is None
    assert autotune.tune([Ctx()], None, "k", candidates=cands, rounds=1) == {1: 8}
    assert len(searched) == 2 and autotune.report("k") == {"1=8": 1.0, "1=2": 2.0}
    assert autotune.tune([Ctx()], None, "k", candidates=cands, rounds=1) == {1: 8} and len(searched) == 2
    # other kernel sources
    monkeypatch.setattr(build, "digest", lambda: "other sources")
    assert autotune.report("k") is None
    autotune.tune([Ctx()], None, "k", candidates=cands, rounds=1)
    assert len(searched) == 4
    assert set(json.loads(path.read_text())) == {"k", "other"}


def test_digest_follows_the_sources(tmp_path, monkeypatch):
    src = tmp_path / "a.cu"
    monkeypatch.setattr(build, "_deps", lambda: [str(src)])
    seen = set()
    for text in ("one", "two", "one"):
        src.write_text(text)
        build.digest.cache_clear()
        seen.add(build.digest())
    build.digest.cache_clear()
    assert len(seen) == 2
