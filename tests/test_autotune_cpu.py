"""Autotuner host logic: batch signatures, candidate choice and the JSON cache
(with a stand-in timer; no GPU)."""
import json

from paper_1705_08266_gb300 import autotune as A


def _descs():
    return [(512, 700, 4, "cdf97", "float32", 0), (65, 4096, 1, "legall53", "int32", 1),
            (3000, 2000, 6, "cdf97", "float32", 0)]


def test_signature_order_independent_and_class_based():
    d = _descs()
    assert A.signature(d) == A.signature(list(reversed(d)))
    # same power-of-two classes -> same signature
    d2 = [(600, 900, 4, "cdf97", "float32", 0)] + d[1:]
    assert A.signature(d2) == A.signature(d)
    # another class, level count, direction or type -> another signature
    for change in [(1100, 700, 4, "cdf97", "float32", 0), (512, 700, 5, "cdf97", "float32", 0),
                   (512, 700, 4, "cdf97", "float32", 1), (512, 700, 4, "cdf97", "float16", 0)]:
        assert A.signature([change] + d[1:]) != A.signature(d)


def test_pick_fastest_and_cache(tmp_path):
    path = str(tmp_path / "tune.json")
    calls = []

    def measure(t):
        calls.append(t)
        if t["fuse_first"] == 1 and t["min_segment"] == 8:
            return None  # candidate not applicable
        return 1.0 + abs(t["warps_per_sm"] - 32) / 10 + (0.5 if t["fuse_first"] == 1 else 0)

    best = A.pick("sig", measure, cache_path=path)
    assert best["warps_per_sm"] == 32 and best["fuse_first"] == 2
    assert len(calls) == len(A.CANDIDATES)
    data = json.load(open(path))
    assert data["nonsep_reduced:sig"]["tuning"] == best
    # second call: from the cache, nothing measured
    calls.clear()
    assert A.pick("sig", measure, cache_path=path) == best
    assert calls == []
    # another scheme is another entry
    A.pick("sig", measure, cache_path=path, scheme="separable")
    assert len(calls) == len(A.CANDIDATES)


def test_corrupt_cache_is_ignored(tmp_path):
    path = tmp_path / "tune.json"
    path.write_text("{not json")
    best = A.pick("s", lambda t: float(t["warps_per_sm"]), cache_path=str(path))
    assert best["warps_per_sm"] == 12
    assert "nonsep_reduced:s" in json.loads(path.read_text())


def test_context_separates_cache_entries(tmp_path):
    """A tuning measured on another device or library build is not reused."""
    path = str(tmp_path / "tune.json")
    calls = []

    def measure(t):
        calls.append(t)
        return float(t["warps_per_sm"])

    A.pick("sig", measure, cache_path=path, context="GPU-A/152sm/lib1")
    n = len(calls)
    A.pick("sig", measure, cache_path=path, context="GPU-A/152sm/lib1")
    assert len(calls) == n  # cached
    A.pick("sig", measure, cache_path=path, context="GPU-B/132sm/lib1")
    assert len(calls) == 2 * n  # measured again
    assert len(json.load(open(path))) == 2


def test_tune_times_the_library_default_first(monkeypatch):
    """Unless told otherwise, tune() offers no tuning at all beside the fixed
    settings; candidates a caller names are taken as they are."""
    from types import SimpleNamespace

    import torch

    from paper_1705_08266_gb300 import dwt2d as D

    seen = {}

    def pick(sig, measure, candidates, cache_path, scheme, context):
        seen["candidates"] = candidates
        return dict(candidates[0])

    monkeypatch.setattr(A, "pick", pick)
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda dev: SimpleNamespace(name="stand-in", multi_processor_count=1))
    jobs = [(torch.zeros(8, 8), torch.zeros(8, 8), 1, "cdf97", 0)]
    best = A.tune(jobs, stream=object())
    assert set(best) == set(A.KNOBS) and not any(best.values())
    D.Tuning(**best)  # every knob of it is one of the library's
    assert seen["candidates"][1:] == A.CANDIDATES
    A.tune(jobs, stream=object(), candidates=A.CANDIDATES[:2])
    assert seen["candidates"] == A.CANDIDATES[:2]
