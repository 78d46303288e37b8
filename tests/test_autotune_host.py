"""Host logic of the autotuner: cache keys and the JSON cache (no GPU needed)."""
import json

import pytest

pytest.importorskip("torch")

from paper_2103_00405_gb300 import autotune as A
from paper_2103_00405_gb300 import workloads as W


@pytest.fixture
def fake_gpu(monkeypatch, tmp_path):
    monkeypatch.setattr(A, "_gpu", lambda: "GB300-test")
    monkeypatch.setenv("RANDTIME_AUTOTUNE_CACHE", str(tmp_path / "cache" / "autotune.json"))
    return tmp_path


def test_batch_key_depends_on_the_size_multiset_not_the_order(fake_gpu):
    specs = [W.random_mass_action(3, m, seed=m) for m in (5, 40, 300)]
    k1 = A.batch_key(specs, 1)
    k2 = A.batch_key(list(reversed(specs)), 1)
    assert k1 == k2
    assert A.batch_key(specs, 2) != k1
    assert A.batch_key(specs[:2], 1) != k1
    assert "GB300-test" in k1


def test_single_key_names_the_shape(fake_gpu):
    spec = W.random_mass_action(7, 90, seed=1)
    assert A.single_key(spec, 64) == "single|GB300-test|M=90|N=7|traj=64"


def test_cache_round_trip_and_cached_choice_is_returned_without_timing(fake_gpu, monkeypatch):
    specs = [W.random_mass_action(3, m, seed=m) for m in (5, 40)]
    key = A.batch_key(specs, 1)
    A._store(key, {"policy": {"thread_max_m": 4, "warp_max_m": 64, "block_threads": 256}})
    A._store("other", {"policy": {}})
    with open(A.cache_path()) as f:
        data = json.load(f)
    assert set(data) == {key, "other"}

    def no_timing(*a, **k):
        raise AssertionError("a cached choice must not be re-timed")

    monkeypatch.setattr(A, "_time", no_timing)
    got = A.tune_batch(specs, None, None, 1)
    assert got == {"thread_max_m": 4, "warp_max_m": 64, "block_threads": 256}


def test_candidates_respect_the_library_limits():
    for c in A.BATCH_CANDIDATES:
        assert 0 <= c["thread_max_m"] <= 8
        assert 0 <= c["warp_max_m"] <= 256
        assert c["block_threads"] in (128, 256, 512)


class _Events:
    def sum(self):
        return self

    def item(self):
        return 1000


def _fake_launches(monkeypatch, times, calls):
    """api.simulate and the timer replaced: a launch takes what `times` says for (mapping, block_threads)."""
    class Net:
        def __init__(self, spec):
            pass

    def simulate(net, x0, t_end, n_traj, seed, max_events, outputs, mapping, block_threads):
        calls.append((mapping, block_threads))
        return dict(n_events=_Events())

    def timed(fn):
        fn()
        return times.get(calls[-1], 10.0)

    monkeypatch.setattr(A.api, "Network", Net)
    monkeypatch.setattr(A.api, "simulate", simulate)
    monkeypatch.setattr(A, "_time", timed)


@pytest.mark.parametrize("m", [3, 12, 100, 700, 9000])
def test_the_librarys_own_choice_is_a_candidate(fake_gpu, monkeypatch, m):
    spec = W.random_mass_action(7, m, seed=1)
    calls = []
    _fake_launches(monkeypatch, {(A.L.RT_MAP_AUTO, 0): 1.0}, calls)
    got = A.tune_single(spec, None, 1.0, 64)
    assert got == dict(mapping=A.L.RT_MAP_AUTO, block_threads=0)
    assert len(calls) == len(set(calls)) > 1  # the named mappings are still timed
    n = len(calls)
    assert A.tune_single(spec, None, 1.0, 64) == got and len(calls) == n  # from the cache


def test_an_entry_tuned_without_the_librarys_choice_is_timed_again(fake_gpu, monkeypatch):
    spec = W.random_mass_action(7, 3, seed=1)
    thread = dict(mapping=A.L.RT_MAP_THREAD, block_threads=128)
    A._store(A.single_key(spec, 64), {"launch": thread, "tried": [[thread, 1.0]]})
    calls = []
    _fake_launches(monkeypatch, {(A.L.RT_MAP_AUTO, 0): 1.0}, calls)
    assert A.tune_single(spec, None, 1.0, 64)["mapping"] == A.L.RT_MAP_AUTO
    other = W.random_mass_action(7, 5, seed=1)
    A._store(A.single_key(other, 64), {"launch": thread})  # an entry that does not say what it tried stands
    n = len(calls)
    assert A.tune_single(other, None, 1.0, 64) == thread and len(calls) == n
