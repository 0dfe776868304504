"""The ensemble autotuner without a device: the library's own choices are a candidate
and can be what is left set, also from the cache, and mixes that differ only in
their members' storage are tuned apart."""
import types

import pytest

from paper_1601_03815_gb300 import ensemble


class FakeEnsemble:
    """Steps take the time that `cost(tuning)` names; tuning None: untouched."""

    def __init__(self, clock, cost, storage=0):
        self.clock, self.cost, self.tuning = clock, cost, None
        self.members = [types.SimpleNamespace(N=50, scheme=1, storage=storage)]

    def reset_tuning(self):
        self.tuning = None

    def set_tuning(self, tile_y=0, zchunk=0, lbe_block=0):
        old = self.tuning or (0, 0, 0)
        self.tuning = tuple(n if n > 0 else o for n, o in zip((tile_y, zchunk, lbe_block), old))

    def step(self, n=1):
        self.clock.now += n * self.cost(self.tuning)


@pytest.fixture
def clock(monkeypatch, tmp_path):
    c = types.SimpleNamespace(now=0.0)
    monkeypatch.setattr(ensemble.time, "perf_counter", lambda: c.now)
    monkeypatch.setenv("KIN_TUNE_CACHE", str(tmp_path))
    return c


def test_the_librarys_choice_is_kept_where_it_is_the_fastest(clock):
    cost = lambda t: 1.0 if t is None else 1.3  # noqa: E731
    ens = FakeEnsemble(clock, cost)
    best = ensemble.autotune(ens)
    assert ens.tuning is None
    assert best["ms_per_step"] == pytest.approx(1e3)
    again = FakeEnsemble(clock, cost)
    again.set_tuning(8, 16, 64)
    ensemble.autotune(again)  # from the cache
    assert again.tuning is None


def test_a_faster_candidate_is_set(clock):
    ens = FakeEnsemble(clock, lambda t: 0.7 if t == (0, 32, 64) else 1.0)
    ensemble.autotune(ens)
    assert ens.tuning == (0, 32, 64)


def test_storage_types_are_tuned_apart(clock):
    ensemble.autotune(FakeEnsemble(clock, lambda t: 0.7 if t == (0, 32, 64) else 1.0, storage=0))
    half = FakeEnsemble(clock, lambda t: 0.7 if t == (0, 8, 128) else 1.0, storage=1)
    ensemble.autotune(half)
    assert half.tuning == (0, 8, 128)
