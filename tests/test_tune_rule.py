"""Host logic of sweep_threads="auto", with the library calls replaced by fakes (no GPU): the
library's own rule is a candidate, and choices timed on another source of the library are not
used."""
import pytest

from paper_2401_07965_gb300 import tune
from tests.test_tune_host import SPEC2, SPEC3, _Fake, cache  # noqa: F401


@pytest.mark.parametrize("rule,expected", [(9.0, 0), (3.0, 0), (2.98, 0), (2.9, 128)])
def test_the_rule_stands_unless_beaten(cache, monkeypatch, rule, expected):  # noqa: F811
    f = _Fake({None: rule, 64: 1.0, 128: 3.0, 256: 2.0, 384: 0.5, 512: 1.5})
    f.install(monkeypatch)
    assert tune.choose_sweep_threads_batch(SPEC2) == expected
    assert f.batches == 1
    assert tune.choose_sweep_threads_batch(SPEC2) == expected  # cached
    monkeypatch.setattr(tune, "_CACHE", {})
    assert tune.choose_sweep_threads_batch(SPEC2) == expected
    assert f.batches == 1
    # the best of the named variants has its own entry
    assert tune.best_sweep_threads_batch(SPEC2) == 128


def test_choices_of_another_source_are_not_used(cache, monkeypatch):  # noqa: F811
    f = _Fake({None: 1.0, 256: 3.0})
    f.install(monkeypatch)
    assert tune.choose_sweep_threads_batch(SPEC3) == 256
    assert tune.best_sweep_groups_batch(SPEC3) in (1, 2)
    n = f.batches
    monkeypatch.setattr(tune, "_source", lambda: "another")
    f.setting = None
    f.rates = {None: 5.0}
    assert tune.choose_sweep_threads_batch(SPEC3) == 0
    assert f.batches == n + 1
