"""The batch-plan tuner keeps a table only where it beats the library's own chunk
lengths, and times the launch modes that differ (no GPU)."""
import os

from paper_2104_03186_gb300 import tune


def test_table_kept_only_where_it_wins():
    assert tune.keep_table(19.80, 19.60)
    assert not tune.keep_table(19.63, 19.80)  # slower
    assert not tune.keep_table(19.80, 19.75)  # within what runs differ by


def test_timed_modes_differ():
    # "auto" runs the per-level launches: timing it ranks noise
    assert set(tune.TIMED_MODES) == set(tune.MODES) - {"auto"}


def test_committed_plan_was_timed_with_the_modes_that_differ():
    if os.path.exists(tune.DEFAULT_OUT):
        plan = tune.load(tune.DEFAULT_OUT)
        assert set(plan["mix_ms"]) == set(tune.TIMED_MODES)
        if plan["entries"]:
            assert tune.keep_table(plan["untuned_ms"], plan["tuned_ms"])
