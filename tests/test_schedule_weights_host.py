"""The shipped scheduler weights by their own record: on held-out batches their picks take no longer than the
default schedule (2 % for ties)."""
import json

from paper_2511_01235_gb300 import scheduler as SCH


def test_the_shipped_weights_lose_nothing_to_the_default_on_heldout_batches():
    with open(SCH.DEFAULT_WEIGHTS) as f:
        ev = json.load(f)["meta"]["heldout_eval"]
    assert ev["learned_ms"] <= 1.02 * ev["default_ms"], ev
