"""The batch autotuner's candidates include the lengths a batch takes by itself, so that
tuning never ends on a slower one (CPU; no GPU needed)."""
import inspect
import os
import re

from paper_0712_0813_gb300 import autotune

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_candidates_include_the_automatic_lengths():
    with open(os.path.join(ROOT, "paper_0712_0813_gb300", "csrc", "ce_batch.cu")) as fh:
        automatic = [int(x) for x in re.findall(r"kItemLen(?:32|64) = (\d+)", fh.read())]
    assert len(automatic) == 2
    candidates = inspect.signature(autotune.autotune_batch).parameters["candidates"].default
    assert set(automatic) <= set(candidates)
