"""The autotuner's own search space: an option that the library accepts and
ignores has one candidate, its default, so that nothing is tuned by noise;
every other option has more, its default among them."""
import os
import re

import pytest

pytest.importorskip("torch")

from paper_2010_14058_gb300 import autotune  # noqa: E402

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "tg.h")


def ignored_options():
    text = open(HEADER).read()
    body = text[text.index("/* Tuning knobs"):text.index("} tg_options;")]
    return {name for name, note in re.findall(r"int32_t (\w+);\s*/\*(.*?)\*/", body, flags=re.S)
            if "accepted and ignored" in note}


def test_ignored_options_have_one_candidate():
    ignored = ignored_options()
    assert {"light_edge_max_degree", "isect_modes"} <= ignored
    for knob, values in autotune.SPACE.items():
        option = "isect_modes" if knob.startswith("isect_bucket_") else knob
        assert autotune.DEFAULTS[knob] in values
        assert (len(values) == 1) == (option in ignored), knob
