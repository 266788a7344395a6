"""Entries of a tuning cache that name no kernel generation, or an older one, were measured on other
kernels: they are not read back (a choice they hold may select another kernel now), and stay in the
file beside the new entry."""
from __future__ import annotations

import json

import pytest

from _fixtures import make_context, make_problem

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("old", ["", "|kernels=1"])
def test_older_entries_are_measured_again(tmp_path, old):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2003_07358_gb300.fhs import fhs_set_autotune
    path = str(tmp_path / "tune.json")
    _, _, prob = make_problem("tiny")
    try:
        fhs_set_autotune(1, path)
        make_context(prob, torch).close()
        with open(path) as f:
            data = json.load(f)
        (key,) = data
        entry = dict(data[key], gram_tc=0, sara_fast=0)
        older = key.split("|kernels=")[0] + old
        with open(path, "w") as f:
            json.dump({older: entry}, f)
        ctx = make_context(prob, torch)
        assert ctx.fhs_get_tuning(0)["source"] == "measured"
        ctx.close()
        with open(path) as f:
            data = json.load(f)
        assert data[older]["gram_tc"] == 0 and set(data) == {older, key}
    finally:
        fhs_set_autotune(0)
