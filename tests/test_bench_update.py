"""The benchmark names the update that a sweep takes, not the parameter's value (CPU)."""
import dataclasses
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_2504_10118_gb300 import synth  # noqa: E402


# (m, levels, minibatch): the update of deterministic = 0, as include/magpie.h states it
@pytest.mark.parametrize("m,levels,minibatch,update", [
    (8, 2, 1024, "ordered"), (8, 2, 1025, "atomic"), (32, 2, 64, "ordered"), (32, 2, 65, "atomic"),
    (64, 4, 63, "ordered"), (64, 4, 64, "atomic"), (64, 4, 65, "atomic"), (64, 4, 200, "atomic"), (64, 5, 8, "atomic"),
    (128, 3, 64, "ordered"), (128, 5, 400, "ordered"), (128, 6, 8, "atomic"), (256, 5, 64, "ordered"),
    (256, 6, 64, "atomic")])
def test_update_of_a_sweep(m, levels, minibatch, update):
    w = dataclasses.replace(synth.WORKLOADS["mid"], m=m, levels=levels, minibatch=minibatch)
    assert bench.update_of(w, 0) == update
    assert bench.update_of(w, 1) == "ordered"


def test_default_workload_takes_one_update():
    assert bench.update_of(synth.WORKLOADS["mid"], 0) == bench.update_of(synth.WORKLOADS["mid"], 1) == "ordered"
