"""A stage of a sweep's ring that never lands is reported, wherever it lies.

A sweep looks for a wait that gave up every third stage, so each plane loop has
to look once more after its last stage (a CTA's layer may hold two planes). The
GPU test runs the same wait and checks over rings of 1 to 10 stages, each stage
lost in turn; the other one checks that both sweeps end their loop that way.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2404_04441_gb300", "csrc")


def test_sweeps_look_after_the_last_stage():
    with open(os.path.join(CSRC, "sweep.cuh")) as f:
        src = f.read()
    loops = [m.end() for m in re.finditer(r"\bring_wait\(", src)]
    assert len(loops) == 2  # sweep_cta and sweep_cta_tc
    for at in loops:
        rest = src[at:src.index("\n  return;", at)]
        assert re.search(r"\n  if \(ring_failed\(failed[^)]*\)\) goto wait_failed;", rest)


@pytest.mark.gpu
@pytest.mark.parametrize("limit_ms", [2, 20])
def test_each_lost_stage_is_seen(wave_lib, limit_ms):
    import torch
    assert wave_lib.wave_selftest_wait(limit_ms * 1_000_000) == -5  # WAVE_ETIMEOUT
    # the context stays usable
    s = wave_lib.WaveSolver((8, 8, 8), (10.0,) * 3, 1e-4, torch.full((8, 8, 8), 2000.0).cuda())
    s.step(3)
    s.synchronize()
    s.close()
