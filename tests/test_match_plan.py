"""What a matcher's plan leaves to the simulator's units: played sets of chains
above the matcher's limit of accesses, whose slots the runs' mix has to hold."""
import ctypes

import torch

from paper_1509_02308_gb300 import capi as C
from paper_1509_02308_gb300 import workloads as W
from test_abi import _describe, _plan


def _mixes(length):
    """16 RANDOM caches that overflow on one chain, and an index array each."""
    cands = [W.Geom(32 * 256, 32, 64, 4, W.RANDOM, k) for k in range(16)]
    array = torch.zeros(64, dtype=torch.int32)
    traces = [(None, length, 0, 8 * 5000, 8), (array, 64, 0, 60, 7)]
    rc, h = _plan(cands, traces)
    assert rc == C.OK
    d = _describe(h)
    C.load().pchase_sim_plan_destroy(ctypes.c_void_p(h.value))
    return d


def test_slots_of_a_match_hold_the_chains_it_leaves_to_the_units():
    d = _mixes(40000)  # above kUniformMatchLen: the matcher's units step them
    assert d["live_slots"] != d["slots"]
    assert d["match_slots"] == d["slots"]
    d = _mixes(20000)  # below it: played, as in other runs
    assert d["match_slots"] == d["live_slots"] != d["slots"]
