"""The reduction's rounds where a taken box is shared by the blocks of a cluster:
leaves of fewer groups of four particles than there are blocks, leaves that
start and end inside a group, more taken boxes in a round than clusters, boxes
of many particles met by one, and more boxes met than a list holds.  Streams and
permutations equal the oracle's byte for byte.
"""
import numpy as np
import pytest

import synth
from test_reduce_gpu import check, pc  # noqa: F401  (pc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [3, 5, 13, 17, 31, 63, 129])
@pytest.mark.parametrize("gen,eb,dt", [("uniform", 1e-3, np.float32), ("cosmology", 3e-3, np.float32),
                                       ("uniform", 1e-7, np.float64)])
def test_small_leaves(pc, oracle_mod, gen, eb, dt, r):
    check(pc, oracle_mod, synth.by_name(gen, 3001, seed=r, dtype=dt), pc.PC_EB_REL, eb, r)


@pytest.mark.parametrize("gen,n,eb,r", [("uniform", 40_003, 1e-5, 15), ("cosmology", 90_001, 2e-4, 12_000),
                                        ("uniform", 20_001, 0.3, 9)])
def test_many_taken_and_many_met(pc, oracle_mod, gen, n, eb, r):
    check(pc, oracle_mod, synth.by_name(gen, n, seed=3, dtype=np.float32), pc.PC_EB_REL, eb, r)
