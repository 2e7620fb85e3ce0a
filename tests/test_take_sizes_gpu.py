"""The reduction's rounds on both sides of its rules on sizes: leaves that have a
cluster of blocks per taken box and leaves that have one block, rounds that take
more boxes than there are clusters, and boxes walked by 128 and by 256 threads.
Streams and permutations equal the oracle's byte for byte.  And a round over many
small leaves takes little longer than one over few large ones.
"""
import numpy as np
import pytest

import synth
from test_reduce_gpu import check, pc  # noqa: F401  (pc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# leaves a particle on both sides of 1024 and 2048; 512 to 2048 leaves
@pytest.mark.parametrize("gen,n,eb,r", [("uniform", 1_200_001, 3e-3, 1100), ("cosmology", 1_049_000, 1e-3, 1025),
                                        ("cosmology", 1_049_000, 1e-3, 1024), ("uniform", 1_100_003, 1e-4, 2049),
                                        ("cosmology", 1_048_576, 3e-3, 2048), ("cosmology", 524_800, 1e-6, 1100)])
def test_both_sides_of_the_rules(pc, oracle_mod, gen, n, eb, r):  # noqa: F811
    check(pc, oracle_mod, synth.by_name(gen, n, seed=r, dtype=np.float32), pc.PC_EB_REL, eb, r)


def _take_us(pc, n, r):
    g = torch.Generator(device="cuda").manual_seed(3)
    pos = torch.rand((n, 3), generator=g, device="cuda")
    c = pc.Compressor(n, pc.PC_F32, pc.config(r, reduce=True))
    c.compress(pos, pc.PC_EB_REL, 1e-3)
    pc.pc_trace_reset()
    pc.pc_trace_enable(True)
    c.compress(pos, pc.PC_EB_REL, 1e-3)
    launches, ms = pc.trace_table()["k_rd_take"]
    pc.pc_trace_enable(False)
    pc.pc_trace_reset()
    return 1e3 * ms / launches


def test_rounds_over_small_leaves_are_short(pc):  # noqa: F811
    """2^24 particles in leaves of 256 against 2^21 in leaves of 4096: a launch of k_rd_take
    takes 1.2 times as long with a block per small box, 5 times with a cluster for each."""
    small, large = _take_us(pc, 1 << 24, 256), _take_us(pc, 1 << 21, 4096)
    print(f"k_rd_take: {small:.1f} us over small leaves, {large:.1f} us over large ones")
    assert small < 3.0 * large
