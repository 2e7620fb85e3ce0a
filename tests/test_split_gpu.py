"""Several k-d levels per launch (csrc/k_split.cu) where it can go wrong: inputs a
particle past a CTA's positions or a tile of the move, one to eight levels in a
launch, 15 and 16-bit codes (seven and six levels, median bins of several codes), two launches
with subroots cut by the CTAs' positions, and ties - few, thousands and more
than the shared-memory list holds - on the split planes.  Streams and
permutations equal the oracle's byte for byte.
"""
import numpy as np
import pytest

import synth
from test_parity_gpu import pc, run_gpu  # noqa: F401  (pc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lattice(n, sides, seed):
    """Points on a lattice of `sides` places per axis (1: a constant coordinate, 0: uniform)."""
    rng = np.random.default_rng(seed)
    cols = [rng.integers(0, s, n).astype(np.float64) if s else rng.uniform(0, 8, n) for s in sides]
    return np.stack(cols, axis=1).astype(np.float32)


# name, positions, bound (value-range-relative), leaf size
CASES = [
    ("one level", lambda: synth.uniform(16_385, seed=1), 1e-3, 8192),
    ("two levels", lambda: synth.uniform(24_577, seed=2), 1e-4, 4096),
    ("five levels", lambda: synth.cosmology(152 * 4096 + 1, seed=3), 1e-4, 4096),
    ("seven levels", lambda: synth.cosmology(524_289, seed=4), 1e-3, 700),
    ("seven levels, a chunk of 16", lambda: synth.uniform(1_048_559, seed=5), 1e-2, 4096),
    ("eight levels", lambda: synth.cosmology(1_100_003, seed=14), 1e-4, 2048),
    ("eight levels, one child each tile", lambda: synth.fluid(1_300_000, seed=15, dtype=np.float32), 1e-4, 4096),
    ("fifteen bits", lambda: synth.uniform(300_007, seed=6), 2e-5, 512),
    ("sixteen bits", lambda: synth.cosmology(400_001, seed=7), 8e-6, 512),
    ("two launches", lambda: synth.cosmology(2_200_003, seed=8), 1e-4, 4096),
    ("two launches, sixteen bits", lambda: synth.uniform(2_300_017, seed=9), 8e-6, 4096),
    ("ties on every plane", lambda: _lattice(200_003, (4, 3, 2), 10), 1e-3, 600),
    ("a constant axis", lambda: _lattice(150_001, (1, 2, 0), 11), 1e-3, 900),
    ("more ties than the list", lambda: _lattice(2_600_001, (1, 2, 50), 12), 1e-3, 4096),
    ("lattice order", lambda: synth.fluid(700_001, seed=13, dtype=np.float32), 1e-3, 4096),
]


@pytest.mark.parametrize("name,points,eb,r", CASES, ids=lambda v: v.replace(" ", "-") if isinstance(v, str) else "")
def test_levels_per_launch_match_the_oracle(pc, oracle_mod, name, points, eb, r):
    pos = points()
    ref, ref_perm = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r)
    got, perm, dec = run_gpu(pc, pos, pc.PC_EB_REL, eb, r, with_perm=True)
    assert got == ref and np.array_equal(perm, ref_perm)
    plain, _, _ = run_gpu(pc, pos, pc.PC_EB_REL, eb, r, with_perm=False)
    assert plain == ref
    assert dec.tobytes() == oracle_mod.decompress(ref).tobytes()
