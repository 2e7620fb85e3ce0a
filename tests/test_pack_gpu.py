"""The packing and the on-chip subtrees at their edges: leaves a particle around
the 128 that a warp packs at once, code widths from a few bits to more than a
word (four particles a lane between 8 and 32 bits, other layouts outside), 16
and 32-bit codes, subnodes whose median bins have to be narrowed (codes spread
unevenly over the full range) and subnodes full of ties.  Streams and
permutations equal the oracle's byte for byte.
"""
import numpy as np
import pytest

import synth
from test_parity_gpu import pc, run_gpu  # noqa: F401  (pc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(pc, oracle_mod, pos, eb, r):
    ref, ref_perm = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r)
    got, perm, dec = run_gpu(pc, pos, pc.PC_EB_REL, eb, r, with_perm=True)
    assert got == ref and np.array_equal(perm, ref_perm)
    plain, _, _ = run_gpu(pc, pos, pc.PC_EB_REL, eb, r, with_perm=False)
    assert plain == ref
    assert dec.tobytes() == oracle_mod.decompress(ref).tobytes()


# leaves of n particles (one leaf: r = n), and of about r
@pytest.mark.parametrize("n,r", [(2, 8), (128, 128), (129, 129), (130, 130), (257, 257), (4097, 130), (5000, 1250),
                                 (11_999, 12_000), (16_384, 4096), (24_576, 384), (32_768, 600)])
@pytest.mark.parametrize("eb", [0.2, 2e-2, 3e-3, 2e-4, 1e-5, 1e-6])
def test_widths_and_leaf_sizes(pc, oracle_mod, n, r, eb):
    _check(pc, oracle_mod, synth.uniform(n, seed=n + r, dtype=np.float64), eb, r)


def _uneven(n, seed):
    """Half the particles in a corner of a thousandth of the box, half spread over it."""
    rng = np.random.default_rng(seed)
    scale = np.where(rng.random(n) < 0.5, 0.25, 256.0)
    return (rng.random((n, 3)) * scale[:, None]).astype(np.float32)


def _few_codes(n, seed):
    rng = np.random.default_rng(seed)
    return rng.integers(0, 5, (n, 3)).astype(np.float32)


@pytest.mark.parametrize("make", [_uneven, _few_codes], ids=["uneven", "few-codes"])
@pytest.mark.parametrize("n,r,eb", [(16_001, 300, 8e-6), (32_700, 4096, 8e-6), (30_011, 520, 1e-3), (1024, 17, 1e-4),
                                    (90_001, 2000, 8e-6)])
def test_narrowed_medians_and_ties(pc, oracle_mod, make, n, r, eb):
    _check(pc, oracle_mod, make(n, n), eb, r)
