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


# float64 positions and bounds on both sides of the fixed-point quantizer's rule (s >= 2^-35 of
# the power of two above the coordinates), on lattice midpoints, with both signs and zeros
@pytest.mark.parametrize("offset,span", [(0.0, 1.0), (-0.5, 1.0), (1e6, 3.0), (-1e9, 0.25), (-3e4, 7e4), (1e-3, 1e-6)])
@pytest.mark.parametrize("eb", [1e-1, 1e-3, 1e-5, 1e-8])
def test_float64_quantizer(pc, oracle_mod, offset, span, eb):
    rng = np.random.default_rng(17)
    pos = offset + span * rng.random((6_000, 3))
    pos[::7] = offset + span * np.round(rng.random((858, 3)) * 64) / 64
    pos[::50] = np.where(rng.random((120, 3)) < 0.5, 0.0 if offset <= 0.0 <= offset + span else offset, pos[::50])
    s = 2 * eb * span
    pos[::11] = np.minimum(offset + s * (rng.integers(0, int(0.5 / eb) - 1, (546, 3)) + 0.5), offset + span)
    _check(pc, oracle_mod, pos, eb, 512)


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
