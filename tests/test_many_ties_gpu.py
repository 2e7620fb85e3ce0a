"""Inputs of many equal coordinates: the ties on a split plane are more than a list
holds (csrc/k_split.cu counts them by warp), in one node and in several, on one
axis and on all, in position order and mixed, with the quota's end in the first
warp, the last one and between, over one launch of levels and two.  Streams and
permutations equal the oracle's byte for byte.  And equal coordinates cost a
compression little beside different ones.
"""
import time

import numpy as np
import pytest

import synth
from test_parity_gpu import pc, run_gpu  # noqa: F401  (pc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _points(kind, n, seed):
    rng = np.random.default_rng(seed)
    p = rng.random((n, 3)) * 256.0
    if kind == "half at the start":
        p[: n // 2] = p[0]
    elif kind == "half at the end":
        p[n // 2:] = p[0]
    elif kind == "half, mixed":
        p[rng.random(n) < 0.5] = p[0]
    elif kind == "a tenth":
        p[n // 3: n // 3 + n // 10] = p[0]
    elif kind == "two points":
        p[:] = np.where(rng.random((n, 1)) < 0.3, p[0], p[1])
    elif kind == "one point but one":
        p[1:] = p[0]
    elif kind == "a plane":
        p[:, 2] = 7.0
    elif kind == "a line":
        p[:, 1:] = 7.0
    elif kind == "four values":
        p = np.floor(p / 64.0)
    elif kind == "eight values, sorted":
        p = np.floor(p / 32.0)
        p = p[np.lexsort(p.T)]
    return p.astype(np.float32)


KINDS = ["half at the start", "half at the end", "half, mixed", "a tenth", "two points", "one point but one", "a plane",
         "a line", "four values", "eight values, sorted"]


@pytest.mark.parametrize("kind", KINDS, ids=lambda k: k.replace(" ", "-"))
@pytest.mark.parametrize("n,eb,r", [(40_007, 1e-3, 600), (300_011, 1e-4, 1000), (2_500_003, 1e-3, 2048),
                                    (4_300_007, 8e-6, 200)])
def test_many_ties(pc, oracle_mod, kind, n, eb, r):  # noqa: F811
    pos = _points(kind, n, seed=n % 19)
    ref, ref_perm = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r)
    got, perm, _ = run_gpu(pc, pos, pc.PC_EB_REL, eb, r, with_perm=True)
    assert got == ref and np.array_equal(perm, ref_perm)
    plain, _, dec = run_gpu(pc, pos, pc.PC_EB_REL, eb, r, with_perm=False)
    assert plain == ref
    assert dec.tobytes() == oracle_mod.decompress(ref).tobytes()


@pytest.mark.parametrize("chunk", [8_193, 16_384, 24_577])
def test_a_list_or_none(pc, oracle_mod, chunk):  # noqa: F811
    """One CTA's positions around the size of the list, all of them ties at once."""
    n = 2 * chunk
    pos = synth.uniform(n, seed=2)
    pos[:, 0] = 1.0
    ref, ref_perm = oracle_mod.compress(pos, oracle_mod.REL, 1e-3, leaf_size=300)
    cfg = pc.config(300, warp_node_max=256)
    got, perm, _ = run_gpu(pc, pos, pc.PC_EB_REL, 1e-3, cfg, with_perm=True)
    assert got == ref and np.array_equal(perm, ref_perm)


def test_ties_cost_little(pc):  # noqa: F811
    """2^26 particles, half of them one point, against 2^26 different ones: 1.5 times the time
    when the ties are counted by warp, 3.5 times when one CTA lists them."""
    n = 1 << 26
    pos = torch.rand((n, 3), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    c = pc.Compressor(n, pc.PC_F32)

    def best():
        times = []
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            c.compress(pos, pc.PC_EB_REL, 1e-4)
            times.append(time.perf_counter() - t0)
        return min(times[1:])

    plain = best()
    pos[: n // 2] = pos[0].clone()
    ties = best()
    print(f"different {plain * 1e3:.2f} ms, half equal {ties * 1e3:.2f} ms")
    assert ties < 2.0 * plain
