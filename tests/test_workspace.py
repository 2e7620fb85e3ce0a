"""The compressor's scratch.  Its size is bounded by what pc_compress_noalloc's
fixed array holds, so the largest inputs that array takes are pinned here (CPU).
On the GPU the streams and permutations equal the oracle's from a workspace full
of stale bytes, at the sizes where the counters of several levels per launch
(csrc/k_split.cu) lie in different places and have different numbers of bins:
inputs with and without spare room for them, with per-level histograms as large
and smaller, 13 and 16-bit codes, and codes that leave no room for them at all.
"""
import numpy as np
import pytest

import synth

# leaf size: the most particles (rounded down) whose scratch is within 48 MiB
NOALLOC = {0: 1_272_000, 64: 473_700, 256: 759_700, 1000: 974_300, 12_000: 1_479_000}


@pytest.fixture(scope="module")
def pc():
    import paper_2404_02826_gb300 as pc
    from paper_2404_02826_gb300 import build as b

    b.build()
    pc.load()
    return pc


@pytest.mark.parametrize("leaf", sorted(NOALLOC))
def test_fixed_scratch_holds_the_same_inputs(pc, leaf):
    for dtype in (pc.PC_F32, pc.PC_F64):
        assert pc.pc_compress_workspace_size(NOALLOC[leaf], dtype, leaf) <= pc.PC_NOALLOC_SCRATCH_BYTES


@pytest.mark.gpu
def test_noalloc_takes_the_largest_input_of_its_array(pc):
    torch = pytest.importorskip("torch")
    n = NOALLOC[0]
    pos = torch.from_numpy(synth.cosmology(n, seed=3)).cuda()
    c = pc.Compressor(n, pc.PC_F32)
    size = c.compress(pos, pc.PC_EB_REL, 1e-4)
    out = torch.empty_like(c.out)
    assert pc.pc_compress_noalloc(pos, pc.PC_EB_REL, 1e-4, out) == size
    assert torch.equal(out[:size], c.out[:size])


# particles, bound, leaf size, nodes split by a warp up to (0: the default), reordered
STALE = [
    (3_019, 1e-4, 1000, 1, True), (3_019, 8e-6, 1000, 1, True),             # 1024 bins
    (9_371, 1e-4, 4096, 0, True), (9_371, 8e-6, 4096, 0, True),             # 4096 bins
    (12_344, 1e-4, 4096, 1, True),
    (5_000, 1e-4, 16, 0, False), (5_000, 8e-6, 16, 512, False),             # in the per-level histograms
    (9_000, 8e-6, 60, 1, True),
    (16_385, 8e-6, 300, 512, False), (18_711, 1e-4, 4096, 0, False),        # in the spare room, ties in shared memory
    (65_536, 1e-4, 500, 0, False), (65_537, 1e-4, 500, 0, False),           # its last size, and the first with a list
    (600_011, 1e-4, 30, 1, False), (600_011, 8e-6, 30, 1, False),           # two launches' worth of levels, one fits
    (2_200_003, 1e-4, 100, 0, False),                                       # two launches
    (40_003, 1e-6, 500, 0, False),                                          # 32-bit codes
]


@pytest.mark.gpu
@pytest.mark.parametrize("perm", [False, True])
@pytest.mark.parametrize("n,eb,r,node_max,reorder", STALE)
def test_stale_workspaces(pc, oracle_mod, n, eb, r, node_max, reorder, perm):
    torch = pytest.importorskip("torch")
    pos = synth.cosmology(n, seed=n % 71)
    ref, ref_perm = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r)
    if reorder:
        ref, ref_perm, _ = oracle_mod.reorder(ref, ref_perm)
    c = pc.Compressor(n, pc.PC_F32, pc.config(r, reorder=reorder, warp_node_max=node_max), perm)
    dpos = torch.from_numpy(pos).cuda()
    other = torch.from_numpy(synth.uniform(n, seed=1)).cuda()
    for first in (None, other):  # full of a pattern, then as a call on other data left it
        if first is None:
            c.ws.fill_(0xA5)
        else:
            c.compress(first, pc.PC_EB_REL, 8e-6)
        size = c.compress(dpos, pc.PC_EB_REL, eb)
        assert c.out[:size].cpu().numpy().tobytes() == ref
        if perm:
            assert np.array_equal(c.perm[:n].cpu().numpy().astype(np.int64), ref_perm)
