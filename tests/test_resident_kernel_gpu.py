"""Compression beside a kernel of somebody else's that stays on an SM for most of a
second: the launch of several levels (csrc/k_split.cu) takes what SMs there are
and does not wait for that one.  Streams equal the oracle's and are there while
the other kernel still runs.
"""
import pytest

import synth
from test_parity_gpu import pc  # noqa: F401  (a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# one launch of a few levels and of eight, two launches
@pytest.mark.parametrize("n,eb,r", [(40_003, 1e-4, 500), (1_100_003, 1e-4, 2048), (2_300_017, 8e-6, 4096)])
def test_an_sm_that_is_taken(pc, oracle_mod, n, eb, r):  # noqa: F811
    pos = synth.cosmology(n, seed=n % 31)
    ref, _ = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r, want_perm=False)
    dpos = torch.from_numpy(pos).cuda()
    c = pc.Compressor(n, pc.PC_F32, r)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    c.compress(dpos, pc.PC_EB_REL, eb, stream=mine)
    c.ws.fill_(0xA5)
    c.out.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(1_500_000_000)  # cycles: 0.7 to 1 s on one SM
        done = torch.cuda.Event()
        done.record()
    sizes = [c.compress(dpos, pc.PC_EB_REL, eb, stream=mine) for _ in range(4)]
    assert not done.query()
    torch.cuda.synchronize()
    assert set(sizes) == {len(ref)}
    assert c.out[:len(ref)].cpu().numpy().tobytes() == ref
