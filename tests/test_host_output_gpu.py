"""Decompression into memory that the host reads: pc_decompress returns when the
decoder's last block has left its error word in host memory, so every position has
to be visible to the host by then.  The output lies in page-locked host memory,
is filled with another pattern before each call and compared on the host straight
after the return, with nothing synchronised in between.
"""
import numpy as np
import pytest

import synth
from test_parity_gpu import pc  # noqa: F401  (a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dtype", [(1_000, np.float32), (100_003, np.float32), (1 << 20, np.float32),
                                     (1 << 20, np.float64)])
def test_positions_are_visible_to_the_host_on_return(pc, oracle_mod, n, dtype):  # noqa: F811
    pos = synth.cosmology(n, seed=n % 97, dtype=dtype)
    ref, _ = oracle_mod.compress(pos, oracle_mod.REL, 1e-3, want_perm=False)
    want = oracle_mod.decompress(ref)
    stream = torch.from_numpy(np.frombuffer(ref, np.uint8).copy()).cuda()
    ws = torch.empty(pc.pc_decompress_workspace_size(n), dtype=torch.uint8, device="cuda")
    out = torch.empty((n, 3), dtype=torch.from_numpy(pos).dtype).pin_memory()
    host = out.numpy()
    torch.cuda.synchronize()
    for k in range(20):
        host.fill(-1.0 - k)
        pc.pc_decompress(stream, out, ws)
        assert np.array_equal(host, want)
