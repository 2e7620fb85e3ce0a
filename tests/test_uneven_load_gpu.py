"""Compressions that run beside others of other sizes: the SMs that a launch of
several levels takes (csrc/k_split.cu) follow the particles in flight.  Large
and small snapshots in one batch, and plain calls from several host threads at
once: every stream equals the same snapshot's alone and, where the oracle is
quick, the oracle's, also with two such launches on part of the SMs, each of
many subroots, from a workspace full of stale bytes.  And a batch of one large
snapshot among small ones takes little longer than the large one alone.
"""
import threading
import time

import numpy as np
import pytest

import synth
from test_parity_gpu import pc  # noqa: F401  (a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# particles, value-range-relative bound, leaf size
ITEMS = [
    (4_300_007, 1e-4, 200),   # two launches, five and four levels
    (2_300_017, 8e-6, 4096),  # two launches, 16-bit codes
    (700_001, 1e-4, 500), (300_007, 1e-3, 4096), (40_003, 8e-6, 60),
    (10_007, 1e-2, 4096), (10_007, 1e-4, 16), (1_000, 1e-3, 64),
]


@pytest.fixture(scope="module")
def snapshots(pc):  # noqa: F811
    """Positions on the device and the streams of lone calls."""
    out = []
    for i, (n, eb, r) in enumerate(ITEMS):
        pos = synth.cosmology(n, seed=60 + i)
        d = torch.from_numpy(pos).cuda()
        c = pc.Compressor(n, pc.PC_F32, r)
        size = c.compress(d, pc.PC_EB_REL, eb)
        out.append((pos, d, c.out[:size].clone()))
    torch.cuda.synchronize()
    return out


def test_lone_calls_match_the_oracle(pc, oracle_mod, snapshots):  # noqa: F811
    for (n, eb, r), (pos, _, alone) in zip(ITEMS, snapshots):
        ref, _ = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r, want_perm=False)
        assert alone.cpu().numpy().tobytes() == ref


@pytest.mark.parametrize("lanes", [2, 8])
def test_uneven_batches(pc, snapshots, lanes):  # noqa: F811
    pick = list(range(len(ITEMS))) + [5] * 6
    jobs = [(snapshots[i][1], pc.PC_EB_REL, ITEMS[i][1], ITEMS[i][2]) for i in pick]
    outs = [torch.empty(pc.pc_compress_bound(ITEMS[i][0], pc.PC_F32, ITEMS[i][2]), dtype=torch.uint8, device="cuda")
            for i in pick]
    ws = torch.empty(pc.pc_compress_batch_workspace_size([(ITEMS[i][0], pc.PC_F32, ITEMS[i][2]) for i in pick], lanes),
                     dtype=torch.uint8, device="cuda")
    for _ in range(3):
        ws.fill_(0xA5)
        sizes, statuses = pc.pc_compress_batch(jobs, outs, ws, lanes)
        assert statuses == [pc.PC_OK] * len(pick)
        for i, o, size in zip(pick, outs, sizes):
            assert torch.equal(o[:size], snapshots[i][2])


def test_host_threads_at_once(pc, snapshots):  # noqa: F811
    torch.cuda.synchronize()
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        i = k % len(ITEMS)
        n, eb, r = ITEMS[i]
        with torch.cuda.stream(st):
            c = pc.Compressor(n, pc.PC_F32, r)
        for _ in range(4):
            size = c.compress(snapshots[i][1], pc.PC_EB_REL, eb, stream=st)
            with torch.cuda.stream(st):
                if not torch.equal(c.out[:size], snapshots[i][2]):
                    bad.append(i)
        st.synchronize()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_a_large_snapshot_keeps_its_sms(pc):  # noqa: F811
    """2^26 particles among fifteen of 10^4: 1.15 times the large one alone when the SMs follow
    the particles, 3.9 times with an even share for every lane."""
    n = 1 << 26
    g = torch.Generator(device="cuda").manual_seed(5)
    pos = torch.rand((n, 3), generator=g, device="cuda")
    ns = [n] + [10_000] * 15
    outs = [torch.empty(pc.pc_compress_bound(m, pc.PC_F32), dtype=torch.uint8, device="cuda") for m in ns]
    ws = torch.empty(pc.pc_compress_batch_workspace_size([(m, pc.PC_F32, 0) for m in ns], 8), dtype=torch.uint8,
                     device="cuda")
    jobs = [(pos[:m], pc.PC_EB_REL, 1e-4, 0) for m in ns]

    def best(call):
        times = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            call()
            times.append(time.perf_counter() - t0)
        return min(times[1:])

    alone = best(lambda: pc.pc_compress(pos, pc.PC_EB_REL, 1e-4, outs[0], ws))
    batch = best(lambda: pc.pc_compress_batch(jobs, outs, ws, 8))
    print(f"alone {alone * 1e3:.2f} ms, batch {batch * 1e3:.2f} ms")
    assert batch < 2.0 * alone
