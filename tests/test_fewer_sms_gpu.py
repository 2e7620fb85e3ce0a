"""Compression on a stream that has a part of the device's SMs (a green context):
the launch of several levels (csrc/k_split.cu), whose CTAs wait for one another,
takes the SMs there are.  Streams, permutations and decoded positions equal the
oracle's.
"""
import ctypes

import numpy as np
import pytest

import synth
from test_parity_gpu import pc  # noqa: F401  (a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SM = 1  # CU_DEV_RESOURCE_TYPE_SM


class Resource(ctypes.Structure):
    """CUdevResource: its type, padding, and (of a union of 48 bytes) the SM count."""
    _fields_ = [("type", ctypes.c_int), ("padding", ctypes.c_ubyte * 92), ("sm_count", ctypes.c_uint),
                ("rest", ctypes.c_ubyte * 44)]


@pytest.fixture(scope="module")
def part():
    """A stream of a green context with a quarter of the SMs or a little more."""
    torch.cuda.synchronize()  # the primary context exists
    cu = ctypes.CDLL("libcuda.so.1")
    names = ("cuDeviceGetDevResource", "cuDevSmResourceSplitByCount", "cuDevResourceGenerateDesc", "cuGreenCtxCreate",
             "cuGreenCtxStreamCreate", "cuGreenCtxDestroy", "cuStreamDestroy_v2")
    if not all(hasattr(cu, n) for n in names):
        pytest.skip("the driver has no green contexts")

    def ok(rc, what):
        if rc != 0:
            pytest.skip(f"{what}: CUDA error {rc}")

    whole, piece, rest = Resource(), Resource(), Resource()
    ok(cu.cuDeviceGetDevResource(0, ctypes.byref(whole), SM), "cuDeviceGetDevResource")
    groups = ctypes.c_uint(1)
    ok(cu.cuDevSmResourceSplitByCount(ctypes.byref(piece), ctypes.byref(groups), ctypes.byref(whole),
                                      ctypes.byref(rest), 0, whole.sm_count // 4), "cuDevSmResourceSplitByCount")
    assert groups.value == 1 and 0 < piece.sm_count < whole.sm_count
    desc, ctx, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    ok(cu.cuDevResourceGenerateDesc(ctypes.byref(desc), ctypes.byref(piece), 1), "cuDevResourceGenerateDesc")
    ok(cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, 0, 1), "cuGreenCtxCreate")
    ok(cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0), "cuGreenCtxStreamCreate")
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


# one launch of a few levels and of eight, two launches, and one within the part's SMs
@pytest.mark.parametrize("n,eb,r", [(300_007, 1e-3, 4096), (1_100_003, 1e-4, 2048), (2_300_017, 8e-6, 4096),
                                    (40_003, 1e-4, 500)])
def test_a_stream_with_fewer_sms(pc, oracle_mod, part, n, eb, r):  # noqa: F811
    pos = synth.cosmology(n, seed=n % 53)
    ref, ref_perm = oracle_mod.compress(pos, oracle_mod.REL, eb, leaf_size=r)
    dpos = torch.from_numpy(pos).cuda()
    c = pc.Compressor(n, pc.PC_F32, r, True)
    plain = pc.Compressor(n, pc.PC_F32, r)
    out = torch.empty_like(dpos)
    for w in (c.ws, plain.ws):
        w.fill_(0xA5)
    torch.cuda.synchronize()
    for _ in range(2):
        size = c.compress(dpos, pc.PC_EB_REL, eb, stream=part)
        assert plain.compress(dpos, pc.PC_EB_REL, eb, stream=part) == size
        c.decompress(c.out, out, size, stream=part)
        part.synchronize()
        assert c.out[:size].cpu().numpy().tobytes() == ref
        assert plain.out[:size].cpu().numpy().tobytes() == ref
        assert np.array_equal(c.perm[:n].cpu().numpy().astype(np.int64), ref_perm)
        assert out.cpu().numpy().tobytes() == oracle_mod.decompress(ref).tobytes()
