"""Calls on a stream that holds part of the chip's SMs (a green context): launches
whose blocks wait for one another need no block that does not fit."""
import ctypes as C

import numpy as np
import pytest

from gpu_util import device, og, torch

pytestmark = pytest.mark.gpu


class _Part:
    """A stream on at least sms of the SMs, by the driver API."""

    def __init__(self, sms):
        self.cu = cu = C.CDLL("libcuda.so.1")
        resource = C.c_char * 144  # CUdevResource: type, padding, union of 48 bytes
        dev, whole, part, rest = C.c_int(), resource(), resource(), resource()
        n, desc = C.c_uint(1), C.c_void_p()
        self.ctx, s = C.c_void_p(), C.c_void_p()
        ok = [cu.cuDeviceGet(C.byref(dev), 0), cu.cuDeviceGetDevResource(dev, whole, 1),
              cu.cuDevSmResourceSplitByCount(part, C.byref(n), whole, rest, 0, sms),
              cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1),
              cu.cuGreenCtxCreate(C.byref(self.ctx), desc, dev, 1)]
        if any(ok):
            pytest.skip(f"no green context here: {ok}")
        assert cu.cuGreenCtxStreamCreate(C.byref(s), self.ctx, 1, 0) == 0
        self.sms = int.from_bytes(part.raw[96:100], "little")
        self.s, self.stream = s, torch.cuda.ExternalStream(s.value)

    def close(self):
        torch.cuda.synchronize()
        self.cu.cuStreamDestroy_v2(self.s)
        self.cu.cuGreenCtxDestroy(self.ctx)


@pytest.mark.parametrize("n", [300, 300_000])
def test_build_and_gradient_on_part_of_the_chip(n):
    dev = device()
    m = og()
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    pos[: n // 2] = np.mod(0.3 + 0.01 * rng.standard_normal((n // 2, 3)), 1.0)
    p = torch.tensor(pos, dtype=torch.float64, device=dev)
    mass = torch.ones(n, dtype=torch.float64, device=dev)
    w = torch.randn((n, 3), device=dev, generator=torch.Generator(dev).manual_seed(1))
    r_s = min(0.1, 0.4 * n ** (-1 / 3))

    def call(stream):
        keys, order = m.keys_sort(p, 1.0, stream=stream)
        tree = m.tree_build(keys, order, p, mass, 1e-4, 1.0, stream=stream)
        return tree.nodes(stream), m.shortrange_accel(tree, r_s, 0.5, stream=stream)[0], \
            m.shortrange_adjoint(tree, r_s, 0.5, w, stream=stream)

    ref = call(None)
    part = _Part(16)
    assert part.sms < torch.cuda.get_device_properties(0).multi_processor_count
    torch.cuda.synchronize()
    got = call(part.stream)
    part.stream.synchronize()
    for k, v in ref[0].items():
        assert torch.equal(got[0][k], v), k
    assert torch.equal(got[1], ref[1])
    for a, b in zip(got[2], ref[2]):  # FP64 sums in any order
        assert (a - b).abs().max() <= 1e-9 * b.abs().max()
    part.close()
