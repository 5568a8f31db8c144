"""Streams of a green context, which run on some of the device's SMs only: the
cooperative launches have to fit them, and every result is the one of an
ordinary stream, bit for bit (gradients: to the order of their atomics)."""

import ctypes as C

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def t2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_15235_gb300 import build_lib
    build_lib.build()
    import paper_2310_15235_gb300 as mod
    mod.load_library()
    return mod


class _Resource(C.Structure):  # CUdevResource of an SM partition
    _fields_ = [("type", C.c_int), ("pad", C.c_ubyte * 92), ("sm_count", C.c_uint),
                ("rest", C.c_ubyte * 44)]


@pytest.fixture()
def small_stream(t2):
    """A stream on about 16 of the SMs."""
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    dev = C.c_int(0)
    assert cu.cuDeviceGet(C.byref(dev), torch.cuda.current_device()) == 0
    whole, part, groups = _Resource(), _Resource(), C.c_uint(1)
    assert cu.cuDeviceGetDevResource(dev, C.byref(whole), 1) == 0
    if cu.cuDevSmResourceSplitByCount(C.byref(part), C.byref(groups), C.byref(whole), None, 0, 16):
        pytest.skip("the driver does not split the SMs")
    assert 0 < part.sm_count < whole.sm_count // 2
    desc, green, stream = C.c_void_p(), C.c_void_p(), C.c_void_p()
    assert cu.cuDevResourceGenerateDesc(C.byref(desc), C.byref(part), 1) == 0
    assert cu.cuGreenCtxCreate(C.byref(green), desc, dev, 1) == 0
    assert cu.cuGreenCtxStreamCreate(C.byref(stream), green, 1, 0) == 0
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    assert cu.cuStreamDestroy_v2(stream) == 0 and cu.cuGreenCtxDestroy(green) == 0


def test_every_cooperative_launch_fits(t2, small_stream):
    # 60k elements: sort, topology, sums and tables each want more blocks than 16 SMs hold
    case = workloads.random_case(60_000, 300, nb=2, seed=601, clumped=True, bucket=3)
    act = case["active"][:20_001]
    rows = torch.as_tensor(act, device="cuda")
    f = [torch.as_tensor(case[k], device="cuda").to(d) for k, d in
         (("pos", torch.float64), ("mass", torch.float32), ("kappa", torch.float32),
          ("lum", torch.float32), ("h", torch.float32))]
    gJ = torch.ones((len(act), 2), device="cuda")

    def run(stream):
        torch.cuda.synchronize()
        tree = t2.build(*f, case["box_lo"], case["box_size"], case["bucket"], stream=stream)
        out = [tree.export("perm"), tree.export("B")]
        out.append(tree.J(rows, 4, 0.5, stream=stream))
        out.append(tree.J(rows, 2, 0.75, flags=t2.BUCKET, stream=stream))
        grads = tree.J_backward(rows, gJ, 2, 0.75, stream=stream)
        plan = t2.Batch([tree], np.array([0, len(act)], np.int64), np.array([0], np.int32), nside=2,
                        theta=0.75, stream=stream)
        out.append(plan.run(rows, stream=stream))
        plan.status(stream=stream)
        torch.cuda.synchronize()
        plan.free()
        tree.free()
        torch.cuda.synchronize()
        return out, grads

    want, gwant = run(None)
    got, ggot = run(small_stream)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    for a, b in zip(ggot, gwant):
        torch.testing.assert_close(a, b, rtol=1e-4, atol=1e-6 * float(b.abs().max()))
