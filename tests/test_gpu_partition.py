"""Contexts on a stream with a part of the device's SMs (a green context): the
persistent launches, whose blocks wait for one another, are cut for the SMs
that the stream has, and a factor cut for more is served by other kernels."""
from __future__ import annotations

import ctypes

import pytest
import torch

import paper_2410_04512_gb300 as sgp
import workloads
from gpu_common import GpuSystem, dev_tensor, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture()
def part_stream(cuda_device):
    """A stream with 32 SMs or more, but not all of them."""
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    dev = ctypes.c_int()
    whole, part, rest = (ctypes.create_string_buffer(256) for _ in range(3))   # CUdevResource, 144 bytes
    desc, green, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    groups = ctypes.c_uint(1)
    calls = [
        lambda: cu.cuDeviceGet(ctypes.byref(dev), 0),
        lambda: cu.cuDeviceGetDevResource(dev, whole, 1),                       # the SMs
        lambda: cu.cuDevSmResourceSplitByCount(part, ctypes.byref(groups), whole, rest, 0, 32),
        lambda: cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
        lambda: cu.cuGreenCtxCreate(ctypes.byref(green), desc, dev, 1),         # (default stream: required)
        lambda: cu.cuGreenCtxStreamCreate(ctypes.byref(stream), green, 1, 0),   # non-blocking: required
    ]
    for c in calls:
        if c() != 0:
            pytest.skip("no green contexts here")
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(green)


@pytest.mark.parametrize("precision", [sgp.PREC_F64, sgp.PREC_MIXED])
def test_solves_on_a_part_of_the_device(part_stream, precision):
    """Bounds as for the persistent launch against the level kernels."""
    c = workloads.ball(n=30011, seed=2115, gamma0=1e-3)
    F = dev_tensor(c.forces())
    whole = sgp.Context(0)
    a = GpuSystem(whole, c, precision=precision)
    ref, _ = whole.pcg_solve(a.M, a.Fac, F, tol=1e-10, precision=precision)
    xr = whole.tree_apply(a.Fac, F)
    torch.cuda.synchronize()
    cx = sgp.Context(0, part_stream)
    with torch.cuda.stream(part_stream):
        b = GpuSystem(cx, c, precision=precision)
        # its own factor: in the persistent launch, on the SMs it has
        cx.launch_count(reset=True)
        v, info = cx.pcg_solve(b.M, b.Fac, F, tol=1e-10, precision=precision)
        assert info.status == 0 and cx.launch_count() <= 100
        w, _ = cx.pcg_solve(b.M, None, F, tol=1e-10, precond=sgp.PRECOND_BLOCK_JACOBI, precision=precision)
        x = cx.tree_apply(b.Fac, F)
        # the whole device's factor
        u, info = cx.pcg_solve(a.M, a.Fac, F, tol=1e-10, precision=precision)
        assert info.status == 0
        y = cx.tree_apply(a.Fac, F)
        part_stream.synchronize()
    for t in (v, w, u):
        assert rel_err(t.cpu().numpy(), ref.cpu().numpy()) <= 1e-8
    for t in (x, y):
        assert rel_err(t.cpu().numpy(), xr.cpu().numpy()) <= 1e-10
