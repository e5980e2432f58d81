"""The FP32 network kernel (warp tiles of 32 samples, 12 warps per CTA) at the
edges of its tiles against the FP64 forward, and its SiLU on its own.

Tolerances: |dr| <= 2e-6 as for every FP32 forward (64-term FP32 sums).  SiLU:
relative 5e-7 for -87 < z (ex2.approx 2^-22, and the roundings of the sum, the
Newton reciprocal and the product, 2^-24 each, and of the exponent's
correction); below -87 (where SiLU is above -1.5e-36) absolute 1e-30."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2206_02937_gb300 import workloads as wl
from tests.test_gpu_mlp import _run, _theta
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("features", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 383, 4863, 4864, 4865, 58369])
def test_tile_edges(n, features):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    u, k = wl.c3(n, seed=40)
    th = _theta(3, gain=1.5)
    ref, _ = omlp.forward(th.astype(np.float32).astype(np.float64),
                          omlp.features(u, k, mode="invariants" if features else "momenta"))
    out, _ = _run(torch, th, u, k, [cg.MODE_MLP_FP32], calibrate=True, features=features)
    assert np.abs(out[cg.MODE_MLP_FP32] - ref).max() <= 2e-6


def test_silu_f32():
    torch_cuda()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    build = os.path.join(HERE, "_build")
    os.makedirs(build, exist_ok=True)
    so = os.path.join(build, "libsilu_f32.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-o", so, os.path.join(HERE, "silu_f32_eval.cu")])
    L = ctypes.CDLL(so)
    L.silu_f32_eval.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
    z = np.concatenate([np.linspace(-110.0, 110.0, 2_000_001), np.geomspace(1e-30, 1e30, 200_001),
                        -np.geomspace(1e-30, 87.0, 200_001), [0.0, -1e4, -1e30, np.nan]]).astype(np.float32)
    out = np.empty_like(z)
    assert L.silu_f32_eval(z.ctypes.data, z.size, out.ctypes.data) == 0
    z64 = z.astype(np.float64)
    with np.errstate(over="ignore", invalid="ignore"):
        exact = z64 / (1.0 + np.exp(-z64))
    inner = z64 > -87.0
    nz = inner & (exact != 0.0) & (np.abs(exact) > 1e-30)
    rel = np.abs(out[nz] / exact[nz] - 1.0)
    print("silu2_f32: max relative error", rel.max(), "mean", rel.mean())
    assert rel.max() <= 5e-7
    low = z64 <= -87.0
    assert np.all(np.abs(out[low] - exact[low])[z64[low] > -1e20] <= 1e-30)
    assert np.isnan(out[-1]) and out[-4] == 0.0


def test_silu_f32_at_the_ends_of_its_range():
    """Infinities, the largest numbers and NaN: z itself above 87 (sigma is 1 to
    FP32), a value between SiLU(-87) = -1.4e-36 and 0 below -87."""
    torch_cuda()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    build = os.path.join(HERE, "_build")
    os.makedirs(build, exist_ok=True)
    so = os.path.join(build, "libsilu_f32_ends.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-o", so, os.path.join(HERE, "silu_f32_eval.cu")])
    L = ctypes.CDLL(so)
    L.silu_f32_eval.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
    top = np.finfo(np.float32).max
    ends = np.concatenate([np.geomspace(87.0, top, 3001), [top, np.inf]]).astype(np.float32)
    z = np.concatenate([ends, -ends, [np.nan]]).astype(np.float32)
    out = np.empty_like(z)
    assert L.silu_f32_eval(z.ctypes.data, z.size, out.ctypes.data) == 0
    high, low = out[:ends.size], out[ends.size:-1]
    assert np.isinf(high[-1]) and high[-1] > 0 and np.all(np.abs(high[:-1].astype(np.float64) / ends[:-1] - 1.0) <= 5e-7)
    assert np.all(low <= 0.0) and np.all(low >= -1.5e-36)
    assert np.isnan(out[-1])


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000, 4097])
def test_calibration_sees_the_samples_alone(n):
    """The FP8 scales are 448 over the largest |input| of each hidden layer over
    the n samples, whatever fills the rest of a tile: against the FP64 maxima, to
    the FP32 forward's 64-term sums (relative 2e-5; biases apart from zero, so that
    a sample of zeros would show)."""
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    th = _theta(7, gain=1.5)
    off = [384, 4544, 8704, 12864]  # the hidden layers' biases
    rng = np.random.default_rng(8)
    for o in off:
        th[o:o + 64] = rng.uniform(1.0, 2.0, 64)
    th = th.astype(np.float32)
    u, k = wl.c3(n, seed=41)
    t = th.astype(np.float64)
    h, want = omlp.features(u, k).T, []
    for l, (o, i) in enumerate(((64, 6), (64, 64), (64, 64))):
        at = (0, 448, 4608)[l]
        want.append(np.abs(h).max())
        z = h @ t[at:at + o * i].reshape(o, i).T + t[at + o * i:at + o * i + o]
        h = z / (1.0 + np.exp(-z))
    want.append(np.abs(h).max())
    ctx = cg.compton_init(1, 1, 1.0, 0.05, 1)
    try:
        cg.compton_mlp_set_params(ctx, th)
        cg.compton_mlp_calibrate(ctx, torch.from_numpy(u).cuda(), torch.from_numpy(k).cuda())
        torch.cuda.synchronize()
        scales = np.frombuffer(cg.compton_mlp_save(ctx)[40:56], np.float32)
    finally:
        cg.compton_destroy(ctx)
    assert np.allclose(scales, 448.0 / np.array(want), rtol=2e-5, atol=0.0)
