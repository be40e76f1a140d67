"""The trace's reciprocal of a direction component against CUDA's correctly rounded
one.  Expected, from the iteration's error analysis: the same bits for every input
whose mantissa is not all ones and whose reciprocal is a normal number; at most one
unit in the last place apart for the others; zeros, infinities and NaN as rounded."""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def reciprocals(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = str(tmp_path_factory.mktemp("reciprocal") / "reciprocal.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-o", so, os.path.join(HERE, "reciprocal", "reciprocal.cu")], check=True, timeout=300)
    fn = ctypes.CDLL(so).reciprocals
    fn.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]

    def run(bits):
        x = bits.to(torch.int32).contiguous()
        own, rounded = torch.empty_like(x), torch.empty_like(x)
        assert fn(x.data_ptr(), x.numel(), own.data_ptr(), rounded.data_ptr(),
                  torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        return own, rounded
    return run


def _check(run, bits):
    """bits: binary32 patterns (int64 tensor)."""
    own, rounded = run(torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits))
    x = torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits).to(torch.int32)
    finite_result = (rounded & 0x7FFFFFFF) < 0x7F800000
    subnormal = (rounded & 0x7FFFFFFF) < 0x00800000
    ones = (x & 0x7FFFFF) == 0x7FFFFF
    loose = finite_result & (subnormal | ones)
    assert torch.equal(own[~loose], rounded[~loose])
    assert ((own[loose] - rounded[loose]).abs() <= 1).all()  # neighbouring patterns of one sign
    return int(loose.sum())


@pytest.mark.parametrize("exponent", [0, 126, 127, 128, 180, 252, 253, 254])
@pytest.mark.parametrize("sign", [0, 1])
def test_every_mantissa(reciprocals, exponent, sign):
    m = torch.arange(2 ** 23, device="cuda", dtype=torch.int64)
    loose = _check(reciprocals, m | exponent << 23 | sign << 31)
    assert loose <= 1 or exponent >= 253


def test_every_exponent_and_special_values(reciprocals):
    g = torch.Generator("cuda").manual_seed(1)
    m = torch.randint(0, 2 ** 23, (4096,), generator=g, device="cuda", dtype=torch.int64)
    edges = torch.tensor([0, 1, 2, 0x3FFFFF, 0x400000, 0x400001, 0x7FFFFD, 0x7FFFFE, 0x7FFFFF], device="cuda")
    m = torch.cat([m, edges])
    e = torch.arange(256, device="cuda", dtype=torch.int64)
    bits = (m[None] | e[:, None] << 23).reshape(-1)
    _check(reciprocals, bits)  # zero, subnormals, infinity and NaN among them
    _check(reciprocals, bits | 2 ** 31)
    clamp = int(torch.tensor(1e-18).view(torch.int32))
    near = torch.arange(clamp - 4096, clamp + 4096, device="cuda", dtype=torch.int64)
    _check(reciprocals, torch.cat([near, near | 2 ** 31]))
