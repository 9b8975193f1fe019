"""The slope of a pixel's ray from the focal length's reciprocal (csrc/sgad_ray.cuh, compiled
here for the host) has the bits of the division for every column of a range of cameras."""
import ctypes
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = """
#include "sgad_ray.cuh"
extern "C" void slopes(const float *a, const float *f, const float *inv_f, float *out, long n)
{
    for (long i = 0; i < n; ++i) out[i] = sgad::ray_slope(a[i], f[i], inv_f[i]);
}
"""


def test_ray_slope_is_the_division(tmp_path):
    src, lib = tmp_path / "s.cpp", tmp_path / "s.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2603_21055_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).slopes
    rng = np.random.default_rng(0)
    f = np.exp(rng.uniform(np.log(2.0), np.log(2e4), 400)).astype(np.float32)
    f[:8] = np.frombuffer(np.array([0x43ffffff, 0x43800001, 0x447fffff, 0x3f7fffff, 0x44160000, 0x3f800001, 0x43fa0000,
                                    0x44000000], np.uint32).tobytes(), np.float32)    # mantissas of ones, of one, whole sizes
    cx = np.where(np.arange(400) % 3 == 0, 0.5 * rng.integers(0, 4000, 400), rng.uniform(0, 2000, 400)).astype(np.float32)
    a = np.arange(4096, dtype=np.float32)[None, :] - cx[:, None]
    a, ff = np.ascontiguousarray(a).ravel(), np.repeat(f, 4096)
    inv, out = (np.float32(1) / ff).astype(np.float32), np.empty_like(a)
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    fn(ptr(a), ptr(ff), ptr(inv), ptr(out), ctypes.c_long(a.size))
    assert np.array_equal(out.view(np.uint32), (a / ff).view(np.uint32))
