"""The march's steps over empty macrocells, on the host: the header the kernel
uses, compiled with the host compiler.  No sample that a step passes over may
lie in another macrocell than the one it starts in, however far the eye is
(float32 distances grow coarser than a vertex cell), and the macrocells'
numbers hold beyond 2^31."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "raymarch_step.h"
using namespace veg;
// Marches one ray through macrocells that are all empty; counts the samples
// passed over that lie in another macrocell, and the steps taken.
extern "C" void walk(const float* eye, const float* d, float ta, float tb, float step, float inv_h,
                     int R, int shift, long long* wrong, long long* steps, long long* samples) {
  MarchRay r;
  for (int c = 0; c < 3; ++c) r.eye[c] = eye[c], r.d[c] = d[c];
  r.ta = ta, r.step = step, r.inv_h = inv_h, r.R = R;
  float g[3], q[3];
  int ic[3], jc[3];
  const int n = (int)floorf((tb - ta) / step);
  const MarchStep over = march_step(r, n, shift);
  for (int k = 0; k < n; ++*steps) {
    march_place(r, k, g, ic);
    const int m[3] = {ic[0] >> shift, ic[1] >> shift, ic[2] >> shift};
    const int next = march_next(r, over, k, n, g, m, shift);
    for (int j = k + 1; j < next; ++j) {
      march_place(r, j, q, jc);
      for (int c = 0; c < 3; ++c)
        if (jc[c] >> shift != m[c]) { ++*wrong; break; }
    }
    *samples += next - k;
    k = next;
  }
}
extern "C" long long macrocell(int x, int y, int z, int cells) {
  const int m[3] = {x, y, z};
  return march_macrocell(m, cells);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("step")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2504_13339_gb300", "csrc"), "-o",
                    str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


def rays(distance, count, rng):
    """Rays from `distance` away through points of the volume, in float32."""
    v = rng.normal(size=(count, 3))
    eye = (distance * v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.float32)
    d = rng.uniform(-0.9, 0.9, (count, 3)) - eye
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    for e, u in zip(eye, d):
        with np.errstate(divide="ignore"):
            a, b = (-1 - e) / u, (1 - e) / u
        ta, tb = np.float32(np.minimum(a, b).max()), np.float32(np.maximum(a, b).min())
        if tb > ta:
            yield e, u, ta, tb


@pytest.mark.parametrize("R,cell,distance,per", [
    (256, 8, 4.0, 0.5), (1024, 8, 600.0, 1.0), (1024, 64, 5000.0, 1.0), (2048, 8, 4.0, 0.5),
    (2048, 8, 300.0, 1.0), (2048, 16, 1000.0, 1.0), (2048, 8, 20000.0, 1.0), (2048, 1, 300.0, 0.1),
    (64, 4, 50000.0, 0.5)])
def test_no_step_leaves_its_macrocell(lib, R, cell, distance, per):
    rng = np.random.default_rng(R + cell)
    f32, p = ctypes.c_float, lambda a: a.ctypes.data_as(ctypes.c_void_p)
    wrong, steps, samples = (ctypes.c_longlong(0) for _ in range(3))
    h = 2.0 / (R - 1)
    for e, u, ta, tb in rays(distance, 60, rng):
        lib.walk(p(e), p(u), f32(ta), f32(tb), f32(per * h), f32(1.0 / h), R,
                 cell.bit_length() - 1, ctypes.byref(wrong), ctypes.byref(steps),
                 ctypes.byref(samples))
    assert samples.value > 0 and wrong.value == 0
    if distance == 4.0:  # near eyes: still a few steps per macrocell
        assert steps.value * cell / per < 4.0 * samples.value


@pytest.mark.parametrize("cells", [1, 32, 1290, 1291, 2047])
def test_macrocell_numbers_beyond_31_bits(lib, cells):
    """1291^3 macrocells and more (vertex cells of 1292^3 vertices) number past
    2^31 - 1."""
    lib.macrocell.restype = ctypes.c_longlong
    for x, y, z in ((0, 0, 0), (cells - 1, 0, cells - 1), (cells - 1,) * 3):
        assert lib.macrocell(x, y, z, cells) == x + cells * (y + cells * z)
