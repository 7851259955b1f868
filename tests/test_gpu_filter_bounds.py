"""The row filter's single-precision face data against exact rationals: every evaluated bound lies
between the true one and E beside it, on the safe side, and its coefficients are as close to the true
ones as four roundings make them (the span kernel's filter).  Likewise the lines that bound a slice's
candidate rows: each lies outside the tet, and no farther than its margin."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2106_01326_gb300 import build as vbuild

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "voxtet_rows.cuh"
using namespace voxtet;
struct In { long long L, nx, ny, nz; int sh, fb, fc, b, c, pad; };
struct Out { float beta, gamma, e, t; };
__global__ void faces(const In *in, Out *out, int n, int strict) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const In q = in[i];
  float a, b, g;
  Out o;
  const float fb = (float)q.fb, fc = (float)q.fc;
  o.e = strict ? face_bound<true>(q.L, q.nx, q.ny, q.nz, q.sh, fb, fc, a, b, g)
               : face_bound<false>(q.L, q.nx, q.ny, q.nz, q.sh, fb, fc, a, b, g);
  o.beta = b;
  o.gamma = g;
  o.t = __fmaf_rn(b, (float)q.b, __fmaf_rn(g, (float)q.c, a));
  out[i] = o;
}
struct Lines { float aL0, kL0, aL1, kL1, aU0, kU0, aU1, kU1, z0, z1; int j0, l0, nb, nc; };
__global__ void lines(const int3 *v, Lines *out, int n, int sh, int res) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  Box bx;
  const int3 V[4] = {v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]};
  tet_box(V, sh, res, res, 0, res, bx);
  RowRange R = {};
  if (bx.nb > 0 && bx.nc > 0) row_range(V, bx, sh, R);
  out[i] = {R.aL0, R.kL0, R.aL1, R.kL1, R.aU0, R.kU0, R.aU1, R.kU1, R.z0, R.z1, bx.j0, bx.l0, bx.nb, bx.nc};
}
extern "C" int run_lines(const int3 *v, Lines *out, int n, int sh, int res) {
  lines<<<(n + 127) / 128, 128>>>(v, out, n, sh, res);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_faces(const In *in, Out *out, int n, int strict) {
  faces<<<(n + 127) / 128, 128>>>(in, out, n, strict);
  return (int)cudaDeviceSynchronize();
}
"""
IN = np.dtype([("L", "<i8"), ("nx", "<i8"), ("ny", "<i8"), ("nz", "<i8"), ("sh", "<i4"), ("fb", "<i4"), ("fc", "<i4"),
               ("b", "<i4"), ("c", "<i4"), ("pad", "<i4")])
OUT = np.dtype([(k, "<f4") for k in ("beta", "gamma", "e", "t")])
U = Fraction(1, 1 << 24)


@pytest.fixture(scope="module")
def dll(tmp_path_factory):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    d = tmp_path_factory.mktemp("faces")
    src, lib = os.path.join(d, "faces.cu"), os.path.join(d, "faces.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([vbuild._nvcc(), *vbuild.NVCC_FLAGS, "-I", vbuild.CSRC, "-shared", "-cudart", "shared", "-o", lib,
                    src], check=True)
    return ctypes.CDLL(lib)


@pytest.fixture(scope="module")
def faces(dll):
    import torch

    def run(cases, strict):
        x = torch.from_numpy(cases.view(np.uint8).copy()).cuda()
        y = torch.zeros(len(cases) * OUT.itemsize, dtype=torch.uint8, device="cuda")
        assert dll.run_faces(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), len(cases), int(strict)) == 0
        return y.cpu().numpy().view(OUT)

    return run


def _log_int(rng, n, hi):
    """Whole numbers of either sign, their size spread over the logarithm of 1 .. hi."""
    x = np.exp(rng.uniform(0.0, np.log(float(hi)), n)).astype(np.int64)
    return np.clip(x, 1, hi - 1) * rng.choice([-1, 1], n)


def _cases(seed, n):
    rng = np.random.default_rng(seed)
    c = np.zeros(n, IN)
    c["sh"] = rng.integers(4, 21, n)
    for k in ("nx", "ny", "nz"):
        # |n 2^sh| stays within the 2^62 of a face's gradient
        c[k] = np.minimum(np.abs(_log_int(rng, n, 1 << 43)), (1 << 62) >> c["sh"].astype(np.int64)) * rng.choice([-1, 1], n)
    c["ny"][rng.random(n) < 0.1] = 0
    c["nz"][rng.random(n) < 0.1] = 0
    c["L"] = _log_int(rng, n, 3 << 61)
    c["fb"] = np.abs(_log_int(rng, n, 8192)) - 1
    c["fc"] = np.abs(_log_int(rng, n, 65536)) - 1
    # faces on multiples of 1/16 in a tenth of the cases
    lat = rng.random(n) < 0.1
    for k in ("ny", "nz"):
        c[k][lat] = rng.integers(-64, 65, lat.sum())
    c["nx"][lat] = rng.choice([-16, -4, -1, 1, 4, 16], lat.sum())
    c["L"][lat] = rng.integers(-4096, 4097, lat.sum()) << (c["sh"][lat].astype(np.int64) - 4)
    c["b"] = rng.integers(0, c["fb"] + 1)
    c["c"] = rng.integers(0, c["fc"] + 1)
    return c


@pytest.mark.parametrize("strict", [False, True])
def test_face_bounds(faces, strict):
    cases = _cases(3 + strict, 20000)
    out = faces(cases, strict)
    certified = 0
    for q, o in zip(cases, out):
        L, nx, ny, nz = (int(q[k]) for k in ("L", "nx", "ny", "nz"))
        alpha = Fraction(-L, nx << int(q["sh"]))
        beta, gamma = Fraction(-ny, nx), Fraction(-nz, nx)
        where = f"{q} {o}"
        # the coefficients: four roundings each, as the span kernel's
        assert abs(Fraction(float(o["beta"])) - beta) <= Fraction(40001, 10000) * U * abs(beta), where
        assert abs(Fraction(float(o["gamma"])) - gamma) <= Fraction(40001, 10000) * U * abs(gamma), where
        t = alpha + beta * int(q["b"]) + gamma * int(q["c"])
        T, E = Fraction(float(o["t"])), Fraction(float(o["e"]))
        S = abs(alpha) + abs(beta) * int(q["fb"]) + abs(gamma) * int(q["fc"])
        assert E <= Fraction(16001, 1000) * U * S, where  # the span kernel's bracket is 16 u S wide
        if E == 0:  # certified: the face takes multiples of 1/16 only, and T' passes no integer that t does not
            certified += 1
            assert all((16 * x).denominator == 1 for x in (alpha, beta, gamma)), where
            E = Fraction(1, 32)
        if (nx < 0) != strict:
            assert t <= T <= t + E, where
        else:
            assert t - E <= T <= t, where
    assert certified > 100



LINES = np.dtype([(k, "<f4") for k in ("aL0", "kL0", "aL1", "kL1", "aU0", "kU0", "aU1", "kU1", "z0", "z1")]
                 + [(k, "<i4") for k in ("j0", "l0", "nb", "nc")])


@pytest.mark.parametrize("res", [16, 512, 4096])
def test_row_range_lines(dll, res):
    """Tets of 1/2000 to 1/2 of the grid, some with edges parallel to y or z.  A slope rounds once, the
    line's evaluation at most twice (4u (|y'| + nb) with the margin's own rounding) and the margin is
    8u (|y'| + nb), so a line in the box is off by 4 to 12 of these units, outwards."""
    import torch

    rng = np.random.default_rng(res)
    n = 3000
    size = np.exp(rng.uniform(np.log(1 / 2000), np.log(0.5), (n, 1, 1)))
    v = (rng.uniform(0.1, 0.9, (n, 1, 3)) + size * rng.uniform(-0.5, 0.5, (n, 4, 3))) * (1 << 20)
    v = np.rint(v).astype(np.int32)
    flat = rng.random(n) < 0.2
    v[flat, 1, 2] = v[flat, 0, 2]
    flat = rng.random(n) < 0.2
    v[flat, 3, 2] = v[flat, 2, 2]
    flat = rng.random(n) < 0.1
    v[flat, 2, 1:] = v[flat, 1, 1:]
    sh = 20 - (res.bit_length() - 1)
    x = torch.from_numpy(v).cuda()
    y = torch.zeros(n * LINES.itemsize, dtype=torch.uint8, device="cuda")
    assert dll.run_lines(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), n, sh, res) == 0
    half, checked = 1 << (sh - 1), 0
    for t, R in zip(v.tolist(), y.cpu().numpy().view(LINES)):
        nb, nc = int(R["nb"]), int(R["nc"])
        if nb <= 0 or nc <= 0:
            continue
        p = sorted((z, w) for _, w, z in t)
        yp = [Fraction(w - half - (int(R["j0"]) << sh), 1 << sh) for _, w in p]
        zp = [Fraction(z - half - (int(R["l0"]) << sh), 1 << sh) for z, _ in p]

        def k(a, b):
            if zp[a] == zp[b]:
                return None if yp[a] == yp[b] else float("inf")
            return (yp[b] - yp[a]) / (zp[b] - zp[a])

        for name, base, edges, pick, out in (("L0", 0, ((0, 1), (0, 2), (0, 3)), min, -1), ("L1", 3, ((0, 3), (1, 3), (2, 3)), max, -1),
                                             ("U0", 0, ((0, 1), (0, 2), (0, 3)), max, 1), ("U1", 3, ((0, 3), (1, 3), (2, 3)), min, 1)):
            slope = pick(s for s in (k(a, b) for a, b in edges) if s is not None)
            if slope == float("inf"):
                assert R["a" + name] == out * np.inf and R["k" + name] == 0
                continue
            unit = U * (abs(yp[base]) + nb)
            z0 = Fraction(float(R["z0" if base == 0 else "z1"]))
            assert z0 == zp[base]
            for c in {0, nc // 3, nc - 1}:
                true = yp[base] + slope * (c - zp[base])
                if not 0 <= true <= nb:
                    continue
                checked += 1
                # the kernel's evaluation, one FMA: a float64 product and sum, rounded, is as close
                got = Fraction(float(np.float32(float(R["k" + name]) * float(c - z0) + float(R["a" + name]))))
                assert 4 * unit <= out * (got - true) <= 12 * unit, (t, name, c)
    assert checked > 1000
