"""split_f64 and join_f64 (a double as a pair of floats and back, on the integer pipe) against the plain
conversions, bit for bit: random signs, exponents and significands over the whole range of doubles, ties of the
first rounding and their neighbours, carries into the next binade, the exponents at which the routines change
over to the conversions, and pairs whose sum lies below the binade of the head."""
import ctypes
import pathlib
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include "kernels.cuh"
__global__ void split_k(int64_t n, const double* v, float* h, float* l) {
  for (int64_t i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) hdg::split_f64(v[i], h[i], l[i]);
}
__global__ void join_k(int64_t n, const float* h, const float* l, double* v) {
  for (int64_t i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) v[i] = hdg::join_f64(h[i], l[i]);
}
extern "C" int split(int64_t n, const double* v, float* h, float* l) {
  split_k<<<256, 256>>>(n, v, h, l);
  return (int)cudaDeviceSynchronize();
}
extern "C" int join(int64_t n, const float* h, const float* l, double* v) {
  join_k<<<256, 256>>>(n, h, l, v);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1807_00086_gb300 import build
    d = tmp_path_factory.mktemp("pairs")
    (d / "pairs.cu").write_text(SOURCE)
    csrc = pathlib.Path(build.__file__).resolve().parent / "csrc"
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", str(csrc),
                    str(d / "pairs.cu"), "-o", str(d / "pairs.so")], check=True)
    return ctypes.CDLL(str(d / "pairs.so"))


def _doubles():
    rng = np.random.default_rng(17)
    n = 1 << 18
    sign = rng.integers(0, 2, n, dtype=np.uint64) << np.uint64(63)
    expo = rng.integers(0, 2047, n, dtype=np.uint64)                  # 2047: infinities, appended below
    edge = np.array([0, 1, 896, 897, 958, 959, 960, 961, 1022, 1023, 1139, 1140, 1141, 1150, 1151, 2046], dtype=np.uint64)
    expo[: n // 2] = rng.choice(np.concatenate([edge, np.arange(955, 1145, dtype=np.uint64)]), n // 2)
    head = rng.integers(0, 1 << 23, n, dtype=np.uint64)
    head[: n // 4] = rng.choice(np.array([0, 1, (1 << 23) - 1, (1 << 23) - 2], dtype=np.uint64), n // 4)
    tail = rng.integers(0, 1 << 29, n, dtype=np.uint64)
    half = 1 << 28
    tail[: n // 2 : 2] = rng.choice(np.array([0, 1, half - 1, half, half + 1, (1 << 29) - 1], dtype=np.uint64), n // 4)
    v = (sign | expo << np.uint64(52) | head << np.uint64(29) | tail).view(np.float64)
    return np.concatenate([v, [np.inf, -np.inf, 0.0, -0.0, 1.0, -1.0]])


def _pair(v):
    with np.errstate(all="ignore"):
        h = v.astype(np.float32)
        return h, (v - h.astype(np.float64)).astype(np.float32)


def _call(fn, n, args, outs):
    import torch
    torch.cuda.synchronize()
    assert fn(ctypes.c_int64(n), *[ctypes.c_void_p(t.data_ptr()) for t in (*args, *outs)]) == 0
    return [t.cpu().numpy() for t in outs]


def _same(a, b):
    nan = np.isnan(a) & np.isnan(b)
    return bool(np.all(nan | (a.view(np.uint32 if a.dtype == np.float32 else np.uint64)
                              == b.view(np.uint32 if b.dtype == np.float32 else np.uint64))))


def test_split(lib):
    import torch
    v = _doubles()
    h, l = _pair(v)
    dev = torch.tensor(v, device="cuda")
    gh, gl = _call(lib.split, v.size, [dev], [torch.empty(v.size, dtype=torch.float32, device="cuda") for _ in range(2)])
    assert _same(gh, h) and _same(gl, l)


def test_join(lib):
    import torch
    rng = np.random.default_rng(18)
    h, l = _pair(_doubles())
    keep = np.isfinite(h)
    h, l = h[keep], l[keep]
    # normalised pairs of every size of l: up to half a unit of the head's last place, also exactly that
    with np.errstate(all="ignore"):
        ulp = np.spacing(np.abs(h)) / np.float32(2)
        ulp = np.where(np.abs(h).view(np.uint32) & np.uint32((1 << 23) - 1), ulp, ulp / np.float32(2)).astype(np.float32)
        part = np.ldexp(rng.uniform(-1, 1, h.size), -rng.integers(0, 60, h.size)).astype(np.float32)
        part[::3] = rng.choice(np.array([-1, 1, 0, -0.5, 0.5], dtype=np.float32), part[::3].size)
        l2 = (ulp * part).astype(np.float32)
    h, l = np.concatenate([h, h]), np.concatenate([l, np.where(np.isfinite(l2), l2, np.float32(0))])
    want = h.astype(np.float64) + l.astype(np.float64)
    got, = _call(lib.join, h.size, [torch.tensor(h, device="cuda"), torch.tensor(l, device="cuda")],
                 [torch.empty(h.size, dtype=torch.float64, device="cuda")])
    assert _same(got, want)
