"""The K-cycle's coefficients from the inner products of its launches, where the
second direction is close to the first and the sums that give it cancel: the
flat kernel and the fused one (an identity in sliced form) against the same
sums in extended precision.

a2 = (w2'.r)/(w2'.w2'), w2' = w2 - beta w1.  FP32 vectors: their products are
exact in float-float and 64 roundoffs of 2^-43 bound a tree of such adds, so
w2'.w2' is off by at most 64 2^-43 of the magnitudes that cancel in it, w2'.r
likewise.  FP64: the same with 2^-53 where the sums do not cancel (more than a
quarter is left), else with the magnitudes of w2' itself, whose elements carry a
roundoff of |w2| + |beta w1|."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import build  # noqa: E402

SRC = r"""
#include "kernels.cuh"
using namespace nbp;
template <typename T> static void flat(const void *y, const void *a, const void *b, long long n, double *kd) {
    k_kdots<T><<<kKdotBlocks, 256>>>((const T *)y, (const T *)a, (const T *)b, n, kd);
}
template <typename VT, typename T, int C, int P>
static void fused(const void *x, void *y, const void *a, const void *b, int n, const long long *ptr, const int *ci,
                  const void *val, double *part, double *kd) {
    SpmvArgs s = {};
    s.nbr = n; s.nslice = (n + C - 1) / C; s.sl_ptr = ptr; s.sl_ci = ci; s.val = val; s.x = x; s.y = y;
    const DotArgs q{a, b, part, kd};
    k_sell_dot<VT, T, C, P><<<grid_exact((long long)s.nslice * C * P), 256>>>(s, q);
}
extern "C" int dots(int form, int dbl, const void *x, void *y, const void *a, const void *b, int n, const long long *ptr,
                    const int *ci, const void *val, double *part, double *kd) {
    if (form == 0) dbl ? flat<double>(x, a, b, n, kd) : flat<float>(x, a, b, n, kd);
    else if (form == 1) dbl ? fused<double, double, 32, 1>(x, y, a, b, n, ptr, ci, val, part, kd)
                            : fused<float, float, 32, 1>(x, y, a, b, n, ptr, ci, val, part, kd);
    else dbl ? fused<double, double, 8, 4>(x, y, a, b, n, ptr, ci, val, part, kd)
             : fused<float, float, 8, 4>(x, y, a, b, n, ptr, ci, val, part, kd);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("kcycle")
    src, so = d / "k.cu", d / "k.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", build.INCLUDE, "-shared", "-o", str(so), str(src)],
                   check=True)
    return ctypes.CDLL(str(so))


def _p(t):
    return ctypes.c_void_p(t.data_ptr() if t is not None else None)


@pytest.mark.parametrize("form", [0, 1, 2])   # flat; fused: 32-row slices with one thread, 8-row with four
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_coefficients_of_close_directions(lib, form, dtype):
    dev = "cuda:0"
    C = (32, 32, 8)[form]
    for n in (1, 31, 255, 257, 4097, 70001):
        slots = (n + C - 1) // C * C
        ptr = torch.arange(0, slots + 1, C, dtype=torch.int64, device=dev)
        ci = torch.arange(slots, dtype=torch.int32, device=dev).clamp(max=n - 1)
        val = torch.zeros(slots, dtype=torch.float32 if dtype is np.float32 else torch.float64, device=dev)
        val[:n] = 1.0
        part = torch.zeros(4 * (slots * 4 // 256 + 1), dtype=torch.float64, device=dev)
        for eps in (1.0, 0.1, 1e-2, 1e-3) if n > 1 else (0.0,):
            rng = np.random.default_rng(n)
            w1 = rng.standard_normal(n).astype(dtype)
            w2 = (-0.7 * w1 + eps * rng.standard_normal(n)).astype(dtype)
            r = rng.standard_normal(n) + (w2 if n > 1 else 0) / max(eps, 1e-3)
            r = (r - (w1 @ r) / (w1 @ w1) * w1).astype(dtype)   # after the first step
            kd = torch.zeros(8 + 4 * 96, dtype=torch.float64, device=dev)
            kd[2] = 0.25
            t = {k: torch.as_tensor(v, device=dev) for k, v in dict(w1=w1, w2=w2, r=r).items()}
            y = torch.zeros_like(t["w1"])
            for x, a, b in ((t["w1"], t["r"], None), (t["w2"], t["w1"], t["r"])):
                assert lib.dots(form, int(dtype is np.float64), _p(x), _p(y), _p(a), _p(b), n, _p(ptr), _p(ci), _p(val), _p(part),
                                _p(kd)) == 0
                if form:
                    assert torch.equal(y, x)
            k = kd.cpu().numpy()
            L1, L2, R = (v.astype(np.longdouble) for v in (w1, w2, r))
            u, s11 = (2.0 ** -43 if dtype is np.float32 else 2.0 ** -53), np.sum(L1 * L1)
            assert abs(k[0] - s11) <= 64 * u * s11
            assert abs(k[1] - np.sum(L1 * R)) <= 64 * u * np.sum(abs(L1 * R))
            beta = np.sum(L2 * L1) / s11
            V = L2 - beta * L1
            ww, wr, s22 = np.sum(V * V), np.sum(V * R), np.sum(L2 * L2)
            if n == 1:   # nothing but rounding is left
                assert k[4] == 0.0 and k[3] == 0.25
                continue
            mag = abs(L2) + abs(beta * L1)
            if dtype is np.float64 and ww < 0.25 * s22:
                dww, dwr = 64 * u * np.sum(abs(V) * mag), 64 * u * np.sum(mag * abs(R))
            else:
                dww, dwr = 64 * u * 2 * s22, 64 * u * np.sum(mag * abs(R))
            a2 = wr / ww
            err = dwr / abs(wr) + dww / ww
            assert err < 0.1
            assert abs(k[4] - a2) <= 1.2 * err * abs(a2), (n, eps)
            assert abs(k[3] - (0.25 - a2 * beta)) <= 1.2 * err * abs(a2 * beta) + 64 * u * (s22 / s11) ** 0.5 * abs(a2) + 1e-15
