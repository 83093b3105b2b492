"""One thread per row in the sums of V threads (k_sell with V > 1, BF16 values)
against k_sellm with V threads: the same bits for every row width from none to
past two rounds of the chains, both slice heights and block sizes, every
epilogue that a batch runs so."""
import ctypes
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
using B = __nv_bfloat16;
template <int BS, int EPI, int C, int V> static void run(const SpmvArgs &a, int one) {
    if (one) k_sell<BS, B, float, EPI, false, C, C == 32 ? 2 : 1, V><<<grid_exact((long long)a.nslice * C), 256>>>(a);
    else k_sellm<BS, B, float, EPI, C, V><<<grid_exact((long long)a.nslice * C * V), 256>>>(a);
}
template <int BS, int EPI, int C> static void by_v(const SpmvArgs &a, int V, int one) {
    if (V == 2) run<BS, EPI, C, 2>(a, one);
    else if (V == 4) run<BS, EPI, C, 4>(a, one);
    else run<BS, EPI, C, 8>(a, one);
}
template <int BS, int C> static void by_epi(const SpmvArgs &a, int epi, int V, int one) {
    if (epi == EPI_RES) by_v<BS, EPI_RES, C>(a, V, one);
    else if (epi == EPI_CHEB) by_v<BS, EPI_CHEB, C>(a, V, one);
    else by_v<BS, EPI_SET, C>(a, V, one);
}
extern "C" int product(int bs, int C, int V, int epi, int one, int n, const long long *ptr, const int *ci, const void *val,
                       const void *x, const void *b, const void *dinv, void *d, void *y, int more) {
    SpmvArgs a = {};
    a.nbr = n; a.nslice = (n + C - 1) / C; a.sl_ptr = ptr; a.sl_ci = ci; a.val = val; a.x = x; a.b = b; a.dinv = dinv; a.d = d;
    a.y = a.xout = y; a.c1f = 0.3f; a.c2f = 0.7f; a.d_read = a.d_write = more;
    a.lr_rev = -1;
    if (bs == 3) C == 32 ? by_epi<3, 32>(a, epi, V, one) : by_epi<3, 8>(a, epi, V, one);
    else C == 32 ? by_epi<1, 32>(a, epi, V, one) : by_epi<1, 8>(a, epi, V, one);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("chains")
    src, so = d / "c.cu", d / "c.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", build.INCLUDE, "-shared", "-o", str(so), str(src)],
                   check=True)
    return ctypes.CDLL(str(so))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("bs", [1, 3])
@pytest.mark.parametrize("C", [8, 32])
def test_the_same_bits(lib, bs, C):
    dev = "cuda:0"
    g = torch.Generator(device=dev).manual_seed(10 * bs + C)
    rnd = lambda *n: torch.randn(*n, device=dev, generator=g)  # noqa: E731
    widths = np.concatenate([np.arange(0, 21), [40, 41, 3, 0, 16, 17]])   # of the slices
    n = C * len(widths) - 5                                               # a ragged last slice
    ptr = torch.as_tensor(np.concatenate([[0], np.cumsum(C * widths)]), dtype=torch.int64, device=dev)
    slots = int(ptr[-1])
    ci = torch.randint(0, n, (slots,), dtype=torch.int32, device=dev, generator=g)
    val = rnd(slots * bs * bs).to(torch.bfloat16)
    x, b, d0 = rnd(n * bs), rnd(n * bs), rnd(n * bs)
    dinv = rnd(n * bs * bs)
    for V in (2, 4, 8):
        for epi, more in ((0, 0), (3, 0), (4, 0), (4, 1)):
            if bs == 1 and epi == 0:
                continue
            got = []
            for one in (0, 1):
                y, d = torch.full_like(x, float("nan")), d0.clone()
                assert lib.product(bs, C, V, epi, one, n, _p(ptr), _p(ci), _p(val), _p(x), _p(b), _p(dinv), _p(d), _p(y), more) == 0
                got.append((y, d))
            assert torch.isfinite(got[0][0]).all()
            assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]), (V, epi, more)
