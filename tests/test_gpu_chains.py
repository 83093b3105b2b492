"""Few threads per row in the sums of V threads (k_sell with V > 1: one, BF16
values; k_sellm with V > T) against k_sellm with V threads: the same bits for
every row width from none to past two rounds of the chains, both slice heights
and block sizes, every epilogue that a batch runs so, BF16 and FP32 values."""
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
// P threads in the sums of V (P == V: as it is); f32: FP32 values, unpaired
template <int BS, typename VT, int EPI, int C, int P, int V> static void run(const SpmvArgs &a) {
    constexpr bool B16 = std::is_same<VT, B>::value;
    constexpr int K = C == 32 && B16 ? 2 : 1;
    const unsigned grid = grid_exact((long long)a.nslice * C * P);
    if constexpr (P == 1 && B16) k_sell<BS, B, float, EPI, false, C, K, V><<<grid, 256>>>(a);
    else k_sellm<BS, VT, float, EPI, C, P, false, K, V><<<grid, 256>>>(a);
}
template <int BS, typename VT, int EPI, int C> static void by_v(const SpmvArgs &a, int V, int P) {
    if (V == 2) P == 2 ? run<BS, VT, EPI, C, 2, 2>(a) : run<BS, VT, EPI, C, 1, 2>(a);
    else if (V == 4) P == 4 ? run<BS, VT, EPI, C, 4, 4>(a) : P == 2 ? run<BS, VT, EPI, C, 2, 4>(a) : run<BS, VT, EPI, C, 1, 4>(a);
    else P == 8 ? run<BS, VT, EPI, C, 8, 8>(a) : P == 4 ? run<BS, VT, EPI, C, 4, 8>(a) : P == 2 ? run<BS, VT, EPI, C, 2, 8>(a) : run<BS, VT, EPI, C, 1, 8>(a);
}
template <int BS, typename VT, int C> static void by_epi(const SpmvArgs &a, int epi, int V, int P) {
    if (epi == EPI_RES) by_v<BS, VT, EPI_RES, C>(a, V, P);
    else if (epi == EPI_CHEB) by_v<BS, VT, EPI_CHEB, C>(a, V, P);
    else by_v<BS, VT, EPI_SET, C>(a, V, P);
}
extern "C" int product(int bs, int C, int V, int epi, int P, int f32, int n, const long long *ptr, const int *ci, const void *val,
                       const void *x, const void *b, const void *dinv, void *d, void *y, int more) {
    SpmvArgs a = {};
    a.nbr = n; a.nslice = (n + C - 1) / C; a.sl_ptr = ptr; a.sl_ci = ci; a.val = val; a.x = x; a.b = b; a.dinv = dinv; a.d = d;
    a.y = a.xout = y; a.c1f = 0.3f; a.c2f = 0.7f; a.d_read = a.d_write = more;
    a.lr_rev = -1;
    if (f32) C == 32 ? by_epi<3, float, 32>(a, epi, V, P) : by_epi<3, float, 8>(a, epi, V, P);
    else if (bs == 3) C == 32 ? by_epi<3, B, 32>(a, epi, V, P) : by_epi<3, B, 8>(a, epi, V, P);
    else C == 32 ? by_epi<1, B, 32>(a, epi, V, P) : by_epi<1, B, 8>(a, epi, V, P);
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


@pytest.mark.parametrize("bs,f32", [(1, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("C", [8, 32])
def test_the_same_bits(lib, bs, f32, C):
    dev = "cuda:0"
    g = torch.Generator(device=dev).manual_seed(10 * bs + C)
    rnd = lambda *n: torch.randn(*n, device=dev, generator=g)  # noqa: E731
    widths = np.concatenate([np.arange(0, 21), [40, 41, 3, 0, 16, 17]])   # of the slices
    n = C * len(widths) - 5                                               # a ragged last slice
    ptr = torch.as_tensor(np.concatenate([[0], np.cumsum(C * widths)]), dtype=torch.int64, device=dev)
    slots = int(ptr[-1])
    ci = torch.randint(0, n, (slots,), dtype=torch.int32, device=dev, generator=g)
    val = rnd(slots * bs * bs).to(torch.float32 if f32 else torch.bfloat16)
    x, b, d0 = rnd(n * bs), rnd(n * bs), rnd(n * bs)
    dinv = rnd(n * bs * bs)
    for V in (2, 4, 8):
        for epi, more in ((0, 0), (3, 0), (4, 0), (4, 1)):
            if bs == 1 and epi == 0:
                continue
            got = []
            for P in (V, *(p for p in (1, 2, 4) if p < V)):
                y, d = torch.full_like(x, float("nan")), d0.clone()
                assert lib.product(bs, C, V, epi, P, f32, n, _p(ptr), _p(ci), _p(val), _p(x), _p(b), _p(dinv), _p(d), _p(y), more) == 0
                got.append((y, d))
            assert torch.isfinite(got[0][0]).all()
            for y, d in got[1:]:
                assert torch.equal(got[0][0], y) and torch.equal(got[0][1], d), (V, epi, more)
