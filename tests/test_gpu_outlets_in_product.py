"""The rank-one factors of the A product, taken inside the product's blocks from
100,000 rows on where the outlets' rows lie close together, by a launch before
it otherwise: outlets in the last and in the first rows, blocks that hold
entries of four outlets that are not the first ones (one of them without
entries), of five, and outlets scattered over all rows; two and one threads
per row, FP64 and FP32.

The product of each row against the oracle's, in FP64: both sides sum at most
16 blocks of three terms and the outlets' terms, so they differ by at most
64 unit roundoffs of the sums of the magnitudes (the outlets' own inner
products, thousands of terms in another order on either side, are FP64 in both
forms: their roundoff is taken with their number of terms)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import Solver  # noqa: E402


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")


def _reversed(d):
    """The same system with its nodes numbered from the other end."""
    N, nnz = d["n_nodes"], len(d["col"])
    out = dict(d)
    out["rowptr"] = np.ascontiguousarray(nnz - d["rowptr"][::-1]).astype(np.int32)
    out["col"] = np.ascontiguousarray(N - 1 - d["col"][::-1]).astype(np.int32)
    for k in "ABCD":
        out[k] = np.ascontiguousarray(d[k][::-1])
    out["out_idx"] = (3 * (N - 1 - d["out_idx"] // 3) + d["out_idx"] % 3).astype(np.int32)
    out["b"] = np.concatenate([d["b"][:3 * N].reshape(N, 3)[::-1].reshape(-1), d["b"][3 * N:][::-1]])
    return out


def _outlets(d, lists, seed=9):
    """d with outlet k on the nodes lists[k], all three components each."""
    rng = np.random.default_rng(seed)
    idx = [np.add.outer(3 * np.asarray(nodes, dtype=np.int64), np.arange(3)).reshape(-1) for nodes in lists]
    out = dict(d)
    out["out_ptr"] = np.cumsum([0] + [len(i) for i in idx]).astype(np.int32)
    out["out_idx"] = np.concatenate(idx).astype(np.int32)
    out["out_val"] = rng.uniform(-1.0, 1.0, len(out["out_idx"]))
    out["r"] = 10.0 ** rng.uniform(2, 4, len(lists))
    out["n_out"] = len(lists)
    return out


def _forms(d):
    N = d["n_nodes"]
    at = 256 * (N // 2 // 256)   # a block of 256 rows in the middle, its 32-row groups too
    yield "last rows", d
    yield "first rows", _reversed(d)
    # outlets 1-4 meet in 32 rows (3 without entries), 0 and 5 lie far away
    yield "four of six", _outlets(d, [range(700), range(at, at + 40), range(at + 20, at + 60), [], range(at + 30, at + 31),
                                      range(N - 900, N)])
    yield "five in a block", _outlets(d, [range(at, at + 9), range(at + 9, at + 18), [at + 18], [at + 19], range(at + 20, at + 40)])
    yield "scattered", _outlets(d, [range(0, N, 29), range(1, N, 31)])


@pytest.mark.parametrize("n", [46, 58])
def test_every_form_against_the_oracle(n):
    d0 = synth.generate(synth.MeshSpec(n, n, n, Re=500.0, seed=4, R=(1e3, 1e4, 1e2)))
    N = d0["n_nodes"]
    assert 100000 < N and (N < 200000) == (n == 46)   # two threads per row, one
    x = np.random.default_rng(6).standard_normal(3 * N).astype(np.float32)
    for name, d in _forms(d0):
        y = oracle.Oracle(d).apply_A(x.astype(np.float64))
        mag = {k: np.abs(v) if k in ("A", "B", "C", "D", "out_val", "r") else v for k, v in d.items()}
        size = oracle.Oracle(mag).apply_A(np.abs(x).astype(np.float64))
        terms = 64 + np.diff(d["out_ptr"]).max()
        s = Solver(d, precision=1)
        s.setup()
        y64 = s.apply_A(_t(x.astype(np.float64)), 0).cpu().numpy()
        y32 = s.apply_A(_t(x), 1).cpu().numpy().astype(np.float64)
        assert (np.abs(y64 - y) <= terms * 2.0 ** -53 * size).all(), name
        assert (np.abs(y32 - y) <= (64 * 2.0 ** -24 + terms * 2.0 ** -53) * size).all(), name
        if name == "first rows":   # and inside a device-driven solve
            z, _ = s.solve(_t(d["b"]), rtol=1e-9)
            r = d["b"] - oracle.Oracle(d).apply_full(z.cpu().numpy())
            assert np.linalg.norm(r) <= 1.01e-9 * np.linalg.norm(d["b"])
        s.close()
