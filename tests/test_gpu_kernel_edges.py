"""Single kernels at the edges of their tiles, compiled from the library's headers: the narrow Cholesky and its reciprocal."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
U = 2.0 ** -53


@pytest.fixture(scope="module")
def E(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("edges") / "edges.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I",
                    os.path.join(HERE, "..", "paper_2607_12550_b200", "csrc"), "-o", so, os.path.join(HERE, "kernel_edges.cu")], check=True)
    torch.zeros(1, device="cuda")
    return ctypes.CDLL(so)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr() if t is not None else None)


def _cholesky(E, n, A=None, parts=None, dead_rel=1e-13):
    kp = (n + 15) // 16 * 16
    A, parts = (None if x is None else torch.from_numpy(x).cuda() for x in (A, parts))
    L = torch.full((n * n + 1,), float("nan"), dtype=torch.float64, device="cuda")
    hi, lo = (torch.full((kp, kp), float("nan"), dtype=torch.float16, device="cuda") for _ in range(2))
    info = torch.zeros(2, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert E.edge_cholesky(_ptr(A), _ptr(parts), 0 if parts is None else parts.shape[0], n, kp, ctypes.c_double(dead_rel), _ptr(L), _ptr(hi), _ptr(lo), _ptr(info)) == 0
    e, status = info.tolist()
    inv = (hi.double() + lo.double()).cpu().numpy()
    assert not inv[n:].any() and not inv[:, n:].any()
    return L[:n * n].view(n, n).t().cpu().numpy(), float(L[-1]), inv[:n, :n], e, status


def _check(G, L, exp2, inv, e, dead):
    """G = L L^T backward: each entry is a sum of up to n products rounded once each, and of the few roundings of a column's scaling
    (reciprocal and reciprocal root of the pivot, seven products of the block's unit factor).  L^-1 row by row from L by substitution,
    rounded to the fp16 pair (22 bits of each entry, subnormal below 2^-24)."""
    n = len(G)
    Lx = L.astype(np.longdouble)
    d = np.sqrt(np.diag(G)).astype(np.longdouble)
    assert not np.triu(L, 1).any() and not L[:, dead].any()
    assert np.all(np.abs(G - Lx @ Lx.T) <= (n + 16) * U * np.outer(d, d)), float((np.abs(G - Lx @ Lx.T) / np.outer(d, d)).max() / U)
    assert np.abs(L).max() < 2.0 ** exp2
    X = np.zeros((n, n), np.longdouble)      # L^-1 on the live directions
    for i in range(n):
        if i not in dead:
            X[i] = -(Lx[i, :i] @ X[:i]) / Lx[i, i]
            X[i, i] = 1 / Lx[i, i]
    bound = 2 * (n + 16) * U * (np.abs(X) @ np.abs(Lx) @ np.abs(X))
    scaled = np.abs(X) * np.longdouble(2.0) ** e
    assert 2.0 ** 9 * (1 - 1e-6) <= scaled.max() < 2.0 ** 10 * (1 + 1e-6)
    assert np.all(np.abs(inv - X * np.longdouble(2.0) ** e) <= 2.0 ** -21 * scaled + 2.0 ** -24 + bound * np.longdouble(2.0) ** e)


def _matrix(kind, n, seed):
    """Gram of a tall matrix of integers below 2^12: exact in fp64."""
    g = np.random.default_rng(seed)
    B = g.integers(-1000, 1001, (n + 40, n)).astype(np.float64)
    dead = []
    if kind == "graded":
        B = np.rint(B * 10.0 ** -np.linspace(0, 2, n))
    elif kind == "close":                    # every second column one entry away from its neighbour (another entry for each pair)
        rows = g.permutation(n + 40)
        for j in range(1, n, 2):
            B[:, j] = B[:, j - 1]
            B[rows[j // 2], j] += 1
    elif kind == "dead":                     # copies: in the first panel, in its own block, in the last one
        for j, of in ((1, 0), (n // 2, n // 2 - 1), (n - 1, 0)):
            if 0 <= of < j < n and j not in dead:
                B[:, j] = B[:, of]
                dead.append(j)
    return (B.T @ B).astype(np.float64), sorted(dead)


# sizes around a tile of eight, around the 128 rows of the Gram's first block, the largest; 1: a matrix of one entry
@pytest.mark.parametrize("kind", ["graded", "close", "dead"])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 17, 74, 127, 128, 129, 138, 151, 152])
def test_cholesky_and_inverse(E, kind, n):
    G, dead = _matrix(kind, n, n)
    L, exp2, inv, e, status = _cholesky(E, n, A=G)
    assert status == (2 if dead else 0)
    _check(G, L, exp2, inv, e, dead)


# partial Grams: fewer than the eight chunks of one round of loads, a remainder; only entries with row <= column exist
@pytest.mark.parametrize("n,chunks", [(8, 1), (26, 7), (74, 8), (129, 11), (152, 32)])
def test_cholesky_of_partial_grams(E, n, chunks):
    kp = (n + 15) // 16 * 16
    parts = np.full((chunks, kp, kp), np.nan, np.float32)
    for c in range(chunks):
        G, _ = _matrix("graded", n, 100 * n + c)
        parts[c, :n, :n] = np.where(np.triu(np.ones((n, n), bool)), G, np.nan)
    G = np.triu(parts[:, :n, :n].astype(np.longdouble).sum(0))
    G = G + np.triu(G, 1).T
    L, exp2, inv, e, status = _cholesky(E, n, parts=parts, dead_rel=5e-7)
    assert status == 0
    _check(G, L, exp2, inv, e, [])


def test_reciprocal_is_correctly_rounded(E):
    g = np.random.default_rng(3)
    m = 1 << 20
    d = np.ldexp(1.0 + g.random(m), g.integers(-990, 990, m))
    d[:4096] = np.ldexp(1.0 + g.integers(0, 2, 4096) * U * 2, g.integers(-100, 100, 4096))      # the smallest fractions
    ones = np.ldexp(2.0 - 2 * U, np.arange(-100, 100))                                          # all ones: to the last place
    x = torch.from_numpy(np.concatenate([d, ones])).cuda()
    out = torch.empty(2 * len(x), dtype=torch.float64, device="cuda")
    assert E.edge_rcp(_ptr(x), _ptr(out), len(x)) == 0
    y, ref = out.view(2, -1).cpu().numpy()
    assert (y[:m] == ref[:m]).all()
    assert np.all(np.abs(y - ref) <= 2 * U * np.abs(ref))


# staging and sums of the projected core: sixteen bytes (r_f a multiple of 8), pairs (even), single entries (odd); 21 rows end inside the second
# half of a block of 32, 72 in a third block.  Saved and loaded handles form it again.
@pytest.mark.parametrize("r_t", [7, 24])
@pytest.mark.parametrize("r_f", [1, 2, 8, 10, 12, 126, 127])
def test_projected_core(r_f, r_t):
    import __graft_entry__ as entry
    entry.build()
    import paper_2607_12550_b200 as pkg
    from tests.helpers import cell_from_handle, cell_view, decode_elementwise_bound
    from oracle import jolt_oracle as O
    B = pkg.load()
    cfg = pkg.synth.CacheConfig("t", 1, 1, 3, 256, n_terms=40, seed=r_f)
    K, V = pkg.synth.make_cache(cfg, device="cuda")
    r_t = min(r_t, 3 * r_f)                  # (no more than the rows of the projected unfolding)
    gs, plans = [0, 1], [(r_t, r_f, 0), (r_t, r_f, 4)]
    h = B.jolt_compress(K, V, gs, plans, B.default_options(seed=4, power_iters=1))
    h2 = B.jolt_deserialize(B.jolt_serialize(h))
    got = []
    for x in (h, h2):
        Ko, Vo = torch.empty(K.shape, device="cuda"), torch.empty(K.shape, device="cuda")
        B.jolt_decompress(x, Ko, Vo, gs)
        got.append((Ko, Vo))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    out = [t.cpu().numpy() for t in got[0]]
    for c, plan in enumerate(plans):
        oc = cell_from_handle(h, c, 3, 256, plan, 4, "f32")
        err = np.abs(cell_view(*out, gs, c) - O.decompress_cell(oc))
        assert np.all(err <= decode_elementwise_bound(oc, "f32")), float(err.max())
    h.free()
    h2.free()
