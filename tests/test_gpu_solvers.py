"""The tridiagonal eigen-solver against the Jacobi solvers (the portable path, bit 4 of the kernel mask off) and against
LAPACK, at the sizes where its kernels change: one CTA up to n = 160 (rows beyond 128 in shared memory), a cluster beyond."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    entry.build()
    import paper_2607_12550_b200 as pkg
    return pkg.load()


def _cache(T, m, rank, noise, seed):
    g = torch.Generator().manual_seed(seed)
    P = torch.randn(T, rank, generator=g) / torch.arange(1, rank + 1)
    X = torch.einsum("tr,mfr->mtf", P, torch.randn(m, 128, rank, generator=g)) + noise * torch.randn(m, T, 128, generator=g)
    return X.view(1, m, T, 128).float().cuda()


def _solve(B, K, V, plan, mask, **opt):
    prev = B.set_fast_path(mask)
    try:
        h = B.jolt_compress(K, V, [0, 1], plan, B.default_options(seed=3, power_iters=1, **opt))
        sig = [h.component(c, 6).astype(np.float64) for c in range(2)]
        UT = [h.component(c, 8).reshape(K.shape[2], -1).astype(np.float64) for c in range(2)]
        h.free()
    finally:
        B.set_fast_path(prev)
    return sig, UT


# sketch width = rank + 10: both sides of 32 (portable solver), 128 (register block), 160 (one CTA), 288 and 544 (rows per lane)
@pytest.mark.parametrize("r_t", [2, 22, 23, 54, 118, 119, 128, 150, 151, 278, 279, 534, 535])
def test_small_svd_matches_jacobi(B, r_t):
    T = 640
    K, V = _cache(T, 6, 40, 0.05, 1), _cache(T, 6, 700, 0.3, 2)
    plan = [(r_t, 128, 4), (r_t, 128, 4)]
    sig, UT = _solve(B, K, V, plan, 0)
    sig2, UT2 = _solve(B, K, V, plan, 16)
    for c in range(2):
        # both solvers return the fp32 rounding of an fp64 solution of the same matrix, up to the Jacobi threshold (1e-7 relative)
        assert np.abs(sig2[c] - sig[c]).max() <= 3e-6 * sig[c][0]
        assert np.abs(UT2[c].T @ UT2[c] - np.eye(r_t)).max() <= 1e-4        # single-precision products of two orthonormal factors
        gap = sig[c][r_t - 1] ** 2 - sig[c][r_t] ** 2
        if gap > 1e-3 * sig[c][0] ** 2:
            assert np.linalg.norm(UT[c] @ UT[c].T - UT2[c] @ UT2[c].T) <= 1e-3


@pytest.mark.parametrize("T", [128, 256, 640, 1024])
def test_exact_token_factor_matches_lapack(B, T):
    m = 2
    K, V = _cache(T, m, 24, 0.02, 5), _cache(T, m, 12, 0.0, 6)              # V: exactly rank 12, a null space of T - 12 (T x T)
    sig, UT = _solve(B, K, V, [(24, 128, 4), (16, 128, 4)], 255, token_mode=B.TOKEN_EXACT)
    for c, X in enumerate((K, V)):
        A = X[0].permute(1, 0, 2).reshape(T, -1).double().cpu().numpy()
        U, s, _ = np.linalg.svd(A, full_matrices=False)
        n = min(T, len(s))
        assert np.abs(sig[c][:n] ** 2 - s[:n] ** 2).max() <= 1e-6 * s[0] ** 2    # fp32 input products, fp64 solve
        r = 24 if c == 0 else 12
        assert np.linalg.norm(UT[c][:, :r] @ UT[c][:, :r].T - U[:, :r] @ U[:, :r].T) <= 1e-4
        assert np.abs(UT[c].T @ UT[c] - np.eye(UT[c].shape[1])).max() <= 1e-5   # a full basis, null directions included


# sketch width = rank + 10: one accumulator up to 152, blocks of 128 columns beyond (edges of the blocks), panels of 32 in the Cholesky
@pytest.mark.parametrize("r_t", [142, 143, 150, 246, 247, 256, 374, 375, 502, 503])
def test_wide_choleskyqr_matches_cuda_core_path(B, r_t):
    T = 768
    K, V = _cache(T, 6, 40, 0.05, 1).half(), _cache(T, 6, 700, 0.3, 2).half()
    K[:, :, :, 64:] = 0          # rank deficient beyond 384 directions: dead pivots in the Gram of the token basis
    plan = [(r_t // 16 * 16 if r_t > 374 else r_t, 128, 4), (r_t, 128, 4)]
    sig, UT = _solve(B, K, V, plan, 255 - 32)
    sig2, UT2 = _solve(B, K, V, plan, 255)
    for c in range(2):
        r = plan[c][0] if c else min(plan[c][0], 384)
        # the flat tail of a sketch with the width of the rank depends on the test matrix; compare down to the widest gap
        # both bases are single precision (hi + lo 22 bits, fp32 accumulation): 2^-20 of the square root of the contraction
        assert np.abs(UT2[c][:, :r].T @ UT2[c][:, :r] - np.eye(r)).max() <= 2e-5
        n = int((sig[c][4:r - 1] / sig[c][5:r]).argmax()) + 5                      # the widest relative gap behind the first
        assert np.abs(sig2[c] - sig[c])[:n].max() <= 1e-5 * sig[c][0]
        energy = (sig[c][:r] ** 2).sum()
        assert abs((sig2[c][:r] ** 2).sum() - energy) <= 1e-6 * energy             # no direction of the range is lost
        assert np.linalg.norm(UT[c][:, :n] @ UT[c][:, :n].T - UT2[c][:, :n] @ UT2[c][:, :n].T) <= 1e-3


def _graded_cache(T, m, seed):
    """A key cache (decaying terms, four outlier channels) and a value cache, as the synthetic caches are made."""
    g = torch.Generator().manual_seed(seed)
    out = []
    for alpha, sigma in ((1.0, 0.05), (0.6, 0.1)):
        n = 256
        q, _ = torch.linalg.qr(torch.randn(128, 128, generator=g, dtype=torch.float64))
        q = (q * 128 ** 0.5)[:, torch.arange(n) % 128]
        w = torch.arange(1, n + 1, dtype=torch.float64) ** -alpha
        p = torch.randn(T, n, generator=g, dtype=torch.float64)
        a = (1.0 + 0.1 * torch.randn(m, n, generator=g, dtype=torch.float64)) * w
        x = (p * a[:, None, :]) @ q.t() + sigma * torch.randn(m, T, 128, generator=g, dtype=torch.float64)
        if not out:
            x[:, :, [5, 37, 70, 101]] *= 10.0
        out.append(x.half().view(1, m, T, 128).cuda())
    return out


def _range_fp64(B, X, cell, seed, k, q):
    """Basis of the range finder with the library's own sketch, in fp64, in the order of the singular values."""
    _, m, T, _ = X.shape
    A = X[0].permute(1, 0, 2).reshape(T, m * 128).double()
    om = torch.from_numpy(B.sketch_host(seed, cell, 0, m * 128, k).astype(np.float64)).cuda().reshape(m * 128, k)
    Q = torch.linalg.qr(A @ om)[0]
    for _ in range(q):
        Q = torch.linalg.qr(A @ torch.linalg.qr(A.T @ Q)[0])[0]
    M = Q.T @ A
    return Q @ torch.linalg.eigh(M @ M.T)[1].flip(1)


def _distance(P, R):
    return max(float((P.T @ P).norm() ** 2 + (R.T @ R).norm() ** 2 - 2 * (P.T @ R).norm() ** 2), 0.0) ** 0.5


# the whole sketch is kept (no oversampling), so the span of the factor is the span of the basis: it has to be as close to the
# fp64 one as with the fp64 Gram and the CUDA-core solve (bit 5 off); what both have is the error of the sweeps
@pytest.mark.parametrize("T,m,k,q", [(2048, 8, 160, 1), (1024, 8, 272, 2), (2048, 8, 400, 1)])
def test_wide_basis_is_as_good_as_the_fp64_one(B, T, m, k, q):
    KV = _graded_cache(T, m, 7)
    got = []
    for mask in (255 - 32, 255):
        prev = B.set_fast_path(mask)
        try:
            h = B.jolt_compress(*KV, [0, 1], [(k, 128, 4)] * 2, B.default_options(seed=7, power_iters=q, oversample=0))
            got.append([torch.from_numpy(h.component(c, 8).reshape(T, k).astype(np.float64)).cuda() for c in (0, 1)])
            h.free()
        finally:
            B.set_fast_path(prev)
    for c in (0, 1):
        R = _range_fp64(B, KV[c], c, 7, k, q)
        # columns of unit length: the rounding of the fp32 factor and of the product with the small SVD's vectors, 2^-23 each
        assert float((got[1][c].T @ got[1][c] - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max()) <= 2.0 ** -22
        assert abs(float(got[1][c].norm() ** 2) / k - 1.0) <= 2.0 ** -24
        for n in (64, k):
            assert _distance(got[1][c][:, :n], R[:, :n]) <= 1.2 * _distance(got[0][c][:, :n], R[:, :n]), (c, n)


# sketch width = cap + 10: portable up to 32, Cholesky in shared memory to 152, in global memory to 288, tridiagonal beyond
@pytest.mark.parametrize("q_cap", [16, 32, 142, 144, 278, 279, 320])
def test_probe_values_give_the_portable_plan(B, q_cap):
    T = 640
    K, V = _cache(T, 6, 40, 0.05, 1).half(), _cache(T, 6, 700, 0.3, 2).half()
    raw = 2 * K.numel() * 2
    opts = B.default_options(seed=3, power_iters=1, q_cap=q_cap)
    got = []
    for mask in (255 - 16, 255):
        prev = B.set_fast_path(mask)
        try:
            sp = B.jolt_probe(K, V, [0, 1], 3.0, opts)
            got.append([sp.plan(raw / r, opts) for r in (2.0, 3.0, 5.0)])
            sp.free()
        finally:
            B.set_fast_path(prev)
    for (p, a), (q, b) in zip(*got):
        # values agree to some 1e-6 of the largest: a near-tie moves one cell by one step of the grid, and nothing else moves
        assert sum(x != y for x, y in zip(p, q)) <= 1, (p, q)
        assert all(abs(x[0] - y[0]) <= 16 and x[1] == y[1] and x[2] == y[2] for x, y in zip(p, q)), (p, q)


# one entry of the cache is no number: the spectra do not exist, and the call has to say so
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("dtype", [torch.float16, torch.float32])
@pytest.mark.parametrize("mask", [255, 255 - 16, 0])
def test_planning_a_cache_that_is_not_finite_fails(B, bad, dtype, mask):
    T = 512
    K, V = _cache(T, 4, 40, 0.05, 1).to(dtype), _cache(T, 4, 70, 0.3, 2).to(dtype)
    raw = 2 * K.numel() * 2
    prev = B.set_fast_path(mask)
    try:
        for opts in (B.default_options(seed=3, q_cap=64), B.default_options(seed=3, q_cap=300),
                     B.default_options(seed=3, token_mode=B.TOKEN_EXACT)):
            for X, at in ((K, (0, 0, 0, 0)), (V, (0, 3, T - 1, 77))):
                keep = X[at].clone()
                X[at] = bad
                for call in (lambda: B.jolt_plan(K, V, [0, 1], raw / 2, opts), lambda: B.jolt_probe(K, V, [0, 1], 2.0, opts)):
                    with pytest.raises(B.JoltError) as e:
                        call()
                    assert e.value.status == B.ENUMERIC
                X[at] = keep
            assert B.jolt_plan(K, V, [0, 1], raw / 2, opts)[1] <= raw / 2
    finally:
        B.set_fast_path(prev)
