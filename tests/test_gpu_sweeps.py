"""The tensor-core sweeps at the edges of their tiles, and calls that follow one another without a wait in between."""
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


def _cache(layers, heads, T, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    P = torch.randn(T, 200, generator=g, device="cuda") / torch.arange(1, 201, device="cuda") ** 0.7
    def make():
        x = torch.einsum("tr,lhfr->lhtf", P, torch.randn(layers, heads, 128, 200, generator=g, device="cuda"))
        return (x + 0.05 * torch.randn(layers, heads, T, 128, generator=g, device="cuda")).half()
    return make(), make()


def _factor(B, K, V, r_t, mask):
    prev = B.set_fast_path(mask)
    try:
        h = B.jolt_compress(K, V, [0, K.shape[0]], [(r_t, 128, 4)] * 2, B.default_options(seed=3, power_iters=1))
        out = []
        for cell, X in ((0, K), (1, V)):
            U = torch.from_numpy(h.component(cell, 8).reshape(X.shape[2], r_t).astype(np.float64)).cuda()
            A = X.reshape(-1, X.shape[2], 128).double().permute(1, 0, 2).reshape(X.shape[2], -1)
            out.append((float((U.T @ U - torch.eye(r_t, device="cuda")).abs().max()), float((U.T @ A).norm() ** 2 / A.norm() ** 2),
                        h.component(cell, 6)[:r_t].astype(np.float64)))
        h.free()
    finally:
        B.set_fast_path(prev)
    return out


# one and several items of two tiles, a ragged last tile of tokens, one pair of heads; column chunks of wide sketches; token segments
@pytest.mark.parametrize("layers,heads,T,r_t", [(1, 2, 128, 16), (1, 2, 384, 32), (3, 2, 640, 64), (1, 6, 1152, 112), (2, 4, 1024, 256), (1, 4, 4224, 64)])
def test_two_tile_sweeps_equal_single_ones(B, layers, heads, T, r_t):
    K, V = _cache(layers, heads, T, 12)
    for (orth, cap, sig), (_, cap1, sig1) in zip(_factor(B, K, V, r_t, 255), _factor(B, K, V, r_t, 255 - 64)):
        # single-precision product of two orthonormal bases; the same operands in the same order of K steps otherwise
        assert orth < 1e-5 and abs(cap - cap1) < 1e-6
        assert np.abs(sig - sig1).max() <= 1e-5 * sig1[0]


# a new sequence's plan, compress and decode, each pass enqueued while the one before it still runs: wide sketches, four cell groups on streams of their own
def test_passes_follow_one_another(B):
    K, V = _cache(8, 4, 8192, 5)
    gs, opts = [0, 2, 4, 6, 8], B.default_options(seed=9, power_iters=2)
    outs = []
    for _ in range(6):
        plan = B.jolt_plan(K, V, gs, K.numel() * 4 / 2.5, opts)[0]
        h = B.jolt_compress(K, V, gs, plan, opts)
        Ko, Vo = torch.empty_like(K), torch.empty_like(V)
        B.jolt_decompress(h, Ko, Vo, gs)
        h.free()
        outs.append((plan, Ko, Vo))
    torch.cuda.synchronize()
    assert max(p[0] for p in outs[0][0]) + 10 > 152          # (a wide sketch)
    for plan, Ko, Vo in outs[1:]:
        assert plan == outs[0][0] and torch.equal(Ko, outs[0][1]) and torch.equal(Vo, outs[0][2])
