"""The streaming attention kernel against the CUDA-core kernels (bit 0 of the kernel mask off) where its shapes change: four
heads a CTA or four chunks of one head, partial head quads and last chunks, ranks that are no multiple of its 32-column blocks,
every code width in both roles."""
import pytest
import torch

import __graft_entry__ as entry

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    entry.build()
    import paper_2607_12550_b200 as pkg
    return pkg.load()


# layers, first layer of the second group, heads, tokens, ranks (K, V) of both groups, bits (K, V) of both groups, queries
@pytest.mark.parametrize("L,g1,H,T,ranks,bits,nq", [
    (2, 1, 1, 128, (8, 8, 16, 40), (8, 1, 1, 8), 1),              # one head a cell: four chunks a CTA, three of them past the end
    (2, 1, 1, 640, (40, 8, 8, 72), (3, 4, 4, 3), 8),
    (2, 1, 2, 768, (0, 8, 32, 0), (2, 8, 8, 2), 4),
    (3, 2, 3, 384, (264, 136, 24, 0), (4, 8, 0, 4), 4),           # six and three heads: a partial quad
    (3, 2, 5, 256, (64, 96, 8, 248), (8, 2, 3, 1), 8),
    (5, 4, 4, 512, (128, 112, 96, 40), (1, 3, 8, 0), 5),
    (4, 2, 10, 9600, (16, 32, 24, 8), (4, 8, 2, 3), 4),           # more than one wave of CTAs: descriptors in the table arena
    (4, 2, 1, 40960, (16, 8, 8, 24), (8, 4, 3, 1), 6),
])
def test_stream_matches_cuda_core_path(B, L, g1, H, T, ranks, bits, nq):
    g = torch.Generator().manual_seed(L * 1000 + T)
    base = torch.randn(L, 1, T, 24, generator=g) @ torch.randn(L, H, 24, 128, generator=g)
    K, V = (base + 0.3 * torch.randn(L, H, T, 128, generator=g)).half().cuda(), (base.flip(0) + torch.randn(L, H, T, 128, generator=g)).half().cuda()
    plan = [(r, 128 if r else 0, b) for r, b in zip(ranks, bits)]
    h = B.jolt_compress(K, V, [0, g1, L], plan, B.default_options(seed=5, power_iters=0))
    Q = torch.randn(L, H, nq, 128, generator=g).cuda()
    Q[0, 0, 0] *= 8.0                                             # a sharp row: one chunk carries the weight
    out = B.jolt_attend(h, Q)
    prev = B.set_fast_path(14)
    try:
        ref = B.jolt_attend(h, Q)
        torch.cuda.synchronize()
    finally:
        B.set_fast_path(prev)
    h.free()
    assert torch.isfinite(out).all()
    # hi + lo fp16 operands (2^-22 each) give scores to 2^-21 of the largest, which is the relative error of a weight; the
    # values' own sums add a few 2^-22
    smax = torch.einsum("lhqf,lhtf->lhqt", Q, K.float()).abs().amax(-1) / 128 ** 0.5
    per_row = (out - ref).norm(dim=-1) / ref.norm(dim=-1)
    assert bool((per_row <= 5e-6 + 2.0 ** -21 * smax).all()), (per_row / smax).max()


@pytest.mark.parametrize("groups", [15, 16])                       # descriptors as a kernel argument / in the table arena
def test_many_layer_groups(B, groups):
    g = torch.Generator().manual_seed(groups)
    K, V = (torch.randn(groups, 2, 256, 128, generator=g).half().cuda() for _ in range(2))
    gs = list(range(groups + 1))
    h = B.jolt_compress(K, V, gs, [(16, 128, 8), (24, 128, 4)] * groups, B.default_options(seed=1, power_iters=0))
    Q = torch.randn(groups, 2, 4, 128, generator=g).cuda()
    out = B.jolt_attend(h, Q)
    prev = B.set_fast_path(14)                                     # (always the table)
    try:
        ref = B.jolt_attend(h, Q)
        torch.cuda.synchronize()
    finally:
        B.set_fast_path(prev)
    h.free()
    # scores of size one: 2^-21 of a weight, and the values' own sums
    assert float(((out - ref).norm(dim=-1) / ref.norm(dim=-1)).max()) <= 1e-5


# the second and third kernel of a call start while their predecessor runs: one head a CTA and four, descriptors by argument and table
@pytest.mark.parametrize("L,H,T,nq", [(2, 1, 512, 4), (4, 8, 1024, 8), (2, 16, 16384, 4)])
def test_calls_in_a_row_use_their_own_queries(B, L, H, T, nq):
    g = torch.Generator().manual_seed(T)
    K, V = (torch.randn(L, H, T, 128, generator=g).half().cuda() for _ in range(2))
    h = B.jolt_compress(K, V, [0, L], [(32, 128, 4), (48, 128, 8)], B.default_options(seed=3, power_iters=0))
    Q = [torch.randn(L, H, nq, 128, generator=g).cuda() * 2.0 ** i for i in range(5)]
    want = []
    for q in Q:
        want.append(B.jolt_attend(h, q))
        torch.cuda.synchronize()
    got = [B.jolt_attend(h, Q[i % 5]) for i in range(25)]
    torch.cuda.synchronize()
    h.free()
    for i, o in enumerate(got):
        assert torch.equal(o, want[i % 5]), i


def test_scratch_of_a_call(B):
    """What a call takes from the device: per head and 128-token chunk the partial values (ranks and features) of four queries, and
    nothing per token."""
    L, H, T, nq, r = 2, 4, 65536, 4, 64
    K, V = (torch.randn(L, H, T, 128, device="cuda").half() for _ in range(2))
    h = B.jolt_compress(K, V, [0, L], [(r, 128, 4), (r, 128, 4)], B.default_options(seed=3, power_iters=0))
    Q = torch.randn(L, H, nq, 128, device="cuda")
    B.jolt_attend(h, Q)
    del K, V
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    B.release_workspace()
    out = torch.empty_like(Q)
    before = torch.cuda.mem_get_info()[0]
    B._check(B.lib.jolt_attend(h.ptr, Q.data_ptr(), nq, 0.1, out.data_ptr(), None))
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    h.free()
    partial = L * H * (T // 128) * 4 * (r + 128 + 2) * 4
    assert taken <= partial * 9 // 8 + (6 << 20), (taken, partial)           # an eighth of headroom, tables, pages of 2 MB
