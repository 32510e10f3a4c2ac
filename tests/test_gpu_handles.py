"""Decode of caches whose cells fall into different kernel classes, and the memory of freed handles used again."""
import time

import pytest
import torch

import __graft_entry__ as entry

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    entry.build()
    import paper_2607_12550_b200 as pkg
    return pkg.load()


def _cache(layers, heads, T, seed, dtype=torch.float16):
    g = torch.Generator().manual_seed(seed)
    P = torch.randn(T, 24, generator=g) / torch.arange(1, 25)
    mk = lambda: (torch.einsum("tr,lhfr->lhtf", P, torch.randn(layers, heads, 128, 24, generator=g)) + 0.1 * torch.randn(layers, heads, T, 128, generator=g)).to(dtype).cuda()
    return mk(), mk()


# keys / values of r_t <= 128, above 128, and ranks the tensor-core kernels do not take, in one call
@pytest.mark.parametrize("plans", [
    [(64, 128, 4), (144, 128, 2), (160, 96, 8), (128, 128, 3)],
    [(48, 64, 2), (32, 128, 4), (50, 128, 4), (176, 128, 1)],
    [(144, 128, 4), (256, 128, 0), (256, 128, 4), (160, 128, 8)],
    [(16, 16, 1), (0, 0, 4), (64, 128, 2), (0, 0, 2)],
])
@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("dtype", [torch.float16, torch.float32])
def test_mixed_cells_decode_like_the_portable_kernels(B, plans, rope, dtype):
    K, V = _cache(3, 2, 384, 5)
    gs = [0, 2, 3]
    h = B.jolt_compress(K, V, gs, plans, B.default_options(seed=4))
    outs = []
    for mask in (0, 255, 255 - 128):
        prev = B.set_fast_path(mask)
        try:
            Ko, Vo = (torch.full(K.shape, float("nan"), dtype=dtype, device="cuda") for _ in range(2))
            for _ in range(2):
                if rope:
                    B.jolt_decompress_rope(h, Ko, Vo, gs, base=10000.0, pos0=17)
                else:
                    B.jolt_decompress(h, Ko, Vo, gs)
                B.check_status(h)
            outs.append((Ko.float(), Vo.float()))
        finally:
            B.set_fast_path(prev)
    # fp16 rounding of the output (twice where keys are rotated by the separate pass) and of the residual operand
    for a, b in zip(outs[0], outs[1]):
        assert float((a - b).norm() / a.norm()) <= 1e-3
    for a, b in zip(outs[1], outs[2]):
        assert float((a - b).norm() / a.norm()) <= 5e-4
    h.free()


def test_memory_of_freed_handles_is_used_again_in_order(B):
    """Handles made, decoded and freed in turn on two streams without a host wait between: every decode sees its own cache."""
    gs = [0, 2, 4]
    plans = [(64, 128, 4), (32, 128, 4)] * 2
    caches = [_cache(4, 4, 1024, 20 + i) for i in range(4)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    opts = B.default_options(seed=4)
    want = []
    for K, V in caches:
        h = B.jolt_compress(K, V, gs, plans, opts)
        o = torch.empty_like(K), torch.empty_like(V)
        B.jolt_decompress(h, *o, gs)
        torch.cuda.synchronize()
        want.append(o)
        h.free()
    got = []
    for i in range(12):
        st = streams[i % 2]
        h = B.jolt_compress(*caches[i % 4], gs, plans, opts, stream=st)
        o = torch.empty_like(caches[0][0]), torch.empty_like(caches[0][1])
        B.jolt_decompress(h, *o, gs, stream=st)
        h.free()                                   # the decode may still be running
        got.append(o)
    torch.cuda.synchronize()
    for i, o in enumerate(got):
        assert torch.equal(o[0], want[i % 4][0]) and torch.equal(o[1], want[i % 4][1]), i
    B.release_workspace()
    h = B.jolt_compress(*caches[1], gs, plans, opts)
    B.jolt_decompress(h, *got[0], gs)
    torch.cuda.synchronize()
    assert torch.equal(got[0][0], want[1][0])
    h.free()


def test_default_stream_decodes_then_another_stream(B):
    """Decodes that follow one another on the default stream leave no event behind; a call on another stream and the free after
    it still come after all of them."""
    g = torch.Generator().manual_seed(3)
    K, V = (torch.randn(2, 4, 1024, 128, generator=g).half().cuda() for _ in range(2))
    plan = [(32, 128, 4), (16, 64, 2)]
    opts = B.default_options(seed=1, power_iters=0)
    side = torch.cuda.Stream()
    h = B.jolt_compress(K, V, [0, 2], plan, opts)
    ref = [torch.empty_like(K), torch.empty_like(V)]
    B.jolt_decompress(h, *ref, [0, 2])
    torch.cuda.synchronize()
    for _ in range(4):
        outs = [[torch.zeros_like(K), torch.zeros_like(V)] for _ in range(4)]
        torch.cuda.synchronize()
        for o in outs[:3]:
            B.jolt_decompress(h, *o, [0, 2])
        B.jolt_decompress(h, *outs[3], [0, 2], stream=side)
        h.free()
        h2 = B.jolt_compress(-K, V.flip(0), [0, 2], plan, opts, stream=side)        # takes over the freed memory
        h2.free()
        h = B.jolt_compress(K, V, [0, 2], plan, opts)
        torch.cuda.synchronize()
        for o in outs:
            assert torch.equal(o[0], ref[0]) and torch.equal(o[1], ref[1])
    h.free()


def _held(stream, seconds=0.2):
    """The stream is busy for about that long (a bounded spin of SM clocks, up to 2 GHz)."""
    with torch.cuda.stream(stream):
        torch.cuda._sleep(int(seconds * 1.9e9))


def _after(stream):
    ev = torch.cuda.Event()
    ev.record(stream)
    return ev


def test_call_on_a_third_stream_waits_for_the_second(B):
    """h1 was decoded on the default stream, h2 is used on stream C (held back): a call that reads h1 on stream A uses the same
    shared memory as C's and comes after it, and both give what they give alone."""
    K, V = _cache(2, 4, 1024, 11)
    gs, plan = [0, 2], [(32, 128, 4), (16, 64, 2)]
    opts = B.default_options(seed=1, power_iters=0)
    h1, h2 = B.jolt_compress(K, V, gs, plan, opts), B.jolt_compress(V, K, gs, plan, opts)
    Q1, Q2 = (torch.randn(2, 4, 4, 128, generator=torch.Generator().manual_seed(i)).cuda() for i in (1, 2))
    o = torch.empty_like(K), torch.empty_like(V)
    want1, want2 = B.jolt_attend(h1, Q1), B.jolt_attend(h2, Q2)
    B.jolt_decompress_rope(h1, *o, gs, base=10000.0, pos0=3)
    torch.cuda.synchronize()
    want_rope = [t.clone() for t in o]
    C, A = torch.cuda.Stream(), torch.cuda.Stream()
    for call in ("attend", "rope"):
        B.jolt_decompress(h1, *o, gs)
        torch.cuda.synchronize()
        _held(C)
        got2 = B.jolt_attend(h2, Q2, stream=C)
        if call == "attend":
            got1 = B.jolt_attend(h1, Q1, stream=A)
        else:
            B.jolt_decompress_rope(h1, *o, gs, base=10000.0, pos0=3, stream=A)
        done = _after(A)
        time.sleep(0.03)
        assert not done.query()
        torch.cuda.synchronize()
        assert torch.equal(got2, want2)
        assert torch.equal(got1, want1) if call == "attend" else torch.equal(o[0], want_rope[0]) and torch.equal(o[1], want_rope[1])
    h1.free(); h2.free()


def test_calls_on_other_handles_come_after_default_stream_decodes_and_before_them(B):
    """Short decodes on the default stream leave no event behind, but a call on another stream comes after them whatever handle
    it reads or makes, and they come after the calls on other streams before them."""
    K, V = _cache(2, 4, 1024, 12)
    gs, plan = [0, 2], [(32, 128, 4), (16, 64, 2)]
    opts = B.default_options(seed=1, power_iters=0)
    h1, h2 = B.jolt_compress(K, V, gs, plan, opts), B.jolt_compress(V, K, gs, plan, opts)
    Q = torch.randn(2, 4, 4, 128, generator=torch.Generator().manual_seed(1)).cuda()
    o = torch.empty_like(K), torch.empty_like(V)
    B.jolt_attend(h2, Q)
    B.jolt_decompress(h2, *o, gs)
    torch.cuda.synchronize()
    C, default = torch.cuda.Stream(), torch.cuda.default_stream()
    for first, then in ((default, C), (C, default)):
        for call in ("attend", "decode"):
            torch.cuda.synchronize()
            B.jolt_decompress(h1, *o, gs)
            torch.cuda.synchronize()
            _held(first)
            B.jolt_decompress(h1, *o, gs, stream=None if first == default else C)
            st = None if then == default else C
            if call == "attend":
                B.jolt_attend(h2, Q, stream=st)
            else:
                B.jolt_decompress(h2, *o, gs, stream=st)
            done = _after(then)
            time.sleep(0.03)
            assert not done.query(), (call, then)
    torch.cuda.synchronize()
    h1.free(); h2.free()


def _free_bytes():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_is_given_back(B):
    """Blocks of freed handles are kept for the next ones, but not against the workspace: a call whose workspace only fits
    without them succeeds, and jolt_release_workspace returns everything to the driver."""
    K = torch.randn(4, 8, 32768, 128, device="cuda", dtype=torch.float16)
    V, gs, opts = K.flip(0).contiguous(), [0, 4], B.default_options(seed=1)
    Ko, Vo = torch.empty(K.shape, dtype=K.dtype), torch.empty(V.shape, dtype=V.dtype)       # host: the call stages 2 x 268 MB
    small = B.jolt_compress(K[:, :, :128], V[:, :, :128], gs, [(0, 0, 8)] * 2, opts)        # what the library allocates once
    B.jolt_decompress(small, K[:, :, :128], V[:, :, :128], gs)
    small.free()
    B.release_workspace()
    base = _free_bytes()
    hs = [B.jolt_compress(K, V, gs, [(0, 0, 8)] * 2, opts) for _ in range(3)]               # 285 MB each
    hs.pop().free()
    hs.pop().free()
    filler = torch.empty(_free_bytes() - (200 << 20), dtype=torch.uint8, device="cuda")
    B.jolt_decompress(hs[0], Ko, Vo, gs)
    del filler
    assert float((Ko.cuda().float() - K.float()).norm() / K.float().norm()) <= 1e-2
    hs[0].free()
    B.release_workspace()
    assert _free_bytes() >= base - (8 << 20)


@pytest.mark.parametrize("bits", [(0, 1), (2, 3), (4, 8)])
@pytest.mark.parametrize("T,tail", [(128, 0), (640, 0), (384, 60)])
def test_rotated_keys_of_the_persistent_kernel(B, bits, T, tail):
    """Every key width, one and several tiles a head, tiles dealt out in chunks: against the per-item kernel (bit 7 off)."""
    K, V = _cache(4, 3, T, 9)
    gs = [0, 2, 4]
    plans = [(32, 128, bits[0]), (48, 128, 4), (128, 96, bits[1]), (16, 128, 2)]
    h = B.jolt_compress(K, V, gs, plans, B.default_options(seed=2, power_iters=0))
    outs = []
    for mask in (255, 255 - 128):
        Ko, Vo = torch.empty_like(K), torch.empty_like(V)
        prev = B.set_fast_path(mask)
        B.set_test_decode_tail(tail, 2)
        try:
            B.jolt_decompress_rope(h, Ko, Vo, gs, base=10000.0, pos0=100)
            torch.cuda.synchronize()
        finally:
            B.set_fast_path(prev)
            B.set_test_decode_tail(0)
        outs.append((Ko, Vo))
    h.free()
    # the same operands, accumulators and rounding in both kernels
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


def _decode_both(B, h, like, gs, rope, tail=0):
    outs = []
    for mask in (255, 255 - 128):
        o = torch.empty_like(like), torch.empty_like(like)
        prev = B.set_fast_path(mask)
        B.set_test_decode_tail(tail, 2)
        try:
            for _ in range(4):                          # on one stream, without a host wait: what follows a decode sees all of it
                o[0].zero_(); o[1].zero_()
                if rope:
                    B.jolt_decompress_rope(h, *o, gs, base=10000.0, pos0=100)
                else:
                    B.jolt_decompress(h, *o, gs)
                outs.append((o[0].clone(), o[1].clone()))
            B.check_status(h)
        finally:
            B.set_fast_path(prev)
            B.set_test_decode_tail(0)
    return outs


# more than two tiles a CTA (640): one cell, half and all but one of them above r_t = 128, keys or values; widths with an
# instantiation of their own and without
@pytest.mark.parametrize("high", [(1,), (0, 5), (0, 2, 4, 6), (1, 3, 5, 7), (0, 1, 2, 4, 5, 6, 7), ()])
@pytest.mark.parametrize("bits", [(4, 8), (2, 3)])
@pytest.mark.parametrize("rope", [False, True])
def test_overlapping_launches_decode_like_one(B, high, bits, rope):
    K, V = _cache(4, 4, 2560, 31)
    gs = [0, 1, 2, 3, 4]
    plans = [(176 if c in high else 48 + 16 * (c % 3), 128, bits[c % 2]) for c in range(8)]
    h = B.jolt_compress(K, V, gs, plans, B.default_options(seed=2, power_iters=0))
    outs = _decode_both(B, h, K, gs, rope)
    h.free()
    for o in outs[1:]:
        assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])


# as test_rotated_keys_of_the_persistent_kernel, with enough tiles for the persistent kernel to take the rotation
@pytest.mark.parametrize("bits", [(0, 1), (2, 3), (4, 8)])
@pytest.mark.parametrize("heads,T,tail", [(40, 128, 0), (8, 640, 0), (13, 384, 60)])
def test_rotated_keys_of_many_tiles(B, bits, heads, T, tail):
    K, V = _cache(4, heads, T, 9)
    gs = [0, 2, 4]
    plans = [(32, 128, bits[0]), (48, 128, 4), (128, 96, bits[1]), (16, 128, 2)]
    h = B.jolt_compress(K, V, gs, plans, B.default_options(seed=2, power_iters=0))
    outs = _decode_both(B, h, K, gs, True, tail)
    h.free()
    for o in outs[1:]:
        assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])
