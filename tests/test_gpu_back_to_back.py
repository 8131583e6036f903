"""Consecutive kernels of a stream overlap their starts.  Runs of calls in which each reads what the call before wrote, or
overwrites what it read, give what the same calls give one at a time, bit for bit."""
import ctypes as C

import pytest
import torch

from paper_2407_09453_b200 import bsp

pytestmark = pytest.mark.gpu


def randn(seed, shape, scale=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, device="cuda", generator=g) * scale


def randi8(seed, shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(-127, 128, shape, device="cuda", generator=g, dtype=torch.int8)


def compare(program, runs=4):
    """program(wait) -> tensors; `wait` is called between the calls and synchronises in the first run only.  The other runs
    queue up behind a kernel of some milliseconds, so that the GPU never waits for the host."""
    want = [t.clone() for t in program(torch.cuda.synchronize)]
    for _ in range(runs):
        torch.cuda._sleep(10_000_000)
        got = program(lambda: None)
        torch.cuda.synchronize()
        for k, (x, y) in enumerate(zip(got, want)):
            assert torch.equal(x, y), k


@pytest.mark.parametrize("N,L,C", [(1, 7, 16), (3, 14, 32), (2, 28, 64), (16, 56, 16)])
def test_small_int8_layers(N, L, C):
    """3x3 layers whose weights stay on chip: their CTAs are small enough to share an SM with those of the next call."""
    lay = bsp.SparseLayer(C, C, 3, 3, 8, 8, torch.int8)
    W = randi8(1, (C, 3, 3, C))
    lay.mask(W, lay.NBo * lay.NBi // 2)
    lay.compact(W)
    shift = torch.full((C,), 7 + (C * 9).bit_length() // 2, dtype=torch.int32, device="cuda")
    X = randi8(2, (N, L, L, C))

    def program(wait):
        a, b = X.clone(), torch.empty_like(X)
        for _ in range(40):
            lay.conv2d_q8(a, None, shift, b, (1, 1), (1, 1))
            wait()
            a, b = b, a
        lay.check()
        return a, b
    compare(program)


@pytest.mark.parametrize("dtype,N,L,C,mid,taps", [("i8", 2, 14, 32, 48, 3), ("i8", 4, 30, 192, 48, 1), ("bf16", 2, 28, 64, 64, 3), ("bf16", 3, 9, 24, 136, 3)])
def test_pairs(dtype, N, L, C, mid, taps):
    i8 = dtype == "i8"
    dt = torch.int8 if i8 else torch.bfloat16
    l1, l2 = bsp.SparseLayer(mid, C, taps, taps, 8, 8, dt), bsp.SparseLayer(C, mid, 1, 1, 8, 8, dt)
    W1 = randi8(3, (mid, taps, taps, C)) if i8 else randn(3, (mid, taps, taps, C), 1.4 / taps / C ** 0.5).to(dt)
    W2 = randi8(4, (C, 1, 1, mid)) if i8 else randn(4, (C, 1, 1, mid), 1.4 / mid ** 0.5).to(dt)
    for lay, W in ((l1, W1), (l2, W2)):
        lay.mask(W, lay.NBo * lay.NBi // 2)
        lay.compact(W)
    s1 = torch.full((mid,), 7 + (C * taps * taps).bit_length() // 2, dtype=torch.int32, device="cuda")
    s2 = torch.full((C,), 7 + mid.bit_length() // 2, dtype=torch.int32, device="cuda")
    X = randi8(5, (N, L, L, C)) if i8 else randn(5, (N, L, L, C)).to(dt)
    xd = bsp.XDesc(N, L, L, 1, 1, taps // 2, taps // 2)
    h1, h2 = l1.handle(), l2.handle()

    def program(wait):
        a, b = X.clone(), torch.empty_like(X)
        for _ in range(24):
            if i8:
                bsp.bsp_conv2d_chain_q8(l1.wd, h1, l2.wd, h2, xd, a, None, s1, 0, None, s2, b, l1.ws)
            else:
                bsp.bsp_conv2d_chain(l1.wd, h1, l2.wd, h2, xd, a, None, 0, None, b, bsp.BF16, l1.ws)
            wait()
            a, b = b, a
        l1.check()
        return a, b
    compare(program)


def test_products_of_different_kinds_take_turns():
    """A product, a pair and a sparse x sparse product by turns: each kernel's tensor memory is free when the next one takes it."""
    C = 64
    lay, l2 = bsp.SparseLayer(C, C, 3, 3, 8, 8, torch.bfloat16), bsp.SparseLayer(C, C, 1, 1, 8, 8, torch.bfloat16)
    for s, q in ((6, lay), (7, l2)):
        W = randn(s, (C, q.wd.H, q.wd.K, C), 1.4 / q.wd.H / C ** 0.5).to(torch.bfloat16)
        q.mask(W, q.NBo * q.NBi // 2)
        q.compact(W)
    sa, sb = bsp.SparseLayer(256, 1024, 1, 1, 8, 8, torch.bfloat16), bsp.SparseLayer(512, 1024, 1, 1, 8, 8, torch.bfloat16)
    for s, q in ((8, sa), (9, sb)):
        W = randn(s, (q.wd.O, 1, 1, 1024)).to(torch.bfloat16)
        q.mask(W, q.NBo * q.NBi // 4)
        q.compact(W)
    X = randn(10, (2, 14, 14, C)).to(torch.bfloat16)
    xd = bsp.XDesc(2, 14, 14, 1, 1, 1, 1)

    def program(wait):
        a, b, Cm = X.clone(), torch.empty_like(X), torch.empty((256, 512), device="cuda")
        for _ in range(12):
            lay.conv2d(a, None, b, (1, 1), (1, 1))
            wait()
            bsp.bsp_spgemm(sa.wd, sa.handle(), sb.wd, sb.handle(), Cm, sa.ws)
            wait()
            bsp.bsp_conv2d_chain(lay.wd, lay.handle(), l2.wd, l2.handle(), xd, b, None, 1, None, a, bsp.BF16, lay.ws)
            wait()
        lay.check(), sa.check()
        return a, b, Cm
    compare(program)


@pytest.mark.parametrize("scope", [bsp.SCOPE_LAYER, bsp.SCOPE_ROW])
@pytest.mark.parametrize("C,canonical", [(256, True), (1024, True), (1024, False), (1088, False)])
def test_set_up_of_weights_that_the_product_before_wrote(C, canonical, scope):
    """Mask, compaction and product by turns, the output of each product being the weights of the next layer: layers of 1024, 16384
    and 18496 blocks, ranked as a whole and by rows, with and without the canonical payload."""
    lay = bsp.SparseLayer(C, C, 1, 1, 8, 8, torch.bfloat16, canonical=canonical)
    W0, X = randn(11, (C, C), C ** -0.5).to(torch.bfloat16), randn(12, (C, C), C ** -0.5).to(torch.bfloat16)
    n_zero = lay.NBo * lay.NBi // 4 if scope == bsp.SCOPE_LAYER else lay.NBi // 4

    def program(wait):
        a, b = W0.clone(), torch.empty_like(W0)
        for _ in range(8):
            lay.mask(a, n_zero, scope=scope)
            wait()
            lay.compact(a)
            wait()
            lay.gemm(X, None, b)
            wait()
            a, b = b, a
        lay.check()
        return (a, b, lay.gamma, lay.row_ptr, lay.col_idx[:lay.nnz]) + ((lay.payload[:lay.nnz * 64],) if canonical else ())
    compare(program)


def test_sparse_operands_that_the_call_before_wrote():
    """fp32: a sparse x sparse product is masked, compacted and multiplied by itself again.  bfloat16: operands pruned again
    between the products, in the tensor-core form and the sparse form."""
    C = 256
    lay = bsp.SparseLayer(C, C, 1, 1, 8, 8, torch.float32)
    W0 = randn(13, (C, C), 0.5 * C ** -0.5)

    def square(wait):
        a, b = W0.clone(), torch.empty_like(W0)
        for _ in range(4):
            lay.mask(a, lay.NBo * lay.NBi // 2)
            wait()
            lay.compact(a)
            wait()
            bsp.bsp_spgemm(lay.wd, lay.handle(), lay.wd, lay.handle(), b, lay.ws)
            wait()
            a, b = b, a
        lay.check()
        return a, b
    compare(square)

    sa, sb = bsp.SparseLayer(512, 1024, 1, 1, 8, 8, torch.bfloat16), bsp.SparseLayer(256, 1024, 1, 1, 8, 8, torch.bfloat16)
    Ws = [(randn(20 + k, (512, 1024)).to(torch.bfloat16), randn(30 + k, (256, 1024)).to(torch.bfloat16)) for k in range(4)]

    def prune(wait):
        out = []
        for quarters in (1, 3):
            for A, B in Ws:
                for q, W in ((sa, A), (sb, B)):
                    q.mask(W, q.NBo * q.NBi * quarters // 4)
                    wait()
                    q.compact(W)
                    wait()
                out.append(torch.empty((512, 256), device="cuda"))
                bsp.bsp_spgemm(sa.wd, sa.handle(), sb.wd, sb.handle(), out[-1], sa.ws)
                wait()
        sa.check(), sb.check()
        return out
    compare(prune)


def test_loads_ahead_only_where_memory_is_mapped():
    """A header seen before the wait may be an old one of memory that held a larger buffer.  Loads go by it only where the allocation reaches
    as far as the descriptor's packed form does; the host decides, to the byte."""
    spans = bsp.lib()._ZN3bsp12packed_spansERK9bsp_wdescPKv
    spans.restype = C.c_bool
    wd = bsp.wdesc(256, 512, 3, 3, 8, 8, bsp.BF16)
    need = bsp.bsp_packed_bytes(wd, 0)
    cudart, base, size = C.CDLL("libcudart.so.12"), C.c_void_p(0), need + 4096
    torch.cuda.synchronize()
    assert cudart.cudaMalloc(C.byref(base), C.c_size_t(size)) == 0
    try:
        for offset, want in ((0, True), (4096, True), (4096 + 256, False), (size - 256, False)):
            assert spans(C.byref(wd), C.c_void_p(base.value + offset)) is want, offset
        assert not spans(C.byref(bsp.wdesc(264, 512, 3, 3, 8, 8, bsp.BF16)), base)
        assert not spans(C.byref(bsp.wdesc(1 << 19, 1 << 19, 1, 1, 8, 8, bsp.BF16)), base)
    finally:
        assert cudart.cudaFree(base) == 0
    assert not spans(C.byref(wd), C.c_void_p(256))
    for dt in (torch.float32, torch.bfloat16, torch.int8):       # (what programs have: tensors)
        for O, I, H in ((64, 64, 1), (512, 512, 3), (1000, 2048, 1)):
            lay = bsp.SparseLayer(O, I, H, H, 8, 8, dt)
            assert spans(C.byref(lay.wd), C.c_void_p(lay.packed.data_ptr()))


@pytest.mark.parametrize("H", [1, 3])
def test_packed_buffer_filled_anew_just_before_the_call(H):
    """A packed buffer that the call before fills for another descriptor (of the same size): whatever a product or a pair saw of it while
    that call still ran, it stores nothing and reports the buffer; filled again for its own, it gives what it gave."""
    C, P = 64, 64
    lays = [bsp.SparseLayer(C, C, H, H, bo, bi, torch.bfloat16) for bo, bi in ((8, 8), (4, 16))]
    W, X = randn(1, (C, H, H, C), 0.1).bfloat16(), randn(2, (P, 8, 8, C)).bfloat16()
    lay2 = bsp.SparseLayer(C, C, 1, 1, 8, 8, torch.bfloat16)
    W2 = randn(3, (C, 1, 1, C), 0.1).bfloat16()
    for lay, w in ((lays[0], W), (lays[1], W), (lay2, W2)):
        lay.mask(w, lay.NBo * lay.NBi // 4)
        lay.compact(w)
    a, b = lays
    shared, pad = a.packed, (H // 2, H // 2)
    xd = bsp.XDesc(P, 8, 8, 1, 1, pad[0], pad[1])

    def calls(Y, Z):
        a.conv2d(X, None, Y, (1, 1), pad)
        bsp.bsp_conv2d_chain(a.wd, a.handle(), lay2.wd, lay2.handle(), xd, X, None, 1, None, Z, bsp.F32, a.ws)

    want = [torch.empty((P, 8, 8, C), device="cuda") for _ in range(2)]
    calls(*want)
    a.check()
    for _ in range(20):
        got = [torch.full((P, 8, 8, C), -7.0, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        torch.cuda._sleep(1_000_000)
        bsp.bsp_compact(b.wd, W, b.gamma, b.row_ptr, b.col_idx, None, shared, b.capacity, b.ws)
        calls(*got)
        with pytest.raises(bsp.BspError) as e:
            a.check()
        assert e.value.status == bsp.ERR_INDEX
        assert all(bool((g == -7.0).all()) for g in got)
        torch.cuda._sleep(1_000_000)
        bsp.bsp_compact(a.wd, W, a.gamma, a.row_ptr, a.col_idx, None, shared, a.capacity, a.ws)
        calls(*got)
        a.check()
        assert all(torch.equal(g, w) for g, w in zip(got, want))
