"""The compiled marshalling of the Python calls (csrc/bsp_call.cpp): every argument arrives as the C ABI declares it, wrong
kinds raise, and refused calls give the library's own status.  No call here reaches a launch."""
import numpy as np
import pytest
import torch

from paper_2407_09453_b200 import bsp, build


class Stream:
    cuda_stream = 0


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def buffers():
    return torch.zeros(64, dtype=torch.int32), torch.zeros(64, dtype=torch.bfloat16)


@pytest.mark.parametrize("nnz", [0, 1, 2 ** 31 + 5])
def test_handle_fields(nnz):
    i, p = buffers()
    h = bsp.bcsr(i, i[1:], None, torch.nn.Parameter(p), nnz)
    assert (h.row_ptr, h.col_idx, h.payload, h.packed, h.nnz) == (i.data_ptr(), i.data_ptr() + 4, None, p.data_ptr(), nnz)


def test_refused_calls_give_the_status_of_the_library():
    i, p = buffers()
    wd, h, xd = bsp.wdesc(64, 64, 1, 1, 8, 8, bsp.BF16), bsp.bcsr(i, i, p, p, 8), bsp.XDesc(1, 1, 1, 1, 1, 0, 0)
    x, s = torch.zeros(4, 64, dtype=torch.bfloat16), Stream()
    lay = bsp.SparseLayer(64, 64, 1, 1, 8, 8, torch.bfloat16, device="cpu")
    y = torch.zeros(4, 64)
    calls = [(bsp.ERR_NULL, lambda: bsp.bsp_gemm(wd, h, None, 4, None, y, bsp.F32, p, s)),
             (bsp.ERR_DTYPE, lambda: bsp.bsp_gemm(wd, h, x, 4, None, y, bsp.I32, p, s)),
             (bsp.ERR_DTYPE, lambda: bsp.bsp_conv2d(wd, h, xd, x, None, y, bsp.I32, p, s)),
             (bsp.ERR_NULL, lambda: bsp.bsp_mask(wd, None, 0, 0, 1, i, None, p, s)),
             (bsp.ERR_CAPACITY, lambda: bsp.bsp_mask(wd, x, 0, 0, 65, i, None, p, s)),
             (bsp.ERR_NULL, lambda: lay.gemm_q8(x, None, None, y.to(torch.int8), s)),
             (bsp.ERR_DTYPE, lambda: lay.gemm(x, None, y.to(torch.int32), s)),
             (bsp.ERR_SHAPE, lambda: lay.conv2d(x.view(4, 1, 1, 64), None, y, (0, 1), (0, 0), s)),
             (bsp.ERR_SHAPE, lambda: lay.conv2d(x.view(4, 1, 1, 64), None, y, (1, 1), (0, -1), s))]
    for want, call in calls:
        with pytest.raises(bsp.BspError) as e:
            call()
        assert e.value.status == want


@pytest.mark.parametrize("call", [lambda n, a: n.gemm(*a), lambda n, a: n.gemm(a[1], *a[1:]), lambda n, a: n.gemm(*a[:-1]),
                                  lambda n, a: n.gemm(*a[:3], 1.5, *a[4:]), lambda n, a: n.gemm(*a[:2], object(), *a[3:])])
def test_wrong_kinds_raise(call):
    i, p = buffers()
    args = [bsp.wdesc(64, 64, 1, 1, 8, 8, bsp.BF16), bsp.bcsr(i, i, p, p, 8), p, 4, None, p, bsp.F32, p, object()]
    with pytest.raises((TypeError, AttributeError)):
        call(bsp._native(), args)


@pytest.mark.parametrize("k,other", [(0, bytes(28)), (0, np.zeros(7, np.int32)), (1, bytes(40)), (2, 4096), (7, 4096), (3, np.int64(4)), (3, torch.tensor(4)),
                                     (6, np.int32(0))], ids=["bytes-wd", "array-wd", "bytes-handle", "address-x", "address-ws", "numpy-P", "tensor-P", "numpy-type"])
def test_only_the_declared_kinds_are_taken(k, other):
    """A descriptor is a ctypes structure, a buffer is an object with data_ptr() and no address, a count is an int: what merely
    has the bytes or converts is refused, as ctypes refuses it."""
    i, p = buffers()
    args = [bsp.wdesc(64, 64, 1, 1, 8, 8, bsp.BF16), bsp.bcsr(i, i, p, p, 8), p, 4, None, p, bsp.F32, p, Stream()]
    args[5] = p[1:]                              # (a misaligned output: a call that got through would be refused by the library)
    with pytest.raises(bsp.BspError):
        bsp.bsp_gemm(*args)
    args[k] = other
    with pytest.raises((TypeError, AttributeError)):
        bsp.bsp_gemm(*args)


@pytest.mark.parametrize("nnz", [np.int64(8), torch.tensor(8), 8.0])
def test_a_layer_takes_any_count(nnz):
    lay, x = bsp.SparseLayer(64, 64, 1, 1, 8, 8, torch.bfloat16, device="cpu"), torch.zeros(4, 64, dtype=torch.bfloat16)
    lay.nnz = nnz
    assert lay.handle().nnz == 8
    with pytest.raises(bsp.BspError):
        lay.gemm(x, None, torch.zeros(4, 64, dtype=torch.int32), Stream())


def test_input_shape_and_output_type():
    lay = bsp.SparseLayer(64, 64, 1, 1, 8, 8, torch.bfloat16, device="cpu")
    x = torch.zeros(4, 64, dtype=torch.bfloat16)
    with pytest.raises(ValueError):
        lay.conv2d(x, None, x, stream=Stream())
    with pytest.raises(KeyError):
        lay.gemm(x, None, x.double(), stream=Stream())


class Buffer:
    """What a layer's calls read of a buffer: a shape, a type and an address."""

    def __init__(self, t):
        self.t, self.shape, self.dtype = t, t.shape, t.dtype

    def data_ptr(self):
        return self.t.data_ptr()


def test_a_layer_takes_any_buffer_with_a_shape_and_a_type():
    lay, s = bsp.SparseLayer(64, 64, 1, 1, 8, 8, torch.bfloat16, device="cpu"), Stream()
    x, y = torch.zeros(4, 1, 1, 64, dtype=torch.bfloat16), torch.zeros(4, 64)
    x2 = x.view(4, 64)
    class Sub(torch.Tensor):
        pass
    for X in (Buffer(x), x.as_subclass(Sub)):
        for Y, want in ((Buffer(y[:0]), bsp.ERR_NULL), (Buffer(y.to(torch.int32)), bsp.ERR_DTYPE)):      # (an empty tensor has no address)
            with pytest.raises(bsp.BspError) as e:
                lay.conv2d(X, None, Y, stream=s)
            assert e.value.status == want
    for X in (Buffer(x2), x2.as_subclass(Sub)):
        with pytest.raises(bsp.BspError) as e:
            lay.gemm(X, None, Buffer(y.to(torch.int32)), s)
        assert e.value.status == bsp.ERR_DTYPE
    for X in (Buffer(x), x):
        with pytest.raises(bsp.BspError) as e:
            lay.conv2d_q8(X, None, None, Buffer(y.to(torch.int8)), stream=s)
        assert e.value.status == bsp.ERR_NULL
    for X in (x2[0].view(64), x.view(2, 2, 64)):                           # any rank: the first extent counts
        with pytest.raises(bsp.BspError) as e:
            lay.gemm_q8(X, None, None, y.to(torch.int8), s)
        assert e.value.status == bsp.ERR_NULL
    with pytest.raises(IndexError):
        lay.gemm(x.sum(), None, y, s)
    with pytest.raises(AttributeError):
        lay.gemm(None, None, y, s)


def test_a_marshalling_of_another_pytorch_is_built_again_and_not_loaded(monkeypatch, tmp_path):
    """It reads tensors in place: what was compiled against other headers must not be loaded, and a build replaces it whatever
    the times of the files say."""
    so = tmp_path / "_bspcall.so"
    so.write_bytes(b"")
    monkeypatch.setattr(build, "CALL", str(so))
    runs = []
    monkeypatch.setattr(build.subprocess, "check_call", lambda cmd: (runs.append(cmd), open(cmd[cmd.index("-o") + 1], "wb").close()))
    monkeypatch.setattr(bsp, "_calls", None)
    with pytest.raises(RuntimeError, match="build"):
        bsp._native()
    build.build_call()
    assert len(runs) == 1 and build.call_is_current()
    build.build_call()
    assert len(runs) == 1
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    with pytest.raises(RuntimeError, match="build"):
        bsp._native()
    build.build_call()
    assert len(runs) == 2 and build.call_is_current()
