"""GPU parity of the position tiles at both ends of the range.  Layers with so few tiles that most SMs would idle: lower
tiles, up to 64 positions by MMAs with M = 64 (16 rows in each quarter of the tensor-memory lanes).  Layers of several waves:
tiles of parts of several images."""
import numpy as np
import pytest
import torch

from oracle import ref
from paper_2407_09453_b200 import synth
from gpu_util import from_dev, gpu_layer, make_bias, make_case, make_x, to_dev
from test_gpu_product import check, run_conv_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1, 15, 17, 33, 63, 64, 65, 129])
@pytest.mark.parametrize("dtype,out", [("bf16", "f32"), ("bf16", "bf16"), ("f32", "f32"), ("i8", "f32")])
def test_rows_and_channels(P, dtype, out):
    """Quarters of the tile that are empty or partly filled; a last channel tile of 24 channels."""
    run_conv_case(901, 1048, 512, 1, 1, 8, 8, dtype, (P, 1, 1, 512), (1, 1), (0, 0), out=out)


@pytest.mark.parametrize("O", [40, 48, 72, 1000])
@pytest.mark.parametrize("P", [7, 64])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("bias", [True, False])
def test_tiles_of_32_channels_end_where_y_does(O, P, dtype, bias):
    """bfloat16 output by rows of 64 bytes: a last tile of 8, 16 or 8 channels of 32, Y in the middle of memory that stays as it was."""
    I = 512
    W = make_case(905, O, I, 1, 1, dtype)
    gamma = synth.random_gamma(906, O // 8, I // 8, O * I // 128)
    X = make_x(907, (P, I), dtype)
    b = make_bias(908, O, dtype) if bias else None
    lay = gpu_layer(W, gamma, 8, 8, dtype)
    memory = torch.full((4096 + P * O + 4096,), -7, dtype=torch.bfloat16, device="cuda")
    Y = memory[4096:4096 + P * O].view(P, O)
    lay.gemm(to_dev(X, dtype), None if b is None else torch.from_numpy(b).cuda(), Y)
    lay.check()
    rp, ci, pl = ref.compact(W, gamma, 8, 8)
    check(from_dev(Y), ref.gemm(O, I, 8, 8, rp, ci, pl.reshape(-1, 8, 8), X, b), dtype, "bf16")
    assert bool((memory[:4096] == -7).all()) and bool((memory[4096 + P * O:] == -7).all())


@pytest.mark.parametrize("O,I,H,K,L,J,N,stride,pad", [
    (64, 176, 3, 3, 27, 27, 1, (1, 1), (1, 1)),      # two rows of the image a tile
    (128, 128, 3, 3, 28, 28, 1, (2, 2), (1, 1)),     # a stride
    (96, 320, 1, 7, 17, 70, 2, (1, 1), (0, 3)),      # a row of the image in two tiles
    (320, 512, 2, 2, 6, 6, 5, (1, 1), (0, 0)),       # several images a tile
])
@pytest.mark.parametrize("dtype", ["bf16", "i8", "f32"])
def test_taps_and_images(O, I, H, K, L, J, N, stride, pad, dtype):
    run_conv_case(911, O, I, H, K, 8, 8, dtype, (N, L, J, I), stride, pad)


@pytest.mark.parametrize("dtype,O,I,H,K,L,J,N,stride", [
    ("bf16", 64, 176, 3, 3, 28, 28, 60, (1, 1)),     # 4 x 4 positions of 8 images, a last tile of 4 images
    ("i8", 320, 144, 3, 3, 17, 17, 52, (1, 1)),      # 2 x 2 positions with clipped columns and rows
    ("f32", 264, 40, 3, 3, 7, 7, 150, (1, 1)),       # a row of 18 images
    ("bf16", 520, 72, 1, 1, 57, 57, 12, (2, 2)),     # strides
])
def test_tiles_of_parts_of_several_images(dtype, O, I, H, K, L, J, N, stride):
    run_conv_case(941, O, I, H, K, 8, 8, dtype, (N, L, J, I), stride, (H // 2, K // 2))


@pytest.mark.parametrize("P,O,I", [(64, 1008, 512), (200, 64, 1024), (5, 80, 640)])
def test_requantised_output(P, O, I):
    W = make_case(921, O, I, 1, 1, "i8")
    gamma = synth.random_gamma(922, O // 8, I // 8, (O // 8) * (I // 8) // 2)
    X, b = make_x(923, (P, 1, 1, I), "i8"), make_bias(924, O, "i8")
    s = synth.uniform_int(925, (O,), 0, 31).astype(np.int32)
    lay = gpu_layer(W, gamma, 8, 8, "i8")
    Y = torch.full((P, O), -7, dtype=torch.int8, device="cuda")
    lay.gemm_q8(torch.from_numpy(X).cuda().view(P, I), torch.from_numpy(b).cuda(), torch.from_numpy(s).cuda(), Y)
    lay.check()
    rp, ci, pl = ref.compact(W, gamma, 8, 8)
    acc = ref.conv2d(W.shape, 8, 8, rp, ci, pl, X, b, (1, 1), (0, 0))
    assert np.array_equal(Y.cpu().numpy(), ref.requant_i8(acc, s).reshape(P, O))
