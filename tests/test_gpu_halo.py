"""GPU parity of stride-1 layers with taps whose input channels fit one stage: the weights stay in shared memory and a tile's
activations arrive once, with the border that its taps reach."""
import numpy as np
import pytest
import torch

from oracle import ref
from paper_2407_09453_b200 import bsp, synth
from gpu_util import gpu_layer, make_bias, make_case, make_x
from test_gpu_product import run_conv_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,I", [("bf16", 8), ("bf16", 16), ("bf16", 24), ("bf16", 32), ("bf16", 40), ("bf16", 64),
                                     ("i8", 16), ("i8", 32), ("i8", 48), ("i8", 64), ("i8", 80), ("f32", 8), ("f32", 16), ("f32", 32)])
def test_input_channels_by_planes_and_rows(dtype, I):
    """One or two planes of 32-byte rows up to 64 bytes of channels, 128-byte rows above; channel tails inside a row."""
    run_conv_case(801, 64, I, 3, 3, 8, 8, dtype, (3, 19, 21, I), (1, 1), (1, 1))


@pytest.mark.parametrize("H,K,L,J,N,pad", [
    (3, 3, 7, 7, 9, (1, 1)),             # several whole images in a tile
    (3, 3, 5, 200, 2, (1, 1)),           # a row of the image in two tiles
    (5, 5, 30, 31, 2, (2, 2)),
    (1, 7, 17, 17, 3, (0, 3)),
    (7, 1, 17, 17, 3, (3, 0)),
    (2, 3, 12, 140, 1, (0, 0)),          # no padding, even taps
    (3, 3, 1, 1, 130, (1, 1)),           # one position an image
    (3, 3, 40, 40, 20, (2, 2)),          # more tiles than SMs, an output larger than the input
])
@pytest.mark.parametrize("dtype,out", [("bf16", "bf16"), ("i8", "i32")])
def test_taps_and_images(H, K, L, J, N, pad, dtype, out):
    run_conv_case(811, 64, 32, H, K, 8, 8, dtype, (N, L, J, 32), (1, 1), pad, out=out if dtype == "bf16" else "f32")


@pytest.mark.parametrize("H,K,L,J,N", [
    (3, 3, 16, 16, 3),                   # two tiles of 8 x 16 an image
    (3, 3, 31, 15, 2),                   # a ragged last column and row of tiles
    (5, 5, 16, 24, 40),                  # more tiles than SMs
    (1, 7, 16, 16, 2),
    (3, 3, 7, 7, 64),                    # two images of seven columns a tile, more tiles than images in one
])
@pytest.mark.parametrize("dtype,I", [("bf16", 16), ("bf16", 32), ("bf16", 64), ("i8", 64), ("i8", 128), ("f32", 32)])
def test_tiles_of_eight_columns(H, K, L, J, N, dtype, I):
    run_conv_case(815, 64, I, H, K, 8, 8, dtype, (N, L, J, I), (1, 1), (H // 2, K // 2))


@pytest.mark.parametrize("dtype,O", [("bf16", 48), ("bf16", 200), ("i8", 136), ("f32", 72)])
def test_channel_tiles(dtype, O):
    """A CTA keeps one channel tile: ragged last tiles, more position tiles than CTAs."""
    run_conv_case(821, O, 32, 3, 3, 8, 8, dtype, (8, 40, 40, 32), (1, 1), (1, 1))


@pytest.mark.parametrize("O,L", [(64, 440), (128, 440), (192, 250), (256, 440), (128, 147)])
def test_requantised_output_of_many_tiles(O, L):
    """Tiles of up to 128 channels use four accumulators in turn, wider ones two: one to eleven tiles a CTA."""
    W = make_case(841, O, 16, 1, 3, "i8")
    gamma = synth.random_gamma(842, O // 8, 2, O // 8)
    X = make_x(843, (1, L, 421, 16), "i8")
    b = make_bias(844, O, "i8")
    s = synth.uniform_int(845, (O,), 1, 12).astype(np.int32)
    lay = gpu_layer(W, gamma, 8, 8, "i8")
    Y = torch.full((1, L, 421, O), -7, dtype=torch.int8, device="cuda")
    lay.conv2d_q8(torch.from_numpy(X).cuda(), torch.from_numpy(b).cuda(), torch.from_numpy(s).cuda(), Y, (1, 1), (0, 1))
    lay.check()
    rp, ci, pl = ref.compact(W, gamma, 8, 8)
    acc = ref.conv2d(W.shape, 8, 8, rp, ci, pl, X, b, (1, 1), (0, 1))
    assert np.array_equal(Y.cpu().numpy().reshape(-1, O), ref.requant_i8(acc, s))


@pytest.mark.parametrize("O", [64, 128])
@pytest.mark.parametrize("case", ["plain", "shift 0", "shift 31", "bias"])
def test_requantised_output(O, case):
    """The short form of the rounding shift, and the cases that must leave it: a shift of 0 or 31, a bias near the rails."""
    W = make_case(831, O, 64, 3, 3, "i8")
    gamma = synth.random_gamma(832, O // 8, 8, O // 2)
    X = make_x(833, (3, 33, 29, 64), "i8")
    b = make_bias(834, O, "i8")
    s = synth.uniform_int(835, (O,), 1, 14).astype(np.int32)
    if case == "shift 0":
        s[::7] = 0
    elif case == "shift 31":
        s[::5] = 31
    elif case == "bias":
        b[::3], b[1::3] = (1 << 31) - 1 - (1 << 24), -(1 << 31) + (1 << 24)
        s[::2] = 25
    lay = gpu_layer(W, gamma, 8, 8, "i8")
    Y = torch.full((3, 33, 29, O), -7, dtype=torch.int8, device="cuda")
    lay.conv2d_q8(torch.from_numpy(X).cuda(), torch.from_numpy(b).cuda(), torch.from_numpy(s).cuda(), Y, (1, 1), (1, 1))
    lay.check()
    rp, ci, pl = ref.compact(W, gamma, 8, 8)
    acc = ref.conv2d(W.shape, 8, 8, rp, ci, pl, X, b, (1, 1), (1, 1))
    assert np.array_equal(Y.cpu().numpy().reshape(-1, O), ref.requant_i8(acc, s))


@pytest.mark.parametrize("N,L,J,I,O1,O2,H,K,relu", [
    (6, 56, 56, 64, 64, 256, 3, 3, 1),   # the weights of layer two stay in shared memory, several tiles a CTA
    (6, 40, 40, 32, 64, 1024, 3, 3, 0),  # ... and stream through their ring
    (9, 7, 7, 16, 128, 200, 3, 3, 1),    # several images a tile, one plane of 32-byte rows, clipped channels
    (2, 17, 33, 40, 72, 64, 1, 7, 1),    # two chunks of T with a tail
    (1, 1, 300, 64, 48, 48, 1, 3, 0),    # T and Y narrower than a chunk
    (12, 56, 56, 48, 64, 112, 3, 3, 1),  # two rounds a tile in the 8-bit form, many tiles a CTA
    (20, 101, 101, 48, 96, 96, 7, 1, 1), # ... whose second epilogue is late: two phases of layer two pass before it looks
    (20, 56, 56, 48, 96, 256, 3, 3, 0),  # ... three and four rounds a tile
    (20, 56, 56, 48, 96, 384, 3, 3, 0),
    (1, 11, 11, 64, 64, 928, 7, 1, 1),   # few tiles: a CTA for each 128 channels of layer two, the last of them clipped
    (24, 14, 14, 32, 64, 1024, 3, 3, 0), # ... for every three of eight, the last with one past the end
    (2, 22, 22, 192, 80, 176, 3, 3, 1),  # ... with layer one loaded tap by tap
    (60, 17, 17, 192, 64, 160, 3, 3, 0), # tiles of parts of several images
    (3, 16, 16, 64, 64, 256, 3, 3, 1),   # tiles of eight columns
    (120, 31, 15, 32, 72, 112, 5, 5, 1), # ... several a CTA, ragged
])
def test_pair_equals_the_two_calls(N, L, J, I, O1, O2, H, K, relu):
    for dtype in ("bf16", "i8"):
        W1, W2 = make_case(841, O1, I, H, K, dtype), make_case(842, O2, O1, 1, 1, dtype)
        ls = []
        for k, W in enumerate((W1, W2)):
            nb = (W.shape[0] // 8) * (W.shape[3] // 8)
            ls.append(gpu_layer(W, synth.random_gamma(843 + k, W.shape[0] // 8, W.shape[3] // 8, nb // 2), 8, 8, dtype))
        l1, l2 = ls
        X = torch.from_numpy(make_x(845, (N, L, J, I), dtype)).cuda()
        b1, b2 = (torch.from_numpy(make_bias(846 + k, O, dtype)).cuda() for k, O in enumerate((O1, O2)))
        pad, P = (H // 2, K // 2), (N, L, J)
        xd = bsp.XDesc(N, L, J, 1, 1, pad[0], pad[1])
        if dtype == "bf16":
            X = X.to(torch.bfloat16)
            T = torch.empty(P + (O1,), dtype=torch.bfloat16, device="cuda")
            l1.conv2d(X, b1, T, (1, 1), pad)
            if relu:
                T.clamp_(min=0)
            for ydt in (torch.bfloat16, torch.float32):
                Ya, Yb = (torch.full(P + (O2,), -7.0, dtype=ydt, device="cuda") for _ in range(2))
                l2.conv2d(T, b2, Ya)
                bsp.bsp_conv2d_chain(l1.wd, l1.handle(), l2.wd, l2.handle(), xd, X, b1, relu, b2, Yb, bsp.dtype_code(ydt), l1.ws)
                l1.check()
                assert torch.equal(Ya, Yb), (dtype, ydt)
            continue
        if I % 16 or O1 % 16 or O2 % 16:
            continue
        s1, s2 = (torch.from_numpy(synth.uniform_int(848 + k, (O,), 8, 13).astype(np.int32)).cuda() for k, O in enumerate((O1, O2)))
        for slow in (False, True):
            if slow:
                s1[0], s2[1] = 0, 31
            T = torch.empty(P + (O1,), dtype=torch.int8, device="cuda")
            l1.conv2d_q8(X, b1, s1, T, (1, 1), pad)
            if relu:
                T.clamp_(min=0)
            Ya, Yb = (torch.full(P + (O2,), -7, dtype=torch.int8, device="cuda") for _ in range(2))
            l2.conv2d_q8(T, b2, s2, Ya)
            bsp.bsp_conv2d_chain_q8(l1.wd, l1.handle(), l2.wd, l2.handle(), xd, X, b1, s1, relu, b2, s2, Yb, l1.ws)
            assert torch.equal(Ya, Yb), (dtype, slow)
            Za, Zb = (torch.full(P + (O2,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
            l2.conv2d(T, b2, Za)
            bsp.bsp_conv2d_chain_q8(l1.wd, l1.handle(), l2.wd, l2.handle(), xd, X, b1, s1, relu, b2, None, Zb, l1.ws)
            l1.check()
            assert torch.equal(Za, Zb), (dtype, slow)
