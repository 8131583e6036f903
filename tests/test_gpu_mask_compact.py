"""GPU parity: Gamma builder and compaction against the CPU oracle, bit for bit, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import ref
from paper_2407_09453_b200 import bsp, synth
from gpu_util import gpu_layer, gpu_mask, from_dev, make_case, to_dev, TORCH_DT

pytestmark = pytest.mark.gpu

SHAPES = [(8, 8), (4, 16), (16, 4)]


@pytest.mark.parametrize("dtype", ["bf16", "f32", "i8"])
@pytest.mark.parametrize("bo,bi", SHAPES)
@pytest.mark.parametrize("norm", [bsp.NORM_L2, bsp.NORM_L1])
def test_scores_and_gamma_bit_exact(dtype, bo, bi, norm):
    O, I, H, K = 96, 160, 3, 3
    W = make_case(101, O, I, H, K, dtype)
    NB = (O // bo) * (I // bi)
    want_s = ref.scores(W, bo, bi, norm)
    for n_zero in (NB // 2, 1, NB - 1):
        g, s, _, _ = gpu_mask(W, bo, bi, dtype, n_zero, norm)
        assert np.array_equal(s.view(np.uint64), want_s.view(np.uint64))      # identical bit patterns
        assert np.array_equal(g, ref.mask(want_s, n_zero))
        assert int((g == 0).sum()) == n_zero                                   # Eq. (2)


@pytest.mark.parametrize("dtype", ["bf16", "i8"])
def test_gamma_row_scope_and_extremes(dtype):
    bo = bi = 8
    O, I, H, K = 64, 256, 1, 1
    W = make_case(103, O, I, H, K, dtype)
    want_s = ref.scores(W, bo, bi)
    g, s, _, _ = gpu_mask(W, bo, bi, dtype, 9, scope=bsp.SCOPE_ROW)
    assert np.array_equal(g, ref.mask(want_s, 9, ref.SCOPE_ROW)) and np.all((g == 0).sum(axis=1) == 9)
    for n_zero in (0, 32):
        g, _, _, _ = gpu_mask(W, bo, bi, dtype, n_zero, scope=bsp.SCOPE_ROW)
        assert np.all(g == (1 if n_zero == 0 else 0))
    NB = g.size
    assert gpu_mask(W, bo, bi, dtype, 0)[0].all() and not gpu_mask(W, bo, bi, dtype, NB)[0].any()


def test_gamma_ties_broken_by_index():
    """int8 scores collide all the time; equal weights make every score equal."""
    bo = bi = 8
    W = np.full((64, 1, 1, 64), 5, dtype=np.int8)
    g, s, _, _ = gpu_mask(W, bo, bi, "i8", 23)
    assert np.array_equal(g.ravel(), np.r_[np.zeros(23, np.uint8), np.ones(41, np.uint8)])
    W = synth.uniform_int(107, (128, 1, 1, 256), -3, 3).astype(np.int8)        # few distinct scores
    want_s = ref.scores(W, bo, bi)
    assert len(np.unique(want_s)) < want_s.size // 2
    for n_zero in (100, 256, 301):
        g, s, _, _ = gpu_mask(W, bo, bi, "i8", n_zero)
        assert np.array_equal(g, ref.mask(want_s, n_zero))


def test_gamma_ties_in_a_layer_of_many_blocks():
    """8192 blocks with few distinct int8 scores: every CTA selects on all keys and counts the equal ones before its share of
    Gamma; equal keys are zeroed lowest index first."""
    bo = bi = 8
    W = synth.uniform_int(131, (512, 1, 1, 1024), -3, 3).astype(np.int8)
    want_s = ref.scores(W, bo, bi)
    assert len(np.unique(want_s)) < want_s.size // 8
    for n_zero in (1, 4097, want_s.size - 1):
        g, s, _, _ = gpu_mask(W, bo, bi, "i8", n_zero)
        assert np.array_equal(g, ref.mask(want_s, n_zero))
    g, _, _, _ = gpu_mask(W, bo, bi, "i8", 40, scope=bsp.SCOPE_ROW)
    assert np.array_equal(g, ref.mask(want_s, 40, ref.SCOPE_ROW))


def test_gamma_large_layer_many_select_passes():
    """More blocks than one pass of the selecting CTA covers (4096x2048 / 8x8 = 131072 blocks)."""
    bo = bi = 8
    W = synth.round_to_bf16(synth.normal(109, (2048, 1, 1, 1024), 1 / 32.0).astype(np.float32))
    want_s = ref.scores(W, bo, bi)
    g, s, _, _ = gpu_mask(W, bo, bi, "bf16", want_s.size // 2)
    assert np.array_equal(s.view(np.uint64), want_s.view(np.uint64))
    assert np.array_equal(g, ref.mask(want_s, want_s.size // 2))


@pytest.mark.parametrize("rows,cols,scope", [
    (19, 27, bsp.SCOPE_LAYER),           # 513 blocks: counted
    (47, 45, bsp.SCOPE_LAYER),           # 2115: the one-launch kernel selects by digits
    (64, 64, bsp.SCOPE_LAYER),           # 4096: the last
    (33, 128, bsp.SCOPE_ROW),            # rows of 128, 256, 257 and 600 in a layer of more than 4096 blocks
    (17, 256, bsp.SCOPE_ROW),
    (17, 257, bsp.SCOPE_ROW),
    (7, 600, bsp.SCOPE_ROW),
])
def test_select_within_one_cta(rows, cols, scope):
    """Distinct float scores, int8 scores with long runs of equal keys, and all keys equal."""
    seg = rows * cols if scope == bsp.SCOPE_LAYER else cols
    for dtype in ("bf16", "i8", "equal"):
        if dtype == "equal":
            W = np.full((rows * 8, 1, 1, cols * 8), 3, dtype=np.int8)
        elif dtype == "i8":
            W = synth.uniform_int(141, (rows * 8, 1, 1, cols * 8), -1, 1).astype(np.int8)
        else:
            W = make_case(142, rows * 8, cols * 8, 1, 1, "bf16")
        want = ref.scores(W, 8, 8)
        for n_zero in (1, seg // 3, seg // 2, seg - 1):
            g, _, _, _ = gpu_mask(W, 8, 8, "bf16" if dtype == "bf16" else "i8", n_zero, scope=scope)
            assert np.array_equal(g, ref.mask(want, n_zero, ref.SCOPE_ROW if scope == bsp.SCOPE_ROW else ref.SCOPE_LAYER)), (dtype, n_zero)


@pytest.mark.parametrize("rows,cols", [
    (17, 241),                           # 4097 blocks, the fewest that every CTA selects on for itself
    (128, 128),
    (145, 113),
    (129, 128),
    (128, 192),                          # 24576, the most
    (157, 157),                          # 24649
    (349, 73),                           # 25477 and
    (256, 256),                          # more: the cooperative select
    (256, 512),
    (24577, 1),                          # the fewest of it
])
def test_ties_across_the_ctas_of_a_select(rows, cols):
    """Layers whose threshold key is held by many blocks, in the shares of many CTAs: few distinct int8 scores, and one score for
    all blocks; the number to zero falls inside a run of equal keys, at its ends and one beside them."""
    NB = rows * cols
    for W in (synth.uniform_int(151, (rows * 8, 1, 1, cols * 8), -1, 1).astype(np.int8), np.full((rows * 8, 1, 1, cols * 8), -2, dtype=np.int8)):
        want = ref.scores(W, 8, 8)
        keys, counts = np.unique(want, return_counts=True)
        run = int(np.argmax(counts))
        below = int(counts[:run].sum())
        assert counts[run] > 100
        for n_zero in sorted({below + 1, below + int(counts[run]) // 2, below + int(counts[run]) - 1, below + int(counts[run]), 1, NB // 3, NB - 1} - {0, NB}):
            g, s, _, _ = gpu_mask(W, 8, 8, "i8", n_zero)
            assert np.array_equal(s, want)
            assert np.array_equal(g, ref.mask(want, n_zero)), n_zero


@pytest.mark.parametrize("rows,cols", [(64, 64), (128, 192), (149, 165), (256, 160)])      # 4096, 24576, 24585 and 40960 blocks
@pytest.mark.parametrize("what", ["infinite first", "mostly zero", "wide range", "two values"])
def test_select_of_uneven_scores(rows, cols, what):
    """Scores that leave most of a histogram's bins empty or lie outside of them, on each kind of select: an infinite weight among the
    blocks that the range is taken from, weights that were pruned before, forty octaves, two values."""
    W = make_case(161, rows * 8, cols * 8, 1, 1, "bf16")
    keep = synth.random_gamma(162, rows, cols, rows * cols // 4).repeat(8, 0).repeat(8, 1).reshape(W.shape)
    if what == "infinite first":
        W[0, 0, 0, 0] = np.inf
    elif what == "mostly zero":
        W = W * keep
    elif what == "wide range":
        W = synth.round_to_bf16((W * np.exp2(np.linspace(-20, 20, rows * 8)).reshape(-1, 1, 1, 1)).astype(np.float32))
    else:
        W = np.where(keep != 0, np.float32(0.5), np.float32(0.25))
    want = ref.scores(W, 8, 8)
    NB = rows * cols
    for n_zero in (1, NB // 10, NB // 2, 3 * NB // 4 + 1, NB - 1):
        g, s, _, _ = gpu_mask(W, 8, 8, "bf16", n_zero)
        assert np.array_equal(s, want)
        assert np.array_equal(g, ref.mask(want, n_zero)), n_zero


def by_key_bits(scores, n_zero, scope):
    """Gamma by the bits of the scores: what the selects order by, NaNs of either sign among them."""
    seg = scores.view(np.uint64).reshape(1, -1) if scope == bsp.SCOPE_LAYER else scores.view(np.uint64)
    g = np.ones(seg.shape, dtype=np.uint8)
    np.put_along_axis(g, np.argsort(seg, axis=1, kind="stable")[:, :n_zero], 0, axis=1)
    return g.reshape(scores.shape)


@pytest.mark.parametrize("rows,cols,scope", [
    (16, 16, bsp.SCOPE_LAYER),           # one launch, the last arriver selects
    (65, 64, bsp.SCOPE_LAYER),           # every CTA selects for itself
    (150, 165, bsp.SCOPE_LAYER),         # the cooperative select
    (8, 300, bsp.SCOPE_ROW),             # a row per CTA
    (129, 150, bsp.SCOPE_ROW),           # rows in a launch of their own
])
@pytest.mark.parametrize("norm", [bsp.NORM_L2, bsp.NORM_L1, bsp.NORM_VAR])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_select_of_scores_that_are_not_numbers(rows, cols, scope, norm, dtype):
    """NaNs of both signs and infinities among the weights, few and more than a warp ranks, with the threshold among ordinary scores and
    among theirs (the last bins of 64 bits)."""
    W0 = make_case(167, rows * 8, cols * 8, 1, 1, dtype)
    rng = np.random.default_rng(168)
    for n_odd in (1, 8, rows * cols // 3):
        W, bits = to_dev(W0, dtype), torch.int32 if dtype == "f32" else torch.int16
        raw = W.reshape(rows, 8, cols, 8)[:, 3, :, 5].contiguous().view(bits)
        odd = [0x7F800000, 0x7FC00000, -0x800000, -0x400000]          # inf, NaN, -inf and a NaN with its sign set
        values = torch.tensor([odd[k % 4] >> (0 if dtype == "f32" else 16) for k in range(n_odd)], dtype=bits, device="cuda")
        raw.view(-1)[torch.from_numpy(rng.choice(rows * cols, n_odd, replace=False)).cuda()] = values.flip(0)
        W.reshape(rows, 8, cols, 8)[:, 3, :, 5] = raw.view(W.dtype)
        lay = bsp.SparseLayer(rows * 8, cols * 8, 1, 1, 8, 8, TORCH_DT[dtype])
        sc = torch.empty((rows, cols), dtype=torch.float64, device="cuda")
        seg = rows * cols if scope == bsp.SCOPE_LAYER else cols
        for n_zero in sorted({1, seg // 2, seg - min(n_odd, 40), seg - 2, seg - 1}):
            for keep in (sc, None):
                lay.mask(W, n_zero, norm, scope, keep)
                lay.check()
                assert np.array_equal(from_dev(lay.gamma).reshape(rows, cols), by_key_bits(from_dev(sc), n_zero, scope)), (n_odd, n_zero)
        assert int((~torch.isfinite(sc)).sum()) == n_odd


@pytest.mark.parametrize("rows", [(5, 128), (5, 129), (5, 4096), (128, 200), (129, 200)])
def test_row_scope_in_one_and_two_launches(rows):
    """Rows that are ranked, selected by the CTA that scores them, and selected in a launch of their own; a few equal keys."""
    W = synth.uniform_int(163, (rows[0] * 8, 1, 1, rows[1] * 8), -3, 3).astype(np.int8)
    want = ref.scores(W, 8, 8)
    for n_zero in (0, 1, rows[1] // 2, rows[1] - 1, rows[1]):
        g, s, _, _ = gpu_mask(W, 8, 8, "i8", n_zero, scope=bsp.SCOPE_ROW)
        assert np.array_equal(s, want)
        assert np.array_equal(g, ref.mask(want, n_zero, ref.SCOPE_ROW)), n_zero


@pytest.mark.parametrize("NBo,NBi", [(9, 512), (17, 496), (16, 513), (8, 600), (40, 1024), (1030, 4), (7, 1040)])
def test_index_without_a_payload(NBo, NBi):
    """row_ptr and col_idx of layers of more than 4096 blocks that keep the packed form only: rows of one and several passes of 512
    entries, of a multiple of 16 and not, numbers of rows that are no multiple of eight, empty and full rows, Gamma at an odd
    address, and a capacity that ends inside a row."""
    W = make_case(153, NBo * 8, NBi * 8, 1, 1, "i8")
    gamma = synth.random_gamma(154, NBo, NBi, NBo * NBi // 2)
    gamma[NBo // 2], gamma[NBo - 1, :], gamma[0, NBi // 3:] = 0, 1, 0
    Wd = to_dev(W, "i8")
    for g in (gamma, np.zeros_like(gamma), np.ones_like(gamma)):
        rp, ci, _ = ref.compact(W, g, 8, 8)
        for capacity, offset in ((NBo * NBi, 0), (NBo * NBi, 1), (max(1, len(ci) - 3), 0)):
            lay = bsp.SparseLayer(NBo * 8, NBi * 8, 1, 1, 8, 8, torch.int8, capacity_blocks=capacity, canonical=False)
            big = torch.zeros(NBo * NBi + 16, dtype=torch.uint8, device="cuda")
            lay.gamma = big[offset:offset + NBo * NBi]
            col_idx = torch.full((NBo * NBi + 1,), -5, dtype=torch.int32, device="cuda")
            lay.col_idx = col_idx
            lay.row_ptr.fill_(-5)
            lay.compact(Wd, torch.from_numpy(np.ascontiguousarray(g)).cuda())
            if len(ci) > capacity:
                with pytest.raises(bsp.BspError) as e:
                    lay.check()
                assert e.value.status == bsp.ERR_CAPACITY
            else:
                lay.check()
            kept = min(len(ci), capacity)
            assert np.array_equal(from_dev(lay.row_ptr), rp)
            assert np.array_equal(from_dev(col_idx)[:kept], ci[:kept]) and bool((col_idx[kept:] == -5).all())


@pytest.mark.parametrize("dtype", ["bf16", "f32", "i8"])
@pytest.mark.parametrize("bo,bi", SHAPES)
def test_compact_bit_exact(dtype, bo, bi):
    O, I, H, K = 128, 96, 3, 2
    W = make_case(113, O, I, H, K, dtype)
    NBo, NBi = O // bo, I // bi
    for nz in ((NBo * NBi) // 2, 0, NBo * NBi, 5):
        gamma = synth.random_gamma(115 + nz, NBo, NBi, nz)
        lay = gpu_layer(W, gamma, bo, bi, dtype)
        rp, ci, pl = ref.compact(W, gamma, bo, bi)
        nnz = len(ci)
        assert np.array_equal(from_dev(lay.row_ptr), rp)
        assert np.array_equal(from_dev(lay.col_idx)[:nnz], ci)
        got = from_dev(lay.payload)[:pl.size].reshape(pl.shape)
        assert np.array_equal(got, pl if dtype != "bf16" else pl.astype(np.float32))
        assert bsp.bsp_compact_nnz(lay.wd, lay.gamma, lay.ws) == nnz


@pytest.mark.parametrize("dtype", ["bf16", "i8"])
@pytest.mark.parametrize("bo,bi", SHAPES)
def test_compact_more_blocks_than_the_single_launch_path_takes(dtype, bo, bi):
    """8192 blocks: Gamma is counted through L2 instead of from shared memory."""
    O, I, H, K = 512, 1024, 1, 1
    W = make_case(123, O, I, H, K, dtype)
    NBo, NBi = O // bo, I // bi
    assert NBo * NBi > 4096
    gamma = synth.random_gamma(125, NBo, NBi, (NBo * NBi) // 3)
    lay = gpu_layer(W, gamma, bo, bi, dtype)
    rp, ci, pl = ref.compact(W, gamma, bo, bi)
    assert np.array_equal(from_dev(lay.row_ptr), rp)
    assert np.array_equal(from_dev(lay.col_idx)[:len(ci)], ci)
    got = from_dev(lay.payload)[:pl.size].reshape(pl.shape)
    assert np.array_equal(got, pl if dtype != "bf16" else pl.astype(np.float32))


@pytest.mark.parametrize("dtype", ["bf16", "i8", "f32"])
def test_mask_and_compact_of_weights_at_an_odd_address(dtype):
    """W starting four bytes into an allocation: the 16-byte loads of the score and copy loops must give way to
    narrower ones, with the same bits out; an address that is not a multiple of four is refused."""
    bo = bi = 8
    O, I, H, K = 64, 72, 3, 3
    W = make_case(127, O, I, H, K, dtype)
    skip = {"bf16": 2, "i8": 4, "f32": 1}[dtype]
    big = torch.empty(W.size + 16, dtype=TORCH_DT[dtype], device="cuda")
    Wd = big[skip:skip + W.size].view(O, H, K, I)
    Wd.copy_(to_dev(W, dtype))
    assert Wd.data_ptr() % 16 == 4
    lay = bsp.SparseLayer(O, I, H, K, bo, bi, TORCH_DT[dtype])
    if dtype != "f32":
        odd = big[1:1 + W.size].view(O, H, K, I)
        with pytest.raises(bsp.BspError) as e:
            lay.mask(odd, 1)
        assert e.value.status == bsp.ERR_SHAPE
    sc = torch.empty(lay.NBo * lay.NBi, dtype=torch.int64 if dtype == "i8" else torch.float64, device="cuda")
    n_zero = lay.NBo * lay.NBi // 2
    lay.mask(Wd, n_zero, scores=sc)
    lay.compact(Wd)
    lay.check()
    want_s = ref.scores(W, bo, bi)
    assert np.array_equal(from_dev(sc).view(np.uint64), want_s.reshape(-1).view(np.uint64))
    g = ref.mask(want_s, n_zero)
    assert np.array_equal(from_dev(lay.gamma).reshape(g.shape), g)
    rp, ci, pl = ref.compact(W, g, bo, bi)
    assert np.array_equal(from_dev(lay.row_ptr), rp) and np.array_equal(from_dev(lay.col_idx)[:len(ci)], ci)
    got = from_dev(lay.payload)[:pl.size].reshape(pl.shape)
    assert np.array_equal(got, pl if dtype != "bf16" else pl.astype(np.float32))


def test_compact_capacity_overflow_is_latched():
    bo = bi = 8
    W = make_case(117, 64, 64, 1, 1, "bf16")
    lay = bsp.SparseLayer(64, 64, 1, 1, bo, bi, torch.bfloat16, capacity_blocks=10)
    gamma = synth.random_gamma(119, 8, 8, 32)
    lay.compact(to_dev(W, "bf16"), torch.from_numpy(gamma).cuda())
    with pytest.raises(bsp.BspError) as e:
        lay.check()
    assert e.value.status == bsp.ERR_CAPACITY
    lay.check()                                                                # cleared after being read


def test_mask_then_compact_round_trip_to_masked_dense():
    bo = bi = 8
    O, I, H, K = 256, 256, 3, 3
    W = make_case(121, O, I, H, K, "bf16")
    g, s, lay, Wd = gpu_mask(W, bo, bi, "bf16", 512)
    lay.compact(Wd)
    lay.check()
    rp, ci = from_dev(lay.row_ptr), from_dev(lay.col_idx)
    pl = from_dev(lay.payload).reshape(-1, bo, H, K, bi)
    back = np.zeros_like(W)
    for l in range(O // bo):
        for n in range(rp[l], rp[l + 1]):
            back[l * bo:(l + 1) * bo, :, :, ci[n] * bi:(ci[n] + 1) * bi] = pl[n]
    assert rp[-1] == 512 and np.array_equal(back, ref.apply_mask(W, g, bo, bi))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("bo,bi", SHAPES)
@pytest.mark.parametrize("H,K,O,I", [(3, 3, 96, 160), (1, 1, 256, 512), (1, 7, 32, 64)])
def test_variance_scores_and_gamma_bit_exact(dtype, bo, bi, H, K, O, I):
    """Variance importance (float weights): blocks get their own offsets so that the mean matters and the ranking
    differs from the L2 one; scores are compared as bit patterns (the kernel keeps the oracle's order of the sums and
    rounds the subtraction, the square and the addition one by one), Gamma bit for bit."""
    W = make_case(131, O, I, H, K, dtype)
    NBo, NBi = O // bo, I // bi
    shift = synth.normal(132, (NBo, NBi), 0.05).astype(np.float32)
    W = W + np.repeat(np.repeat(shift, bo, axis=0), bi, axis=1)[:, None, None, :]
    W = synth.round_to_bf16(W.astype(np.float32)) if dtype == "bf16" else W.astype(np.float32)
    want_s = ref.scores(W, bo, bi, ref.NORM_VAR)
    NB = NBo * NBi
    g, s, _, _ = gpu_mask(W, bo, bi, dtype, NB // 2, bsp.NORM_VAR)
    assert np.array_equal(s.view(np.uint64), want_s.view(np.uint64))
    want_g = ref.mask(want_s, NB // 2)
    assert np.array_equal(g, want_g)
    assert not np.array_equal(want_g, ref.mask(ref.scores(W, bo, bi, ref.NORM_L2), NB // 2))
    g_row, _, _, _ = gpu_mask(W, bo, bi, dtype, 3, bsp.NORM_VAR, bsp.SCOPE_ROW)
    assert np.array_equal(g_row, ref.mask(want_s, 3, ref.SCOPE_ROW))


def test_variance_of_int8_weights_is_refused():
    W = make_case(133, 64, 64, 1, 1, "i8")
    with pytest.raises(bsp.BspError) as e:
        gpu_mask(W, 8, 8, "i8", 4, bsp.NORM_VAR)
    assert e.value.status == bsp.ERR_DTYPE


def test_bounded_wait_runs_out_and_the_workspace_recovers():
    """A count of arrivals that cannot be this launch's: the arrival word in the workspace header is preset (by the host: the
    contract says it starts at zero) so that no CTA of the one-launch Gamma builder, where nobody waits, ever counts
    as the last arriver.  The kernel returns, bsp_check reports BSP_ERR_TIMEOUT once and clears the words of the
    counts, and the next call on the same workspace is bit-exact."""
    W = make_case(141, 128, 128, 3, 3, "bf16")
    lay = bsp.SparseLayer(128, 128, 3, 3, 8, 8, torch.bfloat16)
    Wd = to_dev(W, "bf16")
    lay.ws.view(torch.int32)[2] = 0x40000000          # arrivals so far: far more than any grid
    lay.mask(Wd, 128)
    with pytest.raises(bsp.BspError) as e:
        lay.check()
    assert e.value.status == bsp.ERR_TIMEOUT
    assert lay.ws.view(torch.int32)[:4].abs().sum().item() == 0      # status and barrier words cleared by bsp_check
    lay.check()
    lay.mask(Wd, 128)
    lay.check()
    want = ref.mask(ref.scores(W, 8, 8), 128)
    assert np.array_equal(from_dev(lay.gamma).reshape(16, 16), want)


@pytest.mark.parametrize("preset", [
    0xFFFFFFFF,                          # the count ends one short of the grid: every CTA's wait runs out
    0x40000000,                          # far more arrivals than any grid has: seen at once
])
def test_wait_of_the_cooperative_select_ends_and_the_workspace_recovers(preset):
    """A wait that nothing can satisfy ends by itself: the arrival word is preset as above, on a layer whose CTAs wait for one another
    (more than 24576 blocks)."""
    W = make_case(171, 150 * 8, 165 * 8, 1, 1, "bf16")
    want = ref.mask(ref.scores(W, 8, 8), 9000)
    lay = bsp.SparseLayer(150 * 8, 165 * 8, 1, 1, 8, 8, torch.bfloat16)
    Wd = to_dev(W, "bf16")
    lay.ws.view(torch.int32)[2] = preset - (1 << 32 if preset >= 1 << 31 else 0)
    lay.mask(Wd, 9000)
    with pytest.raises(bsp.BspError) as e:
        lay.check()
    assert e.value.status == bsp.ERR_TIMEOUT
    assert lay.ws.view(torch.int32)[:4].abs().sum().item() == 0
    lay.mask(Wd, 9000)
    lay.check()
    assert np.array_equal(from_dev(lay.gamma).reshape(150, 165), want)


@pytest.mark.parametrize("dtype,norm", [("bf16", bsp.NORM_L2), ("bf16", bsp.NORM_L1), ("bf16", bsp.NORM_VAR), ("f32", bsp.NORM_L2),
                                        ("f32", bsp.NORM_L1), ("f32", bsp.NORM_VAR), ("i8", bsp.NORM_L2), ("i8", bsp.NORM_L1)])
@pytest.mark.parametrize("rows,cols,H,bo,bi", [
    (157, 157, 3, 8, 8),                 # taps: b_o threads score a block
    (150, 165, 1, 8, 8),                 # one tap: a thread does, but for the variance
    (25, 1000, 2, 16, 4),
    (1001, 25, 1, 4, 16),
])
def test_cooperative_select_by_type_measure_and_block(rows, cols, H, bo, bi, dtype, norm):
    """Just above 24576 blocks, with the scores asked for and without (they stay on chip then)."""
    W = make_case(173, rows * bo, cols * bi, H, H, dtype)
    want = ref.scores(W, bo, bi, norm)
    NB = rows * cols
    for n_zero in (1, NB // 2, NB - 1):
        g, s, lay, Wd = gpu_mask(W, bo, bi, dtype, n_zero, norm)
        assert np.array_equal(s.view(np.uint64), want.view(np.uint64))
        assert np.array_equal(g, ref.mask(want, n_zero)), n_zero
        lay.gamma.fill_(7)
        lay.mask(Wd, n_zero, norm)
        lay.check()
        assert np.array_equal(from_dev(lay.gamma).reshape(rows, cols), g), n_zero


@pytest.mark.parametrize("dtype,norm,few", [("bf16", bsp.NORM_L2, False), ("bf16", bsp.NORM_VAR, False), ("i8", bsp.NORM_L2, False), ("i8", bsp.NORM_L1, True)])
def test_cooperative_select_of_slices_that_shared_memory_does_not_hold(dtype, norm, few):
    """1048576 blocks: a CTA's share is more than the 4096 keys that it keeps, and the keys are read again from the scores."""
    O = I = 8192
    g = torch.Generator()
    g.manual_seed(181)
    if dtype == "i8":
        lim = 1 if few else 127
        W = torch.randint(-lim, lim + 1, (O, 1, 1, I), generator=g, dtype=torch.int8).numpy()
    else:
        W = torch.randn((O, 1, 1, I), generator=g).bfloat16().float().numpy()
    want = ref.scores(W, 8, 8, norm)
    NB = want.size
    for n_zero in (1, NB // 2, NB - 1):
        g_, s, lay, Wd = gpu_mask(W, 8, 8, dtype, n_zero, norm)
        assert np.array_equal(s.view(np.uint64), want.view(np.uint64))
        assert np.array_equal(g_, ref.mask(want, n_zero)), n_zero
    lay.gamma.fill_(7)
    lay.mask(Wd, NB // 2, norm)
    lay.check()
    assert np.array_equal(from_dev(lay.gamma).reshape(want.shape), ref.mask(want, NB // 2))
