"""GPU parity of the block-sparse x block-sparse product and of the relative column index against the oracle, through the
C ABI: the product within the fp32-accumulation tolerance (bf16 or fp32 blocks), the index bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import ref
from paper_2407_09453_b200 import bsp, synth
from gpu_util import gpu_layer, make_case, rel_err

pytestmark = pytest.mark.gpu


def run_spgemm(seed, Oa, Ob, I, dtype, fa, fb):
    A = make_case(seed, Oa, I, 1, 1, dtype)
    B = make_case(seed + 10, Ob, I, 1, 1, dtype)
    ga = synth.random_gamma(seed + 1, Oa // 8, I // 8, int(round(fa * (Oa // 8) * (I // 8))))
    gb = synth.random_gamma(seed + 11, Ob // 8, I // 8, int(round(fb * (Ob // 8) * (I // 8))))
    la, lb = gpu_layer(A, ga, 8, 8, dtype), gpu_layer(B, gb, 8, 8, dtype)
    la.nnz, lb.nnz = int(ga.sum()), int(gb.sum())
    Cm = torch.full((Oa, Ob), -7.0, dtype=torch.float32, device="cuda")
    bsp.bsp_spgemm(la.wd, la.handle(), lb.wd, lb.handle(), Cm, la.ws)
    la.check()
    want = ref.spgemm(8, ref.compact(A, ga, 8, 8), ref.compact(B, gb, 8, 8))
    got = Cm.cpu().numpy()
    assert rel_err(got, want) <= 2e-5 if want.any() else np.array_equal(got, want)
    # blocks of C whose rows share no kept column are exactly zero
    share = (ga.astype(np.int32) @ gb.astype(np.int32).T) > 0
    full = np.repeat(np.repeat(share, 8, axis=0), 8, axis=1)
    assert np.all(got[~full] == 0.0)
    return got


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("fa,fb", [(0.5, 0.5), (0.0, 0.75), (0.9, 0.9), (1.0, 0.3)])
def test_spgemm_against_the_oracle(dtype, fa, fb):
    run_spgemm(901, 136, 200, 320, dtype, fa, fb)


def test_spgemm_many_rows_and_long_lists():
    """More rows of B than one sweep of the warps covers, and column lists longer than one 32-entry look-up."""
    run_spgemm(911, 64, 2048, 1024, "bf16", 0.5, 0.5)


@pytest.mark.parametrize("Oa,Ob,I,fa,fb", [
    (256, 512, 1024, 0.25, 0.25),        # 64 columns of C per CTA, reduction split over a cluster
    (264, 456, 1032, 0.3, 0.1),          # the same with ragged tiles and a last chunk of one block column
    (2040, 1032, 264, 0.1, 0.1),         # 128 columns, ragged, odd number of chunks
    (2048, 1800, 776, 0.05, 0.05),       # 256 columns, ragged
    (1840, 1672, 1040, 0.1, 0.1),        # pairs of CTAs, of the last of which one has no rows of A
    (1160, 2048, 2056, 0.2, 0.1),        # ... a row of blocks, and a last chunk of one block column
])
def test_spgemm_tensor_core_tiles(Oa, Ob, I, fa, fb):
    run_spgemm(931, Oa, Ob, I, "bf16", fa, fb)


@pytest.mark.parametrize("Oa,Ob,I,fa,fb", [
    (512, 1024, 520, 0.1, 0.1),          # a CTA an SM, a last chunk of one block column
    (1288, 1032, 264, 0.2, 0.0),         # ragged tiles of one block row and of one block column, two CTAs an SM
    (2048, 1800, 256, 0.8, 0.0),         # one operand sparse
])
def test_spgemm_fp32_tiles(Oa, Ob, I, fa, fb):
    run_spgemm(935, Oa, Ob, I, "f32", fa, fb)


@pytest.mark.parametrize("Oa,Ob,I,keep", [
    (512, 1024, 520, 0.9),               # a CTA an SM, a last chunk of one block column
    (1288, 1032, 264, 0.8),              # ragged tiles of one block row and of one block column, two CTAs an SM
    (1024, 1024, 1000, 0.5),
    (1608, 2000, 128, 0.6),
])
def test_spgemm_fp32_tiles_and_rows_give_the_same_bits(Oa, Ob, I, keep):
    """The count in the handle chooses between the two forms of fp32 operands: tiles for what the masks keep, rows for a count of one.
    Both add the terms of a sum in the same order, and neither multiplies a dropped block: with infinities and NaNs in blocks that
    the other operand dropped in the first, a middle and the last column, and in two that are kept."""
    g = torch.Generator(device="cuda")
    g.manual_seed(961)
    NBk = I // 8
    lays = []
    for k, O in enumerate((Oa, Ob)):
        W = torch.randn((O, 1, 1, I), device="cuda", generator=g)
        gamma = (torch.rand((O // 8, NBk), device="cuda", generator=g) < keep).to(torch.uint8)
        for col in (0, NBk // 2, NBk - 1):
            gamma[:, col] = k
            if k == 0:
                gamma[[0, O // 16, O // 8 - 1], col] = 1          # three rows of A keep the column
                W[[3, (O // 16) * 8 + 1], 0, 0, col * 8 + 2] = torch.tensor([float("inf"), float("nan")], device="cuda")
            else:
                gamma[1::2, col] = 0                             # every second row of B dropped it
        lay = bsp.SparseLayer(O, I, 1, 1, 8, 8, torch.float32)
        lay.compact(W, gamma)
        lay.nnz = int(gamma.sum())
        lay.check()
        lays.append((lay, gamma))
    (la, ga), (lb, gb) = lays
    got = []
    for nnz in ((la.nnz, lb.nnz), (1, 1)):
        la.nnz, lb.nnz = nnz
        Cm = torch.full((Oa, Ob), -7.0, device="cuda")
        bsp.bsp_spgemm(la.wd, la.handle(), lb.wd, lb.handle(), Cm, la.ws)
        la.check()
        got.append(Cm)
    finite = torch.isfinite(got[0])
    assert torch.equal(finite, torch.isfinite(got[1]))
    assert torch.equal(got[0][finite].view(torch.int32), got[1][finite].view(torch.int32))
    odd = torch.zeros((Oa // 8, Ob // 8), dtype=torch.bool, device="cuda")
    odd[0, 0::2] = odd[Oa // 16, 0::2] = True
    odd = odd.repeat_interleave(8, 0).repeat_interleave(8, 1)
    rows = torch.zeros(Oa, dtype=torch.bool, device="cuda")
    rows[[3, (Oa // 16) * 8 + 1]] = True
    assert torch.equal(~finite, odd & rows[:, None])


def test_spgemm_more_rows_than_a_grid_is_high():
    """1048577 block rows of A, one more than 65535 row tiles hold.  Few of them have blocks; the count in the handle says that all
    do, as for a mask that keeps everything (it chooses the kernel)."""
    NBa, NBb, NBk = 16 * 65535 + 1, 8, 64
    rows, cols = [0, 7, 524288, NBa - 1], [0, 5, 63]
    n = len(rows) * len(cols)
    row_ptr = torch.zeros(NBa + 1, dtype=torch.int32, device="cuda")
    for r in rows:
        row_ptr[r + 1:] += len(cols)
    col_idx = torch.tensor(cols * len(rows), dtype=torch.int32, device="cuda")
    payload = torch.randn((n, 8, 8), device="cuda").to(torch.bfloat16)
    lb = bsp.SparseLayer(NBb * 8, NBk * 8, 1, 1, 8, 8, torch.bfloat16)
    B = torch.randn((NBb * 8, NBk * 8), device="cuda").to(torch.bfloat16)
    lb.mask(B, 0)
    lb.compact(B)
    wa = bsp.wdesc(NBa * 8, NBk * 8, 1, 1, 8, 8, bsp.BF16)
    Cm = torch.full((NBa * 8, NBb * 8), -7.0, device="cuda")
    bsp.bsp_spgemm(wa, bsp.bcsr(row_ptr, col_idx, payload, None, NBa * NBk), lb.wd, lb.handle(), Cm, lb.ws)
    lb.check()
    for k, r in enumerate(rows):
        A = torch.zeros((8, NBk, 8), dtype=torch.float64, device="cuda")
        A[:, cols] = payload[k * len(cols):(k + 1) * len(cols)].double().permute(1, 0, 2)
        want = A.reshape(8, -1) @ B.double().T
        assert rel_err(Cm[r * 8:r * 8 + 8].cpu().numpy(), want.cpu().numpy()) <= 2e-5
        Cm[r * 8:r * 8 + 8] = 0.0
    assert not bool(Cm.any())


def test_spgemm_dropped_blocks_hide_non_finite_weights():
    """An infinite weight reaches the blocks of C whose row of B keeps its column, and no other."""
    O, I = 256, 512
    A, B = make_case(941, O, I, 1, 1, "bf16"), make_case(942, O, I, 1, 1, "bf16")
    ga, gb = synth.random_gamma(943, O // 8, I // 8, 200), synth.random_gamma(944, O // 8, I // 8, 200)
    ga[3, 10], gb[:, 10] = 1, 0
    gb[7, 10] = 1
    A[3 * 8 + 2, 0, 0, 10 * 8 + 1] = np.inf
    B[7 * 8:8 * 8, 0, 0, 10 * 8:11 * 8] = 1.0
    la, lb = gpu_layer(A, ga, 8, 8, "bf16"), gpu_layer(B, gb, 8, 8, "bf16")
    Cm = torch.empty((O, O), dtype=torch.float32, device="cuda")
    bsp.bsp_spgemm(la.wd, la.handle(), lb.wd, lb.handle(), Cm, la.ws)
    la.check()
    got = Cm.cpu().numpy()
    hit = np.zeros_like(got, dtype=bool)
    hit[3 * 8 + 2, 7 * 8:8 * 8] = True
    assert np.all(np.isposinf(got[hit])) and np.all(np.isfinite(got[~hit]))
    A[3 * 8 + 2, 0, 0, 10 * 8 + 1] = 0.0
    want = ref.spgemm(8, ref.compact(A, ga, 8, 8), ref.compact(B, gb, 8, 8))
    assert rel_err(np.where(hit, 0.0, got), np.where(hit, 0.0, want)) <= 2e-5


def test_spgemm_pairs_hide_non_finite_weights():
    """The same on pairs of CTAs, in the rows of either."""
    O, I = 2048, 1024
    g = torch.Generator(device="cuda")
    g.manual_seed(951)
    lays, full = [], []
    for k in range(2):
        W = torch.randn((O, 1, 1, I), device="cuda", generator=g).to(torch.bfloat16)
        gamma = (torch.rand((O // 8, I // 8), device="cuda", generator=g) < 0.6).to(torch.uint8)
        if k == 0:
            gamma[3, 10] = gamma[200, 10] = 1
            W[3 * 8 + 2, 0, 0, 10 * 8 + 1] = W[200 * 8 + 5, 0, 0, 10 * 8 + 4] = float("inf")
        else:
            gamma[:, 10] = 0
            gamma[7, 10] = gamma[150, 10] = 1
            W[:, 0, 0, 80:88] = W[:, 0, 0, 80:88].abs() + 1
        lay = bsp.SparseLayer(O, I, 1, 1, 8, 8, torch.bfloat16)
        lay.compact(W, gamma)
        lay.nnz = int(gamma.sum())
        lays.append(lay)
        keep = gamma.bool().repeat_interleave(8, 0).repeat_interleave(8, 1)
        full.append(torch.where(keep, W.reshape(O, I), torch.zeros((), dtype=W.dtype, device="cuda")).double())
    C = torch.empty((O, O), dtype=torch.float32, device="cuda")
    bsp.bsp_spgemm(lays[0].wd, lays[0].handle(), lays[1].wd, lays[1].handle(), C, lays[0].ws)
    lays[0].check()
    hit = torch.zeros_like(C, dtype=torch.bool)
    for r in (3 * 8 + 2, 200 * 8 + 5):
        for b in (7, 150):
            hit[r, b * 8:b * 8 + 8] = True
    assert bool(torch.isposinf(C[hit]).all()) and bool(torch.isfinite(C[~hit]).all())
    want = full[0].nan_to_num(posinf=0.0) @ full[1].T
    assert float((C.double() - want)[~hit].abs().max() / want.abs().max()) <= 2e-5


def test_spgemm_first_calls_from_several_threads():
    """The first calls of a process, at once and each on a stream of its own: every thread finds the device's limits in place."""
    code = """
import threading, torch
from paper_2407_09453_b200 import bsp
def layer(O, seed):
    torch.manual_seed(seed)
    lay = bsp.SparseLayer(O, 512, 1, 1, 8, 8, torch.bfloat16)
    W = torch.randn((O, 1, 1, 512), device="cuda").to(torch.bfloat16)
    lay.mask(W, lay.NBo * lay.NBi // 4)
    lay.compact(W)
    lay.check()
    return lay
jobs = [(layer(256, k), layer(256, k + 100), torch.empty((256, 256), device="cuda"), torch.cuda.Stream(), bsp.new_workspace(256)) for k in range(8)]
torch.cuda.synchronize()
gate, errors = threading.Barrier(8), []
def run(a, b, C, s, ws):
    gate.wait()
    try:
        bsp.bsp_spgemm(a.wd, a.handle(), b.wd, b.handle(), C, ws, s)
        bsp.bsp_check(ws, s)
    except Exception as e:
        errors.append(e)
ts = [threading.Thread(target=run, args=j) for j in jobs]
[t.start() for t in ts], [t.join() for t in ts]
assert not errors, errors
for a, b, C, s, ws in jobs:
    D = torch.empty_like(C)
    bsp.bsp_spgemm(a.wd, a.handle(), b.wd, b.handle(), D, ws)
    bsp.bsp_check(ws)
    assert torch.equal(C, D)
"""
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300, cwd=os.path.dirname(os.path.dirname(os.path.abspath(bsp.__file__))))


def test_spgemm_argument_errors():
    la = bsp.SparseLayer(64, 64, 1, 1, 8, 8, torch.bfloat16)
    lb = bsp.SparseLayer(64, 128, 1, 1, 8, 8, torch.bfloat16)
    Cm = torch.zeros((64, 64), dtype=torch.float32, device="cuda")
    with pytest.raises(bsp.BspError) as e:
        bsp.bsp_spgemm(la.wd, la.handle(), lb.wd, lb.handle(), Cm, la.ws)
    assert e.value.status == bsp.ERR_SHAPE                   # the reduction dimensions differ
    l4 = bsp.SparseLayer(64, 64, 1, 1, 4, 16, torch.bfloat16)
    with pytest.raises(bsp.BspError) as e:
        bsp.bsp_spgemm(la.wd, la.handle(), l4.wd, l4.handle(), Cm, la.ws)
    assert e.value.status == bsp.ERR_BLOCK


def test_relative_index_round_trip_bit_exact():
    W = make_case(921, 256, 1024, 1, 1, "bf16")
    gamma = synth.random_gamma(922, 32, 128, 2500)
    gamma[5, :] = 0                                          # an empty row
    lay = gpu_layer(W, gamma, 8, 8, "bf16")
    nnz = int(gamma.sum())
    rel = torch.full((nnz,), -1, dtype=torch.int32, device="cuda")
    back = torch.full((nnz,), -1, dtype=torch.int32, device="cuda")
    bsp.bsp_index_to_relative(32, lay.row_ptr, lay.col_idx, rel)
    bsp.bsp_index_from_relative(32, lay.row_ptr, rel, back)
    torch.cuda.synchronize()
    rp, ci, _ = ref.compact(W, gamma, 8, 8)
    assert np.array_equal(rel.cpu().numpy(), ref.index_to_relative(rp, ci))
    assert np.array_equal(back.cpu().numpy(), ci)
