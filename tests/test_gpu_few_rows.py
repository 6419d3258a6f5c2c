"""Batches small enough for the few-row kernels (weight-streaming GEMM with its K slices summed inside a cluster, cluster
shrink) at the sizes where their tiles and slices can go wrong: one row up to and beyond a row tile of 128, widths that leave
a half-filled column tile, contractions with an odd number of K-blocks, every rank, plans with per-adapter ranks, strides."""
import numpy as np
import pytest

from oracle import mlora_oracle as orc
from paper_2607_28848_b200 import binding as mb
from paper_2607_28848_b200 import synth
from paper_2607_28848_b200.runner import LayerRun, Session
from test_gpu_parity import TOL, assert_close, run_and_check
from test_gpu_variants import check_dropout

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sess():
    s = Session(0)
    yield s
    s.close()


# (rows, d_in, d_out): K slices 1 to 8; 320 = 2.5 column tiles; 576 and 1088 = an odd number of K-blocks; 300 and 700 rows =
# row tiles of 128 with a remainder; 16384 -> 64: one half-filled column tile in eight slices
SIZES = [(1, 576, 320), (16, 1024, 128), (17, 4096, 192), (64, 1088, 448), (65, 2048, 320), (128, 576, 1024), (129, 1088, 192),
         (255, 512, 320), (256, 4096, 256), (300, 576, 448), (700, 1024, 320), (40, 16384, 64)]


@pytest.mark.parametrize("rank", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("rows,d_in,d_out", SIZES)
def test_few_rows(sess, rows, d_in, d_out, rank):
    w = synth.random_workload(1000 + rows + rank, d_in, d_out, rank, 7, rows, max_seg=max(2, rows // 3), p_finetune=0.5)
    run_and_check(sess, w, synth.make_tensors(w), blocked=True)


@pytest.mark.parametrize("rank", [8, 64])
def test_every_row_its_own_adapter(sess, rank):
    """200 decode rows over 200 adapters: the low-rank operand is many times as deep as the contraction, an odd number of
    groups falls into each row tile and each slice."""
    segs = synth.segments_array([(i, 1, (7 * i) % 211, 0) for i in range(200)] + [(200, 30, 5, 1)])
    w = synth.Workload("own_adapters", 512, 320, rank, 211, "bf16", 230, segs, seed=rank)
    run_and_check(sess, w, synth.make_tensors(w), blocked=True)


def test_rows_of_the_base_model_only(sess):
    """No rank-r launch in front of the GEMM: it has to wait for whatever wrote its input."""
    segs = synth.segments_array([(0, 50, -1, 0)])
    w = synth.Workload("base_only", 1024, 320, 16, 3, "bf16", 50, segs, seed=3)
    t = synth.make_tensors(w, with_grad=False)
    ref = orc.forward(t["X"], t["W"], t["A_all"], t["B_all"], t["scale"], w.segments)["Y"]
    run = LayerRun(sess, w.dtype, t, w.segments, w.n_rows)
    try:
        X = run.X.clone()
        for _ in range(20):                         # the input is written by the launch right in front of the call
            run.X.zero_()
            run.X.add_(X)
            run.forward()
        assert run.status() == mb.MLORA_OK
        assert_close("Y", run.host(run.Y), ref, TOL["bf16"])
    finally:
        run.close()


@pytest.mark.parametrize("rows", [60, 230])
def test_ranked_plans(sess, rows):
    ranks = [16, 64, 32, 16, 48, 8, 16, 64, 24]
    w = synth.random_workload(1300 + rows, 1024, 320, 64, len(ranks), rows, max_seg=12, p_decode=0.5, p_finetune=0.4)
    t = synth.make_tensors(w)
    for a, r in enumerate(ranks):
        t["A_all"][a, r:] = 0
        t["B_all"][a, r:] = 0
    outs = []
    for ar in (None, ranks):
        run = LayerRun(sess, w.dtype, t, w.segments, w.n_rows, adapter_rank=ar)
        try:
            run.forward()
            run.backward()
            assert run.status() == mb.MLORA_OK
            outs.append([run.host(b) for b in (run.Y, run.u_save, run.dX, run.dA, run.dB)])
        finally:
            run.close()
    fwd = orc.forward(t["X"], t["W"], t["A_all"], t["B_all"], t["scale"], w.segments)
    assert_close("Y", outs[1][0], fwd["Y"], TOL["bf16"])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


def test_slices_give_the_same_bits_every_time(sess):
    """The cluster's sums are added in slice order, whoever is done first."""
    w = synth.random_workload(1400, 8192, 512, 16, 5, 90, max_seg=20, p_finetune=0.5)
    t = synth.make_tensors(w)
    run = LayerRun(sess, w.dtype, t, w.segments, w.n_rows)
    try:
        first = None
        for _ in range(5):
            run.forward()
            run.backward()
            got = [run.host(b) for b in (run.Y, run.u_save, run.dX, run.dA, run.dB)]
            if first is None:
                first = got
            assert all(np.array_equal(a, b) for a, b in zip(first, got))
        assert run.status() == mb.MLORA_OK
    finally:
        run.close()


@pytest.mark.parametrize("rows,d_in,d_out,rank", [(1, 33, 31, 4), (7, 97, 131, 5), (9, 256, 257, 8), (130, 511, 65, 16)])
def test_fp32_tiles_of_eight_rows(sess, rows, d_in, d_out, rank):
    """The fp32 product at row, column and contraction remainders of its 8 x 32 tiles and 32-deep blocks."""
    w = synth.random_workload(1500 + rows, d_in, d_out, rank, 3, rows, dtype="f32", max_seg=max(2, rows // 2), p_finetune=0.5)
    run_and_check(sess, w, synth.make_tensors(w))


@pytest.mark.parametrize("save_x", [True, False])
@pytest.mark.parametrize("rank", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("rows", [17, 130, 250])
def test_dropout(sess, rows, rank, save_x):
    """The few-row shrink with the dropout mask: above rank 32 several CTAs share a row, each masks it and one saves it.  Saved
    behind rows of an earlier step; without x_save the forward gives the same Y and u_save."""
    w = synth.random_workload(1600 + rows + rank, 1088, 448, rank, 4, rows, max_seg=max(2, rows // 3), p_finetune=0.7)
    t = synth.make_tensors(w)
    p, seed, base = 0.2, 2 ** 33 + rows, 7
    if save_x:
        check_dropout(sess, w, t, p, seed, base=base, cap=base + w.ft_rows + 5)
        return
    outs = []
    mb.mlora_set_dropout(sess.ctx, p, seed)
    try:
        for keep in (True, False):
            run = LayerRun(sess, w.dtype, t, w.segments, w.n_rows, save_row_base=base, save_x=keep)
            run.forward()
            assert run.status() == mb.MLORA_OK
            outs.append((run.host(run.Y), run.host(run.u_save)))
            run.close()
    finally:
        mb.mlora_set_dropout(sess.ctx, 0.0, 0)
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


# (rows, adapters, rank, d_in, d_out, launches of the shrink, of a reduction): 4096 -> 4096 with 256 adapters is 128 low-rank K-blocks
# in two slices of the few-row GEMM, the two-SM kernel runs them in four and adds these up (64 us against 75); 64 adapters of
# four rows at rank 128 leave the few-row shrink no CTAs along K, the tcgen05 shrink and its finish kernel take them (52 us
# against 110 for the call); the same rows of four adapters stay on the few-row kernels
@pytest.mark.parametrize("rows,adapters,rank,d_in,d_out,shrinks,reductions", [
    (256, 256, 32, 4096, 4096, 1, 1), (256, 64, 128, 8192, 1024, 2, 0), (256, 4, 128, 4096, 1024, 1, 0), (256, 4, 32, 4096, 4096, 1, 0)])
def test_batches_of_many_adapters_leave_the_few_row_kernels(sess, rows, adapters, rank, d_in, d_out, shrinks, reductions):
    n = rows // adapters
    segs = synth.segments_array([(i * n, n, i, 0) for i in range(adapters)])
    t = {"X": np.zeros((rows, d_in)), "W": np.zeros((d_in, d_out)), "A_all": np.zeros((adapters, rank, d_in)),
         "B_all": np.zeros((adapters, rank, d_out)), "scale": np.ones(adapters)}
    run = LayerRun(sess, "bf16", t, segs, rows)
    mb.mlora_profile_enable(sess.ctx, 8)
    try:
        run.forward()
        kinds = list(mb.mlora_profile_collect(sess.ctx)[0])
        assert run.status() == mb.MLORA_OK
        assert (kinds.count(0), kinds.count(6)) == (shrinks, reductions)
    finally:
        mb.mlora_profile_enable(sess.ctx, 0)
        run.close()
