"""Small fp32 layers run in three launches instead of six: the same bits as the separate kernels (kernel variant 1 runs those), at
the remainders of the 8 x 32 tiles, ranks that are no multiple of the four or eight rows taken at a time, with a mask, with a
save base, without dX, accumulating, and with dX in the memory of x_save (which takes the separate launches)."""
import numpy as np
import pytest
import torch

from paper_2607_28848_b200 import binding as mb
from paper_2607_28848_b200 import synth
from paper_2607_28848_b200.runner import LayerRun, Session
from test_gpu_parity import run_and_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sess():
    s = Session(0)
    yield s
    s.close()


SIZES = [(1, 5, 3, 1), (7, 33, 65, 4), (64, 256, 256, 8), (100, 97, 130, 13), (256, 250, 31, 7), (256, 64, 64, 32)]


@pytest.mark.parametrize("rows,d_in,d_out,rank", SIZES)
def test_parity(sess, rows, d_in, d_out, rank):
    w = synth.random_workload(1800 + rows + rank, d_in, d_out, rank, 3, rows, dtype="f32", max_seg=max(2, rows // 2), p_finetune=0.5)
    run_and_check(sess, w, synth.make_tensors(w))


@pytest.mark.parametrize("dropout", [0.0, 0.2])
@pytest.mark.parametrize("rows,d_in,d_out,rank", SIZES)
def test_same_bits_as_the_separate_launches(sess, rows, d_in, d_out, rank, dropout):
    w = synth.random_workload(1900 + rows + rank, d_in, d_out, rank, 3, rows, dtype="f32", max_seg=max(2, rows // 2), p_finetune=0.9)
    t = synth.make_tensors(w)
    outs, launches = [], []
    mb.mlora_set_dropout(sess.ctx, dropout, 5)
    try:
        for path in (0, 1):
            mb.mlora_set_gemm_path(sess.ctx, path)
            run = LayerRun(sess, w.dtype, t, w.segments, w.n_rows, save_row_base=2)
            got = []
            n = mb.mlora_launch_count(sess.ctx)
            run.forward()
            if w.ft_rows:
                run.backward()
            launches.append(mb.mlora_launch_count(sess.ctx) - n)
            got += [x.clone() for x in (run.Y, run.x_save, run.u_save, run.dX, run.dA, run.dB)]
            if w.ft_rows:
                run.backward(accumulate=True, want_dx=False)
                got += [run.dA.clone(), run.dB.clone()]
                run.dX = run.x_save[2:]                     # an output over an operand of the launch before
                run.backward()
                got += [run.x_save.clone(), run.dA.clone(), run.dB.clone()]
            assert run.status() == mb.MLORA_OK
            outs.append(got)
            run.close()
    finally:
        mb.mlora_set_gemm_path(sess.ctx, 0)
        mb.mlora_set_dropout(sess.ctx, 0.0, 0)
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    assert launches == ([3, 6] if w.ft_rows else [1, 2])
