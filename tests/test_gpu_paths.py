"""Kernels that small batches no longer reach by default (they take the few-row kernels), at sizes that still reach them or
under kernel variant 4, which switches the few-row kernels off: the two-SM GEMM with every tile split along K, its reduction,
its epilogue on narrow outputs, and the streaming shrink's gather, block save and dropout mask."""
import pytest
import torch

import test_gpu_parity as parity
import test_gpu_variants as variants
from paper_2607_28848_b200 import binding as mb
from paper_2607_28848_b200 import synth
from paper_2607_28848_b200.runner import LayerRun, Session

pytestmark = pytest.mark.gpu

KIND_REDUCE = 6
SPLIT = [(512, 10880, 2816), (512, 2816, 10880)]       # 22 two-SM tiles of 170 K-blocks in the forward / in the input gradient


@pytest.fixture(scope="module")
def sess():
    s = Session(0)
    yield s
    mb.mlora_set_gemm_path(s.ctx, 0)
    s.close()


def split_workload(rows, d_in, d_out):
    segs = synth.segments_array([(0, rows // 2, 0, 1), (rows // 2, rows - rows // 2, 1, 1)])
    return synth.Workload("every_tile_split", d_in, d_out, 16, 2, "bf16", rows, segs, seed=d_in)


def launch_kinds(sess, run):
    mb.mlora_profile_enable(sess.ctx, 16)
    try:
        run.forward()
        run.backward()
        return list(mb.mlora_profile_collect(sess.ctx)[0])
    finally:
        mb.mlora_profile_enable(sess.ctx, 0)


@pytest.mark.parametrize("path", [0, 4])
@pytest.mark.parametrize("rows,d_in,d_out", SPLIT)
def test_every_tile_split_along_k(sess, rows, d_in, d_out, path):
    w = split_workload(rows, d_in, d_out)
    t = synth.make_tensors(w)
    parity.run_and_check(sess, w, t, path=path, blocked=True)
    mb.mlora_set_gemm_path(sess.ctx, path)
    run = LayerRun(sess, w.dtype, t, w.segments, w.n_rows)
    try:
        assert launch_kinds(sess, run).count(KIND_REDUCE) == (1 if path == 0 else 0)
    finally:
        mb.mlora_set_gemm_path(sess.ctx, 0)
        run.close()


@pytest.mark.parametrize("rows,d_in,d_out", SPLIT)
def test_every_tile_split_along_k_in_a_graph(sess, rows, d_in, d_out):
    w = split_workload(rows, d_in, d_out)
    run = LayerRun(sess, w.dtype, synth.make_tensors(w), w.segments, w.n_rows)
    outs = (run.Y, run.x_save, run.u_save, run.dX, run.dA, run.dB)
    stream = torch.cuda.Stream(device=sess.device)
    try:
        with torch.cuda.stream(stream):
            for _ in range(2):
                run.forward()
                run.backward()
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                run.forward()
                run.backward()
            run.X.copy_(run.X.flip(0))
            run.dY.copy_(run.dY.flip(1))
            run.forward()
            run.backward()
            want = [b.clone() for b in outs]
            for b in outs:
                b.zero_()
            graph.replay()
            stream.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, outs))
        assert run.status() == mb.MLORA_OK
    finally:
        run.close()


@pytest.mark.parametrize("d_in,d_out", [(64, 128), (128, 64), (320, 448), (192, 320)])
def test_two_sm_epilogue_on_narrow_outputs(sess, d_in, d_out):
    parity.test_output_width_not_a_multiple_of_the_column_tile(sess, 4, d_in, d_out)


def test_streaming_shrink_block_save_order(sess):
    """The table of the block-save test with 512 rows of a prompt behind it: too many rows for the few-row shrink."""
    segs = [(0, 8, 0, 1), (16, 8, 0, 1), (8, 8, 0, 1), (24, 8, 0, 1), (64, 32, 1, 1), (32, 32, 1, 1), (96, 96, 2, 1),
            (192, 10, 3, 0), (202, 54, 3, 1), (256, 45, 0, 1), (301, 512, 1, 0)]
    w = synth.Workload("block_save_order", 768, 256, 16, 4, "bf16", 813, synth.segments_array(segs), seed=11)
    parity.run_and_check(sess, w, synth.make_tensors(w), base=5, cap=5 + 291 + 9)


@pytest.mark.parametrize("rank", [8, 16, 32, 64])
def test_streaming_shrink_gathered_and_contiguous_items(sess, rank):
    segs, row = [], 0
    for i in range(60):
        segs.append((row, 1, (i % 6) - 1, 0))
        row += 1
    segs.append((row, 150, 2, 1))
    row += 157                                            # seven rows that no segment covers
    segs.append((row, 90, 4, 0))
    w = synth.Workload("mixed_items", 2048, 320, rank, 5, "bf16", row + 90, synth.segments_array(segs), seed=rank)
    parity.run_and_check(sess, w, synth.make_tensors(w), path=4)


def test_streaming_shrink_dropout_mask_bit_exact(sess):
    mb.mlora_set_gemm_path(sess.ctx, 4)
    try:
        variants.test_dropout_mask_bit_exact(sess)
    finally:
        mb.mlora_set_gemm_path(sess.ctx, 0)
