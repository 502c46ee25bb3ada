"""Prompt GEMMs whose tiles are cut so that every pair of thread blocks gets as much: tiles in two and in more parts, of one and of
several token tiles, partly filled ones, behind whole waves; and of a GEMM that leaves sums for a reduction.  Against 64-bit sums
over the library's own cache, by the measure of the precision tests (the 128-row kernel's error); and bit for bit when repeated
behind other lengths, whose sums lie in the same memory."""
import pytest
import torch

import synth_inputs as si
from tests import test_gpu_precision as prec

pytestmark = pytest.mark.gpu

CAP = 1088


def _errors(sh, lengths, monkeypatch):
    from paper_2412_18910_b200 import Engine
    monkeypatch.setattr(prec, "CAP", CAP)
    e = Engine(sh, si.make_weights(sh), kv_capacity=CAP)
    try:
        out = {}
        for m in lengths + lengths[::-1]:
            e.prefill(0, si.uniform_ids(29, "runs%d" % m, m, sh.vocab))
            feat = e.ada_debug_buffer(0, torch.float32, (1, CAP, sh.d_model))[0, :m].clone()
            if m in out:
                assert torch.equal(feat, out[m][0]), m
                continue
            toks = e.ada_debug_buffer(2, torch.int32, (1, CAP))[0, :m]
            out[m] = feat, prec._off(feat, prec._features(e, sh, 0, torch.arange(m, device=e.dev), toks))
        assert e.ada_get_counters()["status"] == 0
        return {m: x[1] for m, x in out.items()}
    finally:
        e.close()


@pytest.mark.parametrize("shape,lengths", [
    (dict(d_model=2048, n_heads=32, head_dim=64, d_ffn=11264), [129, 205, 256, 300, 517]),
    (dict(d_model=5120, n_heads=40, head_dim=128, d_ffn=688), [205, 1000]),
])
def test_cut_tiles(shape, lengths, monkeypatch):
    sh = si.scaled(si.SHAPES["tiny"], n_layers=1, vocab=272, **shape)
    off = _errors(sh, [100] + lengths, monkeypatch)
    for m in lengths:
        assert off[m] < 1.05 * off[100], (m, off)


def test_flags_that_a_wait_left_behind():
    """A wait that gave up leaves the other pair's flag set (here: all of them): after ada_reset_status the same prompt has the same bits
    again, and no sums of an earlier launch."""
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], n_layers=1, vocab=272, d_model=2048, n_heads=32, head_dim=64, d_ffn=11264)
    e = Engine(sh, si.make_weights(sh), kv_capacity=CAP)
    try:
        feats = []
        flags, counts = 2 * 74 * 8, 64       # the flags and the grid barrier's words lie, in 256 bytes each, before the phase clock
        clock = e.ada_debug_buffer(9, torch.int64, (2560,)).data_ptr() - e.workspace.data_ptr()
        at = clock - 4 * counts - (4 * flags + 255) // 256 * 256
        left = e.workspace[at: at + 4 * flags].view(torch.int32)
        for m in (205, 300, 205):
            e.prefill(0, si.uniform_ids(29, "runs%d" % m, m, sh.vocab))
            feats.append(e.ada_debug_buffer(0, torch.float32, (1, CAP, sh.d_model))[0, :m].clone())
            assert not left.any()
            left.fill_(1)
            e.ada_reset_status()
        assert torch.equal(feats[0], feats[2])
        assert not left.any() and e.ada_get_counters()["status"] == 0
    finally:
        e.close()


def test_rows_of_the_multi_row_gemms():
    """Prompts of 49 to 128 rows bring only as many rows of the planes as they have, in steps of eight: a row's features do not depend on
    how many rows come after it, bit for bit."""
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], n_layers=2, vocab=272, d_model=2048, n_heads=16, head_dim=128, d_ffn=1424)
    ids = si.uniform_ids(31, "rows", 128, sh.vocab)
    e = Engine(sh, si.make_weights(sh), kv_capacity=256)
    try:
        feats = {}
        for m in (128, 49, 127, 56, 57, 64, 88, 89, 120, 121):
            e.prefill(0, ids[:m])
            feats[m] = e.ada_debug_buffer(0, torch.float32, (1, 256, sh.d_model))[0, :m].clone()
            assert torch.equal(feats[m], feats[128][:m]), m
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("shape,lengths", [   # tiles of 32 to 128 prompt rows per thread block, full and with rows to spare, whole and cut
    (dict(d_model=2048, n_heads=32, head_dim=64, d_ffn=5632), [130, 144, 145, 209, 230, 241, 333, 401, 433, 600, 850]),
    (dict(d_model=4096, n_heads=32, head_dim=128, d_ffn=11008), [130, 145, 205, 209, 333, 401, 610]),
])
def test_tile_widths(shape, lengths, monkeypatch):
    sh = si.scaled(si.SHAPES["tiny"], n_layers=1, vocab=272, **shape)
    off = _errors(sh, [100] + lengths, monkeypatch)
    for m in lengths:
        assert off[m] < 1.05 * off[100], (m, off)
