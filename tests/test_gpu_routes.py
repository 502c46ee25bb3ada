"""Tests of the small model again, on models that its cluster kernel (k_small) does not take: heads of 128, d_model above 256, d_ffn
above 1024.  Packed labels and batches on the multi-row path, accepting inside the persistent pass, its grids of 64 thread blocks and
odd slabs, the programmatic chain of decode passes.  test_small_model.py holds k_small's plan to refusing these shapes."""
import pytest
import torch

import synth_inputs as si
from tests import test_gpu_batches as batches, test_gpu_labels as labels, test_gpu_tiny as small

pytestmark = pytest.mark.gpu

WIDE = dict(d_model=512, n_heads=4, head_dim=128, d_ffn=1376)
HEADS64 = dict(d_model=320, n_heads=5, d_ffn=688)
NARROW = dict(d_model=192, n_heads=3, d_ffn=1168, vocab=272, n_layers=1)
MANY_HEADS = dict(d_model=2816, n_heads=44, d_ffn=1408, vocab=1024)     # a batch of three has more heads than a persistent pass takes
SHAPES = [WIDE, HEADS64, NARROW, MANY_HEADS]


def again(test):
    """The parameters of another test."""
    return pytest.mark.parametrize(*next(m for m in test.pytestmark if m.name == "parametrize").args)


def _model(shape):
    import oracle
    sh = si.scaled(si.SHAPES["tiny"], **shape)
    w = si.make_weights(sh)
    return sh, w, si.make_prompts(sh)[0], oracle.Model(sh, w)


@pytest.fixture(scope="module")
def wide():
    return _model(WIDE)


@pytest.fixture(scope="module")
def heads64():
    return _model(HEADS64)


@pytest.fixture(scope="module")
def wide_engine(wide):
    from paper_2412_18910_b200 import Engine
    e = Engine(wide[0], wide[1], max_batch=1, kv_capacity=wide[0].kv_capacity)
    yield e
    e.close()


@pytest.mark.parametrize("batch,shape,one_launch", [(1, WIDE, True), (5, WIDE, True), (6, WIDE, False), (8, WIDE, False), (1, HEADS64, True),
                                                    (2, NARROW, True), (3, MANY_HEADS, False)])
def test_which_kernels_run(batch, shape, one_launch):
    """A verify pass is one launch of matrix products (the persistent kernel) or four a layer and the LM head (the multi-row path)."""
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], **shape)
    e = Engine(sh, si.make_weights(sh), max_batch=batch, kv_capacity=128)
    try:
        for b in range(batch):
            e.prefill(b, si.uniform_ids(61 + b, "route", 9 + b, sh.vocab))
        e.d_draft.zero_()
        e.d_n.fill_(sh.n_max)
        e.ada_profile(True)
        e.ada_verify(e.d_draft, e.d_n, e.d_target)
        assert e.ada_get_profile()["gemm_launches"] == (1 if one_launch else 4 * sh.n_layers + 1)
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@again(labels.test_packed_labels_equal_single_label_passes)
def test_packed_labels(wide, plen, j0, count, cap, batch):
    labels.test_packed_labels_equal_single_label_passes(wide, plen, j0, count, cap, batch)


@again(labels.test_labels_leave_the_sequences_as_they_were)
def test_labels_leave_the_sequences(wide, plen, cap, batch, forced):
    labels.test_labels_leave_the_sequences_as_they_were(wide, plen, cap, batch, forced)


def test_labels_match_the_oracle(wide, wide_engine):
    small.test_labels_over_start_positions_match_the_oracle_and_leave_the_state_alone(wide)
    small.test_label_pass_and_told_the_label_nothing_is_wasted(wide, wide_engine)
    small.test_label_pass_matches_the_oracle_label_on_own_drafts(wide, wide_engine)


@again(batches.test_batches_match_their_sequences)
def test_batches(wide, lengths):
    batches.test_batches_match_their_sequences(wide, lengths)


@again(batches.test_catch_up_rows_of_more_than_one_pass)
def test_catch_up_rows(wide, batch):
    batches.test_catch_up_rows_of_more_than_one_pass(wide, batch)


def test_sequences_that_fill_up(monkeypatch):
    monkeypatch.setitem(si.SHAPES, "tiny", si.scaled(si.SHAPES["tiny"], **WIDE))
    batches.test_step_ends_as_its_parts_do_when_sequences_fill_up()


@pytest.mark.parametrize("vocab", [2048, 2560, 4608, 4864])     # 64, 80 and 144 thread blocks, and all SMs
def test_part_of_the_chip(vocab, monkeypatch):
    monkeypatch.setitem(si.SHAPES, "tiny", si.scaled(si.SHAPES["tiny"], **WIDE))
    batches.test_small_models_on_part_of_the_chip(vocab)


def test_slabs_of_three_columns():
    batches.test_slabs_of_odd_widths(NARROW["d_model"], NARROW["n_heads"], NARROW["d_ffn"], 2)


@again(small.test_long_context_attention_spans_blocks_and_rounds)
def test_long_contexts(heads64, plen):
    small.test_long_context_attention_spans_blocks_and_rounds(heads64, plen)


def test_launch_chain(monkeypatch):
    monkeypatch.setitem(si.SHAPES, "tiny", si.scaled(si.SHAPES["tiny"], **MANY_HEADS))
    small.test_launch_chain_equals_plain_stream_order_bit_for_bit(monkeypatch)
