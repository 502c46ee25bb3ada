"""Decode passes of small models, a thread-block cluster per sequence: tiles that the 16 thread blocks share unevenly or not at
all, K outside whole units, vocabularies of several rounds and on either side of the largest, contexts over and inside the
pieces of eight keys that the thread blocks and their warps are dealt, the most rows and sequences."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from tests import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,batch,prompt", [
    (dict(d_model=128, n_heads=2, d_ffn=144, vocab=272), 1, 1),
    (dict(d_model=192, n_heads=3, d_ffn=688, n_layers=3), 2, 63),
    (dict(d_model=256, n_heads=4, d_ffn=656, vocab=5136, n_max=7), 1, 129),
    (dict(n_max=1), 8, 70),
    (dict(d_ffn=128, n_layers=1), 3, 250),
    (dict(vocab=16384), 1, 20),
    (dict(vocab=16400), 1, 20),
    (dict(), 8, 33),
])
def test_lock_step(shape, batch, prompt):
    import oracle
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], **shape)
    w = si.make_weights(sh)
    m = oracle.Model(sh, w)
    e = Engine(sh, w, max_batch=batch, kv_capacity=512)
    try:
        seqs = []
        for b in range(batch):
            ids = si.uniform_ids(71 + b, "small%d" % b, prompt + 11 * b, sh.vocab)
            seq = m.new_seq(512)
            assert seq.prefill(ids) == e.prefill(b, ids)
            seqs.append(seq)
        res = lockstep.run_lockstep(e, seqs, 3)
        assert not res["failures"], res["failures"]
        e.ada_force_n([sh.n_max] * batch)
        res = lockstep.run_lockstep(e, seqs, 3, n_forced=sh.n_max)
        assert not res["failures"], res["failures"]
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("prompt", [9, 122, 250])
def test_rows_do_not_depend_on_their_pass(tiny, prompt):
    """The same tokens committed one by one, or as a block: features of the target bit for bit, and those of a draft whose catch-up rows
    were one, or all of the block."""
    from paper_2412_18910_b200 import Engine
    sh, w, _, _ = tiny
    ids = si.uniform_ids(5, "rows", prompt, sh.vocab)
    toks = torch.from_numpy(si.uniform_ids(6, "rows", sh.n_max, sh.vocab).astype(np.int32))
    out = []
    for block in (True, False):
        e = Engine(sh, w, kv_capacity=512)
        try:
            e.prefill(0, ids)
            for part in ([toks] if block else list(toks.view(-1, 1))):
                e.d_draft.zero_()
                e.d_draft[0, : len(part)] = part.to(e.dev)
                n = torch.tensor([len(part) - 1], dtype=torch.int32, device=e.dev)
                if not block:          # (the draft head follows token by token)
                    one = torch.ones(1, dtype=torch.int32, device=e.dev)
                    d = torch.zeros_like(e.d_draft)
                    e.ada_draft(one, d)
                e.ada_verify(e.d_draft, n, e.d_target)
                e.ada_force_commit(0, part.to(e.dev), len(part))
            n = torch.full((1,), sh.n_max, dtype=torch.int32, device=e.dev)
            d = torch.zeros_like(e.d_draft)
            e.ada_draft(n, d)
            feat = e.ada_debug_buffer(0, torch.float32, (1, 512, sh.d_model))[0, : prompt + len(toks)].clone()
            dfeat = e.ada_debug_buffer(4, torch.float32, (1, sh.n_max, sh.d_model)).clone()
            assert e.ada_get_counters()["status"] == 0
            out.append((feat, dfeat, d.clone()))
        finally:
            e.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_phase_clock(tiny):
    """ada_debug_buffer 9 of a profiled verify pass: its start, the embedding, five phases a layer, the LM head; nothing where no profile is
    taken."""
    from paper_2412_18910_b200 import Engine
    sh, w, prompt, _ = tiny
    e = Engine(sh, w, kv_capacity=512)
    try:
        e.prefill(0, prompt)
        e.d_draft.zero_()
        e.d_n.fill_(4)
        clock = e.ada_debug_buffer(9, torch.int64, (2560,))
        for profiled in (False, True):
            clock.zero_()
            e.ada_profile(profiled)
            e.ada_verify(e.d_draft, e.d_n, e.d_target)
            at = clock[: 5 * sh.n_layers + 3].tolist()
            assert at == sorted(at) and (min(at) > 0) == profiled and not clock[len(at):].any()
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


def test_passes_behind_a_wait_that_gave_up(tiny):
    """With the time-out bit in the status word every wait that takes long gives up: passes return, what they emit are tokens of the
    vocabulary (or nothing), and behind ada_reset_status the same context decodes in lock step with the oracle."""
    from paper_2412_18910_b200 import Engine
    sh, w, prompt, m = tiny
    e = Engine(sh, w, max_batch=1, kv_capacity=512)
    try:
        e.prefill(0, prompt)
        e.ada_selftest_bounded_wait(0, 1000, torch.zeros(2, dtype=torch.int32, device=e.dev))
        for _ in range(4):
            assert all(0 <= t < sh.vocab for t in e.step()["emitted"][0])
        assert e.ada_get_counters()["status"] & 4
        e.ada_reset_status()
        seq = m.new_seq(512)
        assert seq.prefill(prompt) == e.prefill(0, prompt)
        res = lockstep.run_lockstep(e, [seq], 4)
        assert not res["failures"], res["failures"]
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()
