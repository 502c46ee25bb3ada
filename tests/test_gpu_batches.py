"""Batches of short sequences against one oracle run per sequence, and lengths that differ inside a batch.  The tiny model decodes on
its cluster kernel, a cluster a sequence; test_gpu_routes.py runs the same widths, around the 48 rows of a persistent pass (9 rows a
sequence: 2 to 5 sequences there, 6 and 8 on the multi-row path; rows on both sides of 8, 16 and 32), on a model that it does not take."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from tests import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[8, 8], [1, 0], [8, 3, 5], [1, 8, 8, 8], [8, 8, 8, 8, 8], [2, 1, 0, 3, 1], [8, 7, 8, 1, 8, 8],
                                     [3, 8, 1, 8, 2, 8, 8, 5]])
def test_batches_match_their_sequences(tiny, lengths):
    from paper_2412_18910_b200 import Engine
    sh, w, _, m = tiny
    B = len(lengths)
    e = Engine(sh, w, max_batch=B, kv_capacity=512)
    try:
        seqs = []
        for b in range(B):
            prompt = si.uniform_ids(11 + b, "batch%d" % b, 20 + 37 * b, sh.vocab)
            seq = m.new_seq(512)
            t_o, t_g = seq.prefill(prompt), e.prefill(b, prompt)
            assert t_o == t_g
            seqs.append(seq)
        logits = torch.zeros(B, sh.n_max + 1, sh.vocab, dtype=torch.float32, device=e.dev)
        for it in range(3):
            n = torch.tensor(lengths if it % 2 == 0 else lengths[::-1], dtype=torch.int32, device=e.dev)
            e.d_n.copy_(n)
            e.ada_draft(e.d_n, e.d_draft)
            drafts = []
            dfeat = e.ada_debug_buffer(4, torch.float32, (B, sh.n_max, sh.d_model)).cpu().numpy()
            g_draft = e.d_draft.cpu().numpy()
            for b in range(B):
                nb = int(n[b])
                d_o = np.zeros(0, dtype=np.int32)
                if nb:   # a sequence's own draft: equal, or a flip inside the oracle's margin; then on with the oracle's
                    d_o, d1, d2 = seqs[b].draft(nb)
                    f_o = seqs[b].draft_features(nb)
                    rms = np.sqrt((f_o.astype(np.float64) ** 2).mean(axis=1))
                    for i in range(nb):
                        scale = max(1.0, float(rms[i]))
                        assert np.abs(dfeat[b, i] - f_o[i]).max() < 2e-2 * scale, (it, b, i)
                        if g_draft[b, i] != d_o[i]:
                            assert d1[i] - d2[i] <= lockstep.TOKEN_MARGIN * scale, (it, b, i)
                            break
                    e.d_draft[b, :nb] = torch.from_numpy(np.asarray(d_o, dtype=np.int32)).to(e.dev)
                drafts.append(d_o)
            e.ada_verify(e.d_draft, e.d_n, e.d_target, logits)
            e.ada_accept(e.d_accept, e.d_emitted, e.d_nemit)
            for b in range(B):
                tt_o, _, _, lg_o = seqs[b].verify(drafts[b], want_logits=True)
                rows = int(n[b]) + 1
                assert np.abs(logits[b, :rows].cpu().numpy() - lg_o).max() < 2e-2, (it, b)
                k_o, em_o = seqs[b].accept(drafts[b], tt_o)
                em_g = e.d_emitted.cpu().numpy()[b, : int(e.d_nemit.cpu()[b])]
                if list(em_g) != list(em_o):
                    e.ada_force_commit(b, torch.from_numpy(np.asarray(em_o, dtype=np.int32)).to(e.dev), len(em_o))
        assert e.ada_get_counters()["status"] == 0
        res = lockstep.run_lockstep(e, seqs, 4)
        assert not res["failures"], res["failures"]
    finally:
        e.close()


def test_step_ends_as_its_parts_do_when_sequences_fill_up():
    """ada_step verifies and accepts in one launch; the calls one by one accept in a kernel of their own.  Both from the same
    prompts until one sequence, then the other, has no room for a further step."""
    from paper_2412_18910_b200 import Engine
    sh = si.SHAPES["tiny"]
    w = si.make_weights(sh)
    lens, forced = (41, 13), [4, 5]
    engines = [Engine(sh, w, max_batch=2, kv_capacity=64) for _ in range(2)]
    try:
        for e in engines:
            for b, plen in enumerate(lens):
                e.prefill(b, si.uniform_ids(3 + b, "full%d" % b, plen, sh.vocab))
            e.ada_force_n(forced)
        one, parts = engines
        full = 0
        for it in range(60):
            one.ada_step(one.d_emitted, one.d_nemit, one.d_nused, one.d_accept)
            parts.ada_ldlp_predict(parts.d_n)
            parts.ada_draft(parts.d_n, parts.d_draft)
            parts.ada_verify(parts.d_draft, parts.d_n, parts.d_target)
            parts.ada_accept(parts.d_accept, parts.d_emitted, parts.d_nemit)
            a, p = ([e.d_nemit.cpu().tolist(), e.d_accept.cpu().tolist()] for e in engines)
            assert a == p, it
            for b, k in enumerate(a[0]):
                assert one.d_emitted[b, :k].cpu().tolist() == parts.d_emitted[b, :k].cpu().tolist(), (it, b)
            full += a[0] == [0, 0]
        assert full > 3   # both came to their end
        tok = [e.ada_debug_buffer(2, torch.int32, (2, 64)).cpu() for e in engines]
        assert torch.equal(tok[0], tok[1])
        c = [e.ada_get_counters() for e in engines]
        assert all(c[0][k] == c[1][k] for k in ("n_target", "n_draft", "n_waste", "n_tokens", "status"))
        assert c[0]["status"] in (0, 1)   # (1: lengths were clamped to the room left)
    finally:
        for e in engines:
            e.close()


@pytest.mark.parametrize("batch", [5, 6, 8])
def test_catch_up_rows_of_more_than_one_pass(tiny, batch):
    """Drafts after nine tokens were committed in every sequence: nine catch-up rows a cluster, or (test_gpu_routes.py) 45, 54 and 72,
    which the draft head takes in a persistent pass of up to 48 rows or on the multi-row path."""
    import oracle
    from paper_2412_18910_b200 import Engine
    sh, w, _, m = tiny
    e = Engine(sh, w, max_batch=batch, kv_capacity=512)
    try:
        seqs, prompts, streams = [], [], []
        for b in range(batch):
            prompts.append(si.uniform_ids(23 + b, "catch%d" % b, 30 + 29 * b, sh.vocab))
            streams.append(oracle.decode(m, prompts[b], 40, n_policy=0)["tokens"])
            seqs.append(m.new_seq(512))
            assert seqs[b].prefill(prompts[b]) == e.prefill(b, prompts[b])
        e.ada_force_n([8] * batch)
        res = lockstep.run_lockstep(e, seqs, 2, n_forced=8, forced_stream=streams, prompts=prompts)
        assert not res["failures"], res["failures"]
        assert all(seq.counters()["n_waste"] == 0 for seq in seqs)
        e.ada_force_draft(None)
        res = lockstep.run_lockstep(e, seqs, 2, n_forced=8)     # the heads' own drafts on those cache rows
        assert not res["failures"], res["failures"]
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("batch,wider", [(1, dict(vocab=40960)), (6, dict(vocab=40960)), (2, dict(d_ffn=19200))])
def test_models_that_the_persistent_pass_does_not_hold(batch, wider):
    """Vocabularies above 37 888 and d_ffn above 18 944 (256 and 128 columns for each of 148 thread blocks): prompts, every draft step
    and verify passes on the multi-row path."""
    import oracle
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], **wider)
    w = si.make_weights(sh)
    m = oracle.Model(sh, w)
    e = Engine(sh, w, max_batch=batch, kv_capacity=256)
    try:
        seqs = []
        for b in range(batch):
            prompt = si.uniform_ids(81 + b, "wide%d" % b, 9 + 31 * b, sh.vocab)
            seq = m.new_seq(256)
            assert seq.prefill(prompt) == e.prefill(b, prompt)
            seqs.append(seq)
        e.ada_force_n([8] * batch)
        res = lockstep.run_lockstep(e, seqs, 2, n_forced=8)
        assert not res["failures"], res["failures"]
        e.ada_force_n(None)
        res = lockstep.run_lockstep(e, seqs, 3)
        assert not res["failures"], res["failures"]
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("vocab", [4096, 5120, 9216, 9728])
def test_small_models_on_part_of_the_chip(vocab):
    """Vocabularies of several rounds of the cluster kernel.  On models that it does not take (test_gpu_routes.py): widths around the 64
    thread blocks that the smallest run on, between them and all of the chip, and on either side of its 148 SMs (32 KB of the
    vocabulary matrix to a block).  Prompts of 7 tokens are passes of those grids here too."""
    import oracle
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], vocab=vocab)
    w = si.make_weights(sh)
    m = oracle.Model(sh, w)
    e = Engine(sh, w, max_batch=2, kv_capacity=512)
    try:
        seqs = []
        for b, plen in enumerate((7, 130)):
            prompt = si.uniform_ids(5 + b, "grid%d" % b, plen, vocab)
            seq = m.new_seq(512)
            assert seq.prefill(prompt) == e.prefill(b, prompt)
            seqs.append(seq)
        res = lockstep.run_lockstep(e, seqs, 6)
        assert not res["failures"], res["failures"]
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("d,heads,ffn,batch", [(192, 3, 144, 2), (1088, 17, 400, 2), (4672, 73, 128, 1), (4800, 75, 128, 1)])
def test_slabs_of_odd_widths(d, heads, ffn, batch):
    """Slabs that start on odd columns, thread blocks without a slab, pieces of 64 columns that a slab fills in part, wholly, or
    with a column in a second piece (64 and 65 columns a pair of thread blocks at the largest widths), K outside whole chunks."""
    import oracle
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], n_layers=1, d_model=d, n_heads=heads, head_dim=64, d_ffn=ffn, vocab=272)
    w = si.make_weights(sh)
    m = oracle.Model(sh, w)
    e = Engine(sh, w, max_batch=batch, kv_capacity=128)
    try:
        seqs = []
        for b in range(batch):
            prompt = si.uniform_ids(11 + b, "odd%d" % b, 7 + 13 * b, 272)
            seq = m.new_seq(128)
            assert seq.prefill(prompt) == e.prefill(b, prompt)
            seqs.append(seq)
        res = lockstep.run_lockstep(e, seqs, 4)
        assert not res["failures"], res["failures"]
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("batch", [1, 3, 6])
def test_drafts_do_not_depend_on_batch_mates(batch):
    """A sequence's drafts and draft features bit for bit beside short and beside long sequences (three sequences: every step in
    the persistent pass, and the same bits as alone; six: the first step on the multi-row path), and whatever the length of
    the draft that they belong to.  Sixteen heads: the items of the long batch are more than the thread blocks."""
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], d_model=1024, n_heads=16, d_ffn=1408)
    w = si.make_weights(sh)
    prompt = si.uniform_ids(31, "mates", 300, sh.vocab)

    def draft(B, mate_len, n):
        e = Engine(sh, w, max_batch=B, kv_capacity=512)
        try:
            for b in range(B):
                e.prefill(b, prompt if b == 0 else si.uniform_ids(32 + b, "mate", mate_len, sh.vocab))
            e.d_n.fill_(sh.n_max)
            e.d_n[0] = n
            e.ada_draft(e.d_n, e.d_draft)
            f = e.ada_debug_buffer(4, torch.float32, (B, sh.n_max, sh.d_model))[0, :n].clone()
            assert e.ada_get_counters()["status"] == 0
            return e.d_draft[0, :n].clone(), f
        finally:
            e.close()

    tokens, feats = draft(1 if batch == 3 else batch, 20, sh.n_max)
    for mate_len, n in ((20, sh.n_max), (450, sh.n_max), (450, 3)):
        t, f = draft(batch, mate_len, n)
        assert torch.equal(t, tokens[:n]) and torch.equal(f, feats[:n]), (mate_len, n)


@pytest.mark.parametrize("lengths", [[8, 7], [8, 8], [5, 5, 5], [8, 8, 5], [8, 8, 8], [8, 8, 8, 8, 2], [8, 8, 8, 8, 8]])
def test_verified_rows_do_not_depend_on_batch_mates(lengths):
    """Logits, features and cache rows of verify passes of 17 to 45 rows, heads 128 wide, bit for bit as each sequence alone has
    them: 16 rows at most, whose first keys are requested in the QKV phase; those of more rows wait until the sums that lie in the
    same shared memory are read.  Several cache splits and more than one piece of keys a warp; two layers, so that the cache
    rows of the first are read behind the second's sums; a second pass reads the cache rows that the first left."""
    from paper_2412_18910_b200 import Engine
    sh = si.scaled(si.SHAPES["tiny"], d_model=512, n_heads=4, head_dim=128, d_ffn=1376)
    w = si.make_weights(sh)
    prompts = [si.uniform_ids(41 + b, "rows%d" % b, 700 - 130 * b, sh.vocab) for b in range(len(lengths))]
    drafts = torch.from_numpy(np.stack([si.uniform_ids(51 + b, "draft%d" % b, 2 * sh.n_max, sh.vocab) for b in range(len(lengths))]))

    def verify(members):
        e = Engine(sh, w, max_batch=len(members), kv_capacity=1024)
        try:
            for i, b in enumerate(members):
                e.prefill(i, prompts[b])
            out = []
            for it in range(2):
                e.d_n.copy_(torch.tensor([lengths[b] for b in members], dtype=torch.int32))
                e.d_draft.copy_(drafts[members, it * sh.n_max: (it + 1) * sh.n_max])
                logits = torch.zeros(e.B, sh.n_max + 1, sh.vocab, device=e.dev)
                e.ada_verify(e.d_draft, e.d_n, e.d_target, logits)
                feat = e.ada_debug_buffer(0, torch.float32, (e.B, 1024, sh.d_model))
                pos = [len(prompts[b]) + it for b in members]
                out.append([(logits[i, : lengths[b] + 1].clone(), feat[i, pos[i]: pos[i] + lengths[b] + 1].clone())
                            for i, b in enumerate(members)])
                for i, b in enumerate(members):     # one token on, the same whatever was drafted
                    e.ada_force_commit(i, drafts[b, it: it + 1].to(e.dev).int(), 1)
            assert e.ada_get_counters()["status"] == 0
            return out
        finally:
            e.close()

    together = verify(list(range(len(lengths))))
    for b in range(len(lengths)):
        alone = verify([b])
        for it in range(2):
            for x, y in zip(together[it][b], alone[it][0]):
                assert torch.equal(x, y), (b, it)
