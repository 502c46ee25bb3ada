"""Labels of packed start positions (ada_label_positions) against one label pass per position from a fresh prefill: groups
of eight and a rest, start positions on both sides of a page boundary, drafts that reach into the next page, a sequence
whose cache leaves room for some of them only, and a sequence that is not the first of its engine.  The tiny model's packed passes run
on its cluster kernel; test_gpu_routes.py runs these on the multi-row path."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("plen,j0,count,cap,batch", [
    (80, 57, 17, 512, 1),      # two groups of eight and one; positions 57 .. 73 around the boundary at 64
    (129, 128, 2, 512, 2),     # the first rows of a page
    (200, 183, 9, 320, 1),     # one unused page: position 183 packed, the others (two pages each) in the sequence's own
    (240, 233, 6, 256, 1),     # no unused page
    (70, 1, 3, 512, 1)])       # the start of the text
def test_packed_labels_equal_single_label_passes(tiny, plen, j0, count, cap, batch):
    from paper_2412_18910_b200 import Engine
    sh, w, _, _ = tiny
    text = si.uniform_ids(3, "label%d" % plen, plen, sh.vocab)
    e = Engine(sh, w, max_batch=batch, kv_capacity=cap)
    try:
        b = batch - 1
        e.prefill(b, text)
        before = e.ada_debug_buffer(3, torch.int32, (batch, 8)).clone()
        k = torch.full((count,), -9, dtype=torch.int32, device=e.dev)
        dr = torch.zeros(count, sh.n_max, dtype=torch.int32, device=e.dev)
        tg = torch.zeros(count, sh.n_max + 1, dtype=torch.int32, device=e.dev)
        e.ada_label_positions(b, j0, count, k, dr, tg)
        assert torch.equal(e.ada_debug_buffer(3, torch.int32, (batch, 8)), before)
        feats = e.ada_debug_buffer(0, torch.float32, (batch, cap, sh.d_model))[b, : plen].clone()
        one = Engine(sh, w, max_batch=1, kv_capacity=cap)
        try:
            for i in range(count):
                # the state in which token j was pending: a prompt of the tokens before it, then token j committed
                j = j0 + i
                one.prefill(0, text[:j])
                if j < plen:
                    one.ada_debug_buffer(2, torch.int32, (1, cap))[0, j] = int(text[j])
                one.ada_force_n(None)
                kk = torch.zeros(1, dtype=torch.int32, device=e.dev)
                one.ada_label(kk)
                n = int(min(sh.n_max, cap - j - 2))
                d1 = one.ada_debug_buffer(7, torch.int32, (1, sh.n_max))[0, :n]
                t1 = one.ada_debug_buffer(8, torch.int32, (1, sh.n_max + 1))[0, : n + 1]
                assert torch.equal(dr[i, :n], d1) and bool((dr[i, n:] == -1).all()), (i, dr[i], d1)
                assert torch.equal(tg[i, : n + 1], t1) and bool((tg[i, n + 1:] == -1).all()), (i, tg[i], t1)
                assert int(k[i]) == int(kk)
            one.prefill(0, text)
            ref = one.ada_debug_buffer(0, torch.float32, (1, cap, sh.d_model))[0, :plen]
            assert float((feats - ref).abs().max()) < 2e-2      # the text's own features: as after its prefill
        finally:
            one.close()
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("plen,cap,batch,forced", [
    (180, 256, 1, False),     # no unused page beside a sequence that goes on: every position in the sequence's own pages
    (100, 192, 2, False),     # one unused page: the first positions packed, those that need two pages one by one
    (100, 512, 2, True),      # teacher forcing: one by one
    (20, 512, 6, False)])     # packed, beside a batch of six
def test_labels_leave_the_sequences_as_they_were(tiny, plen, cap, batch, forced):
    """Two engines decode the same prompts; one labels a range of prompt and decoded positions in between, after a verify whose
    outcome is accepted only then.  States, features, cache rows, drafts and choices are the same bits, and so is what follows."""
    from paper_2412_18910_b200 import Engine
    sh, w, _, _ = tiny
    engines = [Engine(sh, w, max_batch=batch, kv_capacity=cap) for _ in range(2)]
    try:
        seq = batch - 1
        kept = []
        for e in engines:
            for b in range(batch):
                e.prefill(b, si.uniform_ids(41 + b, "keep%d" % plen, plen, sh.vocab))
            for _ in range(4):
                e.step()
            e.ada_ldlp_predict(e.d_n)
            if forced:
                g = torch.Generator(e.dev).manual_seed(5)
                e.ada_force_draft(torch.randint(0, sh.vocab, (batch, sh.n_max), generator=g, device=e.dev, dtype=torch.int32))
            e.ada_draft(e.d_n, e.d_draft)
            e.ada_verify(e.d_draft, e.d_n, e.d_target)
            if e is engines[0]:
                last = int(e.ada_debug_buffer(3, torch.int32, (batch, 8))[seq, 0]) - 1
                j0 = max(1, last - 24)
                if forced:
                    j0 = last - 3
                k = torch.zeros(last - j0 + 1, dtype=torch.int32, device=e.dev)
                pools = cap * batch * (sh.n_layers + 1) * sh.d_model * 2 * 2
                base = (-e.workspace.data_ptr()) % 256
                before = e.workspace[base: base + pools].clone()
                e.ada_label_positions(seq, j0, last - j0 + 1, k)
                # cache rows of all positions so far (the packed positions' rows lie in pages that no sequence uses)
                page = sh.n_heads * 64 * sh.head_dim * 2
                used = [i * batch + b for b in range(batch) for i in range((last if b == seq else cap) // 64 + 1) if i * 64 < cap]
                off = 0
                for L in (sh.n_layers, sh.n_layers, 1, 1):
                    size = cap // 64 * batch * L * page
                    a = before[off: off + size].view(-1, L * page)
                    now = e.workspace[base + off: base + off + size].view(-1, L * page)
                    assert torch.equal(a[used], now[used])
                    off += size
            kept.append([e.ada_debug_buffer(n, torch.int32, dims).clone() for n, dims in
                         ((3, (batch, 8)), (7, (batch, sh.n_max)), (8, (batch, sh.n_max + 1)))] +
                        [e.ada_debug_buffer(n, torch.float32, dims).clone() for n, dims in
                         ((4, (batch, sh.n_max, sh.d_model)), (5, (batch, sh.n_max + 1, 2)), (6, (batch, sh.n_max, 2)))])
            e.ada_accept(e.d_accept, e.d_emitted, e.d_nemit)
            e.ada_force_draft(None)
            for _ in range(2):
                e.step()
            assert e.ada_get_counters()["status"] == 0
        assert torch.equal(kept[0][0], kept[1][0])
        for which, extra in ((1, 0), (2, 1), (3, 0), (4, 1), (5, 0)):    # entries past the draft lengths are never written
            for s in range(batch):
                n = int(kept[0][0][s, 2]) + extra
                assert torch.equal(kept[0][which][s, :n], kept[1][which][s, :n]), (which, s)
        lens = [e.ada_debug_buffer(3, torch.int32, (batch, 8))[:, 0].tolist() for e in engines]
        assert lens[0] == lens[1]
        for which, dtype, dims in ((0, torch.float32, (batch, cap, sh.d_model)), (2, torch.int32, (batch, cap))):
            a, b = (e.ada_debug_buffer(which, dtype, dims) for e in engines)
            for s, n in enumerate(lens[0]):
                assert torch.equal(a[s, : n - 1], b[s, : n - 1])
    finally:
        for e in engines:
            e.close()
