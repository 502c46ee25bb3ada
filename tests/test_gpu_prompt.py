"""Prompt passes against the CPU oracle, at the sizes where their tiles end: up to 48 rows (one persistent pass, attention in
groups of 16 rows, rows padded to 8), more than 128 (GEMMs on pairs of CTAs) around multiples of 32 (a tile holds 64, 128, 192
or 256 of them) and around the 1024 rows of one pass (1101: the second pass starts inside a cache page), weight matrices whose rows are no multiple of 128, both head widths, and
a sequence that is not the first of its engine.  The drafts that follow read the caches that the pass wrote."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si

pytestmark = pytest.mark.gpu

# the bound of every feature comparison with the oracle in this directory: its cache is fp32, the library's 16 bits
FEATURE_TOL = 2e-2


def _shape(head_dim):
    tiny = si.SHAPES["tiny"]
    if head_dim == 64:
        return tiny                                   # d_ffn 688 = 5 x 128 + 48
    return si.scaled(tiny, d_model=384, n_heads=3, head_dim=128, d_ffn=1040)


@pytest.fixture(scope="module", params=[64, 128])
def model(request):
    sh = _shape(request.param)
    w = si.make_weights(sh)
    return sh, w, oracle.Model(sh, w)


@pytest.mark.parametrize("plen", [1, 2, 8, 9, 16, 17, 33, 47, 48, 49, 129, 160, 161, 193, 256, 257, 385, 1024, 1025, 1101])
def test_prompt_features_match_the_oracle(model, plen):
    from paper_2412_18910_b200 import Engine
    sh, w, m = model
    cap, seq_id = 1280, 1
    prompt = si.uniform_ids(7, "prompt%d" % plen, plen, sh.vocab)
    e = Engine(sh, w, max_batch=2, kv_capacity=cap)
    try:
        seq = m.new_seq(cap)
        seq.prefill(prompt)
        e.prefill(seq_id, prompt)
        feat = e.ada_debug_buffer(0, torch.float32, (2, cap, sh.d_model))[seq_id, :plen].cpu().numpy()
        err = np.abs(feat - seq.features(0, plen)).max(axis=1)
        assert err.max() < FEATURE_TOL, (int(err.argmax()), float(err.max()))
        if plen > 1:   # the head's own cache: draft features of a chain fed the oracle's tokens
            n = 3
            forced = torch.zeros(2, sh.n_max, dtype=torch.int32)
            t_o = seq.tokens()[-1]
            e.ada_debug_buffer(2, torch.int32, (2, cap))[seq_id, plen] = int(t_o)
            d_o, _, _ = seq.draft(n)
            forced[seq_id, :n] = torch.from_numpy(d_o)
            e.ada_force_draft(forced.to(e.dev))
            e.d_n.fill_(n)
            e.ada_draft(e.d_n, e.d_draft)
            e.ada_force_draft(None)
            dfeat = e.ada_debug_buffer(4, torch.float32, (2, sh.n_max, sh.d_model))[seq_id, :n].cpu().numpy()
            derr = np.abs(dfeat - seq.draft_features(n)).max(axis=1)
            assert derr.max() < FEATURE_TOL, derr
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


@pytest.mark.parametrize("cap,budget", [(512, 5769216), (1280, 12000000), (64, 3817728)])
def test_workspaces_of_shorter_chunks(monkeypatch, cap, budget):
    """Workspaces that hold prompt chunks of 128 rows (of the sizes that the small model asked for when chunks had 128 rows) or of
    some more: the same features as with all the scratch.  One that holds none is refused."""
    from paper_2412_18910_b200 import Engine, binding
    sh = si.SHAPES["tiny"]
    w = si.make_weights(sh)
    real = binding.lib()

    class Budget:
        def __init__(self, nbytes):
            self.nbytes = nbytes

        def __getattr__(self, name):
            return (lambda cfg: self.nbytes) if name == "ada_workspace_bytes" else getattr(real, name)

    def features(nbytes):
        if nbytes:
            monkeypatch.setattr(binding, "lib", lambda: Budget(nbytes))
        try:
            e = Engine(sh, w, max_batch=1, kv_capacity=cap)
        finally:
            monkeypatch.setattr(binding, "lib", lambda: real)
        try:
            m = cap - sh.n_max - 2
            first = e.prefill(0, si.uniform_ids(9, "budget", m, sh.vocab))
            e.step()
            assert e.ada_get_counters()["status"] == 0
            return first, e.ada_debug_buffer(0, torch.float32, (1, cap, sh.d_model))[0, :m].double().clone()
        finally:
            e.close()

    t0, f0 = features(None)
    t1, f1 = features(budget)
    assert t0 == t1
    # another order of 32-bit sums moves about one cache element in 60 by a unit (2^-11 of the element): as a share of the norm
    # 2^-11 / sqrt(60), which no layer passes on whole
    assert float((f1 - f0).norm() / f0.norm()) < 2.0 ** -11 / 60 ** 0.5
    with pytest.raises(binding.AdaError, match="WORKSPACE"):
        features(1000000)
