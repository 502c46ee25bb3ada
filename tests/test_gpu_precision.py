"""Rounding of every route against 64-bit sums.  A row may be read by the 128-row kernel (prompts of 49 to 128 tokens: K splits of
up to 1365 elements, an accumulator each for the hi and the lo products), by CTA pairs (longer prompts) or by the persistent
pass (short prompts, decode passes of up to 48 rows, draft steps).  The tensor core's accumulators drop what lies below their
last bit at every addition, so the error grows with the additions made to one accumulator, and it is what differs between
the routes: the first route's error is the measure, and every other one must stay within a twentieth of it (its rows are
others; nine rows of one sequence scatter by a tenth, and get a fifth).  One accumulator over all of K: 1.2 to 1.35 times the
measure at this width.

The 64-bit reference reads the library's own 16-bit cache, so that no rounding of a cache element hides the sums' error.
"""
import math

import numpy as np
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

D = torch.float64
CAP = 512


@pytest.fixture(scope="module")
def model():
    sh = si.scaled(si.SHAPES["tiny"], d_model=2048, n_heads=32, head_dim=64, d_ffn=5632)
    return sh, si.make_weights(sh)


def _pools(e, sh):
    """Keys and values of target and draft head, [sequence][layer][head][position][channel]: the pools open the workspace,
    [page][layer][head][slot][channel] with page i of sequence b at i B + b and a row's 16-byte chunks XORed with slot & 7."""
    H, hd = sh.n_heads, sh.head_dim
    base, off, out = (-e.workspace.data_ptr()) % 256, 0, []
    chunk = torch.arange(hd // 8, device=e.dev)[None, :] ^ (torch.arange(64, device=e.dev) & 7)[:, None]
    for L in (sh.n_layers, sh.n_layers, 1, 1):
        off = (off + 255) & ~255
        size = CAP * e.B * L * H * hd * 2
        t = e.workspace[base + off: base + off + size].view(torch.float16).view(CAP // 64, e.B, L, H, 64, hd // 8, 8)
        t = torch.gather(t, 5, chunk[None, None, None, None, :, :, None].expand(t.shape))
        out.append(t.permute(1, 2, 3, 0, 4, 5, 6).reshape(e.B, L, H, CAP, hd))
        off += size
    return out


def _norm(h, g, eps):
    return h / torch.sqrt((h * h).mean(-1, keepdim=True) + eps) * g.to(D)


def _layer(w, h, pos, K, V, sh):
    H, hd = sh.n_heads, sh.head_dim
    q = (_norm(h, w["norm_attn"], sh.rms_eps) @ w["wq"].to(D).T).view(-1, H, hd)
    ang = pos.to(D)[:, None] * sh.rope_theta ** (-2.0 * torch.arange(hd // 2, dtype=D, device=h.device) / hd)
    c, s = ang.cos()[:, None, :], ang.sin()[:, None, :]
    x, y = q[..., : hd // 2], q[..., hd // 2:]
    q = torch.cat([x * c - y * s, y * c + x * s], -1)
    n = int(pos.max()) + 1
    z = torch.einsum("thd,hkd->htk", q, K[:, :n].to(D)) / math.sqrt(hd)
    z = z.masked_fill(torch.arange(n, device=h.device)[None, None, :] > pos[None, :, None], float("-inf"))
    h = h + torch.einsum("htk,hkd->thd", z.softmax(-1), V[:, :n].to(D)).reshape(len(pos), -1) @ w["wo"].to(D).T
    u = _norm(h, w["norm_mlp"], sh.rms_eps)
    g = u @ w["w_gate"].to(D).T
    return h + (g / (1 + torch.exp(-g)) * (u @ w["w_up"].to(D).T)) @ w["w_down"].to(D).T


_LAYER = ("norm_attn", "wq", "wo", "norm_mlp", "w_gate", "w_up", "w_down")


def _features(e, sh, b, pos, toks):
    K, V = _pools(e, sh)[:2]
    h = e.w["embed"][toks.long()].to(D)
    for l in range(sh.n_layers):
        h = _layer({n: e.w[n][l] for n in _LAYER}, h, pos, K[b, l], V[b, l], sh)
    return _norm(h, e.w["final_norm"], sh.rms_eps)


def _off(got, want):
    return float((got.to(D) - want).norm() / want.norm())


def _engine(model, lens):
    from paper_2412_18910_b200 import Engine
    sh, w = model
    e = Engine(sh, w, max_batch=len(lens), kv_capacity=CAP)
    for b, m in enumerate(lens):
        e.prefill(b, si.uniform_ids(23 + b, "prec%d" % m, m, sh.vocab))
    return e


def _prompt_error(model, m):
    sh, _ = model
    e = _engine(model, [m])
    try:
        feat = e.ada_debug_buffer(0, torch.float32, (1, CAP, sh.d_model))[0, :m]
        toks = e.ada_debug_buffer(2, torch.int32, (1, CAP))[0, :m]
        return _off(feat, _features(e, sh, 0, torch.arange(m, device=e.dev), toks))
    finally:
        e.close()


@pytest.fixture(scope="module")
def measure(model):
    return _prompt_error(model, 100)


@pytest.mark.parametrize("m", [31, 48, 129, 333])
def test_prompt_routes(model, measure, m):
    assert _prompt_error(model, m) < 1.05 * measure


@pytest.mark.parametrize("lens", [[300], [31, 205, 118], [100, 310, 33, 57], [100, 310, 33, 57, 200]])
def test_decode_routes(model, measure, lens):
    """Verify rows, and draft rows each from the library's own inputs: 9 to 45 rows in all (the longest chains)."""
    sh, _ = model
    e = _engine(model, lens)
    try:
        n = sh.n_max
        e.d_n.fill_(n)
        e.ada_draft(e.d_n, e.d_draft)
        e.ada_verify(e.d_draft, e.d_n, e.d_target)
        feat = e.ada_debug_buffer(0, torch.float32, (e.B, CAP, sh.d_model))
        dfeat = e.ada_debug_buffer(4, torch.float32, (e.B, n, sh.d_model))
        tok = e.ada_debug_buffer(2, torch.int32, (e.B, CAP))
        dk, dv = _pools(e, sh)[2:]
        head = {k: e.w[{"norm_attn": "e_norm_attn", "norm_mlp": "e_norm_mlp"}.get(k, "e_" + k.replace("w_", ""))] for k in _LAYER}
        got, want, dgot, dwant = [], [], [], []
        for b, m in enumerate(lens):
            toks = torch.cat([tok[b, m: m + 1], e.d_draft[b]])
            got.append(feat[b, m: m + n + 1])
            want.append(_features(e, sh, b, torch.arange(m, m + n + 1, device=e.dev), toks))
            x = torch.cat([e.w["embed"][toks[:n].long()].to(D), torch.cat([feat[b, m - 1: m], dfeat[b, : n - 1]]).to(D)], 1)
            dgot.append(dfeat[b])
            dwant.append(_layer(head, x @ e.w["eagle_fc"].to(D).T, torch.arange(m - 1, m - 1 + n, device=e.dev), dk[b, 0], dv[b, 0], sh))
        bound = (1.05 if len(lens) > 1 else 1.2) * measure
        assert _off(torch.cat(got), torch.cat(want)) < bound
        assert _off(torch.cat(dgot), torch.cat(dwant)) < bound
        assert e.ada_get_counters()["status"] == 0
    finally:
        e.close()


def _tree(v):
    """The sum of 32 values as a warp's exchanges make it: pairs 16 apart, then 8, 4, 2, 1."""
    for o in (16, 8, 4, 2, 1):
        v = v + v[..., np.arange(32) ^ o]
    return v[..., 0]


def _pass_row_sum(sq, row, width, ctas, pairs):
    """A row's sum of squares as passes of up to 48 rows form it: per thread block that finishes the row (of a pair that splits K
    each second row) its columns in groups of 32, the groups in order; the thread blocks 32 apart in order, then a tree."""
    c = np.zeros(256, dtype=np.float32)
    for s in range(-(-len(sq) // width)):
        cols = sq[s * width: (s + 1) * width]
        cols = np.concatenate([cols, np.zeros(-len(cols) % 32, dtype=np.float32)]).reshape(-1, 32)
        r = np.float32(0)
        for g in _tree(cols):
            r = r + g
        c[2 * s + row % 2 if pairs else s] = r
    assert -(-len(sq) // width) * (2 if pairs else 1) <= ctas
    lanes = np.zeros(32, dtype=np.float32)
    for k in range(8):
        lanes = lanes + c[32 * k: 32 * k + 32]
    return _tree(lanes)


@pytest.mark.parametrize("d,ffn,width,pairs", [(256, 128, 4, False), (768, 688, 11, True), (1024, 688, 14, True), (1536, 688, 21, True),
                                               (4096, 688, 56, True), (4800, 688, 65, True), (5120, 688, 70, True), (8192, 688, 111, True)])
def test_order_of_a_rows_sum_of_squares(d, ffn, width, pairs):
    """Its last bit moves a row's scale, and with it 16-bit cache elements: the first rows of a short prompt see few keys, and 7B
    features move by 2e-4 of their size with another order.  All layers hand the embedding on, so the final norm's input and every
    square are known; where it holds 1 the features are the row's scale itself."""
    from paper_2412_18910_b200 import Engine
    tiny = si.SHAPES["tiny"]
    hd = 128 if d > 5120 else 64
    sh = si.scaled(tiny, d_model=d, n_heads=d // hd, head_dim=hd, d_ffn=ffn, n_layers=1)
    size = {tiny.d_model: d, 2 * tiny.d_model: 2 * d, tiny.d_ffn: ffn}

    def zeros(a):
        return [zeros(x) for x in a] if isinstance(a, list) else np.zeros([size.get(n, n) for n in a.shape], dtype=np.uint16)

    w = {k: zeros(v[:1] if isinstance(v, list) else v) for k, v in si.make_weights(tiny).items()}
    w["final_norm"][:] = 0x3F80
    w["embed"] = si.normal_bf16(5, "order", (sh.vocab, d))
    w["embed"][:, 0] = 0x3F80
    ids = si.uniform_ids(7, "order", 48, sh.vocab)
    e = Engine(sh, w, kv_capacity=512)
    try:
        e.prefill(0, ids)
        got = e.ada_debug_buffer(0, torch.float32, (1, 512, d))[0, :48, 0].clone()
    finally:
        e.close()
    h = si.bf16_bits_to_f32(w["embed"][ids])
    widest = max(sh.vocab, ffn, 3 * d) * d * 2
    ctas = min(torch.cuda.get_device_properties(0).multi_processor_count, max(64, widest >> 15)) & ~1
    assert width == -(-d // (ctas // 2 if pairs else ctas))     # (the width of a thread block's columns at this size)
    s = np.array([_pass_row_sum(h[t] * h[t], t, width, ctas, pairs) for t in range(48)])
    want = torch.rsqrt(torch.from_numpy(s / np.float32(d) + np.float32(sh.rms_eps)).to(e.dev))
    assert torch.equal(got, want), int((got != want).sum())
