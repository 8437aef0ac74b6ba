"""Replay attention (App. C.4) on the GPU through the C ABI, against the fp64
oracle: the Top-S selection bit for bit, the attention within the bf16 bar."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import _gpu as G   # noqa: E402
M = G.M

RW = synth.ReplayWorkload
SMALL = {
    # GQA 12 / 2, d = 128, S = 16 (short rows below S), ragged batch
    "r_gqa6_d128": RW("r_gqa6_d128", 6, 7, 12, 2, 128, 2, 300, (300, 131), top_s=16, n_full=2),
    # no GQA, d = 64, the paper's S = 128 with rows shorter and longer than S
    "r_mha_d64": RW("r_mha_d64", 4, 4, 4, 4, 64, 3, 400, (400, 128, 129), top_s=128, n_full=1),
    # 16 query heads per key/value head, one long row per entry
    "r_gqa16": RW("r_gqa16", 2, 2, 16, 1, 64, 1, 1000, (1000,), top_s=64, n_full=1),
    # d = 128 on the tensor-core guided kernel: S = 128, 16 heads per group, ragged rows
    "r_gqa16_d128": RW("r_gqa16_d128", 2, 4, 16, 1, 128, 3, 520, (520, 127, 129), top_s=128,
                       n_full=1),
    # d = 128, no GQA, an S that is not a multiple of 4 (partial gather4 groups)
    "r_mha_d128_s99": RW("r_mha_d128_s99", 2, 4, 3, 3, 128, 2, 333, (333, 98), top_s=99, n_full=1),
}


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda()


class ReplayRun:
    def __init__(self, wl, seq=None, batch=None):
        self.wl = wl
        self.h = M.mot_create_replay(M.replay_config_from(wl))
        self.seq = list(wl.seq_lens if seq is None else seq)
        self.batch = len(self.seq) if batch is None else batch
        self.lens = torch.tensor(self.seq, dtype=torch.int32, device="cuda")

    def select(self, g):
        sel = torch.full((self.wl.max_batch, self.wl.max_seq, self.wl.top_s), -7,
                         dtype=torch.int32, device="cuda")
        M.mot_replay_select(self.h, _dev(g), self.lens, self.batch, sel)
        torch.cuda.synchronize()
        return sel.cpu().numpy()

    def attend(self, layer, q, k, v, g):
        out = torch.full((self.wl.max_batch, self.wl.q_heads, self.wl.max_seq, self.wl.head_dim),
                         G.SENTINEL_BF16, dtype=torch.int16, device="cuda")
        M.mot_replay_attention(self.h, layer, _dev(q), _dev(k), _dev(v),
                               None if g is None else _dev(g), self.lens, self.batch, out)
        torch.cuda.synchronize()
        return out


BF16 = synth.WORKLOADS["gpt2s_opt125m"]   # carries the bf16 tolerance of the parity bar


def _f64(bits_t):
    return bits_t.view(torch.bfloat16).double().cpu().numpy()


@pytest.mark.parametrize("name", sorted(SMALL))
def test_selection_is_bit_exact_on_every_row(name):
    wl = SMALL[name]
    g = synth.gen_guide(wl, 3)
    run = ReplayRun(wl)
    sel = run.select(g)
    for b, L in enumerate(wl.seq_lens):
        for u in range(L):
            ref = oracle.replay_select(wl, g, b, u)
            row = sel[b, u]
            np.testing.assert_array_equal(row[:ref.size], ref, err_msg=f"b={b} u={u}")
            assert (row[ref.size:] == -1).all()
        assert (sel[b, L:] == -7).all()   # rows past the sequence are not written


@pytest.mark.parametrize("name", ["r_gqa6_d128", "r_mha_d64"])   # max_seq 300 and 400: scalar and 16-byte loads
def test_selection_ties_and_constant_rows(name):
    wl = SMALL[name].replace(top_s=8)
    N = wl.max_seq
    g = np.zeros((wl.max_batch, N, N), dtype=np.uint16)
    g[0] = 0x4000                                  # every score 2.0: the lowest positions win
    rng = np.random.default_rng(0)
    g[1] = (0x3F80 + rng.integers(0, 3, size=(N, N))).astype(np.uint16)   # three values only
    if wl.batch > 2:   # mixed signs (no exact zeros: -0 and +0 order apart in the 16-bit keys)
        x = rng.standard_normal((N, N)).astype(np.float32)
        g[2] = (x.view(np.uint32) >> 16).astype(np.uint16)
    run = ReplayRun(wl)
    sel = run.select(g)
    for b, L in enumerate(wl.seq_lens):
        for u in range(0, L, 7):
            ref = oracle.replay_select(wl, g, b, u)
            np.testing.assert_array_equal(sel[b, u, :ref.size], ref)


@pytest.mark.parametrize("span", [1, 255, 256, 257, 511, 512, 4097, 0x7EFF])
def test_selection_across_key_ranges(span):
    """Rows whose 16-bit keys span `span` values: the histogram digit's width
    follows the row's range, so spans around 2^8 and 2^9 take the one-pass and
    two-pass cases and their boundary."""
    wl = SMALL["r_mha_d64"].replace(top_s=32)
    N = wl.max_seq
    rng = np.random.default_rng(span)
    base = 0x3C00 if span < 0x4000 else 0x0080        # positive bf16 bit patterns, no NaN or Inf
    g = (base + rng.integers(0, span + 1, size=(wl.max_batch, N, N))).astype(np.uint16)
    g[:, :, 0] = base                                   # the range's ends are present
    g[:, :, 1] = base + span
    run = ReplayRun(wl)
    sel = run.select(g)
    for b, L in enumerate(wl.seq_lens):
        for u in range(0, L, 5):
            ref = oracle.replay_select(wl, g, b, u)
            np.testing.assert_array_equal(sel[b, u, :ref.size], ref, err_msg=f"b={b} u={u}")


@pytest.mark.parametrize("max_seq", [4104, 4099])   # 16-byte and scalar loads
def test_selection_rows_longer_than_the_key_cache(max_seq):
    """Rows past 4,096 positions take the streaming selection (the row read once per pass)."""
    wl = RW("r_long", 2, 2, 4, 1, 64, 1, max_seq, (max_seq,), top_s=128, n_full=1)
    g = synth.gen_guide(wl, 13)
    sel = ReplayRun(wl).select(g)
    rng = np.random.default_rng(max_seq)
    for u in np.unique(np.concatenate([[0, 127, 128, 4095, 4096, max_seq - 1],
                                       rng.integers(129, max_seq, size=40)])):
        ref = oracle.replay_select(wl, g, 0, int(u))
        np.testing.assert_array_equal(sel[0, u, :ref.size], ref, err_msg=f"u={u}")


@pytest.mark.parametrize("name", sorted(SMALL))
def test_attention_matches_oracle(name):
    wl = SMALL[name]
    q, k, v = synth.gen_replay_qkv(wl, 1)
    g = synth.gen_guide(wl, 5)
    run = ReplayRun(wl)
    rng = np.random.default_rng(7)
    for layer in (0, wl.n_full, wl.n_full + 3):
        out = run.attend(layer, q, k, v, None if layer < wl.n_full else g)
        tb, th, tu = [], [], []
        for b, L in enumerate(wl.seq_lens):
            us = np.unique(np.concatenate([[0, 1, L - 1, min(L - 1, wl.top_s), min(L - 1, wl.top_s - 1)],
                                           rng.integers(0, L, size=20)]))
            for u in us:
                for h in rng.choice(wl.q_heads, size=min(4, wl.q_heads), replace=False):
                    tb.append(b); th.append(h); tu.append(u)
        ref = oracle.replay_tokens(wl, layer, q, k, v, g, tb, th, tu)
        got = _f64(out)[tb, th, tu]
        G.assert_parity(BF16, got, ref, f"{name} layer {layer}")
        o = out.cpu().numpy()
        for b, L in enumerate(wl.seq_lens):
            assert (o[b, :, L:] == np.int16(G.SENTINEL_BF16)).all()


@pytest.mark.parametrize("group", [2, 3, 4, 5, 7, 8, 12])
def test_guided_attention_every_group_size(group):
    """The tensor-core guided kernel is instantiated per GQA group size G (the
    query heads of one key/value head): a guided layer with d = 128 and S = 128
    for each G the other tests do not reach, sampled against the oracle."""
    kv = 2 if group <= 4 else 1
    wl = RW(f"r_g{group}", 2, 3, group * kv, kv, 128, 2, 264, (264, 131), top_s=128, n_full=1)
    q, k, v = synth.gen_replay_qkv(wl, 17)
    g = synth.gen_guide(wl, 19)
    run = ReplayRun(wl)
    out = run.attend(2, q, k, v, g)
    rng = np.random.default_rng(group)
    tb, th, tu = [], [], []
    for b, L in enumerate(wl.seq_lens):
        us = np.unique(np.concatenate([[0, 127, 128, L - 1], rng.integers(0, L, size=12)]))
        for u in us:
            for h in range(wl.q_heads):
                tb.append(b); th.append(h); tu.append(u)
    ref = oracle.replay_tokens(wl, 2, q, k, v, g, tb, th, tu)
    G.assert_parity(BF16, _f64(out)[tb, th, tu], ref, f"group {group}")
    o = out.cpu().numpy()
    for b, L in enumerate(wl.seq_lens):
        assert (o[b, :, L:] == np.int16(G.SENTINEL_BF16)).all()


@pytest.mark.parametrize("gain", [0.05, 2.0])
def test_attention_scores_rising_along_the_context(gain):
    """Keys that grow along a common direction of the queries, so a query's scores
    rise with the key position by about `gain` (base 2) per key: the full-attention
    kernel's running max passes its 2^8 margin on later key tiles and rescales O
    and the row sum (gain 0.05: every tile or two by a moderate factor; gain 2:
    every tile, the earlier keys' weight vanishing), and the guided kernel sees
    rows whose selected scores span hundreds of binades. Against the oracle."""
    import _helpers as H
    wl = RW("r_rise", 2, 3, 12, 2, 128, 2, 520, (520, 300), top_s=128, n_full=1)
    q, k, v = synth.gen_replay_qkv(wl, 23)
    g = synth.gen_guide(wl, 29)
    # q . k / sqrt(d) = 128 (gain j / 16) / sqrt(128) ~ 0.7 gain j, about gain j in base 2
    qf = 0.25 * H.bf16_bits_to_f64(q) + 1.0
    j = np.arange(wl.max_seq, dtype=np.float64)[None, None, :, None]
    kf = 0.25 * H.bf16_bits_to_f64(k) + gain * j / 16.0
    q = H.f32_to_bf16_bits(qf.astype(np.float32))
    k = H.f32_to_bf16_bits(kf.astype(np.float32))
    run = ReplayRun(wl)
    rng = np.random.default_rng(31)
    for layer in (0, 2):
        out = run.attend(layer, q, k, v, None if layer < wl.n_full else g)
        tb, th, tu = [], [], []
        for b, L in enumerate(wl.seq_lens):
            us = np.unique(np.concatenate([[0, 127, 128, 255, 256, L - 1], rng.integers(0, L, size=10)]))
            for u in us:
                for h in range(wl.q_heads):
                    tb.append(b); th.append(h); tu.append(u)
        ref = oracle.replay_tokens(wl, layer, q, k, v, g, tb, th, tu)
        G.assert_parity(BF16, _f64(out)[tb, th, tu], ref, f"gain {gain} layer {layer}")


def test_full_size_layer_sampled():
    """Qwen2.5-0.5B -> 1.5B replay shapes (4 x 4096 context, 12 / 2 heads of 128,
    S = 128): one full and one guided layer, in the benchmark's launch configuration."""
    wl = synth.REPLAY_WORKLOADS["replay_qwen05_qwen15"]
    q, k, v = synth.gen_replay_qkv(wl, 2)
    g = synth.gen_guide(wl, 9)
    run = ReplayRun(wl)
    sel = run.select(g)
    rng = np.random.default_rng(11)
    # 256 selection rows per batch entry (both ends, the S boundary, a whole
    # 128-row block and random rows), each bit-exact
    for b in range(wl.batch):
        blk = 128 * int(rng.integers(1, 32))
        us = np.unique(np.concatenate([[0, 127, 128, 4095], np.arange(blk, blk + 128),
                                       rng.integers(0, 4096, size=124)]))
        for u in us:
            ref = oracle.replay_select(wl, g, b, int(u))
            np.testing.assert_array_equal(sel[b, u, :ref.size], ref)
    # 2048 queries per layer: a full layer, a guided layer and the last layer;
    # every query head of one whole 128-query tile of one batch entry included
    for layer in (1, 5, wl.n_layers_tgt - 1):
        out = run.attend(layer, q, k, v, g)
        t0 = 128 * int(rng.integers(0, 32))
        tile_h, tile_u = np.meshgrid(np.arange(wl.q_heads), np.arange(t0, t0 + 128), indexing="ij")
        n = 2048 - tile_h.size
        tb = np.concatenate([np.full(tile_h.size, 3), rng.integers(0, wl.batch, size=n)])
        th = np.concatenate([tile_h.ravel(), rng.integers(0, wl.q_heads, size=n)])
        tu = np.concatenate([tile_u.ravel(), [0, 4095], rng.integers(0, 4096, size=n - 2)])
        ref = oracle.replay_tokens(wl, layer, q, k, v, g, tb, th, tu)
        G.assert_parity(BF16, _f64(out)[tb, th, tu], ref, f"full-size layer {layer}")


def test_full_layers_use_the_tensor_core_kernel():
    """max_seq % 8 == 0: full layers run the tcgen05 attention kernel (after the V
    transpose); guided layers run the selection and the gather kernel."""
    wl = SMALL["r_mha_d64"]
    q, k, v = synth.gen_replay_qkv(wl, 0)
    g = synth.gen_guide(wl, 0)
    run = ReplayRun(wl)
    M.mot_profile_enable(run.h, True)
    run.attend(0, q, k, v, None)
    run.attend(2, q, k, v, g)
    prof = M.mot_profile_read(run.h)
    assert set(prof) == {"replay_vt", "replay_fmha_full", "replay_select", "replay_attn_sparse"}


def test_batch_prefix_and_errors():
    wl = SMALL["r_mha_d64"]
    q, k, v = synth.gen_replay_qkv(wl, 0)
    g = synth.gen_guide(wl, 0)
    run = ReplayRun(wl, batch=2)
    out = run.attend(3, q, k, v, g).cpu().numpy()
    assert (out[2] == np.int16(G.SENTINEL_BF16)).all()    # entry 2 is past `batch`
    dst = torch.empty(out.shape, dtype=torch.int16, device="cuda")
    with pytest.raises(M.MotError) as e:                   # a guided layer needs its map
        M.mot_replay_attention(run.h, 3, _dev(q), _dev(k), _dev(v), None, run.lens, 2, dst)
    assert e.value.status == M.MOT_ERR_INVALID_ARG
    with pytest.raises(M.MotError) as e:
        M.mot_create_replay(M.replay_config_from(wl.replace(head_dim=96)))
    assert e.value.status == M.MOT_ERR_UNSUPPORTED
    with pytest.raises(M.MotError) as e:
        M.mot_create_replay(M.replay_config_from(wl.replace(kv_heads=3)))
    assert e.value.status == M.MOT_ERR_INVALID_ARG


def test_guided_timeout_is_reported_and_recovers():
    """Failure reporting without a fault: with the stall hook the guided kernel's
    first CTA waits for a signal that nothing sends, the wait runs out after the
    short limit, the CTA leaves and the status word reports a timeout. (The kernel
    itself waits for its own copies only, so this covers the report and the next
    call, not an unwinding pipeline.) The next guided layer on the same context
    matches the oracle."""
    wl = SMALL["r_gqa6_d128"]
    q, k, v = synth.gen_replay_qkv(wl, 3)
    g = synth.gen_guide(wl, 6)
    run = ReplayRun(wl)
    layer = wl.n_full + 1
    M.mot_debug_set(run.h, True, 20_000_000)        # about 10 ms of SM cycles
    run.attend(layer, q, k, v, g)
    assert M.mot_get_device_status(run.h) == M.MOT_ERR_TIMEOUT
    assert M.mot_get_device_status(run.h) == M.MOT_OK   # reading cleared it
    M.mot_debug_set(run.h, False, 0)
    out = run.attend(layer, q, k, v, g)
    assert M.mot_get_device_status(run.h) == M.MOT_OK
    rng = np.random.default_rng(5)
    tb, th, tu = [], [], []
    for b, L in enumerate(wl.seq_lens):
        for u in np.unique(np.concatenate([[0, L - 1], rng.integers(0, L, size=12)])):
            for h in rng.choice(wl.q_heads, size=3, replace=False):
                tb.append(b); th.append(h); tu.append(u)
    ref = oracle.replay_tokens(wl, layer, q, k, v, g, tb, th, tu)
    G.assert_parity(BF16, _f64(out)[tb, th, tu], ref, "guided layer after a timeout")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("group,top_s,n", [(1, 1, 70), (4, 31, 130), (5, 32, 131), (8, 33, 99), (6, 64, 201),
                                           (3, 65, 200), (16, 127, 260), (2, 129, 333), (7, 192, 257),
                                           (12, 200, 333)])
def test_gathered_rows_every_unit_size(d, group, top_s, n):
    """The gather kernel at the edges of its units (32, 64 or 128 rows, 64 for larger sets),
    in every form of the probabilities (group sizes up to 4, 8 and 16), with a context that
    is not a multiple of 8 so that the full layer takes it too. Against the oracle, with
    the parity bar of the other replay tests."""
    wl = RW(f"r_u{top_s}", 2, 3, group * 2, 2, d, 2, n, (n, n // 2 + 1), top_s=top_s, n_full=1)
    if n % 8 == 0:
        wl = wl.replace(max_seq=n + 1)
    q, k, v = synth.gen_replay_qkv(wl, 37)
    g = synth.gen_guide(wl, 41)
    run = ReplayRun(wl)
    rng = np.random.default_rng(top_s)
    for layer in (0, 2):
        out = run.attend(layer, q, k, v, None if layer < wl.n_full else g)
        tb, th, tu = [], [], []
        for b, L in enumerate(wl.seq_lens):
            edge = [x for x in (0, 15, 16, 63, 64, top_s - 1, top_s, L - 1) if x < L]
            for u in np.unique(np.concatenate([edge, rng.integers(0, L, size=8)])):
                for h in range(wl.q_heads):
                    tb.append(b); th.append(h); tu.append(int(u))
        ref = oracle.replay_tokens(wl, layer, q, k, v, g, tb, th, tu)
        G.assert_parity(BF16, _f64(out)[tb, th, tu], ref, f"d {d} group {group} S {top_s} layer {layer}")
        o = out.cpu().numpy()
        for b, L in enumerate(wl.seq_lens):
            assert (o[b, :, L:] == np.int16(G.SENTINEL_BF16)).all()


@pytest.mark.parametrize("max_seq", [257, 263, 520, 1030, 2049, 4093])   # every 16-byte phase of a row start
@pytest.mark.parametrize("top_s", [1, 128, 160, 161, 256, 416, 417, 449])
def test_selection_bounds_lists_and_fallback(max_seq, top_s):
    """The bounded selection against numpy, bit for bit: one or two sets of group maxima
    (top_s up to 160 and 416) and the histogram past them; rows whose candidates overflow
    the list (a few values only), rows of distinct scores, mixed signs, and rows holding the
    lowest key (a negative NaN pattern), whose bound cannot separate it from empty slots."""
    wl = RW("r_bound", 2, 2, 1, 1, 64, 2, max_seq, (max_seq, max_seq - 3), top_s=top_s, n_full=1)
    rng = np.random.default_rng(max_seq * 1000 + top_s)
    N = max_seq
    g = rng.integers(0x0080, 0x7F00, size=(2, N, N)).astype(np.uint16)
    g[0, 1::6] = rng.integers(0x3F80, 0x3F84, size=g[0, 1::6].shape).astype(np.uint16)
    g[0, 2::6] = (np.exp(rng.standard_normal(g[0, 2::6].shape)).astype(np.float32).view(np.uint32) >> 16)
    g[0, 3::6] = (rng.standard_normal(g[0, 3::6].shape).astype(np.float32).view(np.uint32) >> 16)
    g[0, 4::6] = np.where(rng.random(g[0, 4::6].shape) < 0.9, 0xFFFF, 0x3F80)
    g[0, 5::6] = np.where(rng.random(g[0, 5::6].shape) < 0.5, 0, 0x3F80)
    g[1, 1::3] = rng.integers(0, 0x0100, size=g[1, 1::3].shape)      # subnormals
    g[1, 2::3, 5::64] = rng.choice([0x7F80, 0x7FC0, 0x8000], size=g[1, 2::3, 5::64].shape)
    sel = ReplayRun(wl).select(g)
    for b, L in enumerate(wl.seq_lens):
        for u in np.unique(np.concatenate([[0, top_s - 1, top_s, 255, 256, L - 1],
                                           rng.integers(0, L, size=60)])):
            if u >= L:
                continue
            bits = g[b, u, :u + 1].astype(np.int64)
            key = np.where(bits >= 0x8000, 0xFFFF - bits, bits | 0x8000)
            ref = np.sort(np.lexsort((np.arange(u + 1), -key))[:top_s])
            np.testing.assert_array_equal(sel[b, u, :ref.size], ref, err_msg=f"b={b} u={u}")
            assert (sel[b, u, ref.size:] == -1).all()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("group,top_s,n", [(1, 128, 99), (2, 64, 63), (4, 128, 99), (6, 128, 99), (16, 128, 99),
                                           (1, 256, 201), (2, 256, 201), (3, 256, 201), (7, 256, 201),
                                           (12, 256, 201)])
def test_probabilities_keep_fp32(d, group, top_s, n):
    """Values +1 and -1 on neighbouring keys that score almost alike: what is left of the weights is
    about 1e-5, so an error of the weights shows. Sets of more than 128 rows, sets of 64-wide heads
    and full layers of a context that is not a multiple of 8 keep fp32 weights. With n keys of weight
    1 / n, fp32 weights are off by about 2^-24 / sqrt(n) (rms) and a sum of two bf16 by 2^-18.8 /
    sqrt(n), which is 2.2e-7 at n = 99; the bound is 2^-24 beside the output's own rounding (2^-9)."""
    import _helpers as H
    wl = RW("r_cancel", 2, 3, group, 1, d, 1, n, (n,), top_s=top_s, n_full=1)
    rng = np.random.default_rng(group + n)
    q = rng.standard_normal((1, group, n, d)).astype(np.float32)
    k = rng.standard_normal((1, 1, n, d)).astype(np.float32) * 0.25
    k[:, :, 1::2] = k[:, :, 0:n - 1:2]
    q[..., 0] *= 2.0 ** -10
    k[:, :, 1::2, 0] += 0.25
    v = np.ones((1, 1, n, d), np.float32)
    v[:, :, 1::2] = -1.0
    v *= 1.0 + np.arange(d, dtype=np.float32) / 64 % 1
    bits = [H.f32_to_bf16_bits(x) for x in (q, k, v)]
    g = synth.gen_guide(wl, 3)
    run = ReplayRun(wl)
    us = np.arange(31, n, 2)   # whole pairs of keys
    for layer in (0, 1) if d == 64 or top_s > 128 else (0,):   # 0: full; 1: guided, over 0..u (u < top_s)
        got = _f64(run.attend(layer, *bits, None if layer == 0 else g))[0][:, us]
        qd, kd, vd = (H.bf16_bits_to_f64(x)[0] for x in bits)
        s = np.einsum("hud,jd->huj", qd[:, us], kd[0]) / np.sqrt(d)
        s[:, np.arange(n)[None] > us[:, None]] = -np.inf
        p = np.exp(s - s.max(2, keepdims=True))
        ref = np.einsum("huj,jd->hud", p / p.sum(2, keepdims=True), vd[0])
        rms = lambda x: float(np.sqrt(np.mean(x * x)))
        assert 1e-6 < rms(ref) < 1e-4
        assert rms(got - ref) <= 2.0 ** -9 * rms(ref) + 2.0 ** -24, (layer, rms(got - ref), rms(ref))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("group,top_s,n", [(1, 100, 131), (2, 40, 67), (4, 200, 261), (6, 128, 195), (12, 130, 197)])
def test_infinities_and_nans(d, group, top_s, n):
    """An infinity in a value row makes infinite what takes the row with a positive weight, in its
    dimension, and nothing else; a key whose score is -inf takes no part, also where whole units of
    keys score -inf; +inf and NaN scores, and infinities of both signs, give NaN. Every query of a
    full layer (n not a multiple of 8) and of a guided layer against the same in numpy."""
    import _helpers as H
    wl = RW("r_inf", 2, 3, group, 1, d, 1, n, (n,), top_s=top_s, n_full=1)
    q, k, v = synth.gen_replay_qkv(wl, 43)
    g = synth.gen_guide(wl, 47)
    q[..., 0] &= 0x7FFF
    q[..., 1] &= 0x7FFF
    q[0, 0, n - 2:, 1] |= 0x8000       # one head's last queries meet k = -inf with a negative q
    run = ReplayRun(wl)
    sel = run.select(g)[0]
    cases = []
    k1, v1 = k.copy(), v.copy()
    v1[0, 0, [3, 60], 17] = 0x7F80     # +inf
    v1[0, 0, n // 2, 18] = 0xFF80      # -inf
    v1[0, 0, 5, 19], v1[0, 0, 9, 19] = 0x7F80, 0xFF80
    v1[0, 0, 20, 20] = 0x7FC0
    cases.append((k1, v1))
    k2, v2 = k.copy(), v.copy()
    k2[0, 0, 1:70, 0] = 0xFF80         # score -inf: more than the first unit of 64 but one key
    k2[0, 0, n - 1, 1] = 0xFF80
    cases.append((k2, v2))
    k3 = k2.copy()
    k3[0, 0, 0, 0] = 0xFF80            # the whole first unit
    cases.append((k3, v2))
    for layer in (0, 1):
        clean = run.attend(layer, q, k, v, None if layer == 0 else g).cpu().numpy()[0]
        for kk, vv in cases:
            out = run.attend(layer, q, kk, vv, None if layer == 0 else g)
            got, raw = _f64(out)[0], out.cpu().numpy()[0]
            qd, kd, vd = (H.bf16_bits_to_f64(x)[0] for x in (q, kk, vv))
            with np.errstate(invalid="ignore", over="ignore"):
                s = np.einsum("hud,jd->huj", qd, np.where(np.isinf(kd[0]), 0, kd[0])) / np.sqrt(d)
                for j, c in zip(*np.nonzero(np.isinf(kd[0]))):
                    s[:, :, j] += qd[:, :, c] * kd[0, j, c]
                for u in range(n):
                    at = np.arange(u + 1) if layer == 0 else sel[u][sel[u] >= 0]
                    p = np.exp(s[:, u, at] - s[:, u, at].max(1, keepdims=True))
                    ref = (p / p.sum(1, keepdims=True)) @ np.where(np.isfinite(vd[0, at]), vd[0, at], 0)
                    for i, c in zip(*np.nonzero(~np.isfinite(vd[0, at]))):
                        ref[:, c] += np.where(p[:, i] > 0, 1.0, np.nan) * vd[0, at[i], c]
                    x = got[:, u]
                    assert (np.isnan(x) == np.isnan(ref)).all(), u
                    assert (x[np.isinf(ref)] == ref[np.isinf(ref)]).all(), u
                    fin = np.isfinite(ref)
                    assert np.isfinite(x[fin]).all(), u
                    if kk is k1:       # scores as before: what is finite has the clean run's bits
                        assert (raw[:, u][fin] == clean[:, u][fin]).all(), u
                    elif fin.any():
                        G.assert_parity(BF16, x[fin], ref[fin], f"layer {layer} u {u}")


@pytest.mark.parametrize("kv,lens", [(5, (40, 0, 33)), (2, (40, 1, 17, 40)), (4, tuple(1 + 13 * b % 40 for b in range(30))),
                                     (7, tuple(40 - b % 3 for b in range(64)))])
@pytest.mark.parametrize("top_s", [24, 130])
def test_every_item_of_ragged_batches(kv, lens, top_s):
    """Items walk over positions and heads in passes of the grid's warps: whole positions, turning to
    the next head with each pass, or (many heads) any part of one. Every row inside its sequence, and
    no other, against numpy."""
    import _helpers as H
    n = 41
    wl = RW("r_items", 2, 3, kv, kv, 64, len(lens), n, lens, top_s=top_s, n_full=1)
    q, k, v = synth.gen_replay_qkv(wl, 53)
    g = synth.gen_guide(wl, 59)
    run = ReplayRun(wl)
    sel = run.select(g)
    qd, kd, vd = (H.bf16_bits_to_f64(x) for x in (q, k, v))
    for layer in (0, 2):
        out = run.attend(layer, q, k, v, None if layer == 0 else g)
        got, raw = _f64(out), out.cpu().numpy()
        s = np.einsum("bhud,bhjd->bhuj", qd, kd) / 8.0
        ref = np.zeros_like(got)
        for b, L in enumerate(lens):
            assert (raw[b, :, L:] == np.int16(G.SENTINEL_BF16)).all()
            for u in range(L):
                at = np.arange(u + 1) if layer == 0 else sel[b, u][sel[b, u] >= 0]
                p = np.exp(s[b, :, u, at] - s[b, :, u, at].max(0))
                ref[b, :, u] = np.einsum("jh,hjd->hd", p / p.sum(0), vd[b][:, at])
        inside = np.arange(n)[None] < np.array(lens)[:, None]
        rows = np.broadcast_to(inside[:, None], got.shape[:3])
        G.assert_parity(BF16, got[rows], ref[rows], f"layer {layer}")
