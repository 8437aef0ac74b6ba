"""The backbone translators' scan in one launch, at the edges of its tiles, chunks and
attention blocks: against the fp64 oracle, and against the staged schedule (which runs
while profiling of the stages is enabled) bit for bit."""
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

W = synth.Workload
# name: (source heads P, d_s, target heads, d_t, E, top_k, lengths, (window start, slots, 128, heads, d_f))
SHAPES = {
    "p5_ds128_dh16": (5, 128, 3, 32, 1, 0, (26, 25, 1), (0, 2, 128, 8, 128)),    # one FFN chunk, 3-token blocks
    "p16_dh64": (16, 64, 2, 64, 2, 1, (8, 9, 17), (1, 3, 128, 2, 256)),           # whole 16-row blocks, two chunks
    "p7_dh32": (7, 64, 4, 32, 3, 0, (18, 19, 37), (0, 2, 128, 4, 768)),           # 126 rows, six chunks
    "p1_dh16": (1, 128, 2, 32, 2, 0, (127, 128, 129), (2, 1, 128, 8, 512)),       # 16-token blocks, one slot
    "p9_top1": (9, 64, 2, 128, 4, 1, (14, 15, 0, 29), (0, 4, 128, 4, 1024)),      # 9 of 16 rows, shorter ring
}


def _run(wl, sk, sv, blob, staged=False):
    h = M.mot_create_bt(*M.bt_config_from(wl))
    M.mot_load_weights(h, blob)
    M.mot_profile_enable(h, staged)
    k, v = G.to_device(wl, sk), G.to_device(wl, sv)
    (bk, dk), (bv, dv) = G.alloc_dst(wl), G.alloc_dst(wl)
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    c0 = M.mot_get_launch_count(h)
    M.mot_translate_bt(h, k, v, lens, wl.batch, dk, dv)
    assert M.mot_get_device_status(h) == M.MOT_OK
    return dk, dv, M.mot_get_launch_count(h) - c0


def _workload(name):
    P, ds, ht, dt, e, top_k, lens, bt = SHAPES[name]
    return W(name, 3, P, ds, 5, ht, dt, e, 0, len(lens), max(lens), "bf16", lens, top_k=top_k, bt=bt)


def _inputs(wl, seed):
    return synth.gen_cache(wl, 0, seed), synth.gen_cache(wl, 1, seed), synth.gen_weights(wl, seed)


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_scan_matches_oracle(name):
    wl = _workload(name)
    sk, sv, blob = _inputs(wl, 5)
    dk, dv, launches = _run(wl, sk, sv, blob)
    sdk, sdv, staged = _run(wl, sk, sv, blob, staged=True)
    assert launches < staged
    tb, ts = zip(*[(b, s) for b, n in enumerate(wl.seq_lens) for s in range(n)])
    tb, ts = np.array(tb), np.array(ts)
    ref = oracle.bt_tokens(wl, sk, sv, blob, tb, ts)
    if 0 < wl.top_k < wl.n_translators:   # tokens whose two best scores nearly tie may go either way
        g = oracle.bt_tokens(wl.replace(top_k=0), sk, sv, blob, tb, ts, want_gate=True)[1]
        top = np.sort(g, axis=2)
        clear = top[:, :, -1] - top[:, :, -2] > 1e-4
    else:
        clear = np.ones((2, tb.size), dtype=bool)
    win = set(wl.bt_window)
    for X, (dst, other) in enumerate(((dk, sdk), (dv, sdv))):
        got = dst.double().cpu().numpy()
        for r, l in enumerate(wl.bt_window):
            rows = got[l][tb, :, ts].reshape(tb.size, -1)
            G.assert_parity(wl, rows[clear[X]], ref[r][X][clear[X]], f"{name} X={X} slot {r}")
        # what is written is exactly what the staged schedule writes
        s = G.sentinel_value(wl)
        assert torch.equal(G.int_view(dst) == s, G.int_view(other) == s)
        for l in range(wl.n_layers_tgt):
            if l not in win:
                assert bool((G.int_view(dst)[l] == s).all())


# more edges: tokens of one row, of two with a longer window, of three and of 13 (one row stays alone)
SAME = dict(SHAPES, **{
    "p2_dh32": (2, 64, 2, 32, 2, 1, (65, 64, 1), (0, 8, 128, 4, 256)),
    "p13_dh64": (13, 128, 2, 32, 2, 0, (9, 10), (1, 3, 128, 2, 128)),
    "p3_dh16": (3, 64, 4, 32, 3, 1, (43, 42, 85), (0, 4, 128, 8, 512)),
    "p1_dh64": (1, 64, 2, 64, 1, 0, (128, 200), (0, 3, 128, 2, 2048)),
})


@pytest.mark.parametrize("seed", [1, 2])
@pytest.mark.parametrize("name", sorted(SAME))
def test_scan_equals_the_staged_kernels_bit_for_bit(name, seed):
    """The same fp32 sums in the same order, rounded to bf16 at the same places."""
    P, ds, ht, dt, e, top_k, lens, bt = SAME[name]
    wl = W(name, 3, P, ds, bt[0] + bt[1] + 1, ht, dt, e, 0, len(lens), max(lens), "bf16", lens, top_k=top_k, bt=bt)
    ins = _inputs(wl, seed)
    scan, staged = _run(wl, *ins), _run(wl, *ins, staged=True)
    assert scan[2] < staged[2]
    for a, b in zip(scan[:2], staged[:2]):
        assert torch.equal(G.int_view(a), G.int_view(b))


def test_scan_keeps_non_finite_tokens_apart():
    """A NaN or infinity in one token's rows makes that token's outputs NaN and leaves every
    other token as it was, also those that share its attention blocks."""
    wl = _workload("p5_ds128_dh16")
    sk, sv, blob = _inputs(wl, 7)
    clean = _run(wl, sk, sv, blob)
    bad = [(0, 3, 0x7FC0), (0, 4, 0x7F80), (1, 24, 0xFF80), (2, 0, 0x7FC0)]
    sk2, sv2 = sk.copy(), sv.copy()
    for b, s, bits in bad:
        for l in range(wl.n_layers_src):
            sk2[l, b, 2, s, 17] = bits
            sv2[l, b, 4, s, 90] = bits
    dirty = _run(wl, sk2, sv2, blob)
    staged = _run(wl, sk2, sv2, blob, staged=True)
    for c, x, y in zip(clean[:2], dirty[:2], staged[:2]):
        for l in wl.bt_window:
            for b, n in enumerate(wl.seq_lens):
                for s in range(n):
                    if any((b, s) == (bb, ss) for bb, ss, _ in bad):
                        assert torch.isnan(x[l, b, :, s].float()).all()
                        assert torch.isnan(y[l, b, :, s].float()).all()
                    else:
                        assert torch.equal(G.int_view(c[l, b, :, s]), G.int_view(x[l, b, :, s]))


def test_no_room_for_every_slot_runs_the_staged_kernels():
    """Where the state rows of all slots (553 MB here) do not fit but those of one slot and of the stages
    do (about 440 MB with the weights), the handle is created all the same and a call runs the staged
    schedule: its launches, and its output bit for bit."""
    lens = (40, 7)
    wl = W("bt_room", 1, 16, 64, 16, 2, 32, 2, 0, 2, 1024, "bf16", lens, bt=(0, 16, 128, 4, 128))
    sk, sv, blob = _inputs(wl, 11)
    want = _run(wl, sk, sv, blob, staged=True)
    k, v = G.to_device(wl, sk), G.to_device(wl, sv)
    (_, dk), (_, dv) = G.alloc_dst(wl), G.alloc_dst(wl)
    lens_d = torch.tensor(lens, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    held = torch.empty(free - (500 << 20), dtype=torch.uint8, device="cuda")
    left = torch.cuda.mem_get_info()[0]
    if not 480 << 20 < left < 520 << 20:
        pytest.skip("the GPU's memory is in use elsewhere")
    try:
        h = M.mot_create_bt(*M.bt_config_from(wl))
    except M.MotError:
        if torch.cuda.mem_get_info()[0] < left - (8 << 20):
            pytest.skip("the GPU's memory is in use elsewhere")
        raise
    del held
    torch.cuda.empty_cache()
    M.mot_load_weights(h, blob)
    c0 = M.mot_get_launch_count(h)
    M.mot_translate_bt(h, k, v, lens_d, wl.batch, dk, dv)
    assert M.mot_get_device_status(h) == M.MOT_OK
    assert M.mot_get_launch_count(h) - c0 == want[2]
    assert torch.equal(G.int_view(dk), G.int_view(want[0]))
    assert torch.equal(G.int_view(dv), G.int_view(want[1]))


@pytest.mark.parametrize("top_k", [0, 1])
def test_profile_of_the_launches_and_of_the_stages(top_k):
    """Profiling as launched times the kernels that an ordinary call runs; the stages' rows are only
    there once their times are asked for."""
    wl = W("bt_prof", 2, 16, 64, 2, 2, 32, 2, 0, 2, 1024, "bf16", (40, 7), top_k=top_k, bt=(0, 2, 128, 4, 128))
    sk, sv, blob = _inputs(wl, 17)
    want = _run(wl, sk, sv, blob)
    torch.cuda.synchronize()
    k, v = G.to_device(wl, sk), G.to_device(wl, sv)
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    (_, dk), (_, dv) = G.alloc_dst(wl), G.alloc_dst(wl)
    rows = 2 * wl.n_translators * 2 * 1024 * 16        # [K/V][E][B][S][P]
    free = torch.cuda.mem_get_info()[0]
    h = M.mot_create_bt(*M.bt_config_from(wl))
    M.mot_load_weights(h, blob)
    used = free - torch.cuda.mem_get_info()[0]
    assert used < rows * 2 * (2 * 128 + 8) + (64 << 20)   # state rows and statistics of both slots
    for level, names in ((M.PROFILE_AS_LAUNCHED, {"bt_gate", "bt_scan", "bt_out_all_slots"}),
                         (M.PROFILE_STAGES, {"bt_gate", "bt_in_ln_gelu", "bt_q", "bt_kv", "bt_attn",
                                             "bt_o_residual_ln", "bt_ffn_fused", "bt_out_gelu_combine"})):
        M.mot_profile_enable(h, level)
        c0 = M.mot_get_launch_count(h)
        M.mot_translate_bt(h, k, v, lens, wl.batch, dk, dv)
        prof = M.mot_profile_read(h)
        routed = {"bt_route"} | ({"bt_pack"} if level == M.PROFILE_STAGES else set()) if top_k else set()
        assert {n for n, (launches, _) in prof.items() if launches} == names | routed
        assert sum(launches for launches, _ in prof.values()) == M.mot_get_launch_count(h) - c0
        if level == M.PROFILE_AS_LAUNCHED:
            assert M.mot_get_launch_count(h) - c0 == want[2]
        assert torch.equal(G.int_view(dk), G.int_view(want[0]))
        assert torch.equal(G.int_view(dv), G.int_view(want[1]))
    assert free - torch.cuda.mem_get_info()[0] > used + rows * 128 * 20
    M.mot_destroy(h)


@pytest.mark.parametrize("top_k", [0, 1])
@pytest.mark.parametrize("staged", [False, True])
def test_output_rows_at_either_alignment(top_k, staged):
    """Targets that start 16 bytes past a 32-byte boundary get the same bits (16-byte stores),
    and nothing around them is written."""
    wl = W("bt_lead", 2, 3, 64, 3, 3, 32, 2, 0, 2, 70, "bf16", (70, 33), top_k=top_k, bt=(0, 2, 128, 4, 128))
    sk, sv, blob = _inputs(wl, 13)
    want = _run(wl, sk, sv, blob, staged)
    h = M.mot_create_bt(*M.bt_config_from(wl))
    M.mot_load_weights(h, blob)
    M.mot_profile_enable(h, staged)
    k, v = G.to_device(wl, sk), G.to_device(wl, sv)
    (bk, dk), (bv, dv) = G.alloc_dst(wl, 8), G.alloc_dst(wl, 8)
    assert dk.data_ptr() % 32 == 16 and want[0].data_ptr() % 32 == 0
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    M.mot_translate_bt(h, k, v, lens, wl.batch, dk, dv)
    assert M.mot_get_device_status(h) == M.MOT_OK
    for buf, got, ref in ((bk, dk, want[0]), (bv, dv, want[1])):
        assert torch.equal(G.int_view(got), G.int_view(ref))
        s = G.sentinel_value(wl)
        assert bool((G.int_view(buf[:8]) == s).all()) and bool((G.int_view(buf[8 + got.numel():]) == s).all())
