"""Kernels of one call that start before their predecessor has finished: each chain of
launches captured into a graph and replayed on inputs written in between, and run call after
call without a synchronisation, bit for bit as when every kernel is timed by itself (which
launches them one after another)."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import _gpu as G   # noqa: E402
M = G.M

W, RW = synth.Workload, synth.ReplayWorkload
SHAPES = {
    "pair": (W("c_pair", 3, 2, 64, 4, 2, 128, 2, 256, 4, 300, "bf16", (300, 129, 1)), M.SCHEDULE_PAIR),
    "onchip": (W("c_onchip", 2, 2, 64, 3, 2, 128, 3, 256, 2, 64, "bf16", (64, 33)), M.SCHEDULE_ONCHIP),
    "fp32": (W("c_fp32", 3, 2, 12, 2, 3, 10, 2, 50, 3, 90, "fp32", (90, 0, 65)), None),
    "fp32_scalar": (W("c_fp32s", 3, 2, 12, 2, 3, 10, 3, 33, 3, 90, "fp32", (90, 0, 65)), None),
    "routed": (W("c_routed", 2, 2, 64, 2, 2, 128, 4, 256, 2, 160, "bf16", (160, 33), top_k=2), None),
    "activations": (W("c_h", 3, 1, 128, 3, 2, 128, 3, 256, 2, 130, "bf16", (130, 7), act_tgt=256), None),
    "backbones": (W("c_bt", 3, 5, 64, 5, 3, 32, 2, 0, 2, 29, "bf16", (29, 14), top_k=1,
                    bt=(0, 3, 128, 8, 256)), None),
    "replay_full": (RW("c_full", 2, 2, 12, 2, 128, 2, 264, (264, 131), top_s=16, n_full=2), None),
    "replay_guided": (RW("c_guided", 2, 2, 12, 2, 128, 2, 263, (263, 131), top_s=64, n_full=1), None),
}


def _bf16(a):
    return torch.from_numpy(a.view("int16")).cuda()


def _chain(name):
    """(handle, inputs of two draws, input buffers, outputs, call(stream))."""
    wl, schedule = SHAPES[name]
    if isinstance(wl, RW):
        h = M.mot_create_replay(M.replay_config_from(wl))
        lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
        draws = [[_bf16(x) for x in (*synth.gen_replay_qkv(wl, s), synth.gen_guide(wl, s))] for s in (1, 2)]
        buf = [x.clone() for x in draws[0]]
        out = [torch.zeros(wl.max_batch, wl.q_heads, wl.max_seq, wl.head_dim, dtype=torch.int16,
                           device="cuda")]
        guided = name == "replay_guided"

        def call(st):
            M.mot_replay_attention(h, 1, buf[0], buf[1], buf[2], buf[3] if guided else None, lens,
                                   len(wl.seq_lens), out[0], st)
        return h, draws, buf, out, call
    act, bt = name == "activations", name == "backbones"
    h = (M.mot_create_h(M.h_config_from(wl)) if act else
         M.mot_create_bt(*M.bt_config_from(wl)) if bt else M.mot_create(M.config_from(wl)))
    M.mot_load_weights(h, synth.gen_weights(wl, 7))
    if schedule is not None:
        M.mot_set_schedule(h, schedule)
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    draws = [[G.to_device(wl, synth.gen_cache(wl, i, s)) for i in range(1 if act else 2)] for s in (1, 2)]
    buf = [x.clone() for x in draws[0]]
    (_, dk), (_, dv) = G.alloc_dst(wl), G.alloc_dst(wl)
    fn = M.mot_translate_h if act else M.mot_translate_bt if bt else M.mot_translate

    def call(st):
        fn(h, *buf, lens, len(wl.seq_lens), dk, dv, st)
    return h, draws, buf, [dk, dv], call


def _bits(out):
    return [G.int_view(t).clone() if t.is_floating_point() else t.clone() for t in out]


def _load(buf, draw):
    for b, x in zip(buf, draw):
        b.copy_(x)


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_chain_captured_and_back_to_back(name):
    h, draws, buf, out, call = _chain(name)
    st = torch.cuda.Stream()
    M.mot_profile_enable(h, M.PROFILE_AS_LAUNCHED)
    want = []
    with torch.cuda.stream(st):
        for d in draws:
            _load(buf, d)
            call(st)
            st.synchronize()
            want.append(_bits(out))
    M.mot_profile_enable(h, False)
    assert any(bool((a != b).any()) for a, b in zip(*want))
    got = []
    with torch.cuda.stream(st):
        for i in (1, 0, 1, 0, 0, 1):
            _load(buf, draws[i])
            call(st)
            got.append((i, _bits(out)))
    st.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        call(st)
    with torch.cuda.stream(st):
        for i in (1, 0, 0, 1):
            _load(buf, draws[i])
            graph.replay()
            got.append((i, _bits(out)))
    st.synchronize()
    for i, o in got:
        assert all(bool((a == b).all()) for a, b in zip(o, want[i]))
    assert name.startswith("replay") or M.mot_get_device_status(h) == M.MOT_OK


def test_a_full_layer_behind_an_empty_one():
    """A full-attention call whose sequences are all empty, directly followed by an ordinary one on the
    same handle: the second transposes V into the workspace that the first's transpose still writes if
    the first's attention grid is complete too early."""
    wl = SHAPES["replay_full"][0].replace(max_seq=2048, seq_lens=(2048, 1300))
    h = M.mot_create_replay(M.replay_config_from(wl))
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    none = torch.zeros_like(lens)
    a, b = [[_bf16(x) for x in synth.gen_replay_qkv(wl, s)] for s in (1, 2)]
    want = torch.zeros(wl.max_batch, wl.q_heads, wl.max_seq, wl.head_dim, dtype=torch.int16, device="cuda")
    M.mot_replay_attention(h, 0, *b, None, lens, 2, want)
    torch.cuda.synchronize()
    outs = [torch.zeros_like(want) for _ in range(20)]
    untouched = torch.full_like(want, 7)
    for o in outs:
        M.mot_replay_attention(h, 0, *a, None, none, 2, untouched)
        M.mot_replay_attention(h, 0, *b, None, lens, 2, o)
    torch.cuda.synchronize()
    assert bool((untouched == 7).all()) and bool((want != 0).any())
    for o in outs:
        assert torch.equal(o, want)
