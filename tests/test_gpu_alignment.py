"""Targets that start 16 bytes past a 32-byte boundary: the GEMM epilogues then store 16-byte
pieces instead of whole 32-byte sectors, the same bits, and nothing around the targets."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import _gpu as G   # noqa: E402
M = G.M

W = synth.Workload
SHAPES = {
    "pair": (W("al_pair", 2, 2, 64, 3, 4, 64, 2, 256, 2, 140, "bf16", (140, 1)), M.SCHEDULE_PAIR),
    "split": (W("al_split", 2, 2, 64, 3, 8, 32, 2, 256, 2, 140, "bf16", (140, 1)), M.SCHEDULE_SPLIT),
    "top1": (W("al_top1", 2, 2, 64, 2, 4, 128, 4, 256, 2, 160, "bf16", (160, 33), top_k=1), None),
    "top2": (W("al_top2", 2, 2, 64, 2, 4, 128, 4, 256, 2, 160, "bf16", (160, 33), top_k=2), None),
    "activations": (W("al_h", 3, 1, 128, 3, 4, 64, 3, 256, 2, 130, "bf16", (130, 7), act_tgt=256), None),
}


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_target_16_bytes_past_a_sector(name):
    wl, schedule = SHAPES[name]
    act = name == "activations"
    h = M.mot_create_h(M.h_config_from(wl)) if act else M.mot_create(M.config_from(wl))
    M.mot_load_weights(h, synth.gen_weights(wl, 3))
    if schedule is not None:
        M.mot_set_schedule(h, schedule)
    src = [G.to_device(wl, synth.gen_cache(wl, i, 3)) for i in range(1 if act else 2)]
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    fn = M.mot_translate_h if act else M.mot_translate
    outs = []
    for lead in (0, 8):
        (bk, dk), (bv, dv) = G.alloc_dst(wl, lead), G.alloc_dst(wl, lead)
        assert dk.data_ptr() % 32 == 2 * lead
        fn(h, *src, lens, len(wl.seq_lens), dk, dv)
        assert M.mot_get_device_status(h) == M.MOT_OK
        s = G.sentinel_value(wl)
        for buf, d in ((bk, dk), (bv, dv)):
            assert bool((G.int_view(buf[:lead]) == s).all())
            assert bool((G.int_view(buf[lead + d.numel():]) == s).all())
        outs.append((G.int_view(dk).clone(), G.int_view(dv).clone()))
    assert all(torch.equal(a, b) for a, b in zip(*outs))
    assert bool((outs[0][0] != G.sentinel_value(wl)).any())


@pytest.mark.parametrize("d", [64, 128])
def test_full_replay_output_16_bytes_past_a_sector(d):
    wl = synth.ReplayWorkload("al_full", 2, 2, 6, 2, d, 2, 264, (264, 131), top_s=16, n_full=2)
    h = M.mot_create_replay(M.replay_config_from(wl))
    q, k, v = (torch.from_numpy(x.view("int16")).cuda() for x in synth.gen_replay_qkv(wl, 5))
    lens = torch.tensor(wl.seq_lens, dtype=torch.int32, device="cuda")
    outs = []
    for lead in (0, 8):
        n = wl.max_batch * wl.q_heads * wl.max_seq * d
        buf = torch.full((lead + n + 64,), G.SENTINEL_BF16, dtype=torch.int16, device="cuda")
        assert buf[lead:].data_ptr() % 32 == 2 * lead
        M.mot_replay_attention(h, 1, q, k, v, None, lens, len(wl.seq_lens), buf[lead:])
        torch.cuda.synchronize()
        assert bool((buf[:lead] == G.SENTINEL_BF16).all()) and bool((buf[lead + n:] == G.SENTINEL_BF16).all())
        outs.append(buf[lead:lead + n].clone())
    assert torch.equal(*outs) and bool((outs[0] != G.SENTINEL_BF16).any())
