"""The SIMT translation path (fp32 caches, and bf16 shapes outside the tensor-core
tiling) at the edges of its 64 x 32 tiles, 64-wide K blocks and four-value pieces,
every element against the fp64 oracle with the parity bars."""
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import _gpu as G   # noqa: E402

W = synth.Workload


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("hs,ds,ht,dt,e,hidden,lens", [
    (1, 4, 1, 1, 1, 1, (1,)),                    # the smallest
    (2, 12, 3, 10, 3, 21, (31, 32, 33)),         # scalar pieces (K of GEMM2 not a multiple of 4)
    (3, 20, 1, 63, 2, 34, (64, 65)),             # K = 60 and 68 around one block
    (5, 13, 2, 33, 1, 64, (127, 128, 129)),      # scalar heads, 65 channels, 66 columns
    (4, 36, 4, 16, 4, 52, (130, 0, 1)),          # K = 144 and 208, whole columns
])
def test_simt_tile_edges(dtype, hs, ds, ht, dt, e, hidden, lens):
    wl = W("simt_edge", 2, hs, ds, 2, ht, dt, e, hidden, len(lens), max(lens), dtype, lens)
    sk, sv, blob = synth.gen_cache(wl, 0, 3), synth.gen_cache(wl, 1, 3), synth.gen_weights(wl, 3)
    run = G.Run(wl, sk, sv, blob)
    assert G.M.mot_get_path(run.h) == 0
    assert run.translate() == G.M.MOT_OK
    rk, rv = oracle.translate_full(wl, sk, sv, blob, wl.seq_lens)
    mask = G.translated_mask_full(wl, wl.seq_lens)
    gk, gv = run.dst_f64()
    G.assert_parity(wl, gk[mask], rk[mask], "K")
    G.assert_parity(wl, gv[mask], rv[mask], "V")
    assert run.canaries_intact() and run.padding_untouched()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("ht,dt,e,hidden,lens", [
    (1, 33, 1, 511, (64,)),           # the longest K that is not split
    (1, 33, 1, 512, (64,)),           # four K blocks each
    (2, 31, 1, 514, (63, 1)),         # scalar pieces: five blocks, and four (two columns in the last)
    (3, 32, 4, 144, (8, 9, 17, 33)),  # nine blocks; whole row groups, and one row past one
    (2, 48, 4, 1024, (70, 5)),        # long K over several tiles
    (12, 64, 4, 1024, (500, 129)),    # long K, more tiles than two per SM
    (12, 64, 2, 512, (200, 129)),     # short K, more tiles than two per SM: not split
])
def test_simt_second_gemm_split_over_pairs(dtype, ht, dt, e, hidden, lens):
    wl = W("simt_pair", 1, 2, 12, 4, ht, dt, e, hidden, len(lens), max(lens), dtype, lens)
    sk, sv, blob = synth.gen_cache(wl, 0, 5), synth.gen_cache(wl, 1, 5), synth.gen_weights(wl, 5)
    run = G.Run(wl, sk, sv, blob)
    assert G.M.mot_get_path(run.h) == 0
    assert run.translate() == G.M.MOT_OK
    rk, rv = oracle.translate_full(wl, sk, sv, blob, wl.seq_lens)
    mask = G.translated_mask_full(wl, wl.seq_lens)
    gk, gv = run.dst_f64()
    G.assert_parity(wl, gk[mask], rk[mask], "K")
    G.assert_parity(wl, gv[mask], rv[mask], "V")
    assert run.canaries_intact() and run.padding_untouched()
