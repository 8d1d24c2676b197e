"""Layouts at the edges of the kernel dispatch: each test names the branch it takes and checks it against the oracle."""
import pytest
import torch

from paper_2506_11886_b200 import fa, synth
from tests.parity_util import layout_of, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(M=256, n_full_k=48, n_full_v=64),               # one pair per team, one round of gather items
    dict(M=256, n_full_k=104, n_full_v=8),               # several rounds on one side only
    dict(M=768, n_full_k=120, n_full_v=128),             # three pairs per team: rows of a round not a multiple of the pairs
    dict(M=512, n_full_k=64, n_full_v=64, d=64, Hkv=3),  # one head per pair of CTAs
])
def test_pair_compress_writes_many_kept_dims(kw):
    shape = synth.Shape("gather", **{**dict(B=2, layers=1, Hq=4, Hkv=4, d=128, L=1777, dtype="bf16", T=2048, L_init=3,
                                            L_local=64), **kw, **({"Hq": kw["Hkv"]} if "Hkv" in kw else {})})
    pair, _ = make_pair(shape, seed=31, P=2, max_mid=shape.T, algo=fa.FA_DECODE_DIRECT)
    pair.check_state()


@pytest.mark.parametrize("B,M,lengths", [
    (5, 256, [0, 2600, 1091, 1092, 70]),                 # empty, long, one below / at the tensor path's 1024 middle tokens, no middle
    (3, 512, [1100, 1155, 1156]),                        # middles of 1032, 1087, 1088 tokens: ragged and whole last blocks
    (66, 256, [1100 + 7 * (b % 9) for b in range(66)]),  # more rows than one launch takes
    (2, 128, [2000, 300]),                               # odd number of row tiles: row by row
])
def test_ragged_compress_in_one_launch_equals_row_by_row(B, M, lengths):
    shape = synth.Shape("ragged", B=B, layers=1, Hq=4, Hkv=2, d=64, L=max(lengths), dtype="bf16", n_full_k=16, n_full_v=24,
                        M=M, T=4096, L_init=4, L_local=64)
    stream = synth.KVStream(shape, seed=5, device="cuda")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    for b, n in enumerate(lengths):
        K[b, n:], V[b, n:] = float("nan"), float("nan")   # rows past a prompt's length are not read
    layout = layout_of(shape, max_mid=shape.T, P=8)
    one = layout_of(shape.with_(B=1), max_mid=shape.T, P=8)
    got, ws = fa.Cache(layout, stream.idx_full_k, stream.idx_full_v), fa.new_workspace(layout)
    got.coef_k.fill_(7.0)
    fa.fa_compress_ragged(layout, got, K, V, lengths, ws)
    for b in sorted({0, 1, B // 2, B - 2, B - 1}):
        ref = fa.Cache(one, stream.idx_full_k, stream.idx_full_v)
        fa.fa_compress(one, ref, K[b:b + 1, :lengths[b]], V[b:b + 1, :lengths[b]], ws)
        for n in ("k_init", "v_init", "k_local", "v_local", "k_mid", "v_mid", "state"):
            assert torch.equal(getattr(got, n)[b], getattr(ref, n)[0]), (b, n)
        for n in ("coef_k", "coef_v"):
            g, r = getattr(got, n)[b], getattr(ref, n)[0]
            # (basis phasors are seeded where a CTA's blocks begin: some bf16 roundings of the basis differ)
            assert (g - r).abs().max() <= 2e-4 * r.abs().max() + 1e-6, (b, n)
    assert fa.fa_poll_status(got) == fa.FA_OK


@pytest.mark.parametrize("kw,P", [
    (dict(L=63, T=64, M=8), 1),                          # one tile, one frequency group, token-major
    (dict(L=200, T=400, M=66), 3),                       # odd class count and period, a frequency more than a warp
    (dict(L=700, T=1024, M=1024, L_init=3, L_local=70), 4),   # more frequencies than threads
    (dict(L=600, T=1024, M=100, n_full_k=0, n_full_v=128, Hq=3), 2),   # three heads in four slots; no kept K, no compressed V dims
])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_direct_decode_tiles_of_tokens(kw, P, dtype):
    shape = synth.Shape("direct", **{**dict(B=2, layers=1, Hq=2, Hkv=1, d=128, dtype=dtype, n_full_k=32, n_full_v=24, L_init=0,
                                            L_local=0, decode_steps=0), **kw})
    pair, _ = make_pair(shape, seed=9, P=P, algo=fa.FA_DECODE_DIRECT, freq="offgrid", max_mid=min(shape.T, shape.L))
    pair.check_state()
    pair.check_decode(synth.queries(shape, seed=9))
    pair.check_decode(synth.queries(shape, seed=9, step=1, peak=6.0))


@pytest.mark.parametrize("Hq,Hkv,B,S,k", [
    (4, 1, 40, 32, 32),      # sixteen lanes to a pair of bins, every class of a head in one batch
    (4, 1, 40, 64, 20),      # fewer frequencies than bins
    (2, 1, 70, 32, 16),      # two heads to a point
    (1, 1, 130, 32, 32),     # one query head: two classes to a transform
    (3, 1, 3, 128, 128),     # an odd number of classes, three heads in four slots
])
def test_decode_short_transforms_many_classes_in_a_batch(Hq, Hkv, B, S, k):
    shape = synth.Shape("short", B=B, layers=1, Hq=Hq, Hkv=Hkv, d=64, L=S * 32 - 5, dtype="bf16", n_full_k=16, n_full_v=24, M=2 * k,
                        T=S * 32, L_init=3, L_local=20, decode_steps=2)
    pair, stream = make_pair(shape, seed=12, P=32, algo=fa.FA_DECODE_FFT, max_mid=shape.T, freq="offgrid")
    pair.check_decode(synth.queries(shape, seed=12))
    K, V = stream.tokens(shape.L, shape.L + 2)
    for t in range(2):
        pair.check_step(synth.queries(shape, seed=12, step=t + 1, peak=3.0), K[:, t], V[:, t])
    pair.check_state()
