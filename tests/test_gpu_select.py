"""Sec. 3.4 on the GPU (fa_select_dims) against the oracle: index sets bit-exact, errors within tolerance.

The synthetic K / V streams hold, per KV head, in-band sinusoid dims (rebuilt almost exactly from the
coefficients) and white-noise dims (not rebuilt): the error gap between the two groups is many
orders of magnitude, so fp32 / bf16 arithmetic cannot change the ranking across the groups; the number
of kept dims equals the number of noise dims, so the selection is unique."""
import numpy as np
import pytest
import torch

from oracle import fa_oracle as fo
from paper_2506_11886_b200 import fa, synth
from tests.parity_util import layout_of, oracle_cfg, to64

pytestmark = pytest.mark.gpu


def _oracle_selection(layout, K, V):
    cfg = oracle_cfg(layout)
    B, L, H, d = K.shape
    mse = np.zeros((B, H, 2, d))
    for side, X in enumerate((to64(K), to64(V))):
        for b in range(B):
            for h in range(H):
                mse[b, h, side] = fo.dim_mse(cfg, X, b, h)
    sets = []
    for side, n_full in enumerate((layout.n_full_k, layout.n_full_v)):
        full, comp = zip(*(fo.select_dims(mse[:, h, side].mean(axis=0), n_full) for h in range(H)))
        sets += [np.stack(full), np.stack(comp)]
    return sets, mse


@pytest.mark.parametrize("dtype,d,L", [("bf16", 128, 900), ("bf16", 64, 333), ("f32", 128, 300)])
def test_select_dims_matches_oracle(dtype, d, L):
    shape = synth.Shape("sel", B=2, layers=1, Hq=4, Hkv=2, d=d, L=L, dtype=dtype, n_full_k=d // 4, n_full_v=3 * d // 8,
                        M=64, T=1024, L_init=4, L_local=32)
    layout = layout_of(shape, max_mid=1024, P=16)
    stream = synth.KVStream(shape, seed=21)
    K, V = stream.tokens(0, L)
    got = fa.fa_select_dims(layout, K.cuda().contiguous(), V.cuda().contiguous())
    torch.cuda.synchronize()
    want_sets, want_mse = _oracle_selection(layout, K, V)
    names = ("idx_full_k", "idx_comp_k", "idx_full_v", "idx_comp_v")
    for name, g, w in zip(names, got[:4], want_sets):
        np.testing.assert_array_equal(g.cpu().numpy(), w, err_msg=name)
    # the generator's own index sets are what the selection must find
    np.testing.assert_array_equal(got[0].cpu().numpy(), stream.idx_full_k.numpy())
    np.testing.assert_array_equal(got[2].cpu().numpy(), stream.idx_full_v.numpy())
    # errors: relative to the largest error of the row (the well-rebuilt dims sit at the arithmetic's floor)
    g_mse = to64(got[4])
    scale = want_mse.max(axis=-1, keepdims=True)
    assert np.abs(g_mse - want_mse).max() <= 5e-3 * scale.max()
    assert (np.abs(g_mse - want_mse) <= 2e-2 * scale + 1e-6).all()


@pytest.mark.parametrize("Hkv,d,M,L", [(3, 128, 256, 1500), (4, 64, 512, 2000), (2, 128, 128, 129 + 36)])
def test_tensor_core_reconstruction_against_oracle_and_fp32_path(Hkv, d, M, L):
    """bf16 prefill tensors take the tcgen05 reconstruction (several pipeline rounds, a ragged last token tile,
    one or two heads per CTA); the same values handed over as fp32 take the fp32 kernel: both against the oracle."""
    shape = synth.Shape("selt", B=2, layers=1, Hq=Hkv, Hkv=Hkv, d=d, L=L, dtype="bf16", n_full_k=d // 4, n_full_v=d // 2,
                        M=M, T=2048, L_init=4, L_local=32)
    layout = layout_of(shape, max_mid=2048, P=16)
    stream = synth.KVStream(shape, seed=23)
    K, V = stream.tokens(0, L)
    got = fa.fa_select_dims(layout, K.cuda().contiguous(), V.cuda().contiguous())
    shape32 = shape.with_(dtype="f32")
    layout32 = layout_of(shape32, max_mid=2048, P=16)
    got32 = fa.fa_select_dims(layout32, K.float().cuda().contiguous(), V.float().cuda().contiguous())
    torch.cuda.synchronize()
    want_sets, want_mse = _oracle_selection(layout, K, V)
    for g, g32, w in zip(got[:4], got32[:4], want_sets):
        np.testing.assert_array_equal(g.cpu().numpy(), w)
        np.testing.assert_array_equal(g32.cpu().numpy(), w)
    scale = want_mse.max(axis=-1, keepdims=True)
    for g_mse in (to64(got[4]), to64(got32[4])):
        assert (np.abs(g_mse - want_mse) <= 2e-2 * scale + 1e-6).all()
    # the noise dims (errors of the order of the signal) agree closely between the two paths
    big = want_mse > 0.1 * scale
    np.testing.assert_allclose(to64(got[4])[big], to64(got32[4])[big], rtol=5e-3)


@pytest.mark.parametrize("kw", [
    dict(L=1024 + 36, M=256, T=4096, Hkv=24),             # shortest middle of this path: five blocks of 192 tokens and one of 64
    dict(L=1152 + 36, M=256, T=4096, Hkv=24), dict(L=1153 + 36, M=256, T=4096, Hkv=24),      # whole blocks, and one token more (odd number: the middle one by itself)
    dict(L=9 * 192 + 36 + 65, M=256, T=4096, B=1, Hkv=29),                   # ten blocks: two tiles of pairs
    dict(L=4096 + 36, M=256, T=4096, B=12, Hkv=1),        # period full; the smallest prefill of this path
    dict(L=2500, M=512, T=16384, d=64, Hkv=21),           # K and V in one item
    dict(L=2222, M=256, T=65536, L_init=0, L_local=1, Hkv=12),    # the longest blocks
    dict(L=16000, M=256, T=16384, B=1, Hkv=32),           # and many of them to a CTA: a ring of four stages, the sets of warps apart
    dict(L=9000, M=512, T=16384, B=1, Hkv=16),            # a ring of eight
    dict(L=1500, M=256, T=5000, Hkv=17),                  # period not a power of two
    dict(L=1500, M=256, T=4096, norm=1, Hkv=17),          # the paper's weights
    dict(L=4095 + 36, M=256, T=4096, B=12, Hkv=1, direct=1),                 # a token less than the smallest: over coefficient rows
])
def test_reconstruction_by_block_moments(kw):
    """Against the same quantity in 64 bits: x~ from its definition (coefficients, weights, basis by phases
    reduced in integers).  Factors carry 2^-17 and coefficients 4e-6: relative to a dim's mean square and to its error (cross term
    2 sqrt(error * mean square) * 2e-5)."""
    kw = dict(kw)
    norm, direct = kw.pop("norm", 0), kw.pop("direct", 0)
    shape = synth.Shape("selm", **{**dict(B=2, layers=1, Hq=2, Hkv=2, d=128, dtype="bf16", n_full_k=32, n_full_v=24, L_init=4, L_local=32), **kw,
                                   "Hq": kw.get("Hkv", 2)})
    layout = layout_of(shape, max_mid=shape.T, P=1 if shape.T == 5000 else 16)
    layout.norm = norm
    stream = synth.KVStream(shape, seed=29, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    got = fa.fa_select_dims(layout, K, V)[4].double()
    n0 = min(shape.L, shape.L_init)
    X = torch.stack([K, V], 3)[:, n0:shape.L - min(shape.L - n0, shape.L_local)].double()            # [B][mid][H][2][d]
    n = X.shape[1]
    ph = (torch.arange(n, device="cuda")[None] * torch.arange(shape.M // 2, device="cuda")[:, None]) % shape.T
    ang = ph.double() * (2 * np.pi / shape.T)
    F = torch.stack([ang.cos(), ang.sin()], 1).reshape(shape.M, n)
    w = torch.full((shape.M,), 2.0 / shape.T, dtype=torch.float64, device="cuda")
    w[:2] = torch.tensor([1.0 / shape.T, 0.0])
    if norm:
        w[:] = 1.0 / (shape.M // 2)
    C = torch.einsum("mj,bjhse->bhsme", F, X)
    want = (torch.einsum("mj,bhsme->bjhse", F * w[:, None], C) - X).square().mean(1)
    power = torch.einsum("mj,bhsme->bjhse", F * w[:, None], C).square().mean(1) + X.square().mean(1)
    ok = (got - want).abs() <= 4e-5 * (want * power).sqrt() + 1e-8 * power
    if direct:                                             # basis and coefficients in bf16: the floor of 1e-6 tells which path ran
        assert not ok.all()
        ok = (got - want).abs() <= 2e-2 * (want * power).sqrt() + 4e-6 * power
    assert ok.all()


def test_not_finite_dims_stay_alone():
    """By block moments, a NaN or an infinity in the middle spoils the error of its dim only (row 1's here), and what the windows hold does not reach the
    errors.  Bound: two runs of the test above, with mean squares of at most 4 for a dim and for what is rebuilt of it."""
    shape = synth.Shape("seln", B=2, layers=1, Hq=24, Hkv=24, d=128, L=1153 + 36, dtype="bf16", n_full_k=32, n_full_v=24, M=256, T=4096, L_init=4, L_local=32)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    K, V = synth.KVStream(shape, seed=29, device="cuda", freq="offgrid").tokens(0, shape.L, work_dtype=torch.float32)
    want = fa.fa_select_dims(layout, K, V)[4]
    for X in (K, V):
        X[:, :4], X[:, -32:] = float("nan"), float("-inf")
    K[1, 4 + 1152, 5, 17], V[1, 4 + 300, 23, 127], V[1, 4, 0, 64] = float("nan"), float("inf"), float("nan")
    got = fa.fa_select_dims(layout, K, V)[4]
    bad = torch.zeros_like(got, dtype=torch.bool)
    for h, side, e in ((5, 0, 17), (23, 1, 127), (0, 1, 64)):
        bad[1, h, side, e] = True
    assert not torch.isfinite(got[bad]).any()
    assert ((got - want).abs() <= 2 * (4e-5 * (want * 8).sqrt() + 1e-8 * 8))[~bad].all()


def test_select_workspace_of_an_older_size():
    """A workspace without room for the moments is taken as before, by the direct contractions."""
    import ctypes as C
    shape = synth.Shape("selw", B=1, layers=1, Hq=32, Hkv=32, d=128, L=2000, dtype="bf16", n_full_k=32, n_full_v=32, M=256, T=4096, L_init=4, L_local=32)
    layout = layout_of(shape, max_mid=4096, P=16)
    K, V = (x.cuda().contiguous() for x in synth.KVStream(shape, seed=3).tokens(0, 2000))
    want = fa.fa_select_dims(layout, K, V)
    mom_row = -(-4096 // 192) * 32 * 256 * 128
    full = C.c_size_t(0)
    assert fa.lib().fa_select_workspace_bytes(C.byref(layout.c()), C.byref(full)) == fa.FA_OK
    for drop in (256, 32 * 128 * 4 * 256 * 2 + 32 * 128 * 4 + mom_row + 8 * mom_row):          # the last bytes; all moments, of both directions
        ws = torch.zeros(full.value - drop, dtype=torch.uint8, device="cuda")
        idx = [torch.zeros_like(t) for t in want[:4]]
        mse = torch.zeros_like(want[4])
        st = fa.lib().fa_select_dims(C.byref(layout.c()), K.data_ptr(), V.data_ptr(), K.stride(0), K.stride(1), K.stride(2), 2000,
                                     *[t.data_ptr() for t in idx], mse.data_ptr(), ws.data_ptr(), ws.numel(), None)
        torch.cuda.synchronize()
        assert st == fa.FA_OK
        for a, b in zip(idx, want[:4]):
            assert torch.equal(a, b)
        torch.testing.assert_close(mse, want[4], rtol=2e-2, atol=4e-6)          # (basis and coefficients in bf16: 1e-6 of the mean square)


def test_select_dims_empty_middle_and_workspace_check():
    shape = synth.Shape("sel0", B=1, layers=1, Hq=2, Hkv=2, d=64, L=20, dtype="bf16", n_full_k=16, n_full_v=8, M=16,
                        T=256, L_init=4, L_local=32)
    layout = layout_of(shape, max_mid=256, P=8)
    stream = synth.KVStream(shape, seed=22)
    K, V = stream.tokens(0, 20)
    got = fa.fa_select_dims(layout, K.cuda().contiguous(), V.cuda().contiguous())
    torch.cuda.synchronize()
    assert not got[4].any()                                                   # no middle: zero errors
    np.testing.assert_array_equal(got[1].cpu().numpy(), np.tile(np.arange(48), (2, 1)))   # lowest indices compressed
    np.testing.assert_array_equal(got[0].cpu().numpy(), np.tile(np.arange(48, 64), (2, 1)))
    assert fa.fa_workspace_bytes(layout) > 0
    import ctypes as C
    out = C.c_size_t(0)
    assert fa.lib().fa_select_workspace_bytes(C.byref(layout.c()), C.byref(out)) == fa.FA_OK and out.value > 0
    small = torch.zeros(256, dtype=torch.uint8, device="cuda")
    idx = [torch.zeros((2, n), dtype=torch.int32, device="cuda") for n in (16, 48, 8, 56)]
    st = fa.lib().fa_select_dims(C.byref(layout.c()), K.cuda().data_ptr(), V.cuda().data_ptr(), K.stride(0), K.stride(1),
                                 K.stride(2), 20, *[t.data_ptr() for t in idx], None, small.data_ptr(), small.numel(), None)
    assert st == fa.FA_ERR_WORKSPACE
