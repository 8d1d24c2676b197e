"""Compression by block moments (fa_compress_mom.cu): where it can go wrong (ends of blocks and boxes, odd head counts, kept
dims on one side only, rows of different length, little scratch), against the oracle and against the direct contraction.

Bounds.  Both factors of the two products are held as two bf16 numbers: 2^-17 relative each, and the dropped lo x lo term and the
truncated expansion (1.5e-5 at the edge of the band, 6e-7 rms) are below that; relative to the largest coefficient of a
head 3e-5 covers four times their sum.  The direct contraction rounds its basis to bf16: 2^-9 a term, averaged over at
least 1024 tokens, within the 1e-3 that the parity suite allows it."""
import math

import pytest
import torch

from paper_2506_11886_b200 import fa, synth
from tests.parity_util import layout_of, make_pair

pytestmark = pytest.mark.gpu

EXACT_KEYS = ("k_init", "v_init", "k_local", "v_local", "k_mid", "v_mid", "state")
MOMENT_REL = 3e-5


def _shape(**kw):
    return synth.Shape("moments", **{**dict(B=1, layers=1, Hq=2, Hkv=2, d=128, L=1500, dtype="bf16", n_full_k=32, n_full_v=32, M=256,
                                            T=4096, L_init=4, L_local=64), **kw})


@pytest.mark.parametrize("kw", [
    dict(L=1024 + 68),                                    # shortest middle of this path; blocks of 192 tokens, the last of 64
    dict(L=1025 + 68), dict(L=1151 + 68), dict(L=1152 + 68), dict(L=1153 + 68),      # one token into, up to, and past a whole block
    dict(L=4096 + 68, B=2),                               # period full
    dict(L=3001, Hkv=3, Hq=3),                            # odd number of heads: one to a pair of CTAs
    dict(L=3001, n_full_k=0, n_full_v=128),               # nothing kept of K, no coefficients of V
    dict(L=3001, n_full_k=120, n_full_v=8),               # eight columns of K, four rounds of the gather on one side
    dict(L=2500, d=64, n_full_k=64, n_full_v=24, Hkv=4, Hq=4),      # K and V in one item
    dict(L=2500, d=64, n_full_k=8, n_full_v=56),
    dict(L=5000, M=512, T=16384, L_local=300),            # blocks of 384 tokens, a window that starts inside a box
    dict(L=3333, M=256, T=65536, L_init=0, L_local=1),    # T / k = 512: the longest blocks, 768 tokens
    dict(L=3000, M=256, T=5000),                          # period not a power of two
])
def test_block_moments_against_oracle(kw):
    shape = _shape(**kw)
    P = 1 if shape.T == 5000 else 8
    pair, _ = make_pair(shape, seed=71, P=P, max_mid=min(shape.T, shape.L), algo=fa.FA_DECODE_DIRECT, freq="offgrid")
    worst = pair.check_state()
    assert worst <= MOMENT_REL


@pytest.mark.parametrize("kw", [
    # blocks folded about the middle of a row (k a multiple of 256): T = 16384, M = 512: blocks of 384 tokens
    dict(L=3 * 384 + 68),                                 # odd number of blocks: the middle one by itself
    dict(L=4 * 384 + 68), dict(L=4 * 384 + 69),           # even; the last block holds one token
    dict(L=5 * 384 + 68 + 63, B=3),
    dict(L=16384 + 68),                                   # period full
    dict(L=5001, Hkv=3, Hq=3, n_full_k=0, n_full_v=128),
    dict(L=4000, n_full_k=0, n_full_v=0),                 # all 256 columns: three stages
    dict(L=4999, d=64, n_full_k=64, n_full_v=24, Hkv=4, Hq=4),
    dict(L=4999, d=64, n_full_k=8, n_full_v=56),
    dict(L=2900, M=1024, T=32768, B=2),                   # two pairs of tiles
    dict(L=3000, M=512, T=10000),                         # period not a power of two
])
def test_folded_blocks(kw):
    """As many rows as it takes for blocks to be folded, against the definition in 64 bits; one row (blocks as they are) likewise; the
    kept dims and windows exactly as by the order-fixed mode."""
    one = _shape(**{**dict(M=512, T=16384), **kw})
    P = 1 if one.T == 10000 else 8
    n0, n_mid = one.L_init, one.L - one.L_init - one.L_local
    pairs = -(-n_mid // (6 * one.T // (one.M // 2) // 64 * 64)) + 1 >> 1
    folded = one.with_(B=-(-700 * 512 // (pairs * one.Hkv * one.M)))       # (700 positions: folded however the moments' items come out)
    ang = ((torch.arange(n_mid, device="cuda")[None] * torch.arange(one.M // 2, device="cuda")[:, None]) % one.T).double() * (2 * math.pi / one.T)
    F = torch.stack([ang.cos(), ang.sin()], 1).reshape(one.M, n_mid)
    for shape in (folded, folded.with_(B=1)):
        layout = layout_of(shape, max_mid=shape.T, P=P)
        stream = synth.KVStream(shape, seed=72, device="cuda", freq="offgrid")
        K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
        ws = fa.new_workspace(layout)
        got, want = _compress(layout, stream, K, V, ws), _cache(layout, stream)
        fa.fa_compress(layout, want, K, V, ws, flags=fa.FA_COMPRESS_ORDERED)
        torch.cuda.synchronize()
        for n in EXACT_KEYS:
            assert torch.equal(getattr(got, n), getattr(want, n)), n
        for X, coef, idx in ((K, got.coef_k, got.idx_comp_k), (V, got.coef_v, got.idx_comp_v)):
            for h in range(shape.Hkv if coef.numel() else 0):
                y = torch.einsum("mj,bje->bme", F, X[:, n0:n0 + n_mid, h][..., idx[h].long()].double())
                assert ((coef[:, h] - y).abs() <= MOMENT_REL * y.abs().amax(dim=(-1, -2), keepdim=True)).all(), h


def test_folded_rows_of_different_length():
    """Rows of odd and even numbers of blocks, one too short for the path, in one call: each as its row alone (too little work to be folded)."""
    shape = _shape(B=5, Hkv=48, Hq=48, L=6000, M=512, T=16384, n_full_k=24, n_full_v=48)       # 768 positions: folded
    layout = layout_of(shape, max_mid=shape.T, P=16)
    stream = synth.KVStream(shape, seed=10, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    lengths = [6000, 700, 1092 + 384, 4 * 384 + 69, 5 * 384 + 68]
    got = _compress(layout, stream, K, V, fa.new_workspace(layout), lengths)
    for b, n in enumerate(lengths):
        one = layout_of(shape.with_(B=1), max_mid=shape.T, P=16)
        c = _cache(one, stream)
        fa.fa_compress(one, c, K[b:b + 1, :n], V[b:b + 1, :n], fa.new_workspace(one))
        torch.cuda.synchronize()
        for side in ("coef_k", "coef_v"):
            x, y = getattr(got, side)[b], getattr(c, side)[0]
            assert ((x - y).abs() <= MOMENT_REL * y.abs().amax(dim=(-1, -2), keepdim=True)).all(), (b, side)
        assert torch.equal(got.state[b], c.state[0])


@pytest.mark.parametrize("l_init,l_local,d", [(0, 0, 128), (4, 63, 128), (64, 64, 64), (70, 65, 128), (1, 700, 64)])
def test_windows_behind_the_projection(l_init, l_local, d):
    """Window rows are the prompt's, slots past them stay, rows of one length (several boxes to a CTA) and of different ones."""
    shape = _shape(B=3, Hkv=4, Hq=4, L=2000 + l_init + l_local, d=d, n_full_k=16, n_full_v=16, L_init=l_init, L_local=l_local)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    stream = synth.KVStream(shape, seed=5, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    for lengths in (None, [shape.L, l_init + l_local + 1100, shape.L - 1]):
        c = _cache(layout, stream)
        for n in ("k_init", "v_init", "k_local", "v_local"):
            getattr(c, n).fill_(3.0)
        ws = fa.new_workspace(layout)
        if lengths:
            fa.fa_compress_ragged(layout, c, K, V, lengths, ws)
        else:
            fa.fa_compress(layout, c, K, V, ws)
        torch.cuda.synchronize()
        assert fa.fa_poll_status(c) == fa.FA_OK
        for b, n in enumerate(lengths or [shape.L] * 3):
            assert c.state[b, :5].tolist() == [l_init, l_local, n - l_init - l_local, 0, 0]
            for X, init, local in ((K, c.k_init, c.k_local), (V, c.v_init, c.v_local)):
                assert torch.equal(init[b], X[b, :l_init].transpose(0, 1)) and torch.equal(local[b], X[b, n - l_local:n].transpose(0, 1))


def _cache(layout, stream):
    """A cache full of old values: what a call has to write is overwritten, slots past the middle stay."""
    c = fa.Cache(layout, stream.idx_full_k, stream.idx_full_v)
    for n in ("coef_k", "coef_v", "k_mid", "v_mid"):
        getattr(c, n).fill_(3.0)
    return c


def _compress(layout, stream, K, V, ws, lengths=None):
    c = _cache(layout, stream)
    if lengths is None:
        fa.fa_compress(layout, c, K, V, ws)
    else:
        fa.fa_compress_ragged(layout, c, K, V, lengths, ws)
    torch.cuda.synchronize()
    assert fa.fa_poll_status(c) == fa.FA_OK
    return c


def _same(a, b, rel):
    for n in EXACT_KEYS:
        assert torch.equal(getattr(a, n), getattr(b, n)), n
    for n in ("coef_k", "coef_v"):
        x, y = getattr(a, n), getattr(b, n)
        den = y.abs().amax(dim=(-1, -2), keepdim=True)
        assert ((x - y).abs() <= rel * den).all(), n


def _row_bytes(layout, n_mid):
    R = min(6 * layout.period // (layout.n_coef // 2) // 64 * 64, 768)
    return -(-n_mid // R) * layout.n_kv_heads * (2 * layout.head_dim - layout.n_full_k - layout.n_full_v) * 128


def _workspace(layout, n_mid, rows, short=0):
    """A workspace with room for the moments of `rows` rows of n_mid middle tokens, less `short` bytes."""
    decode = fa.fa_workspace_bytes(layout) - 8 * layout.batch * _row_bytes(layout, layout.max_mid)
    return torch.zeros(decode + rows * _row_bytes(layout, n_mid) - short, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("strided", [False, True])
def test_groups_of_rows_and_the_direct_contraction_agree(ragged, strided):
    """A workspace with room for all rows, two, one, or none (the direct contraction): the same cache each time, from
    contiguous and from strided prefill tensors, rows of equal and of different length."""
    shape = _shape(B=5, L=2900, n_full_k=24, n_full_v=48)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    stream = synth.KVStream(shape, seed=9, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    if strided:                                           # [B][H][L][2 d], the second half not used
        wide = [torch.full((shape.B, shape.Hkv, shape.L, 256), float("nan"), dtype=X.dtype, device="cuda") for X in (K, V)]
        for w, X in zip(wide, (K, V)):
            w[..., :128] = X.transpose(1, 2)
        K, V = (w[..., :128].transpose(1, 2) for w in wide)
    lengths = [2900, 700, 1092, 1500, 2899] if ragged else None
    full = _compress(layout, stream, K, V, fa.new_workspace(layout), lengths)
    direct = _compress(layout, stream, K, V, _workspace(layout, shape.L - 68, 1, short=1), lengths)
    _same(direct, full, 1e-3)
    for rows in (1, 2, 3, 5):
        ws = _workspace(layout, shape.L - 68, rows)
        _same(_compress(layout, stream, K, V, ws, lengths), full, 2e-6)      # the same products, added in another order
        assert not ws[:4096].any()                        # the barrier counters of the decode call are left alone


@pytest.mark.parametrize("lengths", [
    [300, 700, 2900, 1500, 1092, 2400],                   # the first group short throughout (rooms of four: groups of two)
    [2900, 1500, 300, 700, 2400, 1092],                   # one in the middle
    [2900, 1500, 2400, 1092, 0, 700],                     # the last
    [100, 2900, 50, 2800, 60, 2700],                      # every other row: groups of one
])
def test_groups_without_a_long_row(lengths):
    """Rows too short for the path make up whole groups: two layers' calls back to back in one stream on one workspace, each row as by itself."""
    shape = _shape(B=6, L=2900, Hkv=4, Hq=4, n_full_k=24, n_full_v=48)
    layout, one = layout_of(shape, max_mid=shape.T, P=16), layout_of(shape.with_(B=1), max_mid=shape.T, P=16)
    streams = [synth.KVStream(shape, seed=30 + i, device="cuda", freq="offgrid") for i in range(2)]
    toks = [s.tokens(0, shape.L, work_dtype=torch.float32) for s in streams]
    want = [[_compress(one, s, K[b:b + 1, :n], V[b:b + 1, :n], fa.new_workspace(one)) for b, n in enumerate(lengths)] for s, (K, V) in zip(streams, toks)]
    for rows in (1, 2, 3, 4, 5):
        ws = _workspace(layout, shape.L - 68, rows)
        got = [_cache(layout, s) for s in streams]
        for c, (K, V) in zip(got, toks):
            fa.fa_compress_ragged(layout, c, K, V, lengths, ws)
        torch.cuda.synchronize()
        for c, singles in zip(got, want):
            assert fa.fa_poll_status(c) == fa.FA_OK
            for b, y in enumerate(singles):
                for name in ("k_init", "v_init", "k_local", "v_local", "k_mid", "v_mid", "state"):
                    assert torch.equal(getattr(c, name)[b], getattr(y, name)[0]), (rows, b, name)
                for name in ("coef_k", "coef_v"):
                    a, r = getattr(c, name)[b], getattr(y, name)[0]
                    den = r.abs().amax(dim=(-1, -2), keepdim=True)
                    # (the same products in another order; short rows fp32 sums in another order)
                    assert ((a - r).abs() <= 2e-6 * den).all(), (rows, b, name)


@pytest.mark.parametrize("room,B", [(1, 1), (2, 1), (3, 1), (4, 1), (7, 1), (4, 2)])      # layers whose moments the workspace holds
def test_layers_in_one_call_and_replayed_from_a_graph(room, B):
    """Layers with scratch for one or two layers at a time, with inputs that change between the replays of a graph."""
    shape = _shape(B=B, L=3000, Hkv=4, Hq=4)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    n = 4
    streams = [synth.KVStream(shape, seed=20 + i, device="cuda", freq="offgrid") for i in range(n)]
    toks = [[s.tokens(t, t + shape.L, work_dtype=torch.float32) for s in streams] for t in (0, 1000)]
    K, V = ([torch.empty_like(p[0]) for p in toks[0]] for _ in range(2))
    caches = [_cache(layout, s) for s in streams]
    ws = _workspace(layout, shape.L - 68, room * B)

    def fill(which):
        for i in range(n):
            K[i].copy_(toks[which][i][0]); V[i].copy_(toks[which][i][1])

    fill(0)
    fa.fa_compress_layers([layout] * n, caches, K, V, ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fa.fa_compress_layers([layout] * n, caches, K, V, ws)
    for which in (1, 0, 1):
        fill(which)
        g.replay()
        torch.cuda.synchronize()
        for i in range(n):
            one = _compress(layout, streams[i], *toks[which][i], fa.new_workspace(layout))
            _same(caches[i], one, 2e-6)
    del g
    assert all(fa.fa_poll_status(c) == fa.FA_OK for c in caches)


def _touched(ws, call):
    """First and last byte of a workspace (past the barrier counters) that a call writes."""
    lo, hi = ws.numel(), 0
    for fill in (0x5A, 0xA5):
        ws[4096:] = fill
        call()
        torch.cuda.synchronize()
        at = (ws[4096:] != fill).nonzero()
        if at.numel():
            lo, hi = min(lo, 4096 + int(at[0])), max(hi, 4096 + int(at[-1]))
    return lo, hi


def test_steps_in_front_of_moments():
    """In one workspace a step over layers stays in front of what the compression of the same layout uses, with areas for four layers as for two."""
    shape = _shape(B=8, Hq=32, Hkv=32, L=1500)
    layout = layout_of(shape, max_mid=shape.T, P=32)
    assert fa.fa_launch_count(layout, 7) == 3
    stream = synth.KVStream(shape, seed=6, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    kn, vn = (x[:, 0].contiguous() for x in stream.tokens(shape.L, shape.L + 1, work_dtype=torch.float32))
    caches = [_compress(layout, stream, K, V, fa.new_workspace(layout)) for _ in range(4)]
    qs = [synth.queries(shape, seed=i, device="cuda") for i in range(4)]
    outs = [torch.zeros_like(q) for q in qs]
    args = fa.LayerStep([layout] * 4, caches, qs, [kn] * 4, [vn] * 4, outs)
    target = _cache(layout, stream)
    ends = []
    for less in (0, 16 << 20):                             # (a layer's areas are some 10 MiB)
        ws = torch.zeros(fa.fa_workspace_bytes(layout) - less, dtype=torch.uint8, device="cuda")
        _, end = _touched(ws, lambda: fa.fa_decode_step_layers(args, ws))
        begin, _ = _touched(ws, lambda: fa.fa_compress(layout, target, K, V, ws))
        assert 0 < end < begin < ws.numel()
        ends.append(end)
    assert ends[1] < ends[0]


def test_rows_one_by_one_keep_off_the_decode_areas():
    """Rows that are compressed one at a time (a local window shorter than a box) use the workspace as the whole batch's layout has it."""
    shape = _shape(B=8, Hq=8, Hkv=8, L=2000, L_local=32)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    stream = synth.KVStream(shape, seed=6, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    lengths, ws = [2000, 1999, 1500, 300, 2000, 1200, 1800, 0], fa.new_workspace(layout)
    c = _compress(layout, stream, K, V, ws, lengths)
    q = synth.queries(shape, seed=1, device="cuda")
    out = torch.zeros_like(q)
    _, end = _touched(ws, lambda: fa.fa_decode_attention(layout, c, q, out, ws))
    begin, _ = _touched(ws, lambda: fa.fa_compress_ragged(layout, c, K, V, lengths, ws))
    assert 0 < end < begin < ws.numel()


def test_a_larger_workspace_holds_all_rows_at_once():
    """What a workspace has beyond the size that is asked for serves the moments: eight rows whose moments exceed the 192 MiB of that size."""
    shape = _shape(B=8, Hq=32, Hkv=32, L=16384, M=512, T=16384)
    layout = layout_of(shape, max_mid=shape.T, P=1)
    stream = synth.KVStream(shape, seed=7, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(7)
    K, V = (torch.randn(shape.B, shape.L, shape.Hkv, shape.d, device="cuda", dtype=torch.bfloat16, generator=g) for _ in range(2))
    rows = shape.B * 44 * shape.Hkv * 192 * 128            # (blocks of 384 tokens, an even number of them)
    want = _compress(layout, stream, K, V, fa.new_workspace(layout))
    ws = torch.zeros(fa.fa_workspace_bytes(layout) + (100 << 20), dtype=torch.uint8, device="cuda")
    got = _cache(layout, stream)
    begin, end = _touched(ws, lambda: fa.fa_compress(layout, got, K, V, ws))
    assert end - begin > 0.95 * rows > 192 << 20
    # (segments are cut at other places: 22 pairs of blocks x six additions in the accumulators, each to 2^-23 of what is there)
    _same(got, want, 22 * 6 * 2.0 ** -23)


def test_not_finite_dims_stay_alone():
    """A NaN or an infinity in one dim of one token spoils that dim's coefficients only."""
    shape = _shape(L=2500)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    stream = synth.KVStream(shape, seed=4, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    want = _compress(layout, stream, K, V, fa.new_workspace(layout))
    bad = int(want.idx_comp_k[1, 5])
    kept = int(want.idx_full_k[0, 3])
    K[0, 777, 1, bad] = float("inf")
    K[0, 900, 0, kept] = float("nan")
    got = _compress(layout, stream, K, V, fa.new_workspace(layout))
    rest = torch.ones_like(got.coef_k, dtype=torch.bool)
    rest[0, 1, :, 5] = False
    assert torch.isfinite(got.coef_k[rest]).all() and torch.isfinite(got.coef_v).all()
    assert not torch.isfinite(got.coef_k[0, 1, :, 5]).all()
    den = want.coef_k.abs().max()
    assert ((got.coef_k - want.coef_k).abs()[rest] <= 2e-6 * den).all()


def test_not_finite_dims_stay_alone_in_pairs_of_blocks():
    """The same where blocks are folded (30 rows of three pairs and eight heads), whose sums and differences meet in an operand: a dim with a NaN and an infinity in
    the two blocks of a pair, one with a NaN in the block by itself; windows full of NaN do not reach the middle."""
    shape = _shape(B=30, Hkv=8, Hq=8, M=512, T=16384, L=68 + 4 * 384 + 100)
    layout = layout_of(shape, max_mid=shape.T, P=16)
    stream = synth.KVStream(shape, seed=4, device="cuda", freq="offgrid")
    K, V = stream.tokens(0, shape.L, work_dtype=torch.float32)
    ws = fa.new_workspace(layout)
    want = _compress(layout, stream, K, V, ws)
    for X in (K, V):
        X[:, :4], X[:, -64:] = float("nan"), float("nan")
    K[3, 4 + 10, 1, int(want.idx_comp_k[1, 5])] = float("inf")              # blocks 0 and 4 are a pair, 2 the one in the middle
    K[3, 4 + 4 * 384 + 50, 1, int(want.idx_comp_k[1, 5])] = float("nan")
    V[29, 4 + 2 * 384 + 7, 6, int(want.idx_comp_v[6, 95])] = float("nan")
    K[0, 900, 0, int(want.idx_full_k[0, 3])] = float("nan")
    got = _compress(layout, stream, K, V, ws)
    for side, bad in (("coef_k", (3, 1, 5)), ("coef_v", (29, 6, 95))):
        x, y = getattr(got, side), getattr(want, side)
        rest = torch.ones_like(x, dtype=torch.bool)
        rest[bad[0], bad[1], :, bad[2]] = False
        assert not torch.isfinite(x[bad[0], bad[1], :, bad[2]]).any()
        assert ((x - y).abs()[rest] <= 2e-6 * y.abs().max()).all()          # (comparison with a NaN is false)
