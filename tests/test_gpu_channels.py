"""The channel form of decode and step (fa_decode_chan.cu): layouts at the edges of what it takes, against the oracle and against
the transform kernel.

Bounds.  Outputs: the parity suite's for bf16.  Against the transform kernel on the same cache: the expansion leaves out 5e-10, the
two bf16 numbers of a factor 2^-17, so scores differ by some 2^-16 of the compressed dims' share (below 8 here) and the results
before rounding by some 1e-4; two bf16 roundings of values up to 4 that straddle a boundary differ by 2^-6.  The rms error against
the oracle is the bf16 rounding of p and of the result in both: not above the transform kernel's by more than its own scatter, 5 %."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2506_11886_b200 import fa, synth
from tests.parity_util import OUT_ABS_BF16, make_pair, to64

pytestmark = pytest.mark.gpu

BUFFERS = ("coef_k", "coef_v", "state", "k_init", "v_init", "k_local", "v_local", "k_mid", "v_mid")


def _shape(**kw):
    return synth.Shape("channels", **{**dict(B=8, layers=1, Hq=16, Hkv=8, d=128, L=1500, dtype="bf16", n_full_k=32, n_full_v=32, M=64,
                                             T=4096, L_init=4, L_local=64, decode_steps=2), **kw})


def _like(layout, algo):
    return dataclasses.replace(layout, decode_algo=algo)


@pytest.mark.parametrize("P,kw", [
    (128, dict()),                                        # S = k = 32; two heads
    (128, dict(Hq=8, n_full_k=48, n_full_v=24, L=0)),     # one head, unlike kept dims; an empty cache fills its first window
    (128, dict(Hq=24, L=67, n_full_k=16, n_full_v=64)),   # three heads; the local window full after one step, then the first middle token
    (128, dict(Hq=40, M=48, L=700)),                      # five heads: passes of three and two, step by two calls; k below S
    (128, dict(Hq=64, B=4, Hkv=16, n_full_k=0, L=900)),   # four heads, nothing kept of K
    (128, dict(n_full_v=0, n_full_k=8, L=513, L_init=0)), # nothing kept of V; one token in the second slot
    (128, dict(L=4094, L_init=0, L_local=0)),             # no windows; the last step fills the period
    (512, dict(B=4, d=64, T=16384, Hq=32, L=2200, n_full_k=24, n_full_v=56)),      # most classes; head_dim 64
    (16, dict(B=16, Hkv=32, Hq=32, T=512, L=300, L_local=20)),                     # fewest classes
    (64, dict(B=8, Hkv=16, Hq=64, T=4096, M=128, L=2100, n_full_k=64, n_full_v=64)),       # most kept dims: two stages a warp
    (128, dict(B=4, Hq=32, T=131072, M=2048, L=3000)),    # longest transforms, clusters of four
    (64, dict(B=8, Hq=32, T=65536, M=2048, L=1000, n_full_k=24, n_full_v=24)),     # and in two waves of clusters
    (128, dict(B=6, Hq=24, T=131072, M=40, L=700)),       # eight warps to a CTA, two to an SM: fewer rows than a stage holds
    (128, dict(B=8, Hq=8, T=131072, M=2048, L=900)),      # one head, many rows
    (64, dict(B=8, Hkv=16, Hq=64, T=65536, M=512, L=800)),         # clusters of two that the sixteen warps' sums leave no room for
])
def test_channels_against_oracle(P, kw):
    shape = _shape(**kw)
    pair, stream = make_pair(shape, seed=5, P=P, max_mid=shape.T, freq="offgrid")
    assert fa.fa_launch_count(pair.layout, 7) == 3 and fa.fa_launch_count(_like(pair.layout, fa.FA_DECODE_FFT), 7) == 0
    other, _ = make_pair(shape, seed=5, P=P, max_mid=shape.T, freq="offgrid", algo=fa.FA_DECODE_FFT)
    K, V = stream.tokens(shape.L, shape.L + 2)
    errs = []
    for t in range(3):
        q = synth.queries(shape, seed=t, step=t)
        if t:
            (got, want), (alt, _) = pair.step(q, K[:, t - 1], V[:, t - 1]), other.step(q, K[:, t - 1], V[:, t - 1])
        else:
            (got, want), (alt, _) = pair.decode(q), other.decode(q)
        assert np.abs(got - want).max() <= OUT_ABS_BF16 * max(1.0, np.abs(want).max())
        assert np.abs(got - alt).max() <= 2.0 ** -6 * max(1.0, np.abs(want).max() / 4)
        errs.append((np.square(got - want).mean() ** 0.5, np.square(alt - want).mean() ** 0.5))
    errs = np.square(np.array(errs)).sum(axis=0) ** 0.5
    assert errs[0] <= 1.05 * errs[1] + 1e-7
    pair.check_state()


@pytest.mark.parametrize("M", [50, 62])
@pytest.mark.parametrize("Hq,kw", [(16, dict()), (24, dict(n_full_k=48)), (32, dict(B=4, Hkv=16, Hq=64)), (8, dict(n_full_v=16))])
def test_coefficients_not_in_groups_of_four(M, Hq, kw):
    """Heads' rows of coefficients that end inside 16 bytes, two, three, four heads and one to a pass: not the channel form, and right."""
    shape = _shape(**{**dict(Hq=Hq, M=M, L=700), **kw})
    pair, stream = make_pair(shape, seed=6, P=128, max_mid=shape.T, freq="offgrid")
    assert fa.fa_launch_count(pair.layout, 7) == 0 and fa.fa_launch_count(dataclasses.replace(pair.layout, n_coef=M + 2), 7) == 3
    K, V = stream.tokens(shape.L, shape.L + 2)
    pair.check_decode(synth.queries(shape, seed=1))
    for t in range(2):
        pair.check_step(synth.queries(shape, seed=1, step=t + 1), K[:, t], V[:, t])
    pair.check_state()


@pytest.mark.parametrize("ragged_one_short", [False, True])
def test_channels_ragged_small_workspace_and_graph(ragged_one_short):
    """Rows of different length (empty, inside the windows, long, one that is full after a step and says so at the next); a
    workspace without room for the channels takes the transform kernel, bit for bit; steps over layers replay from a graph on
    another stream as they ran."""
    shape = _shape(Hq=32, L=3900, M=48)
    pair, stream = make_pair(shape, seed=8, P=128, max_mid=shape.L - 68 + 1, freq="offgrid")
    layout, lengths = pair.layout, [3900, 0, 30, 68, 69, 2000, 197, 3899]
    if ragged_one_short:
        lengths[0], lengths[7] = 1, 700
    K, V = (x.cuda() for x in stream.tokens(0, shape.L))
    kn, vn = (x.cuda() for x in stream.tokens(shape.L, shape.L + 2))
    q = synth.queries(shape, seed=3).cuda()
    fft = _like(layout, fa.FA_DECODE_FFT)

    first = fa.Cache(layout, stream.idx_full_k, stream.idx_full_v)
    fa.fa_compress_ragged(layout, first, K, V, lengths, pair.ws)

    def caches():
        out = [fa.Cache(layout, stream.idx_full_k, stream.idx_full_v) for _ in range(2)]
        for c in out:
            for n in BUFFERS:
                getattr(c, n).copy_(getattr(first, n))
        return out

    new = [[x[:, t].contiguous() for x in (kn, vn)] for t in range(2)]

    def two_steps(lay, cs, ws):
        outs = [[torch.empty_like(q) for _ in cs] for _ in range(2)]
        for t in range(2):
            args = fa.LayerStep([lay] * 2, cs, [q] * 2, [new[t][0]] * 2, [new[t][1]] * 2, outs[t])
            fa.fa_decode_step_layers(args, ws)
        return outs

    a, b, c = caches(), caches(), caches()
    outs = two_steps(layout, a, pair.ws)
    less = fa.new_workspace(fft)                          # (48 coefficients: no room for moments in it)
    assert less.numel() < fa.fa_workspace_bytes(layout)
    ref = two_steps(fft, b, less)
    small = two_steps(layout, c, less)
    torch.cuda.synchronize()
    for x, y, z in zip(sum(outs, []), sum(ref, []), sum(small, [])):
        assert torch.equal(y, z)
        assert (x.float() - y.float()).abs().max() <= 2.0 ** -6
    for x, y in zip(a, b):
        for n in BUFFERS[2:]:
            assert torch.equal(getattr(x, n), getattr(y, n)), n
        for n in BUFFERS[:2]:                             # the same push, fused multiply-add or not
            assert torch.allclose(getattr(x, n), getattr(y, n), rtol=1e-6, atol=1e-5)
    d = caches()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            got = two_steps(layout, d, pair.ws)
        g.replay()
    side.synchronize()
    for x, y in zip(sum(got, []), sum(outs, [])):
        assert torch.equal(x, y)
    status = fa.FA_OK if ragged_one_short else fa.FA_ERR_CAPACITY
    assert all(fa.fa_poll_status(x) == status for x in a + b + c + d)
    del g



def test_layers_share_launches_and_depend_on_one_another():
    """Five layers in one call (four side by side, one more) give the bits of single calls; layers that touch one another's memory (a layer's
    result is the next one's query; one cache twice) run one after the other; with a workspace for one layer's areas they do too."""
    shape = _shape(Hq=32, L=900, M=64)
    pair, stream = make_pair(shape, seed=11, P=128, max_mid=shape.T, freq="offgrid")
    layout, n = pair.layout, 5
    assert fa.fa_launch_count(layout, 7) == 3
    kn, vn = (x.cuda() for x in stream.tokens(shape.L, shape.L + n))
    ks, vs = ([x[:, i].contiguous() for i in range(n)] for x in (kn, vn))
    qs = [synth.queries(shape, seed=3, layer=i).cuda() for i in range(n)]

    def caches():
        out = [fa.Cache(layout, stream.idx_full_k, stream.idx_full_v) for _ in range(n)]
        for c in out:
            for name in BUFFERS:
                getattr(c, name).copy_(getattr(pair.gpu, name))
        return out

    def call(cs, q, out, ws=None):
        fa.fa_decode_step_layers(fa.LayerStep([layout] * n, cs, q, ks, vs, out), pair.ws if ws is None else ws)
        torch.cuda.synchronize()

    def one_by_one(cs, q, out):
        for i in range(n):
            fa.fa_decode_step(layout, cs[i], q[i], ks[i], vs[i], out[i], pair.ws)
        torch.cuda.synchronize()

    def same(a, b, ca, cb):
        for x, y in zip(a, b):
            assert torch.equal(x.view(torch.int16), y.view(torch.int16))
        for x, y in zip(ca, cb):
            assert all(torch.equal(getattr(x, m), getattr(y, m)) for m in BUFFERS)
            assert fa.fa_poll_status(x) == fa.FA_OK

    new = lambda: [torch.full_like(q, float("nan")) for q in qs]
    ca, cb, a, b = caches(), caches(), new(), new()
    call(ca, qs, a)
    one_by_one(cb, qs, b)
    same(a, b, ca, cb)
    cc, c = caches(), new()
    call(cc, qs, c, torch.zeros(fa.fa_workspace_bytes(layout) // 3, dtype=torch.uint8, device="cuda"))
    same(c, b, cc, cb)
    # a chain: layer i + 1 asks with layer i's result
    ca, cb, a, b = caches(), caches(), new(), new()
    call(ca, [qs[0]] + a[:-1], a)
    one_by_one(cb, [qs[0]] + b[:-1], b)
    same(a, b, ca, cb)
    # one cache for all: n pushes, each asked after it
    ca, cb, a, b = caches(), caches(), new(), new()
    call([ca[0]] * n, qs, a)
    one_by_one([cb[0]] * n, qs, b)
    same(a, b, ca[:1], cb[:1])
    assert ca[0].state[:, 2].tolist() == [shape.L - 68 + n] * shape.B
