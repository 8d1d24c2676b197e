"""The fp32 contraction of short middles (compress_coef_kernel), both numbers of rows per thread and the line between them, against the
oracle.

Bound: a coefficient is a sum of at most 1023 products, each product and each addition rounded to 2^-24 of what it is then, the basis to
2^-22: as a random walk sqrt(2 * 1023) * 2^-24 + 2^-22 = 3e-6 of the largest coefficient of a head; 1.5e-5 is five times that."""
import pytest

from paper_2506_11886_b200 import fa, synth
from tests.parity_util import make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    # tiles of 64 rows x rows x heads x 2 sides x chunks of 64 tokens against twice the SMs (296)
    dict(B=1, Hkv=8, M=64, L=18 * 64 + 36, T=2048, dtype="f32"),             # 16 x 18 = 288: four rows to a thread
    dict(B=1, Hkv=8, M=64, L=18 * 64 + 37, T=2048, dtype="f32"),             # 16 x 19 = 304: eight; the last chunk holds one token
    dict(B=2, Hkv=8, M=104, L=6 * 64 + 36, T=2048, dtype="bf16"),            # the second tile has 40 of 64 rows
    dict(B=3, Hkv=3, M=40, L=1023 + 36, T=1500, dtype="bf16", n_full_k=0),   # fewer rows than a tile, all columns of K, no power of two
    dict(B=2, Hkv=8, M=64, L=640 + 36, T=1024, dtype="bf16", d=64),
])
def test_short_middles(kw):
    shape = synth.Shape("short", **{**dict(layers=1, d=128, n_full_k=24, n_full_v=40, L_init=4, L_local=32), **kw, "Hq": kw["Hkv"]})
    pair, _ = make_pair(shape, seed=5, P=1, max_mid=min(shape.T, shape.L), algo=fa.FA_DECODE_DIRECT, freq="offgrid")
    assert pair.check_state() <= 1.5e-5
