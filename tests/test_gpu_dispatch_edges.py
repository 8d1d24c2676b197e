"""Layouts at the edges of the kernel dispatch: each test names the branch it takes and checks it against the oracle."""
import pytest

from paper_2506_11886_b200 import fa, synth
from tests.parity_util import make_pair

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
