"""GPU: the one-codeword min-sum kernel on QC codes of check degree above 8, whose
groups of one warp run a form of their own: the same thresholds, counts and
sets as with two and with five warps a codeword, in both storages."""
import pytest

import paper_2208_05795_gb300 as tsx
from test_gpu_batch import _same
from test_gpu_pair_shapes import P, _qc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("decoder", ["nms16", "nms8"])
@pytest.mark.parametrize("mb,nb,Z", [(3, 9, 31), (4, 18, 64), (4, 31, 37), (2, 32, 70)])
def test_one_warp_against_more(mb, nb, Z, decoder):
    code = tsx.load_code(_qc(mb, nb, Z, 50 + nb))
    p = dict(P, kernel=1, cand_end=300, decoder=decoder, **({"sat": 127} if decoder == "nms8" else {}))
    want = tsx.ts_list_view(tsx.enumerate_ts(code, warps_per_cta=2, **p))
    for G in (1, 5):
        _same(tsx.ts_list_view(tsx.enumerate_ts(code, warps_per_cta=G, **p)), want)
