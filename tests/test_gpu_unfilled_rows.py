"""GPU: QC codes of even check degree above 8 that fit a CTA only without rows
filled up to an odd number of words.  Thresholds, decode counts, iterations
and trapping sets of the two-codeword kernels against the one-codeword kernel
(kernel=1, pinned to the oracle elsewhere); which form a code takes is pinned on the
CPU (test_dispatch_cpu.py)."""
import pytest

import paper_2208_05795_gb300 as tsx
from test_gpu_batch import _same
from test_gpu_pair_shapes import P, _qc

pytestmark = pytest.mark.gpu


def _both(code, **more):
    p = dict(P, cand_end=120, **more)
    return tsx.ts_list_view(tsx.enumerate_ts(code, kernel=2, **p)), tsx.ts_list_view(tsx.enumerate_ts(code, kernel=1, **p))


@pytest.mark.parametrize("mb,nb,Z", [(4, 30, 363), (4, 30, 368), (4, 30, 371), (4, 28, 392), (4, 24, 455), (4, 16, 680),
                                     (4, 10, 1080), (3, 12, 1140)])
def test_variable_node_pass_form(mb, nb, Z):
    _same(*_both(tsx.load_code(_qc(mb, nb, Z, 60 + nb))))


@pytest.mark.parametrize("mb,nb,Z,decoder", [(4, 28, 332, "nms16"), (4, 24, 385, "nms16"), (4, 30, 310, "nms16"),
                                             (4, 28, 494, "nms8")])
def test_two_buffer_form(mb, nb, Z, decoder):
    _same(*_both(tsx.load_code(_qc(mb, nb, Z, 70 + nb)), decoder=decoder, **({"sat": 127} if decoder == "nms8" else {})))


@pytest.mark.parametrize("mb,nb,filled,unfilled", [(4, 32, 250, 254), (4, 16, 490, 505)])
def test_sampling_rate_beside_the_line(mb, nb, filled, unfilled):
    """Sampled words' edge updates a millisecond on either side of where the filling stops: a check's words at a
    stride of 16 or 32 words would meet one or two banks and take 3 to 8 times as long."""
    rate = []
    for Z in (filled, unfilled):
        code = tsx.load_code(_qc(mb, nb, Z, 80))
        kw = dict(ebn0_db=3.5, n_samples=3000, job_key=3, K=20)
        rate.append(max(r["edge_updates"] / r["ms"] for r in (tsx.is_fer_estimate(code, [0, 5, 9], **kw) for _ in range(3))))
    assert rate[1] > 0.5 * rate[0]


@pytest.mark.parametrize("decoder", ["nms16", "nms8"])
def test_in_a_batch(decoder):
    shapes = [(4, 28, 332), (4, 9, 50), (4, 24, 385)] if decoder == "nms16" else [(4, 28, 494), (4, 9, 50)]
    codes = [tsx.load_code(_qc(*s, 90)) for s in shapes]
    p = dict(P, cand_end=120, decoder=decoder, **({"sat": 127} if decoder == "nms8" else {}))
    b = tsx.batch_create(codes, p)
    assert b.decode_launches == 1
    tsx.batch_run(b)
    for i, c in enumerate(codes):
        _same(tsx.batch_view(b, i), tsx.ts_list_view(tsx.enumerate_ts(c, kernel=1, **p)))
