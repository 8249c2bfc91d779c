"""GPU: the two-codeword kernels at the edges of their shapes.

The one-codeword kernel (kernel=1, pinned to the oracle elsewhere) decodes
the same candidates of each code; thresholds, decode counts, iterations and
trapping sets are whole numbers and must be equal.  Sizes: row blocks that do
not fill a warp, n not a multiple of 4, check degrees 1, odd, even and 32,
rows of uneven degree (warps that straddle two row blocks), 8-bit storage,
every group width, fewer candidates than groups, and a batch in which a
degree-6 code runs in the large-degree variant."""
import numpy as np
import pytest

import synth
import paper_2208_05795_gb300 as tsx
from test_gpu_batch import _same

pytestmark = pytest.mark.gpu

P = dict(K=12, base_llr=16, amp_steps=6, max_size=2)


def _qc(mb, nb, Z, seed, drop=0.0):
    """Any exponents (short cycles allowed); drop: share of zero blocks, no empty row or column."""
    rng = np.random.default_rng(seed)
    E = rng.integers(0, Z, (mb, nb)).astype(np.int32)
    E[rng.random((mb, nb)) < drop] = -1
    for j in range(nb):
        if (E[:, j] < 0).all():
            E[j % mb, j] = 0
    for i in range(mb):
        if (E[i] < 0).all():
            E[i, i % nb] = 0
    return synth.qc_code(E, Z)


def _csr(n, m, seed, regular):
    rng = np.random.default_rng(seed)
    rows = [np.sort(rng.choice(n, 6 if regular else int(rng.integers(1, 13)), replace=False)) for _ in range(m)]
    ptr = np.zeros(m + 1, np.int32)
    ptr[1:] = np.cumsum([len(r) for r in rows])
    return synth.csr_code(n, m, ptr, np.concatenate(rows))


CODES = {
    "z1": lambda: _qc(6, 12, 1, 1),
    "z5_deg6": lambda: _qc(3, 6, 5, 2),
    "z33_deg6": lambda: _qc(3, 6, 33, 3),
    "deg1": lambda: _qc(3, 9, 7, 4, 0.8),
    "deg8_uneven": lambda: _qc(4, 8, 19, 5, 0.3),
    "deg9": lambda: _qc(3, 9, 31, 6),
    "z153_uneven": lambda: _qc(4, 23, 153, 7, 0.2),
    "deg31": lambda: _qc(3, 31, 37, 8),
    "deg32": lambda: _qc(2, 32, 64, 9),
    "vn_form": lambda: _qc(4, 30, 380, 10, 0.1),
    "csr6": lambda: _csr(203, 101, 11, True),
    "csr6_tiny": lambda: _csr(9, 4, 12, True),
    "csr_uneven": lambda: _csr(150, 77, 13, False),
}


@pytest.mark.parametrize("decoder", ["nms16", "nms8"])
@pytest.mark.parametrize("name", sorted(CODES))
def test_pair_equals_scalar(name, decoder):
    code = tsx.load_code(CODES[name]())
    p = dict(P, decoder=decoder, cand_end=300, **({"sat": 127} if decoder == "nms8" else {}))
    want = tsx.ts_list_view(tsx.enumerate_ts(code, kernel=1, **p))
    for extra in (dict(), dict(cand_end=3), dict(cand_end=1)):
        q = dict(p, **extra)
        ref = want if not extra else tsx.ts_list_view(tsx.enumerate_ts(code, kernel=1, **q))
        _same(tsx.ts_list_view(tsx.enumerate_ts(code, kernel=2, **q)), ref)


@pytest.mark.parametrize("name", ["z33_deg6", "z153_uneven", "csr6"])
@pytest.mark.parametrize("G", [1, 2, 3, 7, 16])
def test_group_widths(name, G):
    code = tsx.load_code(CODES[name]())
    want = tsx.ts_list_view(tsx.enumerate_ts(code, kernel=1, **dict(P, cand_end=200)))
    _same(tsx.ts_list_view(tsx.enumerate_ts(code, kernel=2, warps_per_cta=G, **dict(P, cand_end=200))), want)


@pytest.mark.parametrize("names", [("z33_deg6", "deg9"), ("z5_deg6", "deg8_uneven", "z33_deg6"), ("csr6", "csr_uneven")])
def test_batch_of_mixed_degrees(names):
    codes = [tsx.load_code(CODES[n]()) for n in names]
    p = dict(P, cand_end=150)
    b = tsx.batch_create(codes, p)
    assert b.multi_launch
    tsx.batch_run(b)
    for i, c in enumerate(codes):
        _same(tsx.batch_view(b, i), tsx.ts_list_view(tsx.enumerate_ts(c, kernel=1, **p)))


@pytest.mark.parametrize("Z", [1, 2, 31, 64, 700, 1600, 1850])
def test_degree_six_tables(Z):
    """Rows as node lists (few groups to many), and exponents where the lists do not fit beside one pair."""
    code = tsx.load_code(_qc(3, 6, Z, 30 + Z))
    p = dict(P, max_size=1 if Z == 1 else 2, cand_end=60)
    _same(tsx.ts_list_view(tsx.enumerate_ts(code, kernel=2, **p)), tsx.ts_list_view(tsx.enumerate_ts(code, kernel=1, **p)))


@pytest.mark.parametrize("mb,nb,Z", [(3, 8, 1188), (4, 10, 817), (4, 9, 868)])
def test_sampling_near_the_shared_memory_limit(mb, nb, Z):
    """Codes whose sampling layout has no room for the kept noise, or for rows of odd length: still taken, with the
    log-weights of a shorter list of nodes (which do not depend on the code) and no failure without noise to speak of."""
    code = tsx.load_code(_qc(mb, nb, Z, 40 + nb))
    kw = dict(ebn0_db=12.0, n_samples=6, job_key=3, rate=0.5, K=4, record=True)
    r = tsx.is_fer_estimate(code, [0, 5, 9], **kw)
    small = tsx.is_fer_estimate(tsx.load_code(_qc(3, 6, 16, 1)), [0, 5, 9], **kw)
    assert np.array_equal(r["logw"], small["logw"]) and r["decodes"] == 6
