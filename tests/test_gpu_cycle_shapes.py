"""GPU: the cycle search on general codes, where every node is a representative:
paths listed in fewer buckets than nodes, and prefixes of nodes of large and
uneven degree shared by a warp.  Against the oracle; and the cost of a
representative does not grow with the code, nor much that of a walk with uneven degrees."""
import numpy as np
import pytest

import paper_2208_05795_gb300 as tsx
import synth
from test_gpu_cycle_edges import _check
from test_gpu_pair_shapes import _qc

pytestmark = pytest.mark.gpu


def _rows(n, m, lo, hi, seed):
    """Rows of lo to hi nodes; node i is in row i mod m at least."""
    rng = np.random.default_rng(seed)
    rows = [set(range(c, n, m)) for c in range(m)]
    for r in rows:
        want = int(rng.integers(lo, hi + 1))
        while len(r) < want:
            r.add(int(rng.integers(0, n)))
    ptr = np.zeros(m + 1, np.int32)
    ptr[1:] = np.cumsum([len(r) for r in rows])
    return synth.csr_code(n, m, ptr, np.concatenate([np.sort(list(r)) for r in rows]).astype(np.int32))


# (buckets: 64 to 256 of 700 nodes, one a node at 60; a warp shares its prefixes from 32 K of one step less on)
CODES = {
    "sparse": (lambda: _rows(900, 600, 2, 4, 1), (4, 5, 6)),
    "uneven": (lambda: _rows(700, 400, 2, 8, 2), (4, 5)),
    "uneven_small": (lambda: _rows(120, 80, 2, 5, 3), (4, 5)),
    "hubs": (lambda: _rows(60, 50, 2, 6, 4), (4, 5)),
    "light": (lambda: _rows(300, 200, 3, 3, 5), (4, 5, 6)),
}


@pytest.mark.parametrize("name,lmax", [(k, l) for k, v in CODES.items() for l in v[1]])
def test_general_codes(name, lmax):
    code = CODES[name][0]()
    _check(code, lmax, range(code.n))


@pytest.mark.parametrize("mb,nb,Z,lmax", [(6, 10, 9, 5), (5, 8, 64, 5), (7, 9, 5, 5)])
def test_qc_codes_of_large_degree(mb, nb, Z, lmax):
    code = _qc(mb, nb, Z, 6, 0.3)
    _check(code, lmax, range(0, code.n, code.Z))


def _degree_two(n, m, most, seed):
    """Every node in two rows, rows of up to `most` nodes, the first ones longer."""
    rng = np.random.default_rng(seed)
    rows = [[] for _ in range(m)]
    for v in range(n):
        for c in (v % m, None):
            while c is None or v in rows[c] or len(rows[c]) >= most:
                c = int(m * rng.random() ** 2)
            rows[c].append(v)
    ptr = np.zeros(m + 1, np.int32)
    ptr[1:] = np.cumsum([len(r) for r in rows])
    return synth.csr_code(n, m, ptr, np.concatenate([np.sort(r) for r in rows]).astype(np.int32))


def _ms(code, lmax):
    c = tsx.load_code(code)
    r = [tsx.emd_spectrum(c, lmax) for _ in range(6)]
    return min(x["ms"] for x in r), int(r[0]["walks"].sum())


def test_degree_two_prefixes():
    """Prefixes are counted over the entries a node may have, not over its row filled up to four: with degree 2 those
    of three steps were eight times as many, and walks of up to 6 nodes took
    13 times as long as walks of up to 4, instead of four."""
    code = _degree_two(200, 150, 20, 8)
    _check(code, 5, range(code.n))
    assert _ms(code, 6)[0] < 8 * _ms(code, 4)[0]


def test_cost_of_a_representative():
    """Rows of six nodes, 2,500 and 30,000 nodes: twelve times the representatives, in less than twelve times as long;
    with n words zeroed, scanned and shifted for each representative it grew with the square."""
    ms = []
    for n in (2500, 30000):
        code = tsx.load_code(_rows(n, n // 3, 3, 6, 7))
        ms.append(min(tsx.emd_spectrum(code, 4)["ms"] for _ in range(5)))
    assert ms[1] < 12 * ms[0], ms


def test_time_of_a_walk_in_an_uneven_code():
    """Walks of nodes of large degree are shared out: a walk of a code with rows of 2 to 12 takes at most five times
    as long as one of a code with even rows (13 times where a thread had all that follow its prefix)."""
    t = []
    for lo, hi in ((8, 8), (2, 12)):
        ms, walks = _ms(_rows(300, 200, lo, hi, 9), 4)
        t.append(ms / walks)
    assert t[1] < 5 * t[0], t
