"""GPU: the cycle search at the edges of its shapes, against the oracle: walks
with repeated nodes (small Z), variable degrees above 4, uneven rows, a
search of few prefixes, and a general code whose listed paths are made in more
than one launch."""
import numpy as np
import pytest

import oracle
import paper_2208_05795_gb300 as tsx
import synth
from test_gpu_pair_shapes import _csr, _qc

pytestmark = pytest.mark.gpu

CODES = {
    "z1": lambda: _qc(3, 6, 1, 1),
    "z3_dv6": lambda: _qc(6, 7, 3, 2),
    "z5_uneven": lambda: _qc(4, 9, 5, 3, 0.4),
    "z40": lambda: _qc(3, 10, 40, 4),
    "csr_uneven": lambda: _csr(60, 31, 5, False),
    "csr6_tiny": lambda: _csr(9, 4, 6, True),
}


def _check(code, lmax, starts):
    s = tsx.emd_spectrum(tsx.load_code(code), lmax)
    g = oracle.Graph(code)
    parts = [g.cycle_walks(v, lmax, emd=True) for v in starts]
    assert np.array_equal(s["count2l"][:lmax + 1], sum(p[1] for p in parts))
    assert np.array_equal(s["walks"][:lmax + 1], sum(p[0] for p in parts))


@pytest.mark.parametrize("lmax", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("name", sorted(CODES))
def test_spectrum_edges(name, lmax):
    code = CODES[name]()
    if lmax == 6 and name in ("z3_dv6", "csr_uneven"):
        pytest.skip("minutes of the oracle's time; the same code paths as lmax = 5 and the other codes")
    starts = range(0, code.n, code.Z) if code.kind == "qc" else range(code.n)
    _check(code, lmax, list(starts))


def test_spectrum_in_several_launches():
    # 4 (n + 1) + 8 dv (dc - 1) ... bytes for each of n representatives: above 64 MB together
    rng = np.random.default_rng(7)
    n, m = 4200, 2100
    cols = np.concatenate([rng.permutation(n) for _ in range(3)]).reshape(m, 6)
    for c in range(m):  # (no node twice in a row)
        while len(set(cols[c])) < 6:
            k = int(rng.integers(0, m))
            cols[c, 0], cols[k, 0] = cols[k, 0], cols[c, 0]
            if len(set(cols[k])) < 6:
                cols[c, 0], cols[k, 0] = cols[k, 0], cols[c, 0]
                cols[c] = rng.choice(n, 6, replace=False)
    code = synth.csr_code(n, m, np.arange(0, 6 * m + 1, 6), np.sort(cols, axis=1).ravel().astype(np.int32))
    _check(code, 4, list(range(n)))
