"""GPU: the sampling kernel where its layout gives way at the shared-memory limit
-- the noise on the set's nodes kept, not kept, and rows as they are -- and with a
set of more nodes than are kept: failures and log-weights of every sample against the
oracle, at noise levels where some decodes fail and the others take several
iterations.  Which form a code takes is pinned on the CPU (test_dispatch_cpu.py)."""
import numpy as np
import pytest

import oracle
import paper_2208_05795_gb300 as tsx
from test_gpu_pair_shapes import _qc

pytestmark = pytest.mark.gpu

SETS = {4: [0, 5, 9, 100], 100: list(range(0, 700, 7))}


@pytest.mark.parametrize("a", sorted(SETS))
@pytest.mark.parametrize("mb,nb,Z,ebn0", [(4, 16, 493, 2.5), (4, 16, 494, 2.5), (4, 16, 505, 2.5), (4, 10, 817, 2.0),
                                          (4, 30, 267, 3.4), (4, 30, 270, 3.4), (4, 32, 254, 3.5), (3, 8, 1188, 2.0)])
def test_samples_at_the_limit(mb, nb, Z, ebn0, a):
    code = _qc(mb, nb, Z, 40 + nb)
    kw = dict(ebn0_db=ebn0, mu=0.8, K=20)
    r = tsx.is_fer_estimate(tsx.load_code(code), SETS[a], n_samples=24, job_key=11, record=True, **kw)
    fail, logw = oracle.Graph(code).is_samples(SETS[a], job=11, n=24, **kw)
    assert 0 < fail.sum() and (a > 4 or fail.sum() < 24)
    assert np.array_equal(r["fail"], fail) and np.array_equal(r["logw"], logw)
    assert r["n_fail"] == int(fail.sum()) and r["decodes"] == 24 and r["iterations"] > 2 * 24
