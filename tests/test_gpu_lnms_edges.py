"""GPU: the layered decoder's two-frame kernel at the edges of its shapes,
against the oracle frame by frame (whole numbers, equal): n not a multiple of
4, layers that do not fill a warp, check degrees 1, odd, even and 32, widths
from 2 to 8 bits, normalizations from 1 / 32768 (products beyond 16 bits:
the one-frame kernel) to 1, K = 0, one frame, buffers at odd addresses, and
a code whose two frames do not fit a CTA (the one-frame kernel)."""
import numpy as np
import pytest

import oracle
import paper_2208_05795_gb300 as tsx
from test_gpu_pair_shapes import CODES, _qc

pytestmark = pytest.mark.gpu

MORE = {"one_frame_form": lambda: _qc(4, 32, 430, 21)}
DEF = dict(K=8, llr_bits=4, c2v_bits=4, v2c_bits=6, alpha_num=3, alpha_shift=2)


def _check(code, nf, off=0, **p):
    import torch
    p = dict(DEF, **p)
    g = oracle.Graph(code)
    rng = np.random.default_rng(code.n + nf)
    llr = np.clip(np.round(rng.normal(1.5, 2.5, (nf, code.n))), -128, 127).astype(np.int8)
    llr[::5] = np.abs(llr[::5] % 8)  # (some decode at once)
    def buf(count, dtype):
        b = torch.zeros(count + 8, dtype=dtype, device="cuda")
        return b[off:off + count]
    d = buf(nf * code.n, torch.int8)
    d.copy_(torch.from_numpy(llr.ravel()))
    fail, it, x = buf(nf, torch.uint8), buf(nf, torch.int32), buf(nf * code.n, torch.uint8)
    c = tsx.load_code(code)
    tsx.lnms_decode(c, d.data_ptr(), nf, fail.data_ptr(), it.data_ptr(), x.data_ptr(), **p)
    torch.cuda.synchronize()
    fail, it, x = fail.cpu().numpy(), it.cpu().numpy(), x.cpu().numpy().reshape(nf, -1)
    for f in range(nf):
        of, ox, ok = g.decode_lnms(llr[f].astype(np.int32), **p)
        assert (bool(fail[f]), int(it[f])) == (of, ok) and np.array_equal(x[f], ox), f


QC = [n for n in sorted(CODES) if not n.startswith("csr")]


@pytest.mark.parametrize("name", QC + sorted(MORE))
def test_shapes(name):
    code = {**CODES, **MORE}[name]()
    _check(code, 40 if code.n < 5000 else 6)


@pytest.mark.parametrize("p", [dict(llr_bits=2, c2v_bits=2, v2c_bits=2), dict(llr_bits=8, c2v_bits=8, v2c_bits=8),
                               dict(c2v_bits=8, v2c_bits=3), dict(alpha_num=1, alpha_shift=0),
                               dict(alpha_num=1, alpha_shift=15), dict(alpha_num=32768, alpha_shift=15),
                               dict(alpha_num=500, alpha_shift=9, v2c_bits=8), dict(K=0), dict(K=1)],
                         ids=lambda p: "-".join("%s%s" % kv for kv in sorted(p.items())))
@pytest.mark.parametrize("name", ["deg1", "z33_deg6", "z153_uneven"])
def test_widths_and_normalizations(name, p):
    _check(CODES[name](), 20, **p)


@pytest.mark.parametrize("nf", [1, 2, 3])
@pytest.mark.parametrize("off", [0, 1])
def test_few_frames_and_addresses(nf, off):
    _check(CODES["deg32"](), nf, off)
    _check(CODES["z5_deg6"](), nf, off)
