"""Which kernel a code is decoded by (csrc/decode.cu, host code), on the CPU:
the dispatch is compiled as it stands, with launchers that only say what they
were given.  The codes here are described by their sizes alone."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else shutil.which("nvcc"))
MAIN = r'''
#include <cstdio>
#include "decode.cu"
namespace tsx {
static cudaError_t say(const char *what, const DevCode &g, const LaunchShape &sh) {
    printf("%s %d %d %d %d\n", what, g.row_odd, sh.G, sh.groups, sh.smem_bytes);
    return cudaSuccess;
}
cudaError_t launch_nms16(const DevCode &g, const DecodeParams &, const EnumBuffers &, const LaunchShape &sh, bool pair,
                         cudaStream_t) { return say(pair ? "pair" : "one", g, sh); }
cudaError_t launch_nms16_vn(const DevCode &g, const DecodeParams &, const EnumBuffers &, const LaunchShape &sh,
                            cudaStream_t) { return say("vn", g, sh); }
cudaError_t launch_nms8(const DevCode &g, const DecodeParams &, const EnumBuffers &, const LaunchShape &sh, bool pair,
                        cudaStream_t) { return say(pair ? "pair" : "one", g, sh); }
cudaError_t launch_spa(const DevCode &g, const DecodeParams &, const EnumBuffers &, const LaunchShape &sh,
                       cudaStream_t) { return say("one", g, sh); }
cudaError_t launch_sieve_kernel(const DevCode &, const EnumBuffers &, const LaunchShape &, int, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_batch16(const BatchArgs &, int, bool, int, bool, const LaunchShape &, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_batch8(const BatchArgs &, int, bool, int, bool, const LaunchShape &, cudaStream_t) {
    return cudaSuccess;
}
}
using namespace tsx;
// lines: decoder, rows and columns of the base, Z, least and largest row degree (rows alternate)
int main() {
    int dec, mb, nb, Z, dmin, dmax;
    while (scanf("%d %d %d %d %d %d", &dec, &mb, &nb, &Z, &dmin, &dmax) == 6) {
        DevCode g{};
        g.kind = TSX_CODE_QC; g.n = nb * Z; g.m = mb * Z; g.Z = Z; g.n_b = nb; g.m_b = mb; g.row_odd = 1;
        for (int i = 0; i < mb; i++) {
            const int d = i & 1 ? dmin : dmax;
            g.E += d * Z;
            g.E_odd += (d | 1) * Z;
        }
        g.dv_max = mb; g.dv_min = 1; g.dc_max = dmax; g.dc_min = dmin;
        DecodeParams dp{};
        dp.decoder = dec; dp.K = 20; dp.base_llr = 16; dp.sat = dec == TSX_DEC_NMS_I8 ? 127 : 511;
        dp.alpha_num = 3; dp.alpha_shift = 2; dp.amp_steps = 10;
        if (dec == 100) {  // the sampling kernel
            LaunchShape sh;
            bool noise = false;
            dp.decoder = TSX_DEC_NMS_I16;
            if (plan_is_shape(g, dp, &sh, 152, &noise)) say(noise ? "noise" : "is", g, sh);
            else printf("none 0 0 0 0\n");
            continue;
        }
        const EnumBuffers b{};
        if (dec >= 200) {  // in a multi-code launch with itself
            dp.decoder = dec - 200;
            dp.sat = dp.decoder == TSX_DEC_NMS_I8 ? 127 : 511;
            const DevCode *const gs[2] = {&g, &g};
            const DecodeParams dps[2] = {dp, dp};
            const EnumBuffers bs[2] = {};
            static BatchItem it[2];
            LaunchShape sh;
            int variant = 0;
            if (!plan_batch(gs, dps, bs, nullptr, 2, 152, it, &sh, &variant)) printf("none 0 0 0 0\n");
            else if (it[1].scalar) printf("own 0 0 0 0\n");
            else printf("batch %d %d %d %d\n", it[1].g.row_odd, it[1].G, it[1].groups, sh.smem_bytes);
            continue;
        }
        if (launch_decode(g, dp, b, 0, 0, 0, 152, 0, 100000, nullptr) != cudaSuccess) printf("none 0 0 0 0\n");
    }
}
'''
NMS16, NMS8, SAMPLING, BATCH = 0, 1, 100, 200


@pytest.fixture(scope="module")
def dispatch(tmp_path_factory):
    if not NVCC:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("dispatch")
    (d / "main.cu").write_text(MAIN)
    exe = str(d / "main")
    csrc = os.path.join(ROOT, "paper_2208_05795_gb300", "csrc")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"), "-I", csrc, str(d / "main.cu"), "-o", exe], check=True, timeout=600)

    def run(cases):
        text = "".join("%d %d %d %d %d %d\n" % c for c in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True, timeout=300).stdout
        rows = [line.split() for line in out.splitlines()]
        assert len(rows) == len(cases)
        return [(r[0],) + tuple(int(x) for x in r[1:]) for r in rows]

    return run


@pytest.mark.parametrize("mb,nb,Z", [(4, 30, 365), (4, 30, 368), (4, 30, 371), (4, 28, 392), (4, 24, 455), (4, 22, 500),
                                     (4, 20, 550), (4, 16, 680), (4, 10, 1080), (3, 20, 690), (3, 12, 1140), (5, 16, 560),
                                     (6, 14, 560)])
def test_codes_that_fit_the_variable_node_pass_form_only_with_rows_as_they_are(dispatch, mb, nb, Z):
    assert dispatch([(NMS16, mb, nb, Z, nb, nb)])[0][:2] == ("vn", 0)


@pytest.mark.parametrize("dec,mb,nb,Z", [(NMS16, 4, 28, 332), (NMS16, 4, 24, 385), (NMS16, 4, 30, 310), (NMS8, 4, 28, 494)])
def test_codes_that_fit_two_buffers_only_with_rows_as_they_are(dispatch, dec, mb, nb, Z):
    assert dispatch([(dec, mb, nb, Z, nb, nb)])[0][:2] == ("pair", 0)


def _two_codeword_bytes(mb, nb, Z, posteriors, msg):
    """Shared memory that suffices for a pair of codewords of a full base: the messages, one or two posterior
    buffers, four error patterns, 336 bytes of scratch, and the tables."""
    def up(x):
        return (x + 15) // 16 * 16

    n, E = nb * Z, mb * nb * Z
    tables = up(2 * mb) + up(4 * mb) + up(4 * mb * nb) + up(2 * mb * nb) + up(2 * nb)
    tables += up(4 * nb * mb) + up(2 * nb * mb) + up(4 * nb * mb)
    words = ((n + 31) // 32 + 3) // 4 * 4
    return up(tables) + up(msg * E) + up(4 * posteriors * n) + 16 * words + 336


@pytest.mark.parametrize("mb", range(2, 9))
def test_every_code_with_room_for_two_codewords_has_them(dispatch, mb):
    cases = []
    for nb in range(mb + 1, 33):
        for dec, posteriors, msg in ((NMS16, 1 if nb > 8 else 2, 4), (NMS8, 2, 2)):
            Z = max(z for z in range(1, 32767 // nb + 1) if _two_codeword_bytes(mb, nb, z, posteriors, msg) <= 226 * 1024)
            cases += [(dec, mb, nb, z, nb, nb) for z in range(Z - 3, Z + 1)]
    for c, got in zip(cases, dispatch(cases)):
        assert got[0] in ("pair", "vn"), (c, got)


@pytest.mark.parametrize("mb", range(2, 9))
def test_a_code_decoded_with_two_buffers_is_in_the_multi_code_launch(dispatch, mb):
    """Each of them, alone and in a batch (the batch has one launch bound more or less, so shapes may differ)."""
    cases = [(dec, mb, nb, Z, nb, nb) for nb in range(mb + 1, 33) for dec in (NMS16, NMS8)
             for Z in range(30, 32767 // nb + 1, 3 if nb > 8 else 40)]
    alone = dispatch(cases)
    batch = dispatch([(BATCH + c[0],) + c[1:] for c in cases])
    assert [b[0] == "batch" for b in batch] == [a[0] == "pair" for a in alone]
    assert [b[1] for b in batch if b[0] == "batch"] == [a[1] for a in alone if a[0] == "pair"]


@pytest.mark.parametrize("mb,nb,Z,form", [(4, 16, 493, ("noise", 1)), (4, 16, 494, ("is", 1)), (4, 16, 505, ("is", 0)),
                                          (4, 10, 817, ("is", 0)), (4, 30, 267, ("is", 1)), (4, 30, 270, ("is", 0)),
                                          (4, 32, 254, ("is", 0)), (3, 8, 1188, ("noise", 1))])
def test_sampling_forms(dispatch, mb, nb, Z, form):
    """The set's noise kept ("noise") or not, rows filled up (1) or as they are."""
    assert dispatch([(SAMPLING, mb, nb, Z, nb, nb)])[0][:2] == form
