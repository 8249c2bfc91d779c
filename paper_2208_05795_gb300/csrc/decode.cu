// decode.cu -- host side of the decoding and sieve kernels: shared-memory
// layouts, launch shapes, dispatch, and the compaction of the trapping-set
// hash table.
#include "decode_pair.cuh"

namespace tsx {

// per-decoder translation units
cudaError_t launch_nms16(const DevCode &, const DecodeParams &, const EnumBuffers &, const LaunchShape &, bool pair,
                         cudaStream_t);
cudaError_t launch_nms16_vn(const DevCode &, const DecodeParams &, const EnumBuffers &, const LaunchShape &,
                            cudaStream_t);
cudaError_t launch_nms8(const DevCode &, const DecodeParams &, const EnumBuffers &, const LaunchShape &, bool pair,
                        cudaStream_t);
cudaError_t launch_spa(const DevCode &, const DecodeParams &, const EnumBuffers &, const LaunchShape &, cudaStream_t);
cudaError_t launch_sieve_kernel(const DevCode &, const EnumBuffers &, const LaunchShape &, int is_float,
                                cudaStream_t);
cudaError_t launch_batch16(const BatchArgs &, int, bool qc, int dc_max, bool reg6, const LaunchShape &,
                           cudaStream_t);
cudaError_t launch_batch8(const BatchArgs &, int, bool qc, int dc_max, bool reg6, const LaunchShape &,
                          cudaStream_t);

namespace {

enum { kLayScalar = 0, kLayPair = 1, kLaySieve = 2, kLayIs = 3, kLayPairVn = 4 };

int msg_bytes(int decoder) { return decoder == TSX_DEC_NMS_I8 ? 1 : (decoder == TSX_DEC_SPA_F32 ? 4 : 2); }
constexpr int kPairMiscBytes = 464;  // the two-codeword kernels' scratch where there is room
static_assert(sizeof(PairMisc) <= kPairMiscBytes, "the two-codeword kernels' scratch");
int post_bytes(int decoder) { return decoder == TSX_DEC_SPA_F32 ? 4 : 2; }

// odd_rows: the two-codeword kernels' variant for check degrees above 8 (QC: each row an odd number of words)
// noise: the sampling kernel keeps the noise on the set's nodes
// tight: nothing to spare, for a code that fits a CTA only so (plan)
SlotLayout make_layout(const DevCode &g, int decoder, int kind, bool odd_rows, bool noise, bool tight) {
    SlotLayout L{};
    L.tables_bytes = al16(tab_offsets(g, kind == kLayPairVn ? 2 : kind == kLayPair || kind == kLayIs ? 1 : 0).total);
    const int nw = (g.n + 31) / 32, nx = tight ? nw : (nw + 3) & ~3;
    // message slots: QC edges, or the position-major m x dc_max grid of a CSR code
    const int nmsg = g.kind == TSX_CODE_QC ? g.E : g.m * g.dc_max;
    const int nmsg2 = g.kind == TSX_CODE_QC && odd_rows && g.row_odd ? g.E_odd : nmsg;
    int x = 0;
    if (kind == kLayScalar) {
        L.r_off = x; x += al16(nmsg * msg_bytes(decoder));
        L.p_off = x; x += al16(g.n * post_bytes(decoder));
        L.xa_off = x; x += al16(nw * 4);
        L.xb_off = x; x += al16(nw * 4);
    } else if (kind == kLayPair) {
        const int rsz = decoder == TSX_DEC_NMS_I8 ? 2 : 4;
        L.r_off = x; x += al16(nmsg2 * rsz);
        L.p_off = x; x += al16(2 * g.n * 4);  // current and accumulating posteriors
        L.xa_off = x; x += al16(4 * nx * 4);
        L.xb_off = L.xa_off;
    } else if (kind == kLayPairVn) {
        L.r_off = x; x += al16(nmsg2 * 4);
        L.p_off = x; x += al16(g.n * 4);  // one posterior buffer, rebuilt by the variable-node pass
        L.xa_off = x; x += al16(4 * nx * 4);
        L.xb_off = L.xa_off;
    } else if (kind == kLayIs) {
        L.r_off = x; x += al16(nmsg2 * 4);
        L.p_off = x; x += al16(3 * g.n * 4);  // two posterior buffers and the channel values
        L.xa_off = x; x += al16(nw * 4);      // bitmask of the trapping set
        L.xb_off = x; x += noise ? kIsNoiseBytes : 0;  // the noise on its nodes, or none
    } else {
        int rbytes = 4 * g.m;
        if (rbytes < 2 * g.n) rbytes = 2 * g.n;
        L.r_off = x; x += al16(rbytes);
        L.p_off = x; x += al16(2 * g.n);
        L.xa_off = x; x += al16(nw * 4);
        L.xb_off = L.xa_off;
    }
    const bool pair = kind == kLayPair || kind == kLayPairVn;
    if (!tight && (pair || kind == kLayIs) && g.kind == TSX_CODE_QC && !g.by_rows) L.tables_bytes += al16(4 * g.m_b);
    L.misc_off = x;
    x += al16((int)(pair ? (tight ? sizeof(PairMisc) : kPairMiscBytes) : kind == kLayIs ? kIsMiscBytes : kind == kLaySieve ? sizeof(SieveMisc)
                                                                                               : sizeof(Misc)));
    L.slot_bytes = x;
    return L;
}

// dynamic shared memory of a CTA: 227 KB less 1 KB for the static part (the
// batch kernel's staged item)
constexpr int kSmemCta = 226 * 1024;

// units > 0: how many codeword groups the launch has work for (pairs of
// candidates), where the host knows it.
bool plan(const DevCode &g, int decoder, int kind, int G, int groups, int ctas_per_sm, int num_sms,
          LaunchShape *out, int max_warps = 16, long long units = 0, bool odd_rows = false,
          bool noise = true) {
    LaunchShape sh{};
    // With a little room to spare in each slot (up to 200 bytes), or without where only that fits.  The
    // shapes below were measured with it; a group more from so few bytes can take half of the others' warps
    // (sum-product, 12 groups of two warps: 43 ms, 13 of one: 62).
    int fit = 0;
    for (int tight = 0; tight < 2 && fit < 1; tight++) {
        sh.lay = make_layout(g, decoder, kind, odd_rows || g.dc_max > 8, noise, tight);
        const int room = kSmemCta - sh.lay.tables_bytes;
        fit = room >= sh.lay.slot_bytes ? room / sh.lay.slot_bytes : 0;
    }
    if (fit < 1) return false;
    if (kind == kLaySieve) G = 1;
    if (G <= 0) {
        // As many codeword groups as fit (up to one per warp) and have work, the warps shared among
        // them: while there are fewer pairs than groups, a pair takes the idle ones' warps (200
        // candidates on a 576-node code: one pair to an SM, 9 warps instead of 1, 0.80 -> 0.27 ms).
        int gr = fit < max_warps ? fit : max_warps;
        if (units > 0 && (units + num_sms - 1) / num_sms < gr) gr = (int)((units + num_sms - 1) / num_sms);
        G = max_warps / gr;
        if (G > (g.m + 31) / 32) G = (g.m + 31) / 32;  // the check pass runs over all rows at once: at most one each
        if (G < 1) G = 1;
    }
    if (G > max_warps) G = max_warps;
    int gmax_cta = max_warps / G;  // at most 32 * max_warps threads per CTA
    if (gmax_cta < 1) gmax_cta = 1;
    if (gmax_cta > fit) gmax_cta = fit;
    if (G > 1 && gmax_cta > 15) gmax_cta = 15;  // named barriers 1..15
    if (groups <= 0 || groups > gmax_cta) groups = gmax_cta;
    sh.G = G;
    sh.groups = groups;
    sh.smem_bytes = sh.lay.tables_bytes + groups * sh.lay.slot_bytes;
    sh.num_sms = num_sms;
    sh.per_sm_req = ctas_per_sm;
    sh.ctas = num_sms;
    *out = sh;
    return true;
}

// A two-codeword layout with rows filled up to an odd number of words, or as they are where only
// that fits a CTA (4 bytes a check of even degree: full 4 x 30 bases in the variable-node-pass form
// need it from Z = 364 to 372; the one-codeword kernel takes 58 ms for 3,000 candidates at Z = 368, this form
// 20.3).  Sets g.row_odd.
bool plan_rows(DevCode &g, int decoder, int kind, int G, int groups, int ctas_per_sm, int num_sms, LaunchShape *out,
               int max_warps, long long units, bool odd_rows = false) {
    for (g.row_odd = 1; g.row_odd >= 0; g.row_odd--)
        if (plan(g, decoder, kind, G, groups, ctas_per_sm, num_sms, out, max_warps, units, odd_rows)) return true;
    g.row_odd = 1;
    return false;
}

// the launch bound of the two-codeword kernel variant launch_pair picks for g
int pair_warps(const DevCode &g) {
    const bool reg6 = g.dc_min == 6 && g.dc_max == 6;
    return pair_kernel_warps(reg6 ? 6 : g.dc_max <= 8 ? 8 : 32, reg6);
}

// the two-codeword kernel keeps every biased quantity inside 16 bits
bool pair_ok(const DevCode &g, const DecodeParams &dp) {
    if (dp.decoder == TSX_DEC_SPA_F32) return false;
    const int B = dp.decoder == TSX_DEC_NMS_I8 ? 128 : 1024;
    const long long an_sat = (long long)dp.alpha_num * dp.sat;
    if (an_sat >= 65536) return false;
    const long long rmax = an_sat >> dp.alpha_shift;
    if (rmax > (dp.decoder == TSX_DEC_NMS_I8 ? 127 : B)) return false;
    if ((long long)(g.dv_max + 2) * dp.sat > 0x8000 - B) return false;
    if ((long long)g.dv_max * B > 0x8000 - dp.sat) return false;
    return true;
}

// Whether a QC code of check degree 6 (16-bit messages) takes its rows as
// lists of node numbers in shared memory, as a general code does, instead of
// working each neighbour out from the exponents: one 2-byte load and one add an edge
// instead of an 8-byte load and three adds (2640-node code, 30,000 candidates: 69.8 -> 65.7 ms;
// n = 804: 16.4 -> 14.2; n = 96: 0.60 -> 0.52).  Not where the table (2 bytes an edge) would leave
// a CTA one group instead of two or more: what one group waits for at its barriers costs more
// (16 warps in one group instead of two on an n = 4608 code: + 17 %).
int rows_table(const DevCode &g0, int decoder, int kind, int num_sms, int max_warps, long long units) {
    DevCode g = g0;
    if (g.kind != TSX_CODE_QC || decoder != TSX_DEC_NMS_I16 || g.dc_min != 6 || g.dc_max != 6) return 0;
    LaunchShape with, without;
    g.by_rows = 0;
    if (!plan(g, decoder, kind, 0, 0, 0, num_sms, &without, max_warps, units)) return 0;
    g.by_rows = 1;
    if (!plan(g, decoder, kind, 0, 0, 0, num_sms, &with, max_warps, units)) return 0;
    return with.groups > 1 || without.groups == 1;
}

}  // namespace

cudaError_t launch_decode(const DevCode &g0, const DecodeParams &dp, const EnumBuffers &b, int G, int groups,
                          int ctas_per_sm, int num_sms, int force_scalar, long long n_cand, cudaStream_t st) {
    LaunchShape sh;
    const long long units = (n_cand + 1) / 2;
    DevCode g = g0;
    // the two-codeword kernel where its bounds hold and its layout fits a CTA
    const bool try_pair = !force_scalar && pair_ok(g, dp);
    bool pair = false;
    if (try_pair) {
        g.by_rows = rows_table(g, dp.decoder, kLayPair, num_sms, pair_warps(g), units);
        const auto fits = [&](int kind) {
            return plan_rows(g, dp.decoder, kind, G, groups, ctas_per_sm, num_sms, &sh, pair_warps(g), units);
        };
        pair = fits(kLayPair);
        // QC codes of large check degree whose two-buffer layout does not fit: the variable-node-pass form
        if (!pair && g.kind == TSX_CODE_QC && dp.decoder == TSX_DEC_NMS_I16 && g.dc_max > 8 && fits(kLayPairVn))
            return launch_nms16_vn(g, dp, b, sh, st);
    }
    const int sw = scalar_warps(dp.decoder == TSX_DEC_SPA_F32, g.dc_max);
    if (!pair && !plan(g, dp.decoder, kLayScalar, G, groups, ctas_per_sm, num_sms, &sh, sw, n_cand))
        return cudaErrorInvalidConfiguration;
    // more one-warp groups than 24 fit and have work: the 32-warp form of the sum-product kernel
    if (!pair && sw == 24 && sh.G == 1 && sh.groups == 24)
        plan(g, dp.decoder, kLayScalar, 1, groups, ctas_per_sm, num_sms, &sh, 32, n_cand);
    switch (dp.decoder) {
        case TSX_DEC_NMS_I16: return launch_nms16(g, dp, b, sh, pair, st);
        case TSX_DEC_NMS_I8: return launch_nms8(g, dp, b, sh, pair, st);
        default: return launch_spa(g, dp, b, sh, st);
    }
}

cudaError_t launch_sieve(const DevCode &g, const EnumBuffers &b, int decoder, int num_sms, cudaStream_t st) {
    LaunchShape sh;
    if (!plan(g, decoder, kLaySieve, 1, 0, 0, num_sms, &sh)) return cudaErrorInvalidConfiguration;
    return launch_sieve_kernel(g, b, sh, decoder == TSX_DEC_SPA_F32 ? 1 : 0, st);
}

// variant bits: 1 = QC, 2 = int8 storage, 4 = all check-regular of degree 6,
// bits 8.. = the largest check degree
bool plan_batch(const DevCode *const *g, const DecodeParams *dp, const EnumBuffers *b, const int *G_req, int n,
                int num_sms, BatchItem *items, LaunchShape *common, int *variant) {
    if (n <= 0) return false;
    const int kind = g[0]->kind, dec = dp[0].decoder;
    bool reg6 = true, odd = false;
    int dcmax = 1, smem = 0;
    for (int i = 0; i < n; i++) odd = odd || g[i]->dc_max > 8;  // (the variant follows the largest degree)
    for (int i = 0; i < n; i++) {
        if (g[i]->kind != kind || dp[i].decoder != dec || !pair_ok(*g[i], dp[i])) return false;
        LaunchShape sh;
        int G, groups;
        items[i].scalar = 0;
        DevCode gi = *g[i];
        if (!plan_rows(gi, dec, kLayPair, 1, 1, 0, num_sms, &sh, kBatchWarps, 0, odd)) {
            items[i].scalar = 1;  // decoded by a launch of its own
            continue;
        }
        reg6 = reg6 && g[i]->dc_min == 6 && g[i]->dc_max == 6;
        if (g[i]->dc_max > dcmax) dcmax = g[i]->dc_max;
        if (G_req && G_req[i] > 0) {
            // the requested (tuned) group width, as many groups as fit
            if (!plan_rows(gi, dec, kLayPair, G_req[i], 0, 0, num_sms, &sh, kBatchWarps, 0, odd)) return false;
            G = sh.G;
            groups = sh.groups;
        } else {
            // the single-code launch's automatic shape
            if (!plan_rows(gi, dec, kLayPair, 0, 0, 0, num_sms, &sh, kBatchWarps, 0, odd)) return false;
            G = sh.G;
            groups = sh.groups;
        }
        items[i].g = gi;
        items[i].dp = dp[i];
        items[i].b = b[i];
        items[i].lay = sh.lay;
        items[i].G = G;
        items[i].groups = groups;
        const int need = sh.lay.tables_bytes + groups * sh.lay.slot_bytes;
        if (need > smem) smem = need;
    }
    LaunchShape sh{};
    sh.G = 1;
    sh.groups = kBatchWarps;
    sh.smem_bytes = smem;
    sh.num_sms = num_sms;
    sh.per_sm_req = 0;
    sh.ctas = num_sms;
    *common = sh;
    *variant = (kind == TSX_CODE_QC ? 1 : 0) | (dec == TSX_DEC_NMS_I8 ? 2 : 0) | (reg6 ? 4 : 0) | (dcmax << 8);
    return true;
}

cudaError_t launch_batch(const BatchArgs &items, int n, int variant, const LaunchShape &sh, cudaStream_t st) {
    const bool qc = variant & 1, i8 = variant & 2, reg6 = variant & 4;
    const int dcmax = variant >> 8;
    return i8 ? launch_batch8(items, n, qc, dcmax, reg6, sh, st) : launch_batch16(items, n, qc, dcmax, reg6, sh, st);
}

bool plan_is_shape(DevCode &g, const DecodeParams &dp, LaunchShape *sh, int num_sms, bool *noise) {
    if (!pair_ok(g, dp)) return false;
    g.by_rows = rows_table(g, TSX_DEC_NMS_I16, kLayIs, num_sms, 16, 0);
    // (the launch bounds of is_kernel)
    const int warps = g.kind == TSX_CODE_QC && g.dc_max > 8 ? kIsWarps : 16;
    // with the set's noise kept and rows filled up to odd lengths where there is room for them
    for (int form = 0; form < 3; form++) {
        *noise = form == 0;
        g.row_odd = form < 2;
        if (plan(g, TSX_DEC_NMS_I16, kLayIs, 0, 0, 0, num_sms, sh, warps, 0, false, *noise)) return true;
    }
    return false;
}

bool decode_fits(const DevCode &g, int decoder) {
    LaunchShape sh;
    return plan(g, decoder, kLayScalar, 1, 1, 0, 1, &sh) && plan(g, decoder, kLaySieve, 1, 1, 0, 1, &sh);
}

// ---------------------------------------------------------------------------
// compaction of the hash table
// ---------------------------------------------------------------------------
__global__ void compact_kernel(EnumBuffers b, int *ts_off, int *ts_count, int *ts_thr, int *slot_map) {
    for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s <= b.cap_mask;
         s += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long tag = b.tags[s];
        if (!tag) continue;
        const unsigned idx = atomicAdd(&b.ctr->n_ts, 1u);
        ts_off[idx] = (int)(tag & 0xffffffffull);
        ts_count[idx] = b.t_count[s];
        ts_thr[idx] = b.t_thr[s];
        slot_map[s] = (int)idx;
    }
}

__global__ void remap_kernel(EnumBuffers b, long long n_rec, const int *slot_map) {
    const long long total = (long long)b.ctr->n_cand_total;
    const long long end = b.cand_end < 0 || b.cand_end > total ? total : b.cand_end;
    long long n = end - b.cand_begin;
    if (n > n_rec) n = n_rec;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int s = b.c_slot[i];
        if (s >= 0) b.c_slot[i] = slot_map[s];
    }
}

cudaError_t launch_compact(const EnumBuffers &b, long long n_rec, int *ts_off, int *ts_count, int *ts_thr,
                           int *slot_map, cudaStream_t st) {
    const long long cap = (long long)b.cap_mask + 1;
    int blocks = (int)((cap + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    compact_kernel<<<blocks, 256, 0, st>>>(b, ts_off, ts_count, ts_thr, slot_map);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int rb = (int)((n_rec + 255) / 256);
    if (rb > 4096) rb = 4096;
    if (rb < 1) rb = 1;
    remap_kernel<<<rb, 256, 0, st>>>(b, n_rec, slot_map);
    return cudaGetLastError();
}

}  // namespace tsx
