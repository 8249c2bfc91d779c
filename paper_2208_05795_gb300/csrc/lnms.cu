// lnms.cu -- the simulation decoder of Sec. III (the FER curves of Fig. 2):
// quantized normalized layered min-sum with LLR, check-to-variable and
// variable-to-check widths of 4, 4 and 6 bits and 20 iterations, and the
// frame-error simulation around it.
//
// Readings (the paper names the widths and nothing else): every quantity is
// a signed integer and a w-bit value saturates to +-(2^(w-1) - 1); a layer
// is a row block of the QC base matrix (its checks touch distinct variable
// nodes, so they are updated in parallel); the posterior P_v starts at the
// saturated channel value and is kept at the variable-to-check width; per
// layer and check, q = sat_v2c(P_v - r) for its edges, then
// r = sign * sat_c2v((alpha_num * m) >> alpha_shift) with m the minimum |q|
// of the other edges (sgn 0 = +1), then P_v = sat_v2c(q + r); after each
// full iteration x = [P < 0] and the syndrome is checked (also before the
// first).  Failure: x != 0 at the end.
//
// Two frames per lane (lnms_pair_kernel): a group of G warps owns two frames,
// every shared-memory word holds both frames' posterior or message in 16-bit
// halves with the representation of decode_pair.cuh, lanes take the rows of a
// layer and a barrier separates the layers; a frame that ends is replaced
// while the other goes on.  Codes whose words do not fit a CTA's shared memory, and
// normalizations whose products leave 16 bits, take one frame per group
// (lnms_kernel): P (int8, n) and r (int8, E).  Frames come from a work queue: either the caller's LLRs or BPSK
// over AWGN drawn on the device (the noise generator of the
// importance-sampling kernel, mu = 0), the channel LLR 2 y / sigma^2 scaled,
// rounded half away from zero and saturated to the LLR width.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "decode_pair.cuh"
#include "noise.cuh"

namespace tsx {
namespace {

struct LnmsArgs {
    int K, lim_llr, lim_c2v, lim_v2c, an, as;
    const int8_t *llr;           // [n_frames][n] channel values, or null: drawn noise
    unsigned long long job;      // noise: Philox key
    long long f0;                // noise: sample index of frame 0
    float sigf, cq;              // noise: sigma and the LLR scale 2 llr_scale / sigma^2
    long long n_frames;
    unsigned char *fail;         // [n_frames]
    int *iters;                  // [n_frames] or null
    int *weight;                 // [n_frames] or null: Hamming weight of x (bit errors)
    unsigned char *x_out;        // [n_frames][n] or null
    unsigned long long *queue;   // work queue (frames)
    Counters *ctr;
};

// warps per CTA of the two-frame kernel (its launch bound); 16, 20 and 28 measured within 7 %
constexpr int kLnmsWarps = 24;
static_assert(kLnmsWarps <= kMaxGroupWarps, "the groups' reduction scratch");

struct LnmsLayout {
    int tables_bytes, p_off, r_off, misc_off, slot_bytes;
};

LnmsLayout lnms_layout(const DevCode &g) {
    LnmsLayout L{};
    L.tables_bytes = al16(tab_offsets(g, false).total);
    int x = 0;
    L.p_off = x; x += al16(g.n);
    L.r_off = x; x += al16(g.E);
    L.misc_off = x; x += al16((int)sizeof(Misc));
    L.slot_bytes = x;
    return L;
}

__device__ __forceinline__ int satw(int x, int lim) { return min(max(x, -lim), lim); }

// round half away from zero (exact), clamped before the conversion
__device__ __forceinline__ int round_half_away(float x, int lim) {
    return (int)fminf(fmaxf(roundf(x), (float)-lim), (float)lim);
}

template <int DCMAX>
__global__ void __launch_bounds__(512, 1) lnms_kernel(DevCode g, LnmsArgs a, LnmsLayout lay, int G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SGraph sg = load_tables(g, smem);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp / G;
    unsigned char *slot = smem + lay.tables_bytes + grp * lay.slot_bytes;
    Misc *misc = (Misc *)(slot + lay.misc_off);
    Grp gp;
    gp.G = G;
    gp.T = 32 * G;
    gp.gw = warp - grp * G;
    gp.gt = gp.gw * 32 + lane;
    gp.lane = lane;
    gp.bar = 1 + grp;
    gp.red = misc->red;
    int8_t *P = (int8_t *)(slot + lay.p_off);
    int8_t *R = (int8_t *)(slot + lay.r_off);
    const int n = g.n, Z = g.Z;
    long long my_frames = 0, my_it = 0, my_fail = 0;

    // unsatisfied checks of x = [P < 0] (group total)
    auto unsat = [&]() {
        int u = 0;
        for (int c = gp.gt; c < g.m; c += gp.T) {
            const int i = c / Z, r = c - i * Z;
            const int deg = sg.rdeg[i];
            int par = 0;
            for (int p = 0; p < deg; p++) par ^= P[sg.rjz[i * g.dc_max + p] + wrapZ(r + sg.rs[i * g.dc_max + p], Z)] < 0;
            u += par;
        }
        return gp.sum(u);
    };

    while (true) {
        if (gp.gt == 0) misc->bcast[0] = (long long)atomicAdd(a.queue, 1ull);
        gp.sync();
        const long long f = misc->bcast[0];
        gp.sync();
        if (f >= a.n_frames) break;
        // the channel
        if (a.llr) {
            const int8_t *src = a.llr + f * (long long)n;
            for (int v = gp.gt; v < n; v += gp.T) P[v] = (int8_t)satw(src[v], a.lim_llr);
        } else {
            for (int q = gp.gt; 4 * q < n; q += gp.T) {
                float gq[4];
                normals4(a.job, (unsigned long long)(a.f0 + f), (uint32_t)q, gq);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int v = 4 * q + j;
                    if (v < n) {
                        const float y = hadd(1.0f, hmul(a.sigf, gq[j]));
                        P[v] = (int8_t)round_half_away(hmul(y, a.cq), a.lim_llr);
                    }
                }
            }
        }
        for (int e = gp.gt; e < g.E; e += gp.T) R[e] = 0;
        gp.sync();
        int u = unsat();
        int k = 0;
        while (u != 0 && k < a.K) {
            k++;
            for (int i = 0; i < g.m_b; i++) {
                const int deg = sg.rdeg[i];
                const int e0 = sg.reoff[i];
                const int32_t *rjz = sg.rjz + i * g.dc_max;
                const int16_t *rs = sg.rs + i * g.dc_max;
                for (int r = gp.gt; r < Z; r += gp.T) {
                    int q[DCMAX], vv[DCMAX];
                    int m1 = 1 << 20, m2 = 1 << 20, neg = 0;
#pragma unroll
                    for (int p = 0; p < DCMAX; p++) {
                        if (p < deg) {
                            const int v = rjz[p] + wrapZ(r + rs[p], Z);
                            vv[p] = v;
                            const int qq = satw((int)P[v] - (int)R[e0 + p * Z + r], a.lim_v2c);
                            q[p] = qq;
                            neg ^= qq < 0;
                            const int mag = abs(qq);
                            m2 = min(m2, max(m1, mag));  // the two smallest magnitudes, no branch
                            m1 = min(m1, mag);
                        }
                    }
#pragma unroll
                    for (int p = 0; p < DCMAX; p++) {
                        if (p < deg) {
                            // the smallest of the others: m2 for an edge at the minimum (with a tie m2 = m1)
                            const int mn = abs(q[p]) == m1 ? m2 : m1;
                            int mag = deg == 1 ? a.lim_c2v : satw((a.an * mn) >> a.as, a.lim_c2v);
                            const int rr = (neg ^ (q[p] < 0)) ? -mag : mag;
                            R[e0 + p * Z + r] = (int8_t)rr;
                            P[vv[p]] = (int8_t)satw(q[p] + rr, a.lim_v2c);
                        }
                    }
                }
                gp.sync();
            }
            u = unsat();
        }
        // x = [P < 0]
        int w = 0;
        for (int v = gp.gt; v < n; v += gp.T) {
            const int bit = P[v] < 0;
            w += bit;
            if (a.x_out) a.x_out[f * (long long)n + v] = (unsigned char)bit;
        }
        w = gp.sum(w);
        if (gp.gt == 0) {
            a.fail[f] = w != 0;
            if (a.iters) a.iters[f] = k;
            if (a.weight) a.weight[f] = w;
        }
        my_frames++;
        my_it += k;
        my_fail += w != 0;
        gp.sync();
    }
    if (gp.gt == 0) {
        atomicAdd(&a.ctr->decodes, (unsigned long long)my_frames);
        atomicAdd(&a.ctr->iterations, (unsigned long long)my_it);
        atomicAdd(&a.ctr->edge_updates, (unsigned long long)my_it * (unsigned long long)g.E);
        atomicAdd(&a.ctr->n_fail, (unsigned long long)my_fail);
    }
}

// The same decoder, two frames per lane.  Per edge of two frames the passes
// over a layer's rows take about 34 warp instructions (the one-frame form 75
// per frame).
__global__ void __launch_bounds__(32 * kLnmsWarps, 1) lnms_pair_kernel(DevCode g, LnmsArgs a, SlotLayout lay, int G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SGraph sg = load_tables(g, smem, 1, true);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp / G;
    unsigned char *slot = smem + lay.tables_bytes + grp * lay.slot_bytes;
    Misc *misc = (Misc *)(slot + lay.misc_off);
    Grp gp;
    gp.G = G;
    gp.T = 32 * G;
    gp.gw = warp - grp * G;
    gp.gt = gp.gw * 32 + lane;
    gp.lane = lane;
    gp.bar = 1 + grp;
    gp.red = misc->red;
    unsigned *P = (unsigned *)(slot + lay.p_off);
    unsigned *R = (unsigned *)(slot + lay.r_off);
    const unsigned Pa = saddr(P), Ra = saddr(R), rt0 = saddr(sg.rt);
    const int n = g.n, Z = g.Z;
    const unsigned Z4 = 4u * (unsigned)Z;
    // clamps of the biased words
    const unsigned hi = (kBeta + (unsigned)a.lim_v2c) * 0x00010001u, lo = (kBeta - (unsigned)a.lim_v2c) * 0x00010001u;
    const unsigned limr = (unsigned)a.lim_c2v * 0x00010001u;
    const unsigned amask = (0xFFFFu >> a.as) * 0x00010001u, BAN = kBeta * 0x00010001u * (unsigned)a.an;
    long long my_frames = 0, my_it = 0, my_fail = 0;
    long long f[2];
    int k[2];

    // the next frame of half hh: channel values into its half of P, zero into its half of R
    auto load = [&](int hh) {
        if (gp.gt == 0) misc->bcast[0] = (long long)atomicAdd(a.queue, 1ull);
        gp.sync();
        f[hh] = misc->bcast[0] < a.n_frames ? misc->bcast[0] : -1;
        gp.sync();
        k[hh] = 0;
        uint16_t *Ph = (uint16_t *)P + hh;
        if (f[hh] < 0) {  // an idle half decodes the all-zero word
            for (int v = gp.gt; v < n; v += gp.T) Ph[2 * v] = (uint16_t)kBeta;
        } else if (a.llr) {
            const int8_t *src = a.llr + f[hh] * (long long)n;
            if ((((uintptr_t)a.llr | (uintptr_t)n) & 3) == 0) {
                for (int q = gp.gt; 4 * q < n; q += gp.T) {
                    const char4 c = __ldg((const char4 *)src + q);
                    Ph[8 * q] = (uint16_t)(kBeta + satw(c.x, a.lim_llr));
                    Ph[8 * q + 2] = (uint16_t)(kBeta + satw(c.y, a.lim_llr));
                    Ph[8 * q + 4] = (uint16_t)(kBeta + satw(c.z, a.lim_llr));
                    Ph[8 * q + 6] = (uint16_t)(kBeta + satw(c.w, a.lim_llr));
                }
            } else {
                for (int v = gp.gt; v < n; v += gp.T) Ph[2 * v] = (uint16_t)(kBeta + satw(src[v], a.lim_llr));
            }
        } else {
            for (int q = gp.gt; 4 * q < n; q += gp.T) {
                float gq[4];
                normals4(a.job, (unsigned long long)(a.f0 + f[hh]), (uint32_t)q, gq);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int v = 4 * q + j;
                    if (v < n) {
                        const float y = hadd(1.0f, hmul(a.sigf, gq[j]));
                        Ph[2 * v] = (uint16_t)(kBeta + round_half_away(hmul(y, a.cq), a.lim_llr));
                    }
                }
            }
        }
        // (a word is (r1 << 16) + r0: the other half's message alone)
        for (int e = gp.gt; e < g.E_odd; e += gp.T)
            R[e] = hh == 0 ? (R[e] + 0x8000u) & 0xFFFF0000u : (unsigned)(int)(int16_t)R[e];
    };
    // x = [P < 0] of half hh out: weight, decision, iterations
    auto finish = [&](int hh) {
        int w = 0;
        const unsigned bit = 15u + 16u * hh;
        if (a.x_out && (((uintptr_t)a.x_out | (uintptr_t)n) & 3) == 0) {
            unsigned *dst = (unsigned *)(a.x_out + f[hh] * (long long)n);
            for (int q = gp.gt; 4 * q < n; q += gp.T) {
                const uint4 p = *(const uint4 *)(P + 4 * q);
                const unsigned x = ((~p.x >> bit) & 1u) | (((~p.y >> bit) & 1u) << 8) | (((~p.z >> bit) & 1u) << 16) |
                                   (((~p.w >> bit) & 1u) << 24);
                w += __popc(x);
                dst[q] = x;
            }
        } else {
            for (int v = gp.gt; v < n; v += gp.T) {
                const unsigned x = (~P[v] >> bit) & 1u;
                w += (int)x;
                if (a.x_out) a.x_out[f[hh] * (long long)n + v] = (unsigned char)x;
            }
        }
        w = gp.sum(w);
        if (gp.gt == 0) {
            a.fail[f[hh]] = w != 0;
            if (a.iters) a.iters[f[hh]] = k[hh];
            if (a.weight) a.weight[f[hh]] = w;
        }
        my_frames++;
        my_it += k[hh];
        my_fail += w != 0;
    };
    // byte offset of the p-th node of a row: column block start + (r + shift) mod Z
    auto at = [&](unsigned x, unsigned y, unsigned r4) {
        const unsigned t = r4 + y;
        return Pa + x + __viaddmin_u32(t, 0u - Z4, t);
    };
    auto pos = [&](unsigned rt, int p, unsigned r4) {
        const uint2 e = lds64(rt + 8u * (unsigned)p);
        return at(e.x, e.y, r4);
    };
    auto pos2 = [&](unsigned rt, int p, unsigned r4, unsigned *o) {  // p even: two table entries in one load
        const uint4 e = lds128(rt + 8u * (unsigned)p);
        o[0] = at(e.x, e.y, r4);
        o[1] = at(e.z, e.w, r4);
    };

    for (int e = gp.gt; e < g.E_odd; e += gp.T) R[e] = 0;
    gp.sync();
    load(0);
    load(1);
    gp.sync();
    while (f[0] >= 0 || f[1] >= 0) {
        // unsatisfied checks of x = [P < 0], half 0 in the low 16 bits
        int u = 0;
        for (int i = 0; i < g.m_b; i++) {
            const int deg = sg.rdeg[i];
            const unsigned rt = rt0 + 8u * (unsigned)(i * rt_row(g));
            for (int r = gp.gt; r < Z; r += gp.T) {
                unsigned sp = (deg & 1) ? 0x80008000u : 0u;
                int p = 0;
#pragma unroll 1
                for (; p + 4 <= deg; p += 4) {
                    unsigned o[4];
                    pos2(rt, p, 4u * r, o);
                    pos2(rt, p + 2, 4u * r, o + 2);
                    sp ^= lds32(o[0]) ^ lds32(o[1]) ^ lds32(o[2]) ^ lds32(o[3]);
                }
#pragma unroll 1
                for (; p < deg; p++) sp ^= lds32(pos(rt, p, 4u * r));
                u += (int)((sp >> 15) & 0x00010001u);
            }
        }
        u = gp.sum(u);
        bool fresh = false;
        for (int hh = 0; hh < 2; hh++) {
            if (f[hh] < 0) continue;
            const int uh = hh == 0 ? (u & 0xFFFF) : (u >> 16);
            if (uh != 0 && k[hh] < a.K) continue;
            finish(hh);
            gp.sync();
            load(hh);
            fresh = true;
        }
        if (fresh) {  // u_0 of the new frame first
            gp.sync();
            continue;
        }
        for (int i = 0; i < g.m_b; i++) {
            const int deg = sg.rdeg[i];
            const unsigned rt = rt0 + 8u * (unsigned)(i * rt_row(g));
            for (int r = gp.gt; r < Z; r += gp.T) {
                const unsigned r4 = 4u * (unsigned)r;
                const unsigned ra = Ra + 4u * (unsigned)(sg.reoff[i] + r * (deg | 1));
                unsigned sx = 0, M1 = 0, M2 = 0;  // the two largest beta - |q|
                // q = sat(P - r), left in the message's word
                auto first = [&](auto width, int p) {
                    constexpr int W = decltype(width)::value;
                    unsigned x[W], na[W];
                    if constexpr (W == 1) x[0] = pos(rt, p, r4);
                    else
#pragma unroll
                        for (int e = 0; e < W; e += 2) pos2(rt, p + e, r4, x + e);
#pragma unroll
                    for (int e = 0; e < W; e++) x[e] = lds32(x[e]) - lds32(ra + 4u * (unsigned)(p + e));
#pragma unroll
                    for (int e = 0; e < W; e++) {
                        x[e] = vmaxu2(vminu2(x[e], hi), lo);
                        sx ^= x[e];
                        na[e] = vminu2(x[e], (~x[e]) + 0x00010001u);
                    }
#pragma unroll
                    for (int e = 0; e < W; e++) sts32(ra + 4u * (unsigned)(p + e), x[e]);
                    if constexpr (W == 1) track_max(na[0], M1, M2);
                    else
#pragma unroll
                        for (int e = 0; e < W; e += 2) track_max2(na[e], na[e + 1], M1, M2);
                };
                int p = 0;
#pragma unroll 1
                for (; p + 4 <= deg; p += 4) first(Int<4>{}, p);
                if (deg & 2) {
                    first(Int<2>{}, p);
                    p += 2;
                }
                if (deg & 1) first(Int<1>{}, p);
                // output magnitudes (edge_out of decode_pair.cuh: the saturation keeps o2 - o1 <= min2 - min1)
                unsigned o1 = vminu2(((BAN - M1 * (unsigned)a.an) >> a.as) & amask, limr);
                unsigned o2 = vminu2(((BAN - M2 * (unsigned)a.an) >> a.as) & amask, limr);
                if (deg == 1) o1 = o2 = limr;
                const unsigned S = vadd2(o2, (~M1) + 0x00010001u);
                sx ^= ((deg - 1) & 1) ? 0x80008000u : 0u;
                auto second = [&](auto width, int p) {
                    constexpr int W = decltype(width)::value;
                    unsigned po[W], x[W];
                    if constexpr (W == 1) po[0] = pos(rt, p, r4);
                    else
#pragma unroll
                        for (int e = 0; e < W; e += 2) pos2(rt, p + e, r4, po + e);
#pragma unroll
                    for (int e = 0; e < W; e++) x[e] = lds32(ra + 4u * (unsigned)(p + e));
#pragma unroll
                    for (int e = 0; e < W; e++) {
                        const unsigned na = vminu2(x[e], (~x[e]) + 0x00010001u);
                        const unsigned neg = spread15(sx ^ x[e]);
                        const unsigned w = (vmaxs2(vadd2(na, S), o1) ^ neg) - neg;
                        sts32(ra + 4u * (unsigned)(p + e), w);
                        sts32(po[e], vmaxu2(vminu2(x[e] + w, hi), lo));
                    }
                };
                p = 0;
#pragma unroll 1
                for (; p + 4 <= deg; p += 4) second(Int<4>{}, p);
                if (deg & 2) {
                    second(Int<2>{}, p);
                    p += 2;
                }
                if (deg & 1) second(Int<1>{}, p);
            }
            gp.sync();
        }
        k[0]++;
        k[1]++;
    }
    if (gp.gt == 0) {
        atomicAdd(&a.ctr->decodes, (unsigned long long)my_frames);
        atomicAdd(&a.ctr->iterations, (unsigned long long)my_it);
        atomicAdd(&a.ctr->edge_updates, (unsigned long long)my_it * (unsigned long long)g.E);
        atomicAdd(&a.ctr->n_fail, (unsigned long long)my_fail);
    }
}

constexpr int kSmemCta = 226 * 1024;

struct LnmsShape {
    LnmsLayout lay;
    int G, groups, smem;
};

// shape of the two-frame kernel; false: its words do not fit a CTA, or products alpha_num |q| leave 16 bits
bool lnms_pair_shape(const DevCode &g, const LnmsArgs &a, int num_sms, LaunchShape *sh) {
    if ((long long)a.an * a.lim_v2c > 0xFFFF) return false;
    SlotLayout L{};
    L.tables_bytes = al16(tab_offsets(g, 1).total) + al16(4 * g.m_b);  // (the measured shapes' sizes: see plan())
    int x = 0;
    L.r_off = x; x += al16(4 * g.E_odd);
    L.p_off = x; x += al16(4 * g.n);
    L.misc_off = x; x += al16((int)sizeof(Misc));
    L.slot_bytes = x;
    const int fit = (kSmemCta - L.tables_bytes) / L.slot_bytes;
    if (fit < 1) return false;
    // as many pairs as fit and have work, a layer's rows shared by the warps
    const long long units = (a.n_frames + 1) / 2, per = (units + num_sms - 1) / num_sms;
    int gr = fit < kLnmsWarps ? fit : kLnmsWarps;
    if (per < gr) gr = (int)per;
    int G = kLnmsWarps / gr;
    if (G > (g.Z + 31) / 32) G = (g.Z + 31) / 32;
    int groups = kLnmsWarps / G;
    if (groups > fit) groups = fit;
    if (G > 1 && groups > 15) groups = 15;  // named barriers 1..15
    sh->lay = L;
    sh->G = G;
    sh->groups = groups;
    sh->smem_bytes = L.tables_bytes + groups * L.slot_bytes;
    sh->num_sms = num_sms;
    sh->per_sm_req = 0;
    return true;
}

bool lnms_shape(const DevCode &g, LnmsShape *sh) {
    sh->lay = lnms_layout(g);
    const int fit = (kSmemCta - sh->lay.tables_bytes) / sh->lay.slot_bytes;
    if (fit < 1) return false;
    int G = g.Z / 128;
    if (G < 1) G = 1;
    if (G > 4) G = 4;
    int groups = 16 / G;
    if (groups > fit) groups = fit;
    if (G > 1 && groups > 15) groups = 15;
    sh->G = G;
    sh->groups = groups;
    sh->smem = sh->lay.tables_bytes + groups * sh->lay.slot_bytes;
    return true;
}

template <class Kern>
cudaError_t launch_lnms_t(Kern k, const LnmsShape &sh, int num_sms, cudaStream_t st, const DevCode &g,
                          const LnmsArgs &a) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sh.smem);
    if (e != cudaSuccess) return e;
    const int threads = sh.groups * sh.G * 32;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, sh.smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    k<<<occ * num_sms, threads, sh.smem, st>>>(g, a, sh.lay, sh.G);
    return cudaGetLastError();
}

cudaError_t launch_lnms(const DevCode &g, const LnmsArgs &a, int num_sms, cudaStream_t st) {
    LaunchShape ps{};
    if (lnms_pair_shape(g, a, num_sms, &ps)) return launch_persistent(lnms_pair_kernel, ps, st, g, a, ps.lay, ps.G);
    LnmsShape sh;
    if (!lnms_shape(g, &sh)) return cudaErrorInvalidConfiguration;
    if (g.dc_max <= 8) return launch_lnms_t(lnms_kernel<8>, sh, num_sms, st, g, a);
    return launch_lnms_t(lnms_kernel<32>, sh, num_sms, st, g, a);
}

int lnms_check(const tsx_code *code, const tsx_lnms_params *p) {
    if (!code || !p) return TSX_EINVAL;
    if (p->K < 0 || p->K > 100000) return TSX_EINVAL;
    if (p->llr_bits < 2 || p->llr_bits > 8 || p->c2v_bits < 2 || p->c2v_bits > 8 || p->v2c_bits < 2 ||
        p->v2c_bits > 8)
        return TSX_EINVAL;
    if (p->alpha_shift < 0 || p->alpha_shift > 15 || p->alpha_num < 1 || p->alpha_num > (1 << p->alpha_shift))
        return TSX_EINVAL;
    const DevCode &g = *code_dev(code);
    if (g.kind != TSX_CODE_QC) return TSX_EUNSUPPORTED;  // layers are the row blocks of a QC base
    // every row block is one circulant per column block (distinct variable nodes per layer)
    LnmsShape sh;
    if (!lnms_shape(g, &sh)) return TSX_EUNSUPPORTED;
    return TSX_OK;
}

void fill_args(const tsx_lnms_params *p, LnmsArgs &a) {
    a.K = p->K;
    a.lim_llr = (1 << (p->llr_bits - 1)) - 1;
    a.lim_c2v = (1 << (p->c2v_bits - 1)) - 1;
    a.lim_v2c = (1 << (p->v2c_bits - 1)) - 1;
    a.an = p->alpha_num;
    a.as = p->alpha_shift;
}

}  // namespace
}  // namespace tsx

using namespace tsx;

extern "C" void lnms_params_default(tsx_lnms_params *p) {
    if (!p) return;
    p->K = 20;
    p->llr_bits = 4;
    p->c2v_bits = 4;
    p->v2c_bits = 6;
    p->alpha_num = 3;
    p->alpha_shift = 2;
}

extern "C" void sim_params_default(tsx_sim_params *p) {
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->ebn0_db = 4.0;
    p->rate = 0.0;
    p->llr_scale = 1.0;
    p->max_frames = 100000;
    p->max_errors = 200;
    p->job_key = 0;
    p->frame_begin = 0;
}

extern "C" int lnms_decode(tsx_code *code, const tsx_lnms_params *p, const int8_t *llr, int64_t n_frames,
                           uint8_t *fail, int32_t *iters, uint8_t *x, void *stream) {
    int st = lnms_check(code, p);
    if (st != TSX_OK) return st;
    if (n_frames < 0) return TSX_EINVAL;
    if (n_frames == 0) return TSX_OK;
    if (!llr || !fail) return TSX_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    Counters *ctr = nullptr;
    if (pool_alloc((void **)&ctr, sizeof(Counters), s) != cudaSuccess) return TSX_ENOMEM;
    LnmsArgs a{};
    fill_args(p, a);
    a.llr = llr;
    a.n_frames = n_frames;
    a.fail = fail;
    a.iters = iters;
    a.x_out = x;
    a.ctr = ctr;
    a.queue = &ctr->next_cand;
    if (cudaMemsetAsync(ctr, 0, sizeof(Counters), s) != cudaSuccess ||
        launch_lnms(*code_dev(code), a, code_num_sms(code), s) != cudaSuccess)
        st = TSX_ECUDA;
    cudaFreeAsync(ctr, s);
    return st;
}

extern "C" int lnms_simulate(tsx_code *code, const tsx_lnms_params *p, const tsx_sim_params *sp, void *stream,
                             tsx_sim_result *out, uint8_t *fail_out) {
    int st = lnms_check(code, p);
    if (st != TSX_OK) return st;
    if (!sp || !out || sp->max_frames < 0 || sp->max_errors < 0 || sp->frame_begin < 0 || !(sp->llr_scale > 0.0))
        return TSX_EINVAL;
    memset(out, 0, sizeof(*out));
    const DevCode &g = *code_dev(code);
    const double R = sp->rate > 0.0 ? sp->rate : 1.0 - (double)g.m / g.n;
    if (!(R > 0.0)) return TSX_EINVAL;
    const double s2 = 1.0 / (2.0 * R * std::pow(10.0, sp->ebn0_db / 10.0));
    cudaStream_t s = (cudaStream_t)stream;
    const long long chunk = 1 << 16;
    unsigned char *d_fail = nullptr;
    int *d_w = nullptr, *d_it = nullptr;
    Counters *ctr = nullptr;
    if (cudaMalloc(&d_fail, chunk) != cudaSuccess) return TSX_ENOMEM;
    if (cudaMalloc(&d_w, sizeof(int) * chunk) != cudaSuccess || cudaMalloc(&d_it, sizeof(int) * chunk) != cudaSuccess ||
        cudaMalloc(&ctr, sizeof(Counters)) != cudaSuccess) {
        cudaFree(d_fail);
        cudaFree(d_w);
        cudaFree(d_it);
        return TSX_ENOMEM;
    }
    std::vector<unsigned char> hf(chunk);
    std::vector<int> hw(chunk), hit(chunk);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float ms_total = 0.0f;
    LnmsArgs a{};
    fill_args(p, a);
    a.job = sp->job_key;
    a.sigf = (float)std::sqrt(s2);
    a.cq = (float)(2.0 * sp->llr_scale / s2);
    a.fail = d_fail;
    a.weight = d_w;
    a.iters = d_it;
    a.ctr = ctr;
    a.queue = &ctr->next_cand;
    long long done = 0;
    bool stop = false;
    while (!stop && done < sp->max_frames) {
        const long long nf = std::min<long long>(chunk, sp->max_frames - done);
        a.f0 = sp->frame_begin + done;
        a.n_frames = nf;
        float ms = 0.0f;
        if (cudaMemsetAsync(ctr, 0, sizeof(Counters), s) != cudaSuccess || cudaEventRecord(e0, s) != cudaSuccess ||
            launch_lnms(g, a, code_num_sms(code), s) != cudaSuccess || cudaEventRecord(e1, s) != cudaSuccess ||
            cudaMemcpyAsync(hf.data(), d_fail, nf, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(hw.data(), d_w, sizeof(int) * nf, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(hit.data(), d_it, sizeof(int) * nf, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            st = TSX_ECUDA;
            break;
        }
        ms_total += ms;
        // frames in order up to the one that reaches max_errors
        for (long long i = 0; i < nf; i++) {
            out->frames++;
            out->iterations += hit[i];
            out->edge_updates += (int64_t)hit[i] * g.E;
            if (fail_out) fail_out[done + i] = hf[i];
            if (hf[i]) {
                out->frame_errors++;
                out->bit_errors += hw[i];
                if (sp->max_errors > 0 && out->frame_errors >= sp->max_errors) {
                    stop = true;
                    break;
                }
            }
        }
        done += nf;
    }
    out->ms = ms_total;
    if (out->frames) {
        out->fer = (double)out->frame_errors / out->frames;
        out->ber = (double)out->bit_errors / ((double)out->frames * g.n);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(d_fail);
    cudaFree(d_w);
    cudaFree(d_it);
    cudaFree(ctr);
    return st;
}
