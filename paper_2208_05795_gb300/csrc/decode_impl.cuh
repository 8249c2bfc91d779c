// decode_impl.cuh -- the persistent impulse-decoding kernel (instantiated
// per decoder in decode_i16.cu, decode_i8.cu and decode_spa.cu).
//
// One group of G warps owns one codeword slot in shared memory and runs,
// for each candidate impulse set it pops from a device work queue:
//   * the amplitude bisection (Cole's error impulse, Sec. III): a decode at
//     the largest amplitude, then up to s halvings keeping the failing end;
//   * each decode: flooding message passing from the all-zero codeword with
//     L_v = base everywhere except the impulse nodes, syndrome early exit,
//     and tracking of the error pattern x_k with the fewest unsatisfied
//     checks u_k = w_H(H x_k) from iteration floor(girth/2) on (Sec. III);
//   * on failure: the sieve S1 = Tree(X), else S2 = Tree(TS(X)), with
//     X = supp(x*) u I (Sec. III), the (a,b) classification (Sec. II), the
//     canonical form under the circulant shift and orbit size, and an
//     insert into the device hash table of distinct trapping sets.
// Messages never leave shared memory: per codeword the check-to-variable
// messages R[E] and posteriors P[n]; the variable-to-check messages are
// recomputed as clamp(P_v - r) when a check reads them.  Neighbour indices
// of QC codes come from the exponent matrix: (r + a) mod Z.
#pragma once
#include "fdiv.cuh"
#include "graph.cuh"
#include "kernels.cuh"

namespace tsx {
namespace {  // each decoder translation unit gets its own copy

// ---------------------------------------------------------------------------
// decoder policies
// ---------------------------------------------------------------------------
struct DecNms16 {
    using msg = int16_t;
    using post = int16_t;
    using lv = int;
    static constexpr bool kFloat = false;
};
struct DecNms8 {
    using msg = int8_t;
    using post = int16_t;
    using lv = int;
    static constexpr bool kFloat = false;
};
struct DecSpa {
    using msg = float;
    using post = float;
    using lv = float;
    static constexpr bool kFloat = true;
};

__host__ __device__ inline int al16(int x) { return (x + 15) & ~15; }

// entries in a row of the two-codeword kernels' QC table: even, so that two of them are one 16-byte load
__host__ __device__ inline int rt_row(const DevCode &g) { return (g.dc_max + 1) & ~1; }

struct TabOff {
    int rdeg, reoff, rjz, rs, rt, ct, cdeg, ceoff, cs, ciz;
    int c_ptr, c_vn, v_ptr, v_edge;
    int total;
};

// pair = the tables of the two-codeword kernels: no per-variable edge lists
// for general codes (they have no variable-node pass), and for QC codes the
// column start and shift of each position as one 8-byte entry in byte units
// (pair = 2: and the column entries of the variable-node-pass form)
__host__ __device__ inline TabOff tab_offsets(const DevCode &g, int pair = 0) {
    TabOff o{};
    int x = 0;
    if (pair && g.by_rows) {
        o.c_vn = x; x += al16(g.E * 2);
        o.total = x;
        return o;
    }
    if (g.kind == TSX_CODE_QC) {
        o.rdeg = x; x += al16(g.m_b * 2);
        o.reoff = x; x += al16(g.m_b * 4);
        if (pair) {
            o.rt = x; x += al16(g.m_b * rt_row(g) * 8);
            if (pair == 2) { o.ct = x; x += al16(g.n_b * g.dv_max * 8); }
        } else {
            o.rjz = x; x += al16(g.m_b * g.dc_max * 4);
            o.rs = x; x += al16(g.m_b * g.dc_max * 2);
        }
        o.cdeg = x; x += al16(g.n_b * 2);
        if (!pair) {
            o.ceoff = x; x += al16(g.n_b * g.dv_max * 4);
            o.cs = x; x += al16(g.n_b * g.dv_max * 2);
            o.ciz = x; x += al16(g.n_b * g.dv_max * 4);
        }
    } else {
        o.c_ptr = x; x += al16((g.m + 1) * 2);
        o.c_vn = x; x += al16(g.E * 2);
        o.v_ptr = x; x += al16((g.n + 1) * 2);
        if (!pair) { o.v_edge = x; x += al16(g.E * 2); }
    }
    o.total = x;
    return o;
}

struct SGraph {
    const int16_t *rdeg;
    const int32_t *reoff;  // [m_b] first message of a row block (filled-up rows: see load_tables)
    const int32_t *rjz;
    // two-codeword kernels
    const int2 *rt;       // [m_b * rt_row] {4 rjz, 4 rs}
    const int2 *ct;       // [n_b * dv_max] {message offset, words a row | shift << 8} of the t-th block of a column
                          // (variable-node-pass form only)
    const int16_t *rs, *cdeg;
    const int32_t *ceoff;
    const int16_t *cs;
    const int32_t *ciz;
    const uint16_t *c_ptr, *c_vn, *v_ptr, *v_edge;
};

// First message of row block i where rows are filled up (two-codeword kernels,
// check degree > 8): each row takes an odd number of words.
__device__ __forceinline__ int row_offset(const DevCode &g, int i) {
    int x = 0;
    for (int k = 0; k < i; k++) x += g.Z * (g.rdeg[k] | 1);
    return x;
}

__device__ void copy_bytes(void *dst, const void *src, int bytes) {
    // 16-byte vector copies when both ends allow, else bytes
    const int n16 = bytes >> 4;
    const int4 *s4 = (const int4 *)src;
    int4 *d4 = (int4 *)dst;
    if ((((uintptr_t)src) & 15) == 0) {
        for (int i = threadIdx.x; i < n16; i += blockDim.x) d4[i] = __ldg(s4 + i);
        for (int i = (n16 << 4) + threadIdx.x; i < bytes; i += blockDim.x)
            ((unsigned char *)dst)[i] = ((const unsigned char *)src)[i];
    } else {
        for (int i = threadIdx.x; i < bytes; i += blockDim.x)
            ((unsigned char *)dst)[i] = ((const unsigned char *)src)[i];
    }
}

// filled (QC, two-codeword kernels): the row blocks start where rows of an odd number of words put them
__device__ SGraph load_tables(const DevCode &g, unsigned char *sm, int pair = 0, bool filled = false) {
    TabOff o = tab_offsets(g, pair);
    SGraph s{};
    if (pair && g.by_rows) {
        uint16_t *cv = (uint16_t *)(sm + o.c_vn);
        for (int c = threadIdx.x; c < g.m; c += blockDim.x) {
            const int i = c / g.Z, r = c - i * g.Z;
            for (int p = 0; p < 6; p++) cv[c * 6 + p] = (uint16_t)(g.rjz[i * 6 + p] + wrapZ(r + g.rs[i * 6 + p], g.Z));
        }
        s.c_vn = cv;
        return s;
    }
    if (g.kind == TSX_CODE_QC) {
        copy_bytes(sm + o.rdeg, g.rdeg, g.m_b * 2);
        int *reoff = (int *)(sm + o.reoff);
        for (int i = threadIdx.x; i < g.m_b; i += blockDim.x) reoff[i] = filled ? row_offset(g, i) : g.reoff[i];
        if (pair) {
            int2 *rt = (int2 *)(sm + o.rt);
            const int row = rt_row(g);
            for (int x = threadIdx.x; x < g.m_b * g.dc_max; x += blockDim.x) {
                const int i = x / g.dc_max;
                rt[i * row + x - i * g.dc_max] = make_int2(4 * g.rjz[x], 4 * (int)g.rs[x]);
            }
            s.rt = rt;
            if (pair == 2) {
                int2 *ct = (int2 *)(sm + o.ct);
                for (int x = threadIdx.x; x < g.n_b * g.dv_max; x += blockDim.x) {
                    const int j = x / g.dv_max;
                    if (x - j * g.dv_max >= g.cdeg[j]) continue;
                    const int i = g.ciz[x] / g.Z, p = (g.ceoff[x] - g.reoff[i]) / g.Z;
                    ct[x] = filled ? make_int2(row_offset(g, i) + p, (g.rdeg[i] | 1) | ((int)g.cs[x] << 8))
                                   : make_int2(g.ceoff[x], 1 | ((int)g.cs[x] << 8));
                }
                s.ct = ct;
            }
        } else {
            copy_bytes(sm + o.rjz, g.rjz, g.m_b * g.dc_max * 4);
            copy_bytes(sm + o.rs, g.rs, g.m_b * g.dc_max * 2);
            copy_bytes(sm + o.ciz, g.ciz, g.n_b * g.dv_max * 4);
            copy_bytes(sm + o.ceoff, g.ceoff, g.n_b * g.dv_max * 4);
            copy_bytes(sm + o.cs, g.cs, g.n_b * g.dv_max * 2);
            s.ceoff = (const int32_t *)(sm + o.ceoff);
            s.cs = (const int16_t *)(sm + o.cs);
            s.rjz = (const int32_t *)(sm + o.rjz);
            s.rs = (const int16_t *)(sm + o.rs);
            s.ciz = (const int32_t *)(sm + o.ciz);
        }
        copy_bytes(sm + o.cdeg, g.cdeg, g.n_b * 2);
        s.rdeg = (const int16_t *)(sm + o.rdeg);
        s.reoff = reoff;
        s.cdeg = (const int16_t *)(sm + o.cdeg);
    } else {
        copy_bytes(sm + o.c_ptr, g.c_ptr, (g.m + 1) * 2);
        // (the two-codeword kernels do not depend on the order of checks and edges)
        copy_bytes(sm + o.c_vn, pair && g.c_vnb ? g.c_vnb : g.c_vn, g.E * 2);
        copy_bytes(sm + o.v_ptr, g.v_ptr, (g.n + 1) * 2);
        s.c_ptr = (const uint16_t *)(sm + o.c_ptr);
        s.c_vn = (const uint16_t *)(sm + o.c_vn);
        s.v_ptr = (const uint16_t *)(sm + o.v_ptr);
        if (!pair) {
            copy_bytes(sm + o.v_edge, g.v_edge, g.E * 2);
            s.v_edge = (const uint16_t *)(sm + o.v_edge);
        }
    }
    return s;
}

// ---------------------------------------------------------------------------
// a group of G warps working on one codeword
// ---------------------------------------------------------------------------
struct Grp {
    int G, T, gt, lane, gw, bar;
    int *red;  // reduction scratch (shared): G words for sum(), from kMaxGroupWarps on for sum_pass()
    // Both forms are volatile asm statements with a memory clobber: the two-codeword kernels read
    // shared memory by volatile asm without one, and what was written by ordinary stores has to be
    // ordered before such reads (and ordinary stores after them) in the source already; __syncwarp() is
    // not an asm statement and orders ordinary accesses only.
    __device__ __forceinline__ void sync() const {
        if (G == 1) asm volatile("bar.warp.sync 0xffffffff;" ::: "memory");
        else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(T) : "memory");
    }
    // LOOP: the warps' parts added one after the other (see enum_kernel)
    template <bool LOOP = false>
    __device__ __forceinline__ int sum(int x) const {
        x = __reduce_add_sync(0xffffffffu, x);
        if (G == 1) {
            sync();
            return x;
        }
        if (lane == 0) red[gw] = x;
        sync();
        int s = 0;
        if constexpr (LOOP)
            for (int w = 0; w < G; w++) s += red[w];
        else
            s = __reduce_add_sync(0xffffffffu, lane < G ? red[lane] : 0);
        sync();
        return s;
    }
    // the same on the second scratch bank without the closing barrier: the
    // caller passes a group barrier before its next sum_pass
    __device__ __forceinline__ int sum_pass(int x) const {
        x = __reduce_add_sync(0xffffffffu, x);
        if (G == 1) {
            sync();
            return x;
        }
        if (lane == 0) red[kMaxGroupWarps + gw] = x;
        sync();
        return __reduce_add_sync(0xffffffffu, lane < G ? red[kMaxGroupWarps + lane] : 0);
    }
};

// ---------------------------------------------------------------------------
// single-precision tanh / atanh of the sum-product check update, from their
// series with IEEE-rounded adds, multiplies and divides only (no fused
// multiply-add), so the result is the same on every conforming machine:
//   expm1(x), x >= 0: k = rint(x/ln2), r = (x - k ln2_hi) - k ln2_lo
//     (Cody-Waite reduction), expm1(r) = sum_{i=1..9} r^i/i! by Horner,
//     expm1(x) = 2^k (expm1(r) + 1) - 1 if k != 0;
//   tanh(y) = sgn(y) e / (e + 2), e = expm1(2|y|);
//   atanh(p) = sgn(p) sum_{j=0..8} a^(2j+1)/(2j+1) for a = |p| < 1/4, else
//     sgn(p) log(t)/2, t = (1+a)/(1-a) = m 2^e with m in [sqrt(1/2),
//     sqrt(2)), log t = e ln2 + 2 sum_{j=0..6} s^(2j+1)/(2j+1),
//     s = (m-1)/(m+1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float hadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float hsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float hmul(float a, float b) { return __fmul_rn(a, b); }

__device__ __forceinline__ float spa_expm1_pos(float x) {
    const float k = rintf(hmul(x, 0x1.715476p+0f));
    const float r = hsub(hsub(x, hmul(k, 0x1.62e4p-1f)), hmul(k, 0x1.7f7d1cp-20f));
    float p = 0x1.71de3ap-19f;  // 1/9!
    p = hadd(hmul(p, r), 0x1.a01a02p-16f);
    p = hadd(hmul(p, r), 0x1.a01a02p-13f);
    p = hadd(hmul(p, r), 0x1.6c16c2p-10f);
    p = hadd(hmul(p, r), 0x1.111112p-7f);
    p = hadd(hmul(p, r), 0x1.555556p-5f);
    p = hadd(hmul(p, r), 0x1.555556p-3f);
    p = hadd(hmul(p, r), 0.5f);
    p = hadd(hmul(p, r), 1.0f);
    p = hmul(p, r);
    // 2^k in two factors, both normal (k >= 0; from 252 on the result is infinite with any larger k too)
    const int ki = min((int)k, 252), kh = ki >> 1;
    const float f = hmul(hmul(hadd(p, 1.0f), __int_as_float((kh + 127) << 23)), __int_as_float((ki - kh + 127) << 23));
    return k == 0.0f ? p : hsub(f, 1.0f);
}

__device__ __forceinline__ float spa_tanhf(float y) {
    const float a = fabsf(y);
    const float e = spa_expm1_pos(hadd(a, a));
    // e / (e + 2): e / 2 where e + 2 rounds to 2, and 1 where it rounds to e (a NaN for infinite e, as inf / inf)
    float t = div_tanh(e);
    t = e < 0x1p-24f ? hmul(e, 0.5f) : t;
    t = e < 0x1p26f ? t : hadd(hsub(e, e), 1.0f);
    return y < 0.0f ? -t : t;
}

// (both series always and no branch: two edges' chains interleave)
__device__ __forceinline__ float spa_atanhf(float p) {
    const float a = fabsf(p);
    const float a2 = hmul(a, a);
    float q = 0x1.e1e1e2p-5f;  // 1/17
    q = hadd(hmul(q, a2), 0x1.111112p-4f);
    q = hadd(hmul(q, a2), 0x1.3b13b2p-4f);
    q = hadd(hmul(q, a2), 0x1.745d18p-4f);
    q = hadd(hmul(q, a2), 0x1.c71c72p-4f);
    q = hadd(hmul(q, a2), 0x1.24924ap-3f);
    q = hadd(hmul(q, a2), 0x1.99999ap-3f);
    q = hadd(hmul(q, a2), 0x1.555556p-2f);
    q = hadd(hmul(q, a2), 1.0f);
    const float small = hmul(q, a);
    // t = m 2^e with m in [1/2, 1): for a in [1/4, 1), t >= 5/3 is normal and finite
    const float t = div_atanh(a);
    const int tb = __float_as_int(t);
    int e = (tb >> 23) - 126;
    float m = __int_as_float((tb & 0x7FFFFF) | 0x3F000000);
    const bool up = m < 0x1.6a09e6p-1f;
    m = up ? hadd(m, m) : m;
    e = up ? e - 1 : e;
    const float s = div_log(m);
    const float s2 = hmul(s, s);
    float z = 0x1.3b13b2p-4f;  // 1/13
    z = hadd(hmul(z, s2), 0x1.745d18p-4f);
    z = hadd(hmul(z, s2), 0x1.c71c72p-4f);
    z = hadd(hmul(z, s2), 0x1.24924ap-3f);
    z = hadd(hmul(z, s2), 0x1.99999ap-3f);
    z = hadd(hmul(z, s2), 0x1.555556p-2f);
    z = hadd(hmul(z, s2), 1.0f);
    const float lg = hadd(hmul((float)e, 0x1.62e43p-1f), hmul(hadd(s, s), z));
    float r = a < 0.25f ? small : hmul(0.5f, lg);
    r = a < 1.0f ? r : a;  // (a NaN stays one)
    return p < 0.0f ? -r : r;
}

// misc area of a slot
struct Misc {
    int red[64];
    long long bcast[2];
    unsigned long long okd, okit;  // converged decodes of this group and their iterations
};
// the sieve kernel's (one warp a slot)
struct SieveMisc {
    uint16_t seg[kMaxNb + 2], segw[kMaxNb + 2];
};

// ---------------------------------------------------------------------------
// one decode
// ---------------------------------------------------------------------------
template <class Dec, int DCMAX, bool QC, bool LOOP = false>
struct Decoder {
    using msg = typename Dec::msg;
    using post = typename Dec::post;
    using lv = typename Dec::lv;

    const DevCode &g;
    const SGraph &sg;
    const Grp &gp;
    const DecodeParams &dp;
    post *P;
    msg *R;

    // check pass: returns (group total) unsatisfied checks of x = [P < 0];
    // if writeR, also replaces R by the next check-to-variable messages.
    __device__ __forceinline__ int check_pass(bool first, bool writeR) const {
        int unsat = 0;
        const int Z = g.Z;
        if (QC) {
            int i = gp.gt / Z, r = gp.gt - i * Z;
            for (int c = gp.gt; c < g.m; c += gp.T) {
                const int deg = sg.rdeg[i];
                const int e0 = sg.reoff[i] + r;
                const int32_t *rjz = sg.rjz + i * g.dc_max;
                const int16_t *rs = sg.rs + i * g.dc_max;
                unsat += check_node(first, writeR, deg, e0, Z, [&](int p) {
                    return rjz[p] + wrapZ(r + rs[p], Z);
                });
                r += gp.T;
                while (r >= Z) { r -= Z; i++; }
            }
        } else {
            for (int c = gp.gt; c < g.m; c += gp.T) {
                const int e0 = sg.c_ptr[c];
                const int deg = sg.c_ptr[c + 1] - e0;
                // message (c, p) lives at p*m + c (consecutive lanes, consecutive words)
                unsat += check_node(first, writeR, deg, c, g.m, [&](int p) { return (int)sg.c_vn[e0 + p]; });
            }
        }
        return gp.template sum<LOOP>(unsat);
    }

    template <class NB>
    __device__ __forceinline__ int check_node(bool first, bool writeR, int deg, int e0, int estride,
                                              NB nb) const {
        if constexpr (!Dec::kFloat) {
            const int sat = dp.sat;
            int m1 = sat, m2 = sat, sgn = 0, par = 0;
            int a[DCMAX];
#pragma unroll
            for (int p = 0; p < DCMAX; p++) {
                if (p < deg) {
                    const int v = nb(p);
                    const int Pv = (int)P[v];
                    const int ro = first ? 0 : (int)R[e0 + p * estride];
                    par ^= Pv;
                    const int q = clampi(Pv - ro, -sat, sat);
                    sgn |= (int)((unsigned)q >> 31) << p;
                    const int aa = abs(q);
                    a[p] = aa;
                    m2 = min(m2, max(m1, aa));
                    m1 = min(m1, aa);
                }
            }
            if (writeR) {
                const int o1 = (dp.alpha_num * m1) >> dp.alpha_shift;
                const int o2 = (dp.alpha_num * m2) >> dp.alpha_shift;
                const int tot = __popc(sgn) & 1;
#pragma unroll
                for (int p = 0; p < DCMAX; p++) {
                    if (p < deg) {
                        const int mag = a[p] == m1 ? o2 : o1;
                        const int neg = tot ^ ((sgn >> p) & 1);
                        R[e0 + p * estride] = (msg)(neg ? -mag : mag);
                    }
                }
            }
            return par < 0;
        } else {
            // Rolled loops, each edge's tanh in its message's place until the outputs take it: the
            // series are in the code once each (unrolled over the edges, with the tanhs in
            // registers, the loop missed the instruction cache).  The products over the other
            // edges are taken in ascending order: the edges before p as a running product,
            // the ones after it one by one.
            const float clip = dp.spa_clip;
            int par = 0;
#pragma unroll 2
            for (int p = 0; p < deg; p++) {
                const float Pv = (float)P[nb(p)];
                const float ro = first ? 0.0f : (float)R[e0 + p * estride];
                par ^= Pv < 0.0f;
                if (writeR) R[e0 + p * estride] = (msg)spa_tanhf(__fmul_rn(clampf_(__fsub_rn(Pv, ro), -clip, clip), 0.5f));
            }
            if (writeR) {
                auto out = [&](float prod) {
                    float rr = __fmul_rn(2.0f, spa_atanhf(prod));
                    rr = fabsf(prod) >= 1.0f ? (prod > 0.0f ? clip : -clip) : rr;
                    return clampf_(rr, -clip, clip);
                };
                float pre = 1.0f;
                int p = 0;
#pragma unroll 1
                for (; p + 1 < deg; p += 2) {  // two edges at a time: the same later edges follow in both products
                    const float t0 = (float)R[e0 + p * estride], t1 = (float)R[e0 + (p + 1) * estride];
                    float A = __fmul_rn(pre, t1), B = __fmul_rn(pre, t0);
                    pre = __fmul_rn(B, t1);
#pragma unroll 4
                    for (int p2 = p + 2; p2 < deg; p2++) {
                        const float t = (float)R[e0 + p2 * estride];
                        A = __fmul_rn(A, t);
                        B = __fmul_rn(B, t);
                    }
                    R[e0 + p * estride] = (msg)out(A);
                    R[e0 + (p + 1) * estride] = (msg)out(B);
                }
                if (p < deg) R[e0 + p * estride] = (msg)out(pre);
            }
            return par;
        }
    }

    // posterior of variable node v with channel value L
    __device__ __forceinline__ lv posterior(int v, lv L) const {
        lv acc = L;
        if (QC) {
            const int j = v / g.Z, k = v - j * g.Z;
            const int deg = sg.cdeg[j];
#pragma unroll 4
            for (int t = 0; t < deg; t++) {
                const int idx = j * g.dv_max + t;
                acc = acc + (lv)R[sg.ceoff[idx] + wrapZneg(k - sg.cs[idx], g.Z)];
            }
        } else {
            const int t0 = sg.v_ptr[v], t1 = sg.v_ptr[v + 1];
            for (int t = t0; t < t1; t++) acc = acc + (lv)R[sg.v_edge[t]];
        }
        return acc;
    }

    __device__ __forceinline__ void vn_pass(lv Lbase) const {
        if (QC) {
            const int Z = g.Z;
            int j = gp.gt / Z, k = gp.gt - j * Z;
            for (int v = gp.gt; v < g.n; v += gp.T) {
                const int deg = sg.cdeg[j];
                lv acc = Lbase;
#pragma unroll 4
                for (int t = 0; t < deg; t++) {
                    const int idx = j * g.dv_max + t;
                    acc = acc + (lv)R[sg.ceoff[idx] + wrapZneg(k - sg.cs[idx], Z)];
                }
                P[v] = (post)acc;
                k += gp.T;
                while (k >= Z) { k -= Z; j++; }
            }
        } else {
            for (int v = gp.gt; v < g.n; v += gp.T) {
                const int t0 = sg.v_ptr[v], t1 = sg.v_ptr[v + 1];
                lv acc = Lbase;
                for (int t = t0; t < t1; t++) acc = acc + (lv)R[sg.v_edge[t]];
                P[v] = (post)acc;
            }
        }
    }

    __device__ __forceinline__ void save_x(uint32_t *xw) const {
        for (int base = 0; base < g.n; base += gp.T) {
            const int v = base + gp.gt;
            const bool bit = v < g.n && P[v] < (post)0;
            const unsigned w = __ballot_sync(0xffffffffu, bit);
            const int wi = (base >> 5) + gp.gw;
            if (gp.lane == 0 && (wi << 5) < g.n) xw[wi] = w;
        }
    }

    // Returns true if the decode failed (x_{K_last} != 0); xbest receives x*.
    // K: the iteration limit of this candidate.
    __device__ bool run(const int *I, int nI, lv Lbase, lv Limp, uint32_t *xbest, int &kl, int K) const {
        if (!(Limp < (lv)0)) {  // x_0 = 0: u_0 = 0, success at iteration 0
            kl = 0;
            return false;
        }
        for (int v = gp.gt; v < g.n; v += gp.T) P[v] = (post)Lbase;
        gp.sync();
        if (gp.gt < nI) P[I[gp.gt]] = (post)Limp;
        gp.sync();
        int ubest = 0x7fffffff, u = 0, k = 0;
        bool first = true;
        while (true) {
            u = check_pass(first, k < K);  // u = u_k; R <- R_{k+1}
            first = false;
            if (k >= g.wstart && u < ubest) {
                ubest = u;
                save_x(xbest);
            }
            if (u == 0 || k == K) break;
            vn_pass(Lbase);  // P <- P_{k+1}
            gp.sync();
            if (gp.gt < nI) P[I[gp.gt]] = (post)posterior(I[gp.gt], Limp);
            gp.sync();
            k++;
        }
        kl = k;
        if (k < g.wstart) save_x(xbest);
        int neg = 0;
        if (u == 0)
            for (int v = gp.gt; v < g.n; v += gp.T) neg |= P[v] < (post)0;
        const int any = gp.sum(neg);
        return u != 0 || any != 0;
    }
};

// Iteration limit of candidate idx: K, or its cycle-density budget.
__device__ __forceinline__ int cand_limit(const DecodeParams &dp, const EnumBuffers &b, long long idx) {
    return b.cand_K ? (int)b.cand_K[idx] : dp.K;
}

// ---------------------------------------------------------------------------
// sieving: Tree(), TS(), (a,b)
// ---------------------------------------------------------------------------
// Sets of variable nodes are bitmasks; a warp takes a word of 32 nodes at a
// time and passes over empty words, so the work follows the set's size and not
// the code's: the degrees |N(c) n S| are counted from the set's nodes (shared
// atomics) and not from the checks' rows, and a node's column block comes from
// a multiplication.  (Row by row, with a division by Z per neighbour, three
// counts of every check made the ordered list's second stage
// several times a decoding iteration per pattern.)
template <bool QC>
struct Sieve {
    const DevCode &g;
    const SGraph &sg;
    const Grp &gp;

    // f(check) for every check of v
    template <class F>
    __device__ __forceinline__ void each_check(int v, F f) const {
        if (QC) {
            const int Z = g.Z;
            const int j = Z > 1 ? (int)__umulhi((unsigned)v, 0xFFFFFFFFu / (unsigned)Z + 1u) : v;  // v / Z, v < 2^15
            const int k = v - j * Z, d = sg.cdeg[j], i0 = j * g.dv_max;
            for (int t = 0; t < d; t++) f(sg.ciz[i0 + t] + wrapZneg(k - sg.cs[i0 + t], Z));
        } else {
            const int t1 = sg.v_ptr[v + 1];
            for (int t = sg.v_ptr[v]; t < t1; t++) f((int)g.v_chk[t]);
        }
    }
    // f(v, word index, whether v is in S) for the group's words of S, every lane of a warp together;
    // empty words only with ALL
    template <bool ALL, class F>
    __device__ __forceinline__ void each_word(const uint32_t *S, F f) const {
        const int nw = (g.n + 31) >> 5;
        for (int wi = gp.gw; wi < nw; wi += gp.G) {
            const uint32_t x = S[wi];
            if (!ALL && x == 0) continue;
            f((wi << 5) + gp.lane, wi, (x >> gp.lane) & 1u);
        }
    }

    // deg[c] += 1 for the checks of S's nodes
    __device__ void add_deg(const uint32_t *S, int *deg) const {
        each_word<false>(S, [&](int v, int, bool in) {
            if (in) each_check(v, [&](int c) { atomicAdd(&deg[c], 1); });
        });
    }

    // Tree(S): delete variable nodes with fewer than two checks of degree >= 2
    // until none is left (the 2-core of the induced bipartite graph).
    __device__ void peel(uint32_t *S, int *deg) const {
        while (true) {
            int changed = 0;
            each_word<false>(S, [&](int v, int wi, bool in) {
                bool rm = false;
                if (in) {
                    int live = 0;
                    each_check(v, [&](int c) { live += deg[c] >= 2; });
                    rm = live < 2;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, rm);
                if (mask == 0) return;
                if (gp.lane == 0) S[wi] &= ~mask;
                if (rm) each_check(v, [&](int c) { atomicSub(&deg[c], 1); });
                changed = 1;
            });
            __syncwarp();
            if (!gp.sum(changed)) break;  // (a barrier after the warps' changes, and one after all have read)
        }
    }

    // S <- S u {v not in S : at least two checks of v touch S} (deg = |N(c) n S|); afterwards deg
    // counts the larger set
    __device__ void closure(uint32_t *S, uint32_t *added, int *deg) const {
        each_word<true>(S, [&](int v, int wi, bool in) {
            bool add = false;
            if (v < g.n && !in) {
                int k = 0;
                each_check(v, [&](int c) { k += deg[c] >= 1; });
                add = k >= 2;
            }
            const unsigned mask = __ballot_sync(0xffffffffu, add);
            if (gp.lane == 0) added[wi] = mask;
        });
        gp.sync();  // every count read before any changes
        add_deg(added, deg);
        const int nw = (g.n + 31) >> 5;
        for (int wi = gp.gw; wi < nw; wi += gp.G)
            if (gp.lane == 0) S[wi] |= added[wi];
        gp.sync();
    }

    __device__ int popcount(const uint32_t *S) const {
        const int nw = (g.n + 31) >> 5;
        int c = 0;
        for (int w = gp.gt; w < nw; w += gp.T) c += __popc(S[w]);
        return gp.sum(c);
    }

    // X = xk u I into S, and deg for it
    __device__ void load_x(uint32_t *S, const uint32_t *xk, const int *I, int nI, int *deg) const {
        const int nw = (g.n + 31) >> 5;
        for (int w = gp.gt; w < nw; w += gp.T) {
            uint32_t x = xk[w];
#pragma unroll
            for (int t = 0; t < 4; t++)
                if (t < nI && (I[t] >> 5) == w) x |= 1u << (I[t] & 31);
            S[w] = x;
        }
        for (int c = gp.gt; c < g.m; c += gp.T) deg[c] = 0;
        gp.sync();
        add_deg(S, deg);
        gp.sync();
    }

    // Returns the sieve used (1: S1 = Tree(X), 2: S2 = Tree(TS(X)), 0: both
    // empty); S holds T and deg[c] = |N(c) n T| on return.
    __device__ int run(uint32_t *S, uint32_t *added, const uint32_t *xk, const int *I, int nI, int *deg,
                       int &a) const {
        load_x(S, xk, I, nI, deg);
        peel(S, deg);
        a = popcount(S);
        if (a > 0) return 1;
        load_x(S, xk, I, nI, deg);
        closure(S, added, deg);
        peel(S, deg);
        a = popcount(S);
        return a > 0 ? 2 : 0;
    }

    // b = checks of odd degree in T, elementary = every check degree <= 2
    __device__ void classify(const int *deg, int &b, int &elem) const {
        // odd degrees in bits 0-19 (m < 2^16), and one flag a thread with degrees above 2 at bit 20: a group of
        // T threads sums to less than T 2^20 + 2^16
        int x = 0;
        for (int c = gp.gt; c < g.m; c += gp.T) {
            const int d = deg[c];
            x += d & 1;
            if (d > 2) x |= 1 << 20;
        }
        x = gp.sum(x);
        b = x & 0xFFFFF;
        elem = (x >> 20) == 0;
    }
};

// ---------------------------------------------------------------------------
// canonical key, orbit, hash and insert (warp 0 of the group)
// ---------------------------------------------------------------------------
// Ordered list of the set bits of S (warp 0), returns count.
__device__ int list_bits(const uint32_t *S, int n, uint16_t *list, int lane) {
    const int nw = (n + 31) >> 5;
    int pos = 0;
    for (int base = 0; base < nw; base += 32) {
        const int w = base + lane;
        uint32_t x = w < nw ? S[w] : 0u;
        const int c = __popc(x);
        int incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        int off = pos + incl - c;
        while (x) {
            const int b = __ffs(x) - 1;
            x &= x - 1;
            list[off++] = (uint16_t)(w * 32 + b);
        }
        pos += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    return pos;
}

// Canonical key (QC: smallest sorted tuple over the shifts moving a member
// to k = 0; CSR: the sorted set) into key[], returns the orbit size.
//
// The tuple is smallest where its first element is: only a shift that moves a
// member of the first column block to k = 0 makes that 0, so the candidates
// are that block's members.  Under the shift of its member i the block's
// members are i, i + 1, ... in order, and every further block starts at the
// first member past the wrap, found by bisection.  (Every member a candidate,
// and the wrap found by a scan for each member written, cost a set of a nodes
// a^2 / 10 steps of one warp: the ordered list's sets reach a = 2,500.)
__device__ int canon_key(const DevCode &g, const uint16_t *L, int a, const uint32_t *S, uint16_t *key,
                         uint16_t *segs, uint16_t *segw, int lane) {
    if (g.kind != TSX_CODE_QC) {
        for (int i = lane; i < a; i += 32) key[i] = L[i];
        __syncwarp();
        return 1;
    }
    const int Z = g.Z;
    const unsigned zm = Z > 1 ? 0xFFFFFFFFu / (unsigned)Z + 1u : 0u;
    auto block = [&](int v) { return Z > 1 ? (int)__umulhi((unsigned)v, zm) : v; };  // v / Z, v < 2^15
    // segments of equal column block
    int nseg = 0;
    for (int base = 0; base < a; base += 32) {
        const int i = base + lane;
        const bool mk = i < a && (i == 0 || block(L[i]) != block(L[i - 1]));
        const unsigned mask = __ballot_sync(0xffffffffu, mk);
        if (mk) segs[nseg + __popc(mask & ((1u << lane) - 1))] = (uint16_t)i;
        nseg += __popc(mask);
    }
    if (lane == 0) segs[nseg] = (uint16_t)a;
    __syncwarp();
    const int c0 = segs[1];
    const int k0 = (int)L[0] - block(L[0]) * Z;
    // stabilizer: shifts sigma = k(L[i]) - k(L[0]) of segment-0 members with T + sigma = T
    int stab = 0;
    for (int base = 0; base < c0; base += 32) {
        const int i = base + lane;
        bool ok = i < c0;
        if (ok) {
            const int sig = (int)L[i] - (int)L[0];  // >= 0: same block, ascending
            for (int x = 0; x < a && ok; x++) {
                const int v = L[x];
                const int jz = block(v) * Z;
                int k = v - jz + sig;
                if (k >= Z) k -= Z;
                const int u = jz + k;
                ok = (S[u >> 5] >> (u & 31)) & 1u;
            }
        }
        stab += __popc(__ballot_sync(0xffffffffu, ok));
    }
    // first member of segment sg at or past k = lim
    auto past = [&](int sg, int lim) {
        int lo = segs[sg], hi = segs[sg + 1];
        const int v = block(L[lo]) * Z + lim;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((int)L[mid] >= v) hi = mid;
            else lo = mid + 1;
        }
        return lo;
    };
    // tournament over segment 0's members, 31 against the best so far
    int best = 0;
    for (int base = 1; base < c0; base += 31) {
        const int i = lane == 0 ? best : base + lane - 1;
        bool active = lane == 0 || i < c0;
        const int ki = active ? (int)L[i] : 0;
        bool more = true;
        for (int t = 1, x = i; t < c0 && more; t++) {  // the gaps decide: member i + t less member i, modulo Z
            if (++x >= c0) x -= c0;
            int e = 0x7fffffff;
            if (active) {
                e = (int)L[x] - ki;
                if (e < 0) e += Z;
            }
            const int mn = __reduce_min_sync(0xffffffffu, e);
            active = active && e == mn;
            more = __popc(__ballot_sync(0xffffffffu, active)) > 1;
        }
        const int s = active ? (Z - (ki - (int)L[0] + k0)) : 0;  // shift, 1 .. Z
        for (int sg = 1; sg < nseg && more; sg++) {
            const int st = segs[sg], c = segs[sg + 1] - st;
            const int jz = block(L[st]) * Z;
            int x = active ? past(sg, Z - s) : st;
            for (int t = 0; t < c && more; t++, x++) {
                if (x >= st + c) x -= c;
                int e = 0x7fffffff;
                if (active) {
                    e = (int)L[x] - jz + s;
                    if (e >= Z) e -= Z;
                }
                const int mn = __reduce_min_sync(0xffffffffu, e);
                active = active && e == mn;
                more = __popc(__ballot_sync(0xffffffffu, active)) > 1;
            }
        }
        const unsigned am = __ballot_sync(0xffffffffu, active);
        best = __shfl_sync(0xffffffffu, i, __ffs(am) - 1);
    }
    // the key under best's shift
    const int s = Z - ((int)L[best] - (int)L[0] + k0);  // 1 .. Z
    for (int sg = lane; sg < nseg; sg += 32) segw[sg] = (uint16_t)past(sg, Z - s);
    __syncwarp();
    int sg = 0;
    for (int pos = lane; pos < a; pos += 32) {
        while (segs[sg + 1] <= pos) sg++;
        const int st = segs[sg], en = segs[sg + 1];
        int x = segw[sg] + (pos - st);
        if (x >= en) x -= en - st;
        const int jz = block(L[x]) * Z;
        int k = (int)L[x] - jz + s;
        if (k >= Z) k -= Z;
        key[pos] = (uint16_t)(jz + k);
    }
    __syncwarp();
    return Z / stab;
}

__device__ unsigned long long key_hash(const uint16_t *key, int a, int lane) {
    unsigned long long h = 0;
    for (int i = lane; i < a; i += 32) h += mix64(((unsigned long long)i << 32) | key[i]);
    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    return h + mix64(0xabcdef0000000000ull + (unsigned long long)a);
}

// Space reserved at pool offset off for a key of a nodes that another
// insert of the same key made unnecessary: taken back if nothing was
// reserved after it, else counted as leaked.
__device__ __forceinline__ void pool_giveback(const EnumBuffers &b, long long off, int a) {
    const unsigned long long len = (unsigned long long)(kPoolHdr + a);
    const unsigned long long top = (unsigned long long)(off - 1);  // pool_top before the reservation
    if (atomicCAS(&b.ctr->pool_top, top + len, top) != top + len) atomicAdd(&b.ctr->pool_leaked, len);
}

// Insert / find the key; returns the table slot, -1 on a full table, -2 on
// a pool overflow.  Warp-collective.  The header's flags word ends as the OR
// of the flags of every insert of the key (independent of their order).
__device__ long long ts_insert(const EnumBuffers &b, const uint16_t *key, int a, int bb, int orbit,
                               int flags, int lane) {
    const unsigned long long h = key_hash(key, a, lane);
    const unsigned long long hhi = (h >> 32) << 32;
    unsigned long long slot = h & b.cap_mask;
    long long my_off = -1;
    for (unsigned long long probe = 0; probe <= b.cap_mask; probe++) {
        unsigned long long tag = 0;
        if (lane == 0) tag = *((volatile unsigned long long *)&b.tags[slot]);
        tag = __shfl_sync(0xffffffffu, tag, 0);
        if (tag == 0) {
            if (my_off < 0) {
                long long off = 0;
                // word 0 of the pool is never used, so a tag is never 0
                if (lane == 0) off = 1 + (long long)atomicAdd(&b.ctr->pool_top, (unsigned long long)(kPoolHdr + a));
                off = __shfl_sync(0xffffffffu, off, 0);
                if ((unsigned long long)(off + kPoolHdr + a) > b.pool_cap + 1) {
                    if (lane == 0) atomicOr(&b.ctr->err, kErrPoolOverflow);
                    return -2;
                }
                if (lane == 0) {
                    b.pool[off] = a;
                    b.pool[off + 1] = bb;
                    b.pool[off + 2] = orbit;
                    b.pool[off + 3] = flags;
                }
                for (int i = lane; i < a; i += 32) b.pool[off + kPoolHdr + i] = key[i];
                __threadfence();
                __syncwarp();
                my_off = off;
            }
            unsigned long long old = 0;
            if (lane == 0) old = atomicCAS(&b.tags[slot], 0ull, hhi | (unsigned long long)my_off);
            old = __shfl_sync(0xffffffffu, old, 0);
            if (old == 0) return (long long)slot;
            tag = old;
        }
        if ((tag & 0xffffffff00000000ull) == hhi) {
            __threadfence();
            const long long off = (long long)(tag & 0xffffffffull);
            bool eq = __ldcg(&b.pool[off]) == a;
            if (eq)
                for (int i = lane; i < a && eq; i += 32) eq = __ldcg(&b.pool[off + kPoolHdr + i]) == (int)key[i];
            if (__all_sync(0xffffffffu, eq)) {
                // the sieve bits of a set are the union over every candidate that reached it
                if (lane == 0) {
                    atomicOr(&b.pool[off + 3], flags);
                    if (my_off >= 0) pool_giveback(b, my_off, a);
                }
                return (long long)slot;
            }
        }
        slot = (slot + 1) & b.cap_mask;
    }
    if (lane == 0) {
        atomicOr(&b.ctr->err, kErrTableFull);
        if (my_off >= 0) pool_giveback(b, my_off, a);
    }
    return -1;
}

// ---------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------
template <class Dec, int DCMAX, bool QC, bool LOOP>
__device__ __forceinline__ void scalar_run(const DevCode &g, const DecodeParams &dp, const EnumBuffers &b,
                                           const SlotLayout &lay, int G, const SGraph &sg, unsigned char *smem,
                                           int grp) {
    using lv = typename Dec::lv;
    using post = typename Dec::post;
    using msg = typename Dec::msg;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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
    post *P = (post *)(slot + lay.p_off);
    msg *R = (msg *)(slot + lay.r_off);
    uint32_t *xa = (uint32_t *)(slot + lay.xa_off);
    uint32_t *xb = (uint32_t *)(slot + lay.xb_off);

    Decoder<Dec, DCMAX, QC, LOOP> dec{g, sg, gp, dp, P, R};

    const long long total = (long long)b.ctr->n_cand_total;
    const long long end = b.cand_end < 0 || b.cand_end > total ? total : b.cand_end;
    long long my_dec = 0, my_it = 0, my_eu = 0, my_ok = 0, my_okit = 0;

    lv Lbase;
    if constexpr (Dec::kFloat) Lbase = (lv)clampf_((float)dp.base_llr / 8.0f, -dp.spa_clip, dp.spa_clip);
    else Lbase = (lv)clampi(dp.base_llr, -dp.sat, dp.sat);

    while (true) {
        if (gp.gt == 0) misc->bcast[0] = (long long)atomicAdd(b.queue, 1ull);
        gp.sync();
        const long long idx = b.cand_begin + misc->bcast[0];
        gp.sync();
        if (idx >= end) break;
        const int4 I4 = b.cands[idx];
        int I[4] = {I4.x, I4.y, I4.z, I4.w};
        const int nI = (I4.x >= 0) + (I4.y >= 0) + (I4.z >= 0) + (I4.w >= 0);

        uint32_t *xcur = xa, *xkeep = xb;
        int ndec = 0, nit = 0, kl = 0;
        bool failed = false;
        int thr = -1;
        float thr_f = -1.0f;
        const int Kc = cand_limit(dp, b, idx);
        if constexpr (!Dec::kFloat) {
            int lo = 0, hi = (1 << dp.amp_steps) - 1;
            bool f = dec.run(I, nI, Lbase, (lv)clampi(dp.base_llr - hi, -dp.sat, dp.sat), xcur, kl, Kc);
            ndec++;
            nit += kl;
            if (!f) { my_ok++; my_okit += kl; }
            if (f) {
                failed = true;
                uint32_t *t = xcur; xcur = xkeep; xkeep = t;
                for (int st = 0; st < dp.amp_steps && hi - lo > 1; st++) {
                    const int mid = (lo + hi) >> 1;
                    f = dec.run(I, nI, Lbase, (lv)clampi(dp.base_llr - mid, -dp.sat, dp.sat), xcur, kl, Kc);
                    ndec++;
                    nit += kl;
                    if (!f) { my_ok++; my_okit += kl; }
                    if (f) {
                        hi = mid;
                        uint32_t *t2 = xcur; xcur = xkeep; xkeep = t2;
                    } else {
                        lo = mid;
                    }
                }
                thr = hi;
            }
        } else {
            float lo = 0.0f, hi = 1.0f;
            const float basef = (float)dp.base_llr / 8.0f;
            auto limp = [&](float eps) {
                return (lv)clampf_(__fsub_rn(basef, __fmul_rn(eps, dp.spa_amax)), -dp.spa_clip, dp.spa_clip);
            };
            bool f = dec.run(I, nI, Lbase, limp(hi), xcur, kl, Kc);
            ndec++;
            nit += kl;
            if (!f) { my_ok++; my_okit += kl; }
            if (f) {
                failed = true;
                uint32_t *t = xcur; xcur = xkeep; xkeep = t;
                for (int st = 0; st < dp.amp_steps; st++) {
                    const float mid = __fmul_rn(0.5f, __fadd_rn(lo, hi));
                    f = dec.run(I, nI, Lbase, limp(mid), xcur, kl, Kc);
                    ndec++;
                    nit += kl;
                    if (!f) { my_ok++; my_okit += kl; }
                    if (f) {
                        hi = mid;
                        uint32_t *t2 = xcur; xcur = xkeep; xkeep = t2;
                    } else {
                        lo = mid;
                    }
                }
                thr_f = hi;
            }
        }
        my_dec += ndec;
        my_it += nit;
        my_eu += (long long)nit * g.E;

        // records and the failing decode's x* for the sieve kernel
        gp.sync();
        const long long o = idx - b.rec_base;
        if (failed) {
            uint32_t *dst = b.xstar + o * (long long)b.nw;
            for (int w = gp.gt; w < b.nw; w += gp.T) dst[w] = xkeep[w];
        }
        if (gp.gt == 0) {
            b.c_thr[o] = thr;
            b.c_thr_f[o] = thr_f;
            b.c_slot[o] = -1;
            b.c_flags[o] = 0;
            b.c_decodes[o] = ndec;
            b.c_iters[o] = nit;
        }
        gp.sync();
    }
    if (gp.gt == 0) {
        atomicAdd(&b.ctr->decodes, (unsigned long long)my_dec);
        atomicAdd(&b.ctr->iterations, (unsigned long long)my_it);
        atomicAdd(&b.ctr->edge_updates, (unsigned long long)my_eu);
        atomicAdd(&b.ctr->ok_decodes, (unsigned long long)my_ok);
        atomicAdd(&b.ctr->ok_iters, (unsigned long long)my_okit);
    }
}

// WARPS: launch bound.  Min-sum codes here are the ones the two-codeword
// kernels do not take; the sum-product decoder (check degree <= 8) is bound by
// issue and the latency of its series and divisions, one chain per check and
// warp, so warps in flight count more than registers: on a general (1008, 504)
// code, 5,000 candidates, 12 groups of two warps (24 warps, 80 registers) take 56 ms,
// 13 of one (16 or 20 warps) 96, 28 warps 57 (with divisions by branch; 43 without); small codes fill 32 one-warp
// groups (n = 306: 17.9 ms; 24 warps 22).  Before: 113 and 25.7.
// LOOP: the form for groups of one warp of the min-sum QC codes of check degree above 8.  The check pass unrolled
// over 32 edges fills the registers (about 200 bytes spilled), and the sum over warps by one reduction, which such
// groups do not even reach, changes what is spilled: 4 x 18 blocks, Z = 128, 8,000 candidates, 95 ms, with the
// loop 89; wider groups take the reduction (Z = 300, degree 30: 29.4 against 30.5).
template <class Dec, int DCMAX, bool QC, int WARPS = 16, bool LOOP = false>
__global__ void __launch_bounds__(32 * WARPS, 1) enum_kernel(DevCode g, DecodeParams dp, EnumBuffers b,
                                                    SlotLayout lay, int G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SGraph sg = load_tables(g, smem);
    __syncthreads();
    scalar_run<Dec, DCMAX, QC, LOOP>(g, dp, b, lay, G, sg, smem, (threadIdx.x >> 5) / G);
}

// ---------------------------------------------------------------------------
// the sieve kernel: one warp per failing candidate
// ---------------------------------------------------------------------------
template <bool QC>
__global__ void __launch_bounds__(512, 2) sieve_kernel(DevCode g, EnumBuffers b, SlotLayout lay, int is_float) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SGraph sg = load_tables(g, smem);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *slot = smem + lay.tables_bytes + warp * lay.slot_bytes;
    SieveMisc *misc = (SieveMisc *)(slot + lay.misc_off);
    Grp gp;
    gp.G = 1;
    gp.T = 32;
    gp.gw = 0;
    gp.gt = lane;
    gp.lane = lane;
    gp.bar = 1;
    gp.red = nullptr;  // (one warp reduces in registers)
    int *deg = (int *)(slot + lay.r_off);
    uint16_t *key = (uint16_t *)(slot + lay.r_off);
    uint16_t *L = (uint16_t *)(slot + lay.p_off);
    uint32_t *S = (uint32_t *)(slot + lay.xa_off);
    uint32_t *added = (uint32_t *)L;  // (what a closure adds: done with before the member list is written)
    Sieve<QC> sv{g, sg, gp};

    const long long total = (long long)b.ctr->n_cand_total;
    const long long end = b.cand_end < 0 || b.cand_end > total ? total : b.cand_end;
    const long long n = end - b.cand_begin;
    long long my_acyc = 0;
    while (true) {
        long long o = 0;
        if (lane == 0) o = (long long)atomicAdd(&b.ctr->next_sieve, 1ull);
        o = __shfl_sync(0xffffffffu, o, 0);
        if (o >= n) break;
        const bool failed = is_float ? b.c_thr_f[o] >= 0.0f : b.c_thr[o] >= 0;
        if (!failed) continue;
        const int4 I4 = b.cands[b.cand_begin + o];
        int I[4] = {I4.x, I4.y, I4.z, I4.w};
        const int nI = (I4.x >= 0) + (I4.y >= 0) + (I4.z >= 0) + (I4.w >= 0);
        const uint32_t *xk = b.xstar + o * (long long)b.nw;
        int a = 0;
        const int which = sv.run(S, added, xk, I, nI, deg, a);
        int flags = which;
        long long tslot = -1;
        if (which == 0) {
            flags |= kFlagAcyclic;
            my_acyc++;
        } else {
            int bb, elem;
            sv.classify(deg, bb, elem);
            __syncwarp();
            list_bits(S, g.n, L, lane);
            const int orbit = canon_key(g, L, a, S, key, misc->seg, misc->segw, lane);
            const int thr_ord = is_float ? f2ord(b.c_thr_f[o]) : b.c_thr[o];
            tslot = ts_insert(b, key, a, bb, orbit, elem | (which << 1), lane);
            if (tslot >= 0 && lane == 0) {
                atomicMin(&b.t_thr[tslot], thr_ord);
                atomicAdd(&b.t_count[tslot], 1);
            }
            if (tslot == -2) flags |= kFlagOverflow;
        }
        if (lane == 0) {
            b.c_slot[o] = (int)(tslot >= 0 ? tslot : -1);
            b.c_flags[o] = flags;
        }
        __syncwarp();
    }
    if (lane == 0 && my_acyc) atomicAdd(&b.ctr->acyclic, (unsigned long long)my_acyc);
}


// launches one instantiation of a persistent kernel with every CTA resident
template <class K, class... Args>
cudaError_t launch_persistent(K k, const LaunchShape &sh, cudaStream_t st, Args... args) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sh.smem_bytes);
    if (e != cudaSuccess) return e;
    const int threads = sh.groups * sh.G * 32;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, sh.smem_bytes);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    if (sh.per_sm_req > 0 && sh.per_sm_req < occ) occ = sh.per_sm_req;
    k<<<occ * sh.num_sms, threads, sh.smem_bytes, st>>>(args...);
    return cudaGetLastError();
}

// the scalar kernel (one codeword per group)
template <class Dec>
cudaError_t launch_scalar(const DevCode &g, const DecodeParams &dp, const EnumBuffers &b, const LaunchShape &sh,
                          cudaStream_t st) {
    const bool qc = g.kind == TSX_CODE_QC;
    if constexpr (Dec::kFloat) {
        if (g.dc_max <= 8 && sh.G * sh.groups > 24)
            return qc ? launch_persistent(enum_kernel<Dec, 8, true, 32>, sh, st, g, dp, b, sh.lay, sh.G)
                      : launch_persistent(enum_kernel<Dec, 8, false, 32>, sh, st, g, dp, b, sh.lay, sh.G);
    }
    if (g.dc_max <= 8)
        return qc ? launch_persistent(enum_kernel<Dec, 8, true, scalar_warps(Dec::kFloat, 8)>, sh, st, g, dp, b, sh.lay, sh.G)
                  : launch_persistent(enum_kernel<Dec, 8, false, scalar_warps(Dec::kFloat, 8)>, sh, st, g, dp, b, sh.lay, sh.G);
    if constexpr (!Dec::kFloat) {
        if (qc && sh.G == 1)
            return launch_persistent(enum_kernel<Dec, 32, true, 16, true>, sh, st, g, dp, b, sh.lay, sh.G);
    }
    return qc ? launch_persistent(enum_kernel<Dec, 32, true>, sh, st, g, dp, b, sh.lay, sh.G)
              : launch_persistent(enum_kernel<Dec, 32, false>, sh, st, g, dp, b, sh.lay, sh.G);
}

}  // namespace
}  // namespace tsx
