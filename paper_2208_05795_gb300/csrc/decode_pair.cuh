// decode_pair.cuh -- the fixed-point min-sum impulse decoder, two codewords
// per lane.
//
// A group of G warps owns a pair of codeword slots ("halves" 0 and 1) and
// runs two independent candidates at once: every shared-memory word holds
// the same message or posterior of both codewords, one per 16-bit half, and
// the two halves follow their own bisection and decode schedules (a half
// whose decode ends starts its next decode at once; the other keeps going).
//
// Representation (one 32-bit add or subtract updates both halves, and signs
// and equalities are single bits):
//   message   R' = (r1 << 16) + r0 as one 32-bit number (the low half's borrow is in the high
//             half), or r + 128 in two bytes (8-bit storage, bias B = 128)
//   posterior P' = P + beta in each half, beta = 0x8000; the accumulator starts at
//             L + beta - dv(v) B, so P' = that + sum_c R'
//   extrinsic d = P' - R' (+ B) = q + beta: bit 15 of each half is [q >= 0], the sign of
//             clamp(q); the clamp itself is not applied (edge_d says why it changes nothing)
//   magnitude na = min(d, 2 beta - d) = beta - |q|   (2 beta - x = ~x + 1 per half)
// Every P', d and na stays inside [0, 0xFFFF] per half for
// (dv + 2) sat <= beta - 1024 and rmax <= 1024, which the launcher checks, so
// sums of R' words are exact whatever the order (borrows cancel modulo 2^32);
// both halves always hold values of a valid decode (an idle half keeps
// decoding its last input).  The arithmetic is the same
// min-sum as the scalar decoder: r = sgn * ((alpha_num * min) >> alpha_shift)
// over the other edges of the check, P = L + sum r, q = clamp(P - r).
//
// No variable-node pass: each check adds its new messages into the next
// posterior buffer with shared-memory atomic adds; that buffer starts at L
// in every word.  For QC codes whose two buffers do not fit a CTA, the
// variable-node-pass form (VN) keeps one buffer and rebuilds it from the
// messages after each check pass; it gives the same words.
//
// The first check pass of a decode reads the zero message in its half; a
// check pass in which no half starts a decode skips that masking.
//
// What bounds it: instruction issue and the two 64-lane pipes (integer and
// multiply-add / 16-bit), then shared-memory wavefronts; DRAM is idle.  So
// the steps are chosen by instruction count: 20 warp instructions per edge of
// two codewords in the check pass of a degree-6 check, of which 2.5 loads,
// half a store and one add to shared memory.  Measured on the decode stage
// against the form before it (magnitudes beta + |q|, outputs by two selects,
// 64-bit generic addresses, the bisection's state in every thread's
// registers, one row block at a time): 2640-node (3,6) QC code, 30,000 candidates,
// 99.5 -> 70 ms; degree 16 (n = 4608), 12,000 candidates, 40 -> 26 ms; degree 28
// (n = 11,520), 8,000 candidates, 82 -> 57 ms; Z = 153, degree 23: 26 -> 7.6 ms (the row-block
// loop gave the group Z / 32 = 4 warps).
#pragma once
#include "decode_impl.cuh"

namespace tsx {
namespace {

__device__ __forceinline__ unsigned vmaxu2(unsigned a, unsigned b) {
    unsigned d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ unsigned vminu2(unsigned a, unsigned b) {
    unsigned d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// per-half adds and signed maximum, modulo 2^16 (an add whose result only feeds a maximum is one instruction with it)
__device__ __forceinline__ unsigned vadd2(unsigned a, unsigned b) {
    unsigned d;
    asm("add.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ unsigned vmaxs2(unsigned a, unsigned b) {
    unsigned d;
    asm("max.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ unsigned prmt(unsigned a, unsigned b, unsigned sel) {
    unsigned d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
// 0xFFFF in each half whose bit 15 is set, else 0
__device__ __forceinline__ unsigned spread15(unsigned x) { return prmt(x, x, 0xBB99u); }
// Shared-memory accesses of the check pass by 32-bit address: with pointers
// the compiler keeps 64-bit generic addresses, whose arithmetic doubled the
// large-degree loop (60 warp instructions per edge pair).  Volatile and
// without a memory clobber: none moves across Grp::sync(), which is volatile asm too and has the
// clobber, and the ordinary accesses between two barriers keep their freedom.
__device__ __forceinline__ unsigned saddr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned lds32(unsigned a) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ unsigned lds16(unsigned a) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds64(unsigned a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint4 lds128(unsigned a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts32(unsigned a, unsigned v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts16(unsigned a, unsigned v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void sts64(unsigned a, unsigned x, unsigned y) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void red_add(unsigned a, unsigned v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// M1 >= M2: the two largest of the values so far
__device__ __forceinline__ void track_max(unsigned a, unsigned &M1, unsigned &M2) {
    M2 = vmaxu2(M2, vminu2(M1, a));
    M1 = vmaxu2(M1, a);
}
// two values at once: five operations instead of six (the two maxima of M2 are one
// three-input instruction), and half as long a dependency chain
__device__ __forceinline__ void track_max2(unsigned a, unsigned b, unsigned &M1, unsigned &M2) {
    const unsigned hi = vmaxu2(a, b), lo = vminu2(a, b);
    M2 = vmaxu2(vmaxu2(M2, lo), vminu2(M1, hi));
    M1 = vmaxu2(M1, hi);
}

constexpr unsigned kBeta = 0x8000u;

template <int V>
struct Int {
    static constexpr int value = V;
    __device__ __forceinline__ constexpr operator unsigned() const { return (unsigned)V; }
};

struct PairConst {
    unsigned NS2, amask2;  // NS2: beta - sat
    unsigned BAN2;  // BETA2 * alpha_num: m an = BAN2 - (beta - m) an (mod 2^32)
    int an, as;
};

// Schedule state of one half, in the group's shared memory: written by the
// group's thread 0 where a decode ends, read by the others after a barrier.
// (Held in every thread's registers it cost 30 of them, and every warp ran
// the bookkeeping.)  Narrow types: what the slot takes beyond a code's words decides
// whether codes at the shared-memory limit run two codewords a lane.
struct HalfS {
    long long idx;       // candidate (absolute index), -1: idle
    long long copy_o;    // record of the finished candidate whose x* is to be copied out, -1: none
    int lo, hi;          // bisection
    int nit;
    int K;               // iteration limit of the candidate
    int16_t I[4];        // impulse nodes (n < 2^15)
    int16_t Limp;        // channel LLR of the impulse nodes in the current decode (|Limp| <= sat < 2^13)
    uint8_t nI, st, phase, ndec, failed;  // (at most 21 decodes a candidate)
    uint8_t keep;        // x buffer (0/1) of the last failing decode; the current decode writes the other
    uint8_t copy;        // x buffer to copy out
    uint8_t fail;        // the decode that ended failed
};

__device__ __forceinline__ PairConst pair_const(const DecodeParams &dp) {
    PairConst pc;
    pc.an = dp.alpha_num;
    pc.as = dp.alpha_shift;
    pc.NS2 = (kBeta - (unsigned)dp.sat) * 0x00010001u;
    pc.amask2 = (0xFFFFu >> pc.as) * 0x00010001u;
    pc.BAN2 = kBeta * 0x00010001u * (unsigned)pc.an;
    return pc;
}

struct PairMisc {
    int red[2 * kMaxGroupWarps];
    unsigned long long okd, okit;  // converged decodes of this group and their iterations
    HalfS h[2];
};

// VN: the variable-node-pass form (QC codes): one posterior buffer, rebuilt
// after each check pass from the stored messages, instead of the
// accumulating second buffer -- 4 bytes per node less, for codes whose
// two-buffer layout does not fit a CTA.
// FILL: QC rows of large degree filled up to an odd number of words.  A code that
// fits a CTA only without the filling keeps its messages by position (message p of row r of a block
// Z words after message p - 1), lanes on consecutive words: a check's words together without the
// filling meet the same banks 32 times at degree 32 and 4 times at 28 (two buffers, 3,000 candidates: degree 32,
// Z = 291: 147 ms, by position 16.4; degree 28, Z = 332: 23.3 and 14.9.  Sampling, degree 32,
// Z = 254, 6,000 samples: 24.3 and 3.0).
template <bool QC, int DC, bool EXACT, bool I8, bool VN = false, bool FILL = true>
struct PairDecoder {
    static constexpr int RSZ = I8 ? 2 : 4;  // bytes of one packed message pair
    static constexpr int kB = I8 ? 128 : 0;  // message bias
    static constexpr unsigned kB2 = (unsigned)kB * 0x00010001u;
    const DevCode &g;
    const SGraph &sg;
    const Grp &gp;
    const PairConst &pc;
    unsigned Rb;  // shared address of the packed messages, RSZ bytes per edge

    __device__ __forceinline__ unsigned ldR(unsigned a) const {
        if constexpr (I8) return prmt(lds16(a), 0u, 0x4140u);  // bytes b0, b1 -> halves
        else return lds32(a);
    }
    __device__ __forceinline__ void stR(unsigned a, unsigned v) const {
        if constexpr (I8) sts16(a, prmt(v, 0u, 0x0020u));
        else sts32(a, v);
    }

    // an edge's incoming message; MASK: some half starts a decode in this
    // pass (km is 0 there, 0xFFFF in a half that goes on) and reads the zero message
    template <bool MASK>
    __device__ __forceinline__ unsigned mask_y(unsigned y, unsigned km) const {
        if constexpr (!MASK) return y;
        else if constexpr (I8) return (y & km) | (kB2 & ~km);
        else return ((km & 0xFFFFu) ? (unsigned)(int)(int16_t)y : 0u) + ((km >> 16) ? (y + 0x8000u) & 0xFFFF0000u : 0u);
    }
    template <bool MASK>
    __device__ __forceinline__ unsigned ldy(unsigned a, unsigned km) const {
        return mask_y<MASK>(ldR(a), km);
    }

    // the extrinsic value of one edge without clamping: d = (P - r) + beta, which the launcher's
    // bounds keep inside each half and which has the sign of clamp(P - r),
    // and na = beta - |P - r|.  Where |P - r| > sat the clamped magnitude
    // would be sat: min1 and min2 start at sat, so they come out
    // the same, and such an edge's output is the same too -- it is not the
    // minimum unless min1 = min2 = sat, when both outputs are equal.
    __device__ __forceinline__ void edge_d(unsigned x, unsigned y, unsigned &d, unsigned &na) const {
        d = x - y;
        if constexpr (I8) d += kB2;
        na = neg_abs(d);
    }
    __device__ __forceinline__ static unsigned neg_abs(unsigned d) { return vminu2(d, (~d) + 0x00010001u); }

    // What the outputs of a check's edges share.  Edge p sends the magnitude o2 if |q_p| is min1,
    // else o1 (o = (alpha_num min) >> alpha_shift).  That is
    //   max(o2 + min1 - |q_p|, o1):
    // equal to o2 >= o1 where |q_p| = min1; elsewhere |q_p| >= min2 (also with ties), and
    // o2 - o1 <= min2 - min1 because alpha <= 1 and the floors are of one multiple each, so
    // the first term is at most o1.  One fused add-max per edge.
    struct Outs {
        unsigned S, o1;  // S = o2 + min1 - beta: na + S = o2 + min1 - |q|, modulo 2^16 per half
        unsigned sx;     // sign parity over the edges, less the edge itself once xor-ed with its d
    };
    __device__ __forceinline__ Outs outs(unsigned M1, unsigned M2, unsigned sx, int deg) const {
        Outs o;
        o.o1 = ((pc.BAN2 - M1 * (unsigned)pc.an) >> pc.as) & pc.amask2;
        const unsigned o2 = ((pc.BAN2 - M2 * (unsigned)pc.an) >> pc.as) & pc.amask2;
        o.S = vadd2(o2, (~M1) + 0x00010001u);  // 2 beta - M1 = beta + min1, which is min1 - beta modulo 2^16
        // bit 15 of sx ^ d_p = parity of #(q >= 0) over the other edges;
        // negatives among the others = (deg - 1) - that
        o.sx = sx ^ (((deg - 1) & 1) ? 0x80008000u : 0u);
        return o;
    }
    // the new message B +- o of an edge from its d and na
    __device__ __forceinline__ unsigned edge_out(unsigned d, unsigned na, const Outs &o) const {
        const unsigned neg = spread15(o.sx ^ d);                  // 0xFFFF: others' sign product < 0
        const unsigned mag = vmaxs2(vadd2(na, o.S), o.o1);
        const unsigned r = (mag ^ neg) - neg;
        return I8 ? r + kB2 : r;
    }

    // One check of up to N edges (EX: exactly N), the edges' d and addresses in
    // registers between the two passes.  pv(p): byte offset of P'[v_p]; re(p):
    // address of R'[e_p].  Reads Pc, adds the new messages into Pn (VN form:
    // stores them only).  Returns the unsatisfied flags in bits 0 and 16.
    template <bool MASK, int N, bool EX, class PV, class RE>
    __device__ __forceinline__ int node(int deg, unsigned km, bool writeR, unsigned Pc, unsigned Pn, PV pv,
                                        RE re) const {
        unsigned sp = 0, sx = 0, M1 = pc.NS2, M2 = pc.NS2;
        unsigned q[N], na[N], po[N];
#pragma unroll
        for (int p = 0; p < N; p++) {
            if (EX || p < deg) {
                po[p] = pv(p);
                const unsigned x = lds32(Pc + po[p]);
                const unsigned y = ldy<MASK>(re(p), km);
                sp ^= x;
                edge_d(x, y, q[p], na[p]);
                sx ^= q[p];
                track_max(na[p], M1, M2);
            }
        }
        if (writeR) {
            const Outs o = outs(M1, M2, sx, EX ? N : deg);
#pragma unroll
            for (int p = 0; p < N; p++) {
                if (EX || p < deg) {
                    const unsigned rn = edge_out(q[p], na[p], o);
                    stR(re(p), rn);
                    if constexpr (!VN) red_add(Pn + po[p], rn);
                }
            }
        }
        return unsat2(sp, EX ? N : deg);
    }
    // syndrome bit of each half: sp bit 15 = parity of #(P >= 0), and
    // #(P < 0) = deg - #(P >= 0)
    __device__ __forceinline__ static int unsat2(unsigned sp, int deg) {
        return (int)(((sp ^ ((deg & 1) ? 0x80008000u : 0u)) >> 15) & 0x00010001u);
    }

    // check-regular codes (EXACT, 16-bit storage, DC even): the check's DC
    // message words are contiguous (check-major layout, 4 DC bytes a check)
    // and move as DC/2 8-byte accesses; a warp's 8-byte accesses at a stride
    // of 4 DC bytes = 24 bytes (DC = 6) touch every bank once per half-warp.
    // Otherwise the same steps as node().
    template <bool MASK, class PV>
    __device__ __forceinline__ int node_cm(unsigned ra, unsigned km, bool writeR, unsigned Pc, unsigned Pn,
                                           PV pv) const {
        static_assert(EXACT && !I8 && DC % 2 == 0, "check-major form");
        unsigned sp = 0, sx = 0, M1 = pc.NS2, M2 = pc.NS2;
        unsigned q[DC], na[DC], po[DC];
#pragma unroll
        for (int t = 0; t < DC / 2; t++) {
            const uint2 w = lds64(ra + 8 * t);
#pragma unroll
            for (int e = 0; e < 2; e++) {
                const int p = 2 * t + e;
                po[p] = pv(p);
                const unsigned x = lds32(Pc + po[p]);
                const unsigned y0 = e ? w.y : w.x;
                const unsigned y = mask_y<MASK>(y0, km);
                sp ^= x;
                edge_d(x, y, q[p], na[p]);
                sx ^= q[p];
            }
            track_max2(na[2 * t], na[2 * t + 1], M1, M2);
        }
        if (writeR) {
            const Outs o = outs(M1, M2, sx, DC);
#pragma unroll
            for (int t = 0; t < DC / 2; t++) {
                const unsigned r0 = edge_out(q[2 * t], na[2 * t], o), r1 = edge_out(q[2 * t + 1], na[2 * t + 1], o);
                sts64(ra + 8 * t, r0, r1);
                if constexpr (!VN) {
                    red_add(Pn + po[2 * t], r0);
                    red_add(Pn + po[2 * t + 1], r1);
                }
            }
        }
        return unsat2(sp, DC);
    }

    // large degree: the first pass leaves each edge's extrinsic word d in its
    // message slot (16-bit storage: a slot holds both halves' d), the second
    // reads it back; with 8-bit storage the second pass reloads P and
    // recomputes d.  (Unrolled over up to 32 edges with d in registers, the
    // loop did not fit the instruction cache: 0.57x on a degree-16 code.)
    // ra: address of the check's first message, stride: bytes between its
    // messages.  QC codes keep a check's messages together, an odd number of
    // words a check, so that lanes hit different banks and every offset is a constant (FILL).
    // Edges are taken four at a time, loads first: no load waits behind the
    // stores of the edges before it.
    template <bool MASK, class PV, class PV2, class Stride>
    __device__ __forceinline__ int node_twopass(int deg, unsigned km, bool writeR, unsigned Pc, unsigned Pn,
                                                PV pv, PV2 pv2, unsigned ra, Stride stride) const {
        const unsigned rs = stride;
        unsigned sp = 0, sx = 0, M1 = pc.NS2, M2 = pc.NS2;
        auto first = [&](auto width, int p, unsigned a) {
            constexpr int W = decltype(width)::value;
            unsigned x[W], y[W], na[W];
            if constexpr (W == 1) x[0] = pv(p);
            else
#pragma unroll
                for (int e = 0; e < W; e += 2) pv2(p + e, x + e);
#pragma unroll
            for (int e = 0; e < W; e++) {
                x[e] = lds32(Pc + x[e]);
                y[e] = ldy<MASK>(a + e * rs, km);
            }
#pragma unroll
            for (int e = 0; e < W; e++) {
                sp ^= x[e];
                edge_d(x[e], y[e], y[e], na[e]);
                sx ^= y[e];
            }
            if constexpr (!I8) {
                if (writeR) {
#pragma unroll
                    for (int e = 0; e < W; e++) stR(a + e * rs, y[e]);
                }
            }
            if constexpr (W == 1) track_max(na[0], M1, M2);
            else
#pragma unroll
                for (int e = 0; e < W; e += 2) track_max2(na[e], na[e + 1], M1, M2);
        };
        int p = 0;
        unsigned a = ra;
#pragma unroll 2
        for (; p + 4 <= deg; p += 4, a += 4 * rs) first(Int<4>{}, p, a);
        if (deg & 2) {
            first(Int<2>{}, p, a);
            p += 2;
            a += 2 * rs;
        }
        if (deg & 1) first(Int<1>{}, p, a);
        if (writeR) {
            const Outs o = outs(M1, M2, sx, deg);
            auto second = [&](auto width, int p, unsigned a) {
                constexpr int W = decltype(width)::value;
                unsigned po[W], d[W], na[W];
                if constexpr (W == 1) po[0] = pv(p);
                else
#pragma unroll
                    for (int e = 0; e < W; e += 2) pv2(p + e, po + e);
#pragma unroll
                for (int e = 0; e < W; e++) {
                    if constexpr (!I8) {
                        d[e] = ldR(a + e * rs);
                        na[e] = neg_abs(d[e]);
                    } else {
                        edge_d(lds32(Pc + po[e]), ldy<MASK>(a + e * rs, km), d[e], na[e]);
                    }
                }
#pragma unroll
                for (int e = 0; e < W; e++) d[e] = edge_out(d[e], na[e], o);
#pragma unroll
                for (int e = 0; e < W; e++) {
                    stR(a + e * rs, d[e]);
                    if constexpr (!VN) red_add(Pn + po[e], d[e]);
                }
            };
            p = 0;
            a = ra;
#pragma unroll 2
            for (; p + 4 <= deg; p += 4, a += 4 * rs) second(Int<4>{}, p, a);
            if (deg & 2) {
                second(Int<2>{}, p, a);
                p += 2;
                a += 2 * rs;
            }
            if (deg & 1) second(Int<1>{}, p, a);
        }
        return unsat2(sp, deg);
    }

    // check pass; returns u of half 0 in the low 16 bits and half 1 above (the
    // caller passes a group barrier before the next check pass)
    template <bool MASK>
    __device__ __forceinline__ int check_pass(unsigned km, bool writeR, const unsigned *Pcur,
                                              unsigned *Pnext) const {
        int u = 0;  // unsatisfied checks: half 0 in the low 16 bits, half 1 above
        const unsigned Pc = saddr(Pcur), Pn = saddr(Pnext);
        const int Z = g.Z;
        if constexpr (QC) {
            // all row blocks at once (check c = i Z + r), so that a group may be wider than Z rows
            // and no lane idles at a block's last rows
            const unsigned Z4 = 4u * (unsigned)Z;
            const unsigned zm = Z > 1 ? 0xFFFFFFFFu / (unsigned)Z + 1u : 0u;  // c / Z = umulhi(c, zm), c < 2^16
            const unsigned rt0 = saddr(sg.rt);
            for (int c = gp.gt; c < g.m; c += gp.T) {
                const int i = Z > 1 ? (int)__umulhi((unsigned)c, zm) : c;
                const int r = c - i * Z;
                const unsigned rt = rt0 + 8u * (unsigned)(i * rt_row(g));
                const unsigned r4 = 4u * (unsigned)r;
                const auto at = [&](unsigned x, unsigned y) {  // 4 x column block start, 4 x shift
                    const unsigned t = r4 + y;
                    return x + __viaddmin_u32(t, 0u - Z4, t);  // min(t - Z4, t): t mod Z4
                };
                const auto pv = [&](int p) {
                    const uint2 e = lds64(rt + 8u * (unsigned)p);
                    return at(e.x, e.y);
                };
                const auto pv2 = [&](int p, unsigned *o) {  // positions p and p + 1, p even
                    const uint4 e = lds128(rt + 8u * (unsigned)p);
                    o[0] = at(e.x, e.y);
                    o[1] = at(e.z, e.w);
                };
                if constexpr (EXACT && !I8 && DC % 2 == 0) {
                    u += node_cm<MASK>(Rb + (unsigned)c * (DC * RSZ), km, writeR, Pc, Pn, pv);
                } else {
                    const int deg = EXACT ? DC : sg.rdeg[i];
                    if constexpr (DC <= 8) {
                        const unsigned ra = Rb + (unsigned)((sg.reoff[i] + r) * RSZ), rs = (unsigned)(Z * RSZ);
                        u += node<MASK, DC, EXACT>(deg, km, writeR, Pc, Pn, pv,
                                                   [&](int p) { return ra + (unsigned)p * rs; });
                    } else if constexpr (FILL) {
                        u += node_twopass<MASK>(deg, km, writeR, Pc, Pn, pv, pv2,
                                                Rb + (unsigned)((sg.reoff[i] + r * (deg | 1)) * RSZ), Int<RSZ>{});
                    } else {
                        u += node_twopass<MASK>(deg, km, writeR, Pc, Pn, pv, pv2, Rb + (unsigned)((sg.reoff[i] + r) * RSZ),
                                                (unsigned)(Z * RSZ));
                    }
                }
            }
        } else {
            const unsigned cv = saddr(sg.c_vn);
            const int m = g.m;
            for (int c = gp.gt; c < m; c += gp.T) {
                const int e0 = EXACT ? c * DC : (int)sg.c_ptr[c];  // check-regular: rows of DC edges
                const unsigned cva = cv + 2u * (unsigned)e0;
                const auto pv = [&](int p) { return 4u * lds16(cva + 2u * (unsigned)p); };
                const auto pv2 = [&](int p, unsigned *o) {
                    o[0] = pv(p);
                    o[1] = pv(p + 1);
                };
                if constexpr (EXACT && !I8 && DC % 2 == 0) {
                    // check-regular: messages check-major
                    u += node_cm<MASK>(Rb + (unsigned)(e0 * RSZ), km, writeR, Pc, Pn, pv);
                } else {
                    const int deg = EXACT ? DC : sg.c_ptr[c + 1] - e0;
                    const unsigned ra = Rb + (unsigned)(c * RSZ), rs = (unsigned)(m * RSZ);
                    if constexpr (DC <= 8)
                        u += node<MASK, DC, EXACT>(deg, km, writeR, Pc, Pn, pv,
                                                   [&](int p) { return ra + (unsigned)p * rs; });
                    else u += node_twopass<MASK>(deg, km, writeR, Pc, Pn, pv, pv2, ra, rs);
                }
            }
        }
        return gp.sum_pass(u);
    }

    __device__ __forceinline__ int vdeg(int v) const {
        if constexpr (QC) return sg.cdeg[v / g.Z];
        else return sg.v_ptr[v + 1] - sg.v_ptr[v];
    }

    // the accumulator: L'(v) = L + beta - dv B in both halves (impulse
    // nodes are patched afterwards)
    // a run of equal words, 16 bytes per store where the run is aligned
    __device__ __forceinline__ void fill(unsigned *row, int count, unsigned w) const {
        if (((uintptr_t)row & 15) == 0 && (count & 3) == 0) {
            uint4 *r4 = (uint4 *)row;
            const uint4 w4 = make_uint4(w, w, w, w);
            for (int k = gp.gt; k < (count >> 2); k += gp.T) r4[k] = w4;
        } else {
            for (int k = gp.gt; k < count; k += gp.T) row[k] = w;
        }
    }
    __device__ __forceinline__ void init_accum(unsigned *Pn, int Lb) const {
        if (!I8 || g.dv_min == g.dv_max) {  // no bias to take off, or the same for every node: one value
            const unsigned l = (unsigned)(Lb + (int)kBeta - g.dv_max * kB);
            fill(Pn, g.n, l | (l << 16));
        } else if constexpr (QC) {
            const int Z = g.Z;
            const unsigned zm = Z > 1 ? 0xFFFFFFFFu / (unsigned)Z + 1u : 0u;
            if ((Z & 3) == 0 && ((uintptr_t)Pn & 15) == 0) {  // four nodes of one column block per store
                for (int v = 4 * gp.gt; v < g.n; v += 4 * gp.T) {
                    const unsigned l = (unsigned)(Lb + (int)kBeta - sg.cdeg[__umulhi((unsigned)v, zm)] * kB);
                    const unsigned l2 = l | (l << 16);
                    *(uint4 *)(Pn + v) = make_uint4(l2, l2, l2, l2);
                }
            } else {
                for (int v = gp.gt; v < g.n; v += gp.T) {
                    const int j = Z > 1 ? (int)__umulhi((unsigned)v, zm) : v;
                    const unsigned l = (unsigned)(Lb + (int)kBeta - sg.cdeg[j] * kB);
                    Pn[v] = l | (l << 16);
                }
            }
        } else {
            for (int v = gp.gt; v < g.n; v += gp.T) {
                const unsigned l = (unsigned)(Lb + (int)kBeta - vdeg(v) * kB);
                Pn[v] = l | (l << 16);
            }
        }
    }

    __device__ __forceinline__ static void set_half(unsigned *P, int v, int h, unsigned val) {
        ((uint16_t *)P)[2 * v + h] = (uint16_t)val;
    }
    __device__ __forceinline__ static void add_half(unsigned *P, int v, int h, int delta) {
        uint16_t *q = (uint16_t *)P + 2 * v + h;
        *q = (uint16_t)(*q + delta);
    }

    // the variable-node pass of the VN form (QC): P'(v) = L + beta - dv B +
    // sum of the R' of v's edges in both halves -- the value the accumulating
    // form builds with red.add -- for the baseline channel value L (impulse
    // nodes are corrected afterwards)
    __device__ __forceinline__ void vn_pass(unsigned *P, int Lb) const {
        const int Z = g.Z;
        const unsigned zm = Z > 1 ? 0xFFFFFFFFu / (unsigned)Z + 1u : 0u;  // v / Z = umulhi(v, zm), v < 2^15
        for (int v = gp.gt; v < g.n; v += gp.T) {
            const int j = Z > 1 ? (int)__umulhi((unsigned)v, zm) : v;
            const int k = v - j * Z;
            const int dv = sg.cdeg[j];
            const int2 *ct = sg.ct + j * g.dv_max;  // message offset, stride and shift of the t-th block
            const unsigned l = (unsigned)(Lb + (int)kBeta - dv * kB);
            unsigned acc = l | (l << 16);
            for (int t = 0; t < dv; t++) {
                // block (i, j) with shift s joins row r to column (r + s) mod Z: r = (k - s) mod Z
                const int2 e = ct[t];
                const int r = wrapZneg(k - (e.y >> 8), Z);
                acc += ldR(Rb + (unsigned)((e.x + r * (e.y & 0xFF)) * RSZ));
            }
            P[v] = acc;
        }
    }

    // x_k of half h (P < 0, i.e. bit 15 of the half clear) into a bitmask
    __device__ __forceinline__ void save_x(const unsigned *P, int h, uint32_t *xw) const {
        const unsigned bitpos = 15u + 16u * h;
        for (int base = 0; base < g.n; base += gp.T) {
            const int v = base + gp.gt;
            const bool bit = v < g.n && !((P[v] >> bitpos) & 1u);
            const unsigned w = __ballot_sync(0xffffffffu, bit);
            const int wi = (base >> 5) + gp.gw;
            if (gp.lane == 0 && (wi << 5) < g.n) xw[wi] = w;
        }
    }

    __device__ __forceinline__ int any_neg(const unsigned *P, int h) const {
        const unsigned bitpos = 15u + 16u * h;
        int neg = 0;
        for (int v = gp.gt; v < g.n; v += gp.T) neg |= !((P[v] >> bitpos) & 1u);
        return gp.sum(neg);
    }
};

// The decode loop of one group (G warps, group index grp) over the
// candidate queue of one code; the code's tables are already in sg.  Every
// thread keeps, per half, only what each iteration needs (whether it runs,
// its iteration, its limit, the smallest u_k); the schedule itself is in
// shared memory and is advanced by thread 0 where a decode ends.
template <bool QC, int DC, bool EXACT, bool I8, bool VN = false, bool FILL = true>
__device__ __forceinline__ void pair_run(const DevCode &g, const DecodeParams &dp, const EnumBuffers &b,
                                         const SlotLayout &lay, int G, const SGraph &sg, unsigned char *smem, int grp) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *slot = smem + lay.tables_bytes + grp * lay.slot_bytes;
    PairMisc *misc = (PairMisc *)(slot + lay.misc_off);
    HalfS *const hs = misc->h;
    Grp gp;
    gp.G = G;
    gp.T = 32 * G;
    gp.gw = warp - grp * G;
    gp.gt = gp.gw * 32 + lane;
    gp.lane = lane;
    gp.bar = 1 + grp;
    gp.red = misc->red;
    unsigned *Pbuf = (unsigned *)(slot + lay.p_off);  // [2][n] ([n] in the VN form)
    const int nw = (g.n + 31) >> 5;
    uint32_t *xb = (uint32_t *)(slot + lay.xa_off);  // 4 buffers of nw words: [half][2]

    const PairConst pc = pair_const(dp);
    PairDecoder<QC, DC, EXACT, I8, VN, FILL> dec{g, sg, gp, pc, saddr(slot + lay.r_off)};

    const long long total = (long long)b.ctr->n_cand_total;
    const long long end = b.cand_end < 0 || b.cand_end > total ? total : b.cand_end;
    const int Lb = clampi(dp.base_llr, -dp.sat, dp.sat);
    const int amax = (1 << dp.amp_steps) - 1;
    long long my_dec = 0, my_it = 0;  // (thread 0's)
    int pcur = 0;                     // which posterior buffer holds P_k

    // ---- the schedule (thread 0 of the group) ----
    auto fetch = [&](HalfS &h) {
        const long long idx = b.cand_begin + (long long)atomicAdd(b.queue, 1ull);
        if (idx >= end) {
            h.idx = -1;
            h.nI = 0;
            return;
        }
        const int4 I4 = b.cands[idx];
        h.idx = idx;
        h.I[0] = (int16_t)I4.x; h.I[1] = (int16_t)I4.y; h.I[2] = (int16_t)I4.z; h.I[3] = (int16_t)I4.w;
        h.nI = (I4.x >= 0) + (I4.y >= 0) + (I4.z >= 0) + (I4.w >= 0);
        h.lo = 0; h.hi = amax; h.st = 0; h.phase = 0;
        h.ndec = 0; h.nit = 0; h.failed = 0;
        h.Limp = (int16_t)clampi(dp.base_llr - amax, -dp.sat, dp.sat);
        h.K = cand_limit(dp, b, idx);
    };
    // the candidate's records; its x* is copied out by the whole group afterwards
    auto finish = [&](HalfS &h) {
        const long long o = h.idx - b.rec_base;
        b.c_thr[o] = h.failed ? h.hi : -1;
        b.c_thr_f[o] = -1.0f;
        b.c_slot[o] = -1;
        b.c_flags[o] = 0;
        b.c_decodes[o] = h.ndec;
        b.c_iters[o] = h.nit;
        if (h.failed) {  // (at most one candidate of a half between two decodes: the ones that
            h.copy_o = o;  //  follow it without a decode have not failed)
            h.copy = h.keep;
        }
        my_dec += h.ndec;
        my_it += h.nit;
        fetch(h);
    };
    // the next amplitude of the bisection, or the end of the candidate
    auto next_amp = [&](HalfS &h) {
        if (h.st < dp.amp_steps && h.hi - h.lo > 1) {
            h.st++;
            h.Limp = (int16_t)clampi(dp.base_llr - ((h.lo + h.hi) >> 1), -dp.sat, dp.sat);
        } else {
            finish(h);
        }
    };
    // past trivial decodes (impulse LLR >= 0: every hard decision 0, u_0 = 0, success at
    // iteration 0) until a decode that needs iterations is set up or no candidate is left
    auto settle = [&](HalfS &h) {
        while (h.idx >= 0 && h.Limp >= 0) {
            h.ndec++;
            misc->okd++;
            if (h.phase == 0) {
                finish(h);  // no failure at the largest amplitude
            } else {
                h.lo = (h.lo + h.hi) >> 1;  // the decode at mid succeeded
                next_amp(h);
            }
        }
    };
    // the decode of half h ended at iteration kl
    auto advance = [&](HalfS &h, int kl) {
        h.copy_o = -1;
        h.ndec++;
        h.nit += kl;
        if (!h.fail) {
            misc->okd++;
            misc->okit += kl;
        }
        if (h.phase == 0) {
            if (!h.fail) {
                finish(h);
            } else {
                h.failed = 1;
                h.keep ^= 1;
                h.phase = 1;
                next_amp(h);
            }
        } else {
            const int mid = (h.lo + h.hi) >> 1;
            if (h.fail) {
                h.hi = mid;
                h.keep ^= 1;
            } else {
                h.lo = mid;
            }
            next_amp(h);
        }
        settle(h);
    };

    // half hh of the current posteriors for a new decode: P = L
    auto start_cur = [&](int hh, unsigned *Pc) {
        for (int v = gp.gt; v < g.n; v += gp.T) dec.set_half(Pc, v, hh, (unsigned)(Lb + (int)kBeta));
    };
    // its impulse nodes
    auto patch_cur = [&](int hh, unsigned *Pc) {
        if (gp.gt < hs[hh].nI) dec.set_half(Pc, hs[hh].I[gp.gt], hh, (unsigned)(hs[hh].Limp + (int)kBeta));
    };
    // The accumulator starts at the baseline L' in every word; its impulse
    // nodes get L_imp - L_base added in their half with the check pass's
    // red.adds (threads 0-3: half 0, 4-7: half 1).  The adds are exact and
    // commute: the word's final halves are in range, so no intermediate
    // carry or borrow between the halves survives.
    // Small degrees keep them in registers between the ends of decodes: the
    // loads in a row from the schedule were on the path of every pass (general (1008, 504)
    // code 92.3 -> 90.6 ms, n = 432 7.28 -> 7.13; degree 16 is 1 % slower with them).
    constexpr bool kImpRegs = !VN && DC <= 8;
    unsigned imp_off = 0, imp_add = 0;
    bool imp = false;  // (threads 0-7 with a node)
    auto load_impulse = [&]() {  // (after a barrier)
        if (gp.gt < 8) {
            const int j = gp.gt & 3, hh = gp.gt >> 2;
            imp = j < hs[hh].nI;  // (0 for an idle half)
            if (imp) {
                const unsigned d = (unsigned)(hs[hh].Limp - Lb);
                imp_off = 4u * (unsigned)hs[hh].I[j];
                imp_add = hh ? d << 16 : d;
            }
        }
    };
    auto impulse_adds = [&](unsigned *Pn) {
        if constexpr (kImpRegs) {
            if (imp) red_add(saddr(Pn) + imp_off, imp_add);
        } else if (gp.gt < 8) {
            const int j = gp.gt & 3, hh = gp.gt >> 2;
            if (j < hs[hh].nI) {
                const unsigned d = (unsigned)(hs[hh].Limp - Lb);
                red_add(saddr(Pn + hs[hh].I[j]), hh ? d << 16 : d);
            }
        }
    };
    // VN form: the impulse nodes of half hh after a variable-node pass (built with the baseline L)
    auto patch_vn = [&](int hh, unsigned *Pc) {
        if (gp.gt < hs[hh].nI) dec.add_half(Pc, hs[hh].I[gp.gt], hh, hs[hh].Limp - Lb);
    };

    bool act[2], first[2];
    int k[2], K[2], ub[2];
    auto load_half = [&](int hh) {  // (after a barrier)
        act[hh] = hs[hh].idx >= 0;
        K[hh] = hs[hh].K;
        k[hh] = 0;
        ub[hh] = 0x7fffffff;
        first[hh] = true;
    };

    if (gp.gt == 0) {
        misc->okd = 0;
        misc->okit = 0;
        for (int hh = 0; hh < 2; hh++) {
            hs[hh].keep = 1;
            hs[hh].K = 0;
            hs[hh].copy_o = -1;
            fetch(hs[hh]);
            settle(hs[hh]);
        }
    }
    {
        unsigned *Pc = Pbuf, *Pn = Pbuf + g.n;
        if constexpr (!VN) dec.init_accum(Pn, Lb);
        for (int hh = 0; hh < 2; hh++) start_cur(hh, Pc);  // idle halves too: every word stays a valid decode state
        gp.sync();
        for (int hh = 0; hh < 2; hh++) {
            load_half(hh);
            patch_cur(hh, Pc);
        }
        if constexpr (kImpRegs) load_impulse();
        gp.sync();
    }

    while (act[0] || act[1]) {
        unsigned *Pc = VN ? Pbuf : Pbuf + pcur * g.n, *Pn = VN ? Pbuf : Pbuf + (pcur ^ 1) * g.n;
        const bool wr = (act[0] && k[0] < K[0]) || (act[1] && k[1] < K[1]);
        // u_k of both halves from P_k = Pc; Pn accumulates P_{k+1}
        if constexpr (!VN) impulse_adds(Pn);
        // (the common form -- no half starting, messages written -- compiled without the mask and
        // with writeR constant)
        int us;
        if (wr && !first[0] && !first[1]) {
            us = dec.template check_pass<false>(0u, true, Pc, Pn);
        } else {
            const unsigned km = (first[0] ? 0xFFFF0000u : 0xFFFFFFFFu) & (first[1] ? 0x0000FFFFu : 0xFFFFFFFFu);
            us = dec.template check_pass<true>(km, wr, Pc, Pn);
        }
        bool ended[2] = {false, false};
        bool read_pc = false;  // some thread read P_k after the check pass (uniform)
#pragma unroll
        for (int hh = 0; hh < 2; hh++) {
            if (!act[hh]) continue;
            const int u = hh == 0 ? (us & 0xFFFF) : (us >> 16);
            const bool end_now = u == 0 || k[hh] == K[hh];
            if ((k[hh] >= g.wstart && u < ub[hh]) || (end_now && k[hh] < g.wstart)) {
                ub[hh] = u;
                dec.save_x(Pc, hh, xb + (2 * hh + (hs[hh].keep ^ 1)) * nw);
                read_pc = true;
            }
            if (end_now) {
                const bool fail = u != 0 || dec.any_neg(Pc, hh) != 0;
                if (gp.gt == 0) hs[hh].fail = fail;
                ended[hh] = true;
                read_pc = true;
            }
        }
        if constexpr (VN) {
            // P_{k+1} from the messages just written, in place of P_k
            gp.sync();
            if (wr) dec.vn_pass(Pc, Lb);
        }
        if (ended[0] || ended[1]) {
            gp.sync();  // x buffers and P_k read and written by every thread
            if (gp.gt == 0) {
#pragma unroll
                for (int hh = 0; hh < 2; hh++)
                    if (ended[hh]) advance(hs[hh], k[hh]);
            }
            gp.sync();
#pragma unroll
            for (int hh = 0; hh < 2; hh++) {
                if (!ended[hh]) continue;
                const long long o = hs[hh].copy_o;
                if (o >= 0) {  // x* of the candidate that ended (its buffer is not written before the next barrier)
                    const uint32_t *src = xb + (2 * hh + hs[hh].copy) * nw;
                    uint32_t *dst = b.xstar + o * (long long)b.nw;
                    for (int w = gp.gt; w < nw; w += gp.T) dst[w] = src[w];
                }
                load_half(hh);
                if (act[hh]) start_cur(hh, VN ? Pc : Pn);
            }
            if constexpr (kImpRegs) load_impulse();
        } else if (VN || read_pc) {
            gp.sync();
        }
#pragma unroll
        for (int hh = 0; hh < 2; hh++) {
            if (act[hh] && !ended[hh]) {
                k[hh]++;
                first[hh] = false;
            }
        }
        // the old P_k becomes the next accumulator
        if constexpr (!VN) dec.init_accum(Pc, Lb);
        if (VN || ended[0] || ended[1]) {
            if (ended[0] || ended[1]) gp.sync();  // after start_cur's stores
#pragma unroll
            for (int hh = 0; hh < 2; hh++) {
                if (!act[hh]) continue;
                if (ended[hh]) patch_cur(hh, VN ? Pc : Pn);
                else if constexpr (VN) patch_vn(hh, Pc);
            }
        }
        gp.sync();
        pcur ^= 1;
    }
    if (gp.gt == 0) {
        atomicAdd(&b.ctr->decodes, (unsigned long long)my_dec);
        atomicAdd(&b.ctr->iterations, (unsigned long long)my_it);
        atomicAdd(&b.ctr->edge_updates, (unsigned long long)my_it * (unsigned long long)g.E);
        atomicAdd(&b.ctr->ok_decodes, misc->okd);
        atomicAdd(&b.ctr->ok_iters, misc->okit);
    }
}

template <bool QC, int DC, bool EXACT, bool I8, bool FILL = true>
__global__ void __launch_bounds__(32 * pair_kernel_warps(DC, EXACT), 1)
    pair_kernel(DevCode g, DecodeParams dp, EnumBuffers b, SlotLayout lay, int G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SGraph sg = load_tables(g, smem, 1, DC > 8 && FILL);
    __syncthreads();
    pair_run<QC, DC, EXACT, I8, false, FILL>(g, dp, b, lay, G, sg, smem, (threadIdx.x >> 5) / G);
}

// the VN form for QC codes of large check degree whose two-buffer layout does not fit
template <bool I8, bool FILL>
__global__ void __launch_bounds__(32 * pair_kernel_warps(32, false), 1) pair_vn_kernel(DevCode g, DecodeParams dp, EnumBuffers b,
                                                               SlotLayout lay, int G) {
    extern __shared__ __align__(16) unsigned char smem[];
    const SGraph sg = load_tables(g, smem, 2, FILL);
    __syncthreads();
    pair_run<true, 32, false, I8, true, FILL>(g, dp, b, lay, G, sg, smem, (threadIdx.x >> 5) / G);
}

// One persistent launch over several codes: every CTA works through the
// codes in order, each with its own tables, slot layout and group size,
// taking candidates from that code's queue until it is empty (CTAs move
// on independently, so no code waits for the slowest CTA of another).
// The items are a __grid_constant__ kernel parameter: the decoders read
// each code's description from the constant bank, as the single-code kernel
// does, instead of holding it in registers.
template <bool QC, int DC, bool EXACT, bool I8>
__global__ void __launch_bounds__(32 * kBatchWarps, 1) batch_kernel(const __grid_constant__ BatchArgs args, int n_items) {
    extern __shared__ __align__(16) unsigned char smem[];
    for (int c = 0; c < n_items; c++) {
        const BatchItem &it = args.it[c];
        const bool filled = DC > 8 && it.g.row_odd;
        const SGraph sg = load_tables(it.g, smem, 1, filled);
        __syncthreads();
        const int grp = (threadIdx.x >> 5) / it.G;
        if (grp < it.groups) {
            if constexpr (QC && DC > 8) {
                if (!filled) pair_run<QC, DC, EXACT, I8, false, false>(it.g, it.dp, it.b, it.lay, it.G, sg, smem, grp);
                else pair_run<QC, DC, EXACT, I8>(it.g, it.dp, it.b, it.lay, it.G, sg, smem, grp);
            } else {
                pair_run<QC, DC, EXACT, I8>(it.g, it.dp, it.b, it.lay, it.G, sg, smem, grp);
            }
        }
        __syncthreads();
    }
}

template <bool I8>
cudaError_t launch_pair(const DevCode &g, const DecodeParams &dp, const EnumBuffers &b, const LaunchShape &sh,
                        cudaStream_t st) {
    const bool qc = g.kind == TSX_CODE_QC;
    const bool reg6 = g.dc_min == 6 && g.dc_max == 6;
    if (reg6)
        return qc && !g.by_rows ? launch_persistent(pair_kernel<true, 6, true, I8>, sh, st, g, dp, b, sh.lay, sh.G)
                  : launch_persistent(pair_kernel<false, 6, true, I8>, sh, st, g, dp, b, sh.lay, sh.G);
    if (g.dc_max <= 8)
        return qc ? launch_persistent(pair_kernel<true, 8, false, I8>, sh, st, g, dp, b, sh.lay, sh.G)
                  : launch_persistent(pair_kernel<false, 8, false, I8>, sh, st, g, dp, b, sh.lay, sh.G);
    if (qc && !g.row_odd) return launch_persistent(pair_kernel<true, 32, false, I8, false>, sh, st, g, dp, b, sh.lay, sh.G);
    return qc ? launch_persistent(pair_kernel<true, 32, false, I8>, sh, st, g, dp, b, sh.lay, sh.G)
              : launch_persistent(pair_kernel<false, 32, false, I8>, sh, st, g, dp, b, sh.lay, sh.G);
}

template <bool I8>
cudaError_t launch_batch_t(const BatchArgs &items, int n, bool qc, int dc_max, bool reg6, const LaunchShape &sh,
                           cudaStream_t st) {
    if (reg6)
        return qc ? launch_persistent(batch_kernel<true, 6, true, I8>, sh, st, items, n)
                  : launch_persistent(batch_kernel<false, 6, true, I8>, sh, st, items, n);
    if (dc_max <= 8)
        return qc ? launch_persistent(batch_kernel<true, 8, false, I8>, sh, st, items, n)
                  : launch_persistent(batch_kernel<false, 8, false, I8>, sh, st, items, n);
    return qc ? launch_persistent(batch_kernel<true, 32, false, I8>, sh, st, items, n)
              : launch_persistent(batch_kernel<false, 32, false, I8>, sh, st, items, n);
}

}  // namespace
}  // namespace tsx
