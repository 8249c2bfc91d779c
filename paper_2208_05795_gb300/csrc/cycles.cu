// cycles.cu -- short cycles of the Tanner graph on the device: the EMD
// spectrum of Sec. II (Table II) and the per-node cycle counts behind the
// cycle-density iteration budgets of Sec. III (Table V).
//
// A cycle of length 2l is an exponent chain that closes (Prop. 1, eq. 3): a
// closed walk v0 - c1 - v1 - ... - v_{l-1} - c_l - v0 that never steps
// straight back (c_{t+1} != c_t, v_{t+1} != v_t, c_l != c_1), up to rotation
// and reversal; it may pass a node twice.  Walked from a representative v0
// ((j,0) of a QC code, every node of a general code), the column index of
// every node of a QC walk is the running alternating sum of the exponents,
// and the walk closes exactly when that sum is 0 mod Z.  A walk class with
// rotation period p and r = 1 (its reverse is a rotation) or 2 is met p r
// times over the representatives (per circulant orbit, for a QC code); each
// walk adds 2l / (p r) to hist2[l][EMD], so hist2 / (2l) counts classes --
// Table II's "number of cycles without multiplication by graph automorphism".
// For l <= 3 every such walk is a simple cycle: walks from v of length 2l
// are twice the cycles through v.
//
// The EMD is the number of checks meeting exactly one variable node of the
// walk.
//
// lmax <= 3 (load_code()): one thread per two-step prefix.  Longer walks are
// searched from both ends: the last two steps v_{L-2} - c_{L-1} - v_{L-1} -
// c_L - v0 are fixed by where they start and end, so every two-step path into
// a representative is listed once, by its start (pairs_kernel), and a walk of
// L nodes is a prefix of L - 2 steps and a listed path.  The search visits
// prefixes of lmax - 2 steps instead of lmax - 1 steps and a test of every
// closing check: on Code 1 (4 x 20, Z = 128) 4.2e6 prefixes instead of 2.3e8
// for cycles up to length 10.
#include <algorithm>

#include "graph.cuh"
#include "kernels.cuh"

namespace tsx {
namespace {

constexpr int kLmax = kCycLmax;

template <int D>
struct Depth {
    static constexpr int value = D;
};

__device__ __forceinline__ bool has_check(const DevCode &g, int v, int c) {
    const int d = vn_degree(g, v);
    for (int t = 0; t < d; t++)
        if (vn_check(g, v, t) == c) return true;
    return false;
}

// checks meeting exactly one distinct variable node of vs[0..L-1]
__device__ int emd_of(const DevCode &g, const int *vs, int L) {
    int u[kLmax], nu = 0;
    for (int x = 0; x < L; x++) {
        bool dup = false;
        for (int y = 0; y < nu; y++) dup |= u[y] == vs[x];
        if (!dup) u[nu++] = vs[x];
    }
    int emd = 0;
    for (int x = 0; x < nu; x++) {
        const int d = vn_degree(g, u[x]);
        for (int t = 0; t < d; t++) {
            const int c = vn_check(g, u[x], t);
            bool other = false;
            for (int y = 0; y < nu && !other; y++)
                if (y != x) other = has_check(g, u[y], c);
            emd += !other;
        }
    }
    return emd;
}

// p r of the closed walk vs[0..L-1], cs[1..L] (cs[t] joins vs[t-1] and vs[t mod L])
__device__ int walk_reps(const int *vs, const int *cs, int L) {
    int p = L;
    for (int q = 1; q < L; q++) {
        if (L % q) continue;
        bool ok = true;
        for (int t = 0; t < L && ok; t++) ok = vs[(t + q) % L] == vs[t] && cs[(t + q) % L + 1] == cs[t + 1];
        if (ok) {
            p = q;
            break;
        }
    }
    // the reverse rotated by s: v_{(s-t) mod L} followed by c_{(s-t) mod L} (c_0 = c_L)
    int r = 2;
    for (int sft = 0; sft < L && r == 2; sft++) {
        bool ok = true;
        for (int t = 0; t < L && ok; t++) {
            const int a = ((sft - t) % L + L) % L;
            ok = vs[a] == vs[t] && cs[a == 0 ? L : a] == cs[t + 1];
        }
        if (ok) r = 1;
    }
    return p * r;
}

// walks[rep * (kLmax + 1) + l]: closed walks of l variable nodes from the
// representative; hist2[l * kEmdBins + e]: sum of 2l / (p r) over them by EMD.
// Thread id = (rep, t_1, p_1, t_2, p_2): the walk's first two steps (check t of
// the last node, then node p of that check); the walks that close at the first
// are counted by the thread whose deeper indices are 0.
__global__ void __launch_bounds__(256) short_kernel(DevCode g, int lmax, long long n_prefix, unsigned long long *walks,
                                                    unsigned long long *hist2) {
    const int dvm = g.dv_max, dcm = g.dc_max;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n_prefix;
         id += (long long)gridDim.x * blockDim.x) {
        long long x = id;
        int tt[3], pp[3];
        for (int lvl = 2; lvl >= 1; lvl--) {
            pp[lvl] = (int)(x % dcm);
            x /= dcm;
            tt[lvl] = (int)(x % dvm);
            x /= dvm;
        }
        const int rep = (int)x;
        int vs[kLmax], cs[kLmax + 1];
        vs[0] = rep_vn(g, rep);
        unsigned long long cnt[4] = {0, 0, 0, 0};
        for (int lvl = 1; lvl <= 2; lvl++) {
            const int v = vs[lvl - 1];
            if (tt[lvl] >= vn_degree(g, v)) break;
            const int c = vn_check(g, v, tt[lvl]);
            if (lvl > 1 && c == cs[lvl - 1]) break;
            if (pp[lvl] >= cn_degree(g, c)) break;
            const int u = cn_vn(g, c, pp[lvl]);
            if (u == v) break;
            cs[lvl] = c;
            vs[lvl] = u;
            if (lvl == 1 && (tt[2] || pp[2])) continue;
            // the walks that close here, through a check of u holding v0
            if (lvl < lmax && u != vs[0]) {
                const int dv = vn_degree(g, u);
                for (int t = 0; t < dv; t++) {
                    const int cl = vn_check(g, u, t);
                    if (cl == c || cl == cs[1] || !has_check(g, vs[0], cl)) continue;
                    const int L = lvl + 1;
                    cs[L] = cl;
                    cnt[L]++;
                    if (hist2)
                        atomicAdd(&hist2[L * kEmdBins + emd_of(g, vs, L)],
                                  (unsigned long long)(2 * L / walk_reps(vs, cs, L)));
                }
            }
        }
        for (int L = 2; L <= lmax; L++)
            if (cnt[L]) atomicAdd(&walks[rep * (kLmax + 1) + L], cnt[L]);
    }
}

// ---------------------------------------------------------------------------
// lmax >= 4: prefixes and listed two-step paths
// ---------------------------------------------------------------------------
constexpr unsigned short kNone = 0xFFFFu;

// Adjacency of the code as rows of 16-bit ids (kNone: no such edge): vadj
// [n][dvp], dvp = dv_max filled up to a multiple of 4, and cadj [m][dc_max].
// by_block (QC, m_b <= dvp): a node's check of row block i is entry i, so that two
// nodes' common checks are in the same entry of both rows.
__global__ void adj_kernel(DevCode g, int dvp, int by_block, unsigned short *vadj, unsigned short *cadj) {
    const long long nv = (long long)g.n * dvp, nc = (long long)g.m * g.dc_max;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nv + nc;
         i += (long long)gridDim.x * blockDim.x) {
        if (i < nv) {
            const int v = (int)(i / dvp), t = (int)(i - (long long)v * dvp);
            int x = t < vn_degree(g, v) ? vn_check(g, v, t) : kNone;
            if (by_block) {
                x = kNone;
                for (int q = 0; q < vn_degree(g, v); q++) {
                    const int c = vn_check(g, v, q);
                    if (c / g.Z == t) x = c;
                }
            }
            vadj[i] = (unsigned short)x;
        } else {
            const int c = (int)((i - nv) / g.dc_max), p = (int)((i - nv) - (long long)c * g.dc_max);
            cadj[i - nv] = p < cn_degree(g, c) ? (unsigned short)cn_vn(g, c, p) : kNone;
        }
    }
}

struct Paths {
    DevCode g;
    int dvp, td;                  // row length of vadj, and its entries that may hold a check
    int alone;                    // the walk kernel has by_block rows: a bucket a node, w not stored
    int rep0, nrep;               // representatives of this launch
    const unsigned short *vadj, *cadj;
    // [nrep][nb + 1]: paths of rep0 + r that start at a node w of bucket k = w & mask: ent[off[k] .. off[k + 1])
    unsigned *off;
    int nb, mask;                 // buckets (see launch_cycles)
    uint2 *ent;                   // [nrep][per]: {u | c' << 16, c | w << 16 (alone: c)} of a path w - c - u - c' - v0
    long long per;                // room per representative
};

// One block per representative: the two-step paths w - c - u - c' - v0 with
// u != v0, c != c', w != u (w may be v0), sorted by w's bucket: counted, scanned
// and placed by counters in off.
__global__ void __launch_bounds__(512) pairs_kernel(Paths a) {
    const int r = blockIdx.x, nb = a.nb, dvp = a.dvp, td = a.td, dc = a.g.dc_max;
    const int v0 = rep_vn(a.g, a.rep0 + r);
    unsigned *off = a.off + (long long)r * (nb + 1);
    uint2 *ent = a.ent + (long long)r * a.per;
    for (int w = threadIdx.x; w <= nb; w += blockDim.x) off[w] = 0;
    __syncthreads();
    const int total = td * dc * td * dc;
    auto each = [&](auto f) {
        for (int i = threadIdx.x; i < total; i += blockDim.x) {
            int x = i;
            const int p2 = x % dc;
            x /= dc;
            const int t2 = x % td;
            x /= td;
            const int p1 = x % dc, t1 = x / dc;
            const int c1 = a.vadj[(long long)v0 * dvp + t1];
            if (c1 == kNone) continue;
            const int u = a.cadj[(long long)c1 * dc + p1];
            if (u == kNone || u == v0) continue;
            const int c = a.vadj[(long long)u * dvp + t2];
            if (c == kNone || c == c1) continue;
            const int w = a.cadj[(long long)c * dc + p2];
            if (w == kNone || w == u) continue;
            f(w, u, c1, c);
        }
    };
    each([&](int w, int, int, int) { atomicAdd(&off[(w & a.mask) + 1], 1u); });
    __syncthreads();
    // inclusive scan of off[1 .. nb] in blocks of blockDim
    __shared__ unsigned wsum[16];
    __shared__ unsigned carry;
    if (threadIdx.x == 0) carry = 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int base = 1; base <= nb; base += blockDim.x) {
        __syncthreads();
        const int i = base + threadIdx.x;
        unsigned v = i <= nb ? off[i] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane == 31) wsum[wid] = v;
        __syncthreads();
        unsigned add = carry;
        for (int k = 0; k < wid; k++) add += wsum[k];
        v += add;
        if (i <= nb) off[i] = v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = v;
    }
    __syncthreads();
    // off[w] is the start of w; placing advances it to the end, which is the start of w + 1: shift back
    each([&](int w, int u, int c1, int c) {
        ent[atomicAdd(&off[w & a.mask], 1u)] =
            make_uint2((unsigned)u | ((unsigned)c1 << 16), a.alone ? (unsigned)c : (unsigned)c | ((unsigned)w << 16));
    });
    __syncthreads();
    for (int base = ((nb + blockDim.x) / blockDim.x) * blockDim.x; base >= 0; base -= blockDim.x) {
        const int w = base + threadIdx.x;
        const unsigned x = w >= 1 && w <= nb ? off[w - 1] : 0u;
        __syncthreads();
        if (w <= nb) off[w] = x;
        __syncthreads();
    }
}

// checks meeting exactly one of the L distinct nodes vs[0..L-1], whose rows of
// vadj are compared pair by pair (BLK: by_block rows, the same entries only)
template <int L, int DVP, bool BLK>
__device__ __forceinline__ int emd_distinct(const unsigned short *vadj, const int *vs) {
    unsigned short ch[L][DVP];
#pragma unroll
    for (int x = 0; x < L; x++)
#pragma unroll
        for (int q = 0; q < DVP / 4; q++) *(uint2 *)&ch[x][4 * q] = __ldg((const uint2 *)(vadj + (long long)vs[x] * DVP) + q);
    int emd = 0;
#pragma unroll
    for (int x = 0; x < L; x++)
#pragma unroll
        for (int t = 0; t < DVP; t++) {
            bool other = ch[x][t] == kNone;
#pragma unroll
            for (int y = 0; y < L; y++)
                if (y != x)
#pragma unroll
                    for (int q = 0; q < DVP; q++)
                        if (!BLK || q == t) other |= ch[y][q] == ch[x][t];
            emd += !other;
        }
    return emd;
}

// One thread per prefix of PD steps (PD = LMAX - 2, or LMAX - 3 where that is
// already enough threads); it counts the walks that close two steps after
// its last node (and, PD = LMAX - 3, after each node one step further), and
// those of the shorter prefixes whose deeper indices are 0.  WARP: the lanes of
// a warp share what follows each of their prefixes.
// (four CTAs an SM: 64 registers; left to itself the compiler takes 80 in some forms, 7 % slower)
template <int LMAX, int PD, int DVP, bool BLK, bool WARP>
__global__ void __launch_bounds__(256, 4) walk_kernel(Paths a, long long n_prefix, int share, unsigned long long *walks,
                                                   unsigned long long *hist2) {
    // the CTA's histogram and walk counts, low words and carries
    __shared__ unsigned hs[(kLmax + 1) * kEmdBins], hc[(kLmax + 1) * kEmdBins], ws[kLmax + 1], wc[kLmax + 1];
    for (int i = threadIdx.x; i < (kLmax + 1) * kEmdBins; i += blockDim.x) hs[i] = hc[i] = 0;
    if (threadIdx.x <= kLmax) ws[threadIdx.x] = wc[threadIdx.x] = 0;
    __syncthreads();
    auto add = [](unsigned *lo, unsigned *hi, unsigned x) {
        const unsigned old = atomicAdd(lo, x);
        if (old + x < old) atomicAdd(hi, 1u);
    };
    const int dvp = a.dvp, td = a.td, dc = a.g.dc_max;
    const int lane = threadIdx.x & 31;
    // WARP: the first `share` lanes of a warp take a prefix each, far apart (next to each other they have
    // the same representative, and the walks of a node of large degree would be one warp's)
    const long long threads = (long long)gridDim.x * blockDim.x, warps = threads / 32;
    const long long thread = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (long long base = WARP ? thread / 32 : thread; base < n_prefix; base += WARP ? share * warps : threads) {
        const long long id = WARP ? base + lane * warps : base;
        const bool mine = !WARP || (lane < share && id < n_prefix);
        long long x = mine ? id : 0;
        int tt[PD + 1], pp[PD + 1];
#pragma unroll
        for (int l = PD; l >= 1; l--) {
            pp[l] = (int)(x % dc);
            x /= dc;
            tt[l] = (int)(x % td);
            x /= td;
        }
        const int r = (int)x;
        const unsigned *off = a.off + (long long)r * (a.nb + 1);
        const uint2 *ent = a.ent + (long long)r * a.per;
        int vs[kLmax], cs[kLmax + 1];
        vs[0] = rep_vn(a.g, a.rep0 + r);
        unsigned cnt[LMAX + 1] = {};
        // the walks of D + 2 nodes that continue v_D with a listed path: every step-th from the first on
        auto close = [&](auto depth, int first, int step) {
            constexpr int D = decltype(depth)::value, L = D + 2;
            const int k = BLK ? vs[D] : vs[D] & a.mask;  // (by_block rows: QC, a bucket a node)
            const unsigned e1 = __ldg(off + k + 1);
            for (unsigned e = __ldg(off + k) + first; e < e1; e += step) {
                const uint2 q = __ldg(ent + e);
                if (!BLK && (int)(q.y >> 16) != vs[D]) continue;
                const int u = (int)(q.x & 0xFFFFu), cl = (int)(q.x >> 16), c = BLK ? (int)q.y : (int)(q.y & 0xFFFFu);
                if constexpr (D > 0)
                    if (c == cs[D] || cl == cs[1]) continue;
                vs[D + 1] = u;
                cs[D + 1] = c;
                cs[L] = cl;
                cnt[L]++;
                if (!hist2) continue;
                bool distinct = true;
#pragma unroll
                for (int i = 0; i < L; i++)
#pragma unroll
                    for (int k = i + 1; k < L; k++) distinct = distinct && vs[i] != vs[k];
                // all nodes distinct: no rotation and no reversal gives the same walk, weight 2L / (2L)
                int emd, wt = 1;
                bool fast = false;
                if constexpr (DVP <= 4) fast = distinct;
                if (fast) {
                    if constexpr (DVP <= 4) emd = emd_distinct<L, DVP, BLK>(a.vadj, vs);
                } else {
                    emd = emd_of(a.g, vs, L);
                    if (!distinct) wt = 2 * L / walk_reps(vs, cs, L);
                }
                add(&hs[L * kEmdBins + emd], &hc[L * kEmdBins + emd], (unsigned)wt);
            }
        };
        bool ok = mine;
        // counted once: by the thread whose remaining indices are 0
        auto zero_from = [&](int l0) {
            bool z = true;
#pragma unroll
            for (int l = 1; l <= PD; l++)
                if (l >= l0) z = z && tt[l] == 0 && pp[l] == 0;
            return z;
        };
        if (ok && zero_from(1)) close(Depth<0>{}, 0, 1);
#pragma unroll
        for (int l = 1; l <= PD; l++) {
            if (!ok) break;
            const int c = a.vadj[(long long)vs[l - 1] * dvp + tt[l]];
            ok = c != kNone && (l == 1 || c != cs[l > 1 ? l - 1 : 1]);
            if (!ok) break;
            const int u = a.cadj[(long long)c * dc + pp[l]];
            ok = u != kNone && u != vs[l - 1];
            if (!ok) break;
            cs[l] = c;
            vs[l] = u;
            if (l == 1 && PD > 1 && zero_from(2)) close(Depth<1>{}, 0, 1);
            if constexpr (PD > 2)
                if (l == 2 && zero_from(3)) close(Depth<2>{}, 0, 1);
            if constexpr (PD > 3)
                if (l == 3 && zero_from(4)) close(Depth<3>{}, 0, 1);
        }
        if constexpr (WARP) {
            static_assert(PD == LMAX - 3, "one step further");
            int mv[PD + 1], mc[PD + 1];
#pragma unroll
            for (int l = 0; l <= PD; l++) {
                mv[l] = vs[l];
                mc[l] = l ? cs[l] : 0;
            }
            for (unsigned todo = __ballot_sync(0xffffffffu, ok); todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                const int rs = __shfl_sync(0xffffffffu, r, src);
                off = a.off + (long long)rs * (a.nb + 1);
                ent = a.ent + (long long)rs * a.per;
#pragma unroll
                for (int l = 0; l <= PD; l++) {
                    vs[l] = __shfl_sync(0xffffffffu, mv[l], src);
                    cs[l] = __shfl_sync(0xffffffffu, mc[l], src);
                }
                close(Depth<PD>{}, lane, 32);
                for (int x = lane; x < td * dc; x += 32) {
                    const int t = x / dc, p = x - t * dc;
                    const int c = a.vadj[(long long)vs[PD] * dvp + t];
                    if (c == kNone || c == cs[PD]) continue;
                    const int u = a.cadj[(long long)c * dc + p];
                    if (u == kNone || u == vs[PD]) continue;
                    cs[PD + 1] = c;
                    vs[PD + 1] = u;
                    close(Depth<PD + 1>{}, 0, 1);
                }
                __syncwarp();
            }
        } else if (ok) {
            close(Depth<PD>{}, 0, 1);
            if constexpr (PD < LMAX - 2) {
                // one step further, node by node
                for (int t = 0; t < td; t++) {
                    const int c = a.vadj[(long long)vs[PD] * dvp + t];
                    if (c == kNone || c == cs[PD]) continue;
                    for (int p = 0; p < dc; p++) {
                        const int u = a.cadj[(long long)c * dc + p];
                        if (u == kNone || u == vs[PD]) continue;
                        cs[PD + 1] = c;
                        vs[PD + 1] = u;
                        close(Depth<PD + 1>{}, 0, 1);
                    }
                }
            }
        }
#pragma unroll
        for (int L = 2; L <= LMAX; L++)
            if (cnt[L]) add(&ws[L], &wc[L], cnt[L]);
    }
    __syncthreads();
    // (walks: summed over the representatives, in the row of the launch's first)
    if (threadIdx.x <= LMAX && (ws[threadIdx.x] || wc[threadIdx.x]))
        atomicAdd(&walks[(long long)a.rep0 * (kLmax + 1) + threadIdx.x],
                  ((unsigned long long)wc[threadIdx.x] << 32) + ws[threadIdx.x]);
    if (hist2)
        for (int i = threadIdx.x; i < (kLmax + 1) * kEmdBins; i += blockDim.x)
            if (hs[i] || hc[i]) atomicAdd(&hist2[i], ((unsigned long long)hc[i] << 32) + hs[i]);
}

template <int LMAX, int DVP, bool BLK>
cudaError_t launch_walk(const Paths &a, long long steps, unsigned long long *walks, unsigned long long *hist,
                        int num_sms, cudaStream_t st) {
    // Prefixes of LMAX - 2 steps while they are few, else of one step less with the last step looped over
    // (no id is decoded, and no prefix walked, for each of a check's nodes).  Variable degrees above 4: often
    // uneven, so that a few prefixes have most of the walks, and the EMD of a walk takes long: a warp shares
    // what follows its prefixes then (general code of 1,500 nodes, rows of 2 to 12, walks of 4 nodes:
    // 14.4 -> 2.6 ms; 300 nodes: 86 -> 8.7; 5 x 12 blocks, Z = 60, walks of 5 nodes: 17.4 -> 4.8).
    long long full = a.nrep, less = a.nrep;
    for (int l = 0; l < LMAX - 2; l++) full *= steps;
    for (int l = 0; l < LMAX - 3; l++) less *= steps;
    const bool loop = less >= 32LL * 1024;
    constexpr bool kWarp = DVP > 4;
    const long long np = loop ? less : full, most = (long long)num_sms * 64;
    if (loop) {
        // as many prefixes to a warp as leave every SM enough warps
        const int share = !kWarp ? 1 : (int)std::min<long long>(32, (np + 8 * most - 1) / (8 * most));
        const long long threads = kWarp ? (np + share - 1) / share * 32 : np;
        walk_kernel<LMAX, LMAX - 3, DVP, BLK, kWarp>
            <<<(int)std::min((threads + 255) / 256, most), 256, 0, st>>>(a, np, share, walks, hist);
    } else {
        walk_kernel<LMAX, LMAX - 2, DVP, BLK, false>
            <<<(int)std::min((np + 255) / 256, most), 256, 0, st>>>(a, np, 1, walks, hist);
    }
    return cudaGetLastError();
}

}  // namespace

// Closed walks per representative and length (walks[n_rep][kLmax + 1]; for
// lmax > 3 only their sums over the representatives are there) and,
// if hist is not null, the class-weighted counts per length and EMD
// (hist[kLmax + 1][kEmdBins]); both zeroed here.
cudaError_t launch_cycles(const DevCode &g, int lmax, unsigned long long *walks, unsigned long long *hist,
                          int num_sms, cudaStream_t st) {
    if (lmax < 2 || lmax > kLmax) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(walks, 0, sizeof(unsigned long long) * g.n_rep * (kLmax + 1), st);
    if (e != cudaSuccess) return e;
    if (hist && (e = cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * (kLmax + 1) * kEmdBins, st)) !=
                    cudaSuccess)
        return e;
    if (lmax <= 3) {
        long long n_prefix = g.n_rep;
        for (int l = 0; l < 2; l++) n_prefix *= (long long)g.dv_max * g.dc_max;
        long long blocks = (n_prefix + 255) / 256;
        if (blocks > 1 << 20) blocks = 1 << 20;
        short_kernel<<<(int)blocks, 256, 0, st>>>(g, lmax, n_prefix, walks, hist);
        return cudaGetLastError();
    }
    // working memory: adjacency rows, and the listed paths of as many representatives at a time as
    // fit about 64 MB
    Paths a{};
    a.g = g;
    a.dvp = (g.dv_max + 3) / 4 * 4;
    a.per = (long long)g.dv_max * (g.dc_max - 1) * std::max(1, g.dv_max - 1) * (g.dc_max - 1);
    if (a.per < 1) a.per = 1;
    // Buckets: one a node (so that none holds two), or about three times as many as a representative has
    // paths on average where that is less -- a general code has as many representatives as nodes, and
    // zeroing, scanning and shifting n words for each was most of the call ((3,6) code of 20,000 nodes,
    // walks of 4 nodes: 3.0 -> 0.47 ms; 32,000 nodes: 6.7 -> 0.55).
    const double avg = (double)g.E / g.n * g.E / g.m * g.E / g.n * g.E / g.m;
    a.nb = g.n;
    a.mask = 0xFFFF;
    for (int k = 64; g.kind == TSX_CODE_CSR && k < g.n; k *= 2)
        if (k >= 3.0 * avg) {
            a.nb = k;
            a.mask = k - 1;
            break;
        }
    const long long per_rep = 4LL * (a.nb + 1) + 8 * a.per;
    long long chunk = (64LL << 20) / per_rep;
    if (chunk < 1) chunk = 1;
    if (chunk > g.n_rep) chunk = g.n_rep;
    auto r256 = [](long long x) { return (x + 255) / 256 * 256; };
    const long long b_vadj = r256(2LL * g.n * a.dvp), b_cadj = r256(2LL * g.m * g.dc_max),
                    b_off = r256(4LL * chunk * (a.nb + 1)), b_ent = r256(8LL * chunk * a.per);
    unsigned char *buf = nullptr;
    if ((e = pool_alloc((void **)&buf, (size_t)(b_vadj + b_cadj + b_off + b_ent), st)) != cudaSuccess) return e;
    a.vadj = (unsigned short *)buf;
    a.cadj = (unsigned short *)(buf + b_vadj);
    a.off = (unsigned *)(buf + b_vadj + b_cadj);
    a.ent = (uint2 *)(buf + b_vadj + b_cadj + b_off);
    const long long na = (long long)g.n * a.dvp + (long long)g.m * g.dc_max;
    const bool blk = g.kind == TSX_CODE_QC && g.m_b <= a.dvp;
    a.td = blk ? g.m_b : g.dv_max;
    a.alone = blk && a.dvp <= 4;
    adj_kernel<<<(int)std::min<long long>((na + 255) / 256, 4096), 256, 0, st>>>(
        g, a.dvp, blk ? 1 : 0, (unsigned short *)a.vadj, (unsigned short *)a.cadj);
    e = cudaGetLastError();
    const long long steps = (long long)a.td * g.dc_max;
    for (int r0 = 0; r0 < g.n_rep && e == cudaSuccess; r0 += (int)chunk) {
        a.rep0 = r0;
        a.nrep = (int)std::min<long long>(chunk, g.n_rep - r0);
        pairs_kernel<<<a.nrep, 512, 0, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        auto go = [&](auto l) {
            constexpr int LM = decltype(l)::value;
            if (a.dvp > 4) return launch_walk<LM, 16, false>(a, steps, walks, hist, num_sms, st);
            return blk ? launch_walk<LM, 4, true>(a, steps, walks, hist, num_sms, st)
                       : launch_walk<LM, 4, false>(a, steps, walks, hist, num_sms, st);
        };
        e = lmax == 4 ? go(Depth<4>{}) : lmax == 5 ? go(Depth<5>{}) : go(Depth<6>{});
    }
    cudaFreeAsync(buf, st);
    return e;
}

}  // namespace tsx
