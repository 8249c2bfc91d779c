// kernels.cuh -- launch interfaces of the library's kernels (host side).
#pragma once
#include "tsx_internal.cuh"

namespace tsx {

// ---- candidate generation (cand.cu) -------------------------------------
struct CandArgs {
    DevCode code;
    int max_size;
    const long long *raw_off;  // [n_rep + 1] raw-set offsets per representative
    long long raw_total;
    int *chunk_count;          // [n_chunks]
    const long long *chunk_off;  // [n_chunks + 1]
    int4 *cands;
    Counters *ctr;
};

struct CycleArgs {
    DevCode code;
    int l;              // VNs per cycle
    long long paths;    // path-index space per representative
    int *count;         // [n_rep]
    const long long *off;  // [n_rep + 1] (absolute positions in cands)
    int4 *cands;
    Counters *ctr;
};

cudaError_t launch_ball(const DevCode &g, int *sizes, const int64_t *ptr, int32_t *ball, bool write,
                        cudaStream_t st);
cudaError_t launch_cand_ball(const CandArgs &a, long long n_chunks, bool write, cudaStream_t st);
cudaError_t launch_cand_cycle(const CycleArgs &a, bool write, cudaStream_t st);
// Exclusive scan of n counts into off[0..n], starting at *base (0 if
// null); with add_total the grand total becomes the candidate count.
cudaError_t launch_scan(const int *cnt, long long n, long long *off, const long long *base, Counters *ctr,
                        bool add_total, cudaStream_t st);
long long cand_chunks(long long raw_total);
// Per-candidate iteration limits of the cycle-density budget for the first
// min(bound, candidate count) candidates.
cudaError_t launch_budget(const int4 *cands, long long bound, const int *vweight, int K, int kmin, int wref,
                          uint16_t *cand_K, const Counters *ctr, cudaStream_t st);

// ---- impulse decoding, bisection, extraction, dedupe (decode.cu) --------
struct SlotLayout {
    int tables_bytes;  // shared code tables at the start of the CTA's shared memory
    int r_off, p_off, xa_off, xb_off, misc_off;  // offsets inside a slot
    int slot_bytes;
};

struct LaunchShape {
    int G;           // warps per codeword group
    int groups;      // groups per CTA
    int ctas;        // grid size (persistent), recomputed from the occupancy at launch
    int num_sms;
    int per_sm_req;  // requested CTAs per SM (0 = as many as are resident)
    int smem_bytes;  // dynamic shared memory per CTA
    SlotLayout lay;
};

// One code of a multi-code decode launch.
struct BatchItem {
    DevCode g;
    DecodeParams dp;
    EnumBuffers b;
    SlotLayout lay;
    int G, groups;
    int scalar;  // 1: not in the multi-code launch (its pair layout does not fit a CTA)
};

// All items of a multi-code launch, passed by value as one kernel parameter
// (kernel parameters may take up to 32 KB).
constexpr int kMaxBatch = 64;

// Warps per CTA of the two-codeword kernels (their launch bounds).  Measured
// on the decode stage, fewer registers against more warps in flight:
//   check-regular codes of degree 6: 20 warps (96 registers): 92 ms on a general
//     (1008, 504) code against 95 with 24 warps and 108 with 16
//   degree 7 or 8: 16 warps (20: 4 B spilled, 0.19 -> 0.23 ms on a small job)
//   degree 9 to 32: 24 warps: the n = 11,520 code, one pair to a CTA, 57 ms
//     against 64 with 20 (two checks a thread instead of three); the others within 3 %
__host__ __device__ constexpr int pair_kernel_warps(int dc, bool exact) {
    return dc == 6 && exact ? 20 : dc <= 8 ? 16 : 24;
}
// the one-codeword kernel (the sum-product decoder's codes of small degree: see enum_kernel)
__host__ __device__ constexpr int scalar_warps(bool is_float, int dc) { return is_float && dc <= 8 ? 24 : 16; }
// the multi-code kernel (24: spills, no faster)
constexpr int kBatchWarps = 20;
// the importance-sampling kernel's large-degree form, one sample pair to a CTA on the n = 8,832
// code: 24 warps 43.2 ms for 200,000 samples, 20: 44.1, 18: 46.2, 16: 48.3
constexpr int kIsWarps = 24;
// its groups' shared scratch, and the room for the noise on the set's nodes (isfer.cu)
constexpr int kIsMiscBytes = 320, kIsNoiseBytes = 512;
// warps in a group, at most (the 32-warp form of the sum-product kernel has groups of one)
constexpr int kMaxGroupWarps = 24;
static_assert(pair_kernel_warps(32, false) <= kMaxGroupWarps && pair_kernel_warps(6, true) <= kMaxGroupWarps &&
              scalar_warps(true, 8) <= kMaxGroupWarps && kBatchWarps <= kMaxGroupWarps && kIsWarps <= kMaxGroupWarps,
              "the groups' reduction scratch");
struct BatchArgs {
    BatchItem it[kMaxBatch];
};
static_assert(sizeof(BatchArgs) + 64 <= 32764, "batch kernel parameters above 32 KB");

// Plans a multi-code launch of the two-codewords-per-lane kernel (fills
// items[] on the host and the common shape over the items that take part);
// a code whose pair layout does not fit a CTA's shared memory gets
// scalar = 1 and is left to a launch of its own.  False if the codes cannot
// share one kernel (kind, decoder or 16-bit bounds differ).
bool plan_batch(const DevCode *const *g, const DecodeParams *dp, const EnumBuffers *b, const int *G_req, int n,
                int num_sms, BatchItem *items, LaunchShape *common, int *variant);
// Launches it over the device copy of items[].
cudaError_t launch_batch(const BatchArgs &items, int n, int variant, const LaunchShape &sh, cudaStream_t st);

// Runs the impulse decodes with bisection over the candidates of b and
// writes the per-candidate records and x* of failing candidates.  NMS
// decoders use the two-codeword kernel where its 16-bit bias bounds hold
// (else, or with force_scalar, the one-codeword kernel).  G / groups /
// ctas_per_sm: 0 = automatic.  n_cand: at most this many candidates are
// decoded (0 = not known): few candidates get wide groups.
cudaError_t launch_decode(const DevCode &g, const DecodeParams &dp, const EnumBuffers &b, int G, int groups,
                          int ctas_per_sm, int num_sms, int force_scalar, long long n_cand, cudaStream_t st);

// Sieve (Tree / TS), classification, canonical key and hash insert of every
// failing candidate (reads the records and x* written by the decoder).
cudaError_t launch_sieve(const DevCode &g, const EnumBuffers &b, int decoder, int num_sms, cudaStream_t st);

// Shape of the importance-sampling kernel (two samples per lane) and the form
// of the code's tables and rows (g.by_rows, g.row_odd), and whether the noise on
// the set's nodes is kept; false if the 16-bit bias bounds or the
// shared memory do not allow it.
bool plan_is_shape(DevCode &g, const DecodeParams &dp, LaunchShape *sh, int num_sms, bool *noise);

// Whether one codeword of g fits the shared memory of a CTA.
bool decode_fits(const DevCode &g, int decoder);

// ---- the ordered list of Sec. III (list.cu) --------------------------------
// Whether one group's list-mode slot fits a CTA for iteration limit K.
bool list_fits(const DevCode &g, int K);
// The second stage over the failing candidates of b (after the decode):
// replay at the threshold, sieve every x_k from kstart (0: floor(girth/2),
// -1: ceil of the first stage's average converged iterations), insert.
cudaError_t launch_list(const DevCode &g, const DecodeParams &dp, const EnumBuffers &b, int kstart, int num_sms,
                        cudaStream_t st);

// ---- short cycles (cycles.cu) ------------------------------------------------
constexpr int kCycLmax = 6;     // variable nodes per cycle at most
constexpr int kEmdBins = 128;   // EMD values per length
// Closed walks from the representatives, per representative and number of
// variable nodes (walks[n_rep][kCycLmax + 1]) and, with hist, per number of
// variable nodes and EMD (hist[kCycLmax + 1][kEmdBins]); zeroed first.
// lmax > 3: walks holds only the sums over the representatives, spread over the
// rows; takes working memory (about 64 MB at most) from the stream's pool.
cudaError_t launch_cycles(const DevCode &g, int lmax, unsigned long long *walks, unsigned long long *hist,
                          int num_sms, cudaStream_t st);

// device working memory from the library's pool on the current device (api.cu); freed with cudaFreeAsync
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s);

// accessors of a loaded code (api.cu)
const DevCode *code_dev(const tsx_code *c);
int code_num_sms(const tsx_code *c);
int code_device(const tsx_code *c);
// validates enumeration parameters and extracts the decoder's part
int enum_params_to_decode(const tsx_enum_params *p, DecodeParams *dp);

// Compacts the hash table: assigns each stored trapping set an index,
// writes its pool offset / count / min threshold, and rewrites the
// candidates' slots as indices.
cudaError_t launch_compact(const EnumBuffers &b, long long n_rec, int *ts_off, int *ts_count,
                           int *ts_thr, int *slot_map, cudaStream_t st);

// ---- serving runtime hooks ------------------------------------------------
// enumeration lists (api.cu): device bytes and candidate bound of a list, start (allocate and
// enqueue everything), finish (after the stream passed: results to the host,
// device memory back), delete.  dchunk > 0 splits the decode into launches of
// dchunk candidates; grid_sms > 0 caps the persistent grids at that many SMs.
int list_bytes(tsx_code *code, const tsx_enum_params *params, long long dchunk, long long *bytes,
               long long *cand_bound);
int list_start(tsx_code *code, const tsx_enum_params *params, cudaStream_t s, long long dchunk, int grid_sms,
               tsx_ts_list **out);
long long list_cand_bound(const tsx_ts_list *L);
int list_finish(tsx_ts_list *L);
void list_delete(tsx_ts_list *L);

// importance-sampling jobs (isfer.cu), the same protocol; chunk > 0 splits
// the samples into launches of chunk samples (results do not change).
struct IsJob;
int is_job_bytes(tsx_code *code, const int32_t *ts_vars, int32_t a, const tsx_is_params *p, long long chunk,
                 long long *bytes);
int is_job_start(tsx_code *code, const int32_t *ts_vars, int32_t a, const tsx_is_params *p, cudaStream_t s,
                 long long chunk, int grid_sms, IsJob **out);
int is_job_finish(IsJob *J, tsx_is_result *out, uint8_t *fail_out, double *logw_out);
void is_job_delete(IsJob *J);

}  // namespace tsx
