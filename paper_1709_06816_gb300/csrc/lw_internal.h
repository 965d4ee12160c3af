// lw_internal.h -- declarations shared by the CUDA translation units of liblw.
// Not part of the public C ABI (include/lw.h is).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

struct lw_ctx;

namespace lw {

constexpr int kThreads = 512;            // default threads per CTA of the merge kernel
constexpr int kRowBlock = 32;            // rows per ownership block (one warp)
constexpr int kCacheKeys = 4;            // smallest keys cached per row
constexpr int kPub = 8;                  // entries a CTA of a multi-CTA grid publishes per round
constexpr int kTeam = 64;                // most members (clusters) of a round
constexpr int kSurv = 32;                // most merged clusters a round leaves
constexpr int kEntries = 64;             // most entries a round selects its members from
constexpr int kCand = 512;               // most entries up to a round's pivot
constexpr int kHeadsHi = 64;             // most lists whose heads the pivot takes in
constexpr int kPieces = 4;               // most pieces a refill row is scanned in
constexpr int kPartWords = 8;            // words of a piece: its smallest keys, the bound of the others
constexpr int kSvList = 64;              // places for listed new cells per survivor
constexpr int kRankBits = 4;             // an entry's rank in its row
constexpr unsigned kRankMask = 15u;
constexpr int kBar2 = 32;                // words of the second and third barrier counter and of
constexpr int kBar3 = 48;                // the first conditional merge that must wait (two, by
constexpr int kViol = 8;                 // round parity; kTeam less it, 0: none)
// A chain cut below kRedoBelow merges, and below half its length (and kRedoGap), is
// walked step by step instead.  Never (0) / 16 / always (64), ms: n = 4000, points four
// at a time, complete 59.5 / 17.5 / 17.5; n = 8192 average on a 1/1024 grid 13.9 / 11.9 /
// 11.9; n = 16384 average 27.9 / 24.5 / 24.5; elsewhere within 1 %.
constexpr int kRedoBelow = 16;
constexpr int kRedoGap = 4;
// Merges that a round of the chain must gain to take them on condition: kTieGain, and
// one for every kTiePart that bounds prove (the look costs a barrier that also waits
// for the scans beside it, more so in long rounds).  ms, n = 65536 conformer-like
// complete / n = 4000 integers complete / n = 5000 on a 1/64 grid complete: any 3 merges
// 146.2 / 26.5 / 6.22, any 8 141.7 / 36.5, any 14 141.1 / 39.4; 2 and half of the
// proved ones 141.4 / 24.1 / 6.31, 2 and a quarter 142.1 / 24.0 / 6.22.
constexpr int kTieGain = 2;
constexpr int kTiePart = 4;
// Up to this n a row asks for a refill at one key left; above it at none, and the
// scans start before the selection, in more pieces, with prefetches.  Early saves rounds, late saves scans; ms, early / late: conformer-like, complete,
// n = 8192 9.0 / 9.8, 16384 21.8 / 21.5, 20480 30.2 / 28.2, 24576 40.2 / 34.7, 28000
// 49.8 / 40.9, 65536 234 / 146; on a 1/1024 grid, 20480 complete 30.2 / 31.5, average
// 32.7 / 34.8, single 69.2 / 72.3, 24576 39.8 / 38.0, 41.5 / 41.9, 87.7 / 91.0, 28000
// 48.8 / 44.0, 49.7 / 48.1, 104 / 108.  The line lies where the grids' gain ends;
// continuous distances would have it at 16384.
constexpr long long kRefillEarlyN = 24576;
constexpr int kSurvivorRefillAt = 1;     // the same for a survivor row right after its merge
constexpr int kMaxReq = 256;             // refill requests served per round
constexpr int kReqPerCta = 8;            // refill requests one CTA may make per round
constexpr int kStats = 33;
constexpr uint64_t kNoKey = ~0ull;

// Column word of a published entry: the column, or one of two stop marks.
constexpr unsigned kColMask = 0x3fffffffu;
constexpr unsigned kRowStop = 0x80000000u;   // the row's cache ends here (cells beyond unknown)
constexpr unsigned kHardStop = 0x40000000u;  // the CTA published no entries beyond this one

// ---- the update formula and the bounds of the cells it makes.  Host code too, for
// the test of the bounds: compiled there without contraction of products and sums.
#ifdef __CUDA_ARCH__
#define LW_ON(device, host) device
#else
#define LW_ON(device, host) host
#endif
__host__ __device__ __forceinline__ float mul_rn(float a, float b) { return LW_ON(__fmul_rn(a, b), a * b); }
__host__ __device__ __forceinline__ float add_rn(float a, float b) { return LW_ON(__fadd_rn(a, b), a + b); }
__host__ __device__ __forceinline__ float sub_rn(float a, float b) { return LW_ON(__fsub_rn(a, b), a - b); }
__host__ __device__ __forceinline__ float div_rn(float a, float b) { return LW_ON(__fdiv_rn(a, b), a / b); }
__host__ __device__ __forceinline__ float div_fast(float a, float b) { return LW_ON(__fdividef(a, b), a / b); }
__host__ __device__ __forceinline__ float ll_rn(long long a) { return LW_ON(__ll2float_rn(a), (float)a); }
__host__ __device__ __forceinline__ unsigned bits_of(float a)
{
    unsigned u;
    memcpy(&u, &a, sizeof u);
    return LW_ON(__float_as_uint(a), u);
}
__host__ __device__ __forceinline__ float value_of(unsigned u)
{
    float a;
    memcpy(&a, &u, sizeof a);
    return LW_ON(__uint_as_float(u), a);
}
#undef LW_ON

// The update of Section 4 step 3 from coefficients: the four terms (bh is the
// third) added in printed order, every operation rounded once.
__host__ __device__ __forceinline__ float lw_sum(float ai, float aj, float bh, float ga, float dki, float dkj)
{
    float s = mul_rn(ai, dki);
    s = add_rn(s, mul_rn(aj, dkj));
    s = add_rn(s, bh);
    return add_rn(s, mul_rn(ga, fabsf(sub_rn(dki, dkj))));
}

// Ward's cell (coefficients depend on the third cluster's size fk).
__host__ __device__ __forceinline__ float ward_cell(float fi, float fj, float fs, float fk, float h, float a, float b)
{
    const float T = add_rn(fs, fk);  // (integers below 2^24: exact)
    const float x = div_rn(add_rn(fi, fk), T), y = div_rn(add_rn(fj, fk), T);
    const float z = -div_rn(fk, T);
    return lw_sum(x, y, mul_rn(z, h), 0.0f, a, b);
}

// Table 1 coefficients of a merge of sizes ni, nj at height h: a_i, a_j, b
// times h, g (LK 3, Ward: per cell, see ward_cell).  Centroid: exact integers,
// each converted to float once, one division.
template <int LK>
__host__ __device__ __forceinline__ float4 merge_coefs(int ni, int nj, float h)
{
    float4 co = make_float4(0.5f, 0.5f, mul_rn(0.0f, h), 0.0f);
    if (LK == 0)
        co.w = -0.5f;
    if (LK == 1)
        co.w = 0.5f;
    if (LK == 2 || LK == 5) {
        const float fs = (float)(ni + nj);
        co.x = div_rn((float)ni, fs);
        co.y = div_rn((float)nj, fs);
    }
    if (LK == 5)
        co.z = mul_rn(-div_rn(ll_rn((long long)ni * nj), ll_rn((long long)(ni + nj) * (ni + nj))), h);
    return co;
}

// A lower bound (value bits) of the cells between a merged cluster and others,
// from the bounds la, lb of its two parts' cells (both above the height h): the
// update formula is monotone in both distances, so it is evaluated at the
// bounds, less a margin for its roundings.  Per linkage, rounding errors in
// units of 2^-24: complete: s + |d|/2 >= max(a, b) up to 3 relative, and >=
// min(a, b) without error (rounding is monotone, and so for weighted); single:
// the terms reach the larger distance, 2.5 of the largest value in the matrix;
// weighted: 1 relative; average, centroid: 4 relative; Ward: the weighted mean
// of a and b is a bound for every size of the third cluster (the formula rises
// from it with that size while a, b >= h), at most 12 relative.  The margins
// taken (2e-6 = 33, 8e-6 = 134 units) leave room for the bound's own roundings.
// Values too small for a relative margin, or not finite, give bound 0: the
// round then ends where it would need it.
template <int LK>
__host__ __device__ __forceinline__ unsigned merged_bound(int lab, int lbb, float fi, float fs, float h, unsigned dmax)
{
    const float la = value_of((unsigned)lab), lb = value_of((unsigned)lbb);
    float r;
    if (LK == 0)
        r = fminf(la, lb) - 2.0e-6f * value_of(dmax);
    else if (LK == 1)
        r = fmaxf(fminf(la, lb), fmaxf(la, lb) * (1.0f - 2.0e-6f));
    else if (LK == 4)
        r = fmaxf(fminf(la, lb), (0.5f * la + 0.5f * lb) * (1.0f - 2.0e-6f));
    else {
        const float w = div_fast(fi, fs);
        r = w * la + (1.0f - w) * lb;
        if (LK == 5)
            r = r - w * (1.0f - w) * h;
        r = r * (1.0f - 8.0e-6f);
    }
    if ((lab & lbb) == -1)
        return 0xffffffffu;  // no such cells
    // (a NaN fails both comparisons)
    return r > 1.0e-30f && r < 3.0e38f ? bits_of(r) : 0u;
}

// Status words written by the kernel (values match lw_status).
enum : int { kOk = 0, kErrInput = 2, kErrInternal = 4, kErrTimeout = 5, kErrBounds = 6 };

// Bounds-checked build (-DLW_CHECKED): every global load and store of the
// merge kernel is checked against the job's buffers; one outside them is
// skipped (a load reads zero) and sets the status to kErrBounds with the
// source line in status[2].  For testing: it replaces a memory checker.
constexpr int kCheckRanges = 8;
struct CheckRange {
    const char *base;
    unsigned long long bytes;
};

// One CTA's record at the start of a round: its kPub smallest cache entries
// (key = (bits(value) << 32) | (row << kRankBits) | rank, column word beside
// it), the rows (at most kReqPerCta) that ask for a refill and, in the first
// round, the largest value of its rows.  Two sets, by round parity: a CTA may
// write the next round's while another still reads this one's.
struct __align__(16) RecA {
    unsigned long long key[kPub];
    unsigned int col[kPub];
    int nreq;
    int req[kReqPerCta];
    unsigned dmax;
    int pad[2];
};
static_assert(sizeof(RecA) == kPub * 12 + 48, "record layout");

struct MergeParams {
    float *D;                      // working matrix, rewritten in place: the packed
                                   // upper triangle, or (full = 1) the row-log layout:
                                   // D is an n x n row-major matrix M whose row x is
                                   // current for every column y with stamp[y] <= stamp[x]
    float *TL;                     // full = 1: n x n; TL[x * n + t] = the cell between x
                                   // and the survivor of merge t, written at merge t
    int *stamp;                    // full = 1: [n] merge that last rewrote each slot's
                                   // row (-1: never); cell {x, y} lives in the row of the
                                   // later-stamped slot, and in TL of the other one
    int full;
    long long n;
    long long pitch;               // full = 1: words per row of M and TL (n rounded up
                                   // to a multiple of 4: rows start 16-byte aligned)
    int linkage;                   // Table 1 row: 0 single, 1 complete, 2 group average,
                                   // 3 Ward, 4 weighted average, 5 centroid
    int G;                         // CTAs in the persistent grid
    int aligned16;                 // D is 16-byte aligned (128-bit loads allowed)
    int32_t *merges;               // [2(n-1)] device
    float *heights;                // [n-1]    device
    int *size_g;                   // [n] cluster sizes
    int chunk;                     // rows per chunk of the apply pass (set at launch)
    RecA *recA;                    // [2][G] published entries and refill requests
    unsigned long long *svlist;    // [2][kSurv][kSvList] survivors' new cells below the limit, by
    unsigned long long *svovf;     // round parity, and [2][kSurv] the least that is not listed
    unsigned long long *parts;     // [2][kMaxReq][kPieces][kPartWords] refill lists (top-K of a row's pieces)
    unsigned int *bar;             // grid barrier counters, words 0 and kBar2 (zero at launch)
    int *status;                   // [4] status word [0]; barrier that gave up [1]
    long long *stats;              // [kStats] counters, see lw_get_stats
    unsigned long long timeout_ns; // bound of every device wait
    int skip_arrive_cta;           // failure-detection test: this CTA never reaches the
                                   // first barrier (-1 = off), so the others' bounded
                                   // wait runs out and reports LW_ERR_TIMEOUT
    int timing;                    // accumulate per-phase wall-clock time in stats[8..13]
#ifdef LW_CHECKED
    CheckRange ck[kCheckRanges];   // the job's buffers (checked build only)
    int nck;
#endif
};

// Registers [base, base + bytes) as a buffer the checked kernel may touch
// (no effect in the normal build).
__host__ __device__ inline void check_range(MergeParams &p, const void *base, unsigned long long bytes)
{
#ifdef LW_CHECKED
    if (p.nck < kCheckRanges && base)
        p.ck[p.nck++] = CheckRange{static_cast<const char *>(base), bytes};
#else
    (void)p;
    (void)base;
    (void)bytes;
#endif
}

// Byte offsets of the merge kernel's global scratch inside one workspace
// block (every part 256-byte aligned).  The words from `zero` to `total`
// (barrier, status, stats) must be zero at launch.
struct WorkspaceLayout {
    size_t size, recA, sv, parts, zero, bar, status, stats, total;
};

__host__ __device__ inline WorkspaceLayout workspace_layout(long long n, int G)
{
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    WorkspaceLayout L;
    size_t off = 0;
    L.size = off;   off = up(off + sizeof(int) * (size_t)n);
    L.recA = off;   off = up(off + sizeof(RecA) * 2 * (size_t)G);
    L.sv = off;     off = up(off + 2 * kSurv * (size_t)(8 * (kSvList + 1)));
    L.parts = off;  off = up(off + 8 * kPartWords * (size_t)kMaxReq * kPieces * 2);
    L.zero = off;
    L.bar = off;    off = up(off + 256);
    L.status = off; off = up(off + 4 * sizeof(int));
    L.stats = off;  off = up(off + kStats * sizeof(long long));
    L.total = off;
    return L;
}

// Points p's scratch pointers into a workspace block laid out by L.
__host__ __device__ inline void bind_workspace(MergeParams &p, char *ws, const WorkspaceLayout &L)
{
    p.size_g = reinterpret_cast<int *>(ws + L.size);
    p.recA = reinterpret_cast<RecA *>(ws + L.recA);
    p.svlist = reinterpret_cast<unsigned long long *>(ws + L.sv);
    p.svovf = p.svlist + 2 * kSurv * kSvList;
    p.parts = reinterpret_cast<unsigned long long *>(ws + L.parts);
    p.bar = reinterpret_cast<unsigned int *>(ws + L.bar);
    p.status = reinterpret_cast<int *>(ws + L.status);
#ifdef LW_CHECKED
    p.nck = 0;
#endif
    check_range(p, ws, L.total);
}

// One job of a batch (device table entry).
struct BatchJob {
    float *D;                      // packed upper triangle (device), rewritten in place
    long long n;
    int linkage;
    int pad;
    int32_t *merges;               // [2(n-1)] device
    float *heights;                // [n-1]    device
};

struct BatchParams {
    const BatchJob *jobs;          // [njobs] device
    int njobs;
    long long n_max;               // largest n in the table (sizes shared memory and slots)
    int *queue;                    // next job to take (zero at launch)
    char *ws;                      // one workspace slot per CTA, workspace_layout(n_max, 1)
    int *job_status;               // [njobs] lw_status of each job
    long long *merges_done;        // total merges performed (optional)
    unsigned long long timeout_ns;
    int chunk;                     // rows per chunk of the apply pass (set at launch)
};

// Writes the symmetric n x n matrix `full` (row-major, rows `pitch` words
// apart, diagonal untouched) from the packed upper triangle `packed`, with
// -0 cells as +0; a NaN, infinite or negative cell sets *status to kErrInput.
cudaError_t launch_expand(const float *packed, float *full, long long n, long long pitch, int *status,
                          cudaStream_t stream);

// Row pitch (words) of the row-log layout's n x n matrices.
inline long long log_pitch(long long n) { return (n + 3) & ~3LL; }

// Bytes of dynamic shared memory the merge kernel needs for (n, G) with CTAs
// of nt threads.
int default_grid(long long n, int linkage, int num_sms);
size_t merge_smem_bytes(long long n, int G, int nt);
// Rows per chunk of the apply pass (its new cells are kept in shared memory).
int merge_chunk_rows(long long n, int G, int nt);
// CTA sizes the kernels are built for: 128, 256 or 512 threads (4, 2 or 1
// CTAs per SM by registers; with their static shared memory of some 50 KB a
// one-CTA job leaves room for 3, 2 and 1 at n = 64, for 2, 2 and 1 from 256 to 512
// and for 1 of any size from 1024 on).
// True if a grid of G CTAs of nt threads for n objects fits co-resident on
// the current device.
bool merge_config_ok(long long n, int G, int num_sms, int nt = kThreads);
// Size the context's device workspace for every run of up to n objects, so
// that later runs never allocate (the serving loop reserves its lanes' at
// creation: growing a workspace frees the old one, and cudaFree waits for
// the whole device).  Returns LW_OK or LW_ERR_OOM.
int reserve_workspace(struct ::lw_ctx *ctx, long long n);

// Launch the persistent kernel (CTAs of nt threads) cooperatively on `stream`.
cudaError_t launch_merge(const MergeParams &p, int nt, cudaStream_t stream);
// CTAs of nt threads of the batch kernel that fit on one SM for jobs up to n_max.
int batch_ctas_per_sm(long long n_max, int nt = kThreads);
// Launch the batch kernel (grid CTAs of nt threads, one workspace slot each) on
// `stream`; call batch_ctas_per_sm(bp.n_max, nt) first (it sets the
// shared-memory limit).
cudaError_t launch_batch(const BatchParams &bp, int grid, int nt, cudaStream_t stream);

}  // namespace lw
