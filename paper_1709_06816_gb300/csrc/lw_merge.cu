// lw_merge.cu -- the persistent cooperative Lance-Williams merge kernel.
//
// One launch performs all n - 1 merges of one matrix (Section 4, "Lance-William
// Algorithm", steps 1-4) so that no merge pays a kernel launch.  The paper
// spreads the packed upper triangle over MPI processes and exchanges local
// minima and (i, j, distance) triples by messages (Section 5.3 steps 1-6b); on
// one GB300 the whole triangle sits in HBM, so the "processors" become CTAs,
// the broadcast of local minima becomes a small record per CTA read after a
// grid barrier, and the triple exchange disappears: every CTA addresses rows
// and columns i and j directly.
//
// Work split.  Rows are dealt to CTAs in blocks of 32 consecutive rows,
// round-robin (block q -> CTA q mod G); a CTA "owns" those rows.  The owner
// of row k keeps, in shared memory, the kCacheKeys smallest keys of row k
// (key = (value bits << 32) | column, over live columns c > k) and a bound B:
// every live cell of the row outside the cache has a key above B (B = "none"
// when the cache holds every live cell of the row).
//
// Rounds.  A grid barrier costs about a microsecond on GB300, and a merge by
// itself less, so a round takes as many consecutive merges of the sequential
// iteration as it can prove from one exchange (up to 63, into at most 32 merged
// clusters).  The merges are
// exactly those of the step-by-step algorithm (same pairs, same order, same
// rounded values); only the bookkeeping differs.  One round:
//
//   publish  every CTA publishes its kPub smallest entries: cached keys of its
//      rows, and at the end of a row's list a mark at its bound B.  (A job's
//      only CTA uses its caches directly.)  Barrier 1.
//   selection  every CTA reads all entries, takes the smallest in (value, row,
//      column) order, and makes the rows and columns they name the round's
//      members (at most kTeam): until the next entry would be one member too
//      many, or is a mark of a row without a member, or the last one of a CTA
//      that may have more.  Every cell between live slots that is not among the
//      entries taken is at or above the first entry not taken, TH, or, in a
//      member's row that ended in a mark, at or above that mark.
//   gather  every CTA reads all cells between members; an arrival at barrier 2
//      says that it has.
//   merges  every CTA works out the same merges from those cells: while the
//      smallest cell between members lies below TH, below the marks and below
//      every cell that a merged cluster can have to a slot outside (a lower
//      bound from the operands' bounds), it is the smallest of all, so it is
//      the sequential algorithm's next merge.  Complete, average, weighted and
//      Ward linkage mostly merge disjoint entries: those are taken in one go
//      and the limits checked side by side (the chain); where cells made by the
//      round's own merges cut it short, and for single and centroid linkage,
//      one warp takes the merges step by step.
//   on condition  the bounds for outside cells may end a round that the cells
//      themselves would not (equal values; inversions; values small against the
//      largest, for single linkage).  When that costs a quarter as many merges of a
//      chain as were proved (kTieGain, kTiePart), or as many steps (see simulate),
//      the merges are taken on condition: the new cells are computed and kept
//      back, every CTA looks whether one of its own comes before a merge of the
//      round, and barrier 3 tells which merges stand (settle).
//   apply  behind barrier 2 (no CTA still reads the members' old cells): the new
//      cells D(k, survivor) for every live k, a warp per 32 rows and up to 4
//      survivors, all loads of an item in flight at once; then logs, caches
//      (merged columns leave, new cells at or below B enter) and the
//      survivors' lists: their new cells below a limit go to lists in global
//      memory that every CTA reads after the next barrier 1.
//
// Refills.  A row whose cache is down to one key (n <= kRefillEarlyN: rows are
// short and rounds are what costs) or empty asks for a refill.  In the next
// round the upper half of the warps of each CTA (team B) scans the rows, cut
// in pieces, beside the lower half's (team A's) gather and merges, and then
// joins the apply; for longer rows it starts before the selection.  At the
// start of the round after that the owner takes the list, dropping the columns
// merged meanwhile and replaying the new cells.  A row that empties while its
// bound sits at the front of the merges is rescanned at once by its owner.  A
// job's only CTA refreshes emptied rows itself, a warp per row.
//
// What bounds it.  A round is a chain of short steps: about 40 us at n = 16384
// of which 3 are barrier 1, 6 the selection, 6 the gather, 5 the merges, 7 the
// new cells, 4 caches and lists, 3 publish; the memory traffic of a round (some
// 10 MB) would take under 2 us.  So what counts is merges per round: certifying
// a walk of disjoint entries after an exchange of the new cells' minima (two full
// barriers and about 13 merges per round) took 46.1 ms for n = 16384 average
// linkage, 162.8 ms for single and 16.8 ms for n = 1968 (complete, on one CTA
// then); selecting up to 64 members by a threshold and merging inside them takes
// 24.7, 50.0 and 2.3 ms.  Next, the instructions themselves: each step's code
// runs once or twice per round, so most of it is fetched anew every round
// (n = 2000: 58 % of the SM's instruction cache requests hit, and waiting for
// instructions was the largest stall after barriers, 3.7 of 11 cycles per
// instruction outside them).  That is why no loop below is unrolled unless its
// loads have to be in flight together: it took 5 to 9 % off every grid run (72 %
// of the requests hit since, and the stall is 1.4 cycles per instruction).
//
// Exact arithmetic: every product and sum of the update uses __fmul_rn /
// __fadd_rn / __fsub_rn (never contracted into FMA), the coefficient
// divisions __fdiv_rn; the four terms are added left to right.  The minimum
// is the smallest (value, row, column); values are non-negative floats, so
// their bit patterns order like the values and a 64-bit integer compare of
// (bits << 32 | index) gives the lexicographic order.
//
// Memory model.  L1 is not coherent across SMs, so every load of data that
// another CTA may have written (matrix cells, records, sizes) is an L2 load
// (ld.global.cg) and every store bypasses L1 (st.global.cg).  The barrier:
// __syncthreads, then one thread arrives with a release add (cumulative over
// the CTA's writes ordered before it by the __syncthreads) and later spins
// with acquire loads.  Each spin is bounded by a wall-clock limit after which
// the kernel records LW_ERR_TIMEOUT and returns.

#include "../../include/lw.h"
#include "lw_internal.h"

#include <cstdint>

namespace lw {
namespace {

typedef unsigned long long u64;
constexpr int K = kCacheKeys;

// Global loads and stores of the merge kernel: L2 only (see "Memory model"),
// and in the bounds-checked build (-DLW_CHECKED) checked against the job's
// buffers first (an address outside them is skipped, a load reads zero, and
// the status records kErrBounds and the source line).
#ifdef LW_CHECKED
__device__ __noinline__ bool check_ok(const MergeParams &p, const void *a, unsigned bytes, int line)
{
    const char *c = static_cast<const char *>(a);
    for (int q = 0; q < p.nck; ++q)
        if (c >= p.ck[q].base && c + bytes <= p.ck[q].base + p.ck[q].bytes)
            return true;
    if (atomicCAS(p.status, 0, kErrBounds) == 0)
        atomicExch(p.status + 2, line);
    return false;
}
template <class T>
struct same_type {
    typedef T type;
};
template <class T>
__device__ __forceinline__ T ld_checked(const MergeParams &p, const T *a, int line)
{
    return check_ok(p, a, sizeof(T), line) ? __ldcg(a) : T();
}
template <class T>
__device__ __forceinline__ void st_checked(const MergeParams &p, T *a, typename same_type<T>::type v, int line)
{
    if (check_ok(p, a, sizeof(T), line))
        __stcg(a, v);
}
#define CHECK_PREFETCH(a) check_ok(p, (a), 4, __LINE__)
#define LDCG(a) ld_checked(p, (a), __LINE__)
#define STCG(a, v) st_checked(p, (a), (v), __LINE__)
#else
#define CHECK_PREFETCH(a) true
#define LDCG(a) __ldcg(a)
#define STCG(a, v) __stcg((a), (v))
#endif

__device__ __forceinline__ long long tri_off(long long r, long long n)
{
    return r * n - ((r * (r + 1)) >> 1);
}

__device__ __forceinline__ long long pair_idx(long long a, long long b, long long n)
{
    return a < b ? tri_off(a, n) + (b - a - 1) : tri_off(b, n) + (a - b - 1);
}

// Row r of the working matrix: cell (r, c) at row_base + c (packed: c > r only).
__device__ __forceinline__ long long row_base(const MergeParams &p, long long r)
{
    return p.full ? r * p.pitch : tri_off(r, p.n) - r - 1;
}


__device__ __forceinline__ u64 make_key(float v, unsigned c)
{
    return ((u64)__float_as_uint(v) << 32) | (u64)c;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_relaxed_s32(const int *p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add(unsigned *p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Brings the line of an address into L2.
__device__ __forceinline__ void prefetch_l2(const void *a)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
}

__device__ __forceinline__ u64 global_ns()
{
    u64 t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------------------
// sorted key lists (ascending, padded with kNoKey)
// ---------------------------------------------------------------------------

__device__ __forceinline__ void cswap(u64 &a, u64 &b)
{
    const u64 lo = a < b ? a : b;
    b = a < b ? b : a;
    a = lo;
}

// Insert x into the K smallest: a compare-swap pass; the largest falls off
// (and is returned).
__device__ __forceinline__ u64 list_insert(u64 (&L)[K], u64 x)
{
#pragma unroll
    for (int q = 0; q < K; ++q)
        cswap(L[q], x);
    return x;
}

__device__ __forceinline__ int list_count(const u64 *L)
{
    int c = 0;
#pragma unroll
    for (int q = 0; q < K; ++q)
        c += L[q] != kNoKey;
    return c;
}

// Warp-wide minimum of 64-bit keys with two hardware warp reductions: the
// smallest high word, then the smallest low word among the lanes holding it.
__device__ __forceinline__ u64 warp_u64_min(u64 v)
{
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mhi = __reduce_min_sync(0xffffffffu, hi);
    const unsigned mlo = __reduce_min_sync(0xffffffffu, hi == mhi ? (unsigned)v : 0xffffffffu);
    return ((u64)mhi << 32) | mlo;
}

// KK smallest keys over the sorted lists of a warp (keys are distinct or kNoKey).
template <int KK>
__device__ __forceinline__ void warp_topk(u64 (&L)[KK], u64 (&out)[KK])
{
#pragma unroll
    for (int q = 0; q < KK; ++q) {
        const u64 m = warp_u64_min(L[0]);
        out[q] = m;
        if (m != kNoKey && L[0] == m) {
#pragma unroll
            for (int s = 0; s + 1 < KK; ++s)
                L[s] = L[s + 1];
            L[KK - 1] = kNoKey;
        }
    }
}

// warp_topk over lists that may have dropped keys above their last one, and
// `next`, a lower bound of every key not in out: the next listed one, or just
// above the last key of a full list whose keys are all in out.
__device__ __forceinline__ void warp_topk_next(u64 (&L)[K], u64 (&out)[K], u64 &next)
{
    const u64 end = L[K - 1] == kNoKey ? kNoKey : L[K - 1] + 1;
    warp_topk(L, out);
    next = warp_u64_min(L[0] != kNoKey ? L[0] : end);
}

// Insert x into a sorted list of KK keys; the largest falls off.
template <int KK>
__device__ __forceinline__ void list_insert_n(u64 (&L)[KK], u64 x)
{
#pragma unroll
    for (int q = 0; q < KK; ++q)
        cswap(L[q], x);
}

constexpr unsigned kFull = 0xffffffffu;
constexpr u64 kHi = 0xffffffff00000000ull;
static_assert(K == 4, "sort_list is a 4-input network");
static_assert(kPub % 4 == 0 && kPub >= K, "record layout");
static_assert(kTeam == 64, "a warp's lanes hold two members each; masks of 64 bits");

// Sort a K-list in which any entries were replaced by kNoKey.
__device__ __forceinline__ void sort_list(u64 (&L)[K])
{
    cswap(L[0], L[1]);
    cswap(L[2], L[3]);
    cswap(L[0], L[2]);
    cswap(L[1], L[3]);
    cswap(L[1], L[2]);
}

// A round's members and merges (static shared memory).
struct Team {
    // the members (slots in ascending order), size and bound of the cells
    // outside (value bits), stamp, row base; every cell not between two members
    // is above (thA, thC) = (value << 32 | row, column), or above the member's
    // own bound (lbA, lbC) where a row's cached keys end below that
    int m;
    unsigned thC, thv;
    u64 thA;
    unsigned dmax;               // largest input value (bits)
    int mem[kTeam], mst[kTeam];
    int2 sl[kTeam];
    long long mbase[kTeam];      // cell (slot, c) at mbase + c
    u64 lbA[kTeam];
    unsigned lbC[kTeam];
    float S[kTeam][kTeam + 1];   // cells between members
    unsigned nnv[kTeam], nnc[kTeam];
    u64 mask[kTeam];
    // the entries in key order: members i | j << 8 (0xffff: a bound mark) and
    // value bits; per member the entries it takes part in
    uint2 ent[kEntries];
    u64 em[kTeam];
    int ne;
    int sz0[kTeam];              // sizes before the round
    // the chain: per entry the entries that share a member with it, per member
    // its merge (0xff: none), the cells merge q makes with every member, those
    // between survivors after the round, and the least cell before each merge
    uint2 enm[kEntries];
    unsigned char step[kEntries];
    unsigned char ce[kSurv];     // entry of merge q
    unsigned char ex[kTeam];     // entry that ends a member's row (0xff: none)
    int redo;                    // the chain broke off early: step by step instead
    // merges on condition (tie): they wait for a look at the cells outside, those
    // from `sure` on (cmax: their largest height); taken step by step (steps):
    // how many at most the next time (reach)
    int tie, sure, steps, reach;
    unsigned cmax;
    unsigned char cons[kTeam];   // merge that takes in the cluster of merge q (L: none)
    float X[kSurv][kTeam + 1];
    float C[kSurv][kSurv + 1];
    unsigned lim[kSurv];
    // the round's merges in order: members i | j << 8 and, in the upper half,
    // the merge that made each operand (q + 1; 0: a cell in memory), height
    // bits, sizes; coefficients (a_i, a_j, b times the height, g; not Ward)
    int L;
    int4 rec[kTeam];
    float4 co[kTeam];
    int res[kTeam];
    // the merged clusters still live after the round: the merges that lead to
    // each in order (prog[sfirst[s] .. sfirst[s + 1])), the last of them, slot
    int ns;
    int prog[kTeam], root[kTeam], sfirst[kSurv + 1], sq[kSurv], sslot[kSurv];
    u64 tT[kSurv][K], tB[kSurv]; // smallest keys of the survivor's cells to other survivors
    __device__ int mi(int q) const { return rec[q].x & 0xff; }
    __device__ int mj(int q) const { return (rec[q].x >> 8) & 0xff; }
};

// Static shared memory of a CTA.  ONE: the CTA is its job's only one (no
// records, no refill requests).
template <int NT, bool ONE>
struct Shared {
    static constexpr int W = NT / 32;
    u64 tk[W][kPub];
    u64 tko[kPub], tnext, tnx[W];
    int wcnt[W];
    u64 wmin[W][2];
    int flag;
    int nexec;                   // refill rows served this round
    int exec_row[kMaxReq];
    int nmyreq[2];               // this CTA's requests, by round parity
    int myreq_l[2][kReqPerCta];
    int npieces;                 // pieces per row of the refills served last
    int ninst;                   // refills to install in this round
    int inst_slot[kReqPerCta];
    // candidate entries of the round (unordered), the first kEntries of them in
    // key order, and which of those bring a new row (1) or column (2) or end
    // the selection (4)
    int ncand;
    u64 ckey[kCand];
    unsigned ccol[kCand];
    u64 ekey[kEntries + 1];
    uint2 erc[kEntries + 1];     // row, column word
    unsigned char enew[kEntries];
    int umem[kTeam];
    Team tm;
    // the previous round's survivors and their caches
    int nps;
    int pslot[kSurv];
    u64 svk[kSurv][K], svB[kSurv];
    int svc[kSurv];
    int nptouch;                 // slots the previous round touched
    int ptouch[kTeam];
    unsigned okm[NT / 32];       // rows of the chunk that take the round's merges
    unsigned hit[NT];            // per row of the chunk: new cells that may enter its cache
    int nresc;                   // rows to rescan at once this round
    int item, viol;              // apply pass: next item, first merge that must wait
    unsigned limit, width;       // see the selection
    int svsum;                   // entries of the previous round's survivors' lists
    u64 ppivot;                  // the last round's pivot of the published entries
    u64 pivot;                   // the last round's pivot of the entry selection
    // the job's arrays in dynamic shared memory (see merge_job) and its row split,
    // for the functions kept out of line (the round loop holds as many registers
    // as a CTA may have: inline, they would spill)
    struct {
        unsigned *bitmap, *touched, *wcol;
        u64 *wkey, *ck, *cB;
        float *kvs;
        int *rsize, *rlist, *pend_t, *pend_s, *rstamp;
        unsigned char *ccnt;
        long long Rmax;
        int R, b, G;
    } cx;
    // phase timers and the counters one thread keeps (thread 0, thread 32 for
    // the refill team): here rather than in registers of the round loop
    struct {
        u64 ph[6], xs[8], xscan[2], tmark;
        long long fills, installs, rounds, idle, walk, rescans;
    } ty;
};

// After the main barrier: the list of rows to refill in this round -- every CTA's
// requests in CTA order (deterministic, the same in every CTA), cut at
// kMaxReq.  Thread t holds CTA t's request count and rows.  Sets
// sh.exec_row and sh.nexec; thread b gives this CTA's own requests (list
// pq) their list positions.
template <int NT, bool ONE>
__device__ void exchange_requests(int cnt, const int (&rq)[kReqPerCta], int b, Shared<NT, ONE> &sh, int pq,
                                  int *pend_t, int *pend_s)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(kFull, inc, off);
        if (lane >= off)
            inc += o;
    }
    if (lane == 31)
        sh.wcnt[warp] = inc;
    __syncthreads();
    int base = 0;
#pragma unroll 1
    for (int w = 0; w < warp; ++w)
        base += sh.wcnt[w];
    const int off0 = base + inc - cnt;
#pragma unroll
    for (int q = 0; q < kReqPerCta; ++q) {
        if (q < cnt && off0 + q < kMaxReq)
            sh.exec_row[off0 + q] = rq[q];
    }
    if ((int)threadIdx.x == b) {
        // this CTA's own requests (list pq) get their positions
#pragma unroll 1
        for (int q = 0; q < cnt; ++q) {
            const int l = sh.myreq_l[pq][q];
            if (off0 + q < kMaxReq)
                pend_s[l] = off0 + q;
            else
                pend_t[l] = -1;  // not served: the row may ask again
        }
    }
    if (warp == 0) {
        int tot = lane < (NT / 32) ? sh.wcnt[lane] : 0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            tot += __shfl_xor_sync(kFull, tot, off);
        if (lane == 0)
            sh.nexec = tot < kMaxReq ? tot : kMaxReq;
    }
    __syncthreads();
}

// Barrier of the threads that work together: the whole CTA (TB == NT), or
// its last TB threads (named barrier 1).
template <int NT, int TB>
__device__ __forceinline__ void team_sync()
{
    static_assert(TB % 32 == 0 && TB <= NT, "a team is whole warps");
    if constexpr (TB == NT)
        __syncthreads();
    else
        asm volatile("bar.sync 1, %0;" ::"n"(TB) : "memory");
}

// KK smallest keys over every thread's sorted list, for a team of the CTA's
// last TB threads (default: all of them); result in sh.tko, and in sh.tnext a
// lower bound of every other key (team threads).
template <int NT, bool ONE, int KK, int TB = NT>
__device__ void block_topk(u64 (&L)[KK], Shared<NT, ONE> &sh)
{
    constexpr int W0 = (NT - TB) / 32;  // first warp of the team
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u64 w[KK];
    u64 end = L[KK - 1] == kNoKey ? kNoKey : L[KK - 1] + 1;
    warp_topk(L, w);
    u64 nx = warp_u64_min(L[0] != kNoKey ? L[0] : end);
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < KK; ++q)
            sh.tk[warp][q] = w[q];
        sh.tnx[warp] = nx;
    }
    team_sync<NT, TB>();
    if (warp == W0) {
        u64 M[KK];
#pragma unroll
        for (int q = 0; q < KK; ++q)
            M[q] = lane < TB / 32 ? sh.tk[W0 + lane][q] : kNoKey;
        end = lane < TB / 32 ? sh.tnx[W0 + lane] : kNoKey;
        warp_topk(M, w);
        nx = warp_u64_min(M[0] != kNoKey ? M[0] : end);
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < KK; ++q)
                sh.tko[q] = w[q];
            sh.tnext = nx;
        }
    }
    team_sync<NT, TB>();
}

// Grid-wide barrier, split in two so that a CTA can do work that nobody
// waits for between arriving and waiting.  arrive: __syncthreads, then one
// thread adds to the counter with release semantics (the CTA's writes so far
// are published).  wait: that thread spins with acquire loads until every
// CTA has arrived, bounded by a wall-clock limit; returns false when the run
// must stop (this CTA gave up, or another CTA flagged an error).
// Two counters: one for the start of a round, one for "every CTA holds the
// members' cells" (see merge_job).
__device__ __forceinline__ void grid_arrive(const MergeParams &p, unsigned *bar, unsigned &epoch)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        epoch += 1;
        if (p.G > 1)
            red_release_add(bar, 1u);
    }
}

template <int NT, bool ONE, class F>
__device__ bool grid_wait(const MergeParams &p, const unsigned *bar, unsigned epoch, Shared<NT, ONE> &sh, F &&sync)
{
    if (threadIdx.x == 0) {
        int st = 0;
        if (p.G > 1) {
            const unsigned target = epoch * (unsigned)p.G;
            const u64 t0 = global_ns();
            unsigned spins = 0;
            while (ld_acquire_u32(bar) < target) {
                if ((++spins & 255u) == 0) {
                    st = ld_relaxed_s32(p.status);
                    if (st != 0)
                        break;
                    if (global_ns() - t0 > p.timeout_ns) {
                        atomicCAS(p.status, 0, kErrTimeout);
                        atomicCAS(p.status + 1, 0, (int)epoch);
                        st = kErrTimeout;
                        break;
                    }
                }
            }
        }
        sh.flag = st;
    }
    sync();
    return sh.flag == 0;
}

template <int NT, bool ONE>
__device__ bool grid_wait(const MergeParams &p, const unsigned *bar, unsigned epoch, Shared<NT, ONE> &sh)
{
    return grid_wait(p, bar, epoch, sh, [] { __syncthreads(); });
}

// Live-column test against the CTA's copy of the liveness bitmap.
// (slots fit 24 bits: 32-bit indices are half the instructions)
__device__ __forceinline__ bool live(const unsigned *bitmap, long long c)
{
    const unsigned i = (unsigned)c;
    return (bitmap[i >> 5] >> (i & 31u)) & 1u;
}

// Adds one input cell to a per-lane list during the initial scan: checks it
// (finite and >= 0), rewrites -0 as +0 in memory, and keeps the K smallest.
__device__ __forceinline__ void init_cell(float v, long long q, unsigned c, const MergeParams &p,
                                          u64 (&L)[K], int &bad, unsigned &mx)
{
    unsigned u = __float_as_uint(v);
    if (u > 0x7f7fffffu) {
        if (u == 0x80000000u) {
            STCG(p.D + q, 0.0f);
            u = 0u;
        } else {
            bad = 1;
            return;
        }
    }
    mx = u > mx ? u : mx;
    // a key not below the list's largest cannot enter it (an exact test of
    // the whole key: cells tying on the value are common and go no further)
    const u64 key = ((u64)u << 32) | (u64)c;
    if (key >= L[K - 1])
        return;
    list_insert(L, key);
}

// K smallest keys of row r (all columns are live at launch), computed by one
// warp that also validates every cell of the row.
__device__ void warp_row_topk(const MergeParams &p, long long r, u64 (&out)[K], u64 &next, int &bad, unsigned &mx)
{
    const long long n = p.n;
    const int lane = threadIdx.x & 31;
    const long long start = row_base(p, r) + r + 1;
    const long long end = start + (n - r - 1);
    const long long base_c = r + 1 - start;  // column of flat index q is q + base_c
    u64 L[K];
#pragma unroll
    for (int q = 0; q < K; ++q)
        L[q] = kNoKey;
    long long a0 = p.aligned16 ? ((start + 3) & ~3LL) : end;
    if (a0 > end)
        a0 = end;
    const long long a1 = a0 + ((end - a0) & ~3LL);
    for (long long q = start + lane; q < a0; q += 32)
        init_cell(LDCG(p.D + q), q, (unsigned)(q + base_c), p, L, bad, mx);
    for (long long q = a1 + lane; q < end; q += 32)
        init_cell(LDCG(p.D + q), q, (unsigned)(q + base_c), p, L, bad, mx);
    // 128-bit body, four loads in flight per lane
    long long q = a0 + 4 * lane;
    for (; q + 3 * 128 < a1; q += 4 * 128) {
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            x[u] = LDCG(reinterpret_cast<const float4 *>(p.D + q + 128 * u));
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long qq = q + 128 * u;
            const unsigned c = (unsigned)(qq + base_c);
            init_cell(x[u].x, qq, c, p, L, bad, mx);
            init_cell(x[u].y, qq + 1, c + 1, p, L, bad, mx);
            init_cell(x[u].z, qq + 2, c + 2, p, L, bad, mx);
            init_cell(x[u].w, qq + 3, c + 3, p, L, bad, mx);
        }
    }
    for (; q < a1; q += 128) {
        const float4 x = LDCG(reinterpret_cast<const float4 *>(p.D + q));
        const unsigned c = (unsigned)(q + base_c);
        init_cell(x.x, q, c, p, L, bad, mx);
        init_cell(x.y, q + 1, c + 1, p, L, bad, mx);
        init_cell(x.z, q + 2, c + 2, p, L, bad, mx);
        init_cell(x.w, q + 3, c + 3, p, L, bad, mx);
    }
    warp_topk_next(L, out, next);
}

// Eight 16-byte pieces of a packed row (j0, j0 + stride, .. below j1; column of
// word q: q + base_c), live cells into a sorted list: all loads in flight, one
// comparison per cell, and one copy of the insertion for the few that pass (a
// copy per cell made this scan 47 KB of instructions, and fetching them cost
// more than running them).
__device__ __forceinline__ void take_batch(const MergeParams &p, long long j0, int stride, long long j1,
                                           long long base_c, const unsigned *bitmap, u64 (&L)[K], long long &cnt)
{
    const float4 *D4 = reinterpret_cast<const float4 *>(p.D);
    float v[8][4];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const long long j = j0 + (long long)u * stride;
        const float4 x = j < j1 ? LDCG(D4 + j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        v[u][0] = x.x; v[u][1] = x.y; v[u][2] = x.z; v[u][3] = x.w;
    }
    const int c0 = (int)((j0 << 2) + base_c);
    unsigned in = 0u;
    int had = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        // (the index, not the value: a cell may be NaN once the recurrence overflowed)
        if (j0 + (long long)u * stride < j1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = c0 + 4 * u * stride + e;
                const unsigned on = (bitmap[c >> 5] >> (c & 31)) & 1u;
                had += (int)on;
                // the whole key: ties on the value stop here
                if (make_key(v[u][e], (unsigned)c) < L[K - 1])
                    in |= on << (4 * u + e);
            }
        }
    }
    cnt += had;
#pragma unroll 1
    for (; in != 0u; in &= in - 1u) {
        const int i = __ffs(in) - 1;
        float x = v[0][0];
#pragma unroll
        for (int q = 1; q < 32; ++q)
            x = i == q ? v[q >> 2][q & 3] : x;
        const u64 key = make_key(x, (unsigned)(c0 + 4 * (i >> 2) * stride + (i & 3)));
        if (key < L[K - 1])
            list_insert(L, key);
    }
}

// block_topk of K-lists, out of line: it is called at the end of every scan.
template <int NT, bool ONE, int TB>
__device__ __noinline__ void block_topk_call(u64 a, u64 b, u64 c, u64 d, Shared<NT, ONE> &sh)
{
    u64 L[K] = {a, b, c, d};
    block_topk<NT, ONE, K, TB>(L, sh);
}

// K smallest keys of row r over live columns, computed by the whole CTA (a
// refill, or a row whose cache emptied).  Adds the live cells read to
// `live_cells`.  Result in sh.tko.
// (Row scans are kept out of line: inside the round loop's register
// allocation their loads in flight would be spilled.)
template <int NT, bool ONE, int TB = NT>
__device__ __noinline__ void block_row_topk(const MergeParams &p, long long r, int piece, int np,
                                            const unsigned *bitmap, Shared<NT, ONE> &sh, long long &live_cells)
{
    const int ts = threadIdx.x - (NT - TB);  // thread of the team
    const long long n = p.n;
    const long long start = row_base(p, r) + r + 1;
    const long long end = start + (n - r - 1);
    const long long base_c = r + 1 - start;
    u64 L[K];
#pragma unroll
    for (int q = 0; q < K; ++q)
        L[q] = kNoKey;
    long long cnt = 0;
    auto take = [&](float v, long long q) {
        const long long c = q + base_c;
        if (live(bitmap, c)) {
            ++cnt;
            const u64 key = make_key(v, (unsigned)c);
            if (key < L[K - 1])  // the whole key: ties on the value stop here
                list_insert(L, key);
        }
    };
    // unaligned head and tail one word per thread; the body as 16-byte loads,
    // eight in flight per thread (dead cells are read and dropped: the row is
    // contiguous, latency and not bandwidth bounds the scan)
    long long a0 = p.aligned16 ? ((start + 3) & ~3LL) : end;
    if (a0 > end)
        a0 = end;
    const long long a1 = a0 + ((end - a0) & ~3LL);
    // (head, then tail)
#pragma unroll 1
    for (int part = piece == 0 ? 0 : 1; part < (piece == np - 1 ? 2 : 1); ++part)
#pragma unroll 1
        for (long long q = (part ? a1 : start) + ts; q < (part ? end : a0); q += TB)
            take(LDCG(p.D + q), q);
    const long long part = ((a1 - a0) >> 2) / np;
    const long long jb = (a0 >> 2) + part * piece;
    const long long j1 = piece == np - 1 ? a1 >> 2 : jb + part;
#pragma unroll 1
    for (long long j0 = jb + ts; j0 < j1; j0 += 8 * TB)
        take_batch(p, j0, TB, j1, base_c, bitmap, L, cnt);
    live_cells += cnt;
    block_topk_call<NT, ONE, TB>(L[0], L[1], L[2], L[3], sh);
}
// block_row_topk in the row-log layout, column by column: live column c > r
// holds its current cell in row r of M when c's stamp is not after r's, and
// otherwise in r's log at c's stamp (written by that merge).  The stamps are
// read beside the row (16-byte pieces of both, two of each per thread and
// batch), then the log cells of the columns stamped after r: two dependent
// reads per batch and no pass over the merge list.  (A deeper batch holds
// more registers across the call, and the caller, the round loop, then
// spills: two pieces measured fastest.)  p.D and p.stamp are 16-byte aligned
// (rows are, the pitch being a multiple of 4).  Columns stamped tskip or
// later are left out: a scan that runs while other CTAs apply the round's
// merges skips the columns they rewrite, whose log cells may not be there
// yet.  The first batch gives a bound when the row has more than one: the 5th
// smallest of the team's per-thread minima is the key of a real cell with at
// least four real cells below it, so no cell above it can be among the row's
// five smallest (the lists and the bound of the rest); after it only cells at
// or below it reach the lists.  Piece
// `piece` of np equal pieces of the row.  Result in sh.tko.
template <int NT, bool ONE, int TB = NT>
__device__ __noinline__ void block_row_topk_cols(const MergeParams &p, long long r, int piece, int np,
                                                 int tskip, const unsigned *bitmap, Shared<NT, ONE> &sh,
                                                 long long &live_cells, u64 *tlog = nullptr)
{
    const int ts = threadIdx.x - (NT - TB);  // thread of the team
    const u64 tm0 = tlog && ts == 0 ? global_ns() : 0;
    const long long n = p.n;
    const int sr = LDCG(p.stamp + r);
    const float *row = p.D + r * p.pitch;
    const float *log = p.TL + r * p.pitch;
    u64 L[K];
#pragma unroll
    for (int q = 0; q < K; ++q)
        L[q] = kNoKey;
    long long cnt = 0;
    auto one = [&](long long c) {
        if (live(bitmap, c)) {
            const int sc = LDCG(p.stamp + c);
            if (sc >= tskip)
                return;
            ++cnt;
            const float v = sc > sr ? LDCG(log + sc) : LDCG(row + c);
            const u64 key = make_key(v, (unsigned)c);
            if (key < L[K - 1])
                list_insert(L, key);
        }
    };
    long long c_a = (r + 4) & ~3LL;  // first multiple of 4 above r
    if (c_a > n)
        c_a = n;
    const long long c_b = c_a + ((n - c_a) & ~3LL);
    // (head, then tail)
#pragma unroll 1
    for (int end = piece == 0 ? 0 : 1; end < (piece == np - 1 ? 2 : 1); ++end)
#pragma unroll 1
        for (long long c = (end ? c_b : r + 1) + ts; c < (end ? n : c_a); c += TB)
            one(c);
    {
        constexpr int U = 2;
        const float4 *R4 = reinterpret_cast<const float4 *>(row);
        const int4 *S4 = reinterpret_cast<const int4 *>(p.stamp);
        const long long part = ((c_b - c_a) >> 2) / np;
        const long long j0a = (c_a >> 2) + part * piece;
        const long long j1 = piece == np - 1 ? c_b >> 2 : j0a + part;
        if (tskip < 0x7fffffff && n > kRefillEarlyN) {
            // the piece's lines of the row, and an equal part of the log's words
            // that live columns may need unless those are few: read at the
            // memory's rate now instead of a sector per column later (n = 65536
            // complete: 22.0 us of scans per round without, 18.5 with; nothing
            // gained where a piece is a batch or two)
            for (long long j = (j0a & ~7LL) + 8LL * ts; j < j1; j += 8LL * TB)
                if (CHECK_PREFETCH(R4 + j))
                    prefetch_l2(R4 + j);
            const long long words = tskip - sr;
            if (words <= 4 * (n - tskip)) {
                const long long w0 = sr + words * piece / np, w1 = sr + words * (piece + 1) / np;
                for (long long j = (w0 & ~31LL) + 32LL * ts; j < w1; j += 32LL * TB)
                    if (j >= 0 && CHECK_PREFETCH(log + j))
                        prefetch_l2(log + j);
            }
        }
        // a bound from the first batch only pays when more batches follow
        bool first = j1 - j0a > (long long)U * TB;
        u64 thr = kNoKey;
        for (long long j0 = j0a + ts;; j0 += U * TB) {
            if (!first && j0 >= j1)
                break;  // (every thread of the team runs a first batch: it holds a barrier)
            float v[U][4];
            int sc[U][4];
            unsigned m4[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long long j = j0 + (long long)u * TB;
                m4[u] = 0u;
                if (j < j1) {
                    const float4 a = LDCG(R4 + j);
                    const int4 b = LDCG(S4 + j);
                    v[u][0] = a.x; v[u][1] = a.y; v[u][2] = a.z; v[u][3] = a.w;
                    sc[u][0] = b.x; sc[u][1] = b.y; sc[u][2] = b.z; sc[u][3] = b.w;
                    const long long c = j << 2;
                    m4[u] = (bitmap[c >> 5] >> (c & 31)) & 15u;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (((m4[u] >> e) & 1u) && sc[u][e] > sr) {
                        if (sc[u][e] < tskip)
                            v[u][e] = LDCG(log + sc[u][e]);
                        else
                            m4[u] &= ~(1u << e);
                    }
            }
            if (first) {
                u64 mn = kNoKey;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const long long c = (j0 + (long long)u * TB) << 2;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const u64 k = make_key(v[u][e], (unsigned)(c + e));
                        if (((m4[u] >> e) & 1u) && k < mn)
                            mn = k;
                    }
                }
                block_topk_call<NT, ONE, TB>(mn, kNoKey, kNoKey, kNoKey, sh);
                thr = sh.tnext;
                first = false;
            }
            // one copy of the insertion for the few cells that pass (see take_batch)
            unsigned in = 0u;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long long c = (j0 + (long long)u * TB) << 2;
                cnt += __popc(m4[u]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const u64 k = make_key(v[u][e], (unsigned)(c + e));
                    if (k <= thr && k < L[K - 1])
                        in |= m4[u] & (1u << e) ? 1u << (4 * u + e) : 0u;
                }
            }
#pragma unroll 1
            for (; in != 0u; in &= in - 1u) {
                const int i = __ffs(in) - 1;
                float x = v[0][0];
#pragma unroll
                for (int q = 1; q < 4 * U; ++q)
                    x = i == q ? v[q >> 2][q & 3] : x;
                const u64 k = make_key(x, (unsigned)(((j0 + (long long)(i >> 2) * TB) << 2) + (i & 3)));
                if (k < L[K - 1])
                    list_insert(L, k);
            }
        }
    }
    live_cells += cnt;
    block_topk_call<NT, ONE, TB>(L[0], L[1], L[2], L[3], sh);
    if (tlog && ts == 0)
        tlog[1] += global_ns() - tm0;
}

// K smallest keys of row r over live columns, computed by one warp (the
// rows of a one-CTA job are refreshed this way, several warps side by side).
// Adds the live cells read to `live_cells`.  Result in out (all lanes).
__device__ __noinline__ void warp_row_refresh(const MergeParams &p, long long r, const unsigned *bitmap,
                                              u64 (&out)[K], u64 &next, long long &live_cells)
{
    const int lane = threadIdx.x & 31;
    const long long start = row_base(p, r) + r + 1;
    const long long end = start + (p.n - r - 1);
    const long long base_c = r + 1 - start;
    u64 L[K];
#pragma unroll
    for (int q = 0; q < K; ++q)
        L[q] = kNoKey;
    long long cnt = 0;
    auto take = [&](float v, long long q) {
        const long long c = q + base_c;
        if (live(bitmap, c)) {
            ++cnt;
            const u64 key = make_key(v, (unsigned)c);
            if (key < L[K - 1])  // the whole key: ties on the value stop here
                list_insert(L, key);
        }
    };
    long long a0 = p.aligned16 ? ((start + 3) & ~3LL) : end;
    if (a0 > end)
        a0 = end;
    const long long a1 = a0 + ((end - a0) & ~3LL);
#pragma unroll 1
    for (int part = 0; part < 2; ++part)  // head, tail
#pragma unroll 1
        for (long long q = (part ? a1 : start) + lane; q < (part ? end : a0); q += 32)
            take(LDCG(p.D + q), q);
    const long long j1 = a1 >> 2;
#pragma unroll 1
    for (long long j0 = (a0 >> 2) + lane; j0 < j1; j0 += 8 * 32)
        take_batch(p, j0, 32, j1, base_c, bitmap, L, cnt);
    live_cells += cnt;
    warp_topk_next(L, out, next);
}

// Merge q for a row of size nk: the new cell from its two cells.
__device__ __forceinline__ float merge_cell(const Team &tm, int linkage, int q, float a, float b, float nk)
{
    if (linkage == 3) {
        const int4 rec = tm.rec[q];
        return ward_cell((float)rec.z, (float)rec.w, (float)(rec.z + rec.w), nk, __int_as_float(rec.y), a, b);
    }
    const float4 co = tm.co[q];
    return lw_sum(co.x, co.y, co.z, co.w, a, b);
}

// The step-by-step iteration among a round's members, as far as no other cell
// can come first; run by one warp, lane l holding members l and l + 32.  Only
// cells at or below the bound matter: per member row a mask of them (columns
// above the row) and the smallest one are kept in registers.
//
// One warp issues a step's instructions one after another, so their number is
// its time: everything is computed for all 64 members without branches, and
// what rarely happens (a lost minimum with other cells below the bound, a new
// cell below it, equal values at a bound) sits behind votes.
template <bool B>
struct Flag {
    static constexpr bool value = B;
};

template <int LK>
__device__ __noinline__ void simulate_steps(Team &tm, int reach, int &L_out, int &sure_out)
{
    const int lane = threadIdx.x & 31;
    const int m = tm.m;
    const unsigned thv = tm.thv;
    constexpr unsigned kNone = 0xffffffffu;
    unsigned nv[2], nc[2], lbv[2];
    u64 mk[2];
    bool lv[2];
    float fk[2];
    float *row[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int a = lane + 32 * h;
        lv[h] = a < m;
        nv[h] = lv[h] ? tm.nnv[a] : kNone;
        nc[h] = lv[h] ? tm.nnc[a] : kNone;
        mk[h] = lv[h] ? tm.mask[a] : 0ull;
        lbv[h] = lv[h] ? (unsigned)tm.sl[a].y : kNone;
        fk[h] = lv[h] ? (float)tm.sl[a].x : 1.0f;
        row[h] = tm.S[a];
        tm.res[a] = 0;
    }
    u64 merged = 0ull;
    int L = 0, sure = -1;
    __syncwarp();
    // `most` merges at most; false: a merge was not proved, but nothing known comes
    // before it
    auto run = [&](auto cond, int most) -> bool {
        while (L < most) {
            const bool sec = nv[1] < nv[0] || (nv[1] == nv[0] && nc[1] < nc[0]);
            const unsigned v1 = sec ? nv[1] : nv[0], c1 = sec ? nc[1] : nc[0];
            const unsigned hb = __reduce_min_sync(kFull, v1);
            const unsigned lbmin = __reduce_min_sync(kFull, lbv[0] < lbv[1] ? lbv[0] : lbv[1]);
            const unsigned code = __reduce_min_sync(kFull, v1 == hb ? c1 : kNone);
            if (code == kNone)
                return true;
            const int i = (int)(code >> 8), j = (int)(code & 0xffu);
            if (hb >= lbmin) {
                // equal values: whole keys against the bounds that are keys (those
                // of merged clusters are values; on condition thv, so that the bound of
                // the cells not listed is still asked)
                const u64 kA = ((u64)hb << 32) | (unsigned)tm.mem[i];
                const unsigned kC = (unsigned)tm.mem[j];
                bool ok = kA < tm.thA || (kA == tm.thA && kC < tm.thC), proved = true;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int a = lane + 32 * h;
                    if (lv[h]) {
                        if ((merged >> a) & 1ull)
                            proved = proved && hb < lbv[h];
                        else
                            ok = ok && (kA < tm.lbA[a] || (kA == tm.lbA[a] && kC < tm.lbC[a]));
                    }
                }
                if (!__all_sync(kFull, ok))
                    return true;
                if (!decltype(cond)::value && !__all_sync(kFull, proved))
                    return false;
            }
            float ca[2], cb[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                ca[h] = row[h][i];
                cb[h] = row[h][j];
            }
            const int2 si = tm.sl[i], sj = tm.sl[j];
            const float hgt = __uint_as_float(hb);
            const float fi = (float)si.x, fj = (float)sj.x, fs = (float)(si.x + sj.x);
            const float4 co = merge_coefs<LK>(si.x, sj.x, hgt);
            const u64 bi = 1ull << i, bj = 1ull << j;
            bool low[2], lost[2];
            float v[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = lane + 32 * h;
                if constexpr (decltype(cond)::value)
                    tm.X[L - sure][k] = ca[h];  // (steps_undo puts it back)
                v[h] = LK == 3 ? ward_cell(fi, fj, fs, fk[h], hgt, ca[h], cb[h])
                               : lw_sum(co.x, co.y, co.z, co.w, ca[h], cb[h]);
                row[h][i] = v[h];
                tm.S[i][k] = v[h];
                lv[h] = lv[h] && k != j;
                low[h] = lv[h] && k != i && __float_as_uint(v[h]) <= thv;
                const unsigned c = nc[h] & 0xffu;
                lost[h] = (c == (unsigned)i || c == (unsigned)j) && k != i;  // (a column above k)
                mk[h] &= ~(bi | bj);
                nv[h] = lost[h] || k == j ? kNone : nv[h];
                nc[h] = lost[h] || k == j ? kNone : nc[h];
            }
            const unsigned nbits = decltype(cond)::value ? thv : merged_bound<LK>(si.y, sj.y, fi, fs, hgt, tm.dmax);
            merged |= bi;
            const unsigned more = __ballot_sync(kFull, (lost[0] && mk[0] != 0ull && lv[0]) || (lost[1] && mk[1] != 0ull && lv[1]));
            const unsigned l0 = __ballot_sync(kFull, low[0]), l1 = __ballot_sync(kFull, low[1]);
            if (more) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = lane + 32 * h;
                    if (lost[h] && lv[h]) {
#pragma unroll 1
                        for (u64 q = mk[h]; q; q &= q - 1) {
                            const int c = __ffsll((long long)q) - 1;
                            const unsigned x = __float_as_uint(row[h][c]), y = (unsigned)(k << 8 | c);
                            if (x < nv[h] || (x == nv[h] && y < nc[h])) {
                                nv[h] = x;
                                nc[h] = y;
                            }
                        }
                    }
                }
            }
            unsigned ri = kNone, rc = kNone;
            u64 rm = 0ull;
            if (l0 | l1) {
                // new cells at or below the bound: those of rows k < i, and row i's
                unsigned w[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = lane + 32 * h;
                    const unsigned x = __float_as_uint(v[h]), y = (unsigned)(k << 8 | i);
                    if (low[h] && k < i) {
                        mk[h] |= bi;
                        if (x < nv[h] || (x == nv[h] && y < nc[h])) {
                            nv[h] = x;
                            nc[h] = y;
                        }
                    }
                    w[h] = low[h] && k > i ? x : kNone;
                }
                rm = (((u64)l1 << 32) | l0) & ~((bi << 1) - 1ull);
                ri = __reduce_min_sync(kFull, w[0] < w[1] ? w[0] : w[1]);
                const unsigned k0 = w[0] == ri ? (unsigned)lane : 64u, k1 = w[1] == ri ? (unsigned)lane + 32u : 64u;
                const unsigned kk = __reduce_min_sync(kFull, k0 < k1 ? k0 : k1);
                rc = rm ? ((unsigned)i << 8 | kk) : kNone;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = lane + 32 * h;
                if (k == i) {
                    mk[h] = rm;
                    nv[h] = ri;
                    nc[h] = rc;
                    lbv[h] = nbits;
                    fk[h] = fs;
                }
                if (k == j) {
                    mk[h] = 0ull;
                    lbv[h] = kNone;
                }
            }
            const int qi = tm.res[i], qj = tm.res[j];
            __syncwarp();
            if (lane == 0) {
                tm.rec[L] = make_int4(i | j << 8 | qi << 16 | qj << 24, (int)hb, si.x, sj.x);
                if (LK != 3)
                    tm.co[L] = co;
                tm.res[i] = L + 1;
                tm.sl[i] = make_int2(si.x + sj.x, (int)nbits);
            }
            ++L;
            __syncwarp();
        }
        return true;
    };
    if (!run(Flag<false>(), kTeam - 1)) {
        // from here on condition: the merged clusters' cells will be looked at
        sure = L;
        if (reach >= L) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                lbv[h] = lv[h] && ((merged >> (lane + 32 * h)) & 1ull) ? thv : lbv[h];
            run(Flag<true>(), min(L + reach, kTeam - 1));
        }
    }
    L_out = L;
    sure_out = sure < 0 ? L : sure;
}

// Takes back merges V .. L - 1 of simulate_steps (all on condition): the cells
// between members are again those after V merges.
__device__ __forceinline__ void steps_undo(Team &tm, int L, int V, int sure)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int e = L - 1; e >= V; --e) {
        const int i = tm.mi(e);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            const float x = tm.X[e - sure][k];
            tm.S[k][i] = x;
            tm.S[i][k] = x;
        }
        __syncwarp();
    }
}

// The first L merges of simulate_steps (their cells between members in S): those
// that lead to each survivor, in order, and the survivors' cells to one another.
__device__ __noinline__ void steps_program(Team &tm, int L)
{
    const int lane = threadIdx.x & 31;
    const bool dep = __any_sync(kFull, (lane < L && ((unsigned)tm.rec[lane].x >> 16) != 0u) ||
                                           (lane + 32 < L && ((unsigned)tm.rec[lane + 32].x >> 16) != 0u));
    tm.cons[lane] = (unsigned char)L;
    tm.cons[lane + 32] = (unsigned char)L;
    int ns = L;
    if (!dep) {
        // every merge joins two clusters of the round before: its own survivor
        // (at most kSurv of them, two members each)
        if (lane < L) {
            tm.prog[lane] = lane;
            tm.sfirst[lane] = lane;
            tm.sq[lane] = lane;
            tm.sslot[lane] = tm.mem[tm.mi(lane)];
        }
    } else {
        tm.root[lane] = lane;
        tm.root[lane + 32] = lane + 32;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int q = lane + 32 * h;
            if (q < L) {
                const int x = tm.rec[q].x;
                const int si = (x >> 16) & 0xff, sj = (x >> 24) & 0xff;
                if (si) {
                    tm.root[si - 1] = q;  // (merge q consumes that result)
                    tm.cons[si - 1] = (unsigned char)q;
                }
                if (sj) {
                    tm.root[sj - 1] = q;
                    tm.cons[sj - 1] = (unsigned char)q;
                }
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int it = 0; it < 6; ++it) {
            const int x0 = tm.root[tm.root[lane]], x1 = tm.root[tm.root[lane + 32]];
            __syncwarp();
            tm.root[lane] = x0;
            tm.root[lane + 32] = x1;
            __syncwarp();
        }
        int rt[2];
        rt[0] = lane < L ? tm.root[lane] : -1;
        rt[1] = lane + 32 < L ? tm.root[lane + 32] : -1;
        const unsigned e0 = __ballot_sync(kFull, rt[0] == lane), e1 = __ballot_sync(kFull, rt[1] == lane + 32);
        const u64 ends = ((u64)e1 << 32) | e0;
        ns = __popcll(ends);
        // survivor of merge q: rank of its last merge among the last merges
        int sidx[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
            sidx[h] = rt[h] >= 0 ? __popcll(ends & ((1ull << rt[h]) - 1ull)) : -1;
        // merges of survivor s: masks of both halves
        unsigned w0 = 0u, w1 = 0u, g0 = 0u, g1 = 0u, g10 = 0u;
#pragma unroll 1
        for (int s = 0; s < ns; ++s) {
            const unsigned x0 = __ballot_sync(kFull, sidx[0] == s), x1 = __ballot_sync(kFull, sidx[1] == s);
            if (lane == s) {
                w0 = x0;
                w1 = x1;
            }
            if (sidx[0] == s)
                g0 = x0;
            if (sidx[1] == s) {
                g10 = x0;
                g1 = x1;
            }
        }
        const int len = __popc(w0) + __popc(w1);
        int inc = len;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(kFull, inc, off);
            if (lane >= off)
                inc += o;
        }
        const int first = inc - len;
        const unsigned below = (1u << lane) - 1u;
        const int f0 = __shfl_sync(kFull, first, sidx[0] & 31), f1 = __shfl_sync(kFull, first, sidx[1] & 31);
        if (sidx[0] >= 0)
            tm.prog[f0 + __popc(g0 & below)] = lane;
        if (sidx[1] >= 0)
            tm.prog[f1 + __popc(g10) + __popc(g1 & below)] = lane + 32;
        if (lane < ns)
            tm.sfirst[lane] = first;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int q = lane + 32 * h;
            if (rt[h] == q && q < L) {
                tm.sq[sidx[h]] = q;
                tm.sslot[sidx[h]] = tm.mem[tm.mi(q)];
            }
        }
    }
    if (lane == 0) {
        tm.sfirst[ns] = L;
        tm.L = L;
        tm.ns = ns;
    }
    __syncwarp();
    if (lane < ns) {
        const int a = tm.mi(tm.sq[lane]);
#pragma unroll 1
        for (int s = 0; s < ns; ++s)
            tm.C[s][lane] = tm.S[tm.mi(tm.sq[s])][a];
    }
    __syncwarp();
}

// The round's merges by simulate_steps (warp 0, the members' cells in S and
// their minima ready).  For single and centroid linkage, whose merges mostly
// take part in one another, and where the chain (below) breaks off early for
// that reason.  The bounds of the cells outside are weak there (single: a margin
// of the matrix's largest value; centroid: up to a quarter of the height; zeros
// and equal values anywhere), so the merges go on past them, on condition,
// `reach` of them: twice as many as stood the last time (and 2).  They have to be
// as many as the proved ones: the steps take a warp's time, the look some 7 us of a
// round's 35, and some are put off again.  Single linkage, ms, ended at the bounds /
// half as many / as many: n = 5500 on a 1/1024 grid 14.1 / 15.2 / 14.5, n = 16384
// 55.6 / 52.9 / 50.0, n = 9000 conformer-like 42.1 / 13.5 / 14.7, n = 4000 points four
// at a time 58.0 / 16.9 / 16.9; n = 3000 centroid 56.5 / 22.2 / 22.2.
__device__ __noinline__ void simulate(Team &tm, int linkage)
{
    const int lane = threadIdx.x & 31;
    const int reach = tm.reach;
    int L, sure;
    switch (linkage) {
    case 0: simulate_steps<0>(tm, reach, L, sure); break;
    case 1: simulate_steps<1>(tm, reach, L, sure); break;
    case 2: simulate_steps<2>(tm, reach, L, sure); break;
    case 3: simulate_steps<3>(tm, reach, L, sure); break;
    case 4: simulate_steps<4>(tm, reach, L, sure); break;
    default: simulate_steps<5>(tm, reach, L, sure); break;
    }
    const bool tie = L > sure && L - sure >= sure;
    if (!tie) {
        steps_undo(tm, L, sure, sure);
        L = sure;
    }
    unsigned top = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (lane + 32 * h >= sure && lane + 32 * h < L)
            top = max(top, (unsigned)tm.rec[lane + 32 * h].y);
    top = __reduce_max_sync(kFull, top);
    if (lane == 0) {
        tm.tie = tie;
        tm.sure = sure;
        tm.steps = 1;
        tm.cmax = top;
    }
    steps_program(tm, L);
}

// ---- the round's merges where they follow the entries (complete, group and
// weighted average, Ward): the chain of entries that share no member, each
// the next merge of the step-by-step iteration unless a cell made by an
// earlier one comes first.  The chain is taken by bit scans; then every cell
// its merges make between members is computed at once and compared.

// Warp 0: the chain.  Lane q gets the entry of merge q; returns their number.
// A step is a bit scan and one shared-memory read.
__device__ __forceinline__ int chain_select(Team &tm)
{
    const int lane = threadIdx.x & 31;
    unsigned lo, hi;
    {
        bool in[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = lane + 32 * h;
            in[h] = e < tm.ne && tm.ent[e].x != 0xffffu;
            if (in[h]) {
                const unsigned x = tm.ent[e].x;
                const u64 w = tm.em[x & 0xffu] | tm.em[x >> 8];
                tm.enm[e] = make_uint2((unsigned)w, (unsigned)(w >> 32));
            }
            tm.step[e] = 0xff;
        }
        lo = __ballot_sync(kFull, in[0]);
        hi = __ballot_sync(kFull, in[1]);
    }
    __syncwarp();
    int L = 0, mine = 0;
    while ((lo | hi) != 0u && L < kSurv) {
        const int e = lo ? __ffs(lo) - 1 : __ffs(hi) + 31;
        const uint2 w = tm.enm[e];
        lo &= ~w.x;
        hi &= ~w.y;
        mine = lane == L ? e : mine;
        ++L;
    }
    if (lane < L) {
        const uint2 w = tm.ent[mine];
        const int i = (int)(w.x & 0xffu), j = (int)(w.x >> 8);
        tm.rec[lane] = make_int4(i | j << 8, (int)w.y, tm.sz0[i], tm.sz0[j]);
        tm.ce[lane] = (unsigned char)mine;
        tm.step[i] = (unsigned char)lane;
        tm.step[j] = (unsigned char)lane;
    }
    tm.lim[lane] = 0xffffffffu;
    if (lane == 0)
        tm.L = L;
    __syncwarp();
    return L;
}

// Warp q of a team of nw: coefficients of merges q, q + nw, .. and the cells
// X[q][k] they make with every member k (those of later merges included).
template <int LK>
__device__ __forceinline__ void chain_cells_made(Team &tm, int q0, int nw)
{
    const int lane = threadIdx.x & 31;
    const int L = tm.L;
#pragma unroll 1
    for (int q = q0; q < L; q += nw) {
        const int4 rec = tm.rec[q];
        const int i = rec.x & 0xff, j = (rec.x >> 8) & 0xff;
        const float hgt = __int_as_float(rec.y);
        const float4 co = merge_coefs<LK>(rec.z, rec.w, hgt);
        if (LK != 3 && lane == 0)
            tm.co[q] = co;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            const float a = tm.S[k][i], b = tm.S[k][j];
            tm.X[q][k] = LK == 3 ? ward_cell((float)rec.z, (float)rec.w, (float)(rec.z + rec.w), (float)tm.sz0[k],
                                             hgt, a, b)
                                 : lw_sum(co.x, co.y, co.z, co.w, a, b);
        }
    }
}

// Then, for merge q and every later merge p (lane p): the smallest cell that
// merge q made and that is there when p comes (value bits, lim[p] the least
// over q): the cells X[q] to members that no merge takes and to those that
// merges p and later take, and C[q][c], the cell to cluster c after merges q
// and c, for the merges c between.
template <int LK>
__device__ __forceinline__ void chain_limits(Team &tm, int q0, int nw)
{
    const int lane = threadIdx.x & 31;
    const int L = tm.L, m = tm.m;
    const unsigned thv = tm.thv;
#pragma unroll 1
    for (int q = q0; q < L; q += nw) {
        const int4 rq = tm.rec[q];
        unsigned xy = 0xffffffffu, cc = 0xffffffffu, un = 0xffffffffu;
        if (lane > q && lane < L) {
            const int4 rc = tm.rec[lane];
            const float a = tm.X[q][rc.x & 0xff], b = tm.X[q][(rc.x >> 8) & 0xff];
            const float c = merge_cell(tm, LK, lane, a, b, (float)(rq.z + rq.w));
            tm.C[q][lane] = c;
            tm.C[lane][q] = c;
            const unsigned ua = __float_as_uint(a), ub = __float_as_uint(b);
            xy = ua < ub ? ua : ub;
            cc = __float_as_uint(c);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            if (k < m && tm.step[k] == 0xff) {
                const unsigned u = __float_as_uint(tm.X[q][k]);
                un = u < un ? u : un;
            }
        }
        // (cells above the bound of the round never matter)
        if (__any_sync(kFull, xy <= thv || cc <= thv || un <= thv)) {
            un = __reduce_min_sync(kFull, un);
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned y = __shfl_down_sync(kFull, xy, d), z = __shfl_up_sync(kFull, cc, d);
                if (lane + d < 32)
                    xy = y < xy ? y : xy;
                if (lane >= d)
                    cc = z < cc ? z : cc;
            }
            const unsigned z = __shfl_up_sync(kFull, cc, 1);  // the merges before p only
            if (lane > q && lane < L) {
                unsigned v = un < xy ? un : xy;
                v = z < v ? z : v;
                if (v <= thv)
                    atomicMin(&tm.lim[lane], v);
            }
        }
    }
}

// Warp 0: the merges of the chain that the step-by-step iteration takes, lane
// p for merge p.  It has to be smaller than (1) every cell earlier merges made
// between members (lim; equal values end the chain), (2) the cells not listed
// that no earlier merge changed: it comes before the marks that end the rows
// of the members not merged before it, (3) the cells earlier merges made with
// clusters outside.  For (3) there are bounds (see merged_bound); where they
// would cost merges (values tied with the bound of the round, or within its
// margin), the merges that pass (1) and (2) are taken on condition: the cells
// are computed before anything is written, and every CTA is asked whether one
// comes first (tie; only with `allow`).  The first merge is the smallest cell
// of all.
template <int LK>
__device__ __forceinline__ void chain_accept(Team &tm, bool allow)
{
    const int lane = threadIdx.x & 31;
    const int L = tm.L;
    constexpr unsigned kNone = 0xffffffffu;
    unsigned own = 0xffu, made = kNone, un = 0xffu, hb = kNone, e = 0u;
    if (lane < L) {
        const int4 rec = tm.rec[lane];
        const int i = rec.x & 0xff, j = (rec.x >> 8) & 0xff;
        own = min(tm.ex[i], tm.ex[j]);
        e = tm.ce[lane];
        hb = (unsigned)rec.y;
        made = merged_bound<LK>(tm.sl[i].y, tm.sl[j].y, (float)rec.z, (float)(rec.z + rec.w), __int_as_float(rec.y),
                                0u);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = lane + 32 * h;
        if (k < tm.m && tm.step[k] == 0xff)
            un = min(un, (unsigned)tm.ex[k]);
    }
    un = __reduce_min_sync(kFull, un);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_down_sync(kFull, own, d), z = __shfl_up_sync(kFull, made, d);
        if (lane + d < 32)
            own = min(own, y);
        if (lane >= d)
            made = min(made, z);
    }
    const unsigned z = __shfl_up_sync(kFull, made, 1);
    const bool in = lane > 0 && lane < L;
    const unsigned made_first = __ballot_sync(kFull, in && hb >= tm.lim[lane]);
    const unsigned bad = __ballot_sync(kFull, in && e >= min(un, own)) | made_first;
    const unsigned out = __ballot_sync(kFull, in && hb >= z) | bad;
    const int most = bad ? __ffs(bad) - 1 : L, sure = out ? __ffs(out) - 1 : L;
    const bool tie = allow && most >= sure + kTieGain && kTiePart * (most - sure) >= sure;
    const int La = tie ? most : sure;
    if (lane < La) {
        tm.prog[lane] = lane;
        tm.sfirst[lane] = lane;
        tm.sq[lane] = lane;
        tm.cons[lane] = (unsigned char)La;
        tm.sslot[lane] = tm.mem[tm.mi(lane)];
    }
    if (lane == 0) {
        tm.sfirst[La] = La;
        tm.L = La;
        tm.ns = La;
        tm.tie = tie;
        tm.sure = sure;
        tm.steps = 0;
        tm.cmax = La > 0 ? (unsigned)tm.rec[La - 1].y : 0u;
        // a cell made between members comes first: many merges are still known
        tm.redo = most < L && ((made_first >> most) & 1u) && most < kRedoBelow && 2 * most < L + kRedoGap;
    }
    __syncwarp();
}

// The chain's cells, limits and accepted prefix, by team A (the whole CTA in a
// one-CTA job).
template <int NT, bool ONE>
__device__ __noinline__ void chain_phase(Team &tm, int linkage, bool allow)
{
    constexpr int WA = ONE ? NT / 32 : NT / 64, TA = WA * 32;
    const int warp = threadIdx.x >> 5;
    auto sync_a = [&]() {
        if constexpr (ONE)
            __syncthreads();
        else
            asm volatile("barrier.cta.sync.aligned 3, %0;" ::"n"(TA) : "memory");
    };
    switch (linkage) {
    case 1: chain_cells_made<1>(tm, warp, WA); break;
    case 2: chain_cells_made<2>(tm, warp, WA); break;
    case 3: chain_cells_made<3>(tm, warp, WA); break;
    default: chain_cells_made<4>(tm, warp, WA); break;
    }
    sync_a();
    if (linkage == 3)
        chain_limits<3>(tm, warp, WA);
    else
        chain_limits<2>(tm, warp, WA);
    sync_a();
    if (warp == 0) {
        switch (linkage) {
        case 1: chain_accept<1>(tm, allow); break;
        case 4: chain_accept<4>(tm, allow); break;
        default: chain_accept<2>(tm, allow); break;
        }
    }
    sync_a();
}

// Merges on condition: a cell v of row k that merge q made, and that is there
// until merge cons[q] takes its cluster in.  Does it come before one of the
// merges meanwhile that no bound proved?  The first such goes to *viol.
__device__ __noinline__ void outside_check(const Team &tm, int q, unsigned vb, unsigned k, int *viol)
{
    const unsigned x = (unsigned)tm.mem[tm.mi(q)];
    const u64 kA = ((u64)vb << 32) | min(k, x);
    const unsigned kC = max(k, x);
    const int last = min((int)tm.cons[q], tm.L - 1);
#pragma unroll 1
    for (int e = max(q + 1, tm.sure); e <= last; ++e) {
        const int4 rec = tm.rec[e];
        const u64 eA = ((u64)(unsigned)rec.y << 32) | (unsigned)tm.mem[rec.x & 0xff];
        if (eA > kA || (eA == kA && (unsigned)tm.mem[(rec.x >> 8) & 0xff] > kC)) {
            atomicMin(viol, e);
            break;
        }
    }
}

// Merges f + 1 .. f + len - 1 of a survivor's program for row k, whose first
// merge gave v: the new cell after the last one (CHECK: each is checked; a copy of
// its own, the call would cost the others registers).  An operand is a cell in
// memory or the result of an earlier merge of the program, mostly of the one
// just before.
template <bool ONE, bool CHECK>
__device__ __noinline__ float chain_cells(const MergeParams &p, const Team &tm, int f, int len, float v, float nk,
                                          long long k, int sk, bool ok, int *viol)
{
    float tmp[kTeam];
    const bool full = !ONE && p.full;
    const long long bk = row_base(p, k);
    auto load = [&](int a) -> float {
        if (!ok)
            return 0.0f;
        if (full)
            return LDCG(tm.mst[a] >= sk ? p.D + tm.mbase[a] + k : p.TL + tm.mbase[a] + sk);
        const long long x = tm.mem[a];
        return LDCG(p.D + (k > x ? tm.mbase[a] + k : bk + x));
    };
    int prev = tm.prog[f];
#pragma unroll 1
    for (int e = 1; e < len; ++e) {
        const int q = tm.prog[f + e];
        const int x = tm.rec[q].x;
        const int si = ((x >> 16) & 0xff) - 1, sj = ((x >> 24) & 0xff) - 1;
        if (si != prev && sj != prev)
            tmp[prev] = v;
        const float a = si < 0 ? load(x & 0xff) : si == prev ? v : tmp[si];
        const float b = sj < 0 ? load((x >> 8) & 0xff) : sj == prev ? v : tmp[sj];
        v = merge_cell(tm, p.linkage, q, a, b, nk);
        if (CHECK && ok && __float_as_uint(v) <= tm.cmax)
            outside_check(tm, q, __float_as_uint(v), (unsigned)k, viol);
        prev = q;
    }
    return v;
}

// Adds a key to a survivor's list in global memory: every place holds the
// smallest key that came to it, by column; a larger one goes on to a second
// place, and from there to the bound of the keys not listed.  So the smallest
// of many equal values stay (they lie in neighbouring columns), where a list in
// order of arrival runs over with any of them and leaves a bare mark, which
// costs a round without a merge (n = 5000, one value everywhere, Ward: 7029
// rounds, 2300 of them without a merge).
__device__ __forceinline__ void list_add(u64 *list, u64 *ovf, u64 key)
{
    static_assert(kSvList == 64, "places by six bits of the column");
    u64 old = atomicMin(list + ((unsigned)key & 63u), key);
    u64 x = old > key ? old : key;
    if (x == kNoKey)
        return;
    const unsigned c = (unsigned)x;
    old = atomicMin(list + ((c + (c >> 6) + 32u) & 63u), x);
    x = old > x ? old : x;
    if (x != kNoKey)
        atomicMin(ovf, x);
}

// Pieces per row when nexec refill rows are served by G CTAs.
// Long rows: about two per CTA (a CTA with one more than the others holds the
// round up by less; n = 65536 complete: one per CTA 166 ms, two 161).  Shorter
// ones: one (two: n = 8191 2 % slower, each piece pays a reduction).
__device__ __forceinline__ int scan_pieces(int G, int nexec, bool early)
{
    const int np = nexec > 0 ? (early ? 2 : 1) * G / nexec : 1;
    return np < 1 ? 1 : np > kPieces ? kPieces : np;
}

// Entry of the published lists: (value bits << 32) | (row << kRankBits) | rank,
// unique and ordered like (value, row, column).
__device__ __forceinline__ u64 entry_key(u64 cell_key, u64 rowbits, unsigned rank)
{
    return (cell_key & kHi) | rowbits | rank;
}

// The largest key, or one in between, such that lo to hi of the counted ones
// are at or below it (all of them, up to `top`, if they are no more than hi;
// fewer if the keys next to it are too many): gallops from the smallest key
// by way of `guess`, then bisects.  Every thread calls it and gets the same.
template <class F>
__device__ __forceinline__ u64 find_pivot(F &&count, u64 least, u64 top, u64 guess, int lo_n, int hi_n)
{
    if (count(top) <= hi_n)
        return top;
    u64 lo = least, hi = top, step = 1ull << 42;
    u64 mid = guess > lo && guess < hi ? guess : lo + (step < hi - lo ? step : (hi - lo) / 2);
    bool open = true;  // hi not met yet
    while (true) {
        const int c = count(mid);
        if (c > hi_n) {
            hi = mid;
            open = false;
        } else if (c < lo_n) {
            lo = mid;
        } else {
            return mid;
        }
        if (hi - lo <= 1)
            return lo;
        mid = lo + (hi - lo) / 2;
        if (open && lo - least + step < mid - lo) {
            mid = lo + (lo - least) + step;
            step *= 2;
        }
    }
}

// The new cells D(k, survivor) of Section 4 step 3 for the rows l0 .. l0 + rows
// of a CTA outside the round's merges: into kvs (kvs[q * (kSurv + 1) + s]:
// chunk row q, survivor s) and into memory (kStore); with merges on condition
// each is compared with the later merges and goes to kvs only (kKeep: the CTA's
// rows are one chunk) or nowhere (kCheck).  A warp takes 32 rows and up to 4
// survivors at a time from a counter (team B comes in when its scans are
// done): 8 loads in flight per thread; the rows of a warp are consecutive, so
// row cells are read and written in whole lines.
constexpr int kStore = 0, kKeep = 1, kCheck = 2;
template <int NT, bool ONE>
__device__ __forceinline__ void new_cells(const MergeParams &p, Shared<NT, ONE> &sh, int l0, int rows, int ns, int mode)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int b = sh.cx.b, G = ONE ? 1 : sh.cx.G;
    auto rows_at = [&](int l) -> long long {
        return (long long)(ONE ? l : (b + G * (l >> 5)) * kRowBlock + (l & 31));
    };
    constexpr int KVP = kSurv + 1;
    const long long n = p.n;
    const bool full = !ONE && p.full;
    const unsigned *bitmap = sh.cx.bitmap, *touched = sh.cx.touched;
    float *kvs = sh.cx.kvs;
    const int *rsize = sh.cx.rsize, *rstamp = sh.cx.rstamp;
    const int nblk = rows / 32;
    int *const viol = mode != kStore ? &sh.viol : nullptr;
    constexpr int U = 4;  // (8: 6 % slower at n = 1968 and 16384, twice the instructions)
    // (fewer survivors at a time when that leaves no warp without an item)
    int ug = U;
    while (ug > 2 && nblk * ((ns + ug / 2 - 1) / (ug / 2)) <= NT / 32)
        ug /= 2;
    const int ng = (ns + ug - 1) / ug;
    // (a warp takes the next item: team B comes in when its scans are done)
    const int nit = nblk * ng;
    while (true) {
        int it = 0;
        if (lane == 0)
            it = atomicAdd(&sh.item, 1);
        it = __shfl_sync(kFull, it, 0);
        if (it >= nit)
            break;
        const int blk = it % nblk, s0 = (it / nblk) * ug;
        const int l = l0 + blk * 32 + lane;
        const long long k = rows_at(l);
        const bool ok = k < n && live(bitmap, k) && !live(touched, k);
        const unsigned okb = __ballot_sync(kFull, ok);
        if (s0 == 0 && lane == 0)
            sh.okm[blk] = okb;
        if (okb == 0)
            continue;
        const float nk = (float)rsize[l];
        const long long bk = row_base(p, k);
        const int sk = full ? rstamp[l] : 0;
        const unsigned bhi = (unsigned)(sh.cx.cB[l] >> 32);
        unsigned hm = 0u;
        // cell (k, member): packed, row x for k > x (consecutive k of a
        // warp read consecutive words) and row k for k < x; row-log
        // layout, row x of M when x was stamped no earlier than k, else
        // x's log at k's stamp (words of one contiguous range)
        auto cell = [&](int a) -> const float * {
            if (full)
                return sh.tm.mst[a] >= sk ? p.D + sh.tm.mbase[a] + k : p.TL + sh.tm.mbase[a] + sk;
            const long long x = sh.tm.mem[a];
            return p.D + (k > x ? sh.tm.mbase[a] + k : bk + x);
        };
        float va[U], vb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = s0 + u;
            va[u] = 0.0f;
            vb[u] = 0.0f;
            if (u < ug && s < ns && ok) {
                const int q = sh.tm.prog[sh.tm.sfirst[s]];
                const int x = sh.tm.rec[q].x;
                va[u] = LDCG(cell(x & 0xff));
                vb[u] = LDCG(cell((x >> 8) & 0xff));
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = s0 + u;
            if (u >= ug || s >= ns)
                break;
            const int f = sh.tm.sfirst[s], len = sh.tm.sfirst[s + 1] - f;
            const int q = sh.tm.prog[f];
            float v = merge_cell(sh.tm, p.linkage, q, va[u], vb[u], nk);
            if (viol && ok && __float_as_uint(v) <= sh.tm.cmax)
                outside_check(sh.tm, q, __float_as_uint(v), (unsigned)k, viol);
            if (len > 1)
                v = viol ? chain_cells<ONE, true>(p, sh.tm, f, len, v, nk, k, sk, ok, viol)
                         : chain_cells<ONE, false>(p, sh.tm, f, len, v, nk, k, sk, ok, viol);
            if (ok && mode != kCheck) {
                const long long x = sh.tm.sslot[s];
                kvs[(size_t)(blk * 32 + lane) * KVP + s] = v;
                if (x > k && __float_as_uint(v) <= bhi)
                    hm |= 1u << s;
                if (mode == kKeep) {
                    // (written when every merge stands)
                } else if (full) {
                    // row x is rewritten whole; row k keeps its stale copy
                    // and the new value goes to k's log (below)
                    STCG(p.D + x * p.pitch + k, v);
                } else {
                    STCG(p.D + (k > x ? row_base(p, x) + k : bk + x), v);
                }
            }
        }
        if (hm != 0u)
            atomicOr(&sh.hit[blk * 32 + lane], hm);
    }
}

// Merges taken on condition (the whole CTA, out of line: rounds without such
// merges do not pay for it): the new cells first; every CTA looks whether one
// of its own comes before a merge of the round that no bound proved, and
// barrier 3 tells the first such, V.  Merges from V on wait for another round.
// Returns 1 if the new cells are in kvs and in memory already, -1 if a wait ran
// out.
template <int NT, bool ONE>
__device__ __noinline__ int settle(const MergeParams &p, Shared<NT, ONE> &sh, int par, unsigned &epoch3)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = sh.cx.b, G = ONE ? 1 : sh.cx.G;
    auto row_of = [&](int l) -> long long {
        return (long long)(ONE ? l : (b + G * (l >> 5)) * kRowBlock + (l & 31));
    };
    constexpr int W = NT / 32, KVP = kSurv + 1;
    Team &tm = sh.tm;
    const int R = sh.cx.R, CH = p.chunk;
    unsigned *touched = sh.cx.touched;
    const bool full = !ONE && p.full, one_chunk = sh.cx.Rmax <= CH;
    const int L = tm.L, ns = tm.ns;
#pragma unroll 1
    for (int l0 = 0; l0 < R; l0 += CH) {
        new_cells(p, sh, l0, R - l0 < CH ? R - l0 : CH, ns, one_chunk ? kKeep : kCheck);
        __syncthreads();
        if (l0 + CH < R) {
            if (tid == 0)
                sh.item = 0;
            __syncthreads();
        }
    }
    if (!ONE) {
        if (tid == 0 && sh.viol < L)
            atomicMax(p.bar + kViol + par, (unsigned)(kTeam - sh.viol));
        grid_arrive(p, p.bar + kBar3, epoch3);
        if (!grid_wait(p, p.bar + kBar3, epoch3, sh))
            return -1;
        if (tid == 0)
            sh.viol = kTeam - ld_relaxed_s32(reinterpret_cast<const int *>(p.bar + kViol + par));
        __syncthreads();
    }
    const int V = sh.viol < L ? sh.viol : L;
    if (V == L && one_chunk) {
#pragma unroll 1
        for (int it = warp; it < R / 32 * ns; it += W) {
            const int blk = it / ns, s = it % ns;
            const int l = blk * 32 + lane;
            const long long k = row_of(l), x = tm.sslot[s];
            if ((sh.okm[blk] >> lane) & 1u)
                STCG(full ? p.D + x * p.pitch + k : p.D + (k > x ? row_base(p, x) + k : row_base(p, k) + x),
                     sh.cx.kvs[(size_t)l * KVP + s]);
        }
        if (tid == 0 && tm.steps)
            tm.reach = min(max(2 * (V - tm.sure) + 2, 4), kSurv);
        return 1;
    }
    sh.hit[tid] = 0u;
    if (V < L) {
#pragma unroll 1
        for (int q = V + tid; q < L; q += NT) {
            const int x = tm.mem[tm.mi(q)], y = tm.mem[tm.mj(q)];
            atomicAnd(&touched[x >> 5], ~(1u << (x & 31)));
            atomicAnd(&touched[y >> 5], ~(1u << (y & 31)));
        }
        __syncthreads();
        // (a slot may take part in merges of both sides)
#pragma unroll 1
        for (int q = tid; q < V; q += NT) {
            const int x = tm.mem[tm.mi(q)], y = tm.mem[tm.mj(q)];
            atomicOr(&touched[x >> 5], 1u << (x & 31));
            atomicOr(&touched[y >> 5], 1u << (y & 31));
        }
        if (tm.steps) {
            if (warp == 0) {
                steps_undo(tm, L, V, tm.sure);
                steps_program(tm, V);
            }
        } else if (tid == 0) {
            tm.sfirst[V] = V;
            tm.L = V;
            tm.ns = V;
        }
    }
    if (tid == 0) {
        sh.item = 0;
        if (tm.steps)
            tm.reach = min(max(2 * (V - tm.sure) + 2, 4), kSurv);
    }
    __syncthreads();
    return 0;
}

// The record for round rr: this CTA's kPub smallest entries (cached keys and
// bound marks of its rows) and its refill requests of round rr - 1.  Also lists
// the refills to install in round rr (served in round rr - 1).
template <int NT, bool ONE>
__device__ __forceinline__ void publish(const MergeParams &p, Shared<NT, ONE> &sh, int rr)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = sh.cx.b, G = ONE ? 1 : sh.cx.G;
    auto rows_at = [&](int l) -> long long {
        return (long long)(ONE ? l : (b + G * (l >> 5)) * kRowBlock + (l & 31));
    };
    constexpr int W = NT / 32;
    const int R = sh.cx.R;
    const long long Rmax = sh.cx.Rmax;
    const u64 *ck = sh.cx.ck, *cB = sh.cx.cB;
    const unsigned char *ccnt = sh.cx.ccnt;
    const int *pend_t = sh.cx.pend_t;
    auto slot_of = [&](long long r) -> int { return (int)(((unsigned)r / kRowBlock / (unsigned)G) * kRowBlock + ((unsigned)r & 31u)); };
    RecA *rec = p.recA + (size_t)(rr & 1) * G + b;
    // a pivot that takes in at least kPub rows' first entries, then the
    // entries up to it in order by counting
    u64 head = kNoKey;
#pragma unroll 1
    for (int l = tid; l < R; l += NT) {
        const int c = ccnt[l];
        const u64 B = cB[l];
        if (c > 0 || B != kNoKey) {
            const u64 e = entry_key(c > 0 ? ck[l] : B, (u64)rows_at(l) << kRankBits, 0);
            head = e < head ? e : head;
        }
        if (rr >= 2 && pend_t[l] == rr - 2) {
            const int s2 = atomicAdd(&sh.ninst, 1);
            sh.inst_slot[s2] = l;
        }
    }
    auto entry_at = [&](int l, int q, int c, u64 &e) -> u64 {
        const u64 x = q < c ? ck[(size_t)q * Rmax + l] : cB[l];
        e = x == kNoKey ? kNoKey : entry_key(x, (u64)rows_at(l) << kRankBits, q);
        return x;
    };
    if (R > 4 * NT) {
        // (a CTA of few threads with very many rows: the entries behind few
        // heads could outnumber kCand)
        u64 Lst[kPub];
#pragma unroll
        for (int q = 0; q < kPub; ++q)
            Lst[q] = kNoKey;
#pragma unroll 1
        for (int l = tid; l < R; l += NT) {
            const int c = ccnt[l];
#pragma unroll 1
            for (int q = 0; q <= c; ++q) {
                u64 e;
                entry_at(l, q, c, e);
                if (e < Lst[kPub - 1])
                    list_insert_n(Lst, e);
            }
        }
        block_topk(Lst, sh);
        if (tid < kPub) {
            const u64 key = sh.tko[tid];
            unsigned col = 0;
            if (key != kNoKey) {
                const int l = slot_of((long long)((unsigned)key >> kRankBits));
                const int q = (int)((unsigned)key & kRankMask);
                col = q < ccnt[l] ? (unsigned)ck[(size_t)q * Rmax + l] : kRowStop | (unsigned)cB[l];
                if (tid == kPub - 1)
                    col |= kHardStop;
            }
            STCG(&rec->key[tid], key);
            STCG(&rec->col[tid], col);
        }
    } else {
        {
            const u64 x = warp_u64_min(head);
            if (lane == 0)
                sh.wmin[warp][0] = x;
        }
        if (tid == 0)
            sh.ncand = 0;
        __syncthreads();
        const u64 gmin = warp_u64_min(lane < W ? sh.wmin[lane][0] : kNoKey);
        auto count = [&](u64 x) -> int { return __syncthreads_count(head <= x && head != kNoKey); };
        const u64 pivot = find_pivot(count, gmin, kNoKey, sh.ppivot, kPub, 3 * kPub);
        int have = 0;
        if (head <= pivot && head != kNoKey) {
#pragma unroll 1
            for (int l = tid; l < R; l += NT) {
                const int c = ccnt[l];
#pragma unroll 1
                for (int q = 0; q <= c; ++q) {
                    u64 e;
                    entry_at(l, q, c, e);
                    have += e <= pivot && e != kNoKey;
                }
            }
        }
        int at = have;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(kFull, at, off);
            if (lane >= off)
                at += o;
        }
        {
            int base = 0;
            if (lane == 31 && at > 0)
                base = atomicAdd(&sh.ncand, at);
            base = __shfl_sync(kFull, base, 31);
            at = base + at - have;
        }
        if (have > 0) {
#pragma unroll 1
            for (int l = tid; l < R; l += NT) {
                const int c = ccnt[l];
#pragma unroll 1
                for (int q = 0; q <= c; ++q) {
                    u64 e;
                    const u64 x = entry_at(l, q, c, e);
                    if (e == kNoKey || e > pivot)
                        break;
                    if (at < kCand) {
                        sh.ckey[at] = e;
                        sh.ccol[at] = q < c ? (unsigned)x : kRowStop | (unsigned)x;
                    }
                    ++at;
                }
            }
        }
        __syncthreads();
        if (tid == 0)
            sh.ppivot = pivot;
        // (at most 3 * kPub threads of 4 rows and K + 1 entries each: they fit)
        static_assert(3 * kPub * 4 * (K + 1) <= kCand, "published entries fit");
        const int N = sh.ncand < kCand ? sh.ncand : kCand;
#pragma unroll 1
        for (int c0 = (tid >> 5) * 8; c0 < N; c0 += NT / 4) {
            const int c = c0 + (lane >> 2);
            const u64 key = c < N ? sh.ckey[c] : kNoKey;
            int rank = 0;
#pragma unroll 1
            for (int f = lane & 3; f < N; f += 4)
                rank += sh.ckey[f] < key;
            rank += __shfl_xor_sync(kFull, rank, 1);
            rank += __shfl_xor_sync(kFull, rank, 2);
            if (c < N && (lane & 3) == 0 && rank < kPub) {
                STCG(&rec->key[rank], key);
                // (more entries may follow the last: none is published)
                STCG(&rec->col[rank], sh.ccol[c] | (rank == kPub - 1 ? kHardStop : 0u));
            }
        }
        if (tid >= N && tid < kPub) {
            STCG(&rec->key[tid], kNoKey);
            STCG(&rec->col[tid], 0u);
        }
    }
    if (tid == 0) {
        const int par = (rr - 1) & 1;
        int nq = rr >= 1 ? sh.nmyreq[par] : 0;
        nq = nq < kReqPerCta ? nq : kReqPerCta;
        if (rr >= 1)
            sh.nmyreq[par] = nq;
        int rows[kReqPerCta];
#pragma unroll
        for (int q = 0; q < kReqPerCta; ++q)
            rows[q] = q < nq ? (int)rows_at(sh.myreq_l[par][q]) : -1;
        uint4 *dst = reinterpret_cast<uint4 *>(&rec->nreq);
        STCG(dst + 0, make_uint4((unsigned)nq, (unsigned)rows[0], (unsigned)rows[1], (unsigned)rows[2]));
        STCG(dst + 1, make_uint4((unsigned)rows[3], (unsigned)rows[4], (unsigned)rows[5], (unsigned)rows[6]));
        STCG(dst + 2, make_uint4((unsigned)rows[7], sh.tm.dmax, 0u, 0u));
    }
}

// All n - 1 merges of one job, run by CTA b of the job's G CTAs (every CTA
// of the job calls this with the same p).  smem_raw: merge_smem_bytes(n, G)
// bytes of dynamic shared memory.
template <int NT, bool ONE>
__device__ void merge_job(const MergeParams &p, const int b, unsigned char *smem_raw, Shared<NT, ONE> &sh)
{
    constexpr int W = NT / 32;
    // the team that selects the round's merges (warps 0 .. WA - 1: all of them in
    // a one-CTA job); the other half of a grid's CTA installs and serves refills
    // beside it
    constexpr int WA = ONE ? W : W / 2, TA = WA * 32;
    constexpr int P = K + 1;  // one-CTA job: keys kept per survivor
    constexpr int KVP = kSurv + 1;
    const long long n = p.n;
    const int G = ONE ? 1 : p.G;
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const long long nb = (n + kRowBlock - 1) / kRowBlock;      // row blocks
    const long long my_blocks = b < nb ? (nb - b + G - 1) / G : 0;
    const int R = (int)(my_blocks * kRowBlock);                 // owned row slots
    const long long Rmax = ((nb + G - 1) / G) * kRowBlock;
    const long long nwords = (n + 31) / 32;
    const int CH = p.chunk;                                     // rows per chunk of the apply pass
    const bool full = !ONE && p.full;
    const int refill_at = n <= kRefillEarlyN ? 1 : 0;
    const bool early = !ONE && n > kRefillEarlyN;  // team B scans beside the selection as well

    // dynamic shared memory: liveness bitmap; slots touched by the round's
    // merges; the published entries of every CTA; per owned slot l: cache
    // keys (key q of slot l at ck[q * Rmax + l]: consecutive threads read
    // consecutive words), bound, size, rescan list, pending refill (round,
    // list position), stamp, key count; the new cells of one chunk of rows
    // (their addresses are kept in shared memory too: as registers they would be
    // live all through the round loop)
    if (threadIdx.x == 0) {
        unsigned char *q0 = smem_raw;
        auto &cx = sh.cx;
        cx.bitmap = reinterpret_cast<unsigned *>(q0);
        q0 += (nwords * 4 + 15) & ~15LL;
        cx.touched = reinterpret_cast<unsigned *>(q0);
        q0 += (nwords * 4 + 15) & ~15LL;
        cx.wkey = reinterpret_cast<u64 *>(q0);
        q0 += ONE ? 0 : (size_t)G * kPub * 8;
        cx.ck = reinterpret_cast<u64 *>(q0);
        q0 += (size_t)Rmax * K * 8;
        cx.cB = reinterpret_cast<u64 *>(q0);
        q0 += (size_t)Rmax * 8;
        cx.wcol = reinterpret_cast<unsigned *>(q0);
        q0 += ONE ? 0 : (size_t)G * kPub * 4;
        cx.kvs = reinterpret_cast<float *>(q0);  // kvs[q * KVP + s]: chunk row q, survivor s
        q0 += (size_t)CH * KVP * 4;
        cx.rsize = reinterpret_cast<int *>(q0);
        cx.rlist = cx.rsize + Rmax;
        q0 += (size_t)Rmax * 8;
        cx.pend_t = reinterpret_cast<int *>(q0);
        cx.pend_s = cx.pend_t + Rmax;
        cx.rstamp = cx.pend_s + Rmax;  // row-log layout: each owned row's stamp
        q0 += ONE ? 0 : (size_t)Rmax * 12;
        cx.ccnt = q0;
        cx.Rmax = Rmax;
        cx.R = R;
        cx.b = b;
        cx.G = G;
    }
    __syncthreads();
    unsigned *const &bitmap = sh.cx.bitmap, *const &touched = sh.cx.touched, *const &wcol = sh.cx.wcol;
    u64 *const &wkey = sh.cx.wkey, *const &ck = sh.cx.ck, *const &cB = sh.cx.cB;
    float *const &kvs = sh.cx.kvs;
    int *const &rsize = sh.cx.rsize, *const &rlist = sh.cx.rlist, *const &pend_t = sh.cx.pend_t;
    int *const &pend_s = sh.cx.pend_s, *const &rstamp = sh.cx.rstamp;
    unsigned char *const &ccnt = sh.cx.ccnt;

    auto row_of = [&](int l) -> long long {
        return (long long)(ONE ? l : (b + G * (l >> 5)) * kRowBlock + (l & 31));
    };
    auto owner_of = [&](long long r) -> int { return ONE ? 0 : (int)((unsigned)r / kRowBlock % (unsigned)G); };
    auto slot_of = [&](long long r) -> int {
        return ONE ? (int)r : (int)(((unsigned)r / kRowBlock / (unsigned)G) * kRowBlock + ((unsigned)r & 31u));
    };
    auto cache_load = [&](u64 (&L)[K], int l) {
#pragma unroll
        for (int q = 0; q < K; ++q)
            L[q] = ck[(size_t)q * Rmax + l];
    };
    auto cache_store = [&](int l, const u64 *L) {
#pragma unroll
        for (int q = 0; q < K; ++q)
            ck[(size_t)q * Rmax + l] = L[q];
    };
    // a refill request for slot l in round r (list par = r & 1)
    auto request = [&](int l, int r) {
        const int par = r & 1;
        const int q = atomicAdd(&sh.nmyreq[par], 1);
        if (q < kReqPerCta) {
            sh.myreq_l[par][q] = l;
            pend_t[l] = r;
        }
    };

    // per-phase wall-clock totals of this CTA (thread 0), when timing is on
    auto &ty = sh.ty;
    if (tid == 0) {
#pragma unroll 1
        for (int q = 0; q < 6; ++q)
            ty.ph[q] = 0;
#pragma unroll 1
        for (int q = 0; q < 8; ++q)
            ty.xs[q] = 0;
        ty.xscan[0] = ty.xscan[1] = ty.tmark = 0;
        ty.fills = ty.installs = ty.rounds = ty.idle = ty.walk = ty.rescans = 0;
    }
    // (the whole of warp 0, every lane with the same values: a branch on the
    // thread index would leave lane 0 running apart from its warp)
    auto lap = [&](u64 &acc) {
        if (p.timing && warp == 0) {
            const u64 now = __shfl_sync(kFull, global_ns(), 0);
            const u64 was = ty.tmark, sum = acc;
            __syncwarp();
            acc = sum + (now - was);
            ty.tmark = now;
            __syncwarp();
        }
    };

    long long st_fill_cells = 0, st_resc_cells = 0;

    // ---- setup
    sh.hit[tid] = 0u;
#pragma unroll 1
    for (long long w = tid; w < nwords; w += NT) {
        const long long live_n = n - w * 32;
        bitmap[w] = live_n >= 32 ? 0xffffffffu : ((1u << live_n) - 1u);
        touched[w] = 0u;
    }
#pragma unroll 1
    for (int l = tid; l < R; l += NT) {
        rsize[l] = 1;
        if (!ONE) {
            pend_t[l] = -1;
            rstamp[l] = -1;
        }
    }
#pragma unroll 1
    for (long long r = (long long)b * NT + tid; r < n; r += (long long)G * NT) {
        STCG(p.size_g + r, 1);
        if (full)
            STCG(p.stamp + r, -1);
    }
    if (!ONE && b == 0) {
#pragma unroll 1
        for (int q = tid; q < 2 * kSurv * (kSvList + 1); q += NT)
            STCG(p.svlist + q, kNoKey);  // (svovf behind it)
    }
    if (tid == 0) {
        sh.ninst = 0;
        sh.npieces = 1;
        sh.nexec = 0;
        sh.nmyreq[0] = 0;
        sh.nmyreq[1] = 0;
        sh.nps = 0;
        sh.nptouch = 0;
        sh.nresc = 0;
        sh.tm.dmax = 0u;
        sh.tm.reach = 4;
        sh.pivot = 0ull;
        sh.ppivot = 0ull;
        sh.limit = sh.width = 0u;
    }
    __syncthreads();

    // ---- phase 0: validate the matrix and fill the caches of owned rows
    // (one warp per owned row; the rows of a CTA are spread over the whole
    // triangle, so every CTA reads about the same number of cells)
    {
        int bad = 0;
        unsigned mx = 0u;
#pragma unroll 1
        for (int l = warp; l < R; l += W) {
            const long long r = row_of(l);
            u64 top[K], next = kNoKey;
#pragma unroll
            for (int q = 0; q < K; ++q)
                top[q] = kNoKey;
            if (r < n - 1)
                warp_row_topk(p, r, top, next, bad, mx);
            if (lane == 0) {
                cache_store(l, top);
                ccnt[l] = (unsigned char)list_count(top);
                cB[l] = next;
            }
        }
        if (bad)
            atomicCAS(p.status, 0, kErrInput);
        mx = __reduce_max_sync(kFull, mx);
        if (lane == 0)
            atomicMax(&sh.tm.dmax, mx);
    }
    __syncthreads();
    unsigned epoch = 0, epoch2 = 0, epoch3 = 0;
    if (p.timing && tid == 0)
        ty.tmark = global_ns();

    long long t = 0;   // merges done
    const long long max_rounds = 2 * n + 64;
#pragma unroll 1
    for (int r = 0;; ++r) {
        const int par = r & 1;
        if (r > max_rounds) {
            // no progress: a stop mark that no refill lifts (every CTA sees the
            // same count and leaves here together)
            if (tid == 0)
                atomicCAS(p.status, 0, kErrInternal);
            return;
        }
        if (!ONE) {
            publish(p, sh, r);
            lap(ty.ph[5]);
            if (b == p.skip_arrive_cta)
                return;
            grid_arrive(p, p.bar, epoch);
            if (!grid_wait(p, p.bar, epoch, sh))
                return;
            lap(ty.ph[0]);
        }
        if (r == 0) {
            // (the input's check)
            if (tid == 0)
                sh.flag = ld_relaxed_s32(p.status);
            __syncthreads();
            if (sh.flag != 0)
                return;
        }
        if (tid == 0) {
            sh.nmyreq[par] = 0;
            sh.ncand = 0;
            sh.svsum = 0;
        }

        // ---- every CTA's published entries and refill requests
        if (!ONE) {
            const RecA *recs = p.recA + (size_t)par * G;
            int rcnt = 0;
            int rq[kReqPerCta];
#pragma unroll
            for (int q = 0; q < kReqPerCta; ++q)
                rq[q] = -1;
            if (tid < G) {
                const uint4 *src = reinterpret_cast<const uint4 *>(&recs[tid].nreq);
                const uint4 w3 = LDCG(src), w4 = LDCG(src + 1), w5 = LDCG(src + 2);
                rcnt = (int)w3.x;
                rq[0] = (int)w3.y;
                rq[1] = (int)w3.z;
                rq[2] = (int)w3.w;
                rq[3] = (int)w4.x;
                rq[4] = (int)w4.y;
                rq[5] = (int)w4.z;
                rq[6] = (int)w4.w;
                rq[7] = (int)w5.x;
                if (r == 0)
                    atomicMax(&sh.tm.dmax, w5.y);
            }
            // keys and column words, entry q of CTA g at [q * G + g]
            constexpr int KW = kPub / 2, CW = kPub / 4;  // 16-byte words of both
#pragma unroll 1
            for (int w = tid; w < (KW + CW) * G; w += NT) {
                const int g = w / (KW + CW), part = w % (KW + CW);
                const uint4 v = LDCG(reinterpret_cast<const uint4 *>(recs + g) + part);
                if (part < KW) {
                    wkey[(2 * part) * G + g] = ((u64)v.y << 32) | v.x;
                    wkey[(2 * part + 1) * G + g] = ((u64)v.w << 32) | v.z;
                } else {
                    const int q = 4 * (part - KW);
                    wcol[q * G + g] = v.x;
                    wcol[(q + 1) * G + g] = v.y;
                    wcol[(q + 2) * G + g] = v.z;
                    wcol[(q + 3) * G + g] = v.w;
                }
            }
            exchange_requests(rcnt, rq, b, sh, par ^ 1, pend_t, pend_s);
            lap(ty.xs[5]);
        }
        epoch2 += 1;

        if (!ONE) {
            // ---- the caches of the previous round's survivors: every cell of a
            // survivor's row below that round's limit is in its list (those pushed
            // out of it: not below svovf) or among the cells to other survivors
            const int nsv = sh.nps;
#pragma unroll 1
            for (int s = warp; s < nsv; s += W) {
                const size_t at = (size_t)(par ^ 1) * kSurv + s;
                const u64 ovf = LDCG(p.svovf + at);
                const ulonglong2 y2 = LDCG(reinterpret_cast<const ulonglong2 *>(p.svlist + at * kSvList) + lane);
                u64 B = kNoKey;
                u64 x = y2.x, x2 = y2.y;
                const int cnt = __popc(__ballot_sync(kFull, x != kNoKey)) + __popc(__ballot_sync(kFull, x2 != kNoKey));
                // (C still holds the previous round's)
                u64 x3 = kNoKey;
                if (lane < nsv && sh.pslot[lane] > sh.pslot[s])
                    x3 = make_key(sh.tm.C[s][lane], (unsigned)sh.pslot[lane]);
                if (lane == 0)
                    B = ovf;
                else if (lane == 1)
                    B = sh.limit == 0xffffffffu ? kNoKey : (u64)sh.limit << 32;
                B = warp_u64_min(B);
                int c = 0;
#pragma unroll 1
                for (int q = 0; q <= K; ++q) {
                    u64 y = x < x2 ? x : x2;
                    y = x3 < y ? x3 : y;
                    y = warp_u64_min(y);
                    x = x == y ? kNoKey : x;
                    x2 = x2 == y ? kNoKey : x2;
                    x3 = x3 == y ? kNoKey : x3;
                    if (q < K) {
                        if (lane == 0)
                            sh.svk[s][q] = y < B ? y : kNoKey;
                        c += y < B;
                    } else {
                        B = y < B ? y : B;
                    }
                }
                if (lane == 0) {
                    atomicAdd(&sh.svsum, cnt < 8 ? cnt : 8);
                    sh.svB[s] = B;
                    sh.svc[s] = c;
                    const long long row = sh.pslot[s];
                    if (owner_of(row) == b) {
                        const int l = slot_of(row);
                        cache_store(l, sh.svk[s]);
                        ccnt[l] = (unsigned char)c;
                        cB[l] = B;
                        if (c <= kSurvivorRefillAt && B != kNoKey)
                            request(l, r);
                    }
                }
            }
            // ---- refills served in the previous round: take the row's list,
            // then replay that round's merges (the scan ran before them, or
            // while they were being written)
            const int ninst = sh.ninst;
            const int ipar = par ^ 1;
            const int inp = sh.npieces;  // pieces per row of the previous round
            const int nps = sh.nps;
#pragma unroll 1
            for (int s2 = W - 1 - warp; s2 < ninst; s2 += W) {
                const int l = sh.inst_slot[s2];
                const int pos = pend_s[l];
                const long long row = row_of(l);
                // (one key per lane, kPartWords lanes per piece, then the K smallest
                // of them; B, a lower bound of the row's other cells)
                u64 M[K], B;
                {
                    const int q1 = lane % kPartWords;
                    u64 x = kNoKey;
                    if (lane < inp * kPartWords && q1 <= K)
                        x = LDCG(p.parts + ((size_t)ipar * kMaxReq + pos) * kPieces * kPartWords + lane);
                    u64 y = q1 < K ? x : kNoKey;
#pragma unroll
                    for (int q = 0; q < K; ++q) {
                        M[q] = warp_u64_min(y);
                        y = y == M[q] ? kNoKey : y;
                    }
                    B = warp_u64_min(q1 == K ? x : y);
                }
                // the new cells (row, survivor) of the previous round, one lane each
                const long long base = row_base(p, row);  // cell (row, c) at base + c
                u64 xr = kNoKey;
                if (lane < nps) {
                    const long long ia = sh.pslot[lane];
                    if (ia > row)
                        xr = make_key(LDCG(full ? p.D + ia * p.pitch + row : p.D + base + ia), (unsigned)ia);
                }
                // keys whose column a merge of that round retired or rewrote go
#pragma unroll
                for (int q = 0; q < K; ++q)
                    if (M[q] != kNoKey && live(touched, (unsigned)M[q]))
                        M[q] = kNoKey;
                sort_list(M);
                int c = list_count(M);
#pragma unroll 1
                for (unsigned w = __ballot_sync(kFull, xr < B); w; w &= w - 1) {
                    const u64 x = __shfl_sync(kFull, xr, __ffs(w) - 1);
                    if (x < B) {
                        const u64 out = list_insert(M, x);
                        if (c == K)
                            B = out;
                        else
                            ++c;
                    }
                }
                if (lane == 0) {
                    cache_store(l, M);
                    ccnt[l] = (unsigned char)c;
                    cB[l] = B;
                    pend_t[l] = -1;
                }
            }
            if (tid == TA)
                ty.installs += ninst;
            __syncthreads();
        }
        // (the previous round's bits; the selection's barriers follow)
#pragma unroll 1
        for (int q = tid; q < sh.nptouch; q += NT)
            atomicAnd(&touched[sh.ptouch[q] >> 5], ~(1u << (sh.ptouch[q] & 31)));
        lap(ty.xs[0]);

        // Team A's barrier (the whole CTA in a one-CTA job).
        auto sync_a = [&]() {
            if constexpr (ONE)
                __syncthreads();
            else
                asm volatile("barrier.cta.sync.aligned 3, %0;" ::"n"(TA) : "memory");
        };
        // The selection's threads: the whole CTA, or (long rows: their scans take
        // longer than the rest of a round, so team B begins at once) team A.
        const int TS = early ? TA : NT;
        auto sync_s = [&]() {
            if constexpr (ONE)
                __syncthreads();
            else
                asm volatile("barrier.cta.sync.aligned 5, %0;" ::"r"(TS) : "memory");
        };
        auto count_s = [&](bool x) -> int {
            if constexpr (ONE) {
                return __syncthreads_count(x);
            } else {
                unsigned c;
                asm volatile("{ .reg .pred q; setp.ne.u32 q, %1, 0; barrier.cta.red.popc.aligned.u32 %0, 5, %2, q; }"
                             : "=r"(c)
                             : "r"((unsigned)x), "r"(TS)
                             : "memory");
                return (int)c;
            }
        };
        int bad = 0;
        if (!early || warp < WA) {
            // ---- selection: a pivot such that the entries up to it number some
            // fifty to a hundred.  A thread's head is its smallest entry.
            {
                u64 head = kNoKey, hard = kNoKey;
                if (ONE) {
#pragma unroll 1
                    for (int l = tid; l < R; l += TS) {
                        const int c = ccnt[l];
                        const u64 B = cB[l];
                        if (c > 0 || B != kNoKey) {
                            const u64 e = entry_key(c > 0 ? ck[l] : B, (u64)l << kRankBits, 0);
                            head = e < head ? e : head;
                        }
                    }
                } else {
#pragma unroll 1
                    for (int g = tid; g < G; g += TS) {
                        const u64 x = wkey[g], y = wkey[(kPub - 1) * G + g];  // (a list that is full may go on)
                        head = x < head ? x : head;
                        hard = y < hard ? y : hard;
                    }
                }
                // survivors' heads (every warp counts them itself)
                u64 svh = kNoKey;
                const int nps = ONE ? 0 : sh.nps;
                if (lane < nps && (sh.svc[lane] > 0 || sh.svB[lane] != kNoKey))
                    svh = entry_key(sh.svc[lane] > 0 ? sh.svk[lane][0] : sh.svB[lane],
                                    (u64)sh.pslot[lane] << kRankBits, 0);
                {
                    const u64 x = warp_u64_min(head), y = warp_u64_min(hard);
                    if (lane == 0) {
                        sh.wmin[warp][0] = x;
                        sh.wmin[warp][1] = y;
                    }
                }
                sync_s();
                u64 gmin = warp_u64_min(32 * lane < TS ? sh.wmin[lane][0] : kNoKey);
                hard = warp_u64_min(32 * lane < TS ? sh.wmin[lane][1] : kNoKey);
                const u64 sv = warp_u64_min(svh);
                gmin = sv < gmin ? sv : gmin;
                auto count = [&](u64 x) -> int {
                    return count_s(head <= x && head != kNoKey) +
                           (ONE ? 0 : __popc(__ballot_sync(kFull, svh <= x && svh != kNoKey)));
                };
                u64 pivot = hard;
                int want = kHeadsHi;
                while (true) {
                    pivot = find_pivot(count, gmin, hard, sh.pivot, want * 5 / 8, want);
                    // every entry up to the pivot: counted per thread, placed by a
                    // scan of the warp and one addition per warp
                    int have = 0, svn = 0;
                    const bool svw = !ONE && 32 * (warp + 1) == TS;
                    if (head <= pivot && head != kNoKey) {
                        if (ONE) {
#pragma unroll 1
                            for (int l = tid; l < R; l += TS) {
                                const int cc = ccnt[l];
                                const u64 B = cB[l];
                                const u64 rowbits = (u64)l << kRankBits;
#pragma unroll 1
                                for (int q = 0; q < cc; ++q)
                                    have += entry_key(ck[(size_t)q * Rmax + l], rowbits, q) <= pivot;
                                have += B != kNoKey && entry_key(B, rowbits, cc) <= pivot;
                            }
                        } else {
#pragma unroll 1
                            for (int g = tid; g < G; g += TS) {
#pragma unroll
                                for (int q = 0; q < kPub; ++q) {
                                    const u64 e = wkey[q * G + g];
                                    have += e <= pivot && e != kNoKey;
                                }
                            }
                        }
                    }
                    if (svw && svh <= pivot && svh != kNoKey) {
                        const u64 rowbits = (u64)sh.pslot[lane] << kRankBits;
                        const int cc = sh.svc[lane];
                        const u64 B = sh.svB[lane];
#pragma unroll 1
                        for (int q = 0; q < cc; ++q)
                            svn += entry_key(sh.svk[lane][q], rowbits, q) <= pivot;
                        svn += B != kNoKey && entry_key(B, rowbits, cc) <= pivot;
                    }
                    int at = have + svn;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int o = __shfl_up_sync(kFull, at, off);
                        if (lane >= off)
                            at += o;
                    }
                    {
                        int base = 0;
                        if (lane == 31 && at > 0)
                            base = atomicAdd(&sh.ncand, at);
                        base = __shfl_sync(kFull, base, 31);
                        at = base + at - (have + svn);
                    }
                    auto put = [&](u64 key, unsigned col) {
                        if (at < kCand) {
                            sh.ckey[at] = key;
                            sh.ccol[at] = col;
                        }
                        ++at;
                    };
                    if (have > 0) {
                        if (ONE) {
#pragma unroll 1
                            for (int l = tid; l < R; l += TS) {
                                const int cc = ccnt[l];
                                const u64 B = cB[l];
                                const u64 rowbits = (u64)l << kRankBits;
#pragma unroll 1
                                for (int q = 0; q < cc; ++q) {
                                    const u64 x = ck[(size_t)q * Rmax + l];
                                    const u64 e = entry_key(x, rowbits, q);
                                    if (e > pivot)
                                        break;
                                    put(e, (unsigned)x);
                                }
                                if (B != kNoKey && entry_key(B, rowbits, cc) <= pivot)
                                    put(entry_key(B, rowbits, cc), kRowStop | (unsigned)B);
                            }
                        } else {
#pragma unroll 1
                            for (int g = tid; g < G; g += TS) {
#pragma unroll 1
                                for (int q = 0; q < kPub; ++q) {
                                    const u64 e = wkey[q * G + g];
                                    if (e > pivot || e == kNoKey)
                                        break;
                                    put(e, wcol[q * G + g]);
                                }
                            }
                        }
                    }
                    if (svn > 0) {
                        const u64 rowbits = (u64)sh.pslot[lane] << kRankBits;
                        const int cc = sh.svc[lane];
                        const u64 B = sh.svB[lane];
#pragma unroll 1
                        for (int q = 0; q < cc; ++q) {
                            const u64 x = sh.svk[lane][q];
                            const u64 e = entry_key(x, rowbits, q);
                            if (e <= pivot)
                                put(e, (unsigned)x);
                        }
                        if (B != kNoKey && entry_key(B, rowbits, cc) <= pivot)
                            put(entry_key(B, rowbits, cc), kRowStop | (unsigned)B);
                    }
                    sync_s();
                    if (sh.ncand <= kCand)
                        break;
                    // too many entries behind so few heads: take fewer heads
                    want = want / 2 > 1 ? want / 2 : 1;
                    sync_s();
                    if (tid == 0)
                        sh.ncand = 0;
                    hard = pivot;
                    sync_s();
                }
                const int N = sh.ncand;
                // key order by counting (entries are distinct), four threads per entry
#pragma unroll 1
                for (int c0 = (tid >> 5) * 8; c0 < N; c0 += TS / 4) {
                    const int c = c0 + (lane >> 2);
                    const u64 key = c < N ? sh.ckey[c] : kNoKey;
                    int rank = 0;
#pragma unroll 1
                    for (int f = lane & 3; f < N; f += 4)
                        rank += sh.ckey[f] < key;
                    rank += __shfl_xor_sync(kFull, rank, 1);
                    rank += __shfl_xor_sync(kFull, rank, 2);
                    if (c < N && (lane & 3) == 0 && rank <= kEntries) {
                        sh.ekey[rank] = key;
                        sh.erc[rank] = make_uint2((unsigned)key >> kRankBits, sh.ccol[c]);
                    }
                }
                if (tid == 0)
                    sh.pivot = pivot;
                sync_s();
                // which entries bring a row or column that no earlier one has
                const int E = N < kEntries ? N : kEntries;
                // (eight threads per entry)
#pragma unroll 1
                for (int c0 = (tid >> 5) * 4; c0 < E; c0 += TS / 8) {
                    const int e = c0 + (lane >> 3);
                    const uint2 w = e < E ? sh.erc[e] : make_uint2(0u, 0u);
                    const unsigned row = w.x, col = w.y & kColMask;
                    int in = 0;
#pragma unroll 1
                    for (int f = lane & 7; f < e; f += 8) {
                        const uint2 o = sh.erc[f];
                        const unsigned fc = o.y & kColMask;
                        const bool mark = (o.y & kRowStop) != 0;  // (a mark brings no member)
                        in |= !mark && (o.x == row || fc == row) ? 1 : 0;
                        in |= !mark && (o.x == col || fc == col) ? 2 : 0;
                    }
                    in |= __shfl_xor_sync(kFull, in, 1);
                    in |= __shfl_xor_sync(kFull, in, 2);
                    in |= __shfl_xor_sync(kFull, in, 4);
                    if (e < E && (lane & 7) == 0) {
                        if (w.y & kHardStop)
                            sh.enew[e] = 4;
                        else if (w.y & kRowStop)
                            sh.enew[e] = (in & 1) ? 0 : 4;
                        else
                            sh.enew[e] = (unsigned char)(~in & 3);
                    }
                }
                sync_s();
                if (warp == 0) {
                    // the selection ends at the bound of a row without a member, at the
                    // last entry of a CTA (the ones behind it are not known), at kTeam
                    // members, or with the list; lane l looks at two entries
                    const int e0 = 2 * lane;
                    const int f0 = e0 < E ? sh.enew[e0] : 4, f1 = e0 + 1 < E ? sh.enew[e0 + 1] : 4;
                    const int a0 = __popc(f0 & 3), a1 = __popc(f1 & 3);
                    int inc = a0 + a1;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int o = __shfl_up_sync(kFull, inc, off);
                        if (lane >= off)
                            inc += o;
                    }
                    int at = inc - a0 - a1, stop = kEntries;
                    if ((f1 & 4) || inc > kTeam)
                        stop = e0 + 1;
                    if ((f0 & 4) || at + a0 > kTeam)
                        stop = e0;
                    stop = (int)__reduce_min_sync(kFull, (unsigned)stop);
                    // entries left out of a list that ends at a pivot lie above its last
                    const bool cut = stop == E && N <= kEntries && pivot != kNoKey;
                    if (cut && E >= 2)
                        stop = E - 1;
                    int mm = 0;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int f = q ? f1 : f0;
                        if (e0 + q < stop) {
                            const uint2 w = sh.erc[e0 + q];
                            if (f & 1)
                                sh.umem[at++] = (int)w.x;
                            if (f & 2)
                                sh.umem[at++] = (int)(w.y & kColMask);
                            mm = at;
                        }
                    }
                    mm = (int)__reduce_max_sync(kFull, (unsigned)mm);
                    if (lane == 0) {
                        sh.tm.ne = stop;
                        sh.tm.m = mm;
                        // every cell not listed is at or above the first entry not taken
                        u64 A = kNoKey;
                        unsigned C = 0xffffffffu;
                        if (stop < N) {
                            A = (sh.ekey[stop] & kHi) | sh.erc[stop].x;
                            C = sh.erc[stop].y & kColMask;
                        } else if (cut && E == 1) {
                            A = (sh.ekey[0] & kHi) | sh.erc[0].x;
                            C = (sh.erc[0].y & kColMask) + 1u;
                        }
                        sh.tm.thA = A;
                        sh.tm.thC = C;
                        const unsigned tv = (unsigned)(A >> 32);
                        sh.tm.thv = tv;
                        if (!ONE) {
                            // survivors' cells below a limit above the bound are listed;
                            // its distance follows the lists' lengths
                            const unsigned v0 = E > 0 ? (unsigned)(sh.ekey[0] >> 32) : tv;
                            unsigned w = sh.width;
                            if (w == 0u)
                                w = tv > v0 && tv < 0x7f800000u ? 8u * min(tv - v0, 0x100000u) : 0u;
                            else if (nps > 0 && sh.svsum < 4 * nps)
                                w += w / 2;
                            else if (nps > 0 && sh.svsum > 6 * nps)
                                w -= w / 4;
                            sh.width = w = min(max(w, 64u), 0x4000000u);
                            sh.limit = tv < 0x7f000000u ? min(tv + w, 0x7f800000u) : 0xffffffffu;
                        }
                        ty.walk += stop;
                    }
                }
                sync_s();
            }
            const int m = sh.tm.m, ne = sh.tm.ne;
            {
                // members in slot order, with their sizes, stamps and bounds: eight
                // threads per member
#pragma unroll 1
                for (int a0 = (tid >> 5) * 4; a0 < m; a0 += TS / 8) {
                    const int a = a0 + (lane >> 3), part = lane & 7;
                    const int x = a < m ? sh.umem[a] : -1;
                    const bool in = x >= 0 && x < n;
                    bad |= a < m && !in;
                    int sz = 0, st = 0;
                    if (part == 0 && in) {
                        sz = LDCG(p.size_g + x);
                        if (full)
                            st = LDCG(p.stamp + x);
                    }
                    int rank = 0;
#pragma unroll 1
                    for (int q = part; q < m; q += 8)
                        rank += sh.umem[q] < x;
                    u64 A = kNoKey;
                    unsigned C = 0u, ex = 0xffu;
#pragma unroll 1
                    for (int e = part; e < ne; e += 8) {
                        const uint2 w = sh.erc[e];
                        if ((w.y & kRowStop) && w.x == (unsigned)x) {
                            A = (sh.ekey[e] & kHi) | (unsigned)x;
                            C = w.y & kColMask;
                            ex = (unsigned)e;
                        }
                    }
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        rank += __shfl_xor_sync(kFull, rank, o);
                        ex = min(ex, __shfl_xor_sync(kFull, ex, o));
                        const u64 A2 = __shfl_xor_sync(kFull, A, o);
                        const unsigned C2 = __shfl_xor_sync(kFull, C, o);
                        if (A2 < A) {
                            A = A2;
                            C = C2;
                        }
                    }
                    if (part == 0 && in) {
                        sh.tm.mem[rank] = x;
                        sh.tm.sz0[rank] = sz;
                        sh.tm.em[rank] = 0ull;
                        {
                            const unsigned lv = (unsigned)(A >> 32), tv = sh.tm.thv;
                            sh.tm.sl[rank] = make_int2(sz, (int)(lv < tv ? lv : tv));
                        }
                        sh.tm.mst[rank] = st;
                        sh.tm.mbase[rank] = row_base(p, x);
                        sh.tm.lbA[rank] = A;
                        sh.tm.lbC[rank] = C;
                        sh.tm.ex[rank] = (unsigned char)ex;
                    }
                }
            }
            // every CTA read the same records and selected the same way, so every
            // CTA takes this exit together
            bad = count_s(bad != 0);
            {
                // the entries by member (eight threads per entry)
#pragma unroll 1
                for (int c0 = (tid >> 5) * 4; c0 < ne; c0 += TS / 8) {
                    const int e = c0 + (lane >> 3);
                    const uint2 w = e < ne ? sh.erc[e] : make_uint2(0u, kRowStop);
                    unsigned at = 0xffffu;
                    if (!(w.y & kRowStop)) {
                        const int row = (int)w.x, col = (int)(w.y & kColMask);
                        at = 0u;
#pragma unroll 1
                        for (int a = lane & 7; a < m; a += 8) {
                            const int x = sh.tm.mem[a];
                            at |= x == row ? (unsigned)a : x == col ? (unsigned)a << 8 : 0u;
                        }
                    }
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1)
                        at |= __shfl_xor_sync(kFull, at, o);
                    if (e < ne && (lane & 7) == 0) {
                        sh.tm.ent[e] = make_uint2(at, (unsigned)(sh.ekey[e] >> 32));
                        if (at != 0xffffu) {
                            atomicOr(&sh.tm.em[at & 0xffu], 1ull << e);
                            atomicOr(&sh.tm.em[at >> 8], 1ull << e);
                        }
                    }
                }
                sync_s();
                lap(ty.xs[1]);
            }
        }
        {
            if (warp < WA && bad) {
                if (tid == 0) {
                    atomicCAS(p.status, 0, kErrInternal);
                    sh.flag = kErrInternal;
                }
                if constexpr (ONE)
                    __syncthreads();
                else
                    asm volatile("barrier.cta.sync.aligned 3, %0;\n\tbarrier.cta.arrive.aligned 4, %1;" ::"n"(TA), "n"(NT)
                                 : "memory");
            } else if (warp < WA) {
                const int m = sh.tm.m;
                // ---- the cells between members: pair (a, a + d mod kTeam); warp 0
                // takes the chain while its loads are on their way
                const int linkage = p.linkage;
                const bool chain = linkage != 0 && linkage != 5;
                constexpr int ALL = kTeam * kTeam / 2, U = (ALL + TA - 1) / TA > 8 ? 8 : (ALL + TA - 1) / TA;
#pragma unroll 1
                for (int e0 = tid; e0 < ALL; e0 += U * TA) {
                    float v[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int e = e0 + u * TA;
                        const int a = e & (kTeam - 1), c = (a + (e / kTeam) + 1) & (kTeam - 1);
                        v[u] = 0.0f;
                        if (e < ALL && a < m && c < m) {
                            // row-log layout: the cell is current in the row of M
                            // whose slot was stamped later (both rows hold the input
                            // value while neither has merged)
                            const int x = sh.tm.mem[a], y = sh.tm.mem[c];
                            const bool of_a = full ? sh.tm.mst[a] >= sh.tm.mst[c] : x < y;
                            v[u] = LDCG(p.D + (of_a ? sh.tm.mbase[a] + y : sh.tm.mbase[c] + x));
                        }
                    }
                    if (chain && warp == 0 && e0 == tid)
                        chain_select(sh.tm);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int e = e0 + u * TA;
                        const int a = e & (kTeam - 1), c = (a + (e / kTeam) + 1) & (kTeam - 1);
                        if (e < ALL && a < m && c < m) {
                            sh.tm.S[a][c] = v[u];
                            sh.tm.S[c][a] = v[u];
                        }
                    }
                }
                sync_a();
                // (nobody rewrites a member's cell, size or stamp before every CTA got here)
                if (!ONE && tid == 0)
                    red_release_add(p.bar + kBar2, 1u);
                if (full) {
                    // the lines of the members' rows that the merges will read
                    const int nblk = R / 32;
#pragma unroll 1
                    for (int e = tid; e < m * nblk; e += TA) {
                        const long long k = row_of((e / m) * 32);
                        const float *line = p.D + sh.tm.mbase[e % m] + k;
                        if (k < n && CHECK_PREFETCH(line))
                            prefetch_l2(line);
                    }
                }
                lap(ty.xs[2]);
                if (chain)
                    chain_phase<NT, ONE>(sh.tm, linkage, Rmax <= CH);
                if (!chain || sh.tm.redo) {
                    // per member row (columns above it): which cells are at or below
                    // the bound, and the smallest of them
                    const unsigned thv = sh.tm.thv;
#pragma unroll 1
                    for (int a = warp; a < m; a += WA) {
                        const unsigned v0 = __float_as_uint(sh.tm.S[a][lane]);
                        const unsigned v1 = __float_as_uint(sh.tm.S[a][lane + 32]);
                        const bool o0 = lane > a && lane < m && v0 <= thv;
                        const bool o1 = lane + 32 > a && lane + 32 < m && v1 <= thv;
                        const unsigned b0 = __ballot_sync(kFull, o0), b1 = __ballot_sync(kFull, o1);
                        unsigned v = 0xffffffffu, c = 0xffffffffu;
                        if (b0 | b1) {
                            const unsigned w0 = o0 ? v0 : 0xffffffffu, w1 = o1 ? v1 : 0xffffffffu;
                            v = __reduce_min_sync(kFull, w0 < w1 ? w0 : w1);
                            const unsigned k0 = o0 && v0 == v ? (unsigned)lane : 64u;
                            const unsigned k1 = o1 && v1 == v ? (unsigned)lane + 32u : 64u;
                            c = (unsigned)a << 8 | __reduce_min_sync(kFull, k0 < k1 ? k0 : k1);
                        }
                        if (lane == 0) {
                            sh.tm.nnv[a] = v;
                            sh.tm.nnc[a] = c;
                            sh.tm.mask[a] = ((u64)b1 << 32) | b0;
                        }
                    }
                    sync_a();
                    if (warp == 0)
                        simulate(sh.tm, linkage);
                }
                sync_a();
                lap(ty.xs[3]);
                // the merges wait until every CTA holds the members' cells; then the
                // slots they take part in are marked, and slot j retires (Section 4
                // step 2)
                if (grid_wait(p, p.bar + kBar2, epoch2, sh, sync_a)) {
                    // (on condition: j retires when the merge stands, with the
                    // bookkeeping, so that the scans beside it leave no column out)
                    const int L = sh.tm.L;
                    const bool tie = sh.tm.tie != 0;
#pragma unroll 1
                    for (int q = tid; q < 2 * L; q += TA) {
                        const int x = sh.tm.mem[q < L ? sh.tm.mi(q) : sh.tm.mj(q - L)];
                        atomicOr(&touched[x >> 5], 1u << (x & 31));
                        if (q >= L && !tie)
                            atomicAnd(&bitmap[x >> 5], ~(1u << (x & 31)));
                    }
                }
                if (tid == 0) {
                    sh.item = 0;
                    sh.viol = kTeam;
                }
                if constexpr (ONE)
                    __syncthreads();
                else
                    asm volatile("barrier.cta.sync.aligned 3, %0;\n\tbarrier.cta.arrive.aligned 4, %1;" ::"n"(TA), "n"(NT)
                                 : "memory");
                lap(ty.ph[3]);
            } else if constexpr (!ONE) {
                constexpr int TB = NT - TA;
                // ---- the refills asked for in the previous round, served now by
                // team B (row s of the list by CTA G - 1 - s mod G: rows are
                // owned in blocks of 32 from CTA 0 up, so the last CTAs own a block
                // fewer and take the scans first): the K smallest keys of the row
                // over live columns.  Other CTAs may already be writing this
                // round's merges: the columns those touch are dropped when the
                // owner installs the list and replays the round.
                // A row is cut in pieces when there are CTAs for them: a whole row
                // scanned by one CTA outlasts the steps beside it, and every other
                // CTA would wait for it.
                const int nexec = sh.nexec;
                const int np = scan_pieces(G, nexec, early);
#pragma unroll 1
                for (int w = G - 1 - b; w < nexec * np; w += G) {
                    const int s2 = w / np, piece = w % np;
                    const long long rr = sh.exec_row[s2];
                    if (rr < 0 || rr >= n - 1)
                        continue;  // the same for every thread of the team
                    if (full)
                        block_row_topk_cols<NT, ONE, TB>(p, rr, piece, np, (int)t, bitmap, sh, st_fill_cells,
                                                         p.timing ? ty.xscan : nullptr);
                    else
                        block_row_topk<NT, ONE, TB>(p, rr, piece, np, bitmap, sh, st_fill_cells);
                    if (tid - TA < K + 1)
                        STCG(p.parts + (((size_t)par * kMaxReq + s2) * kPieces + piece) * kPartWords + (tid - TA),
                             tid - TA < K ? sh.tko[tid - TA] : sh.tnext);
                }
                if (tid == TA)
                    ty.fills += nexec;
                // (team A does not wait: it begins with the new cells)
                asm volatile("barrier.cta.sync.aligned 4, %0;" ::"n"(NT) : "memory");
            }
        }
        if (sh.flag != 0)
            return;  // (a wait ran out, here or in another CTA)
        lap(ty.ph[2]);
        const int m = sh.tm.m;
        int L = sh.tm.L, ns = sh.tm.ns;
        const bool tie = sh.tm.tie != 0;


        // ---- apply the L merges to every live row k outside them, a chunk of
        // rows at a time; per chunk (1) the new cells D(k, survivor) of
        // Section 4 step 3, a warp per 32 rows and 4 survivors, stored and kept
        // in kvs, (2) per survivor the smallest of them above it, NT / kSurv
        // threads each, and the rows' caches, a thread each
        auto bookkeeping = [&]() {
            if (!ONE) {
                // (every CTA has read the previous round's lists)
#pragma unroll 1
                for (int q = b * NT + tid; q < kSurv * kSvList; q += G * NT)
                    STCG(p.svlist + (par ^ 1) * kSurv * kSvList + q, kNoKey);
                if (b == 0 && tid < kSurv)
                    STCG(p.svovf + (par ^ 1) * kSurv + tid, kNoKey);
                if (b == 0 && tid == 0)
                    STCG(p.bar + kViol + (par ^ 1), 0u);
            }
            if (b == 0) {
#pragma unroll 1
                for (int q = tid; q < L; q += NT) {
                    STCG(p.merges + 2 * (t + q), (int32_t)sh.tm.mem[sh.tm.mi(q)]);
                    STCG(p.merges + 2 * (t + q) + 1, (int32_t)sh.tm.mem[sh.tm.mj(q)]);
                    STCG(p.heights + t + q, __int_as_float(sh.tm.rec[q].y));
                }
                if (tid < ns)
                    STCG(p.size_g + sh.tm.sslot[tid], sh.tm.rec[sh.tm.sq[tid]].z + sh.tm.rec[sh.tm.sq[tid]].w);
            }
#pragma unroll 1
            for (int q = tid; q < 2 * L; q += NT) {
                const int x = sh.tm.mem[q < L ? sh.tm.mi(q) : sh.tm.mj(q - L)];
                if (tie && q >= L)
                    atomicAnd(&bitmap[x >> 5], ~(1u << (x & 31)));
                if (owner_of(x) == b) {
                    const int l = slot_of(x);
                    ccnt[l] = 0;
                    cB[l] = kNoKey;
                    if (!ONE)
                        pend_t[l] = -1;
                }
            }
            if (tid < ns) {
                const int x = sh.tm.sslot[tid];
                sh.pslot[tid] = x;
                const int tq = (int)(t + sh.tm.sq[tid]);
                // row-log layout: the last merge rewrites row x (every CTA writes the
                // same value, so each one sees the new stamps in its own rescans)
                if (full)
                    STCG(p.stamp + x, tq);
                if (owner_of(x) == b) {
                    const int l = slot_of(x);
                    rsize[l] = sh.tm.rec[sh.tm.sq[tid]].z + sh.tm.rec[sh.tm.sq[tid]].w;
                    if (!ONE)
                        rstamp[l] = tq;
                }
            }
            if (tid == 0) {
                sh.ninst = 0;
                sh.nps = ns;
                if (!ONE)
                    sh.npieces = scan_pieces(G, sh.nexec, early);
            }
            // slots to clear from `touched` after the next round
#pragma unroll 1
            for (int a = tid; a < m; a += NT)
                sh.ptouch[a] = sh.tm.mem[a];
            if (tid == 0)
                sh.nptouch = m;
        };
        constexpr int TPP = NT / kSurv;
        const int ra = tid / TPP, rpart = tid % TPP;
        u64 ps[P];
#pragma unroll
        for (int q = 0; q < P; ++q)
            ps[q] = kNoKey;
        bool kept = false;  // the new cells are in kvs and in memory already
        if (tie) {
            const int k = settle<NT, ONE>(p, sh, par, epoch3);
            if (k < 0)
                return;
            kept = k != 0;
            L = sh.tm.L;
            ns = sh.tm.ns;
        }
#pragma unroll 1
        for (int l0 = 0; l0 < R; l0 += CH) {
            const int rows = R - l0 < CH ? R - l0 : CH;
            if (!kept) {
                new_cells(p, sh, l0, rows, ns, kStore);
                __syncthreads();
            }
            lap(ty.xs[4]);
            if (l0 == 0) {
                bookkeeping();
                // one CTA: the survivors' smallest cells to other survivors (those to the
                // other members are among their owners' new cells), a lane each
#pragma unroll 1
                for (int s = warp; ONE && s < ns; s += W) {
                    u64 x = kNoKey;
                    if (lane < ns && sh.tm.sslot[lane] > sh.tm.sslot[s])
                        x = make_key(sh.tm.C[s][lane], (unsigned)sh.tm.sslot[lane]);
#pragma unroll
                    for (int q = 0; q <= K; ++q) {
                        const u64 y = warp_u64_min(x);
                        x = x == y ? kNoKey : x;
                        if (lane == 0) {
                            if (q < K)
                                sh.tm.tT[s][q] = y;
                            else
                                sh.tm.tB[s] = y;  // bounds the others
                        }
                    }
                }
                if (b == 0) {
#pragma unroll 1
                    for (int e = tid; e < ns * ns; e += NT) {
                        const int x = e / ns, y = e % ns;
                        if (x < y) {  // (the later last merge has the larger index)
                            const float v = sh.tm.C[x][y];
                            if (full) {
                                STCG(p.D + (long long)sh.tm.sslot[y] * p.pitch + sh.tm.sslot[x], v);
                                STCG(p.TL + (long long)sh.tm.sslot[x] * p.pitch + t + sh.tm.sq[y], v);
                            } else {
                                STCG(p.D + pair_idx(sh.tm.sslot[x], sh.tm.sslot[y], n), v);
                            }
                        }
                    }
                }
            }
            if (full) {
                // row k's log at the survivors' last merges, from kvs: lane per
                // survivor, so a row's words of the round go out together (by
                // rows they would be one sector each)
                const int sq = lane < ns ? sh.tm.sq[lane] : 0;
#pragma unroll 1
                for (int q = warp; q < rows; q += W) {
                    if (lane < ns && ((sh.okm[q >> 5] >> (q & 31)) & 1u))
                        STCG(p.TL + row_of(l0 + q) * p.pitch + t + sq, kvs[(size_t)q * KVP + lane]);
                }
            }
            if (ra < ns) {
                const long long ia = sh.tm.sslot[ra];
#pragma unroll 4
                for (int q = rpart; q < rows; q += TPP) {
                    const unsigned vb = __float_as_uint(kvs[(size_t)q * KVP + ra]);
                    const bool in = (sh.okm[q >> 5] >> (q & 31)) & 1u;
                    if (ONE) {
                        if (in && vb <= (unsigned)(ps[P - 1] >> 32)) {
                            const long long kq = row_of(l0 + q);
                            const u64 key = ((u64)vb << 32) | (unsigned)kq;
                            if (kq > ia && key < ps[P - 1])
                                list_insert_n(ps, key);
                        }
                    } else if (in && vb < sh.limit) {
                        const long long kq = row_of(l0 + q);
                        if (kq > ia) {
                            const size_t at = (size_t)par * kSurv + ra;
                            list_add(p.svlist + at * kSvList, p.svovf + at, ((u64)vb << 32) | (unsigned)kq);
                        }
                    }
                }
            }
#pragma unroll 1
            for (int q = tid; q < rows; q += NT) {
                const int l = l0 + q;
                const long long k = row_of(l);
                unsigned hm = sh.hit[q];
                sh.hit[q] = 0u;
                if (!(k < n && live(bitmap, k) && !live(touched, k)))
                    continue;
                int c = ccnt[l];
                u64 B = cB[l];
                if (ns > 0) {
                    u64 Cc[K];
                    cache_load(Cc, l);
                    bool drop = false;
#pragma unroll
                    for (int e = 0; e < K; ++e) {
                        if (Cc[e] != kNoKey && live(touched, (unsigned)Cc[e])) {
                            Cc[e] = kNoKey;
                            drop = true;
                        }
                    }
                    bool dirty = drop;
                    if (drop) {
                        sort_list(Cc);
                        c = list_count(Cc);
                    }
                    const float *kr = kvs + (size_t)q * KVP;
#pragma unroll 1
                    for (; hm != 0u; hm &= hm - 1u) {
                        const int s = __ffs(hm) - 1;
                        const unsigned vb = __float_as_uint(kr[s]);
                        const long long x = sh.tm.sslot[s];
                        const u64 key = ((u64)vb << 32) | (unsigned)x;
                        if (key < B) {
                            const u64 out = list_insert(Cc, key);
                            dirty = true;
                            if (c == K)
                                B = out;
                            else
                                ++c;
                        }
                    }
                    if (dirty) {
                        cache_store(l, Cc);
                        ccnt[l] = (unsigned char)c;
                        cB[l] = B;
                    }
                }
                if (ONE) {
                    // one CTA: no one else to ask, refill right after this pass
                    if (c == 0 && B != kNoKey)
                        rlist[atomicAdd(&sh.nresc, 1)] = l;
                } else if (c == 0 && B != kNoKey && (unsigned)(B >> 32) <= sh.tm.thv) {
                    // live cells remain, none is cached, and the bound sits at
                    // the front of the merges: its bare mark would hold the next
                    // rounds up until a refill lands, so rescan now
                    rlist[atomicAdd(&sh.nresc, 1)] = l;
                    pend_t[l] = -1;
                } else if (c <= refill_at && B != kNoKey && pend_t[l] < 0) {
                    // (a cache that holds every live cell of its row needs no refill)
                    request(l, r);
                }
            }
            if (l0 + CH < R) {
                if (tid == 0)
                    sh.item = 0;
                __syncthreads();
            }
        }
        // a one-CTA job: per survivor, over the TPP threads
        if constexpr (ONE) {
            __syncthreads();  // (the members' lists)
            u64 out[P];
#pragma unroll
            for (int q = 0; q < P; ++q)
                out[q] = ps[q];
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) {
                u64 x[P];
#pragma unroll
                for (int q = 0; q < P; ++q)
                    x[q] = __shfl_xor_sync(kFull, out[q], o);
#pragma unroll
                for (int q = 0; q < P; ++q)
                    list_insert_n(out, x[q]);
            }
            {
                // the smallest cells of the survivor's row: to other rows (the last of
                // out bounds the rest) and to survivors
                if (ra < ns && rpart == 0) {
                    const int l = slot_of(sh.tm.sslot[ra]);
                    u64 M[K], next = out[P - 1];
#pragma unroll
                    for (int q = 0; q < K; ++q)
                        M[q] = out[q < P - 1 ? q : 0];
#pragma unroll
                    for (int q = 0; q < K; ++q) {
                        const u64 x = list_insert(M, sh.tm.tT[ra][q]);
                        next = x < next ? x : next;
                    }
                    next = sh.tm.tB[ra] < next ? sh.tm.tB[ra] : next;
                    cache_store(l, M);
                    ccnt[l] = (unsigned char)list_count(M);
                    cB[l] = next;
                }
            }
        }
        __syncthreads();
        lap(ty.xs[6]);
        // ---- rows whose cache emptied
        {
            const int nresc = sh.nresc;
            if (ONE) {
#pragma unroll 1
                for (int q = warp; q < nresc; q += W) {
                    const int l = rlist[q];
                    u64 top[K], next;
                    warp_row_refresh(p, row_of(l), bitmap, top, next, st_resc_cells);
                    if (lane == 0) {
                        cache_store(l, top);
                        ccnt[l] = (unsigned char)list_count(top);
                        cB[l] = next;
                    }
                }
            } else {
#pragma unroll 1
                for (int q = 0; q < nresc; ++q) {
                    const int l = rlist[q];
                    if (full)
                        block_row_topk_cols(p, row_of(l), 0, 1, 0x7fffffff, bitmap, sh, st_resc_cells);
                    else
                        block_row_topk(p, row_of(l), 0, 1, bitmap, sh, st_resc_cells);
                    if (tid == 0) {
                        cache_store(l, sh.tko);
                        ccnt[l] = (unsigned char)list_count(sh.tko);
                        cB[l] = sh.tnext;
                    }
                }
            }
            if (nresc > 0)
                __syncthreads();  // the rescanned caches before anyone reads them
            if (tid == 0) {
                ty.rescans += nresc;
                sh.nresc = 0;
                ++ty.rounds;
                ty.idle += L == 0;
            }
        }
        lap(ty.xs[7]);
        t += L;
        if (t >= n - 1)
            break;  // that was the last merge
        __syncthreads();
    }

    if (p.stats) {
        u64 *St = reinterpret_cast<u64 *>(p.stats);
        atomicAdd(St + 5, (u64)st_fill_cells);
        atomicAdd(St + 15, (u64)st_resc_cells);
        if (tid == (ONE ? 32 : TA)) {
            atomicAdd(St + 6, (u64)ty.installs);
            if (b == 0)
                St[4] = (u64)ty.fills;  // every CTA read the same request lists
            if (p.timing) {
                atomicAdd(St + 24, ty.xscan[0]);
                atomicAdd(St + 25, ty.xscan[1]);
            }
        }
        if (tid == 0) {
            atomicAdd(St + 14, (u64)ty.rescans);
            if (b == 0) {
                St[0] = (u64)ty.rounds;
                St[1] = (u64)ty.idle;
                St[2] = (u64)((n - 1) * (n - 2) / 2);  // m_t - 2 cells per merge
                St[7] = (u64)ty.walk;
                St[3] = (u64)G;
            }
            if (p.timing) {
                ty.ph[1] += ty.xs[5] + ty.xs[0] + ty.xs[1] + ty.xs[2] + ty.xs[3];
                ty.ph[5] += ty.xs[4] + ty.xs[6] + ty.xs[7];
#pragma unroll 1
                for (int q = 0; q < 6; ++q)
                    atomicAdd(St + 8 + q, ty.ph[q]);
#pragma unroll 1
                for (int q = 0; q < 8; ++q)
                    atomicAdd(St + 16 + q, ty.xs[q]);
            }
        }
    }
}

template <int NT, int MINB, bool ONE>
__global__ void __launch_bounds__(NT, MINB) merge_kernel(MergeParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared<NT, ONE> sh;
    merge_job<NT, ONE>(p, blockIdx.x, smem_raw, sh);
}

// Many independent jobs in one persistent launch: each CTA takes the next job
// from a queue (atomicAdd on a counter) and runs all its merges alone (a
// one-CTA job needs no grid barrier), then takes another, until the queue is
// empty.  CTA c keeps its scratch in workspace slot c.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) batch_kernel(BatchParams bp)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared<NT, true> sh;
    __shared__ int job;
    const WorkspaceLayout L = workspace_layout(bp.n_max, 1);
    char *ws = bp.ws + (size_t)blockIdx.x * L.total;
    long long merges_done = 0;
    while (true) {
        if (threadIdx.x == 0)
            job = atomicAdd(bp.queue, 1);
        __syncthreads();
        const int jb = job;
        if (jb >= bp.njobs)
            break;
        const BatchJob J = bp.jobs[jb];
        MergeParams p;
        p.D = J.D;
        p.TL = nullptr;
        p.stamp = nullptr;
        p.full = 0;
        p.n = J.n;
        p.pitch = J.n;
        p.linkage = J.linkage;
        p.G = 1;
        p.chunk = bp.chunk;
        p.aligned16 = ((uintptr_t)J.D & 15u) == 0;
        p.merges = J.merges;
        p.heights = J.heights;
        bind_workspace(p, ws, L);
        check_range(p, J.D, (unsigned long long)J.n * (unsigned long long)(J.n - 1) / 2 * sizeof(float));
        check_range(p, J.merges, 8ull * (unsigned long long)(J.n > 1 ? J.n - 1 : 0));
        check_range(p, J.heights, 4ull * (unsigned long long)(J.n > 1 ? J.n - 1 : 0));
        p.stats = nullptr;
        p.timeout_ns = bp.timeout_ns;
        p.skip_arrive_cta = -1;
        p.timing = 0;
        // the slot keeps the previous job's words: clear the ones that must start at zero
#pragma unroll 1
        for (size_t q = threadIdx.x; q < (L.total - L.zero) / 4; q += NT)
            reinterpret_cast<int *>(ws + L.zero)[q] = 0;
        __syncthreads();
        if (J.n > 1)
            merge_job<NT, true>(p, 0, smem_raw, sh);
        __syncthreads();
        if (threadIdx.x == 0) {
            bp.job_status[jb] = J.n > 1 ? LDCG(p.status) : 0;
            merges_done += J.n > 1 ? J.n - 1 : 0;
        }
    }
    if (threadIdx.x == 0 && bp.merges_done)
        atomicAdd(reinterpret_cast<unsigned long long *>(bp.merges_done), (unsigned long long)merges_done);
}

// The symmetric matrix from the packed triangle, one 32 x 32 tile of the
// upper triangle per CTA (32 x 8 threads): the tile is read row by row and
// written both as it is and transposed through shared memory, so every
// global access of a warp is 32 consecutive words.
__global__ void __launch_bounds__(256) expand_kernel(const float *__restrict__ P, float *__restrict__ F,
                                                     long long n, long long pitch, int *status)
{
    __shared__ float tile[32][33];
    const long long tr = blockIdx.y, tc = blockIdx.x;
    if (tr > tc)
        return;
    const int tx = threadIdx.x, ty = threadIdx.y;
    int bad = 0;
#pragma unroll 1
    for (int yy = ty; yy < 32; yy += 8) {
        const long long r = tr * 32 + yy, c = tc * 32 + tx;
        float v = 0.0f;
        if (c > r && c < n) {
            v = __ldg(P + tri_off(r, n) + (c - r - 1));
            const unsigned u = __float_as_uint(v);
            if (u == 0x80000000u)
                v = 0.0f;  // -0 reads as +0 from here on
            else if (u > 0x7f7fffffu)
                bad = 1;   // NaN, infinite or negative
            F[r * pitch + c] = v;
        }
        tile[yy][tx] = v;
    }
    __syncthreads();
#pragma unroll 1
    for (int yy = ty; yy < 32; yy += 8) {
        const long long c = tc * 32 + yy, r = tr * 32 + tx;
        if (c > r && c < n)
            F[c * pitch + r] = tile[tx][yy];
    }
    if (bad)
        atomicCAS(status, 0, kErrInput);
}

}  // namespace

cudaError_t launch_expand(const float *packed, float *full, long long n, long long pitch, int *status,
                          cudaStream_t stream)
{
    const long long nb = (n + 31) / 32;
    if (nb > 65535)
        return cudaErrorInvalidValue;
    expand_kernel<<<dim3((unsigned)nb, (unsigned)nb), dim3(32, 8), 0, stream>>>(packed, full, n, pitch, status);
    return cudaGetLastError();
}

namespace {

// The kernel instantiations: CTA size nt and the CTAs per SM its registers allow.
const void *merge_fn(int nt, int G)
{
    if (G == 1) {
        switch (nt) {
        case 128: return (const void *)merge_kernel<128, 4, true>;
        case 256: return (const void *)merge_kernel<256, 2, true>;
        default: return (const void *)merge_kernel<512, 1, true>;
        }
    }
    switch (nt) {
    case 128: return (const void *)merge_kernel<128, 4, false>;
    case 256: return (const void *)merge_kernel<256, 2, false>;
    default: return (const void *)merge_kernel<512, 1, false>;
    }
}

const void *batch_fn(int nt)
{
    switch (nt) {
    case 128: return (const void *)batch_kernel<128, 4>;
    case 256: return (const void *)batch_kernel<256, 2>;
    default: return (const void *)batch_kernel<512, 1>;
    }
}

size_t static_smem(int nt, int G)
{
    if (G == 1) {
        switch (nt) {
        case 128: return sizeof(Shared<128, true>) + 16;
        case 256: return sizeof(Shared<256, true>) + 16;
        default: return sizeof(Shared<512, true>) + 16;
        }
    }
    switch (nt) {
    case 128: return sizeof(Shared<128, false>);
    case 256: return sizeof(Shared<256, false>);
    default: return sizeof(Shared<512, false>);
    }
}

// Dynamic shared memory for n objects on G CTAs of nt threads with chunks of
// `chunk` rows: two bitmaps; published entries (keys, column words); per slot
// K keys, bound, size, rescan list entry and key count, on a grid also the
// pending refill (round, position) and the stamp; the new cells of a chunk.
size_t smem_for(long long n, int G, int chunk)
{
    const long long nb = (n + kRowBlock - 1) / kRowBlock;
    const long long Rmax = ((nb + G - 1) / G) * kRowBlock;
    const long long words = (((n + 31) / 32) * 4 + 15) & ~15LL;
    const long long row = 8 * K + 8 + 8 + 1 + (G > 1 ? 12 : 0);
    return (size_t)(2 * words + (G > 1 ? (long long)G * kPub * 12 : 0) + (long long)chunk * (kSurv + 1) * 4 +
                    ((Rmax * row + 15) & ~15LL));
}

}  // namespace

// CTAs for n objects when the caller names no number.  One up to 416 objects: a
// block of 32 rows per CTA and grid barriers are no faster there (complete, ms,
// one CTA / grid: n = 300 0.62 / 0.70, n = 400 0.83 / 0.77, n = 512 1.07 / 1.01,
// n = 1000 3.04 / 1.44, n = 2048 12.0 / 2.5).  Centroid linkage makes few merges
// per round, so a grid's barriers weigh more: n = 400 2.9 / 3.8, n = 600 5.8 / 5.4,
// n = 1000 10.3 / 8.1, n = 1152 13.6 / 9.5, n = 2048 32.1 / 15.6; up to 1152 objects
// it stays on one SM, where a grid would take 19 to 36 of them for 7 to 30 % of the
// time.  Above, one CTA per block up to 64 of them, then one per two blocks
// (rounded up: with n = 5003, 157 blocks, 78 CTAs leave three blocks to one of
// them; complete 5.70, average 5.83, packed 5.61, on 79 CTAs 5.64, 5.71, 5.51;
// n = 7001, 109 / 110 CTAs, 7.82 / 7.64), at most one per SM (complete: n = 3500
// 64 CTAs 4.06, 96 3.97; n = 4096 64 CTAs 4.73, 128 4.47; average: n = 5003 79 CTAs
// 5.71, 152 5.63; n = 6500 102 7.21, 128 7.17): the last percent would take
// twice the SMs.  Single linkage (the merges of a round are worked out one by one,
// and every CTA repeats them) is as fast on fewer CTAs with the same most blocks
// per CTA and takes those (n = 16384, 128 / 152 CTAs: distances on a 1/1024 grid
// 52.7 / 53.4, continuous 27.8 / 27.6; Ward 23.0 / 21.5).
int default_grid(long long n, int linkage, int num_sms)
{
    const long long nb = (n + kRowBlock - 1) / kRowBlock;
    if (n <= (linkage == LW_CENTROID ? 1152 : 416))
        return 1;
    long long G = nb <= 64 ? nb : nb > 128 ? (nb + 1) / 2 : 64;
    if (G > num_sms)
        G = num_sms;
    if (linkage == LW_SINGLE) {
        const long long per = (nb + G - 1) / G, even = (nb + per - 1) / per;
        if (10 * even <= 9 * G)
            G = even;
    }
    return (int)G;
}

int merge_chunk_rows(long long n, int G, int nt)
{
    const long long nb = (n + kRowBlock - 1) / kRowBlock;
    const long long Rmax = ((nb + G - 1) / G) * kRowBlock;
    const int most = (int)(Rmax < nt ? Rmax : nt);
    // half a CTA's threads per chunk if that lets as many CTAs share an SM as
    // the registers allow, else whatever fits at all
    const long long sm = 228 * 1024, cta = 227 * 1024, fixed = (long long)static_smem(nt, G);
    const long long share = sm / (kThreads / nt) - 1024 - fixed;
#pragma unroll 1
    for (int c = most; c >= 32 && 2 * c >= most; c = (c / 2) & ~31)
        if ((long long)smem_for(n, G, c) <= share)
            return c;
    int c = most;
    while (c > 32 && (long long)smem_for(n, G, c) > cta - fixed)
        c = c / 2 >= 32 ? (c / 2) & ~31 : 32;
    return c;
}

size_t merge_smem_bytes(long long n, int G, int nt)
{
    return smem_for(n, G, merge_chunk_rows(n, G, nt));
}

namespace {

// Lets a kernel's launches have all the dynamic shared memory that a CTA can have;
// false if smem bytes are more than that.  Always the same value: the attribute
// belongs to the function, and another thread may be between setting it for a
// smaller job and launching that.
bool allow_smem(const void *fn, int nt, int G, size_t smem)
{
    int dev = 0, limit = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    const long long most = (long long)limit - (long long)static_smem(nt, G);
    return (long long)smem <= most &&
           cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) == cudaSuccess;
}

int fit_per_sm(const void *fn, int nt, int G, size_t smem)
{
    if (!allow_smem(fn, nt, G, smem))
        return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, nt, smem) != cudaSuccess)
        return 0;
    return per_sm;
}

}  // namespace

bool merge_config_ok(long long n, int G, int num_sms, int nt)
{
    // the first G threads read the CTAs' records
    if (G < 1 || G > num_sms || G > nt)
        return false;
    return fit_per_sm(merge_fn(nt, G), nt, G, merge_smem_bytes(n, G, nt)) >= 1;
}

int batch_ctas_per_sm(long long n_max, int nt)
{
    return fit_per_sm(batch_fn(nt), nt, 1, merge_smem_bytes(n_max, 1, nt));
}

cudaError_t launch_batch(const BatchParams &bp, int grid, int nt, cudaStream_t stream)
{
    // batch_ctas_per_sm(bp.n_max, nt) has set the kernel's shared-memory limit
    // (this launch may be recorded into a graph, where no attribute is set)
    const size_t smem = merge_smem_bytes(bp.n_max, 1, nt);
    BatchParams q = bp;
    q.chunk = merge_chunk_rows(bp.n_max, 1, nt);
    void *args[] = {&q};
    return cudaLaunchKernel(batch_fn(nt), dim3(grid), dim3(nt), args, smem, stream);
}

cudaError_t launch_merge(const MergeParams &p, int nt, cudaStream_t stream)
{
    const size_t smem = merge_smem_bytes(p.n, p.G, nt);
    const void *fn = merge_fn(nt, p.G);
    if (!allow_smem(fn, nt, p.G, smem)) {
        const cudaError_t e = cudaGetLastError();
        return e != cudaSuccess ? e : cudaErrorInvalidValue;
    }
    MergeParams q = p;
    q.chunk = merge_chunk_rows(p.n, p.G, nt);
    void *args[] = {&q};
    return cudaLaunchCooperativeKernel(fn, dim3(p.G), dim3(nt), args, smem, stream);
}

}  // namespace lw
