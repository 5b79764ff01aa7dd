// sim_kernel.cu -- the simulation of FCFS, LJF, SJF and ISJL on sm_103a.
//
// One warp simulates one (instance, run) task; a persistent grid of warps
// pulls tasks from a global counter.  The model is the paper's token-step one
// (Section 2): in step k, requests with A_i <= k join the pending queue Q(k),
// requests that finished in step k - 1 leave the batch (c_i = k), the policy
// admits (FCFS, LJF of Algorithm 1, SJF, ISJL of Algorithm 2 in Section 3.4's
// rolling form), every running request processes token r_i = a_i + 1, and the
// step costs W += |S| max r, E += sum (max r - r_i), extent, T_busy (Section 5,
// Eq. batch-cost-progress and the decomposition).
//
// The kernel jumps from event to event (arrival, completion, o_1's delay
// expiry) and adds the cost of the L steps in between in closed form: the
// running set is constant there and progress moves in lockstep, so every
// counter equals the step-by-step sum.  Admissions happen only at events:
// between events the running set, the KV reservation and the queue are
// unchanged and A_max only grows, so a step that could not start a request is
// followed by steps that cannot either.  While LJF has a batch running or
// ISJL's gate is shut, completions that do not change the running set's
// earliest or latest start are served in the same pass (a completion window).
// (Advancing every running request in every step takes 1.1 to 3.7 times as long
// over the measured sweeps and nowhere less.)
// While a queue head waits, ISJL without a binding budget, and FCFS and SJF where a
// queue builds up, serve up to 32 completions in a pass (a batch).
// Arrivals that cannot start anything before the next completion are released
// at that completion, and an admission that starts several requests does so
// up to 32 (ISJL plan entries: all) at a time, with the same outcome as one
// start at a time.
//
// Layout.  Worker (batch slot) w lives in lane w % 32, register row w / 32,
// so a warp holds B <= 32 * SPL workers.  Values that change only at events
// (next arrival, start range, KV reservation) are kept as warp-uniform scalars.
// The pending queue is a bitset over the instance's request positions sorted by
// (o desc, index asc) -- the longest pending request is the lowest set bit --
// with a summary word per 32 words, in shared memory.  ISJL plans are per-worker
// FIFO lists linked through a global scratch array.  Many instances of at most 32
// requests go to tiny_kernel.cu instead (the rule is in launch_sim).
#include <algorithm>
#include <climits>
#include <cstdint>

#include "sim_internal.cuh"

namespace isjl {
namespace {

constexpr int32_t kNone = -1;
// ISJL whose budget no request's length exceeds: it never plans (o_2 <= alpha) and
// its gate never shuts, so it starts the longest pending request that fits
constexpr int kPolicyLpt = ISJL_POLICY_ISJL_BETA + 1;
// SJF and FCFS where a queue builds up (queue_builds_up): with batches of completions
constexpr int kPolicySjfQueue = ISJL_POLICY_ISJL_BETA + 2;
constexpr int kPolicyFcfsQueue = ISJL_POLICY_ISJL_BETA + 3;
constexpr uint32_t kEmpty = 0xFFFFFFFFu;   // key of a slot that holds no running request

// bits of a running request's key that hold its register row
template <int SPL> __host__ __device__ constexpr int row_bits() { return SPL >= 16 ? 4 : SPL >= 8 ? 3 : SPL >= 4 ? 2 : SPL >= 2 ? 1 : 0; }

struct WarpSmem {
    uint32_t *key;    // [32][SPL] completion step, lane and row of the request on a slot (kEmpty: none)
    uint32_t *swap;   // [32] words that lanes leave for one another
    int2 *slot;       // [B] request on worker w: start step, reserved KV (its planning length); in Phase ONE,
                      //     w's last plan entry (-1: none) and w's packing budget, then its pack sum
    uint32_t *slink;  // [B] plan link of worker w's next ISJL plan entry (0: none)
    int32_t *slong;   // [B] long request o_j planned on worker j (1 <= j < n_long)
    uint32_t *pend0;  // [words0] bit p: sorted position p is pending
    uint32_t *pend1;  // [words1] bit w: pend0[w] != 0
};

__host__ __device__ inline int smem_words_per_warp(int spl, int B, int words0, int words1) {
    int w = (spl > 1 ? 32 * spl : 0) + 32 + 4 * B + words0 + words1;
    return (w + 3) & ~3;  // keep every warp's block 16-byte aligned
}

// copy one word from global to this lane's shared memory without waiting for it
__device__ __forceinline__ void copy_async(uint32_t *smem, const int32_t *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
// fetch the line of a word into the caches without waiting for it
__device__ __forceinline__ void prefetch(const int32_t *gmem) { asm volatile("prefetch.global.L1 [%0];" :: "l"(gmem)); }
// wait for this lane's copies
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// lowest worker whose row bit is set in the per-lane mask m
__device__ __forceinline__ int lowest_worker(uint32_t m, int lane) {
    const int v = m ? ((__ffs(m) - 1) << 5) + lane : INT_MAX;
    const int r = __reduce_min_sync(kFull, v);
    return r == INT_MAX ? -1 : r;
}
// acc += a * b into a 64-bit accumulator with one wide multiply-add
__device__ __forceinline__ void mad_wide(int64_t &acc, uint32_t a, uint32_t b) {
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// warp sum of a 64-bit value (modulo 2^64) by three independent 32-bit warp
// reductions of its 22-, 22- and 20-bit pieces (each piece's sum is below 2^27)
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
    const uint32_t a = __reduce_add_sync(kFull, (uint32_t)v & 0x3FFFFFu);
    const uint32_t b = __reduce_add_sync(kFull, (uint32_t)(v >> 22) & 0x3FFFFFu);
    const uint32_t c = __reduce_add_sync(kFull, (uint32_t)(v >> 44));
    return (uint64_t)a + ((uint64_t)b << 22) + ((uint64_t)c << 44);
}

__device__ __forceinline__ int64_t warp_sum64(int64_t v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(kFull, v, s);
    return v;
}

// first pending sorted position >= p, INT_MAX if none (uniform call)
__device__ __forceinline__ int bs_next(const WarpSmem &S, int words0, int words1, int p, int lane) {
    const int w0 = p >> 5;
    if (w0 >= words0) return INT_MAX;
    const uint32_t v = S.pend0[w0] & (~0u << (p & 31));
    if (v) return (w0 << 5) + __ffs(v) - 1;
    const int q = w0 + 1;
    if (q >= words0) return INT_MAX;
    const int w1 = q >> 5;
    const uint32_t u = S.pend1[w1] & (~0u << (q & 31));
    if (u) {
        const int ww = (w1 << 5) + __ffs(u) - 1;
        return (ww << 5) + __ffs(S.pend0[ww]) - 1;
    }
#pragma unroll 1
    for (int b1 = w1 + 1; b1 < words1; b1 += 32) {
        const int idx = b1 + lane;
        const uint32_t x = idx < words1 ? S.pend1[idx] : 0u;
        const unsigned b = __ballot_sync(kFull, x != 0u);
        if (b) {
            const int l = __ffs(b) - 1;
            const uint32_t xx = __shfl_sync(kFull, x, l);
            const int ww = ((b1 + l) << 5) + __ffs(xx) - 1;
            return (ww << 5) + __ffs(S.pend0[ww]) - 1;
        }
    }
    return INT_MAX;
}

__device__ __forceinline__ void bs_clear(const WarpSmem &S, int p, int lane) {
    if (lane == 0) {
        const int w = p >> 5;
        const uint32_t v = S.pend0[w] & ~(1u << (p & 31));
        S.pend0[w] = v;
        if (!v) S.pend1[w >> 5] &= ~(1u << (w & 31));
    }
    __syncwarp();
}

// highest pending sorted position, -1 if none (uniform call)
__device__ __forceinline__ int bs_last(const WarpSmem &S, int words1, int lane) {
#pragma unroll 1
    for (int b1 = (words1 - 1) & ~31; b1 >= 0; b1 -= 32) {
        const int idx = b1 + lane;
        const uint32_t x = idx < words1 ? S.pend1[idx] : 0u;
        const unsigned b = __ballot_sync(kFull, x != 0u);
        if (b) {
            const int l = 31 - __clz(b);
            const uint32_t xx = __shfl_sync(kFull, x, l);
            const int ww = ((b1 + l) << 5) + 31 - __clz(xx);
            return (ww << 5) + 31 - __clz(S.pend0[ww]);
        }
    }
    return -1;
}

// highest pending sorted position <= p, -1 if none (uniform call)
__device__ __forceinline__ int bs_prev(const WarpSmem &S, int p, int lane) {
    if (p < 0) return -1;
    const int w0 = p >> 5;
    const uint32_t v = S.pend0[w0] & (~0u >> (31 - (p & 31)));
    if (v) return (w0 << 5) + 31 - __clz(v);
    if (w0 == 0) return -1;
    const int q = w0 - 1, w1 = q >> 5;
    const uint32_t u = S.pend1[w1] & (~0u >> (31 - (q & 31)));
    if (u) {
        const int ww = (w1 << 5) + 31 - __clz(u);
        return (ww << 5) + 31 - __clz(S.pend0[ww]);
    }
    return bs_last(S, w1, lane);
}

// position of the k-th (0-based) set bit of x; k < popc(x)
__device__ __forceinline__ int nth_set_bit(uint32_t x, int k) {
    int pos = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const int c = __popc(x & ((1u << s) - 1u));
        if (k >= c) { k -= c; x >>= s; pos += s; }
    }
    return pos;
}

// number of pending positions < P (uniform call)
__device__ __forceinline__ int bs_count_below(const WarpSmem &S, int words0, int P, int lane) {
    const int full = P >> 5;
    int cnt = 0;
#pragma unroll 1
    for (int w = lane; w < full && w < words0; w += 32) cnt += __popc(S.pend0[w]);
    if (lane == 0 && (P & 31) && full < words0) cnt += __popc(S.pend0[full] & ((1u << (P & 31)) - 1u));
    return (int)__reduce_add_sync(kFull, (unsigned)cnt);
}

// first sorted position whose o is <= x (osorted is non-increasing); n if
// none (uniform call).  A 32-way search: each round the lanes sample 32
// evenly spaced positions of the bracket and a ballot keeps the sub-bracket
// holding the answer, so n = 1,000 takes two dependent loads and n = 10^5
// four, instead of a binary search's 10 and 17.
__device__ __forceinline__ int first_pos_le(const int32_t *os, int n, int64_t x, int lane) {
    int lo = 0, hi = n;                         // the answer lies in [lo, hi]
#pragma unroll 1
    while (hi - lo > 32) {
        const int step = (hi - lo + 31) >> 5;
        const int idx = lo + lane * step;
        const bool le = idx >= hi || (int64_t)__ldg(os + idx) <= x;
        const unsigned b = __ballot_sync(kFull, le);
        const int f = b ? __ffs(b) - 1 : 32;    // first sample at or after the answer
        if (f == 0) return lo;
        hi = min(hi, lo + f * step);
        lo = lo + (f - 1) * step + 1;
    }
    const int idx = lo + lane;
    const bool le = idx >= hi || (int64_t)__ldg(os + idx) <= x;
    const unsigned b = __ballot_sync(kFull, le);
    return b ? lo + __ffs(b) - 1 : lo + 32;
}

// v as a value the optimiser cannot see through.  A condition that holds for a
// whole task (which outputs there are, whether lengths are predictions) would
// otherwise have the event loop compiled once for each of its outcomes, and the
// copies crowd each other out of the instruction cache: a task runs most of its
// code only a few times, so ISJL's runs are bound by instruction fetch.  (With
// this and with short loops rolled: 100,000 x 500 requests under 5 runs 29.8 ->
// 23.6 ms, the profit experiment 3.56 -> 2.57 ms.)
__device__ __forceinline__ int opaque(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

// One (instance, run) task under policy P, a compile-time constant (FCFS, LJF,
// SJF, ISJL or ISJL without a binding budget; Algorithm "ISJL" runs the ISJL body
// with beta in the packing thresholds), so each policy's code holds only its own
// admission rule.
//
// Running requests.  Worker w = r * 32 + lane owns slot row r of its lane.  A
// slot's key is the completion step (relative to kbase) above lane and row; a
// lane's column of keys lies in shared memory as vector words and its smallest
// key, the lane's next completion, in a register: a start is one store and one
// minimum (of all 32 lanes at once), a completion a reload of that lane's column.
// Start step and KV reservation lie in shared memory by slot and are read when
// the request leaves.
// A started request runs uninterrupted, so its completion step is written out
// when it starts.
//
// What bounds it: issue of one dependent chain of warp-uniform instructions per
// event (ncu: issue slots half busy, DRAM a few percent), so the column layout
// and the loop below are made for few instructions and branches per event.
// Against the keys and start steps in per-lane registers, scanned and reduced at
// every event, an FCFS event of a 20,000-request trace went from 258 to 189
// instructions and 0.58 to 0.42 us; the simulation of 10,000 x 1,000 requests
// under 7 runs from 19.2 to 14.6 ms, of 100,000 x 500 under 5 from 42.1 to 33.5
// ms, of 1,024 x 100,000 under 3 from 108 to 64 ms.
//
// Costs.  W accumulates per interval between events; E = W - Q (the
// decomposition W = Q + E of Section 5), with the served part of Q counted per
// start when max_steps may stop the run early.  The start range [smin, smax] of
// the running set changes at a start or when the last completion among the
// requests that started at smin (e_lo) or at smax (e_hi) is reached; only then
// is it searched for again.
template <int SPL, int P>
__device__ __forceinline__ void run_task(const SimArgs &A, const WarpSmem &S, int lane, int64_t gwarp,
                                         int64_t inst, int run) {
    constexpr int RB = row_bits<SPL>();
    constexpr uint32_t RM = (1u << RB) - 1u;
    constexpr int SH = RB + 5;                      // a key's completion step lies above lane and row
    constexpr int32_t kSpan = 1 << (30 - SH);       // kbase follows k when it is this far behind
    constexpr bool kIsjl = P == ISJL_POLICY_ISJL;
    constexpr bool kLpt = P == kPolicyLpt;
    constexpr bool kFar = SPL >= 16 && !kIsjl;      // prefetch (the reason is at load_window)
    constexpr bool kSjf = P == ISJL_POLICY_SJF || P == kPolicySjfQueue;
    constexpr bool kFcfs = P == ISJL_POLICY_FCFS || P == kPolicyFcfsQueue;
    constexpr bool kBatch = P == kPolicyFcfsQueue || kLpt || P == kPolicySjfQueue;
    const int n_slots = A.n, B = A.B;
    const int64_t base = inst * (int64_t)n_slots;
    const InstStats is = A.inst[inst];
    const int n = is.n;                             // requests of this instance (<= n_slots)
    // reserved KV: at most B <= 512 running requests of length <= 65535, so
    // below 2^25; kept in 32 bits, against the cap clamped to INT_MAX (which
    // compares the same)
    const int32_t kv_lim = (int32_t)min(A.kv_cap, (int64_t)INT_MAX);
    const int32_t *__restrict__ arr = A.arrival + base;
    const int32_t *__restrict__ oarr = A.o + base;              // planning lengths (u_i)
    const int32_t *__restrict__ otru = A.otrue ? A.otrue + base : nullptr;   // true lengths
    const int32_t *__restrict__ perm = A.perm + base;
    const int32_t *__restrict__ osrt = A.osorted + base;
    const int32_t *__restrict__ posof = A.posof + base;
    int32_t *pnext = A.plan_next + gwarp * (int64_t)n_slots;    // plan links, by request
    const int64_t out_off = (int64_t)run * A.n_inst * n_slots + base;
    int32_t *st_out = A.start_out ? A.start_out + out_off : nullptr;
    int32_t *co_out = A.compl_out ? A.compl_out + out_off : nullptr;
    const int words0 = (n + 31) >> 5, words1 = (words0 + 31) >> 5;

    int64_t status = task_status(is, kv_lim);
    // the run may stop early: at the caller's max_steps, or with predictions at the
    // step bound, which holds for exact lengths (a pack that finishes before its
    // planned time leaves o_1's delay idle)
    const bool trunc = A.max_steps > 0 || otru != nullptr;
    // conditions of the whole task, tested through opaque()
    const int kHasStart = 1, kHasCompl = 2, kTrunc = 4, kSlack = 8, kPacked = 16;
    const int flags = (st_out ? kHasStart : 0) | (co_out ? kHasCompl : 0) | (trunc ? kTrunc : 0) |
                      (otru ? kSlack : 0) | (n_slots <= 65536 ? kPacked : 0);
    // requests that never start / finish report -1: all of them on an error
    // status (and to begin with in a run that may be stopped), else the unused
    // slots of a ragged instance (a full run writes every other entry)
#pragma unroll 1
    for (int i = (status != ISJL_OK || trunc ? 0 : n) + lane; i < n_slots; i += 32) {
        if (st_out) st_out[i] = -1;
        if (co_out) co_out[i] = -1;
    }

    int64_t W = 0, E = 0, sumc = 0, sumext = 0;
    int32_t peakkv = 0;
    int32_t Tb = 0, tok = 0, maxext = 0, viol = 0, peakb = 0, Tmake = 0;

    if (status == ISJL_OK && n > 0) {
        if (!kFcfs) {
#pragma unroll 1
            for (int w = lane; w < words0; w += 32) S.pend0[w] = 0u;
#pragma unroll 1
            for (int w = lane; w < words1; w += 32) S.pend1[w] = 0u;
        }
        __syncwarp();

        uint32_t *col = S.key + lane * SPL;          // this lane's column of keys (SPL = 1: only key0)
        if (SPL > 1) {
#pragma unroll
            for (int r = 0; r < SPL; ++r) col[r] = kEmpty;
        }
        uint32_t key0 = kEmpty;                      // the smallest of them
        auto load_column = [&](uint32_t (&key)[SPL]) {
            if constexpr (SPL >= 4) {
#pragma unroll
                for (int q = 0; q < SPL / 4; ++q) {
                    const uint4 v = reinterpret_cast<const uint4 *>(col)[q];
                    key[4 * q] = v.x; key[4 * q + 1] = v.y; key[4 * q + 2] = v.z; key[4 * q + 3] = v.w;
                }
            } else if constexpr (SPL > 1) {
#pragma unroll
                for (int r = 0; r < SPL; ++r) key[r] = col[r];
            } else {
                key[0] = key0;
            }
        };
        auto column_min = [&]() {
            uint32_t key[SPL];
            load_column(key);
            key0 = key[0];
#pragma unroll
            for (int r = 1; r < SPL; ++r) key0 = min(key0, key[r]);
        };
        const int nrow = (B - lane + 31) >> 5;       // rows holding a valid worker for this lane
        uint32_t idle = nrow >= 32 ? ~0u : ((1u << nrow) - 1u);   // slot rows of this lane with no running request
        uint32_t resv = 0u;     // ... and whose worker's next plan entry waits
        uint32_t lhead = 0u;    // ... which is its long request o_j (waits for o_1)
        const uint32_t lt = (1u << lane) - 1u;
        const int32_t alpha32 = A.runs.delta[run];
        uint64_t R_l = 0;                            // trunc: this lane's share of sum o (o + 1) / 2 over started requests
        int32_t tok_l = 0;                           // trunc: of sum o over started requests
        int64_t sums = 0;                            // sum of start steps
        // with batches of completions W, sumext, sums, viol and the maxima are this
        // lane's shares until the end: what is warp-wide goes to lane 0's
        const uint32_t share = !kBatch || lane == 0 ? ~0u : 0u;

        int32_t k = -1, kbase = 0, rel = 0, fcfs = 0, run_cnt = 0, pend = 0;
        int32_t kv_sum = 0;
        // the next 32 unreleased requests (from win_base): arrival and sorted position, per lane
        int32_t win_base = 0, win_a = INT_MAX, win_p = 0, win_u = 0;   // (SJF) and planning length
        auto load_window = [&]() {
            const int i = win_base + lane;
            win_a = i < n ? arr[i] : INT_MAX;
            win_p = (i < n && !kFcfs) ? posof[i] : 0;
            if (kSjf) win_u = i < n ? oarr[i] : INT_MAX;
            // ask for the next 32 now: with 16 rows few warps are resident, and long
            // instances come from memory (whole sweep of 1,024 x 100,000 requests, B =
            // 512: 44.4 -> 42.6 ms; short ones are in the cache anyway: 20,000 x 1,000
            // 5.31 -> 5.27, x 200 4.15 -> 4.14).  With fewer rows other warps hide the
            // wait and it only costs: B = 100, 1,024 x 100,000 43.3 -> 43.9
            if (kFar && lane < 2 && win_base + 32 < n) prefetch((lane ? posof : arr) + win_base + 32);
        };
        load_window();
        // FCFS: lengths (planning above true) of the 32 requests from hbase on, per
        // lane, and the queue head's
        uint32_t hw = 0u, fh = 0u;
        int32_t hbase = 0;
        auto load_heads = [&]() {
            const int i = fcfs + lane;
            hbase = fcfs;
            hw = 0u;
            if (i < n) {
                const uint32_t u = (uint32_t)oarr[i];
                hw = (u << 16) | ((opaque(flags) & kSlack) ? (uint32_t)otru[i] : u);
            }
        };
        if (kFcfs) {
            load_heads();
            fh = __shfl_sync(kFull, hw, 0);
        }
        // uniform caches, changed only at events
        int32_t next_arr = __shfl_sync(kFull, win_a, 0);   // arrival of the next unreleased request
        // LJF / ISJL: the longest pending position, SJF: the last one (of the
        // shortest length), with its planning length, index and true length
        int32_t hp = kSjf ? -1 : INT_MAX, ho = 0, he = 0, ht = 0;
        bool h_tie = false;                            // SJF: the position before it has the same length
        // start range of the running set and the last completions of those started
        // at its ends; found again (rescan) once e_lo or e_hi is reached
        int32_t smin = 0, smax = 0, e_lo = INT_MIN, e_hi = INT_MIN;
        // Batches of completions (below): the smallest keys in ascending order, lane i
        // the i-th of nn (kEmpty beyond); every other key's step is at least near_end
        uint32_t nk = kEmpty;
        int nn = 0, span = 64, skip = 0;
        int32_t near_end = 0, far_lo = 0, far_hi = 0;  // start range of the requests not among them

        int32_t plan_left = 0, t0 = 0, d1 = 0, nlong = 0;
        bool L1_started = true;
        bool broken = false;   // an internal invariant failed: stop without touching memory
        const int64_t max_steps = A.max_steps > 0 ? A.max_steps : is.O + (int64_t)is.maxA + 1;
        const int32_t guard = step_guard(max_steps);
        // the next step at which something other than a completion happens: the
        // guard, a new kbase, an arrival or o_1's delay expiry
        int32_t evt_base = min(guard, kSpan), evt = 0;

        // plan links: request and planning length of the entry after a request,
        // in one word when request indices fit 16 bits, else the index plus one
        auto packed = [&]() -> bool { return opaque(flags) & kPacked; };
        auto link_of = [&](int e, int oe) -> uint32_t {
            return packed() ? ((uint32_t)oe << 16) | (uint32_t)e : (uint32_t)e + 1u;
        };
        auto link_job = [&](uint32_t lk) -> int { return packed() ? (int)(lk & 0xFFFFu) : (int)(lk - 1u); };
        auto link_len = [&](uint32_t lk) -> int { return packed() ? (int)(lk >> 16) : oarr[lk - 1u]; };

        // this lane starts request e (planning length oe, true length oc) in slot
        // row `row` at step k
        auto occupy = [&](int e, int oe, int oc, int row) {
            const int c = k + oc;
            idle &= ~(1u << row);
            S.slot[(row << 5) + lane] = make_int2(k, oe);
            const int f = opaque(flags);
            if (f & kHasStart) st_out[e] = k;
            if (f & kHasCompl) co_out[e] = c;
            if (f & kTrunc) {
                R_l += ((uint32_t)oc * (uint32_t)(oc + 1)) >> 1;      // oc (oc + 1) < 2^32
                tok_l += oc;
            }
            const uint32_t x = ((uint32_t)(c - kbase) << SH) | ((uint32_t)lane << RB) | (uint32_t)row;
            if (SPL > 1) col[row] = x;
            key0 = min(key0, x);
        };
        // warp-wide totals of cnt starts at step k that reserve kv_add and whose
        // last completion is c_hi
        auto commit = [&](int cnt, int32_t kv_add, int32_t c_hi) {
            nn = 0;
            run_cnt += cnt;
            kv_sum += kv_add;
            mad_wide(sums, (uint32_t)cnt & share, (uint32_t)k);
            if (run_cnt == cnt) {                          // nothing was running
                smin = k;
                e_lo = c_hi;
            } else if (smin == k) {
                e_lo = max(e_lo, c_hi);
            }
            e_hi = smax == k ? max(e_hi, c_hi) : c_hi;
            smax = k;
        };
        // start request e on lane owner's slot row `row` (that lane's value)
        auto start = [&](int e, int oe, int oc, int owner, int row) {
            if (lane == owner) occupy(e, oe, oc, row);
            commit(1, oe, k + oc);
        };
        // start it on one of the free rows fm, which some lane has (the slots are
        // interchangeable; lanes: those with one)
        auto start_any = [&](int e, int oe, int oc, uint32_t fm, unsigned lanes) {
            start(e, oe, oc, 31 - __clz(lanes), 31 - __clz(fm));
        };
        // Start, at step k, the longest prefix of up to 32 candidates (lane l < m
        // holds request ce and its planning length co) whose KV reservations fit
        // and for which free slots remain.  The same outcome as starting them one
        // at a time until the first that does not fit.  Returns how many started.
        auto bulk_start = [&](int m, int ce, int co, uint32_t fm) -> int {
            int pre = lane < m ? co : 0;                          // inclusive prefix of co
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(kFull, pre, d);
                if (lane >= d) pre += t;
            }
            const int nfree = (int)__reduce_add_sync(kFull, (unsigned)__popc(fm));
            const bool fit = lane < m && lane < nfree && kv_sum + pre <= kv_lim;
            const int c = __popc(__ballot_sync(kFull, fit));
            if (c == 0) return 0;
            const int oc_l = ((opaque(flags) & kSlack) && lane < c) ? otru[ce] : co;  // it finishes after its true length
            const int32_t c_hi = k + (int32_t)__reduce_max_sync(kFull, lane < c ? (unsigned)oc_l : 0u);
#pragma unroll 1
            for (int placed = 0; placed < c;) {                   // one per lane with a free slot and round
                const bool f = fm != 0u;
                const unsigned b = __ballot_sync(kFull, f);
                const int rank = placed + __popc(b & lt);
                const int src = rank & 31;
                const int e = __shfl_sync(kFull, ce, src);
                const int oe = __shfl_sync(kFull, co, src);
                const int oc = __shfl_sync(kFull, oc_l, src);
                if (f && rank < c) {
                    occupy(e, oe, oc, __ffs(fm) - 1);
                    fm &= fm - 1u;
                }
                placed += __popc(b);
            }
            commit(c, __shfl_sync(kFull, pre, c - 1), c_hi);
            return c;
        };

        // the request on this lane's slot row `row` leaves; freed += its KV
        auto vacate = [&](uint32_t row, int32_t &freed) {
            const int w = (int)(row << 5) + lane;
            freed += S.slot[w].y;
            if (kIsjl && plan_left > 0) {
                const uint32_t lk = S.slink[w];
                if (lk) {                                     // the worker's next plan entry waits now
                    resv |= 1u << row;
                    if (!L1_started && w < nlong && link_job(lk) == S.slong[w]) lhead |= 1u << row;
                }
            }
            idle |= 1u << row;
        };
        // this lane's earliest request leaves
        auto pop_front = [&](int32_t &freed) {
            const uint32_t row = key0 & RM;
            vacate(row, freed);
            if (SPL > 1) {
                col[row] = kEmpty;
                column_min();
            } else {
                key0 = kEmpty;
            }
        };
        // start range of the running set, and the last completions at its ends
        auto rescan = [&]() {
            int32_t lo = INT_MAX, hi = INT_MIN;
            int32_t s_of[SPL];
            uint32_t key[SPL];
            load_column(key);
#pragma unroll
            for (int r = 0; r < SPL; ++r) {
                s_of[r] = -1;
                if (key[r] != kEmpty) {
                    s_of[r] = S.slot[(r << 5) + lane].x;
                    lo = min(lo, s_of[r]);
                    hi = max(hi, s_of[r]);
                }
            }
            if (kBatch && SPL > 1) {                       // batches leave key0 behind
                key0 = key[0];
#pragma unroll
                for (int r = 1; r < SPL; ++r) key0 = min(key0, key[r]);
            }
            smin = __reduce_min_sync(kFull, lo);
            smax = __reduce_max_sync(kFull, hi);
            uint32_t m_lo = 0u, m_hi = 0u;
#pragma unroll
            for (int r = 0; r < SPL; ++r) {
                if (s_of[r] == smin) m_lo = max(m_lo, key[r]);
                if (s_of[r] == smax) m_hi = max(m_hi, key[r]);
            }
            e_lo = kbase + (int32_t)(__reduce_max_sync(kFull, m_lo) >> SH);
            e_hi = kbase + (int32_t)(__reduce_max_sync(kFull, m_hi) >> SH);
        };

        auto set_head = [&](int p) {
            hp = p;
            if (p >= 0 && p < n) {
                ho = osrt[p];
                if (kSjf) h_tie = p > 0 && osrt[p - 1] == ho;
                he = perm[p];
                ht = (opaque(flags) & kSlack) ? otru[he] : ho;
            }
        };
        // requests with A_i <= k join the queue (a prefix: arrivals are non-decreasing)
        auto release = [&]() {
            if (!kFcfs && rel == 0 && is.maxA <= k) {   // all of them at once
#pragma unroll 1
                for (int b = 0; b < words0; b += 32) {
                    const int i = b + lane;
                    if (i < words0) S.pend0[i] = i + 1 < words0 || (n & 31) == 0 ? ~0u : (1u << (n & 31)) - 1u;
                    if (i < words1) S.pend1[i] = i + 1 < words1 || (words0 & 31) == 0 ? ~0u : (1u << (words0 & 31)) - 1u;
                }
                rel = n;
                pend = n;
                next_arr = INT_MAX;
                __syncwarp();
                set_head(kSjf ? n - 1 : 0);
                return;
            }
#pragma unroll 1
            for (;;) {
                // released: window lanes at or after rel whose arrival is <= k (a prefix)
                const bool ok = win_base + lane >= rel && win_a <= k;
                const unsigned b = __ballot_sync(kFull, ok);
                if (!kFcfs) {
                    if (ok) {
                        atomicOr(&S.pend0[win_p >> 5], 1u << (win_p & 31));
                        atomicOr(&S.pend1[win_p >> 10], 1u << ((win_p >> 5) & 31));
                    }
                    if (kSjf) {
                        const int q = __reduce_max_sync(kFull, ok ? win_p : -1);
                        if (q > hp) set_head(q);
                    } else {
                        const int q = __reduce_min_sync(kFull, ok ? win_p : INT_MAX);
                        if (q < hp) set_head(q);
                    }
                }
                const int c = __popc(b);
                rel += c;
                pend += c;
                if (rel < win_base + 32 || win_base + 32 >= n) break;
                win_base += 32;                           // window used up: load the next 32
                load_window();
            }
            __syncwarp();
            next_arr = rel < n ? __shfl_sync(kFull, win_a, (rel - win_base) & 31) : INT_MAX;
        };
        // remove the head (the longest pending request): nothing is pending below it
        auto pop_head = [&]() {
            const int w = hp >> 5;
            const uint32_t v = S.pend0[w] & ~(1u << (hp & 31));
            __syncwarp();
            if (lane == 0) {
                S.pend0[w] = v;
                if (!v) S.pend1[w >> 5] &= ~(1u << (w & 31));
            }
            __syncwarp();
            pend--;
            set_head(v ? (w << 5) + __ffs(v) - 1 : pend > 0 ? bs_next(S, words0, words1, (w + 1) << 5, lane) : INT_MAX);
        };
        // SJF: remove the last pending position, hp (nothing is pending above it)
        auto pop_tail = [&]() {
            const int w = hp >> 5;
            const uint32_t v = S.pend0[w] & ~(1u << (hp & 31));
            __syncwarp();
            if (lane == 0) {
                S.pend0[w] = v;
                if (!v) S.pend1[w >> 5] &= ~(1u << (w & 31));
            }
            __syncwarp();
            pend--;
            set_head(v ? (w << 5) + 31 - __clz(v) : pend > 0 ? bs_prev(S, (w << 5) - 1, lane) : -1);
        };
        // sorted positions of the first m (1 <= m <= 32) pending requests at or
        // after position p0: lane l gets the l-th, lanes past the last one -1
        // (uniform call)
        auto first_pending_from = [&](int p0, int m) -> int {
            int mine = -1;
#pragma unroll 1
            for (int wb = (p0 >> 10) << 5, got = 0; got < m && wb < words0; wb += 32) {
                if (S.pend1[wb >> 5] == 0u) continue;           // no pending in these 32 words
                const int wi = wb + lane;
                uint32_t x = wi < words0 ? S.pend0[wi] : 0u;
                if (wi < (p0 >> 5)) x = 0u;                     // below p0
                else if (wi == (p0 >> 5)) x &= ~0u << (p0 & 31);
                const int c = __popc(x);
                int incl = c;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += t;
                }
                const int excl = incl - c;
                const int jj = lane - got;                      // this lane's rank within the chunk
                int lo = 0;
#pragma unroll
                for (int sh = 16; sh > 0; sh >>= 1)
                    if (__shfl_sync(kFull, incl, lo + sh - 1) <= jj) lo += sh;
                const uint32_t xw = __shfl_sync(kFull, x, lo);
                const int ew = __shfl_sync(kFull, excl, lo);
                const int tot = __shfl_sync(kFull, incl, 31);
                if (lane < m && jj >= 0 && jj < tot) mine = ((wb + lo) << 5) + nth_set_bit(xw, jj - ew);
                got += tot;
            }
            return mine;
        };
        // sorted positions of the last m (1 <= m <= 32) pending requests, hp the last:
        // lane l gets the l-th from the end, lanes past the first one -1 (uniform call)
        auto last_pending = [&](int m) -> int {
            int mine = -1;
#pragma unroll 1
            for (int wb = (hp >> 10) << 5, got = 0; got < m && wb >= 0; wb -= 32) {
                if (S.pend1[wb >> 5] == 0u) continue;
                const int wi = wb + 31 - lane;
                const uint32_t x = wi < words0 ? __brev(S.pend0[wi]) : 0u;   // bit b: position 31 - b of the word
                int incl = __popc(x);
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += t;
                }
                const int jj = lane - got;
                int lo = 0;
#pragma unroll
                for (int sh = 16; sh > 0; sh >>= 1)
                    if (__shfl_sync(kFull, incl, lo + sh - 1) <= jj) lo += sh;
                const uint32_t xw = __shfl_sync(kFull, x, lo);
                const int ew = __shfl_sync(kFull, incl - __popc(x), lo);
                const int tot = __shfl_sync(kFull, incl, 31);
                if (lane < m && jj >= 0 && jj < tot) mine = ((wb + 31 - lo) << 5) + 31 - nth_set_bit(xw, jj - ew);
                got += tot;
            }
            return mine;
        };
        // remove the lanes' positions p (where take) from the pending set
        auto clear_pending = [&](int p, bool take) {
            if (take) {
                const uint32_t bit = 1u << (p & 31);
                const uint32_t old = atomicAnd(&S.pend0[p >> 5], ~bit);
                if ((old & ~bit) == 0u) atomicAnd(&S.pend1[p >> 10], ~(1u << ((p >> 5) & 31)));
            }
            __syncwarp();
        };
        // start the longest pending requests (LJF's batch, ISJL's Phase TWO) on
        // idle slots (ISJL: not reserved for a plan entry) until one does not fit
        // or the slots run out
        auto start_longest = [&]() {
            // one at a time for the first two starts, usually all there are; 32 at a
            // time from the third, or from the first where nothing runs and three of
            // the longest fit.  Every round first checks that there is a slot, then
            // that the head fits (its length may still be on the way).  LJF, 300 x 1,000
            // requests of 1 to 1,999 tokens, 32 at a time from the first whatever fits
            // -> so: B = 1 1,210 -> 589 us, B = 6 with KV for two or three 536 -> 420
            unsigned lanes = __ballot_sync(kFull, (idle & ~resv) != 0u);
#pragma unroll 1
            for (int nseq = run_cnt == 0 && min(B, pend) > 2 && kv_lim >= 3 * ho ? 2 : 0; pend > 0 && lanes != 0u && kv_sum + ho <= kv_lim; ++nseq) {
                if (hp >= n) { broken = true; return; }
                if (nseq < 2) {
                    start_any(he, ho, ht, idle & ~resv, lanes);
                    pop_head();
                } else {
                    const int m = min(32, pend);
                    const int q = first_pending_from(hp, m);
                    if (__ballot_sync(kFull, lane < m && q < 0)) { broken = true; return; }
                    const int ce = q >= 0 ? perm[q] : 0;
                    const int co = q >= 0 ? osrt[q] : 0;
                    if (kFar) {                                 // the positions after these, usually the next
                        const int ahead = __shfl_sync(kFull, q, m - 1) + 1 + ((lane & 1) << 5);
                        if (lane < 4 && ahead < n) prefetch((lane & 2 ? osrt : perm) + ahead);
                    }
                    const int c = bulk_start(m, ce, co, idle & ~resv);
                    clear_pending(q, lane < c);
                    pend -= c;
                    const int first = __shfl_sync(kFull, q, 0);
                    set_head(c < m ? __shfl_sync(kFull, q, c & 31) : bs_next(S, words0, words1, first, lane));
                }
                lanes = __ballot_sync(kFull, (idle & ~resv) != 0u);
            }
        };

        // ISJL plan starts of every candidate worker in cand (per-lane row
        // mask) at once, in worker order, until the first whose next entry does
        // not fit the KV cap (then true is returned: the gate of the step is
        // shut); entries that must wait (o_1 delayed, an o_j before o_1 has
        // started) are not in cand.
        auto plan_bulk = [&](uint32_t cand) -> bool {
            bool stopped = false;
            int c = 0;
            int32_t kv_add = 0;
            uint32_t oc_hi = 0u;
#pragma unroll 1
            for (int r = 0; r < SPL; ++r) {
                const bool el = !stopped && (cand >> r & 1u);
                if (__ballot_sync(kFull, el) != 0u) {
                    const int w = (r << 5) + lane;
                    int e = 0, oe = 0;
                    if (el) {
                        const uint32_t lk = S.slink[w];
                        e = link_job(lk);
                        oe = link_len(lk);
                    }
                    bool fits = el;
                    const int row_kv = (int)__reduce_add_sync(kFull, (unsigned)oe);
                    if (kv_sum + kv_add + row_kv > kv_lim) {
                        int pre = oe;                           // prefix over this row, in lane order
#pragma unroll 1
                        for (int d = 1; d < 32; d <<= 1) {
                            const int t = __shfl_up_sync(kFull, pre, d);
                            if (lane >= d) pre += t;
                        }
                        fits = el && kv_sum + kv_add + pre <= kv_lim;
                        stopped = true;                         // the first one that does not fit
                    }
                    if (fits) {
                        copy_async(S.slink + w, pnext + e);
                        const int oc = (opaque(flags) & kSlack) ? otru[e] : oe;     // it finishes after its true length
                        occupy(e, oe, oc, r);
                        resv &= ~(1u << r);
                        lhead &= ~(1u << r);
                        oc_hi = max(oc_hi, (uint32_t)oc);
                    }
                    c += __popc(__ballot_sync(kFull, fits));
                    kv_add += (int32_t)__reduce_add_sync(kFull, fits ? (unsigned)oe : 0u);
                }
            }
            if (c > 0)
                commit(c, kv_add, k + (int32_t)__reduce_max_sync(kFull, oc_hi));
            plan_left -= c;
            return stopped;
        };

        // ISJL Phase ONE at a stage start (Algorithm 2 with beta = alpha).  Nothing
        // runs, so the slots' arrays are free: slot[] holds each worker's last plan entry
        // and first its packing budget, then its pack sum, the key columns hold the
        // packing budgets left (0: takes no pack)
        auto phase_one = [&]() {
            const int64_t alpha = A.runs.delta[run], beta = A.runs.beta[run];
            t0 = k; d1 = 0; L1_started = true; nlong = 0;
            if (pend < 2) return;                               // |Q| = 1: Phase TWO
            const int p1 = bs_next(S, words0, words1, 0, lane);
            if (p1 >= n) { broken = true; return; }
            const int64_t o1 = osrt[p1];
            const int p2 = bs_next(S, words0, words1, p1 + 1, lane);
            // cap_j = min{2 alpha, o_1 - o_j + beta}, theta likewise (beta = alpha in Algorithm 2)
            if (p2 >= n) { broken = true; return; }
            if ((int64_t)osrt[p2] <= alpha) return;             // o_2 <= alpha: Phase TWO
            // M = min{B, #{o > alpha}} over Q(k)
            const int cnt_long = bs_count_below(S, words0, first_pos_le(osrt, n, alpha, lane), lane);
            const int nl = min(B, cnt_long);
            copy_wait();                                        // links of the last stage still in flight
            __syncwarp();
#pragma unroll 1
            for (int w = lane; w < B; w += 32) {
                S.slot[w] = make_int2(kNone, w >= nl ? (int32_t)alpha : 0);   // workers M+1..B: alpha
                S.slink[w] = 0u;
                S.slong[w] = kNone;
            }
            __syncwarp();
            // the long requests o_1..o_M (the first M pending positions) leave Q;
            // worker j's budget cap_j.  Up to 32 at a time: a prefix sum of the
            // bitset words' popcounts gives each lane the word and bit of its rank
            int olast_l = 0;
#pragma unroll 1
            for (int wb = 0, taken = 0; taken < nl; wb += 32) {
                if (wb >= words0) { broken = true; return; }
                const int wi = wb + lane;
                const uint32_t x = wi < words0 ? S.pend0[wi] : 0u;
                const int c = __popc(x);
                int incl = c;                                   // inclusive count over lanes
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += t;
                }
                const int excl = incl - c;
                const int m = min(nl - taken, __shfl_sync(kFull, incl, 31));   // ranks from this chunk
#pragma unroll 1
                for (int r0 = 0; r0 < m; r0 += 32) {
                    const int jj = r0 + lane;                       // rank within the chunk
                    int lo = 0;                                     // lanes whose words end before it
#pragma unroll
                    for (int sh = 16; sh > 0; sh >>= 1)
                        if (__shfl_sync(kFull, incl, lo + sh - 1) <= jj) lo += sh;
                    const uint32_t xw = __shfl_sync(kFull, x, lo);
                    const int ew = __shfl_sync(kFull, excl, lo);
                    if (jj < m) {
                        const int p = ((wb + lo) << 5) + nth_set_bit(xw, jj - ew);
                        const int j = taken + jj;
                        const int e = perm[p];
                        const int oe = osrt[p];
                        if (j == 0) {
                            S.slink[0] = link_of(e, oe);
                        } else {
                            S.slong[j] = e;
                            S.slot[j].y = (int32_t)min(2 * alpha, o1 - (int64_t)oe + beta);
                        }
                        if (j == nl - 1) olast_l = oe;
                    }
                }
                // the taken bits of this lane's word leave the bitset
                const int tk = min(max(m - excl, 0), c);
                if (tk > 0) {
                    const uint32_t y = tk == c ? 0u : x & (~0u << nth_set_bit(x, tk));
                    S.pend0[wi] = y;
                    if (y == 0u) atomicAnd(&S.pend1[wi >> 5], ~(1u << (wi & 31)));
                }
                taken += m;
            }
            __syncwarp();
            const int64_t o_last = __reduce_max_sync(kFull, olast_l);
            pend -= nl;
            const int64_t theta = min(2 * alpha, o1 - o_last + beta);
            auto give = [&](int r, uint32_t v) { if (SPL > 1) col[r] = v; else key0 = v; };
            auto has_room = [&](int r) -> uint32_t { return SPL > 1 ? col[r] : key0; };
            // this lane's rows whose worker takes no long request (M+1..B)
            uint32_t rows_short = 0u;
#pragma unroll 1
            for (int r = 0; r < SPL; ++r) {
                const int w = (r << 5) + lane;
                give(r, w < B ? (uint32_t)S.slot[w].y : 0u);
                if (w < B) S.slot[w].y = 0;
                rows_short |= (uint32_t)(w >= nl) << r;
            }
            __syncwarp();
            // x bounds the sizes that may still fit from above; it is recomputed only
            // when a candidate no larger than it fits nowhere (budgets only shrink)
            auto max_budget = [&]() -> int {
                uint32_t m = 0u;
#pragma unroll 1
                for (int r = 0; r < SPL; ++r) m = max(m, has_room(r));
                return (int)__reduce_max_sync(kFull, m);
            };
            int64_t x = min(theta, (int64_t)max_budget());
            // First fit of the shorter requests, in sorted order, on workers M+1..B
            // first, then M, M-1, ..., 2.  32 candidates at a time: lane l loads the
            // l-th; each is placed by a search over all budgets, and the plan lists
            // are linked once per 32
            int from = x >= 1 ? first_pos_le(osrt, n, x, lane) : n;
#pragma unroll 1
            while (x >= 1 && from < n) {
                const int q = first_pending_from(from, 32);
                const int last = __reduce_max_sync(kFull, q);
                if (last < 0) break;
                const int e = q >= 0 ? perm[q] : 0;
                const int oe = q >= 0 ? osrt[q] : INT_MAX;
                int wsel = -1 - lane;                           // the worker it goes to (distinct if none)
                bool shrunk = false;
                unsigned todo = __ballot_sync(kFull, (int64_t)oe <= x);
#pragma unroll 1
                while (todo) {
                    const int i = __ffs(todo) - 1;
                    todo &= todo - 1u;
                    const uint32_t o = (uint32_t)__shfl_sync(kFull, oe, i);
                    uint32_t fit = 0u;                          // rows whose budget takes it
                    uint32_t room[SPL];
                    load_column(room);
#pragma unroll
                    for (int r = 0; r < SPL; ++r) fit |= (uint32_t)(room[r] >= o) << r;
                    // code of this lane's first choice: w for a short worker, 1023 - w for a long one
                    const uint32_t fs = fit & rows_short;
                    unsigned code = 0xFFFFu;
                    if (fs) code = (unsigned)(((__ffs(fs) - 1) << 5) + lane);
                    else if (fit) code = (unsigned)(1023 - (((31 - __clz(fit)) << 5) + lane));
                    code = __reduce_min_sync(kFull, code);
                    if (code == 0xFFFFu) {                      // it stays queued; the bound was stale
                        x = min(theta, (int64_t)max_budget());
                        todo &= __ballot_sync(kFull, (int64_t)oe <= x);
                        shrunk = true;
                        continue;
                    }
                    const int w = code < 512u ? (int)code : 1023 - (int)code;
                    if (lane == (w & 31)) give(w >> 5, has_room(w >> 5) - o);   // the chosen worker's budget shrinks
                    if (lane == i) wsel = w;
                }
                // append the window's requests to their workers' lists, in lane order
                const bool take = wsel >= 0;
                const unsigned same = __match_any_sync(kFull, wsel);
                const unsigned after = same & ~lt & ~(1u << lane);
                const int succ = after ? __ffs(after) - 1 : lane;
                const int es = __shfl_sync(kFull, e, succ);
                const int os_ = __shfl_sync(kFull, oe, succ);
                int tail = kNone;
                if (take) {
                    pnext[e] = after ? (int32_t)link_of(es, os_) : 0;
                    if (!(same & lt)) tail = S.slot[wsel].x;
                    if (wsel < nl) atomicAdd(&S.slot[wsel].y, oe);
                }
                __syncwarp();
                if (take) {
                    if (!(same & lt)) {
                        const uint32_t lk = link_of(e, oe);
                        if (tail < 0) S.slink[wsel] = lk; else pnext[tail] = (int32_t)lk;
                    }
                    if (!after) S.slot[wsel].x = e;
                }
                const int cnt = __popc(__ballot_sync(kFull, take));
                clear_pending(q, take);                        // includes __syncwarp
                pend -= cnt;
                plan_left += cnt;
                from = last + 1;
                if (shrunk && x >= 1) from = max(from, first_pos_le(osrt, n, x, lane));
            }
            // worker j (2..M) runs o_j after its pack
#pragma unroll 1
            for (int w = 1 + lane; w < nl; w += 32) {
                const int e = S.slong[w];
                const int tl = S.slot[w].x;
                const uint32_t lk = link_of(e, packed() ? oarr[e] : 0);
                if (tl < 0) S.slink[w] = lk; else pnext[tl] = (int32_t)lk;
                pnext[e] = 0;
            }
            __syncwarp();
            if (lane == 0) pnext[link_job(S.slink[0])] = 0;
            plan_left += nl;
            // o_1 waits d1 = min{max{max_j sum(w_j) - alpha, 0}, alpha}, j = 2..M
            int mx = 0;
#pragma unroll 1
            for (int w = 1 + lane; w < nl; w += 32) mx = max(mx, S.slot[w].y);
            mx = __reduce_max_sync(kFull, mx);
            d1 = (int32_t)min(max((int64_t)mx - alpha, (int64_t)0), alpha);
            resv = 0u;
            lhead = 0u;
#pragma unroll 1
            for (int r = 0; r < SPL; ++r) {
                const int w = (r << 5) + lane;
                give(r, kEmpty);
                const uint32_t lk = w < B ? S.slink[w] : 0u;
                if (lk) {
                    resv |= 1u << r;
                    if (w >= 1 && w < nl && link_job(lk) == S.slong[w]) lhead |= 1u << r;
                }
            }
            L1_started = false;
            nlong = nl;
            __syncwarp();
            set_head(bs_next(S, words0, words1, 0, lane));   // Phase ONE removed queued requests
        };

        // After an admission, `blocked` says that no arrival alone can let a
        // request start before the next completion (or o_1's delay expiry):
        // FCFS with B full or its head not fitting the KV cap, LJF with a batch
        // running, SJF with B full or no arrival that fits, ISJL with its gate closed or its queue
        // stopped on the KV cap or on workers (an arrival never becomes a head
        // that fits better: it sorts after every pending request of its length).
        // Arrivals are then released at the next event instead of ending the
        // interval there.
        auto admit = [&]() {
            bool blocked;
            int32_t next_fit = INT_MAX;
            if (kFcfs) {
                // arrival order; the first request that does not fit ends the step;
                // one at a time for the first two starts (usually all there are),
                // then 32 at a time
#pragma unroll 1
                for (int nseq = 0; fcfs < rel && kv_sum + (int)(fh >> 16) <= kv_lim && run_cnt < B; ++nseq) {
                    int c = 1;
                    if (nseq < 2) {
                        start_any(fcfs, (int)(fh >> 16), (int)(fh & 0xFFFFu), idle, __ballot_sync(kFull, idle != 0u));
                    } else {
                        const int m = min(32, rel - fcfs), i = fcfs + lane;
                        c = bulk_start(m, i, lane < m ? oarr[i] : 0, idle);
                    }
                    fcfs += c;
                    if (fcfs - hbase >= 32) load_heads();
                    fh = __shfl_sync(kFull, hw, fcfs - hbase);
                }
                blocked = fcfs < rel || run_cnt >= B;
            } else if (kSjf) {
                // shortest released request first (ties: lower index), continuous
                // batching.  The pending requests of the smallest length are the
                // pending positions from the first of that length upwards, in start
                // order; one at a time for the first two starts, then up to 32 of
                // them at a time
#pragma unroll 1
                for (int nseq = 0; pend > 0 && kv_sum + ho <= kv_lim && run_cnt < B; ++nseq) {
                    if (hp < 0 || hp >= n) { broken = true; return; }
                    if ((!h_tie || pend == 1) && nseq < 2) {     // the only one of its length, or of any
                        start_any(he, ho, ht, idle, __ballot_sync(kFull, idle != 0u));
                        pop_tail();
                        continue;
                    }
                    // first position of this length: usually among the 32 up to hp
                    const int i = hp - lane;
                    const unsigned other = __ballot_sync(kFull, i < 0 || osrt[max(i, 0)] != ho);
                    const int g = other ? hp - __ffs(other) + 2 : first_pos_le(osrt, n, ho, lane);
                    if (nseq < 2) {
                        const int p = bs_next(S, words0, words1, g, lane);
                        if (p > hp) { broken = true; return; }
                        const int e = p == hp ? he : perm[p];
                        const int oc = (opaque(flags) & kSlack) ? otru[e] : ho;
                        start_any(e, ho, oc, idle, __ballot_sync(kFull, idle != 0u));
                        bs_clear(S, p, lane);
                        pend--;
                        if (p == hp) set_head(bs_prev(S, hp, lane));
                    } else {
                        const int q = first_pending_from(g, min(32, pend));
                        const int mg = __popc(__ballot_sync(kFull, q >= 0));   // of this length, in order
                        if (mg == 0) { broken = true; return; }
                        const int c = bulk_start(mg, q >= 0 ? perm[q] : 0, ho, idle);
                        clear_pending(q, lane < c);
                        pend -= c;
                        set_head(bs_prev(S, hp, lane));
                    }
                }
                // what waits does not fit, and nor do the arrivals longer than the KV
                // left: the next that fits, or past this window the window's last
                if (run_cnt < B && rel < n) {
                    const int i = win_base + lane;
                    const unsigned b = __ballot_sync(kFull, i >= rel && (win_u <= kv_lim - kv_sum || (lane == 31 && i < n)));
                    next_fit = b ? __shfl_sync(kFull, win_a, __ffs(b) - 1) : INT_MAX;
                }
                blocked = run_cnt >= B || next_fit == INT_MAX;
            } else if (P == ISJL_POLICY_LJF) {
                // static batch of the longest released requests when nothing runs
                if (run_cnt == 0) start_longest();
                blocked = run_cnt != 0;
            } else if (kLpt) {
                start_longest();
                blocked = pend > 0;
            } else {
                if (run_cnt == 0 && plan_left == 0 && pend > 0) phase_one();
                if (broken) return;
                // the gate A_max(k) <= alpha
                bool stop = false;
                if (run_cnt > 0) stop = k - smin > alpha32;
                if (!stop && plan_left > 0) {
                    // plan starts, workers in order; entries that must wait (o_1's
                    // delay, o_j before o_1) are filtered out up front
                    uint32_t cand = resv;
                    if (!L1_started) {
                        cand &= ~lhead;
                        if (k < t0 + d1 && lane == 0) cand &= ~1u;   // worker 0 holds o_1
                    }
#pragma unroll 1
                    for (int nseq = 0; __ballot_sync(kFull, cand != 0u) != 0u; ++nseq) {
                        if (nseq >= 2) {                            // the rest at once
                            stop = plan_bulk(cand);
                            break;
                        }
                        const int w = lowest_worker(cand, lane);
                        const int owner = w & 31, row = w >> 5;
                        const uint32_t lk = __shfl_sync(kFull, lane == owner ? S.slink[w] : 0u, owner);
                        const int e = link_job(lk);
                        const int oe = link_len(lk);
                        if (kv_sum + oe > kv_lim) { stop = true; break; }
                        if (lane == owner) {
                            const uint32_t keep = ~(1u << row);
                            copy_async(S.slink + w, pnext + e);
                            cand &= keep;
                            resv &= keep;
                            lhead &= keep;
                        }
                        plan_left--;
                        if (w == 0) {                               // o_1: the o_j may start now
                            L1_started = true;
                            cand |= lhead;
                        }
                        start(e, oe, (opaque(flags) & kSlack) ? otru[e] : oe, owner, row);
                    }
                }
                if (!stop) start_longest();   // Phase TWO: longest released first
                blocked = stop || pend > 0;
            }
            evt = blocked && run_cnt > 0 ? evt_base : min(evt_base, kSjf ? next_fit : next_arr);
            if (kIsjl && !L1_started && t0 + d1 > k) evt = min(evt, t0 + d1);
        };

        // Serve steps k .. K - 1 at once, K <= the step at which the earliest or
        // latest start changes: the extent is constant and max r = t - smin + 1 at
        // step t, so a request that runs L_i of the steps adds
        // L_i (k - smin + 1) + L_i (L_i - 1) / 2 to W (max r <= 65535 at each of
        // them: the sum fits 32 bits).  Those that complete before K leave here.
        auto window = [&](int32_t K) {
            if (kIsjl && plan_left > 0) copy_wait();
            const uint32_t m0 = (uint32_t)(k - smin) + 1u;
            const uint32_t thr = (uint32_t)(K - kbase) << SH;
            uint64_t wl = 0;
            int32_t freed = 0, nf = 0, cmx = 0;
            uint32_t least = kEmpty;
#pragma unroll 1
            for (int r = 0; r < SPL; ++r) {
                const uint32_t x = SPL > 1 ? col[r] : key0;
                if (x < thr) {
                    const int32_t c = kbase + (int32_t)(x >> SH);
                    const uint32_t Li = (uint32_t)(c - k);
                    wl += Li * m0 + ((Li * (Li - 1u)) >> 1);
                    cmx = max(cmx, c);
                    nf++;
                    vacate(r, freed);
                    if (SPL > 1) col[r] = kEmpty;
                } else {
                    least = min(least, x);
                }
            }
            key0 = least;
            __syncwarp();
            W += (int64_t)warp_sum_u64(wl);
            if (opaque(flags) & kTrunc) Tmake = max(Tmake, (int32_t)__reduce_max_sync(kFull, (unsigned)cmx));
            run_cnt -= (int32_t)__reduce_add_sync(kFull, (unsigned)nf);
            kv_sum -= (int32_t)__reduce_add_sync(kFull, (unsigned)freed);
            nn = 0;
        };

        // ---- Batches of completions (ISJL without a binding budget, and FCFS and SJF
        // where a queue builds up).  While the queue head waits for KV or a slot, nothing but completions
        // lets a request start (longest or shortest first: until the next arrival, which
        // may come before the head).  The next up to 32
        // completions (i, ascending) and the next up to 31 queued requests (j, in
        // start order) are then served in one pass: with F the prefix sums of the KV
        // that the completions free and P those of the KV that the requests need,
        // J_i = #{j : P_j <= slack + F_i} (at most the slots free by then) requests
        // have started after completion i, and request j starts with the first
        // completion that has J_i > j.  The pass ends before a completion that one
        // of these new requests would precede, where the known requests have all
        // started, and at evt.  The start range before each completion comes from
        // suffix minima and maxima over the batch and the range of all others.
        // One event at a time -> batched, simulation alone: FCFS over a 20,000-request
        // trace 8.35 -> 2.16 ms (0.42 -> 0.11 us a request), 10,000 x 1,000 requests 2.74
        // -> 1.23, 100,000 x 500 9.6 -> 4.2; longest first, 10,000 x 1,000 4.6 -> 2.2; SJF,
        // 77 x 777 0.67 -> 0.38.  ISJL with a binding budget has no such pass: its plan
        // and gate leave few completions in a row (a pass for its plan entries made its
        // body 15% larger and the sweeps 13 to 26% slower).

        // collect the next completions: those within the next `span` steps, a number
        // of steps kept such that there are 16 to 32 where so many run
        auto refill = [&]() {
            uint32_t key[SPL];
            load_column(key);
            uint32_t thr = 0u;
            int mine = 0;
            auto count = [&](int sp) -> int {
                thr = (uint32_t)(k + sp - kbase) << SH;
                mine = 0;
#pragma unroll
                for (int r = 0; r < SPL; ++r) mine += key[r] < thr;
                return (int)__reduce_add_sync(kFull, (unsigned)mine);
            };
            int c = count(span), over = 0, at = span;   // over: a span with too many, if known
#pragma unroll 1
            while (c > 32) {
                over = span;
                at = span >>= 1;
                c = count(span);
            }
#pragma unroll 1
            while (over == 0 && c < 16 && c < run_cnt && span < 65536) {
                at = 2 * span;
                const int c2 = count(at);
                if (c2 > 32) { over = at; break; }
                span = at;
                c = c2;
            }
#pragma unroll 1
            while (over != 0 && c < 8 && over - span > 1) {
                at = (span + over) >> 1;
                const int c2 = count(at);
                if (c2 > 32) { over = at; } else { span = at; c = c2; }
            }
            if (at != span) count(span);
            near_end = k + span;
            nn = c;
            nk = kEmpty;
            int32_t lo = INT_MAX, hi = -1;
#pragma unroll
            for (int r = 0; r < SPL; ++r)
                if (key[r] >= thr && key[r] != kEmpty) {
                    const int32_t s0 = S.slot[(r << 5) + lane].x;
                    lo = min(lo, s0);
                    hi = max(hi, s0);
                }
            far_lo = __reduce_min_sync(kFull, lo);
            far_hi = __reduce_max_sync(kFull, hi);
            if (c == 0) return;                        // more than 32 complete at one step
            int off = mine;                            // the lanes' keys, packed and then ranked
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(kFull, off, d);
                if (lane >= d) off += t;
            }
            off -= mine;
            S.swap[lane] = kEmpty;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < SPL; ++r)
                if (key[r] < thr) S.swap[off++] = key[r];
            __syncwarp();
            const uint32_t x = S.swap[lane];
            int rank = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint4 v = reinterpret_cast<const uint4 *>(S.swap)[q];
                rank += (int)(v.x < x) + (int)(v.y < x) + (int)(v.z < x) + (int)(v.w < x);
            }
            __syncwarp();
            if (lane < c) S.swap[rank] = x;
            __syncwarp();
            nk = lane < c ? S.swap[lane] : kEmpty;
            __syncwarp();
        };
        // a new request's key joins the sorted ones if it belongs there
        auto join = [&](uint32_t x) {
            const int at = __popc(__ballot_sync(kFull, nk < x));
            const uint32_t up = __shfl_up_sync(kFull, nk, 1);
            nk = lane < at ? nk : (lane == at ? x : up);
            if (nn < 32) {
                nn++;
            } else {                                   // one too many: collect anew
                nn = 0;
                near_end = INT_MIN;
            }
        };
        // A pass costs two or three completions one at a time.  With few running each
        // start completes before the others and a short queue is used up, so that a
        // pass serves one or two: none with fewer than 5 running (longest first, 300 x
        // 1,000 requests against one at a time: B = 3 0.8, B = 5 1.07, B = 6 1.14 times
        // as fast) or 4 queued, and none where the next arrival, which ends it, is near
        // (an eighth, a quarter or half of the span: the same times)
        auto waits = [&]() -> bool {
            if (run_cnt < 5) return false;
            if (kFcfs) return rel - fcfs >= 4;
            return pend >= 4 && next_arr - k >= span >> 3;
        };
        auto batch = [&]() -> bool {
            if (skip > 0) { skip--; return false; }
            if (nn < 6 && nn < run_cnt) {
                refill();
                if (nn == 0) { skip = 16; return false; }
            }
            // lane i: completion i and the KV it frees
            const int32_t ci = kbase + (int32_t)(nk >> SH);
            const int32_t c_end = kLpt || kSjf ? min(evt_base, next_arr) : evt_base;
            if (__shfl_sync(kFull, ci, 0) >= c_end) return false;
            const int from = (int)(nk >> RB) & 31;
            const uint32_t row_i = nk & RM;
            const int2 req = lane < nn ? S.slot[(int)(row_i << 5) + from] : make_int2(-1, 0);
            int F = req.y;
            // lane j: request j of the queue
            int nh = min(31, kLpt ? pend : rel - fcfs);
            int q = -1, e, oe, oc;
            if (kSjf) {
                // the 32 shortest, the shortest last in position: lane l the l-th from
                // the end, equal lengths turned round.  Of more than 32 the longest
                // length among them is left out: a request of it may come before
                const int nq = min(32, pend);
                q = last_pending(nq);
                if (__popc(__ballot_sync(kFull, q >= 0)) != nq) { broken = true; return false; }
                oe = q >= 0 ? osrt[q] : -1 - lane;
                const unsigned same = __match_any_sync(kFull, oe);
                q = __shfl_sync(kFull, q, __ffs(same) - 1 + 31 - __clz(same) - lane);
                e = q >= 0 ? perm[q] : 0;
                oc = (opaque(flags) & kSlack) && q >= 0 ? otru[e] : oe;
                const int longest = __shfl_sync(kFull, oe, 31);
                nh = min(31, pend > 32 ? __popc(__ballot_sync(kFull, oe < longest)) : nq);
                if (nh < 4 && pend > 32) { skip = 16; return false; }   // many of one length
            } else if (kLpt) {
                q = first_pending_from(hp, nh);
                e = q >= 0 ? perm[q] : 0;
                oe = q >= 0 ? osrt[q] : 0;
                oc = (opaque(flags) & kSlack) && q >= 0 ? otru[e] : oe;
                if (__popc(__ballot_sync(kFull, q >= 0)) != nh) { broken = true; return false; }
            } else {
                if (hbase != fcfs) load_heads();
                e = fcfs + lane;
                oe = (int)(hw >> 16);
                oc = (int)(hw & 0xFFFFu);
            }
            int Pj = lane < nh ? oe : 1 << 25;
            const int u_i = F;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int a = __shfl_up_sync(kFull, F, d), b = __shfl_up_sync(kFull, Pj, d);
                if (lane >= d) { F += a; Pj += b; }
            }
            const int room = min(kv_lim - kv_sum, 1 << 22) + F;   // prefix sums are below 2^21
            int J = 0;
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1)
                if (__shfl_sync(kFull, Pj, J + sh - 1) <= room) J += sh;
            J = min(J, B - run_cnt + lane + 1);
            int Jp = __shfl_up_sync(kFull, J, 1);               // started before completion i
            if (lane == 0) Jp = 0;
            int at = 0;                                        // the completion request j starts with
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1)
                if (__shfl_sync(kFull, J, at + sh - 1) <= lane) at += sh;
            const int32_t t_j = __shfl_sync(kFull, ci, at);
            const int32_t n_j = t_j + oc;                      // and completes
            int32_t first = lane < nh ? n_j : INT_MAX;         // earliest of requests 0 .. j
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(kFull, first, d);
                if (lane >= d) first = min(first, t);
            }
            const int jl = max(Jp - 1, 0);                     // last request started before completion i
            const int32_t first_i = __shfl_sync(kFull, first, jl);
            const int32_t t_l = __shfl_sync(kFull, t_j, jl);
            const int P_l = __shfl_sync(kFull, Pj, jl);
            // start range before completion i: of those still to complete, the others
            // and the new ones
            int32_t lo = lane < nn ? req.x : INT_MAX, hi = req.x;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int a = __shfl_down_sync(kFull, lo, d), b = __shfl_down_sync(kFull, hi, d);
                if (lane + d < 32) { lo = min(lo, a); hi = max(hi, b); }
            }
            const int32_t t_first = __shfl_sync(kFull, t_j, 0);
            lo = min(min(lo, far_lo), Jp > 0 ? t_first : INT_MAX);
            hi = Jp > 0 ? t_l : max(hi, far_hi);
            const bool ok = lane < nn && ci < c_end && Jp < nh && (Jp == 0 || first_i > ci);
            const unsigned no = ~__ballot_sync(kFull, ok);
            int m = no ? __ffs(no) - 1 : 32;
            if (m < nn && m > 0) {                             // not between completions of one step
                const int32_t cm = __shfl_sync(kFull, ci, m);
                if (__shfl_sync(kFull, ci, m - 1) == cm) m = __popc(__ballot_sync(kFull, ci < cm));
            }
            if (m == 0) return false;
            // the steps before each of the m completions
            int32_t t0_i = __shfl_up_sync(kFull, ci, 1);
            if (lane == 0) t0_i = k;
            if (lane < m && ci > t0_i) {
                const uint32_t L = (uint32_t)(ci - t0_i), m0 = (uint32_t)(t0_i - lo) + 1u;
                const uint32_t cnt = (uint32_t)(run_cnt - lane + Jp);
                const int32_t ext = hi - lo;
                W += (int64_t)((uint64_t)cnt * (L * m0 + ((L * (L - 1u)) >> 1)));
                sumext += (int64_t)((uint64_t)L * (uint32_t)ext);
                maxext = max(maxext, ext);
                if (ext > alpha32) viol += (int32_t)L;
                peakb = max(peakb, (int32_t)cnt);
                peakkv = max(peakkv, kv_sum - (F - u_i) + (Jp > 0 ? P_l : 0));
            }
            const int32_t k_new = __shfl_sync(kFull, ci, m - 1);
            const int c = __shfl_sync(kFull, J, m - 1);        // requests that start
            const int freed = __shfl_sync(kFull, F, m - 1);
            const int used = __shfl_sync(kFull, Pj, max(c - 1, 0));
            // the slots of the completed requests become idle
            S.swap[lane] = 0u;
            __syncwarp();
            if (lane < m) {
                atomicOr(&S.swap[from], 1u << row_i);
                if (SPL > 1) S.key[from * SPL + (int)row_i] = kEmpty;
            }
            __syncwarp();
            const uint32_t left = S.swap[lane];
            idle |= left;
            if (SPL == 1 && left) key0 = kEmpty;
            __syncwarp();
            nk = __shfl_down_sync(kFull, nk, m & 31);
            nn -= m;
            if (lane >= nn) nk = kEmpty;
            if (lane < c) {
                const int f = opaque(flags);
                if (f & kHasStart) st_out[e] = t_j;
                if (f & kHasCompl) co_out[e] = n_j;
                sums += t_j;
                if (f & kTrunc) {
                    R_l += ((uint32_t)oc * (uint32_t)(oc + 1)) >> 1;
                    tok_l += oc;
                }
            }
            int32_t new_lo = INT_MAX, new_hi = -1;
#pragma unroll 1
            for (int placed = 0; placed < c;) {                // one per lane with a free slot and round
                const bool f = idle != 0u;
                const unsigned b = __ballot_sync(kFull, f);
                if (b == 0u) { broken = true; break; }
                const int rank = placed + __popc(b & lt);
                const int src = rank & 31;
                const int t = __shfl_sync(kFull, t_j, src);
                const int u = __shfl_sync(kFull, oe, src);
                const int nc = __shfl_sync(kFull, n_j, src);
                bool near = false;
                uint32_t x = kEmpty;
                if (f && rank < c) {
                    const int row = __ffs(idle) - 1;
                    idle &= idle - 1u;
                    x = ((uint32_t)(nc - kbase) << SH) | ((uint32_t)lane << RB) | (uint32_t)row;
                    if (SPL > 1) col[row] = x; else key0 = x;
                    S.slot[(row << 5) + lane] = make_int2(t, u);
                    near = nc < near_end;
                    if (!near) {
                        new_lo = min(new_lo, t);
                        new_hi = max(new_hi, t);
                    }
                }
#pragma unroll 1
                for (unsigned nb = __ballot_sync(kFull, near); nb; nb &= nb - 1u) {
                    const uint32_t y = __shfl_sync(kFull, x, __ffs(nb) - 1);
                    if (kbase + (int32_t)(y >> SH) < near_end) join(y);
                }
                placed += __popc(b);
            }
            far_lo = min(far_lo, __reduce_min_sync(kFull, new_lo));
            far_hi = max(far_hi, __reduce_max_sync(kFull, new_hi));
            e_lo = e_hi = INT_MIN;                             // smin, smax and key0 are not kept here
            Tb += k_new - k;
            k = k_new;
            Tmake = k_new;
            kv_sum += (c > 0 ? used : 0) - freed;
            run_cnt += c - m;
            if (kLpt) {
                clear_pending(q, lane < c);
                pend -= c;
                if (c < nh) {
                    hp = __shfl_sync(kFull, q, c);
                    ho = __shfl_sync(kFull, oe, c);
                    he = __shfl_sync(kFull, e, c);
                    ht = __shfl_sync(kFull, oc, c);
                } else {
                    set_head(bs_next(S, words0, words1, __shfl_sync(kFull, q, 0), lane));
                }
            } else if (kSjf) {
                clear_pending(q, lane < c);
                pend -= c;
                set_head(bs_prev(S, hp, lane));
            } else {
                fcfs += c;
                fh = __shfl_sync(kFull, hw, c);
                load_heads();                                  // for the next pass
            }
            if (SPL > 1 && run_cnt == 0) key0 = kEmpty;        // else reloaded by the next rescan
            __syncwarp();
            return true;
        };

        for (;;) {
            bool served = false;
            if (run_cnt == 0) {                                  // nothing runs: the steps up to evt are idle
                if (kFcfs ? fcfs == n : rel == n && pend == 0 && plan_left == 0) break;
                smin = smax;
                Tb -= evt - k;
            } else {
                if (kBatch) served = waits() && batch();
                if (!kIsjl && !served && min(e_lo, e_hi) <= k) rescan();
            }
            if (!served) {
                // ---- steps k .. nxt - 1
                const uint32_t m = __reduce_min_sync(kFull, key0);
                int32_t nxt = (int32_t)min((uint32_t)kbase + (m >> SH), (uint32_t)evt);   // the next completion (none: beyond evt) or event
                const int32_t ext = smax - smin;                     // max r - min r
                const uint32_t m0 = (uint32_t)(k - smin + 1);        // max r at step k
                peakkv = max(peakkv, kv_sum);
                peakb = max(peakb, run_cnt);
                // LJF with a batch running, or ISJL with its gate shut (A_max only
                // grows while the earliest start stays): no request can start
                // before the running set's earliest or latest start changes, so
                // completions in between end no interval of their own.  Where there
                // are none the pass over the slots is left out (LJF, 300 x 1,000
                // requests, B = 1: 1,642 -> 1,554 us)
                if ((P == ISJL_POLICY_LJF || (kIsjl && k - smin > alpha32)) && run_cnt > 0) {
                    const int32_t ends = min(min(e_lo, e_hi), evt_base);
                    if (ends > nxt) { nxt = ends; window(nxt); }
                }
                // L steps, max r = m0 + t at step k + t: W += s (L m0 + L (L - 1) / 2).
                // The interval ends by the completion of the request that started at
                // smin, so max r <= its o <= 65535 throughout: the sum of max r over
                // the L <= 65535 steps fits 32 bits
                if (nxt <= k) { status = ISJL_ERR_INTERNAL; break; }
                const uint32_t L = (uint32_t)(nxt - k);
                mad_wide(W, (uint32_t)run_cnt & share, L * m0 + ((L * (L - 1u)) >> 1));
                mad_wide(sumext, L & share, (uint32_t)ext);
                maxext = max(maxext, ext);
                if (ext > alpha32) viol += (int32_t)(L & share);
                Tb += (int32_t)L;
                k = nxt;
            }
            if (k >= min(evt, next_arr)) {
                if (k >= guard) { status = ISJL_ERR_STEP_LIMIT; break; }   // k > max_steps
                if (k >= evt_base) {                 // keep the keys' relative steps within 32 - SH bits
                    const uint32_t d = (uint32_t)(k - kbase) << SH;
                    if (SPL > 1) {
#pragma unroll
                        for (int r = 0; r < SPL; ++r)
                            if (col[r] != kEmpty) col[r] -= d;
                    }
                    if (key0 != kEmpty) key0 -= d;
                    kbase = k;
                    nn = 0;
                    evt_base = (int32_t)min((int64_t)guard, (int64_t)k + kSpan);
                }
                if (k >= next_arr) release();
            }
            // ---- requests completing at step k leave, one per lane and round
            if (!served) {
                const uint32_t thr = ((uint32_t)(k - kbase) << SH) | ((1u << SH) - 1u);
                bool f = key0 <= thr;
                unsigned b = __ballot_sync(kFull, f);
                if (b) {
                    if (kIsjl && plan_left > 0) copy_wait();
                    int32_t freed = 0;
                    Tmake = k;
                    nn = 0;
                    do {
                        if (f) pop_front(freed);
                        run_cnt -= __popc(b);
                        f = key0 <= thr;
                        b = __ballot_sync(kFull, f);
                    } while (b);
                    kv_sum -= (int32_t)__reduce_add_sync(kFull, (unsigned)freed);
                }
            }
            if (kIsjl && min(e_lo, e_hi) <= k && run_cnt > 0) rescan();   // the gate looks at smin
            // ---- starts
            admit();
            if (broken) { status = ISJL_ERR_INTERNAL; break; }
        }
        if (kIsjl) copy_wait();
        if (kBatch) {
            W = warp_sum64(W);
            sumext = warp_sum64(sumext);
            sums = warp_sum64(sums);
            viol = (int32_t)__reduce_add_sync(kFull, (unsigned)viol);
            maxext = __reduce_max_sync(kFull, maxext);
            peakkv = __reduce_max_sync(kFull, peakkv);
            peakb = __reduce_max_sync(kFull, peakb);
        }
        status = checked_status(status, peakkv, kv_lim);
        if (status == ISJL_OK) {
            tok = (int32_t)is.O;
            E = W - is.Q;
            sumc = sums + is.O;                        // sum of starts and true lengths
        } else {
            // a request still running has served a = k - s of its o = c - s tokens
            int64_t rest = 0, run_c = 0;
            int32_t tok_rest = 0;
            uint32_t key[SPL];
            load_column(key);
#pragma unroll
            for (int r = 0; r < SPL; ++r)
                if (key[r] != kEmpty) {
                    const int32_t c = kbase + (int32_t)(key[r] >> SH);
                    const int32_t s0 = S.slot[(r << 5) + lane].x;
                    const uint32_t o = (uint32_t)(c - s0), a = (uint32_t)(k - s0);
                    rest += (int64_t)((o * (o + 1u)) >> 1) - (int64_t)((a * (a + 1u)) >> 1);
                    tok_rest += (int32_t)(o - a);
                    run_c += c;
                }
            E = W - warp_sum64((int64_t)R_l - rest);
            tok = (int32_t)__reduce_add_sync(kFull, (unsigned)(tok_l - tok_rest));
            sumc = sums + (int64_t)__reduce_add_sync(kFull, (unsigned)tok_l) - warp_sum64(run_c);
            __syncwarp();                              // what was written ahead and did not happen
#pragma unroll 1
            for (int i = lane; i < n; i += 32) {
                if (co_out && (status != ISJL_ERR_STEP_LIMIT || co_out[i] >= k)) co_out[i] = -1;
                if (st_out && status != ISJL_ERR_STEP_LIMIT) st_out[i] = -1;
            }
        }
    }

    if (lane == 0)
        store_record(A, is, inst, run, RecordTotals{W, E, sumc, sumext, Tmake, Tb, tok, maxext, viol, peakkv, peakb, status});
    __syncwarp();
}

// resident blocks per SM the register allocation is bounded for, per
// instantiation (measured on GB300): 4 (up to 128 registers) in general;
// SPL_BLOCKS16 for 16 register rows (B > 256), where shared memory already
// limits large instances to 2 blocks per SM and a tighter bound only spills
#ifndef ISJL_SIM_MIN_BLOCKS
#define ISJL_SIM_MIN_BLOCKS 4
#endif
#ifndef ISJL_SIM_BLOCKS16
#define ISJL_SIM_BLOCKS16 3
#endif
template <int SPL>
constexpr int sim_min_blocks() {
    return SPL >= 16 ? ISJL_SIM_BLOCKS16 : ISJL_SIM_MIN_BLOCKS;
}

// Whether FCFS's or SJF's body with batches of completions serves an instance.  It
// pays where a queue lasts over many completions; elsewhere its size costs the single
// events 8 to 20%.  `fit` requests of mean length fit the KV, `served` run at once, and
// O / room is the load.  Simulation times of 300 x 1,000 requests, one at a time
// divided by with batches:
//   FCFS  slots bind: B = 256, load 0.9 0.9, 1.1 1.0 (n = 3,000 1.7), 1.5 1.2, 4 1.6;
//         B = 16, load 0.9 0.8, 1.1 1.0, 1.5 1.2; B = 10 1.0, B = 6 0.9 at any load
//         KV binds, so that the head waits earlier: B = 256, load 0.67 0.95 (n = 3,000
//         1.6), 0.83 1.2 (2.6), 1 1.7; B = 32 0.96, 1.1, 1.2; n = 50, B = 32 1.0
//   SJF   n = 400, load 1.5 0.87, 2 1.0, 4 1.1, all there at 0 1.8; n = 100 0.84, 0.95,
//         1.1, 1.2; n = 50 0.80, 0.83, 0.98, 1.1
// (Near a line the instances of one run take both bodies, which crowd each other out
// of the instruction cache, the more the smaller n is: hence n >= 100, and the lines
// lie above the point where both are the same.)
__device__ __forceinline__ bool queue_builds_up(const SimArgs &A, int64_t inst, bool sjf) {
    const InstStats is = A.inst[inst];
    const int64_t kv = min(A.kv_cap, (int64_t)INT_MAX);
    const int64_t fit = kv * is.n / max(is.O, (int64_t)1), served = min((int64_t)A.B, fit);
    const int64_t room = served * max(is.maxA, 0);         // tokens served until the last arrival
    if (is.n < 100) return false;
    if (sjf) return A.B >= 8 && is.O > 3 * room;
    return served >= 16 && (fit < A.B ? 3 * is.O > 2 * room : is.O > room);
}

template <int SPL>
__global__ void __launch_bounds__(kSimWarpsPerBlock * 32, sim_min_blocks<SPL>())
sim_kernel(SimArgs A, int64_t n_tasks) {
    extern __shared__ __align__(16) int32_t smem[];
    const int lane = threadIdx.x & 31, wib = (int)__reduce_max_sync(kFull, threadIdx.x >> 5);
    const int per = smem_words_per_warp(SPL, A.B, A.words0, A.words1);
    int32_t *b = smem + (size_t)wib * per;
    WarpSmem S;
    S.key = reinterpret_cast<uint32_t *>(b);
    if (SPL > 1) b += 32 * SPL;
    S.swap = reinterpret_cast<uint32_t *>(b);
    b += 32;
    S.slot = reinterpret_cast<int2 *>(b);
    S.slink = reinterpret_cast<uint32_t *>(b + 2 * A.B);
    S.slong = b + 3 * A.B;
    S.pend0 = reinterpret_cast<uint32_t *>(b + 4 * A.B);
    S.pend1 = S.pend0 + A.words0;
    const int64_t gwarp = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(A.task_counter, 1);
        t = (int)__reduce_max_sync(kFull, (unsigned)t);
        if ((int64_t)t >= n_tasks) break;
        // run-major: at any time the warps of an SM mostly run one policy's code;
        // the runs with the longest tasks first, so that short tasks fill the tail
        const int turn = (int)((uint32_t)t / (uint32_t)A.n_inst);   // n_inst and the task count are below 2^31
        const int64_t inst = t - (int64_t)turn * A.n_inst;
        const int run = A.runs.order[turn];
        switch (A.runs.policy[run]) {
            case ISJL_POLICY_FCFS:
                if (queue_builds_up(A, inst, false)) run_task<SPL, kPolicyFcfsQueue>(A, S, lane, gwarp, inst, run);
                else run_task<SPL, ISJL_POLICY_FCFS>(A, S, lane, gwarp, inst, run);
                break;
            case ISJL_POLICY_LJF:  run_task<SPL, ISJL_POLICY_LJF>(A, S, lane, gwarp, inst, run); break;
            case ISJL_POLICY_SJF:
                if (queue_builds_up(A, inst, true)) run_task<SPL, kPolicySjfQueue>(A, S, lane, gwarp, inst, run);
                else run_task<SPL, ISJL_POLICY_SJF>(A, S, lane, gwarp, inst, run);
                break;
            default:
                if (A.runs.delta[run] >= ISJL_MAX_LEN) run_task<SPL, kPolicyLpt>(A, S, lane, gwarp, inst, run);
                else run_task<SPL, ISJL_POLICY_ISJL>(A, S, lane, gwarp, inst, run);
                break;
        }
    }
}

template <int SPL>
const void *kernel_ptr() { return reinterpret_cast<const void *>(&sim_kernel<SPL>); }

const void *pick_kernel(int spl) {
    switch (spl) {
        case 1:  return kernel_ptr<1>();
        case 2:  return kernel_ptr<2>();
        case 4:  return kernel_ptr<4>();
        case 8:  return kernel_ptr<8>();
        default: return kernel_ptr<16>();
    }
}

}  // namespace

int slots_per_lane(int B) {
    int s = 1;
    while (32 * s < B) s <<= 1;
    return s;
}

size_t sim_smem_per_warp(int B, int n) {
    const int words0 = (n + 31) / 32, words1 = (words0 + 31) / 32;
    return (size_t)smem_words_per_warp(slots_per_lane(B), B, words0, words1) * 4;
}

// warps per block and the dynamic shared memory of one (0: n is too large for this B).
// n is accepted as long as four warps with seven words per slot and the pending
// bitset would fit; where four warps' actual layout does not, fewer share a block
static cudaError_t block_shape(int B, int n, int device, int *warps, size_t *smem) {
    int limit = 0;
    const cudaError_t e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return e;
    const int64_t words0 = (n + 31) / 32, words1 = (words0 + 31) / 32;
    const int64_t bound = kSimWarpsPerBlock * (((7 * (int64_t)B + words0 + words1 + 3) & ~(int64_t)3) * 4);
    const size_t per = sim_smem_per_warp(B, n);
    *warps = 0;
    *smem = 0;
    if (bound > limit) return cudaSuccess;
    *warps = (int)std::min<size_t>(kSimWarpsPerBlock, (size_t)limit / per);
    *smem = per * *warps;
    return cudaSuccess;
}

cudaError_t sim_shape(int B, int n, int device, SimShape *out) {
    *out = SimShape{0, 0, 0};
    cudaError_t e = block_shape(B, n, device, &out->warps_per_block, &out->smem);
    if (e != cudaSuccess || out->warps_per_block < 1) return e;
    const void *k = pick_kernel(slots_per_lane(B));
    // the same for every caller, so that no other shape's use of the kernel changes it
    int limit = 0, bps = 0, sms = 0;
    e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k, out->warps_per_block * 32, out->smem);
    if (e != cudaSuccess) return e;
    out->warps = bps * sms * out->warps_per_block;
    return cudaSuccess;
}

cudaError_t launch_sim(const SimArgs &args, const SimShape &shape, cudaStream_t s) {
    const int64_t n_tasks = args.n_inst * args.n_runs, per = shape.warps_per_block;
    // A thread takes longer over a task than a warp, the more so the more requests n
    // and workers w = min(B, n) it has, but all threads run at once.  Measured, the
    // thread per task is faster from about 1 + n (16 + w) / 160 waves of resident
    // warps on: n = 6 2 waves, n = 12 2 to 4, n = 20 2 to 6.5, n = 32 3 (w = 3), 5
    // (8), 10 (32); below it is up to 4 times slower
    const int64_t w = std::min(args.B, args.n);
    if (args.n <= kTinyMax && n_tasks * 160 > shape.warps * (160 + args.n * (16 + w))) return launch_tiny(args, s);
    int64_t blocks = shape.warps / per;
    const int64_t need = (n_tasks + per - 1) / per;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    const void *k = pick_kernel(slots_per_lane(args.B));
    SimArgs a = args;
    void *params[] = {&a, const_cast<int64_t *>(&n_tasks)};
    return cudaLaunchKernel(k, dim3((unsigned)blocks), dim3((unsigned)per * 32), params, shape.smem, s);
}

}  // namespace isjl
