// tiny_kernel.cu -- instances of at most 32 requests, one thread per (instance,
// run) task.
//
// The pending queue, the running workers and a worker's pack are each one 32-bit
// mask, so a task needs no cooperation: a thread steps through its own events with
// the same rules as the warp kernel (sim_kernel.cu), and a warp runs 32 tasks of one
// run.  Requests are known by their sorted position (o desc, index asc): the longest
// pending request is the lowest set bit, the shortest the highest, and a pack runs in
// position order.  Per-worker and per-request words lie in shared memory, word i of
// thread t at i * threads + t, so threads of a warp never share a bank.
//
// A warp per task spends its 32 lanes, its set-up and cold instructions on a few
// events.  Measured, warp -> thread per task: 4,096 instances of 6 requests, B = 3,
// 5 runs 141 -> 26 us; 50,000 of 20, B = 8 2,310 -> 223 us; 50,000 of 32, B = 32
// 2,210 -> 1,233 us.  Latency bound (an event is a walk over the running workers), so
// it needs many tasks: see the rule in launch_sim.
#include <climits>
#include <cstdint>

#include "sim_internal.cuh"

namespace isjl {
namespace {

constexpr int kTinyThreads = 64;

// word i of this thread's column
struct Column {
    int32_t *p;
    int stride;
    __device__ __forceinline__ int32_t &operator[](int i) const { return p[i * stride]; }
};

__device__ __forceinline__ int lowest(uint32_t m) { return __ffs((int)m) - 1; }
__device__ __forceinline__ uint32_t low_bits(int n) { return n >= 32 ? ~0u : (1u << n) - 1u; }

// position of the k-th (0-based) set bit of m
__device__ __forceinline__ int kth_bit(uint32_t m, int k) {
    for (; k > 0; --k) m &= m - 1u;
    return lowest(m);
}

// words of shared memory per thread: completion, start, request and pack of each
// worker, and the planning lengths
__host__ __device__ inline int tiny_words(int B, int n) { return 4 * min(B, n) + n; }

__device__ __forceinline__ void tiny_task(const SimArgs &A, int64_t inst, int run, int32_t *smem, int stride) {
    const InstStats is = A.inst[inst];
    const int n = is.n, n_slots = A.n, policy = A.runs.policy[run];
    const bool isjl = policy == ISJL_POLICY_ISJL || policy == ISJL_POLICY_ISJL_BETA;
    const int64_t base = inst * (int64_t)n_slots;
    const int32_t kv_lim = (int32_t)min(A.kv_cap, (int64_t)INT_MAX);
    const int32_t alpha = A.runs.delta[run];
    const int32_t *arr = A.arrival + base, *perm = A.perm + base, *osrt = A.osorted + base, *posof = A.posof + base;
    const int32_t *otru = A.otrue ? A.otrue + base : nullptr;
    const int64_t out_off = (int64_t)run * A.n_inst * n_slots + base;
    int32_t *st_out = A.start_out ? A.start_out + out_off : nullptr;
    int32_t *co_out = A.compl_out ? A.compl_out + out_off : nullptr;

    RecordTotals t{};
    t.status = task_status(is, kv_lim);
    const bool trunc = A.max_steps > 0 || otru != nullptr;   // the run may stop early (as in sim_kernel.cu)
    for (int i = t.status != ISJL_OK || trunc ? 0 : n; i < n_slots; ++i) {   // what never starts or finishes
        if (st_out) st_out[i] = -1;
        if (co_out) co_out[i] = -1;
    }
    if (t.status == ISJL_OK && n > 0) {
        // more workers than requests change nothing: a pack is opened on the lowest
        // short worker that takes it, and requests that are running need one each
        const int B = min(A.B, n), dim = min(A.B, n_slots);
        const Column C{smem, stride}, S{smem + dim * stride, stride}, J{smem + 2 * dim * stride, stride},
            K{smem + 3 * dim * stride, stride}, U{smem + 4 * dim * stride, stride};
        for (int p = 0; p < n; ++p) U[p] = osrt[p];
        const uint32_t workers = low_bits(B);
        uint32_t pend = 0u, busy = 0u;
        uint32_t plan = 0u;                 // workers with a plan entry left
        uint32_t longs = 0u, long_left = 0u;   // the stage's long requests; workers whose own has not started
        int k = -1, evt = 0, rel = 0, fcfs = 0, run_cnt = 0, kv = 0;
        int t0 = 0, d1 = 0;
        bool L1_started = true;
        const int64_t max_steps = A.max_steps > 0 ? A.max_steps : is.O + (int64_t)is.maxA + 1;
        const int guard = step_guard(max_steps);

        auto start = [&](int p, int w) {
            const int e = perm[p], u = U[p];
            C[w] = k + (otru ? otru[e] : u);
            S[w] = k;
            J[w] = p;
            busy |= 1u << w;
            run_cnt++;
            kv += u;
            if (st_out) st_out[e] = k;
        };
        // Algorithm 2's Phase ONE (nothing runs: C holds the packing budgets left, S
        // the pack sums)
        auto phase_one = [&]() {
            t0 = k;
            d1 = 0;
            L1_started = true;
            if (__popc(pend) < 2) return;
            const int o1 = U[lowest(pend)];
            if (U[lowest(pend & (pend - 1u))] <= alpha) return;      // o_2 <= alpha: Phase TWO
            const int beta = A.runs.beta[run];                       // alpha < 65535 here
            int nl = 0, o_last = 0;
            longs = 0u;
            for (uint32_t m = pend; m && nl < B; m &= m - 1u) {
                const int p = lowest(m);
                if (U[p] <= alpha) break;
                o_last = U[p];
                C[nl] = nl ? min(2 * alpha, o1 - o_last + beta) : 0;
                longs |= 1u << p;
                nl++;
            }
            for (int w = 0; w < B; ++w) {
                if (w >= nl) C[w] = alpha;
                S[w] = 0;
                K[w] = 0;
            }
            pend &= ~longs;
            plan = long_left = low_bits(nl);
            const int theta = min(2 * alpha, o1 - o_last + beta);
            for (uint32_t m = pend; m; m &= m - 1u) {                // first fit: M+1..B, then M, ..., 2
                const int p = lowest(m), u = U[p];
                if (u > theta) continue;
                int w = nl;
                while (w < B && C[w] < u) ++w;
                if (w == B) {
                    w = nl - 1;
                    while (w > 0 && C[w] < u) --w;
                    if (w <= 0) continue;                            // it stays queued
                }
                C[w] -= u;
                S[w] += u;
                K[w] |= (int32_t)(1u << p);
                plan |= 1u << w;
                pend &= ~(1u << p);
            }
            int packs = 0;
            for (int w = 1; w < nl; ++w) packs = max(packs, S[w]);
            d1 = min(max(packs - alpha, 0), alpha);
            L1_started = false;
        };

        for (;;) {
            if (run_cnt == 0 && (policy == ISJL_POLICY_FCFS ? fcfs == n : rel == n && pend == 0u && plan == 0u)) break;
            int c_min = INT_MAX, s_lo = INT_MAX, s_hi = INT_MIN;
            int64_t s_sum = 0;
            for (uint32_t m = busy; m; m &= m - 1u) {
                const int w = lowest(m), s = S[w];
                c_min = min(c_min, C[w]);
                s_lo = min(s_lo, s);
                s_hi = max(s_hi, s);
                s_sum += s;
            }
            const int nxt = min(c_min, evt);
            t.peak_kv = max(t.peak_kv, kv);
            if (nxt <= k || nxt == INT_MAX) t.status = ISJL_ERR_INTERNAL;
            t.status = checked_status(t.status, kv, kv_lim);
            if (t.status != ISJL_OK) break;
            if (run_cnt > 0) {                                       // steps k .. nxt - 1
                const int64_t L = nxt - k;
                const int ext = s_hi - s_lo;
                t.W += run_cnt * (L * (k - s_lo + 1) + L * (L - 1) / 2);
                t.E += L * (s_sum - (int64_t)run_cnt * s_lo);
                t.sum_extent += L * ext;
                t.max_extent = max(t.max_extent, ext);
                if (ext > alpha) t.violations += (int32_t)L;
                t.T_busy += (int32_t)L;
                t.token_adv += (int32_t)(run_cnt * L);
                t.peak_batch = max(t.peak_batch, run_cnt);
            }
            k = nxt;
            if (k >= guard) { t.status = ISJL_ERR_STEP_LIMIT; break; }
            for (; rel < n && arr[rel] <= k; ++rel) pend |= 1u << posof[rel];
            s_lo = INT_MAX;
            for (uint32_t m = busy; m; m &= m - 1u) {
                const int w = lowest(m);
                if (C[w] == k) {
                    const int p = J[w];
                    busy &= ~(1u << w);
                    run_cnt--;
                    kv -= U[p];
                    t.sum_completion += k;
                    t.T_make = k;
                    if (co_out) co_out[perm[p]] = k;
                } else {
                    s_lo = min(s_lo, S[w]);
                }
            }
            if (policy == ISJL_POLICY_FCFS) {
                for (; fcfs < rel && run_cnt < B; ++fcfs) {
                    const int p = posof[fcfs];
                    if (kv + U[p] > kv_lim) break;
                    start(p, lowest(workers & ~busy));
                }
            } else if (policy == ISJL_POLICY_SJF) {
                while (pend && run_cnt < B) {
                    int p = 31 - __clz((int)pend);                   // of its length, the lowest index first
                    const int u = U[p];
                    if (kv + u > kv_lim) break;
                    for (int q = p - 1; q >= 0 && U[q] == u; --q)
                        if (pend >> q & 1u) p = q;
                    pend &= ~(1u << p);
                    start(p, lowest(workers & ~busy));
                }
            } else {
                bool stop = policy == ISJL_POLICY_LJF && run_cnt > 0;
                if (isjl) {
                    if (run_cnt == 0 && plan == 0u && pend) phase_one();
                    stop = run_cnt > 0 && k - s_lo > alpha;          // the gate
                    for (uint32_t m = stop ? 0u : plan & ~busy; m; m &= m - 1u) {
                        const int w = lowest(m);
                        const uint32_t pack = (uint32_t)K[w];
                        if (!pack && (w == 0 ? k < t0 + d1 : !L1_started)) continue;   // o_1 delayed, o_j before o_1
                        const int p = pack ? lowest(pack) : kth_bit(longs, w);
                        if (kv + U[p] > kv_lim) { stop = true; break; }
                        if (pack) K[w] = (int32_t)(pack & (pack - 1u));
                        else { long_left &= ~(1u << w); if (w == 0) L1_started = true; }
                        if (!K[w] && !(long_left >> w & 1u)) plan &= ~(1u << w);
                        start(p, w);
                    }
                }
                while (!stop && pend) {                              // LJF's batch, Phase TWO
                    const uint32_t idle = workers & ~busy & ~plan;
                    const int p = lowest(pend);
                    if (!idle || kv + U[p] > kv_lim) break;
                    pend &= ~(1u << p);
                    start(p, lowest(idle));
                }
            }
            evt = min(guard, rel < n ? arr[rel] : INT_MAX);
            if (!L1_started && t0 + d1 > k) evt = min(evt, t0 + d1);
        }
    }
    if (t.status == ISJL_ERR_INTERNAL)
        for (int i = 0; i < n; ++i) {
            if (st_out) st_out[i] = -1;
            if (co_out) co_out[i] = -1;
        }
    store_record(A, is, inst, run, t);
}

__global__ void __launch_bounds__(kTinyThreads) tiny_kernel(SimArgs A, int64_t n_tasks) {
    extern __shared__ int32_t tiny_smem[];
    const int64_t t = (int64_t)blockIdx.x * kTinyThreads + threadIdx.x;
    if (t >= n_tasks) return;
    const int turn = (int)((uint32_t)t / (uint32_t)A.n_inst);   // n_inst and the task count are below 2^31
    tiny_task(A, t - (int64_t)turn * A.n_inst, A.runs.order[turn], tiny_smem + threadIdx.x, kTinyThreads);
}

}  // namespace

cudaError_t launch_tiny(const SimArgs &args, cudaStream_t s) {
    const int64_t n_tasks = args.n_inst * args.n_runs;
    const size_t smem = sizeof(int32_t) * kTinyThreads * (size_t)tiny_words(args.B, args.n);   // at most 40 KB
    tiny_kernel<<<(unsigned)((n_tasks + kTinyThreads - 1) / kTinyThreads), kTinyThreads, smem, s>>>(args, n_tasks);
    return cudaGetLastError();
}

}  // namespace isjl
