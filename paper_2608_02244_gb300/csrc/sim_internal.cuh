// sim_internal.cuh -- internal definitions shared by the simulator's kernels
// and its C-ABI host code (not part of the public interface).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "isjl_sim.h"

namespace isjl {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarp = 32;
constexpr int kSimWarpsPerBlock = 4;         // 128-thread blocks for the simulation kernel
constexpr int kSortSmallMax = 4096;           // bitonic in shared memory up to this n
constexpr int kRadixThreads = 1024;           // threads of the large-n radix sort

// Per-instance facts derived once per call (policy independent).
struct InstStats {
    int64_t O;        // sum o_i (true lengths)
    int64_t Q;        // sum o_i (o_i + 1) / 2
    int64_t sumA;     // sum of arrivals
    int32_t maxo;     // largest planning length u_i (= o_i without slack): KV feasibility
    int32_t maxA;     // largest arrival
    int32_t status;   // ISJL_OK, ISJL_ERR_INVALID_ARG or ISJL_ERR_INFEASIBLE (o_i < 1)
    int32_t n;        // requests of this instance (its first n slots)
};

// (policy, delta) list of one sweep, passed by value to the kernel.
struct RunList {
    int32_t policy[ISJL_MAX_RUNS];
    int32_t delta[ISJL_MAX_RUNS];
    int32_t beta[ISJL_MAX_RUNS];    // ISJL packing slack: delta, or Algorithm "ISJL"'s beta
    int32_t order[ISJL_MAX_RUNS];   // the runs in the order their tasks are handed out
};

// floor((sqrt(17) - 1) / 4 * alpha) exactly: the largest m with (4m + alpha)^2 <= 17 alpha^2
inline int32_t isjl_beta(int32_t alpha) {
    if (alpha > 1000000) return alpha;   // no plan exists when alpha >= every length
    const int64_t a = alpha;
    int64_t m = (int64_t)(0.780776406404415 * (double)alpha);
    while (m > 0 && (4 * m + a) * (4 * m + a) > 17 * a * a) m--;
    while ((4 * (m + 1) + a) * (4 * (m + 1) + a) <= 17 * a * a) m++;
    return (int32_t)m;
}
inline int32_t run_beta(int32_t policy, int32_t delta) {
    return policy == ISJL_POLICY_ISJL_BETA ? isjl_beta(delta) : delta;
}

// the list of a sweep.  Runs with long tasks go first, so that short ones fill the
// tail: SJF, then ISJL from the largest budget down, FCFS, LJF.  Single runs of
// 10,000 x 1,000 requests: SJF 4.4 ms, ISJL at inf / 1,024 / 256 / 64 / 16 2.3 / 3.9 /
// 1.8 / 1.0 / 0.8, FCFS 1.4, LJF 0.6.  All 7 but SJF take 9.40 ms, in the caller's
// order 9.65; 3,000 x 1,000 with predictions under 7 runs 2.93 against 3.27, 1,500 x
// 701 under all policies 0.95 against 0.96, 1,024 x 100,000 under 3 with B = 100 43
// against 55.  By the single runs 1,024 would come before inf: measured too, that is
// slower (9.71 and 3.17 ms)
inline RunList run_list(int32_t n_runs, const int32_t *policies, const int32_t *deltas) {
    RunList r{};
    auto rank = [&](int32_t i) -> int64_t {
        switch (policies[i]) {
            case ISJL_POLICY_SJF: return (int64_t)1 << 33;
            case ISJL_POLICY_FCFS: return -1;
            case ISJL_POLICY_LJF: return -2;
            default: return deltas[i];
        }
    };
    for (int32_t i = 0; i < n_runs; ++i) {
        r.policy[i] = policies[i];
        r.delta[i] = deltas[i];
        r.beta[i] = run_beta(policies[i], deltas[i]);
        int32_t at = i;                             // stable insertion, the highest rank first
        for (; at > 0 && rank(r.order[at - 1]) < rank(i); --at) r.order[at] = r.order[at - 1];
        r.order[at] = i;
    }
    return r;
}

// launch shape of the simulation kernel for one B and n
struct SimShape {
    int warps_per_block;       // 0: n is too large for this B
    int warps;                 // resident warps
    size_t smem;               // dynamic shared memory per block
};

struct SimArgs {
    const int32_t *arrival;    // [N] instance-major
    const int32_t *o;          // [N] planning length u_i = prompt + output (+ slack)
    const int32_t *otrue;      // [N] true length o_i, or null when there is no slack
    const int32_t *perm;       // [N] sorted position -> request index within its instance
    const int32_t *osorted;    // [N] o at each sorted position (non-increasing)
    const int32_t *posof;      // [N] request index -> sorted position
    const InstStats *inst;     // [n_inst]
    int32_t *plan_next;        // [resident warps * n] ISJL plan links (scratch)
    isjl_record *records;      // [n_runs * n_inst]
    int32_t *start_out;        // [n_runs * N] or null
    int32_t *compl_out;        // [n_runs * N] or null
    int32_t *task_counter;     // work queue head, zeroed by the derive kernel
    int32_t *dev_status;       // first nonzero status of the launch
    int64_t n_inst;
    int32_t n;
    int32_t B;
    int64_t kv_cap;
    int64_t max_steps;         // 0 = per-instance automatic bound
    int32_t n_runs;
    int32_t words0;            // ceil(n / 32): level-0 words of the pending bitset
    int32_t words1;            // ceil(words0 / 32): level-1 summary words
    double c, tau, p0;
    RunList runs;
};

// status of a task before it runs: the instance's, an infeasible length or an
// instance beyond the step counter's range (with exact lengths every schedule ends by
// sum o + max arrival, with predictions the default step bound ends it there)
__device__ __forceinline__ int64_t task_status(const InstStats &is, int32_t kv_lim) {
    if (is.status != ISJL_OK) return is.status;
    if (is.maxo > kv_lim) return ISJL_ERR_INFEASIBLE;
    return is.O + (int64_t)is.maxA + 1 >= (int64_t)(1 << 30) ? ISJL_ERR_INVALID_ARG : ISJL_OK;
}

// the first step that a run of max_steps >= 1 steps does not serve (k > max_steps);
// INT32_MAX, which no run reaches, for every bound beyond the step numbers
__host__ __device__ __forceinline__ int32_t step_guard(int64_t max_steps) {
    return (int32_t)min((uint64_t)max_steps + 1u, (uint64_t)INT32_MAX);   // (unsigned: max_steps may be INT64_MAX)
}

// a run's status given its largest reservation so far: every start is checked
// against the cap, so a reservation beyond it is a library bug
__host__ __device__ __forceinline__ int64_t checked_status(int64_t status, int32_t peak_kv, int32_t kv_lim) {
    return peak_kv > kv_lim ? ISJL_ERR_INTERNAL : status;
}

// what a simulation kernel counted for one task
struct RecordTotals {
    int64_t W, E, sum_completion, sum_extent;
    int32_t T_make, T_busy, token_adv, max_extent, violations, peak_kv, peak_batch;
    int64_t status;
};

// one thread writes the task's record
__device__ __forceinline__ void store_record(const SimArgs &A, const InstStats &is, int64_t inst, int run,
                                             const RecordTotals &t) {
    isjl_record R;
    const bool bad_input = t.status == ISJL_ERR_INVALID_ARG || t.status == ISJL_ERR_INFEASIBLE;
    R.T_make = bad_input ? 0 : t.T_make;
    R.T_busy = bad_input ? 0 : t.T_busy;
    R.O = bad_input ? 0 : is.O;
    R.Q = bad_input ? 0 : is.Q;
    R.W = t.W;
    R.E = t.E;
    R.token_adv = t.token_adv;
    R.sum_completion = t.sum_completion;
    R.sum_latency = bad_input ? 0 : t.sum_completion - is.sumA;
    R.sum_extent = t.sum_extent;
    R.max_extent = t.max_extent;
    R.violations = t.violations;
    R.kv_violations = t.peak_kv > A.kv_cap;   // (and then status is INTERNAL, see checked_status)
    R.peak_kv = t.peak_kv;
    R.peak_batch = t.peak_batch;
    R.status = t.status;
    if (bad_input) {
        R.c_T = R.tau_Q = R.tau_E = R.cost = R.revenue = R.profit = R.throughput = R.ael = 0.0;
    } else {
        // cost decomposition C = tau Q + c T + tau E, no contraction
        R.c_T = __dmul_rn(A.c, (double)t.T_busy);
        R.tau_Q = __dmul_rn(A.tau, (double)is.Q);
        R.tau_E = __dmul_rn(A.tau, (double)t.E);
        R.cost = __dadd_rn(__dadd_rn(R.c_T, R.tau_Q), R.tau_E);
        R.revenue = __dmul_rn(A.p0, (double)is.O);
        R.profit = __dsub_rn(R.revenue, R.cost);
        R.throughput = t.T_make > 0 ? __ddiv_rn((double)is.O, (double)t.T_make) : 0.0;
        R.ael = is.n > 0 ? __ddiv_rn((double)t.sum_completion, (double)is.n) : 0.0;
    }
    A.records[(int64_t)run * A.n_inst + inst] = R;
    if (t.status != ISJL_OK) atomicCAS(A.dev_status, 0, (int32_t)t.status);
}

// host-side launchers (defined in the .cu files)
cudaError_t launch_derive(const int32_t *arrival, const int32_t *prompt, const int32_t *output,
                          const int32_t *count, const int32_t *slack, int32_t *o, int32_t *otrue,
                          InstStats *inst, int32_t *counter, int32_t *dev_status, int64_t n_inst, int32_t n,
                          cudaStream_t s);
cudaError_t launch_sort(const int32_t *o, const InstStats *inst, int32_t *perm, int32_t *osorted, int32_t *posof,
                        int32_t *tmp, int64_t n_inst, int32_t n, cudaStream_t s);
cudaError_t sim_shape(int B, int n, int device, SimShape *out);
cudaError_t launch_sim(const SimArgs &args, const SimShape &shape, cudaStream_t s);
// instances of at most kTinyMax requests, one thread per task
constexpr int kTinyMax = 32;
cudaError_t launch_tiny(const SimArgs &args, cudaStream_t s);
cudaError_t launch_summarize(const isjl_record *records, int64_t n_inst, int32_t n_runs,
                             const RunList &runs, int32_t kv_cap, isjl_summary *out, cudaStream_t s);
size_t sim_smem_per_warp(int B, int n);
int slots_per_lane(int B);

}  // namespace isjl
