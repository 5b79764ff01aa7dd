// prep_kernels.cu -- per-instance preparation and cross-instance summaries.
//
//   derive     o_i = prompt_i + output_i (Section 2), input validation and the
//              policy-independent totals O = sum o_i and
//              Q = sum o_i (o_i + 1) / 2 (Eq. intrinsic-resource-cost)
//   sort       the order o_1 >= o_2 >= ... of Algorithms 1 and 2 (ties by
//              index): a permutation, its inverse and the sorted lengths;
//              bitonic in one warp's registers up to 1,024 requests, in shared
//              memory up to 4,096, a stable two-pass LSD radix sort beyond
//   summarize  per-run totals over all instances, a fixed-order reduction
#include <climits>
#include <cstddef>
#include <cstdint>

#include "sim_internal.cuh"

namespace isjl {
namespace {

constexpr int kSortThreads = 256;
constexpr int kWarpSortMax = 1024;        // one warp sorts an instance in registers up to this n
constexpr int kPrepWarps = 4;             // warps per block of the warp-per-instance kernels

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(kFull, v, s);
    return v;
}
template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v = max(v, __shfl_xor_sync(kFull, v, s));
    return v;
}

// kThreads threads per instance, one block of them or, for one warp, kPrepWarps
// instances per block.  A warp suffices up to 1,024 requests (100,000 x 500: 317
// -> 221 us against a block of 256 threads, whose reduction outlasts its two
// loads per thread); instances of 10^5 take 1,024 threads (1,024 of them: 584 ->
// 420 us).  The first thread also zeroes the simulation's work counter and status.
template <int kThreads>
__global__ void __launch_bounds__(kThreads == 32 ? 32 * kPrepWarps : kThreads)
derive_kernel(const int32_t *__restrict__ arrival, const int32_t *__restrict__ prompt,
              const int32_t *__restrict__ output, const int32_t *__restrict__ count,
              const int32_t *__restrict__ slack, int32_t *__restrict__ o, int32_t *__restrict__ otrue,
              InstStats *inst, int32_t *counter, int32_t *dev_status, int64_t n_inst, int32_t n_slots) {
    constexpr bool kOneWarp = kThreads == 32;
    if (blockIdx.x == 0 && threadIdx.x == 0) { *counter = 0; *dev_status = 0; }
    const int64_t id = kOneWarp ? (int64_t)blockIdx.x * kPrepWarps + (threadIdx.x >> 5) : (int64_t)blockIdx.x;
    if (id >= n_inst) return;                           // (kOneWarp: no block barrier follows)
    const int t0 = kOneWarp ? threadIdx.x & 31 : threadIdx.x;
    const int64_t base = id * n_slots;
    int64_t O = 0, Q = 0, sumA = 0;
    int32_t maxo = 0, maxA = 0, invalid = 0, infeasible = 0;
    int32_t n = count ? count[id] : n_slots;
    if (n < 0 || n > n_slots) { invalid = 1; n = 0; }
#pragma unroll 4
    for (int i = t0; i < n; i += kThreads) {
        const int32_t a = arrival[base + i], p = prompt[base + i], q = output[base + i];
        const int32_t before = i > 0 ? arrival[base + i - 1] : 0;
        const int32_t e = slack ? slack[base + i] : 0;
        const int64_t oi = (int64_t)p + q;
        const int64_t ui = oi + e;                  // planning length (Robust-ISJL's u_i)
        if (a < 0 || p < 0 || q < 0 || e < 0 || before > a || ui > ISJL_MAX_LEN)
            invalid = 1;
        else if (oi < 1) infeasible = 1;
        const bool ok = oi >= 0 && ui <= ISJL_MAX_LEN && e >= 0;
        const int32_t oc = ok ? (int32_t)oi : 0;
        const int32_t uc = ok ? (int32_t)ui : 0;
        o[base + i] = uc;
        if (otrue) otrue[base + i] = oc;
        O += oc;
        Q += (int64_t)oc * (oc + 1) / 2;
        sumA += a;
        maxo = max(maxo, uc);
        maxA = max(maxA, a);
    }
    O = warp_sum(O); Q = warp_sum(Q); sumA = warp_sum(sumA);
    maxo = warp_max(maxo); maxA = warp_max(maxA);
    invalid = warp_max(invalid); infeasible = warp_max(infeasible);
    InstStats st{};
    if (kOneWarp) {
        st.O = O; st.Q = Q; st.sumA = sumA; st.maxo = maxo; st.maxA = maxA;
    } else {
        __shared__ int64_t s64[3][kThreads / 32];
        __shared__ int32_t s32[4][kThreads / 32];
        const int wid = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            s64[0][wid] = O; s64[1][wid] = Q; s64[2][wid] = sumA;
            s32[0][wid] = maxo; s32[1][wid] = maxA; s32[2][wid] = invalid; s32[3][wid] = infeasible;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 0; w < kThreads / 32; ++w) {
                st.O += s64[0][w]; st.Q += s64[1][w]; st.sumA += s64[2][w];
                st.maxo = max(st.maxo, s32[0][w]); st.maxA = max(st.maxA, s32[1][w]);
                invalid |= s32[2][w]; infeasible |= s32[3][w];
            }
    }
    if (t0 == 0) {
        st.status = invalid ? ISJL_ERR_INVALID_ARG : (infeasible ? ISJL_ERR_INFEASIBLE : ISJL_OK);
        st.n = n;
        inst[id] = st;
    }
}

__device__ __forceinline__ uint32_t len_key(int32_t o) {   // larger o sorts first
    const int32_t c = o < 0 ? 0 : (o > ISJL_MAX_LEN ? ISJL_MAX_LEN : o);
    return (uint32_t)(ISJL_MAX_LEN - c);
}

// n <= 1,024: one warp sorts an instance's keys (65535 - o) << 16 | index in
// registers, E per lane (position lane * E + j), by a bitonic network whose strides
// below E stay within a lane and whose others are shuffles; no barrier.  Bound by
// the three arrays it writes (100,000 x 500 requests: 1,466 -> 270 us against the
// network in shared memory with a block barrier per stage; 10,000 x 1,000: 324 ->
// 66 us).
template <int E>
__device__ __forceinline__ void merge_in_lane(uint32_t (&key)[E]) {   // each lane's bitonic run, ascending
#pragma unroll
    for (int stride = E / 2; stride > 0; stride >>= 1)
#pragma unroll
        for (int j = 0; j < E; ++j)
            if ((j & stride) == 0) {
                const uint32_t a = key[j], b = key[j + stride];
                key[j] = min(a, b);
                key[j + stride] = max(a, b);
            }
}

template <int E>
__global__ void __launch_bounds__(32 * kPrepWarps)
sort_warp_kernel(const int32_t *__restrict__ o, const InstStats *__restrict__ inst, int32_t *__restrict__ perm,
                 int32_t *__restrict__ osorted, int32_t *__restrict__ posof, int64_t n_inst, int32_t n_slots) {
    constexpr int kPad = 32 * E + E;              // one word of padding per 32: lane * E + j is free of conflicts
    __shared__ uint32_t sorted[kPrepWarps][kPad];
    __shared__ int32_t place[kPrepWarps][32 * E];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t id = (int64_t)blockIdx.x * kPrepWarps + wib;
    if (id >= n_inst) return;
    const int64_t base = id * n_slots;
    const int n = inst[id].n;
    uint32_t key[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int t = j * 32 + lane;
        key[j] = t < n ? (len_key(o[base + t]) << 16) | (uint32_t)t : 0xffffffffu;
    }
    // runs of 2 .. E within a lane: a run descends where its index has the next bit
#pragma unroll
    for (int size = 2; size <= E; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int j = 0; j < E; ++j)
                if ((j & stride) == 0) {
                    const bool down = size < E ? (j & size) != 0 : (lane & 1) != 0;
                    const uint32_t lo = min(key[j], key[j + stride]), hi = max(key[j], key[j + stride]);
                    key[j] = down ? hi : lo;
                    key[j + stride] = down ? lo : hi;
                }
    // runs of 2 .. 32 lanes; a descending run is sorted ascending on the complements
#pragma unroll 1
    for (int size = 2; size <= 32; size <<= 1) {
        const uint32_t flip = (lane & size) ? 0xffffffffu : 0u;
#pragma unroll
        for (int j = 0; j < E; ++j) key[j] ^= flip;
#pragma unroll 1
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const bool lower = (lane & stride) == 0;
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const uint32_t b = __shfl_xor_sync(kFull, key[j], stride);
                key[j] = lower ? min(key[j], b) : max(key[j], b);
            }
        }
        merge_in_lane<E>(key);
#pragma unroll
        for (int j = 0; j < E; ++j) key[j] ^= flip;
    }
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int p = lane * E + j;
        sorted[wib][p + (p >> 5)] = key[j];
        if (p < n) place[wib][key[j] & 0xffffu] = p;
    }
    __syncwarp();
    for (int t = lane; t < n; t += 32) {
        const uint32_t k = sorted[wib][t + (t >> 5)];
        perm[base + t] = (int32_t)(k & 0xffffu);
        osorted[base + t] = ISJL_MAX_LEN - (int32_t)(k >> 16);
        posof[base + t] = place[wib][t];
    }
}

// n <= 4096: keys (65535 - o) << 16 | index, bitonic sort in shared memory
__global__ void __launch_bounds__(kSortThreads)
sort_small_kernel(const int32_t *__restrict__ o, const InstStats *__restrict__ inst, int32_t *__restrict__ perm,
                  int32_t *__restrict__ osorted, int32_t *__restrict__ posof, int32_t n_slots, int32_t npow2) {
    extern __shared__ uint32_t key[];
    const int64_t base = (int64_t)blockIdx.x * n_slots;
    const int32_t n = inst[blockIdx.x].n;
    for (int t = threadIdx.x; t < npow2; t += kSortThreads)
        key[t] = t < n ? (len_key(o[base + t]) << 16) | (uint32_t)t : 0xffffffffu;
    for (int size = 2; size <= npow2; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < npow2; t += kSortThreads) {
                const int u = t ^ stride;
                if (u > t) {
                    const bool up = (t & size) == 0;
                    const uint32_t x = key[t], y = key[u];
                    if ((x > y) == up) { key[t] = y; key[u] = x; }
                }
            }
        }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < n; p += kSortThreads) {
        const uint32_t k = key[p];
        const int idx = (int)(k & 0xffffu);
        perm[base + p] = idx;
        osorted[base + p] = ISJL_MAX_LEN - (int32_t)(k >> 16);
        posof[base + idx] = p;
    }
}

// large n: stable LSD radix sort on the 16-bit key, two 8-bit passes, one block
// per instance.  Both passes' digit counts come from one read of the lengths.  A
// pass goes over the elements in tiles: each warp owns 32 * kRadixItems consecutive
// ones and ranks them in order with its own counts (lanes of one digit found by
// votes), the counts are summed over the warps per digit, and every element is
// written to its place.  All reads but the last gather are coalesced (1,024 x
// 100,000 requests: 13.7 -> 4.4 ms against one contiguous chunk per thread, whose
// lanes read 32 different lines each time).
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixItems = 4;

// the lanes with this lane's 8-bit digit, among those with `there`: eight votes (a
// match instruction takes a step per distinct digit, up to 32)
__device__ __forceinline__ unsigned same_digit(uint32_t d, bool there) {
    unsigned same = __ballot_sync(kFull, there);
#pragma unroll
    for (int bit = 0; bit < 8; ++bit) {
        const bool one = d >> bit & 1u;
        const unsigned b = __ballot_sync(kFull, one);
        same &= one ? b : ~b;
    }
    return same;
}

__global__ void __launch_bounds__(kRadixThreads)
sort_radix_kernel(const int32_t *__restrict__ o, const InstStats *__restrict__ inst, int32_t *__restrict__ perm,
                  int32_t *__restrict__ osorted, int32_t *__restrict__ posof, int32_t *__restrict__ tmp,
                  int32_t n_slots) {
    __shared__ uint32_t cnt[kRadixWarps][256];    // a tile's elements per warp and digit, then their first place
    __shared__ uint32_t first[2][256];            // per pass and digit: elements before it, then the next place
    const int64_t base = (int64_t)blockIdx.x * n_slots;
    const int32_t n = inst[blockIdx.x].n;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const uint32_t lt = (1u << lane) - 1u;
    for (int d = tid; d < 512; d += kRadixThreads) first[d >> 8][d & 255] = 0u;
    __syncthreads();
    for (int b = 0; b < n; b += kRadixThreads) {
        const int i = b + tid;
        const uint32_t k = i < n ? len_key(o[base + i]) : 0u;
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {    // one addition per warp and distinct digit
            const uint32_t d = (k >> (8 * pass)) & 255u;
            const unsigned same = same_digit(d, i < n);
            if (i < n && (same & lt) == 0u) atomicAdd(&first[pass][d], (uint32_t)__popc(same));
        }
    }
    __syncthreads();
    if (wid < 2) {                                // exclusive scan of 256 counts by one warp per pass
        uint32_t v[8], sum = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { v[j] = first[wid][lane * 8 + j]; sum += v[j]; }
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += t;
        }
        uint32_t run = incl - sum;
#pragma unroll
        for (int j = 0; j < 8; ++j) { first[wid][lane * 8 + j] = run; run += v[j]; }
    }
    for (int pass = 0; pass < 2; ++pass) {
        for (int tile = 0; tile < n; tile += kRadixThreads * kRadixItems) {
            for (int j = tid; j < kRadixWarps * 256; j += kRadixThreads) cnt[j >> 8][j & 255] = 0u;
            __syncthreads();                      // (also: the last pass's and tile's places and writes are done)
            // the index of an element, with its second digit above (n < 2^24), and its rank
            uint32_t item[kRadixItems], rank[kRadixItems];
#pragma unroll
            for (int j = 0; j < kRadixItems; ++j) {
                const int i = tile + wid * 32 * kRadixItems + j * 32 + lane;
                uint32_t d = 256u;                // no element
                item[j] = 0u;
                if (i < n) {
                    if (pass == 0) {
                        const uint32_t k = len_key(o[base + i]);
                        item[j] = (uint32_t)i | (k & 0xff00u) << 16;
                        d = k & 255u;
                    } else {
                        item[j] = (uint32_t)tmp[base + i];
                        d = item[j] >> 24;
                    }
                }
                const unsigned same = same_digit(d, d < 256u);
                const uint32_t before = d < 256u ? cnt[wid][d] : 0u;
                __syncwarp();
                if (d < 256u && (same & lt) == 0u) cnt[wid][d] = before + (uint32_t)__popc(same);
                __syncwarp();
                rank[j] = (before + (uint32_t)__popc(same & lt)) | d << 16;   // rank < 32 * kRadixItems
            }
            __syncthreads();
            for (int d = tid; d < 256; d += kRadixThreads) {
                uint32_t run = first[pass][d];
                for (int w = 0; w < kRadixWarps; ++w) {
                    const uint32_t v = cnt[w][d];
                    cnt[w][d] = run;
                    run += v;
                }
                first[pass][d] = run;
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kRadixItems; ++j) {
                const uint32_t d = rank[j] >> 16;
                if (d < 256u) {
                    const int pos = (int)(cnt[wid][d] + (rank[j] & 0xffffu));
                    if (pass == 0) {
                        tmp[base + pos] = (int32_t)item[j];
                    } else {
                        const int idx = (int)(item[j] & 0xffffffu);
                        perm[base + pos] = idx;
                        osorted[base + pos] = ISJL_MAX_LEN - (int32_t)len_key(o[base + idx]);
                        posof[base + idx] = pos;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// A cluster of kSumBlocks blocks per run.  A warp reads whole records, lane f field
// f, so the reads are coalesced and each lane keeps one total; warps, then blocks
// (through the first block's shared memory), are summed in a fixed order.  One block
// per run with a thread per record left most of the GPU idle: 5 runs of 100,000
// records 741 -> 140 us, 5 of 4,096 41 -> 14 us.
constexpr int kSumThreads = 512;
constexpr int kSumWarps = kSumThreads / 32;
constexpr int kSumBlocks = 8;
constexpr int kFields = sizeof(isjl_record) / 8;            // 16 integers, then 8 doubles
constexpr int kFieldMaxExtent = 10, kFieldStatus = 15, kFieldInts = 16;
static_assert(kFields == 24 && offsetof(isjl_record, max_extent) == 8 * kFieldMaxExtent &&
              offsetof(isjl_record, status) == 8 * kFieldStatus && offsetof(isjl_record, c_T) == 8 * kFieldInts,
              "record layout");

struct FieldTotal { int64_t total, ok, first_bad; };        // total: an integer or the bits of a double

// combine two totals of field f, in this order
__device__ __forceinline__ void add_total(FieldTotal &a, const FieldTotal &b, int f) {
    if (f >= kFieldInts) a.total = __double_as_longlong(__dadd_rn(__longlong_as_double(a.total), __longlong_as_double(b.total)));
    else if (f == kFieldMaxExtent) a.total = max(a.total, b.total);
    else a.total += b.total;
    a.ok += b.ok;
    a.first_bad = min(a.first_bad, b.first_bad);
}

__global__ void __cluster_dims__(kSumBlocks, 1, 1) __launch_bounds__(kSumThreads)
summarize_kernel(const isjl_record *__restrict__ rec, int64_t n_inst, RunList runs, int32_t kv_cap,
                 isjl_summary *out) {
    __shared__ FieldTotal part[kSumWarps][32];
    __shared__ FieldTotal blocks[kSumBlocks][32];           // the first block's is used
    // a block's shared memory may be written by another only once it has started:
    // every thread arrives here and waits before the stores; reading the records
    // comes in between, so that the wait is over by then
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    const int run = blockIdx.x / kSumBlocks, block = blockIdx.x % kSumBlocks;
    const int wid = threadIdx.x >> 5, f = threadIdx.x & 31;
    const int64_t *words = reinterpret_cast<const int64_t *>(rec + (int64_t)run * n_inst);
    FieldTotal t{0, 0, INT64_MAX};
    if (f < kFields) {
        constexpr int kAhead = 8;                           // records loaded before the first is added
        constexpr int64_t kStride = kSumBlocks * kSumWarps;
        for (int64_t i0 = block * kSumWarps + wid; i0 < n_inst; i0 += kAhead * kStride) {
            int64_t v[kAhead];
#pragma unroll
            for (int j = 0; j < kAhead; ++j) {
                const int64_t i = i0 + j * kStride;
                v[j] = i < n_inst ? words[i * kFields + f] : (f == kFieldMaxExtent ? INT64_MIN : 0);
            }
#pragma unroll
            for (int j = 0; j < kAhead; ++j) {
                const int64_t i = i0 + j * kStride;
                const bool there = f == kFieldStatus && i < n_inst, good = v[j] == ISJL_OK;
                add_total(t, FieldTotal{v[j], there && good, there && !good ? i : INT64_MAX}, f);
            }
        }
    }
    part[wid][f] = t;
    __syncthreads();
    asm volatile("barrier.cluster.wait;" ::: "memory");     // all blocks of the cluster run
    if (wid == 0) {
        for (int w = 1; w < kSumWarps; ++w) add_total(t, part[w][f], f);
        // the first block's shared memory, through the cluster
        uint32_t local = (uint32_t)__cvta_generic_to_shared(&blocks[block][f]), remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(local));
        asm volatile("st.shared::cluster.b64 [%0], %1;" :: "r"(remote), "l"(t.total) : "memory");
        asm volatile("st.shared::cluster.b64 [%0], %1;" :: "r"(remote + 8), "l"(t.ok) : "memory");
        asm volatile("st.shared::cluster.b64 [%0], %1;" :: "r"(remote + 16), "l"(t.first_bad) : "memory");
    }
    // (not .aligned: lanes of different fields have taken different branches)
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (block != 0 || wid != 0) return;
    t = blocks[0][f];
    for (int b = 1; b < kSumBlocks; ++b) add_total(t, blocks[b][f], f);
    part[0][f] = t;
    __syncwarp();
    if (f == 0) {
        auto i64 = [&](int k) { return part[0][k].total; };
        auto f64 = [&](int k) { return __longlong_as_double(part[0][k].total); };
        const int64_t bad = part[0][kFieldStatus].first_bad;
        isjl_summary S;
        S.policy = runs.policy[run];
        S.delta = runs.delta[run];
        S.kv_cap = kv_cap;
        S.status = bad == INT64_MAX ? ISJL_OK : (int32_t)rec[(int64_t)run * n_inst + bad].status;
        S.n_instances = n_inst;
        S.n_ok = part[0][kFieldStatus].ok;
        S.T_make = i64(0); S.T_busy = i64(1); S.O = i64(2); S.Q = i64(3); S.W = i64(4); S.E = i64(5);
        S.token_adv = i64(6); S.sum_completion = i64(7); S.sum_latency = i64(8); S.sum_extent = i64(9);
        S.max_extent = i64(kFieldMaxExtent); S.violations = i64(11); S.kv_violations = i64(12);
        S.c_T = f64(16); S.tau_Q = f64(17); S.tau_E = f64(18);
        S.cost = f64(19); S.revenue = f64(20); S.profit = f64(21);
        out[run] = S;
    }
}

}  // namespace

cudaError_t launch_derive(const int32_t *arrival, const int32_t *prompt, const int32_t *output,
                          const int32_t *count, const int32_t *slack, int32_t *o, int32_t *otrue,
                          InstStats *inst, int32_t *counter, int32_t *dev_status, int64_t n_inst, int32_t n,
                          cudaStream_t s) {
    if (n <= kWarpSortMax)
        derive_kernel<32><<<(unsigned)((n_inst + kPrepWarps - 1) / kPrepWarps), 32 * kPrepWarps, 0, s>>>(
            arrival, prompt, output, count, slack, o, otrue, inst, counter, dev_status, n_inst, n);
    else if (n <= 16384)
        derive_kernel<256><<<(unsigned)n_inst, 256, 0, s>>>(arrival, prompt, output, count, slack, o, otrue, inst,
                                                            counter, dev_status, n_inst, n);
    else
        derive_kernel<1024><<<(unsigned)n_inst, 1024, 0, s>>>(arrival, prompt, output, count, slack, o, otrue, inst,
                                                              counter, dev_status, n_inst, n);
    return cudaGetLastError();
}

template <int E>
static void launch_sort_warp(const int32_t *o, const InstStats *inst, int32_t *perm, int32_t *osorted, int32_t *posof,
                             int64_t n_inst, int32_t n, cudaStream_t s) {
    sort_warp_kernel<E><<<(unsigned)((n_inst + kPrepWarps - 1) / kPrepWarps), 32 * kPrepWarps, 0, s>>>(
        o, inst, perm, osorted, posof, n_inst, n);
}

cudaError_t launch_sort(const int32_t *o, const InstStats *inst, int32_t *perm, int32_t *osorted, int32_t *posof,
                        int32_t *tmp, int64_t n_inst, int32_t n, cudaStream_t s) {
    if (n <= 32) launch_sort_warp<1>(o, inst, perm, osorted, posof, n_inst, n, s);
    else if (n <= 128) launch_sort_warp<4>(o, inst, perm, osorted, posof, n_inst, n, s);
    else if (n <= 256) launch_sort_warp<8>(o, inst, perm, osorted, posof, n_inst, n, s);
    else if (n <= 512) launch_sort_warp<16>(o, inst, perm, osorted, posof, n_inst, n, s);
    else if (n <= kWarpSortMax) launch_sort_warp<32>(o, inst, perm, osorted, posof, n_inst, n, s);
    else if (n <= kSortSmallMax) {
        int npow2 = 1;
        while (npow2 < n) npow2 <<= 1;
        sort_small_kernel<<<(unsigned)n_inst, kSortThreads, npow2 * sizeof(uint32_t), s>>>(o, inst, perm, osorted,
                                                                                         posof, n, npow2);
    } else {
        sort_radix_kernel<<<(unsigned)n_inst, kRadixThreads, 0, s>>>(o, inst, perm, osorted, posof, tmp, n);
    }
    return cudaGetLastError();
}

cudaError_t launch_summarize(const isjl_record *records, int64_t n_inst, int32_t n_runs, const RunList &runs,
                             int32_t kv_cap, isjl_summary *out, cudaStream_t s) {
    summarize_kernel<<<n_runs * kSumBlocks, kSumThreads, 0, s>>>(records, n_inst, runs, kv_cap, out);
    return cudaGetLastError();
}

}  // namespace isjl
