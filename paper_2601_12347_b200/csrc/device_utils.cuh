// Small device-side building blocks: warp/block scans, bit tricks, vector reductions to global.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sweep_rule.h"

namespace rp {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// First statement of every kernel.  The kernels of a batch are launched with programmatic stream
// serialisation: a kernel may be scheduled while its predecessor is still running, so that launch
// latency overlaps execution (a batch is a chain of some fifty short kernels).  The wait returns
// once every prerequisite grid has completed and its memory operations are visible, so nothing a
// kernel reads can be stale; the trigger then lets the successor be scheduled in turn.  Without a
// programmatic dependency both instructions are no-ops.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// inclusive warp scan
template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(FULL, x, o);
        if (lane_id() >= o) x += y;
    }
    return x;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

// Exclusive block scan for blocks of up to 1024 threads; `total` receives the block sum.
// scratch: 33 entries of T in shared memory.
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T x, T* scratch, T& total) {
    const int lane = lane_id(), warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
    T inc = warp_inclusive_scan(x);
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T s = lane < nwarp ? scratch[lane] : T(0);
        T si = warp_inclusive_scan(s);
        scratch[lane] = si - s;
        if (lane == 31) scratch[32] = si;
    }
    __syncthreads();
    T base = scratch[warp];
    total = scratch[32];
    __syncthreads();
    return base + inc - x;
}

// 16-byte vector reduction into global memory (sm_90+): four fp32 adds in one request.
__device__ __forceinline__ void red_add_v4(float* addr, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w)
                 : "memory");
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// largest i in [0, n) with a[i] <= x, for ascending a with a[0] <= x
__device__ __forceinline__ int upper_row(const int64_t* a, int n, int64_t x) {
    int lo = 0, hi = n;  // invariant: a[lo] <= x, (hi == n or a[hi] > x)
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (a[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// How the warps of a kernel share `total` equal units of work: chunk by chunk, handed out by ticket.  Registers allow
// these kernels four to six resident blocks per SM, so with a fixed split over a grid of eight per SM the last blocks
// began when the first ones ended, and under overlapped launches the residency is uneven besides (48-float push of 19 M
// messages on the dense graph: 0.91 ms with the fixed split, 1.15 ms replayed from a captured chain, 0.82 ms by ticket;
// 44-float push of 53 M messages on the graph of 233 K vertices: 1.97 -> 0.93 ms).  Where there is no second round -- few
// units -- the warps keep fixed chunks of the small size and nobody touches the counter.
// The ticket of the next chunk is asked for before the present one is worked on.
//
// A walk that adds into rows by vertex id can be told how many rows there are and how wide they are.  Where the rows it
// is likely to reach (half of them) outgrow L2 and each receives several messages, the walk is made twice, over the lower
// and then over the upper half of the ids, in the order of the tickets: more of the rows are then still in L2 when their
// next message arrives.  (2.4 M rows of 48 floats, 20 M messages: whole chain 1.56 -> 1.49 ms; of 104 floats: 4.12 ->
// 3.74; three and four passes are no better, eight are slower than one: every pass reads and sorts out all ids again.)
struct TicketWalk {
    long long total, at;
    int chunk, next, *ticket;
    int passes, per_pass, first_id;
    unsigned span;
    __device__ __forceinline__ TicketWalk(int* t, long long n, int small, int large, int rows = 0, int row_floats = 0)
        : total(n), ticket(t), passes(1), per_pass(0), first_id(0), span(0x80000000u) {
        const long long warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
        chunk = small;
        if (n <= nwarps * small) {   // (as many warps as there are units for, an eighth of the small chunk at least)
            ticket = nullptr;
            chunk = max(max(small >> 3, 1), (int)(((unsigned)n + (unsigned)nwarps - 1u) / (unsigned)nwarps));
            at = warp * chunk;
            return;
        }
        if (n > nwarps * large * 2) chunk = large;
        if (n >= 2ll * rows && (long long)rows * row_floats * 2 >= WALK_TWICE) {
            passes = 2;
            if (n > nwarps * chunk * 8) chunk *= 4;   // (26 M messages of 48 floats: 1.12 -> 1.00 ms in chunks of 1024; in one pass, 50 M of 44 floats, 256 is the better by a hundredth)
            per_pass = (int)((n + chunk - 1) / chunk);
            span = (unsigned)(rows + 1) / 2u;
        }
        take();
        advance();
    }
    __device__ __forceinline__ bool has() const { return at < total; }
    __device__ __forceinline__ void take() {
        if (ticket && lane_id() == 0) next = atomicAdd(ticket, 1);
    }
    __device__ __forceinline__ void advance() {
        if (!ticket) { at = total; return; }
        int t = __shfl_sync(FULL, next, 0);
        if (passes > 1) {
            const int pass = t / per_pass;
            t = pass < passes ? t - pass * per_pass : per_pass;
            first_id = pass * (int)span;
        }
        at = (long long)t * chunk;
    }
};

// The entries [base, base + cnt_total) of a list, delivered 32 at a time as deliver(id, weight, count), an entry per lane
// below count.  With `filter` only ids of [first_id, first_id + span): they are collected in `queue` (the warp's own
// WALK_QUEUE entries of shared memory) until there are 32 of them.
constexpr int WALK_QUEUE = 160;

template <bool WEIGHTED, typename F>
__device__ __forceinline__ void walk_entries(const int32_t* __restrict__ col, const float* __restrict__ w, int64_t base, int cnt_total,
                                             const TicketWalk& walk, int2* queue, F deliver) {
    const int lane = lane_id();
    if (walk.passes == 1) {
        for (int j0 = 0; j0 < cnt_total; j0 += 32) {
            const bool have = j0 + lane < cnt_total;
            deliver(have ? col[base + j0 + lane] : 0, (WEIGHTED && w && have) ? w[base + j0 + lane] : 1.0f, min(32, cnt_total - j0));
        }
        return;
    }
    const unsigned lt = (1u << lane) - 1u;
    int held = 0;
    for (int j0 = 0; j0 < cnt_total || held > 0; j0 += 128) {
        if (j0 < cnt_total) {
            int v[4];
            float a[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = min(j0 + 32 * k + lane, cnt_total - 1);
                v[k] = col[base + j];
                a[k] = (WEIGHTED && w) ? w[base + j] : 1.0f;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool in = j0 + 32 * k + lane < cnt_total && (unsigned)(v[k] - walk.first_id) < walk.span;
                const unsigned m = __ballot_sync(FULL, in);
                if (in) queue[held + __popc(m & lt)] = make_int2(v[k], __float_as_int(a[k]));
                held += __popc(m);
            }
        }
        __syncwarp();
        // full groups, and at the end of the list the rest
        int done = 0;
        while (held - done >= 32 || (j0 + 128 >= cnt_total && done < held)) {
            const int cnt = min(32, held - done);
            const int2 x = queue[done + min(lane, cnt - 1)];
            deliver(x.x, __int_as_float(x.y), cnt);
            done += cnt;
        }
        const int rest = held - done;
        const int2 x = queue[done + min(lane, max(rest - 1, 0))];
        __syncwarp();
        if (lane < rest) queue[lane] = x;
        __syncwarp();
        held = rest;
    }
}

}  // namespace rp
