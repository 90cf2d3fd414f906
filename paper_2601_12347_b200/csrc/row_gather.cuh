// Summing rows over in-lists: the part that the gathers share.
//
// A warp works on a run of in-list entries, which may be the lists of up to 32 sinks laid end to end or a piece of one
// long list.  It takes the run 128 entries at a time (four ids per lane, those of the next 128 on their way meanwhile),
// puts what is to be summed into a queue of its own in shared memory, and then walks the queue: the lanes form as many
// groups as rows fit side by side (a row takes a lane per 16 bytes), every group goes through a contiguous part of the
// queue with eight rows always on their way, adds up in registers and delivers the sum by one reduction per piece when the
// sink changes.
//
// What bounds it: the rate at which L2 serves scattered rows, 15.4 ps per row of 48 floats (12.4 TB/s), 25 at 104 and 63
// at 256 floats (16.3 TB/s), measured on lists alone.  A warp per sink that asks for ids, then for rows, then for the
// next sink's ids, and takes two rows of 12 pieces with 32 lanes only, spends 24 ps per row of 48 floats: most lists are
// shorter than the rows that should be on their way, and each is a chain of four trips to memory.
#pragma once

#include "device_utils.cuh"
#include "ripple_internal.cuh"

namespace rp {

constexpr int RG_WINDOW = 128;    // entries asked for at a time: four per lane
constexpr int RG_DRAIN = 64;      // a filtered queue is walked when it holds this many
constexpr int RG_CAP = RG_DRAIN + RG_WINDOW;
constexpr int RG_NEW = (int)0x80000000;   // on a queued row: its sink is not that of the entry before

// How the lanes share a row of `ld` floats: G groups, lane = (group, piece).
struct RowLanes {
    int G, sub, ql, nq;
    __device__ __forceinline__ explicit RowLanes(int ld) : nq(ld >> 2) {
        const int w = min(nq, 32), lane = lane_id();
        G = 32 / w;
        sub = lane / w;
        ql = lane - sub * w;
    }
};

// rows on their way per group
template <int NV>
__host__ __device__ constexpr int rg_unroll() { return NV == 1 ? 8 : NV == 2 ? 4 : NV == 4 ? 2 : 1; }

template <int NV>
__device__ __forceinline__ void rg_zero(float4 (&acc)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <int NV>
__device__ __forceinline__ void rg_deliver(const RowLanes& g, const float4 (&acc)[NV], float* dst) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int q = g.ql + 32 * k;
        if (q < g.nq) red_add_v4(dst + 4 * q, acc[k]);
    }
}

// A warp's queue in shared memory.
template <bool WGT>
struct RowQueue {
    int* row;      // row of M to add, with RG_NEW where the sink changes
    int* sink;
    float* w;      // its factor
    __device__ __forceinline__ void put(int at, int r, int v, float f) const {
        row[at] = r;
        sink[at] = v;
        if (WGT) w[at] = f;
    }
    __host__ __device__ static constexpr int bytes(int cap) { return cap * (WGT ? 12 : 8); }
    __device__ __forceinline__ RowQueue(void* base, int cap) : row((int*)base), sink((int*)base + cap), w((float*)base + 2 * cap) {}
};

// Adds the n > 0 queued rows up.  ONE: all for the same sink, into acc, which the caller delivers; else each sink's sum
// is delivered to its row of dst.  The steps that all groups have in full go without looking at bounds, their rows read
// four to an instruction: the walk is as much bound by the instructions issued as by L2 (six and a 16-byte load per row
// and lane, two more where sinks change; 16 and 30 with a check of its own for every row took 17 and 29 ps per row of 48 floats).
template <int NV, bool WGT, bool ONE>
__device__ __forceinline__ void rg_walk(const RowLanes& g, const RowQueue<WGT>& q, int n, const float* __restrict__ M, int ld,
                                        float* dst, float4 (&acc)[NV]) {
    constexpr int UNR = rg_unroll<NV>(), VEC = UNR < 4 ? UNR : 4;
    const int run = ((n + g.G - 1) / g.G + 3) & ~3;              // (so that every group's rows are aligned)
    const bool idle = g.sub >= g.G;                              // lanes without a group follow the first one
    const int j0 = idle ? 0 : min(n, g.sub * run), end = idle ? 0 : min(n, j0 + run);
    const int full = max(0, n - (g.G - 1) * run) / UNR * UNR;    // what every group has in whole steps
    const float4* mine[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) mine[k] = reinterpret_cast<const float4*>(M) + (g.ql + 32 * k < g.nq ? g.ql + 32 * k : 0);
    const int nq = ld >> 2;
    float4 x[UNR][NV];
    auto fetch = [&](int t, int r) {
#pragma unroll
        for (int k = 0; k < NV; ++k) x[t][k] = __ldg(mine[k] + (size_t)(ONE ? r : r & ~RG_NEW) * nq);
    };
    auto rows = [&](int (&r)[UNR], int j) {
#pragma unroll
        for (int t = 0; t < UNR; t += VEC) {
            if (VEC == 4) *reinterpret_cast<int4*>(&r[t]) = *reinterpret_cast<const int4*>(q.row + j + t);
            else
#pragma unroll
                for (int u = 0; u < VEC; ++u) r[t + u] = q.row[j + t + u];
        }
    };
    auto use = [&](int t, float w) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            if (WGT) {
                acc[k].x += w * x[t][k].x; acc[k].y += w * x[t][k].y; acc[k].z += w * x[t][k].z; acc[k].w += w * x[t][k].w;
            } else {
                acc[k].x += x[t][k].x; acc[k].y += x[t][k].y; acc[k].z += x[t][k].z; acc[k].w += x[t][k].w;
            }
        }
    };
    auto done = [&](int j) {   // the sink of the entry before j has all of its rows
        if (!idle) rg_deliver<NV>(g, acc, dst + (size_t)q.sink[j - 1] * ld);
        rg_zero<NV>(acc);
    };
    int b = 0;
    if (full) {
        int r[UNR];
        rows(r, j0);
        if (!ONE) r[0] &= ~RG_NEW;
#pragma unroll
        for (int t = 0; t < UNR; ++t) fetch(t, r[t]);
        for (; b + UNR < full; b += UNR) {
            int rn[UNR];
            rows(rn, j0 + b + UNR);
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                if (!ONE && r[t] < 0) done(j0 + b + t);
                use(t, WGT ? q.w[j0 + b + t] : 1.0f);
                fetch(t, rn[t]);   // (the next row is asked for as soon as this one is used)
            }
            if (!ONE)
#pragma unroll
                for (int t = 0; t < UNR; ++t) r[t] = rn[t];
        }
#pragma unroll
        for (int t = 0; t < UNR; ++t) {
            if (!ONE && r[t] < 0) done(j0 + b + t);
            use(t, WGT ? q.w[j0 + b + t] : 1.0f);
        }
        b += UNR;
    }
    for (; b < run; b += UNR) {
        int r[UNR];
#pragma unroll
        for (int t = 0; t < UNR; ++t) {
            r[t] = q.row[min(j0 + b + t, n - 1)];
            fetch(t, r[t] & ~RG_NEW);
        }
#pragma unroll
        for (int t = 0; t < UNR; ++t) {
            const int j = j0 + b + t;
            if (j >= end) break;
            if (!ONE && r[t] < 0 && j > j0) done(j);
            use(t, WGT ? q.w[j] : 1.0f);
        }
    }
    if (!ONE) {
        if (end > j0) rg_deliver<NV>(g, acc, dst + (size_t)q.sink[end - 1] * ld);
        rg_zero<NV>(acc);
    }
}

// All groups have worked for the same sink: their sums meet and are delivered.
template <int NV>
__device__ __forceinline__ void rg_finish_one(const RowLanes& g, float* dst, float4 (&acc)[NV]) {
    if (NV == 1) {
        const float4 own = acc[0];
        for (int s = 1; s < g.G; ++s) {
            const int from = (g.ql + s * g.nq) & 31;
            acc[0].x += __shfl_sync(FULL, own.x, from); acc[0].y += __shfl_sync(FULL, own.y, from);
            acc[0].z += __shfl_sync(FULL, own.z, from); acc[0].w += __shfl_sync(FULL, own.w, from);
        }
    }
    if (g.sub == 0) rg_deliver<NV>(g, acc, dst);
    rg_zero<NV>(acc);   // (the lanes without a group have added up what was not theirs)
}

// The lists of up to 32 sinks, one per lane, laid end to end: entry f lies at `at` and belongs to sink `v`.
struct TileRun {
    static constexpr bool ONE = false;
    int ex, v, total;        // entries before this lane's list; its sink
    int64_t delta;           // where its entry f lies: delta + f
    __device__ __forceinline__ TileRun(int v_, int64_t start, int entries) : v(v_) {
        const int inc = warp_inclusive_scan(entries);
        ex = inc - entries;
        total = __shfl_sync(FULL, inc, 31);
        delta = start - ex;
    }
    __device__ __forceinline__ void locate(int f, int64_t& at, int& sink) const {
        int s = 0;           // the last list that begins at or before f (an empty one lies before the list it shares its begin with)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int e = __shfl_sync(FULL, ex, s + o);
            if (e <= f) s += o;
        }
        at = __shfl_sync(FULL, delta, s) + f;
        sink = __shfl_sync(FULL, v, s);
    }
};

// The lists of `cnt` sinks from position i0 of `list` (null: ids are positions), but for those of more than long_list entries;
// with `only`, those whose bit is set there.
struct TileLists {
    int v, deg;
    int64_t start;
    __device__ __forceinline__ TileLists(const Side& in, const int32_t* list, long long i0, int cnt, const uint32_t* only = nullptr)
        : v(0), deg(0), start(0) {
        if (lane_id() < cnt) {
            v = list ? list[i0 + lane_id()] : (int)i0 + lane_id();
            if (only && !(only[v >> 5] >> (v & 31) & 1u)) return;
            deg = in.deg[v];
            start = in.start[v];
        }
    }
    __device__ __forceinline__ TileRun run(int long_list) const { return TileRun(v, start, deg > long_list ? 0 : deg); }
};

// Tiles by ticket on large graphs (the next ticket is asked for before the tile is worked on); evenly where there are few.
struct TileDeal {
    int *ticket, at, stride, asked;
    __device__ __forceinline__ explicit TileDeal(int* t) : ticket(t) {
        at = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        stride = (gridDim.x * blockDim.x) >> 5;
        asked = 0;
        ask();
    }
    __device__ __forceinline__ void ask() { if (ticket && lane_id() == 0) asked = atomicAdd(ticket, 1); }
    __device__ __forceinline__ int first() { return take(at); }
    __device__ __forceinline__ int next() { at += stride; return take(at); }
    __device__ __forceinline__ int take(int even) {
        if (!ticket) return even;
        const int t = __shfl_sync(FULL, asked, 0);
        ask();
        return t;
    }
};

// Work items for the kernel that follows: pieces of the long lists of a tile, (sink, piece), and what the tile's run has
// beyond its first piece, (-1 - tile, piece).  One addition to the counter per tile: counters that every warp adds to take a
// nanosecond or two per addition (one per list: 0.2 ms on the graph of 233 K vertices, 0.5 on that of 2.4 M).
__device__ __forceinline__ void rg_queue_rest(const TileLists& t, int tile, int total, int long_list, int item, int piece, int2* items, int* n_items) {
    const int lane = lane_id();
    const int rest = total > piece ? (total + piece - 1) / piece - 1 : 0;
    const int mine = t.deg > long_list ? (t.deg + item - 1) / item : 0;
    const int inc = warp_inclusive_scan(mine), lists = __shfl_sync(FULL, inc, 31);
    if (rest + lists == 0) return;
    int first = 0;
    if (lane == 0) first = atomicAdd(n_items, rest + lists);
    first = __shfl_sync(FULL, first, 0);
    for (int k = lane; k < rest; k += 32) items[first + k] = make_int2(-1 - tile, k + 1);
    first += rest;
    for (unsigned many = __ballot_sync(FULL, mine > 0); many; many &= many - 1) {
        const int b = __ffs(many) - 1, row = __shfl_sync(FULL, t.v, b), n = __shfl_sync(FULL, mine, b), at = first + __shfl_sync(FULL, inc - mine, b);
        for (int k = lane; k < n; k += 32) items[at + k] = make_int2(row, k);
    }
}

// A piece of one list.
struct ListRun {
    static constexpr bool ONE = true;
    int v, total;
    int64_t first;
    __device__ __forceinline__ ListRun(int v_, int64_t first_, int n) : v(v_), total(n), first(first_) {}
    __device__ __forceinline__ void locate(int f, int64_t& at, int& sink) const { at = first + f; sink = v; }
};

// One window of ids of a run, four per lane (beyond the end: id -1).
template <bool STORED_W, typename RUN>
struct IdWindow {
    int u[4], v[RUN::ONE ? 1 : 4];
    float w[STORED_W ? 4 : 1];
    __device__ __forceinline__ int sink(int k) const { return v[RUN::ONE ? 0 : k]; }
    __device__ __forceinline__ float weight(int k) const { return STORED_W ? w[STORED_W ? k : 0] : 1.0f; }
    __device__ __forceinline__ void request(const RUN& run, const Side& in, int f0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int f = f0 + 32 * k + lane_id();
            int64_t at;
            run.locate(f, at, v[RUN::ONE ? 0 : k]);
            u[k] = -1;
            if (f < run.total) u[k] = in.col[at];
            if (STORED_W) w[STORED_W ? k : 0] = f < run.total && in.w ? in.w[at] : 1.0f;
        }
    }
};

// RG_NEW for the lanes of `m` whose sink is not that of the lane of `m` before them; `last` is the sink queued before them
// and becomes that of the last of them.
__device__ __forceinline__ int rg_new_sink(unsigned m, int v, int& last) {
    const unsigned before = m & ((1u << lane_id()) - 1u);
    const int prev = __shfl_sync(FULL, v, before ? 31 - __clz(before) : 0);
    const int flag = v != (before ? prev : last) ? RG_NEW : 0;
    if (m) last = __shfl_sync(FULL, v, 31 - __clz(m));
    return flag;
}

}  // namespace rp
