// Delta-message scatter (Send + Aggregate of Sec. 3.3.1) and the bootstrap aggregation.
//
// S^l is the persistent, un-normalised inbox: S^l_v = sum_{u in In(v)} c_u m_u with m_u = h^{l-1}_u,
// or, for a layer whose output is narrower than its input, m_u = W_n^T h^{l-1}_u (aggregation is
// linear, so the neighbour transform can be applied to the few sender rows before the scatter
// instead of to the many sink rows after it; messages and inbox rows then have the output width).
// For hop l
//   S_v += sum over surviving and added edges (u, v) with u in C_{l-1} of D_u
//        + sum over added edges   (u, v) of M_u       (M_u = c_old(u) m_old(u): what the walk
//        - sum over deleted edges (u, v) of M_u        above did not, or wrongly did, deliver)
// with D_u = c_new m_new - c_old m_old the sender's delta row (Sec. 3.3.3: changed vertex; added
// edge = old contribution 0; deleted edge = new contribution 0; weighted form alpha h - alpha h-).
//
// push: the out-edges of the senders are cut into equal chunks; a warp keeps the sender's delta
//       row in registers and issues one 16-byte vector reduction per lane and edge (narrow rows:
//       several edges per warp instruction).
// sweep: the in-lists of all vertices, or of the marked ones, are read, sources that are senders kept (a filter, then the
//       position map), their delta rows summed in registers, and a sink's accumulator touched once.
#include "row_gather.cuh"

#include <algorithm>

namespace rp {

__device__ __forceinline__ float coef_from_degree(int deg) {
    return deg > 0 ? 1.0f / sqrtf((float)deg) : 0.0f;
}

__device__ __forceinline__ void add4(float4& a, const float4& x, float c) {
    a.x += c * x.x; a.y += c * x.y; a.z += c * x.z; a.w += c * x.w;
}

// ---------------------------------------------------------------------------------------------
// bootstrap: S_v for every vertex by gathering over in-edges (Eq. 1)
// LPR lanes hold one row (NV float4 slots each); a warp works on 32 / LPR in-neighbours at a time.
// ---------------------------------------------------------------------------------------------
// acc += sum over in-list entries [j_begin, j_end) of row v of c_u * M_u; LPR lanes hold one row
// (NV float4 slots each), a warp works on 32 / LPR neighbours per step, several steps in flight.
template <int NV, int LPR>
__device__ __forceinline__ void spmm_accumulate(float4 (&acc)[NV], const Side& in, int v, int j_begin, int j_end,
                                                const int32_t* __restrict__ deg_out, int src_norm,
                                                const float* __restrict__ M, int ld) {
    const int lane = lane_id(), nq = ld >> 2;
    constexpr int EPI = 32 / LPR;
    const int sub = lane / LPR, ql = lane % LPR;
    const int64_t base = in.start[v];
    for (int j0 = j_begin; j0 < j_end; j0 += 32) {
        int mine = j0 + lane < j_end ? in.col[base + j0 + lane] : 0;
        // stored edge weights (weighted sum with per-edge weights): the entry's weight is its coefficient
        float mine_w = (in.w && j0 + lane < j_end) ? in.w[base + j0 + lane] : 1.0f;
        int cnt = min(32, j_end - j0);
        constexpr int UNR = NV == 1 ? 8 : 4;   // rows in flight per lane group (48 floats, rebuilt hop of 123 M entries: 8 is 0.3 ms faster than 4)
        for (int j = 0; j < cnt; j += UNR * EPI) {
            int u[UNR];
            float cu[UNR];
            float4 x[UNR][NV];
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const int jj = j + t * EPI + sub;
                u[t] = __shfl_sync(FULL, mine, jj & 31);
                const float wj = __shfl_sync(FULL, mine_w, jj & 31);
                cu[t] = 0.f;
                if (jj < cnt) cu[t] = src_norm ? coef_from_degree(deg_out[u[t]]) : wj;
                else u[t] = -1;
            }
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const float4* row = reinterpret_cast<const float4*>(M + (size_t)max(u[t], 0) * ld);
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const int q = ql + LPR * k;
                    x[t][k] = (u[t] >= 0 && q < nq) ? __ldg(row + q) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int t = 0; t < UNR; ++t)
#pragma unroll
                for (int k = 0; k < NV; ++k) add4(acc[k], x[t][k], cu[t]);
        }
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) {
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            acc[k].x += __shfl_xor_sync(FULL, acc[k].x, o);
            acc[k].y += __shfl_xor_sync(FULL, acc[k].y, o);
            acc[k].z += __shfl_xor_sync(FULL, acc[k].z, o);
            acc[k].w += __shfl_xor_sync(FULL, acc[k].w, o);
        }
    }
}

// S_v = sum over In(v) of c_u M_u for a list of sinks (or for every vertex): the bootstrap's aggregation and the
// rebuilding form of a hop.  A warp takes the lists of 32 sinks at a time, laid end to end (see row_gather.cuh), zeroes
// their rows and adds to them; a list too long for that is queued in pieces for the kernel below, a warp per piece.
// All 124 M in-edges of the graph of 2.4 M vertices, 48 floats per row: 2.99 -> 2.24 to 2.46 ms (a warp per sink and a trip to
// memory for every step of a list -> this); 100 floats: 4.9 -> 4.3 to 4.75 ms.
struct RowSums {
    Side in;
    const int32_t* list;        // sinks (null: every vertex)
    const int* n_dev;           // their number on the device (null: n_host)
    int n_host;
    const int32_t* deg_out;
    int src_norm;
    const float* M;
    int ld;
    float* S;
    int2* items;                // (sink, piece) of the long lists
    int* n_items;
    int* ticket;
    int take;                   // sinks per tile
    int long_list, item, piece; // lists of more than long_list entries go in pieces of `item`, tiles of more than `piece` in such
    float* budget;              // a row gathered anew has spent nothing
};

template <int NV, bool WGT, typename RUN>
__device__ __forceinline__ void sum_rows(const RowLanes& g, const RUN& run, const RowSums& a, const RowQueue<WGT>& q, float4 (&acc)[NV], int begin = 0) {
    const int lane = lane_id();
    IdWindow<WGT, RUN> nx;
    nx.request(run, a.in, begin);
    for (int f0 = begin; f0 < run.total; f0 += RG_WINDOW) {
        const int n = min(RG_WINDOW, run.total - f0);
        int last = -1;
        __syncwarp();   // the window before has been walked
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int u = nx.u[k], v = nx.sink(k), at = 32 * k + lane;
            const int flag = RUN::ONE ? 0 : rg_new_sink(__ballot_sync(FULL, u >= 0), v, last);
            if (u >= 0) q.put(at, u | flag, v, WGT && a.src_norm ? coef_from_degree(a.deg_out[u]) : nx.weight(k));
        }
        __syncwarp();
        nx.request(run, a.in, f0 + RG_WINDOW);
        rg_walk<NV, WGT, RUN::ONE>(g, q, n, a.M, a.ld, a.S, acc);
    }
}

constexpr int SUM_T = 256;

template <int NV, bool WGT>
__global__ void __launch_bounds__(SUM_T, NV == 1 ? 3 : 1)
k_sum_rows(const Ctl* ctl, int l, int only_if_rebuilding, const __grid_constant__ RowSums a) {
    pdl_enter();
    if (only_if_rebuilding && (ctl->abort || !ctl->regather[l])) return;
    __shared__ __align__(16) char s_q[SUM_T / 32][RowQueue<WGT>::bytes(RG_WINDOW)];
    const int n = a.n_dev ? *a.n_dev : a.n_host, lane = lane_id();
    const RowQueue<WGT> q(s_q[threadIdx.x >> 5], RG_WINDOW);
    const RowLanes g(a.ld);
    float4 acc[NV];
    rg_zero<NV>(acc);
    TileDeal deal(a.take == 32 ? a.ticket : nullptr);
    for (int tile = deal.first();; tile = deal.next()) {
        const long long i0 = (long long)a.take * tile;
        if (i0 >= n) break;
        const int cnt = (int)min((long long)a.take, n - i0);
        const TileLists t(a.in, a.list, i0, cnt);
        if (a.budget && lane < cnt) a.budget[t.v] = 0.f;
        TileRun run = t.run(a.long_list);
        for (int r0 = 0; r0 < cnt; r0 += g.G) {   // the rows start from zero
            const int r = r0 + g.sub, row = __shfl_sync(FULL, t.v, r & 31);
            if (g.sub < g.G && r < cnt) {
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const int p = g.ql + 32 * k;
                    if (p < g.nq) *reinterpret_cast<float4*>(a.S + (size_t)row * a.ld + 4 * p) = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
        rg_queue_rest(t, tile, run.total, a.long_list, a.item, a.piece, a.items, a.n_items);
        run.total = min(run.total, a.piece);
        sum_rows<NV, WGT>(g, run, a, q, acc);
    }
}

template <int NV, bool WGT>
__global__ void __launch_bounds__(SUM_T, NV == 1 ? 3 : 1)
k_sum_rows_long(const Ctl* ctl, int l, int only_if_rebuilding, const __grid_constant__ RowSums a, int* ticket) {
    pdl_enter();
    if (only_if_rebuilding && (ctl->abort || !ctl->regather[l])) return;
    __shared__ __align__(16) char s_q[SUM_T / 32][RowQueue<WGT>::bytes(RG_WINDOW)];
    const int n = *a.n_items;
    if (n == 0) return;
    const RowQueue<WGT> q(s_q[threadIdx.x >> 5], RG_WINDOW);
    const RowLanes g(a.ld);
    float4 acc[NV];
    rg_zero<NV>(acc);
    TicketWalk walk(ticket, n, 1, 4);
    for (; walk.has(); walk.advance()) {
        const int from = (int)walk.at, to = min(n, from + walk.chunk);
        walk.take();
        for (int it = from; it < to; ++it) {
            const int2 w = a.items[it];
            if (w.x < 0) {
                const int tile = -1 - w.x;
                const long long i0 = (long long)a.take * tile;
                TileRun run = TileLists(a.in, a.list, i0, (int)min((long long)a.take, (a.n_dev ? *a.n_dev : a.n_host) - i0)).run(a.long_list);
                run.total = min(run.total, (w.y + 1) * a.piece);
                sum_rows<NV, WGT>(g, run, a, q, acc, w.y * a.piece);
                continue;
            }
            const int deg = a.in.deg[w.x];
            const ListRun run(w.x, a.in.start[w.x] + (int64_t)w.y * a.item, min(a.item, deg - w.y * a.item));
            sum_rows<NV, WGT>(g, run, a, q, acc);
            rg_finish_one<NV>(g, a.S + (size_t)w.x * a.ld, acc);
        }
    }
}

static_assert(RP_ANEW_CHUNK >= RP_ITEM_MIN, "the item buffer is sized by it");

// How the lists are cut: pieces of which every warp of the device gets a few, so that none is still at one when the others
// have run out.
template <typename A>
static void cut_lists(const Ctx* c, A& a) {
    const long long per_warp = (long long)c->stats.num_edges / (c->n_sm * 64);
    a.item = RP_ITEM_MIN;
    while (a.item < 1024 && 2 * a.item <= per_warp) a.item *= 2;
    a.piece = std::min(a.item, 512);
    a.long_list = std::min(a.item, 256);
    a.take = c->N >= 32 * 64 * c->n_sm ? 32 : 8;   // (32 sinks from two tiles per warp)
}

static void launch_row_sums(Ctx* c, int l, RowSums a, bool only_if_rebuilding) {
    cut_lists(c, a);
    const bool wgt = c->weighted || a.src_norm;
#define SUMS(NV, WGT)                                                                                                     \
    do {                                                                                                                  \
        RP_LAUNCH(c, (k_sum_rows<NV, WGT>), RP_RESIDENT(c, (k_sum_rows<NV, WGT>), SUM_T), SUM_T, 0, (const Ctl*)c->ctl, l, (int)only_if_rebuilding, a); \
        RP_LAUNCH(c, (k_sum_rows_long<NV, WGT>), RP_RESIDENT(c, (k_sum_rows_long<NV, WGT>), SUM_T), SUM_T, 0, (const Ctl*)c->ctl, l, (int)only_if_rebuilding, a, &c->ctl->hub_ticket[l]); \
    } while (0)
    RP_PIECES_DISPATCH(a.ld, wgt, SUMS);
#undef SUMS
}

// The few rows that the fold sends back to be gathered anew.  The chain waits for the longest chunk, so a whole block takes
// one, 32 entries per warp, and adds its warps' sums up in shared memory before they reach the row (which the fold has
// zeroed): ten rows of the weighted sum on the sparse graph 63 us with a warp per 256 entries, 10 us so; a hub of 26 000
// entries, whose row 800 separate additions would queue for, 45 -> 15 us.
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_spmm_anew(Side in, const int32_t* __restrict__ deg_out, int src_norm, const float* __restrict__ M, int ld, float* S,
            const int2* __restrict__ items, const int* __restrict__ n_items) {
    pdl_enter();
    extern __shared__ __align__(16) float part[];   // [8][ld]
    const int n = *n_items, warp = threadIdx.x >> 5, lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    constexpr int PER_WARP = RP_ANEW_CHUNK / 8;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int2 w = items[it];
        const int deg = in.deg[w.x], j0 = w.y * RP_ANEW_CHUNK + warp * PER_WARP;
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        spmm_accumulate<NV, LPR>(acc, in, w.x, j0, min(deg, j0 + PER_WARP), deg_out, src_norm, M, ld);
        __syncthreads();   // the sums of the item before have been read
        if (sub == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const int q = ql + LPR * k;
                if (q < nq) *reinterpret_cast<float4*>(part + warp * ld + 4 * q) = acc[k];
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < nq; q += blockDim.x) {
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k = 0; k < 8; ++k) add4(t, *reinterpret_cast<const float4*>(part + k * ld + 4 * q), 1.0f);
            red_add_v4(S + (size_t)w.x * ld + 4 * q, t);
        }
    }
}

static RowSums row_sums(Ctx* c, int l) {
    RowSums a{};
    a.in = c->side[1];
    a.deg_out = c->side[0].deg;
    a.src_norm = c->src_norm;
    a.M = c->pre[l] ? c->P[l] : c->H[l - 1];
    a.ld = c->ws[l];
    a.S = c->S[l];
    a.items = c->items;
    a.n_items = &c->ctl->work_counter[(l - 1) & 7];
    a.ticket = &c->ctl->regather_ticket[l];
    return a;
}

void spmm_full(Ctx* c, int l) {
    if (c->pre[l]) project_full(c, l);
    RowSums a = row_sums(c, l);
    a.n_host = c->N;
    launch_row_sums(c, l, a, false);
}

// ---------------------------------------------------------------------------------------------
// edge-change records
// ---------------------------------------------------------------------------------------------
// Messages of the net edge changes: S_v += sign * w * M_r with M_r = c_old m_old of the record's
// source (= c_new m_new - D_u if the source is a sender of this hop, c m otherwise) and w the edge's
// stored weight (1 without stored weights).  One warp per record; rows have the inbox width.
// A pushing hop delivers them in the walk's launch (both only add to the accumulator), by the last blocks of the grid:
// the pushes launch eight blocks per SM, of which registers admit three to five at a time, so on a large walk these
// blocks begin when others run out of tickets.  A swept hop delivers them in the sweep's first launch.  The bulk push and
// hops that are always rebuilt have a launch of their own for them.
struct RecMsgs {
    const Rec* rec;
    int src_norm;
    const int32_t* deg_out;
    const int32_t* posmap;
    const float* Mrows;
};

__device__ __forceinline__ void d_scatter_records(const Ctl* ctl, const RecMsgs& a, const float* __restrict__ D, int ld, float* S) {
    const int n = ctl->n_rec;
    const int nwarps = (gridDim.x * blockDim.x) >> 5, warp = nwarps - 1 - (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = lane_id(), nq = ld >> 2;
    for (int r = warp; r < n; r += nwarps) {
        if (a.rec[r].silent) continue;   // partitioned execution: the source's worker sends for this edge
        const int u = a.rec[r].u;
        const int p = a.posmap[u];
        const float4* hrow = reinterpret_cast<const float4*>(a.Mrows + (size_t)u * ld);
        const float cn = a.src_norm ? coef_from_degree(a.deg_out[u]) : 1.0f;
        const float sgn = (float)a.rec[r].sign * a.rec[r].w;
        float* dst = S + (size_t)a.rec[r].v * ld;
        for (int q = lane; q < nq; q += 32) {
            float4 h = __ldg(hrow + q);
            float4 m = make_float4(cn * h.x, cn * h.y, cn * h.z, cn * h.w);
            if (p >= 0) {
                float4 d = __ldg(reinterpret_cast<const float4*>(D + (size_t)p * ld) + q);
                m.x -= d.x; m.y -= d.y; m.z -= d.z; m.w -= d.w;
            }
            red_add_v4(dst + 4 * q, make_float4(sgn * m.x, sgn * m.y, sgn * m.z, sgn * m.w));
        }
    }
}

__global__ void k_scatter_records(Ctl* ctl, int l, const RecMsgs recs, const float* __restrict__ D, int ld, float* S) {
    pdl_enter();
    if (ctl->abort || ctl->regather[l]) return;
    d_scatter_records(ctl, recs, D, ld, S);
}

// ---------------------------------------------------------------------------------------------
// push scatter
// ---------------------------------------------------------------------------------------------
constexpr int PUSH_CHUNK = 64, PUSH_CHUNK_LARGE = 256;  // edges per warp work item

template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_scatter_push(Ctl* ctl, int l, const int32_t* __restrict__ senders, const int64_t* __restrict__ coff,
               Side out, const float* __restrict__ D, int ld, float* S, uint32_t* bitmap,
               const RecMsgs recs, int rows) {
    pdl_enter();
    if (ctl->abort || ctl->pull[l] || ctl->regather[l]) return;
    d_scatter_records(ctl, recs, D, ld, S);
    const int nC = ctl->nC[l - 1];
    if (nC == 0) return;
    const int64_t E = coff[nC];
    const int lane = lane_id(), nq = ld >> 2;
    constexpr int EPI = 32 / LPR;
    const int sub = lane / LPR, ql = lane % LPR;
    __shared__ int2 s_queue[8][WALK_QUEUE];
    int2* queue = s_queue[threadIdx.x >> 5];
    TicketWalk walk(&ctl->walk_ticket[l], E, PUSH_CHUNK, PUSH_CHUNK_LARGE, rows, ld);
    for (; walk.has(); walk.advance()) {
        const int64_t e0 = walk.at, e1 = min(e0 + walk.chunk, E);
        walk.take();
        int i = upper_row(coff, nC, e0);
        int64_t e = e0;
        while (e < e1) {
            const int64_t row_end = coff[i + 1];
            if (row_end <= e) { ++i; continue; }
            const int64_t seg_end = min(e1, row_end);
            const int64_t base = out.start[senders[i]] + (e - coff[i]);
            float4 d[NV];
            const float4* drow = reinterpret_cast<const float4*>(D + (size_t)i * ld);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int q = ql + LPR * k;
                d[k] = q < nq ? __ldg(drow + q) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            const int cnt_total = (int)(seg_end - e);
            walk_entries<true>(out.col, out.w, base, cnt_total, walk, queue, [&](int mine, float mine_w, int cnt) {
                // (stored edge weights: the message along an edge is the sender's delta row times the edge's weight)
                // every sink joins the hop's affected set (same walk as the frontier's): one lane per
                // edge, 32 edges per instruction
                if (lane < cnt) {
                    const uint32_t m = 1u << (mine & 31);
                    if (!(bitmap[mine >> 5] & m)) atomicOr(&bitmap[mine >> 5], m);
                }
                for (int j = 0; j < cnt; j += EPI) {
                    int jj = j + sub;
                    int v = __shfl_sync(FULL, mine, jj & 31);
                    const float a = __shfl_sync(FULL, mine_w, jj & 31);
                    if (jj < cnt) {
                        float* dst = S + (size_t)v * ld;
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            int q = ql + LPR * k;
                            if (q < nq) red_add_v4(dst + 4 * q, make_float4(a * d[k].x, a * d[k].y, a * d[k].z, a * d[k].w));
                        }
                    }
                }
            });
            e = seg_end;
            ++i;
        }
    }
}

// Packed form for row widths that do not divide a warp (48 floats = 12 lanes, 40 floats = 10):
// messages are laid end to end over the lanes of consecutive instructions (8 messages over 3
// instructions for 12 lanes), so every reduction instruction carries 32 active lanes instead of
// 24.  Lane t of instruction i serves float4 slot (32 i + t) % NQ of message (32 i + t) / NQ.
// WEIGHTED: edges carry stored weights, the message along an edge is the delta row times its weight.
template <int NQ, bool WEIGHTED>
__global__ void __launch_bounds__(256)
k_scatter_push_packed(Ctl* ctl, int l, const int32_t* __restrict__ senders, const int64_t* __restrict__ coff,
                      Side out, const float* __restrict__ D, float* S, uint32_t* bitmap,
                      const RecMsgs recs, int rows) {
    pdl_enter();
    constexpr int LCM = NQ == 12 ? 96 : NQ == 10 ? 160 : NQ * 32;
    constexpr int NI = LCM / 32, G = LCM / NQ, LD = NQ * 4;
    if (ctl->abort || ctl->pull[l] || ctl->regather[l]) return;
    d_scatter_records(ctl, recs, D, LD, S);
    const int nC = ctl->nC[l - 1];
    if (nC == 0) return;
    const int64_t E = coff[nC];
    const int lane = lane_id();
    int msg_of[NI], slot_of[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) { msg_of[i] = (32 * i + lane) / NQ; slot_of[i] = (32 * i + lane) % NQ; }
    __shared__ int2 s_queue[8][WALK_QUEUE];
    int2* queue = s_queue[threadIdx.x >> 5];
    TicketWalk walk(&ctl->walk_ticket[l], E, PUSH_CHUNK, PUSH_CHUNK_LARGE, rows, LD);
    for (; walk.has(); walk.advance()) {
        const int64_t e0 = walk.at, e1 = min(e0 + walk.chunk, E);
        walk.take();
        int i = upper_row(coff, nC, e0);
        int64_t e = e0;
        while (e < e1) {
            const int64_t row_end = coff[i + 1];
            if (row_end <= e) { ++i; continue; }
            const int64_t seg_end = min(e1, row_end);
            const int64_t base = out.start[senders[i]] + (e - coff[i]);
            float4 d[NI];
            const float4* drow = reinterpret_cast<const float4*>(D + (size_t)i * LD);
#pragma unroll
            for (int k = 0; k < NI; ++k) d[k] = __ldg(drow + slot_of[k]);
            const int cnt_total = (int)(seg_end - e);
            walk_entries<WEIGHTED>(out.col, out.w, base, cnt_total, walk, queue, [&](int mine, float mine_w, int cnt) {
                if (lane < cnt) {
                    const uint32_t m = 1u << (mine & 31);
                    if (!(bitmap[mine >> 5] & m)) atomicOr(&bitmap[mine >> 5], m);
                }
                for (int g0 = 0; g0 < cnt; g0 += G) {
#pragma unroll
                    for (int k = 0; k < NI; ++k) {
                        const int idx = g0 + msg_of[k];
                        const int v = __shfl_sync(FULL, mine, idx & 31);
                        float4 m4 = d[k];
                        if (WEIGHTED) {
                            const float a = __shfl_sync(FULL, mine_w, idx & 31);
                            m4 = make_float4(a * m4.x, a * m4.y, a * m4.z, a * m4.w);
                        }
                        if (idx < cnt) red_add_v4(S + (size_t)v * LD + 4 * slot_of[k], m4);
                    }
                }
            });
            e = seg_end;
            ++i;
        }
    }
}

// Bulk form of the push scatter: the sender's delta row is staged in shared memory once per work
// item, and each lane then delivers it along one out-edge with a single bulk reduction
// (cp.reduce.async.bulk ... add.f32: the copy engine adds the whole row, 16-byte aligned, into the
// sink's row in global memory).  One instruction per message instead of one per 16 bytes of it.
// Measured on the dense graph it takes exactly as long as the vector-reduction form (hop 2 at 48
// floats 1.14 against 1.12 ms, at 256 floats 6.15 against 6.18 ms): the additions are retired by
// the L2 slices at the same rate whoever issues them, so the form is selectable
// (RIPPLE_SCATTER_PUSH_BULK), not the default.
// Every lane closes its bulk operations of a work item into one group; before a staging buffer
// (two per warp) is rewritten each lane waits until its group that read the buffer has done so,
// and before the warp leaves, until all its groups have completed.
constexpr int PUSH_BULK_CHUNK = 128;  // edges per warp work item

__device__ __forceinline__ void bulk_reduce_add_f32(float* gdst, const float* smem_src, uint32_t bytes) {
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(gdst),
                 "r"((uint32_t)__cvta_generic_to_shared(smem_src)), "r"(bytes)
                 : "memory");
}

__global__ void __launch_bounds__(256)
k_scatter_push_bulk(Ctl* ctl, int l, const int32_t* __restrict__ senders, const int64_t* __restrict__ coff,
                    Side out, const float* __restrict__ D, int ld, float* S, uint32_t* bitmap) {
    pdl_enter();
    extern __shared__ __align__(16) float stage_all[];
    if (ctl->abort || ctl->pull[l] || ctl->regather[l]) return;
    const int nC = ctl->nC[l - 1];
    if (nC == 0) return;
    const int64_t E = coff[nC];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const int lane = lane_id(), nq = ld >> 2;
    float* stage = stage_all + (size_t)(threadIdx.x >> 5) * 2 * ld;
    int buf = 0;
    for (int64_t e0 = (int64_t)warp * PUSH_BULK_CHUNK; e0 < E; e0 += (int64_t)nwarps * PUSH_BULK_CHUNK) {
        const int64_t e1 = min(e0 + PUSH_BULK_CHUNK, E);
        int i = upper_row(coff, nC, e0);
        int64_t e = e0;
        while (e < e1) {
            const int64_t row_end = coff[i + 1];
            if (row_end <= e) { ++i; continue; }
            const int64_t seg_end = min(e1, row_end);
            const int64_t base = out.start[senders[i]] + (e - coff[i]);
            // this buffer was last read by the bulk operations of two segments ago
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            __syncwarp();
            float* row = stage + (size_t)buf * ld;
            const float4* drow = reinterpret_cast<const float4*>(D + (size_t)i * ld);
            for (int q = lane; q < nq; q += 32) reinterpret_cast<float4*>(row)[q] = __ldg(drow + q);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic stores -> visible to the copy engine
            __syncwarp();
            const int cnt_total = (int)(seg_end - e);
            for (int j0 = 0; j0 < cnt_total; j0 += 32) {
                if (j0 + lane < cnt_total) {
                    const int v = out.col[base + j0 + lane];
                    const uint32_t m = 1u << (v & 31);
                    if (!(bitmap[v >> 5] & m)) atomicOr(&bitmap[v >> 5], m);
                    bulk_reduce_add_f32(S + (size_t)v * ld, row, (uint32_t)ld * 4u);
                }
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            buf ^= 1;
            e = seg_end;
            ++i;
        }
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------
// sweeping form of the delta scatter: every in-list is read once and the delta rows of the senders in it are summed in
// registers, so that a sink's accumulator row takes one addition where the push makes one per message.
//
// Whether an id is a sender's is first asked of a filter in shared memory, which every block fills from the sender list:
// one bit per vertex on graphs of up to 2^19 of them, else one of 2^19 bits per id by a multiplicative hash; the position
// map, one trip to L2, is asked about the few that pass.  The delta rows are few and stay in L2.
//
// What bounds it: the trips to memory of a window and of the rows on their way with 20 warps per SM, at 59 to 65 % of L1TEX, 42
// to 54 % of the issue slots and 37 to 55 % of L2 (30 M edges, 7.6 M rows of 256 floats: 0.59 ms, 12.3 TB/s out of L2).
// ---------------------------------------------------------------------------------------------
constexpr int SWEEP_BITS = 19;
// One block per SM: as many threads as leave them the registers that the rows on their way and the ids of the next window
// take, 102 where a lane has one or two pieces of a row (with 1024 and 768 threads 300 to 580 bytes a thread were spilled, now
// 4 to 200, none at four pieces; eight spill 192 to 364, and 384 threads without are no faster).  49 M rows of 44 floats, 115 M
// edges: 1469 -> 1269 us; 24 M of 256 floats, 124 M edges: 2141 -> 1988; 33 M of 128: 1482 -> 1261.
template <int NV>
__host__ __device__ constexpr int sweep_threads() { return NV <= 2 ? 640 : 512; }

struct Sweep {
    Side in;
    const int32_t* senders;
    const int32_t* posmap;
    const float* D;
    int ld;
    float* dS;
    uint32_t* bitmap;
    int2* items;
    int N, filter_words;
    int take, long_list, item, piece;   // see RowSums
};

struct SenderFilter {
    const uint32_t* bits;
    bool on;
    uint32_t mul;
    int shift;               // the word of an id: (id * mul) >> shift; its bit: the id's lowest five
    __device__ __forceinline__ uint32_t hit(int id) const { return bits[(uint32_t)id * mul >> shift] >> (id & 31) & 1u; }
    // (filling the filter costs a cycle per sender, a look-up that it spares 0.005 of one; and hashed it lets a quarter of
    // the others through at 2^17 senders)
    __device__ __forceinline__ SenderFilter(const Ctl* ctl, int l, const Sweep& a, uint32_t* smem) : bits(smem) {
        const int nC = ctl->nC[l - 1];
        const bool exact = a.N <= 1 << SWEEP_BITS;
        mul = exact ? 1u : 2654435761u;
        shift = exact ? 5 : 32 - (SWEEP_BITS - 5);
        on = 192ll * nC <= ctl->num_edges && (exact || nC <= 1 << (SWEEP_BITS - 2));
        if (!on) return;
        for (int i = threadIdx.x; i < a.filter_words; i += blockDim.x) smem[i] = 0u;
        __syncthreads();
#pragma unroll 4
        for (int i = threadIdx.x; i < nC; i += blockDim.x) {
            const int id = a.senders[i];
            atomicOr(&smem[(uint32_t)id * mul >> shift], 1u << (id & 31));
        }
        __syncthreads();
    }
};

// The queue's first `held` ids become rows of D by the position map, which has the last word: what it does not know leaves
// the queue.  Returns how many stay; `reached` takes, per lane, bits of the sinks reached.
template <bool WGT, bool ONE>
__device__ __forceinline__ int sweep_resolve(const RowQueue<WGT>& q, int held, const int32_t* __restrict__ posmap, unsigned& reached) {
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    int p[RG_CAP / 32];
#pragma unroll
    for (int k = 0; k < RG_CAP / 32; ++k) p[k] = 32 * k + lane < held ? posmap[q.row[32 * k + lane]] : -1;
    int n = 0, last = -1;
#pragma unroll
    for (int k = 0; k < RG_CAP / 32; ++k) {
        if (32 * k >= held) break;
        const unsigned m = __ballot_sync(FULL, p[k] >= 0);
        if (m == 0) continue;
        const int v = ONE ? 0 : q.sink[32 * k + lane];
        const float w = WGT ? q.w[32 * k + lane] : 1.0f;
        const int flag = ONE ? 0 : rg_new_sink(m, v, last), at = n + __popc(m & lt);
        if (WGT || !ONE) __syncwarp();
        if (p[k] >= 0) {
            q.row[at] = p[k] | flag;
            if (!ONE) q.sink[at] = v;
            if (WGT) q.w[at] = w;
            reached |= ONE ? 1u : 1u << (v & 31);
        }
        n += __popc(m);
    }
    __syncwarp();
    return n;
}

// Adds the delta rows of the senders in a piece of one list to acc; returns, per lane, whether there were any.  The ids are
// read four to a lane from the aligned place before the piece, two windows ahead.
template <int NV, bool WGT>
__device__ __forceinline__ unsigned sweep_list(const RowLanes& g, int64_t first, int n, const Sweep& a, const SenderFilter& filter,
                                               const RowQueue<WGT>& q, float4 (&acc)[NV]) {
    const int lane = lane_id(), lead = (int)(first & 3), total = lead + n;
    const int32_t* const from = a.in.col + (first - lead);
    auto ids = [&](int f) { return f < total ? *reinterpret_cast<const int4*>(from + f) : make_int4(0, 0, 0, 0); };   // (a list's last piece may reach into its slack)
    unsigned reached = 0;
    int held = 0;
    int4 x0 = ids(4 * lane), x1 = ids(RG_WINDOW + 4 * lane);
    for (int f0 = 0; f0 < total; f0 += RG_WINDOW) {
        int u[4] = {x0.x, x0.y, x0.z, x0.w};
        x0 = x1;
        x1 = ids(f0 + 2 * RG_WINDOW + 4 * lane);
        unsigned m = 0xfu;
        if (f0 < lead || f0 + RG_WINDOW > total) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int f = f0 + 4 * lane + k;
                if (f < lead || f >= total) {
                    u[k] = 0;
                    m &= ~(1u << k);
                }
            }
        }
        if (filter.on) m &= filter.hit(u[0]) | filter.hit(u[1]) << 1 | filter.hit(u[2]) << 2 | filter.hit(u[3]) << 3;
        if (__any_sync(FULL, m)) {
            const int c = __popc(m), inc = warp_inclusive_scan(c);
            int at = held + inc - c;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (m >> k & 1u) {
                    q.row[at] = u[k];
                    if (WGT) q.w[at] = a.in.w ? a.in.w[first - lead + f0 + 4 * lane + k] : 1.0f;
                    ++at;
                }
            held += __shfl_sync(FULL, inc, 31);
        }
        if (held == 0 || (held < RG_DRAIN && f0 + RG_WINDOW < total)) continue;
        __syncwarp();
        const int rows = sweep_resolve<WGT, true>(q, held, a.posmap, reached);
        if (rows) rg_walk<NV, WGT, true>(g, q, rows, a.D, a.ld, a.dS, acc);
        __syncwarp();
        held = 0;
    }
    return reached;
}

// Adds the delta rows of the senders in a tile's run to their sinks' accumulator rows; returns, per lane, bits of the sinks
// reached.
template <int NV, bool WGT>
__device__ __forceinline__ unsigned sweep_tile(const RowLanes& g, const TileRun& run, const Sweep& a, const SenderFilter& filter,
                                               const RowQueue<WGT>& q, float4 (&acc)[NV], int begin) {
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    unsigned reached = 0;
    int held = 0;
    IdWindow<WGT, TileRun> nx;
    nx.request(run, a.in, begin);
    for (int f0 = begin; f0 < run.total; f0 += RG_WINDOW) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = nx.u[k] >= 0 && (!filter.on || filter.hit(max(nx.u[k], 0)));
            const unsigned m = __ballot_sync(FULL, in);
            if (in) q.put(held + __popc(m & lt), nx.u[k], nx.sink(k), nx.weight(k));
            held += __popc(m);
        }
        nx.request(run, a.in, f0 + RG_WINDOW);
        if (held == 0 || (held < RG_DRAIN && f0 + RG_WINDOW < run.total)) continue;
        __syncwarp();
        const int rows = sweep_resolve<WGT, false>(q, held, a.posmap, reached);
        if (rows) rg_walk<NV, WGT, false>(g, q, rows, a.D, a.ld, a.dS, acc);
        __syncwarp();
        held = 0;
    }
    return reached;
}

// Steps of `take` consecutive vertices per warp; longer lists are queued for the kernel below.
template <int NV, bool WGT>
__global__ void __launch_bounds__(sweep_threads<NV>(), 1)
k_sweep(Ctl* ctl, int l, const __grid_constant__ Sweep a, const RecMsgs recs) {
    pdl_enter();
    if (ctl->abort || !ctl->pull[l] || ctl->regather[l]) return;
    extern __shared__ __align__(16) uint32_t s_dyn[];
    d_scatter_records(ctl, recs, a.D, a.ld, a.dS);
    if (ctl->nC[l - 1] == 0) return;
    const SenderFilter filter(ctl, l, a, s_dyn);
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const RowQueue<WGT> q(reinterpret_cast<char*>(s_dyn + a.filter_words) + warp * RowQueue<WGT>::bytes(RG_CAP), RG_CAP);
    const RowLanes g(a.ld);
    float4 acc[NV];
    rg_zero<NV>(acc);
    const uint32_t* const only = ctl->pull[l] == SWEEP_MARKED ? a.bitmap : nullptr;
    TileDeal deal(a.take == 32 ? &ctl->gather_ticket[l] : nullptr);
    for (int tile = deal.first();; tile = deal.next()) {
        const long long v0 = (long long)a.take * tile;
        if (v0 >= a.N) break;
        const int cnt = (int)min((long long)a.take, a.N - v0);
        if (only && !(only[v0 >> 5] >> (v0 & 31) & (cnt < 32 ? (1u << cnt) - 1u : FULL))) continue;
        const TileLists t(a.in, nullptr, v0, cnt, only);
        TileRun run = t.run(a.long_list);
        rg_queue_rest(t, tile, run.total, a.long_list, a.item, a.piece, a.items, &ctl->gather_items[l]);
        run.total = min(run.total, a.piece);
        const unsigned reached = __reduce_or_sync(FULL, sweep_tile<NV, WGT>(g, run, a, filter, q, acc, 0));
        if (reached && lane == 0) atomicOr(&a.bitmap[v0 >> 5], reached);   // (a tile lies within a word)
    }
}

template <int NV, bool WGT>
__global__ void __launch_bounds__(sweep_threads<NV>(), 1)
k_sweep_long(Ctl* ctl, int l, const __grid_constant__ Sweep a) {
    pdl_enter();
    if (ctl->abort || !ctl->pull[l] || ctl->regather[l]) return;
    extern __shared__ __align__(16) uint32_t s_dyn[];
    const int n = ctl->gather_items[l];
    if (n == 0) return;
    const SenderFilter filter(ctl, l, a, s_dyn);
    const int warp = threadIdx.x >> 5;
    const RowQueue<WGT> q(reinterpret_cast<char*>(s_dyn + a.filter_words) + warp * RowQueue<WGT>::bytes(RG_CAP), RG_CAP);
    const RowLanes g(a.ld);
    float4 acc[NV];
    rg_zero<NV>(acc);
    const uint32_t* const only = ctl->pull[l] == SWEEP_MARKED ? a.bitmap : nullptr;
    TicketWalk walk(&ctl->gather_long_ticket[l], n, 1, 4);
    for (; walk.has(); walk.advance()) {
        const int from = (int)walk.at, to = min(n, from + walk.chunk);
        walk.take();
        for (int it = from; it < to; ++it) {
            const int2 w = a.items[it];
            if (w.x < 0) {
                const long long v0 = (long long)a.take * (-1 - w.x);
                TileRun run = TileLists(a.in, nullptr, v0, (int)min((long long)a.take, a.N - v0), only).run(a.long_list);
                run.total = min(run.total, (w.y + 1) * a.piece);
                const unsigned sinks = __reduce_or_sync(FULL, sweep_tile<NV, WGT>(g, run, a, filter, q, acc, w.y * a.piece));
                if (sinks && lane_id() == 0) atomicOr(&a.bitmap[v0 >> 5], sinks);
                continue;
            }
            const int deg = a.in.deg[w.x];
            const bool reached = __any_sync(FULL, sweep_list<NV, WGT>(g, a.in.start[w.x] + (int64_t)w.y * a.item, min(a.item, deg - w.y * a.item), a, filter, q, acc));
            if (!reached) continue;
            rg_finish_one<NV>(g, a.dS + (size_t)w.x * a.ld, acc);
            const uint32_t m = 1u << (w.x & 31);
            if (lane_id() == 0 && !(a.bitmap[w.x >> 5] & m)) atomicOr(&a.bitmap[w.x >> 5], m);
        }
    }
}

template <int NV>
static size_t sweep_smem(int filter_words, bool wgt) {
    return sizeof(uint32_t) * (size_t)filter_words + (size_t)(sweep_threads<NV>() / 32) * (size_t)(wgt ? RowQueue<true>::bytes(RG_CAP) : RowQueue<false>::bytes(RG_CAP));
}

// One-time attributes of the instances that this context's layers launch (setting them loads a kernel, half a millisecond).
void sweep_prepare(const Ctx* c) {
    for (int l = 1; l <= c->L; ++l) {
        const bool sums = c->weighted || c->src_norm;
        // the rows that many lists name are served by L1, so the sums ask for as much of it as their queues leave
#define PREP(NV, WGT)                                                                                              \
    do {                                                                                                           \
        cudaFuncSetAttribute(k_sum_rows<NV, WGT>, cudaFuncAttributePreferredSharedMemoryCarveout, 25);           \
        cudaFuncSetAttribute(k_sum_rows_long<NV, WGT>, cudaFuncAttributePreferredSharedMemoryCarveout, 25);      \
    } while (0)
        RP_PIECES_DISPATCH(c->ws[l], sums, PREP);
#undef PREP
        // likewise the pushes, which look every sink up in the frontier's bitmap (behind a tensor-core update, with 28 KB of L1
        // left, 26 M messages of 48 floats made the whole batch 1.41 ms instead of 1.28, 50 M of 44 floats 1.73 instead of 1.61)
        const int ld = c->ws[l];
#define PREP(NV, LPR) cudaFuncSetAttribute(k_scatter_push<NV, LPR>, cudaFuncAttributePreferredSharedMemoryCarveout, 35)
        if (ld == 48 && c->weighted) cudaFuncSetAttribute(k_scatter_push_packed<12, true>, cudaFuncAttributePreferredSharedMemoryCarveout, 35);
        else if (ld == 48) cudaFuncSetAttribute(k_scatter_push_packed<12, false>, cudaFuncAttributePreferredSharedMemoryCarveout, 35);
        else if (ld == 40 && c->weighted) cudaFuncSetAttribute(k_scatter_push_packed<10, true>, cudaFuncAttributePreferredSharedMemoryCarveout, 35);
        else if (ld == 40) cudaFuncSetAttribute(k_scatter_push_packed<10, false>, cudaFuncAttributePreferredSharedMemoryCarveout, 35);
        else RP_WIDTH_DISPATCH(ld, PREP);
#undef PREP
        if (c->n_local > 0) continue;
        // and the sweeps, for all but the filter and the queues of the one block
#define PREP(NV, WGT)                                                                                                      \
    do {                                                                                                                   \
        const int smem = (int)sweep_smem<NV>(1 << (SWEEP_BITS - 5), WGT), share = div_up(100 * (smem + 1024), 228 << 10);  \
        cudaFuncSetAttribute(k_sweep<NV, WGT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);                         \
        cudaFuncSetAttribute(k_sweep<NV, WGT>, cudaFuncAttributePreferredSharedMemoryCarveout, share);                     \
        cudaFuncSetAttribute(k_sweep_long<NV, WGT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);                    \
        cudaFuncSetAttribute(k_sweep_long<NV, WGT>, cudaFuncAttributePreferredSharedMemoryCarveout, share);                \
    } while (0)
        RP_PIECES_DISPATCH(c->ws[l], c->weighted, PREP);
#undef PREP
    }
}

static void launch_sweep(Ctx* c, int l, const int32_t* senders, const float* D, const RecMsgs& recs) {
    Sweep a{};
    a.in = c->side[1];
    a.senders = senders;
    a.posmap = c->posmap;
    a.D = D;
    a.ld = c->ws[l];
    a.dS = c->dS[l];
    a.bitmap = c->bitmap;
    a.items = c->items;
    a.N = c->N;
    a.filter_words = std::min(1 << (SWEEP_BITS - 5), (div_up(c->N, 32) + 3) & ~3);   // (the queues behind it are aligned)
    cut_lists(c, a);
#define SWEEP(NV, WGT)                                                                                                                      \
    do {                                                                                                                                    \
        RP_LAUNCH(c, (k_sweep<NV, WGT>), c->n_sm, sweep_threads<NV>(), sweep_smem<NV>(a.filter_words, WGT), c->ctl, l, a, recs);                          \
        RP_LAUNCH(c, (k_sweep_long<NV, WGT>), c->n_sm, sweep_threads<NV>(), sweep_smem<NV>(a.filter_words, WGT), c->ctl, l, a);                           \
    } while (0)
    RP_PIECES_DISPATCH(a.ld, c->weighted, SWEEP);
#undef SWEEP
}

// A sink that lost at least as many in-edges as it keeps is rebuilt from its in-list, whatever
// form the hop takes: subtracting most of a sum leaves the rounding of the large old value on the
// small new one (a hub emptied by a vertex deletion kept 2e-3 where exact zeros belong), while
// gathering the survivors costs no more than the deletions did.  One warp per such row; its
// pending message sums are dropped with it.
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_regather_rows(Ctl* ctl, int l, const Rec* __restrict__ rec, Side in, const int32_t* __restrict__ deg_out,
                int src_norm, const float* __restrict__ M, int ld, float* __restrict__ S, float* __restrict__ dS,
                float* budget, const int32_t* __restrict__ senders, int32_t* posmap, int self_term,
                const int32_t* __restrict__ A_prev, uint32_t* bitmap, int chores_only) {
    pdl_enter();
    // Two chores of the hop ride along with this kernel, the last of the hop's delta form, whatever form
    // the hop takes.  The hop's senders are no longer looked up by anyone: their entries of the position
    // map are cleared.  And the members of A_l that no walk finds are marked: the sinks of
    // net edge changes, and A_{l-1} for models with a self term.
    {
        const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsize = gridDim.x * blockDim.x;
        const int nC = ctl->nC[l - 1];
        for (int i = gtid; i < nC; i += gsize) posmap[senders[i]] = -1;
        if (!ctl->abort) {
            for (int i = gtid; i < ctl->n_rec; i += gsize) {
                const int v = rec[i].v;
                atomicOr(&bitmap[v >> 5], 1u << (v & 31));
            }
            if (self_term)
                for (int i = gtid; i < ctl->nA[l - 1]; i += gsize) {
                    const int v = A_prev[i];
                    atomicOr(&bitmap[v >> 5], 1u << (v & 31));
                }
        }
    }
    // (a worker of a partitioned execution cannot gather a row anew: remote in-neighbours' rows live elsewhere)
    if (ctl->abort || ctl->regather[l] || chores_only) return;
    const int n = ctl->n_rec;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const int lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    for (int r = warp; r < n; r += nwarps) {
        if (!rec[r].rep[1]) continue;          // one record per distinct sink
        const int v = rec[r].v;
        const int deg = in.deg[v], lost = in.cnt_del[v];
        if (lost == 0 || lost < deg) continue;
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        spmm_accumulate<NV, LPR>(acc, in, v, 0, deg, deg_out, src_norm, M, ld);
        if (sub == 0) {
            float4* dst = reinterpret_cast<float4*>(S + (size_t)v * ld);
            float4* pend = reinterpret_cast<float4*>(dS + (size_t)v * ld);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int q = ql + LPR * k;
                if (q < nq) { dst[q] = acc[k]; pend[q] = make_float4(0.f, 0.f, 0.f, 0.f); }
            }
        }
        if (budget && lane == 0) budget[v] = 0.f;
    }
}

// Form of hop l, decided on the device once the senders and their out-degree sum are known.
//
// Delta form: the out-edges of the senders each carry one message, added to the sink's accumulator by vector reductions
// (push), or every in-list is read and the senders' delta rows in it are summed in registers (sweep).
//
// Rebuilding form: once the senders' out-edges are most of the graph, reading every in-edge of
// the affected sinks once and overwriting their aggregates costs less than one reduction per
// message: a gathered row is a plain load, a delivered message a read-modify-write in L2.  The
// rebuilt aggregate also sheds whatever rounding the deltas had left in it.  threshold = the
// share of all edges above which the hop rebuilds (<= 0: never).  With the default threshold a hop
// of fewer than min_messages messages pushes regardless: on a graph of a million edges neither
// form is throughput-bound, and the edge-balanced push is the more parallel of the two (measured
// on the sparse graph, 256 floats per row: 0.24 ms pushed, 0.26 to 0.47 ms rebuilt).
//
// Between push and sweep, where both are in the chain, the cheaper one is taken (see sweep_pays): what the batch before
// carried says nothing about this one.  (Three layers on the graph of 124 M edges, one update after a thousand: hop 2 carries
// 2 K messages of 256 floats, which a sweep chosen by the batch before took 0.5 ms for.)
__global__ void k_choose_direction(Ctl* ctl, int l, int mode, float threshold, long long min_messages, int sweep, int N,
                                   int width) {
    pdl_enter();
    const int nC = ctl->nC[l - 1];
    int re = 0;
    const unsigned long long msgs = ctl->E[l] + (unsigned long long)ctl->n_rec;
    if (mode == RIPPLE_SCATTER_REGATHER) re = 1;
    else if (mode == RIPPLE_SCATTER_AUTO && threshold > 0.f) {
        re = (double)msgs >= (double)threshold * (double)ctl->num_edges && ctl->num_edges > 0 &&
             msgs >= (unsigned long long)min_messages;
    }
    if (nC == 0 && ctl->n_rec == 0) re = 0;
    if (mode == RIPPLE_SCATTER_PULL)
        ctl->pull[l] = sweep_reads_all((double)msgs, (double)ctl->num_edges) ? SWEPT : SWEEP_MARKED;
    else ctl->pull[l] = sweep && sweep_pays((double)msgs, (double)nC, (double)ctl->num_edges, (double)N, width) ? SWEPT : PUSHED;
    ctl->regather[l] = re;
}

// Messages of one batch are first summed among themselves in dS (zero outside a batch) and reach
// the cached aggregate as one addition per affected row.  A hub's aggregate is large and receives
// thousands of small messages per batch; adding each of them to it directly rounds every time at
// the aggregate's magnitude, and the error random-walks with the number of messages (measured
// drift 1e-4 of the value after 100 batches).  Folding keeps it at one rounding per row and batch.
//
// Even that one rounding per batch adds up, and it is taken at the magnitude the row has at the
// time: a sink that loses the edge from a hub keeps, on its now small aggregate, the rounding of
// the large value it held before (on the unnormalised-sum stack rows differ by four orders of
// magnitude).  So every row keeps a budget: the sum over its folds of max|S_v|^2, in units of one
// fp32 rounding.  Once that exceeds tau^2 max|S_v,new|^2 the row is gathered anew from its in-list
// (Sec. 3.2's scoped recomputation, for this one row) and the budget starts again.  tau^2 is
// scaled per vertex by a fixed factor in [0.5, 1), so that rows touched by every batch do not all
// come due in the same batch.  A row that comes due is zeroed and its in-list queued, in chunks,
// for k_spmm_anew.
__global__ void __launch_bounds__(256)
k_fold_deltas(Ctl* ctl, int l, const int32_t* __restrict__ A, int ld, float* S, float* dS, float* budget,
              float tau2, const int32_t* __restrict__ deg_in, int2* items) {
    pdl_enter();
    if (ctl->abort || ctl->regather[l]) return;   // a rebuilt aggregate has no pending sums
    const int n = ctl->nA[l];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const int lane = lane_id(), nq = ld >> 2;
    for (int i = warp; i < n; i += nwarps) {
        const int v = A[i];
        const size_t off = (size_t)v * ld;
        float4* s = reinterpret_cast<float4*>(S + off);
        float4* d = reinterpret_cast<float4*>(dS + off);
        float m_old = 0.f, m_new = 0.f;
        for (int q = lane; q < nq; q += 32) {
            float4 x = s[q], y = d[q];
            m_old = fmaxf(m_old, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
            x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
            m_new = fmaxf(m_new, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
            s[q] = x;
            d[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (!budget) continue;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            m_old = fmaxf(m_old, __shfl_xor_sync(FULL, m_old, o));
            m_new = fmaxf(m_new, __shfl_xor_sync(FULL, m_new, o));
        }
        const float m = fmaxf(m_old, m_new);
        const float spent = budget[v] + m * m;
        const float limit = tau2 * (0.5f + (float)(mix64((uint64_t)v) & 255u) * (1.0f / 512.0f)) * m_new * m_new;
        if (!(spent > limit)) {     // also taken if anything overflowed to inf or nan
            if (lane == 0) budget[v] = spent;
            continue;
        }
        // the row comes due: zero it and queue its in-list, in chunks, for k_spmm_anew
        __syncwarp();
        for (int q = lane; q < nq; q += 32) s[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int deg = deg_in[v];
        const int nch = (deg + RP_ANEW_CHUNK - 1) / RP_ANEW_CHUNK;
        int first = 0;
        if (lane == 0) {
            if (nch) first = atomicAdd(&ctl->rebuild_items[l], nch);
            budget[v] = 0.f;
            atomicAdd(&ctl->n_rebuilt[l], 1);
        }
        first = __shfl_sync(FULL, first, 0);
        for (int ch = lane; ch < nch; ch += 32) items[first + ch] = make_int2(v, ch);
    }
}

void fold_deltas(Ctx* c, int l) {
    if (c->fused_fold[l]) return;   // folded inside the row update's epilogue
    const float* M = c->pre[l] ? c->P[l] : c->H[l - 1];
    int2* items = c->items;
    const int ld = c->ws[l];
    RP_LAUNCH(c, k_fold_deltas, RP_RESIDENT(c, k_fold_deltas, 256), 256, 0, c->ctl, l, c->A[l], ld, c->S[l], c->dS[l], c->Eb[l],
              c->rebuild_tau2, c->side[1].deg, items);
    if (!c->Eb[l]) return;
#define HUBS(NV, LPR)                                                                                              \
    RP_LAUNCH(c, (k_spmm_anew<NV, LPR>), c->n_sm * 4, 256, sizeof(float) * 8 * (size_t)ld, c->side[1], c->side[0].deg, \
              (int)c->src_norm, M, ld, c->S[l], (const int2*)items, (const int*)&c->ctl->rebuild_items[l])
    RP_WIDTH_DISPATCH(ld, HUBS);
#undef HUBS
}

void choose_direction(Ctx* c, int l) {
    // nothing to decide for a pushing hop: the control block's flags are already zero after its reset
    if (!c->rebuild_armed[l] && !c->sweep_armed[l] &&
        (c->scatter_mode == RIPPLE_SCATTER_AUTO || c->scatter_mode == RIPPLE_SCATTER_PUSH ||
         c->scatter_mode == RIPPLE_SCATTER_PUSH_BULK)) return;
    RP_LAUNCH(c, k_choose_direction, 1, 1, 0, c->ctl, l, c->scatter_mode, c->rebuild_armed[l] ? c->regather_threshold[l] : -1.f, c->regather_min_messages, c->sweep_armed[l], c->N, c->ws[l]);
}

// delta form of hop l (does nothing on the device if the hop rebuilds)
void scatter_layer(Ctx* c, int l, int n) {
    const int ld = c->ws[l];
    const float* D = c->D[(l - 1) & 1];
    const int32_t* senders = sender_list(c, l - 1);
    const int T = 256;
    const int grid = c->n_sm * 8;
    // Edge records: M_r = c_old m_old of the record's source = c_new m_new - D_u for a sender.  A
    // layer that transforms first keeps m = P^l rows up to date for the senders, whatever form the
    // hop takes, and builds its records from them directly.
    const float* Dm = D;
    const float* Mrows = c->H[l - 1];
    if (c->pre[l]) {
        sender_transform(c, l);
        Dm = c->Dt;
        Mrows = c->P[l];
    }
    if (c->timing) cudaEventRecord(c->ev_sc[2 * l], c->stream);
    const RecMsgs recs{c->rec, (int)c->src_norm, c->side[0].deg, c->posmap, Mrows};
    bool recs_done = false;
#define PUSH(NV, LPR) RP_LAUNCH(c, (k_scatter_push<NV, LPR>), grid, T, 0, c->ctl, l, senders, c->coff, c->side[0], Dm, ld, c->dS[l], c->bitmap, recs, c->N)
    // (rows too wide for two staging buffers per warp in the default shared-memory allowance take the ordinary form)
    if (c->scatter_mode == RIPPLE_SCATTER_PUSH_BULK && !c->weighted && (size_t)8 * 2 * ld * sizeof(float) <= (48u << 10)) {
        RP_LAUNCH(c, k_scatter_push_bulk, grid, T, (size_t)8 * 2 * ld * sizeof(float), c->ctl, l, senders, c->coff,
                  c->side[0], Dm, ld, c->dS[l], c->bitmap);
    } else if (c->scatter_mode != RIPPLE_SCATTER_PULL && c->scatter_mode != RIPPLE_SCATTER_REGATHER) {
#define PACKED(NQ, WGT) RP_LAUNCH(c, (k_scatter_push_packed<NQ, WGT>), grid, T, 0, c->ctl, l, senders, c->coff, c->side[0], Dm, c->dS[l], c->bitmap, recs, c->N)
        if (ld == 48 && c->weighted) PACKED(12, true);
        else if (ld == 48) PACKED(12, false);
        else if (ld == 40 && c->weighted) PACKED(10, true);
        else if (ld == 40) PACKED(10, false);
#undef PACKED
        else RP_WIDTH_DISPATCH(ld, PUSH);
        recs_done = true;
    }
#undef PUSH
    if (c->sweep_armed[l]) {
        launch_sweep(c, l, senders, Dm, recs);
        recs_done = true;
    }
    if (c->timing) cudaEventRecord(c->ev_sc[2 * l + 1], c->stream);
    if (n > 0) {
        if (!recs_done)
            RP_LAUNCH(c, k_scatter_records, std::min(div_up(n, T / 32), c->n_sm * 8), T, 0, c->ctl, l, recs, Dm, ld, c->dS[l]);
        const float* rows = c->pre[l] ? c->P[l] : c->H[l - 1];
#define ROWS(NV, LPR) RP_LAUNCH(c, (k_regather_rows<NV, LPR>), std::min(div_up(n, T / 32), c->n_sm * 8), T, 0, c->ctl, l, c->rec, c->side[1], c->side[0].deg, (int)c->src_norm, rows, ld, c->S[l], c->dS[l], c->Eb[l], senders, c->posmap, (int)c->self_term, c->A[l - 1], c->bitmap, (int)(c->n_local > 0))
        RP_WIDTH_DISPATCH(ld, ROWS);
#undef ROWS
    }
}

// rebuilding form of hop l (does nothing on the device unless the hop rebuilds); needs the list A_l
void regather_layer(Ctx* c, int l) {
    if (!c->rebuild_armed[l]) return;
    if (c->timing) cudaEventRecord(c->ev_rg[2 * l], c->stream);
    RowSums a = row_sums(c, l);   // (P^l rows of the senders are already current)
    a.list = c->A[l];
    a.n_dev = &c->ctl->nA[l];
    a.budget = c->Eb[l];
    launch_row_sums(c, l, a, true);
    if (c->timing) cudaEventRecord(c->ev_rg[2 * l + 1], c->stream);
}

// ---------------------------------------------------------------------------------------------
// diagnostic: the rate at which the device retires the 16-byte vector reductions the push scatter
// is made of, on rows drawn pseudo-randomly from a window of n_rows rows
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_probe_reductions(float* buf, long long n_rows, int nq, long long n_messages, unsigned long long seed, int pattern) {
    pdl_enter();
    const long long total = n_messages * nq;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long m = t / nq;
        const int q = (int)(t - m * nq);
        long long row;
        if (pattern == 1) row = m % n_rows;                                    // consecutive rows
        else {
            const unsigned long long h = mix64((unsigned long long)m + seed);
            row = (long long)(h % (unsigned long long)n_rows);                  // uniformly random rows
            if (pattern == 2) {                                                 // popular rows: position = u^3
                const double u = (double)(h >> 11) * (1.0 / 9007199254740992.0);
                row = (long long)(u * u * u * (double)n_rows);
            }
        }
        red_add_v4(buf + (size_t)row * (4 * nq) + 4 * q, make_float4(1.f, 1.f, 1.f, 1.f));
    }
}

// diagnostic: the rate at which the device serves whole rows read from pseudo-random places of a
// window of n_rows rows, with the lane layout of the gathering kernels (LPR lanes per row, 32 / LPR
// rows per warp instruction), eight instructions in flight per warp and nothing else going on: what
// a gather over in-lists could reach if its indices cost nothing
template <int LPR>
__global__ void __launch_bounds__(256)
k_probe_gathers(const float* __restrict__ buf, unsigned long long n_rows, int nq, long long n_gathers,
                unsigned long long seed, float* sink) {
    pdl_enter();
    constexpr int EPI = 32 / LPR, UNR = 8;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int lane = lane_id(), sub = lane / LPR, ql = lane % LPR;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long g0 = warp * (UNR * EPI); g0 < n_gathers; g0 += nwarps * (UNR * EPI)) {
        for (int q0 = 0; q0 < nq; q0 += LPR) {
            float4 x[UNR];
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const long long g = g0 + t * EPI + sub;
                // uniform row index without a 64-bit division: high half of hash x n_rows
                const unsigned long long row = __umul64hi(mix64((unsigned long long)g + seed), n_rows);
                const float4* p = reinterpret_cast<const float4*>(buf + (size_t)row * (4 * nq));
                x[t] = (q0 + ql < nq && g < n_gathers) ? __ldg(p + q0 + ql) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int t = 0; t < UNR; ++t) add4(acc, x[t], 1.0f);
        }
    }
    if (acc.x + acc.y + acc.z + acc.w == 12345.678f) sink[0] = acc.x;   // keeps the loads alive
}

}  // namespace rp

extern "C" ripple_status ripple_probe_reduction_rate(int32_t device, int64_t n_rows, int32_t row_floats,
                                                     int64_t n_messages, int32_t pattern, float* ms_out) {
    if (pattern < 0 || pattern > 2) return RIPPLE_ERR_INVALID_ARG;
    if (n_rows < 1 || row_floats < 4 || (row_floats & 3) || n_messages < 1 || !ms_out) return RIPPLE_ERR_INVALID_ARG;
    if (device >= 0 && cudaSetDevice(device) != cudaSuccess) return RIPPLE_ERR_CUDA;
    float* buf = nullptr;
    const size_t bytes = sizeof(float) * (size_t)n_rows * (size_t)row_floats;
    if (cudaMalloc(&buf, bytes) != cudaSuccess) { cudaGetLastError(); return RIPPLE_ERR_OOM; }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int n_sm = 1;
    cudaGetDevice(&device);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, device);
    cudaMemset(buf, 0, bytes);
    float best = 0.f;
    for (int rep = 0; rep < 4; ++rep) {   // the first pass warms up
        cudaEventRecord(e0);
        rp::k_probe_reductions<<<n_sm * 8, 256>>>(buf, n_rows, row_floats / 4, n_messages, 0x9E37ull * (rep + 1), pattern);
        cudaEventRecord(e1);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0 && (best == 0.f || ms < best)) best = ms;
    }
    cudaError_t e = cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(buf);
    *ms_out = best;
    return e == cudaSuccess ? RIPPLE_OK : RIPPLE_ERR_CUDA;
}

extern "C" ripple_status ripple_probe_gather_rate(int32_t device, int64_t n_rows, int32_t row_floats,
                                                  int64_t n_gathers, float* ms_out) {
    if (n_rows < 1 || row_floats < 4 || (row_floats & 3) || n_gathers < 1 || !ms_out) return RIPPLE_ERR_INVALID_ARG;
    if (device >= 0 && cudaSetDevice(device) != cudaSuccess) return RIPPLE_ERR_CUDA;
    float* buf = nullptr;
    const size_t bytes = sizeof(float) * (size_t)n_rows * (size_t)row_floats;
    if (cudaMalloc(&buf, bytes + 16) != cudaSuccess) { cudaGetLastError(); return RIPPLE_ERR_OOM; }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int n_sm = 1;
    cudaGetDevice(&device);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, device);
    cudaMemset(buf, 0, bytes + 16);
    float best = 0.f;
    for (int rep = 0; rep < 4; ++rep) {   // the first pass warms up
        cudaEventRecord(e0);
        const int nq = row_floats / 4;
        float* sink = buf + (size_t)n_rows * row_floats;
        const unsigned long long seed = 0x9E37ull * (rep + 1);
        if (nq <= 8) rp::k_probe_gathers<8><<<n_sm * 8, 256>>>(buf, (unsigned long long)n_rows, nq, n_gathers, seed, sink);
        else if (nq <= 16) rp::k_probe_gathers<16><<<n_sm * 8, 256>>>(buf, (unsigned long long)n_rows, nq, n_gathers, seed, sink);
        else rp::k_probe_gathers<32><<<n_sm * 8, 256>>>(buf, (unsigned long long)n_rows, nq, n_gathers, seed, sink);
        cudaEventRecord(e1);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0 && (best == 0.f || ms < best)) best = ms;
    }
    cudaError_t e = cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(buf);
    *ms_out = best;
    return e == cudaSuccess ? RIPPLE_OK : RIPPLE_ERR_CUDA;
}
