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
// pull: a warp per affected sink walks its in-list, keeps only sources that are senders
//       (position map), sums their delta rows in registers and touches S_v once.
#include "device_utils.cuh"
#include "ripple_internal.cuh"

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
// In-lists longer than this are cut into chunks handled by separate warps.  A warp gathers about
// three neighbours per microsecond at 256 floats per row, so one 2048-neighbour row used to keep a
// single warp busy for 0.7 ms, longer than everything else of a hop on the sparse graph.
constexpr int SPMM_HUB_DEGREE = 256;
constexpr int SPMM_HUB_CHUNK = 256;
static_assert(SPMM_HUB_CHUNK >= RP_ANEW_CHUNK && SPMM_HUB_DEGREE >= RP_ANEW_CHUNK, "the item buffer is sized by RP_ANEW_CHUNK");

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

// One warp per vertex.  A vertex with a long in-list only zeroes its row here and queues
// (vertex, chunk) work items for k_spmm_hubs, so that no single warp walks thousands of neighbours.
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_spmm_pull(int N, Side in, const int32_t* __restrict__ deg_out, int src_norm,
            const float* __restrict__ M, int ld, float* __restrict__ S, int2* items, int* n_items, int* ticket) {
    pdl_enter();
    const int lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    // vertices are handed out in runs of eight by ticket: in-lists differ in length
    for (;;) {
        int v0 = 0;
        if (lane == 0) v0 = atomicAdd(ticket, 8);
        v0 = __shfl_sync(FULL, v0, 0);
        if (v0 >= N) break;
    for (int v = v0; v < min(v0 + 8, N); ++v) {
        const int deg = in.deg[v];
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (deg > SPMM_HUB_DEGREE) {
            const int nch = (deg + SPMM_HUB_CHUNK - 1) / SPMM_HUB_CHUNK;
            int first = 0;
            if (lane == 0) first = atomicAdd(n_items, nch);
            first = __shfl_sync(FULL, first, 0);
            for (int ch = lane; ch < nch; ch += 32) items[first + ch] = make_int2(v, ch);
        } else {
            spmm_accumulate<NV, LPR>(acc, in, v, 0, deg, deg_out, src_norm, M, ld);
        }
        if (sub == 0) {
            float4* dst = reinterpret_cast<float4*>(S + (size_t)v * ld);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int q = ql + LPR * k;
                if (q < nq) dst[q] = acc[k];
            }
        }
    }
    }
}

// The chunks of the long in-lists, one warp per 256-entry chunk; chunk sums are added to the row,
// which the kernel that queued the chunks has zeroed.
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_spmm_hubs(Side in, const int32_t* __restrict__ deg_out, int src_norm, const float* __restrict__ M, int ld,
            float* S, const int2* __restrict__ items, const int* __restrict__ n_items, int* ticket) {
    pdl_enter();
    const int lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    const int n = *n_items;
    if (n == 0) return;
    TicketWalk walk(ticket, n, 1, 1);
    for (; walk.has(); walk.advance()) {
        const int2 w = items[walk.at];
        walk.take();
        const int deg = in.deg[w.x];
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        spmm_accumulate<NV, LPR>(acc, in, w.x, w.y * SPMM_HUB_CHUNK, min(deg, (w.y + 1) * SPMM_HUB_CHUNK), deg_out,
                                 src_norm, M, ld);
        if (sub == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int q = ql + LPR * k;
                if (q < nq) red_add_v4(S + (size_t)w.x * ld + 4 * q, acc[k]);
            }
        }
    }
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

void spmm_full(Ctx* c, int l) {
    const int ld = c->ws[l];
    const float* M = c->H[l - 1];
    if (c->pre[l]) {
        project_full(c, l);
        M = c->P[l];
    }
    const int grid = c->n_sm * 16, T = 256;
    int2* items = c->items;
    int* n_items = &c->ctl->work_counter[(l - 1) & 7];
#define SPMM(NV, LPR)                                                                                              \
    do {                                                                                                           \
        RP_LAUNCH(c, (k_spmm_pull<NV, LPR>), grid, T, 0, c->N, c->side[1], c->side[0].deg, (int)c->src_norm, M,   \
                  ld, c->S[l], items, n_items, &c->ctl->regather_ticket[l]);                                      \
        RP_LAUNCH(c, (k_spmm_hubs<NV, LPR>), grid, T, 0, c->side[1], c->side[0].deg, (int)c->src_norm, M, ld,     \
                  c->S[l], items, n_items, &c->ctl->hub_ticket[l]);                                                \
    } while (0)
    RP_WIDTH_DISPATCH(ld, SPMM);
#undef SPMM
}

// ---------------------------------------------------------------------------------------------
// edge-change records
// ---------------------------------------------------------------------------------------------
// Messages of the net edge changes: S_v += sign * w * M_r with M_r = c_old m_old of the record's
// source (= c_new m_new - D_u if the source is a sender of this hop, c m otherwise) and w the edge's
// stored weight (1 without stored weights).  One warp per record; rows have the inbox width.
// A pushing hop delivers them in the walk's launch (both only add to the accumulator), by the last blocks of the grid:
// the pushes launch eight blocks per SM, of which registers admit three to five at a time, so on a large walk these
// blocks begin when others run out of tickets.  A gathering hop, whose gather stores the rows it finishes, delivers them
// afterwards in a launch of their own.
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
// gathering form of the delta scatter: per affected sink, the delta rows of the senders among its
// in-neighbours are summed in registers and reach the accumulator row as ONE addition.  The sender
// delta rows are few (they stay in L2) and are read with plain loads; no
// accumulator row is touched more than once.  It pays where a message is wide: 256-float
// messages cost the push one kilobyte of read-modify-write each in the L2 slices and evict each
// other's accumulator rows in between.
//
// A warp examines GATHER_WINDOW in-list entries at a time (four per lane, their position-map
// lookups in flight together), compacts the hits into shared memory and then gathers them like
// the bootstrap gather does: LPR lanes per row, 32 / LPR rows per step, several steps in flight.
// ---------------------------------------------------------------------------------------------
constexpr int GATHER_WINDOW = 128;
constexpr int GATHER_LONG = 512;     // longer in-lists are cut into work items of GATHER_ITEM entries
constexpr int GATHER_ITEM = 256;
static_assert(GATHER_ITEM >= RP_ANEW_CHUNK && GATHER_LONG >= RP_ANEW_CHUNK, "the item buffer is sized by RP_ANEW_CHUNK");
constexpr int GATHER_TAKE = 8;       // sinks per ticket

template <int NV, int LPR>
__device__ __forceinline__ bool gather_accumulate(float4 (&acc)[NV], const Side& in, int v, int j_begin, int j_end,
                                                  const int32_t* __restrict__ posmap, const float* __restrict__ D,
                                                  int ld, int2* hits) {
    const int lane = lane_id(), nq = ld >> 2;
    constexpr int EPI = 32 / LPR;
    constexpr int UNR = NV <= 2 ? 4 : 2;
    constexpr int PER_LANE = GATHER_WINDOW / 32;
    const int sub = lane / LPR, ql = lane % LPR;
    const int64_t base = in.start[v];
    const unsigned lt = (1u << lane) - 1u;
    bool any = false;
    for (int j0 = j_begin; j0 < j_end; j0 += GATHER_WINDOW) {
        int u[PER_LANE], p[PER_LANE];
        float w[PER_LANE];
#pragma unroll
        for (int k = 0; k < PER_LANE; ++k) {
            const int j = j0 + 32 * k + lane;
            u[k] = j < j_end ? in.col[base + j] : -1;
            w[k] = (in.w && j < j_end) ? in.w[base + j] : 1.0f;
        }
#pragma unroll
        for (int k = 0; k < PER_LANE; ++k) p[k] = u[k] >= 0 ? posmap[u[k]] : -1;
        int cnt = 0;
        __syncwarp();   // the hits of the window before have all been read
#pragma unroll
        for (int k = 0; k < PER_LANE; ++k) {
            const unsigned m = __ballot_sync(FULL, p[k] >= 0);
            if (p[k] >= 0) hits[cnt + __popc(m & lt)] = make_int2(p[k], __float_as_int(w[k]));
            cnt += __popc(m);
        }
        __syncwarp();
        if (cnt == 0) continue;
        any = true;
        for (int j = 0; j < cnt; j += UNR * EPI) {
            int pj[UNR];
            float a[UNR];
            float4 x[UNR][NV];
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const int jj = j + t * EPI + sub;
                pj[t] = -1;
                a[t] = 0.f;
                if (jj < cnt) {
                    const int2 h = hits[jj];
                    pj[t] = h.x;
                    a[t] = __int_as_float(h.y);
                }
            }
#pragma unroll
            for (int t = 0; t < UNR; ++t) {
                const float4* row = reinterpret_cast<const float4*>(D + (size_t)max(pj[t], 0) * ld);
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const int q = ql + LPR * k;
                    x[t][k] = (pj[t] >= 0 && q < nq) ? __ldg(row + q) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int t = 0; t < UNR; ++t)
#pragma unroll
                for (int k = 0; k < NV; ++k) add4(acc[k], x[t][k], a[t]);
        }
    }
    if (any) {
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
    return any;
}

// One warp per affected sink; a sink with a long in-list only queues (sink, chunk) work items.
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_scatter_gather(Ctl* ctl, int l, const int32_t* __restrict__ A, Side in, const int32_t* __restrict__ posmap,
                 const float* __restrict__ D, int ld, float* dS, int2* items) {
    pdl_enter();
    __shared__ int2 s_hits[8][GATHER_WINDOW];
    if (ctl->abort || !ctl->pull[l] || ctl->regather[l]) return;
    const int nA = ctl->nA[l];
    const int lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    int2* hits = s_hits[threadIdx.x >> 5];
    // sinks are handed out in runs of GATHER_TAKE by ticket: in-lists differ in length by orders of magnitude,
    // and the grid need not match the number of resident blocks
    for (;;) {
        int i0 = 0;
        if (lane == 0) i0 = atomicAdd(&ctl->gather_ticket[l], GATHER_TAKE);
        i0 = __shfl_sync(FULL, i0, 0);
        if (i0 >= nA) break;
    for (int i = i0; i < min(i0 + GATHER_TAKE, nA); ++i) {
        const int v = A[i];
        const int deg = in.deg[v];
        if (deg > GATHER_LONG) {
            const int nch = (deg + GATHER_ITEM - 1) / GATHER_ITEM;
            int first = 0;
            if (lane == 0) first = atomicAdd(&ctl->gather_items[l], nch);
            first = __shfl_sync(FULL, first, 0);
            for (int ch = lane; ch < nch; ch += 32) items[first + ch] = make_int2(v, ch);
            continue;
        }
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!gather_accumulate<NV, LPR>(acc, in, v, 0, deg, posmap, D, ld, hits)) continue;
        if (sub == 0) {
            // the accumulator is zero outside a batch and this is the hop's first kernel to touch the row
            // (edge records are added after it): a plain store
            float4* dst = reinterpret_cast<float4*>(dS + (size_t)v * ld);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const int q = ql + LPR * k;
                if (q < nq) dst[q] = acc[k];
            }
        }
    }
    }
}

// the chunks of the long in-lists: several warps add into the same accumulator row
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_scatter_gather_long(Ctl* ctl, int l, Side in, const int32_t* __restrict__ posmap, const float* __restrict__ D, int ld,
                      float* dS, const int2* __restrict__ items) {
    pdl_enter();
    __shared__ int2 s_hits[8][GATHER_WINDOW];
    if (ctl->abort || !ctl->pull[l] || ctl->regather[l]) return;
    const int n = ctl->gather_items[l];
    const int lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    int2* hits = s_hits[threadIdx.x >> 5];
    // items by ticket: they are equally long, but the senders among their entries are not equally many
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&ctl->gather_long_ticket[l], 1);
        it = __shfl_sync(FULL, it, 0);
        if (it >= n) break;
        const int2 w = items[it];
        const int deg = in.deg[w.x];
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!gather_accumulate<NV, LPR>(acc, in, w.x, w.y * GATHER_ITEM, min(deg, (w.y + 1) * GATHER_ITEM), posmap, D, ld,
                                        hits))
            continue;
        if (sub == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const int q = ql + LPR * k;
                if (q < nq) red_add_v4(dS + (size_t)w.x * ld + 4 * q, acc[k]);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// rebuilding hop (scoped recomputation of the aggregates, the "RC" strategy of Sec. 3.2 applied to
// one hop): S_v of every affected vertex is gathered again over In_new(v) from the current rows
// ---------------------------------------------------------------------------------------------
template <int NV, int LPR>
__global__ void __launch_bounds__(256)
k_regather(Ctl* ctl, int l, const int32_t* __restrict__ A, Side in, const int32_t* __restrict__ deg_out,
           int src_norm, const float* __restrict__ M, int ld, float* __restrict__ S, int2* items,
           int* n_items, float* budget) {
    pdl_enter();
    if (ctl->abort || !ctl->regather[l]) return;
    const int nA = ctl->nA[l];
    const int lane = lane_id(), nq = ld >> 2;
    const int sub = lane / LPR, ql = lane % LPR;
    // rows are handed out in runs of eight by ticket (the grid need not match the number of resident blocks)
    for (;;) {
        int i0 = 0;
        if (lane == 0) i0 = atomicAdd(&ctl->regather_ticket[l], 8);
        i0 = __shfl_sync(FULL, i0, 0);
        if (i0 >= nA) break;
    for (int i = i0; i < min(i0 + 8, nA); ++i) {
        const int v = A[i];
        const int deg = in.deg[v];
        float4 acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (deg > SPMM_HUB_DEGREE) {   // zero the row here, chunks are added by k_spmm_hubs
            const int nch = (deg + SPMM_HUB_CHUNK - 1) / SPMM_HUB_CHUNK;
            int first = 0;
            if (lane == 0) first = atomicAdd(n_items, nch);
            first = __shfl_sync(FULL, first, 0);
            for (int ch = lane; ch < nch; ch += 32) items[first + ch] = make_int2(v, ch);
        } else {
            spmm_accumulate<NV, LPR>(acc, in, v, 0, deg, deg_out, src_norm, M, ld);
        }
        if (sub == 0) {
            float4* dst = reinterpret_cast<float4*>(S + (size_t)v * ld);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int q = ql + LPR * k;
                if (q < nq) dst[q] = acc[k];
            }
        }
        if (budget && lane == 0) budget[v] = 0.f;   // a freshly gathered row has spent nothing
    }
    }
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
                float* budget, const int32_t* __restrict__ senders, int32_t* posmap, int mark, int self_term,
                const int32_t* __restrict__ A_prev, uint32_t* bitmap, int chores_only) {
    pdl_enter();
    // Two chores of the hop ride along with this kernel, the last of the hop's delta form, whatever form
    // the hop takes.  The hop's senders are no longer looked up by anyone: their entries of the position
    // map are cleared.  And (mark) the members of A_l that no out-list walk finds are marked: the sinks of
    // net edge changes, and A_{l-1} for models with a self term.
    {
        const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsize = gridDim.x * blockDim.x;
        const int nC = ctl->nC[l - 1];
        for (int i = gtid; i < nC; i += gsize) posmap[senders[i]] = -1;
        if (mark && !ctl->abort) {
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
// Delta form: the out-edges of the senders each carry one message, added to the sink's aggregate
// by a vector reduction (push), or gathered per sink over the senders among its in-neighbours
// (k_scatter_gather: chosen on the host, per hop, for wide messages from few senders; slower than
// the push for narrow rows because of the per-edge membership lookup).
//
// Rebuilding form: once the senders' out-edges are most of the graph, reading every in-edge of
// the affected sinks once and overwriting their aggregates costs less than one reduction per
// message: a gathered row is a plain load, a delivered message a read-modify-write in L2.  The
// rebuilt aggregate also sheds whatever rounding the deltas had left in it.  threshold = the
// share of all edges above which the hop rebuilds (<= 0: never).  With the default threshold a hop
// of fewer than min_messages messages pushes regardless: on a graph of a million edges neither
// form is throughput-bound, and the edge-balanced push is the more parallel of the two (measured
// on the sparse graph, 256 floats per row: 0.24 ms pushed, 0.26 to 0.47 ms rebuilt).
__global__ void k_choose_direction(Ctl* ctl, int l, int mode, int gather, float threshold, long long min_messages) {
    pdl_enter();
    const int nC = ctl->nC[l - 1];
    int re = 0;
    if (mode == RIPPLE_SCATTER_REGATHER) re = 1;
    else if (mode == RIPPLE_SCATTER_AUTO && threshold > 0.f) {
        const unsigned long long msgs = ctl->E[l] + (unsigned long long)ctl->n_rec;
        re = (double)msgs >= (double)threshold * (double)ctl->num_edges && ctl->num_edges > 0 &&
             msgs >= (unsigned long long)min_messages;
    }
    if (nC == 0 && ctl->n_rec == 0) re = 0;
    ctl->pull[l] = gather;
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
    if (!c->rebuild_armed[l] && !c->pull_hop[l] &&
        (c->scatter_mode == RIPPLE_SCATTER_AUTO || c->scatter_mode == RIPPLE_SCATTER_PUSH ||
         c->scatter_mode == RIPPLE_SCATTER_PUSH_BULK)) return;
    RP_LAUNCH(c, k_choose_direction, 1, 1, 0, c->ctl, l, c->scatter_mode, (int)c->pull_hop[l],
              c->rebuild_armed[l] ? c->regather_threshold[l] : -1.f, c->regather_min_messages);
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
#define PUSH(NV, LPR) RP_LAUNCH(c, (k_scatter_push<NV, LPR>), grid, T, 0, c->ctl, l, senders, c->coff, c->side[0], Dm, ld, c->dS[l], c->bitmap, recs, c->N)
    int2* gather_items = c->items;
    const RecMsgs recs{c->rec, (int)c->src_norm, c->side[0].deg, c->posmap, Mrows};
    bool recs_done = false;
#define PULL(NV, LPR)                                                                                                  \
    do {                                                                                                               \
        RP_LAUNCH(c, (k_scatter_gather<NV, LPR>), grid, T, 0, c->ctl, l, c->A[l], c->side[1], c->posmap, Dm, ld,      \
                  c->dS[l], gather_items);                                                                             \
        RP_LAUNCH(c, (k_scatter_gather_long<NV, LPR>), grid, T, 0, c->ctl, l, c->side[1], c->posmap, Dm, ld, c->dS[l], \
                  (const int2*)gather_items);                                                                          \
    } while (0)
    // (rows too wide for two staging buffers per warp in the default shared-memory allowance take the ordinary form)
    if (c->scatter_mode == RIPPLE_SCATTER_PUSH_BULK && !c->weighted && (size_t)8 * 2 * ld * sizeof(float) <= (48u << 10)) {
        RP_LAUNCH(c, k_scatter_push_bulk, grid, T, (size_t)8 * 2 * ld * sizeof(float), c->ctl, l, senders, c->coff,
                  c->side[0], Dm, ld, c->dS[l], c->bitmap);
    } else if (!c->pull_hop[l] && c->scatter_mode != RIPPLE_SCATTER_REGATHER) {
#define PACKED(NQ, WGT) RP_LAUNCH(c, (k_scatter_push_packed<NQ, WGT>), grid, T, 0, c->ctl, l, senders, c->coff, c->side[0], Dm, c->dS[l], c->bitmap, recs, c->N)
        if (ld == 48 && c->weighted) PACKED(12, true);
        else if (ld == 48) PACKED(12, false);
        else if (ld == 40 && c->weighted) PACKED(10, true);
        else if (ld == 40) PACKED(10, false);
#undef PACKED
        else RP_WIDTH_DISPATCH(ld, PUSH);
        recs_done = true;
    }
    if (c->pull_hop[l]) RP_WIDTH_DISPATCH(ld, PULL);
#undef PUSH
#undef PULL
    if (c->timing) cudaEventRecord(c->ev_sc[2 * l + 1], c->stream);
    if (n > 0) {
        if (!recs_done)
            RP_LAUNCH(c, k_scatter_records, std::min(div_up(n, T / 32), c->n_sm * 8), T, 0, c->ctl, l, recs, Dm, ld, c->dS[l]);
        const float* rows = c->pre[l] ? c->P[l] : c->H[l - 1];
#define ROWS(NV, LPR) RP_LAUNCH(c, (k_regather_rows<NV, LPR>), std::min(div_up(n, T / 32), c->n_sm * 8), T, 0, c->ctl, l, c->rec, c->side[1], c->side[0].deg, (int)c->src_norm, rows, ld, c->S[l], c->dS[l], c->Eb[l], senders, c->posmap, (int)(!c->pull_hop[l]), (int)c->self_term, c->A[l - 1], c->bitmap, (int)(c->n_local > 0))
        RP_WIDTH_DISPATCH(ld, ROWS);
#undef ROWS
    }
}

// rebuilding form of hop l (does nothing on the device unless the hop rebuilds); needs the list A_l
void regather_layer(Ctx* c, int l) {
    if (!c->rebuild_armed[l]) return;
    const int ld = c->ws[l];
    const float* M = c->pre[l] ? c->P[l] : c->H[l - 1];   // P^l rows of the senders are already current
    const int grid = c->n_sm * 16, T = 256;
    int2* items = c->items;
    int* n_items = &c->ctl->work_counter[(l - 1) & 7];
    if (c->timing) cudaEventRecord(c->ev_rg[2 * l], c->stream);
#define REGATHER(NV, LPR)                                                                                          \
    do {                                                                                                           \
        RP_LAUNCH(c, (k_regather<NV, LPR>), grid, T, 0, c->ctl, l, c->A[l], c->side[1], c->side[0].deg,           \
                  (int)c->src_norm, M, ld, c->S[l], items, n_items, c->Eb[l]);                                     \
        RP_LAUNCH(c, (k_spmm_hubs<NV, LPR>), grid, T, 0, c->side[1], c->side[0].deg, (int)c->src_norm, M, ld,     \
                  c->S[l], items, n_items, &c->ctl->hub_ticket[l]);                                                \
    } while (0)
    RP_WIDTH_DISPATCH(ld, REGATHER);
#undef REGATHER
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
