// Affected-row layer update (Compute + Prepare of Sec. 3.3.1): gather the inputs of Update^l for the
// rows of A_l, multiply by the layer weights, add bias, apply the activation, write h^l_v in
// place and emit the delta row D_v = c_new h_new - c_old h_old for the next hop (Sec. 3.3.3).
//
// Two forms of the same contraction, chosen on the device from the row count:
//   SIMT fp32    register-tiled GEMM whose A operand is gathered by row id (this file); used
//                while the affected set is too small to be a real dense contraction;
//   tensor core  tcgen05 TF32 with a 3-term split that keeps fp32 accuracy (layer_update_tc.cu).
// A launch takes one or two problems: the neighbour and the self projection of a layer's senders read the same rows.
#include "layer_update.cuh"

#include <algorithm>

namespace rp {

// K is walked in chunks of 64: every thread has eight independent 16-byte loads in flight per chunk
// (four pieces of a gathered A row, four of the weights).  With chunks of 16 a small frontier -- a
// handful of tiles, so nothing to overlap with -- paid one trip to L2 per 16 columns of K: 20 to 27 us
// for a few dozen rows, half of the latency of a batch of one update.
constexpr int BM = 64, BN = 64, BK = 64, TM = 4, TN = 4;

// A frontier of a few rows (a batch of a few updates at the first hops) is nothing but latency: the tiled form
// walks K in chunks, each a round trip to L2 behind the last, and gives the device a tile per 64 rows.  While all items of
// 16 rows and 32 output columns fit on the device at once the same kernel takes another route: a block stages the rows of
// its item in shared memory (256 entries of K at a time), its eight warps each take an eighth of them with every weight
// load independent of the others (one round trip in all), the partial sums meet in shared memory and the ordinary epilogue
// finishes the rows.  (Two projections of some 900 rows, K = 256, 40 columns: 31 -> 13 us; 20 rows, K = 602, 256
// columns: 49 -> 18.)
constexpr int FEW_ROWS = 16, FEW_K = 256, FEW_COLS = 32;

__device__ __forceinline__ int upd_few_items(const UpdParams& p, int n) {
    return ((p.n_cols + FEW_COLS - 1) / FEW_COLS) * ((n + FEW_ROWS - 1) / FEW_ROWS);
}

__device__ __forceinline__ bool upd_few(const UpdParams& p, int n) {
    return n > 0 && p.K > 0 && upd_few_items(p, n) <= (int)gridDim.x;
}

__device__ __forceinline__ void update_few_rows(const UpdParams& p, int n_all, int first, float* A_s, float* red, int* row_id,
                                                float* row_scale) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int groups = (p.n_cols + FEW_COLS - 1) / FEW_COLS, items = upd_few_items(p, n_all);
    for (int item = first; item < items; item += gridDim.x) {
        const int g = item % groups, r0 = (item / groups) * FEW_ROWS;
        const int n = min(FEW_ROWS, n_all - r0);   // rows of this block: compact indices r0 .. r0 + n - 1
        __syncthreads();
        if (tid < n) {
            const int v = p.list ? p.list[r0 + tid] : r0 + tid;
            row_id[tid] = v;
            row_scale[tid] = upd_row_scale(p, v);
        }
        const int c = g * FEW_COLS + lane;
        float acc[FEW_ROWS];
#pragma unroll
        for (int r = 0; r < FEW_ROWS; ++r) acc[r] = 0.f;
        for (int k0 = 0; k0 < p.K; k0 += FEW_K) {
            const int kn = min(FEW_K, p.K - k0), kq = kn >> 2;
            __syncthreads();
            for (int it = tid; it < n * kq; it += blockDim.x) {
                const int r = it / kq, k = 4 * (it - r * kq);
                *reinterpret_cast<float4*>(A_s + r * FEW_K + k) = upd_load_a(p, row_id[r], r0 + r, k0 + k, row_scale[r]);
            }
            __syncthreads();
            const int kper = (kn + 7) >> 3, k_begin = warp * kper, k_end = min(kn, k_begin + kper);
#pragma unroll 8
            for (int k = k_begin; k < k_end; ++k) {
                const float wv = c < p.n_cols ? __ldg(p.W + (size_t)(k0 + k) * p.ldw + c) : 0.f;
#pragma unroll
                for (int r = 0; r < FEW_ROWS; ++r)
                    if (r < n) acc[r] = fmaf(A_s[r * FEW_K + k], wv, acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < FEW_ROWS; ++r) red[(warp * FEW_ROWS + r) * FEW_COLS + lane] = acc[r];
        __syncthreads();
        if (tid < n * (FEW_COLS / 4)) {
            const int r = tid / (FEW_COLS / 4), q = tid - r * (FEW_COLS / 4), col = g * FEW_COLS + 4 * q;
            if (col < p.n_cols) {
                float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int w = 0; w < 8; ++w) {
                    const float4 x = *reinterpret_cast<const float4*>(red + (w * FEW_ROWS + r) * FEW_COLS + 4 * q);
                    h.x += x.x; h.y += x.y; h.z += x.z; h.w += x.w;
                }
                upd_epilogue4(p, row_id[r], r0 + r, col, h, row_scale[r]);
            }
        }
    }
}

// FEW: the instantiation that small batches launch also holds the few-row form.  Large batches launch the one
// without it: with the few-row code inlined beside it the tiled form, unchanged in registers and shared memory,
// made a batch of 1000 updates on the dense graph 0.3 ms slower (1.65 -> 2.0 ms) once the kernels of the chain
// overlap their launches, and calling the few-row form out of line cost the small batches 10 us of the 30 it saves.
template <bool FEW>
__global__ void __launch_bounds__(256)
k_update_rows(const Ctl* ctl, const __grid_constant__ UpdPair pair) {
    pdl_enter();
    if (ctl->abort) return;
    __shared__ __align__(16) float As[BK][BM + 4];
    __shared__ __align__(16) float Bs[BK][BN];
    __shared__ int row_id[BM];
    __shared__ float row_scale[BM];
    int used = 0;   // work items of the problems before: the next one starts at the block after the last of them
    for (int pi = 0; pi < pair.n; ++pi) {
    const UpdParams& p = pair.p[pi];
    const int n = upd_rows(p);
    if (upd_use_tc(p, n) || upd_use_narrow(p, n)) continue;
    const int first = (int)((blockIdx.x + gridDim.x - (unsigned)used % gridDim.x) % gridDim.x);
    if (FEW && upd_few(p, n)) {
        static_assert(sizeof(As) >= sizeof(float) * FEW_ROWS * FEW_K && sizeof(Bs) >= sizeof(float) * 8 * FEW_ROWS * FEW_COLS,
                      "the few-row form borrows the tiles' shared memory");
        update_few_rows(p, n, first, &As[0][0], &Bs[0][0], row_id, row_scale);
        used += upd_few_items(p, n);
        continue;
    }
    const int row_tiles = (n + BM - 1) / BM, col_tiles = (p.n_cols + BN - 1) / BN;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    used += row_tiles * col_tiles;
    for (int tile = first; tile < row_tiles * col_tiles; tile += gridDim.x) {
        const int rt = tile / col_tiles, ct = tile - rt * col_tiles;
        const int r0 = rt * BM, c0 = ct * BN;
        __syncthreads();
        if (tid < BM) {
            int i = r0 + tid, v = -1;
            float sc = 0.f;
            if (i < n) {
                v = p.list ? p.list[i] : i;
                sc = upd_row_scale(p, v);
            }
            row_id[tid] = v;
            row_scale[tid] = sc;
        }
        __syncthreads();
        float acc[TM][TN];
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int b = 0; b < TN; ++b) acc[a][b] = 0.f;

        const int ar = tid >> 2, ak = (tid & 3) * 4;   // A tile: row ar, k offsets ak + 16 j .. + 3, j = 0..3
        const int bk = tid >> 4, bn = (tid & 15) * 4;  // B tile: k rows bk + 16 j, cols bn..bn+3
        for (int k0 = 0; k0 < p.K; k0 += BK) {
            float4 a[4], b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                a[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                const int v = row_id[ar], k = k0 + ak + 16 * j;
                if (v >= 0 && k < p.K) a[j] = upd_load_a(p, v, r0 + ar, k, row_scale[ar]);
                b[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                const int kb = k0 + bk + 16 * j;
                if (kb < p.K && c0 + bn < p.n_cols)
                    b[j] = __ldg(reinterpret_cast<const float4*>(p.W + (size_t)kb * p.ldw + c0 + bn));
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                As[ak + 16 * j + 0][ar] = a[j].x; As[ak + 16 * j + 1][ar] = a[j].y;
                As[ak + 16 * j + 2][ar] = a[j].z; As[ak + 16 * j + 3][ar] = a[j].w;
                *reinterpret_cast<float4*>(&Bs[bk + 16 * j][bn]) = b[j];
            }
            __syncthreads();
            const int kmax = min(BK, p.K - k0);
#pragma unroll 16
            for (int k = 0; k < kmax; ++k) {
                float4 av = *reinterpret_cast<const float4*>(&As[k][ty * TM]);
                float4 bv = *reinterpret_cast<const float4*>(&Bs[k][tx * TN]);
                const float ar4[4] = {av.x, av.y, av.z, av.w};
                const float br4[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int a2 = 0; a2 < TM; ++a2)
#pragma unroll
                    for (int b2 = 0; b2 < TN; ++b2) acc[a2][b2] = fmaf(ar4[a2], br4[b2], acc[a2][b2]);
            }
        }
        const int col = c0 + tx * TN;
        if (col < p.n_cols) {
#pragma unroll
            for (int a2 = 0; a2 < TM; ++a2) {
                const int lr = ty * TM + a2, v = row_id[lr];
                if (v < 0) continue;
                upd_epilogue4(p, v, r0 + lr, col, make_float4(acc[a2][0], acc[a2][1], acc[a2][2], acc[a2][3]),
                              row_scale[lr]);
            }
        }
    }
    }
}

// Outputs of at most 48 columns over many rows (the last layers of the configurations: 47 and 40 classes, as the
// neighbour and the self projection of a million senders): the 64 x 64 tile above leaves a quarter of its threads
// multiplying zero columns, and it waits for every chunk of K before it multiplies it.  Here a tile is 256 rows x 48
// columns.  The gathered rows arrive through a ring of NST stages filled by cp.async, 16 entries of K per stage and
// row, NST - 1 chunks ahead of the one being multiplied and without passing through registers.  A warp owns six
// columns (its loads of the weights are uniform: one broadcast), a lane the eight rows ty, ty + 32, ...; it reads
// four entries of K per row with one 16-byte load (rows are 20 floats apart in a stage, so the loads of eight
// consecutive lanes fall into eight different 16-byte bank groups).  The factor on the A operand is per row: it is
// applied to the finished sums.  The finished tile goes through shared memory once more so that the epilogue sees
// 16-byte pieces of rows.  One source per A entry: the operand alpha h + scale S of GIN layers stays with the tiled form.
constexpr int NBM = 256, NBN = 48, NBK = 16, NTM = 8, NTN = 6, NST = 4, NARROW_MIN_ROWS = 65536;
constexpr int NAS_LD = NBK + 4, NCS_LD = NBN + 4;
constexpr size_t NARROW_SMEM = sizeof(float) * ((size_t)NST * NBM * NAS_LD + 2 * NBK * NBN + 2 * NBM) + sizeof(int) * NBM;
static_assert(NST * NBM * NAS_LD >= (NBM / 2) * NCS_LD, "the finished half tile is staged in the ring");

__device__ __forceinline__ void cp_async16_zfill(float* smem_dst, const float* gptr, bool valid) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem_dst);
    const int bytes = valid ? 16 : 0;      // (0: sixteen zero bytes are written, nothing is read)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(gptr), "r"(bytes) : "memory");
}

__global__ void __launch_bounds__(256, 2)
k_update_rows_narrow(const Ctl* ctl, UpdParams p) {
    pdl_enter();
    if (ctl->abort) return;
    extern __shared__ __align__(16) float nsm[];
    float* ring = nsm;                                   // [NST][NBM][NAS_LD], later the finished tile, half at a time
    float* Bs = ring + (size_t)NST * NBM * NAS_LD;       // [2][NBK][NBN]
    float* row_scale = Bs + 2 * NBK * NBN;               // [NBM]
    float* row_fac = row_scale + NBM;                    // [NBM]
    int* row_id = reinterpret_cast<int*>(row_fac + NBM); // [NBM]
    const int n = upd_rows(p);
    if (!upd_use_narrow(p, n)) return;
    const int row_tiles = (n + NBM - 1) / NBM, chunks = (p.K + NBK - 1) / NBK;
    const int tid = threadIdx.x, tx = tid >> 5, ty = tid & 31;
    for (int rt = blockIdx.x; rt < row_tiles; rt += gridDim.x) {
        const int r0 = rt * NBM;
        __syncthreads();
        {
            const int i = r0 + tid;
            int v = -1;
            float sc = 0.f;
            if (i < n) {
                v = p.list ? p.list[i] : i;
                sc = upd_row_scale(p, v);
            }
            row_id[tid] = v;
            row_scale[tid] = sc;
            row_fac[tid] = p.a_mode == A_DENSE ? 1.0f : p.a_mode == A_SELF ? p.alpha : sc;
        }
        __syncthreads();
        float acc[NTM][NTN];
#pragma unroll
        for (int a2 = 0; a2 < NTM; ++a2)
#pragma unroll
            for (int b2 = 0; b2 < NTN; ++b2) acc[a2][b2] = 0.f;
        // this thread's part of a chunk of A: rows ar + 64 s, entries ak .. ak + 3 of the chunk
        const int ar = tid >> 2, ak = (tid & 3) * 4;
        const float* src[4];
#pragma unroll
        for (int s2 = 0; s2 < 4; ++s2) {
            const int r = ar + 64 * s2, v = row_id[r];
            src[s2] = nullptr;
            if (v >= 0) {
                if (p.a_mode == A_DENSE) src[s2] = p.Hprev + (size_t)(r0 + r) * p.ld_h;
                else if (p.a_mode == A_SELF) src[s2] = p.Hprev + (size_t)v * p.ld_h;
                else src[s2] = p.S + (size_t)v * p.ld_s;
            }
        }
        auto request = [&](int c) {      // chunk c of A into its stage (beyond K: an empty group keeps the count)
            if (c < chunks) {
                float* stage = ring + (size_t)(c % NST) * NBM * NAS_LD;
                const int k = c * NBK + ak;
#pragma unroll
                for (int s2 = 0; s2 < 4; ++s2) {
                    const bool ok = src[s2] && k < p.K;
                    cp_async16_zfill(stage + (ar + 64 * s2) * NAS_LD + ak, ok ? src[s2] + k : p.W, ok);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // this thread's piece of a chunk of the weights (192 threads): row bk of the chunk, columns 4 bq .. 4 bq + 3
        const int bk = tid / (NBN / 4), bq = tid - bk * (NBN / 4);
        auto load_b = [&](int c) {
            float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
            if (bk < NBK && c * NBK + bk < p.K && 4 * bq < p.n_cols)
                b = __ldg(reinterpret_cast<const float4*>(p.W + (size_t)(c * NBK + bk) * p.ldw + 4 * bq));
            return b;
        };
#pragma unroll
        for (int c = 0; c < NST - 1; ++c) request(c);
        float4 b = load_b(0);
        for (int c = 0; c < chunks; ++c) {
            float* Bc = Bs + (c & 1) * NBK * NBN;
            if (bk < NBK) *reinterpret_cast<float4*>(Bc + bk * NBN + 4 * bq) = b;
            asm volatile("cp.async.wait_group %0;" ::"n"(NST - 2) : "memory");   // this thread's pieces of chunk c are in
            __syncthreads();                  // everyone's are, the weights too; and chunk c - 1 has been multiplied
            request(c + NST - 1);             // into the stage that chunk c - 1 has left
            b = load_b(c + 1);
            const float* stage = ring + (size_t)(c % NST) * NBM * NAS_LD;
            const int kmax = min(NBK, p.K - c * NBK);      // a multiple of four
            for (int k = 0; k < kmax; k += 4) {
                float4 av[NTM];
#pragma unroll
                for (int a2 = 0; a2 < NTM; ++a2)
                    av[a2] = *reinterpret_cast<const float4*>(stage + (a2 * 32 + ty) * NAS_LD + k);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const float2 w0 = *reinterpret_cast<const float2*>(Bc + (k + kk) * NBN + tx * NTN);
                    const float2 w1 = *reinterpret_cast<const float2*>(Bc + (k + kk) * NBN + tx * NTN + 2);
                    const float2 w2 = *reinterpret_cast<const float2*>(Bc + (k + kk) * NBN + tx * NTN + 4);
                    const float bv[NTN] = {w0.x, w0.y, w1.x, w1.y, w2.x, w2.y};
#pragma unroll
                    for (int a2 = 0; a2 < NTM; ++a2) {
                        const float x = kk == 0 ? av[a2].x : kk == 1 ? av[a2].y : kk == 2 ? av[a2].z : av[a2].w;
#pragma unroll
                        for (int b2 = 0; b2 < NTN; ++b2) acc[a2][b2] = fmaf(x, bv[b2], acc[a2][b2]);
                    }
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // the finished tile, 128 rows at a time, through shared memory to the epilogue
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            __syncthreads();
#pragma unroll
            for (int a2 = 0; a2 < NTM / 2; ++a2) {
                const int r = (half * (NTM / 2) + a2) * 32 + ty;
                const float f = row_fac[r];
#pragma unroll
                for (int b2 = 0; b2 < NTN; ++b2)
                    ring[(a2 * 32 + ty) * NCS_LD + tx * NTN + b2] = f * acc[half * (NTM / 2) + a2][b2];
            }
            __syncthreads();
            for (int it = tid; it < (NBM / 2) * (NBN / 4); it += 256) {
                const int lr = it / (NBN / 4), q = it - lr * (NBN / 4);
                const int r = half * (NBM / 2) + lr, v = row_id[r];
                if (v < 0 || 4 * q >= p.n_cols) continue;
                const float4 h = *reinterpret_cast<const float4*>(&ring[lr * NCS_LD + 4 * q]);
                upd_epilogue4(p, v, r0 + r, 4 * q, h, row_scale[r]);
            }
        }
    }
}

void narrow_prepare() {
    cudaFuncSetAttribute(k_update_rows_narrow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NARROW_SMEM);
}

// K = 0: the layer's self projection and transformed aggregate are both cached, so the update is elementwise (bias +
// cached terms + activation).  HBM bound: per row of d floats it reads S, its pending sums and Z and writes S, zeros and h
// (24 d bytes; 12 d where the aggregate was gathered anew and nothing is pending).  A thread takes one 16-byte piece of a
// row, two pieces per round with all their loads asked for before either is used; pieces are numbered through the rows,
// so that any width keeps every lane busy.
constexpr int EW_U = 2, EW_ROUNDS = 4;

__global__ void __launch_bounds__(256)
k_update_rows_elementwise(const Ctl* ctl, const __grid_constant__ UpdParams p) {
    pdl_enter();
    if (ctl->abort) return;
    const unsigned n = (unsigned)upd_rows(p), nq = (unsigned)p.n_cols >> 2, inv = 0xffffffffu / nq + 1u;   // x / nq = umulhi(x, inv), x small
    const bool fold = p.addend_rw && !(p.rebuilt && *p.rebuilt);
    const float* const srows = p.addend_rw ? p.addend_rw : p.addend;
    // Runs of pieces by ticket: with a fixed stride from run to run a block kept meeting the same memory channels, and the
    // slowest block took half as long again as the fastest (1.15 M rows of 256 floats: 1.41 -> 1.06 ms).
    constexpr unsigned RUN = 256 * EW_U * EW_ROUNDS;
    __shared__ unsigned s_run;
    unsigned next = 0;
    if (threadIdx.x == 0) next = (unsigned)atomicAdd(p.ticket, 1);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) { s_run = next; next = (unsigned)atomicAdd(p.ticket, 1); }
        __syncthreads();
        const unsigned long long first = (unsigned long long)s_run * RUN;
        unsigned row0 = (unsigned)(first / nq);
        const unsigned rem_first = (unsigned)(first - (unsigned long long)row0 * nq);
        if (row0 >= n) break;
#pragma unroll 1
        for (int round = 0; round < EW_ROUNDS; ++round) {
        const unsigned rem0 = rem_first + 256u * EW_U * (unsigned)round;
        unsigned i[EW_U], col[EW_U];
        int v[EW_U];
        bool on[EW_U];
#pragma unroll
        for (int u = 0; u < EW_U; ++u) {
            const unsigned off = rem0 + 256u * u + threadIdx.x, dr = nq == 1 ? off : __umulhi(off, inv);
            i[u] = row0 + dr;
            col[u] = 4u * (off - dr * nq);
            on[u] = i[u] < n;
            v[u] = on[u] ? (p.list ? p.list[i[u]] : (int)i[u]) : 0;
        }
        float sc[EW_U];
        float4 s[EW_U], d[EW_U], z[EW_U], o[EW_U];
#pragma unroll
        for (int u = 0; u < EW_U; ++u) {
            // (pieces beyond the last read row 0 and are dropped)
            s[u] = d[u] = z[u] = o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            sc[u] = upd_row_scale(p, v[u]);
            const size_t at = (size_t)v[u] * p.ld_add + col[u];
            if (srows) s[u] = *reinterpret_cast<const float4*>(srows + at);
            if (fold) d[u] = *reinterpret_cast<const float4*>(p.addend_delta + at);
            if (p.addend2) z[u] = *reinterpret_cast<const float4*>(p.addend2 + at);
            if (p.Dout) o[u] = upd_load_old(p, v[u], col[u]);
        }
#pragma unroll
        for (int u = 0; u < EW_U; ++u) {
            if (!on[u]) continue;
            const size_t at = (size_t)v[u] * p.ld_add + col[u];
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p.bias) h = __ldg(reinterpret_cast<const float4*>(p.bias + col[u]));
            if (fold) {
                s[u].x += d[u].x; s[u].y += d[u].y; s[u].z += d[u].z; s[u].w += d[u].w;
                *reinterpret_cast<float4*>(p.addend_rw + at) = s[u];
                *reinterpret_cast<float4*>(p.addend_delta + at) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            h.x += sc[u] * s[u].x; h.y += sc[u] * s[u].y; h.z += sc[u] * s[u].z; h.w += sc[u] * s[u].w;
            h.x += z[u].x; h.y += z[u].y; h.z += z[u].z; h.w += z[u].w;
            if (p.act == RIPPLE_ACT_RELU) {
                h.x = fmaxf(h.x, 0.f); h.y = fmaxf(h.y, 0.f); h.z = fmaxf(h.z, 0.f); h.w = fmaxf(h.w, 0.f);
            }
            if (p.Dout) {
                float cn = 1.f, co = 1.f;
                if (p.src_norm) {
                    const int dold = p.deg_out_old[v[u]];
                    cn = coef_deg(p.deg_out[v[u]]);
                    co = dold >= 0 ? coef_deg(dold) : cn;
                }
                *reinterpret_cast<float4*>(p.Dout + (size_t)i[u] * p.ld_o + col[u]) =
                    p.dout_old ? o[u] : make_float4(cn * h.x - co * o[u].x, cn * h.y - co * o[u].y, cn * h.z - co * o[u].z, cn * h.w - co * o[u].w);
            }
            *reinterpret_cast<float4*>(p.Hout + (size_t)v[u] * p.ld_o + col[u]) = h;
        }
        }
    }
}

// Launches every form that the row counts can call for; exactly one of them does the work of each problem (decided on
// the device).
// `over`: the hop whose list (A_over or C_over) the rows come from.
// `both`: the weights of two problems over the same rows, side by side.
static void launch_update(Ctx* c, UpdPair& u, int over, const TcW* const (&tw)[2], const TcW* both = nullptr) {
    if (u.p[0].K == 0) {
        RP_LAUNCH(c, k_update_rows_elementwise, RP_RESIDENT(c, k_update_rows_elementwise, 256), 256, 0, c->ctl, u.p[0]);
        return;
    }
    UpdPair tc{};      // the problems that have a tensor-core twin
    bool apart = false;   // narrow ones: each alone, unless their weights lie side by side
    for (int i = 0; i < u.n; ++i) {
        UpdParams& p = u.p[i];
        p.tc_mode = TC_OFF;
        p.narrow_min_rows = 0;
        // The forms for many rows are only put into the chain when the last batch's frontiers (or a whole-graph pass)
        // were large enough for them; without them the tiled SIMT form takes whatever comes.
        if (!c->tc_armed[over] && p.list) continue;
        if (tw[i]->w && !(tw[i]->pieces && p.a_mode == A_SUM) && c->gemm_mode != RIPPLE_GEMM_FP32) {
            p.tc_mode = c->gemm_mode == RIPPLE_GEMM_TF32 && !tw[i]->pieces ? TC_TF32 : TC_TF32X3;
            p.tc_min_rows = RP_TC_MIN_ROWS;
            p.tc_withhold = c->debug_tc_withhold;
            p.tc_w = tw[i]->w; p.tc_groups = tw[i]->groups; p.tc_chunks = tw[i]->chunks;
            tc.p[tc.n++] = p;
            apart |= tw[i]->pieces;
        } else if (p.n_cols <= NBN && p.a_mode != A_SUM) {
            // narrow outputs over many rows have a form of their own
            p.narrow_min_rows = NARROW_MIN_ROWS;
        }
    }
    if (c->few_rows_form && u.p[0].list) RP_LAUNCH(c, k_update_rows<true>, c->n_sm * 4, 256, 0, c->ctl, u);
    else if (u.p[0].list || tc.n < u.n || c->N < RP_TC_MIN_ROWS) RP_LAUNCH(c, k_update_rows<false>, c->n_sm * 4, 256, 0, c->ctl, u);
    for (int i = 0; i < u.n; ++i)
        if (u.p[i].narrow_min_rows) RP_LAUNCH(c, k_update_rows_narrow, c->n_sm * 2, 256, NARROW_SMEM, c->ctl, u.p[i]);
    if (tc.n == 2 && apart && both && both->w && tc.p[0].list == tc.p[1].list) tc.p[0].tc_w = both->w;
    else if (tc.n == 2 && apart) {
        UpdPair second{};
        second.p[second.n++] = tc.p[1];
        tc.n = 1;
        launch_update_tc(c, second, true);
    }
    if (tc.n) launch_update_tc(c, tc, apart);
}

static void launch_update(Ctx* c, const UpdParams& p, int over, const TcW& tw) {
    UpdPair u{};
    u.p[0] = p;
    u.n = 1;
    launch_update(c, u, over, {&tw, &tw});
}

// P^l_u = W_n^T h^{l-1}_u (all rows if `full`)
static UpdParams neighbour_problem(Ctx* c, int l, bool full) {
    const LayerDev& ly = c->layer[l];
    UpdParams p{};
    p.list = full ? nullptr : sender_list(c, l - 1);
    p.n_dev = full ? nullptr : &c->ctl->nC[l - 1];
    p.n_host = c->N;
    p.a_mode = A_SELF; p.epi_mode = EPI_COMMIT; p.alpha = 1.0f;
    p.Hprev = c->H[l - 1]; p.ld_h = c->ld[l - 1];
    p.K = ly.ld_in;
    p.W = ly.kind == RIPPLE_LAYER_SAGE ? ly.W1 + (size_t)ly.ld_in * ly.ld_out : ly.W1;
    p.ldw = c->ws[l]; p.bias = nullptr; p.n_cols = c->ws[l];
    p.act = RIPPLE_ACT_IDENTITY; p.Hout = c->P[l]; p.ld_o = c->ws[l];
    p.src_norm = c->src_norm; p.deg_out = c->side[0].deg; p.deg_out_old = c->deg_out_old;
    return p;
}

// Z^l_v = W_self^T h^{l-1}_v for the rows whose h^{l-1} changed (all rows at bootstrap).  SAGE
// layers keep this self projection cached: it is recomputed where the layer's input changed
// (A_{l-1}), not where its output is needed (A_l, usually far larger).  The affected-row update
// then contracts over the aggregate only (half the K of [h || x]); for a layer that also
// transforms before the scatter nothing is left to contract.
static UpdParams self_problem(Ctx* c, int l, bool full) {
    const LayerDev& ly = c->layer[l];
    UpdParams p{};
    p.list = full ? nullptr : c->A[l - 1];
    p.n_dev = full ? nullptr : &c->ctl->nA[l - 1];
    p.n_host = c->N;
    p.a_mode = A_SELF; p.epi_mode = EPI_COMMIT; p.alpha = 1.0f;
    p.Hprev = c->H[l - 1]; p.ld_h = c->ld[l - 1];
    p.K = ly.ld_in; p.W = ly.W1; p.ldw = ly.ld_out; p.n_cols = ly.ld_out;
    p.act = RIPPLE_ACT_IDENTITY; p.Hout = c->Z[l]; p.ld_o = ly.ld_out;
    return p;
}

static void project(Ctx* c, int l, const UpdParams& nbr, bool full) {
    const LayerDev& ly = c->layer[l];
    UpdPair u{};
    u.p[0] = nbr;
    u.n = 1;
    if (c->Z[l]) u.p[u.n++] = self_problem(c, l, full);   // the same rows: one launch for both products
    launch_update(c, u, l - 1, {&ly.tc_nbr, &ly.tc_self}, &ly.tc_both);
}

void project_full(Ctx* c, int l) { project(c, l, neighbour_problem(c, l, true), true); }

// Layers that transform before the scatter keep P^l_u = W_n^T h^{l-1}_u for every vertex.  For the
// senders of hop l (rows whose h^{l-1}, or whose source coefficient, changed) this recomputes the
// row, commits it and emits the transformed delta message c_new P_new - c_old P_old as a compact
// row.  Because the next batch subtracts exactly the value cached here, the deltas of successive
// batches telescope: the aggregate tracks the cached rows without a rounding drift of its own.
// The senders' self projections (their rows are those of A_{l-1}) are computed along with them.
void sender_transform(Ctx* c, int l) {
    UpdParams p = neighbour_problem(c, l, false);
    p.Dout = c->Dt;
    project(c, l, p, false);
}

void self_project(Ctx* c, int l, bool full) {
    if (!c->Z[l] || c->pre[l]) return;   // (a layer that transforms first has done it with the neighbour projection)
    launch_update(c, self_problem(c, l, full), l - 1, c->layer[l].tc_self);
}

void update_rows(Ctx* c, int l, bool full) {
    const LayerDev& ly = c->layer[l];
    const bool pre = c->pre[l];
    UpdParams p{};
    p.list = full ? nullptr : c->A[l];
    p.n_dev = full ? nullptr : &c->ctl->nA[l];
    p.n_host = c->N;
    p.ticket = &c->ctl->ew_ticket[l];
    p.Hprev = c->H[l - 1]; p.ld_h = c->ld[l - 1];
    p.S = c->S[l]; p.ld_s = c->ws[l];
    p.alpha = 1.0f;
    p.agg = c->agg;
    p.deg_in = c->side[1].deg;
    p.src_norm = c->src_norm;
    p.deg_out = c->side[0].deg;
    p.deg_out_old = c->deg_out_old;
    if (pre) {
        p.addend = c->S[l]; p.ld_add = c->ws[l];
        if (!full && c->fused_fold[l]) { p.addend_rw = c->S[l]; p.addend_delta = c->dS[l]; p.rebuilt = &c->ctl->regather[l]; }   // fold_deltas is skipped for these layers
    }
    // the last hop sends nothing, and a layer that transforms first makes its messages from the projections it keeps
    // (P_new - P_old): it never looks at delta rows, nor does anyone need the row's previous value then
    float* dout = (full || l == c->L || c->pre[l + 1]) ? nullptr : c->D[l & 1];
    p.dout_old = rp_monotonic(c->agg);
    if (ly.kind == RIPPLE_LAYER_GIN) {
        // hidden = relu(W1^T ((1 + eps) h + x) + b1), kept as compact rows
        p.a_mode = pre ? A_SELF : A_SUM; p.epi_mode = EPI_TEMP; p.alpha = 1.0f + ly.eps;
        p.K = ly.ld_in; p.W = ly.W1; p.ldw = ly.ld_hid; p.bias = ly.b1; p.n_cols = ly.ld_hid;
        p.act = RIPPLE_ACT_RELU; p.Hout = c->T; p.ld_o = ly.ld_hid; p.Dout = nullptr;
        launch_update(c, p, l, ly.tc_main);
        p.a_mode = A_DENSE; p.epi_mode = EPI_COMMIT; p.addend = nullptr; p.addend_rw = nullptr; p.addend_delta = nullptr;
        p.Hprev = c->T; p.ld_h = ly.ld_hid;
        p.K = ly.ld_hid; p.W = ly.W2; p.ldw = ly.ld_out; p.bias = ly.b2; p.n_cols = ly.ld_out;
        p.act = ly.act; p.Hout = c->H[l]; p.ld_o = ly.ld_out; p.Dout = dout;
        launch_update(c, p, l, ly.tc_2);
        return;
    }
    p.epi_mode = EPI_COMMIT;
    if (ly.kind == RIPPLE_LAYER_SAGE) {
        p.a_mode = A_AGG;
        p.K = pre ? 0 : ly.ld_in;       // transformed aggregate: nothing left to multiply
        p.addend2 = c->Z[l];            // cached W_self^T h_v
    } else {
        p.a_mode = A_AGG;
        p.K = pre ? 0 : ly.ld_in;   // transformed inbox: nothing left to multiply
    }
    p.W = ly.kind == RIPPLE_LAYER_SAGE ? ly.W1 + (size_t)ly.ld_in * ly.ld_out : ly.W1;   // neighbour matrix
    p.ldw = ly.ld_out; p.bias = ly.b1; p.n_cols = ly.ld_out;
    p.act = ly.act; p.Hout = c->H[l]; p.ld_o = ly.ld_out; p.Dout = dout;
    if (!pre) p.ld_add = ly.ld_out;   // leading dimension of the cached projection
    launch_update(c, p, l, ly.tc_main);
}

// ---------------------------------------------------------------------------------------------
// hop 0: feature replacement rows and their deltas; one warp per vertex of A_0
// ---------------------------------------------------------------------------------------------
__global__ void k_feature_rows(Ctl* ctl, const ripple_update* __restrict__ ups, const float* __restrict__ feat,
                               int d0, const int32_t* __restrict__ A0, const int32_t* __restrict__ feat_last,
                               int src_norm, const int32_t* __restrict__ deg_out,
                               const int32_t* __restrict__ deg_out_old, float* H0, int ld, float* D, int keep_old) {
    pdl_enter();
    if (ctl->abort) return;
    const int n = ctl->nA[0];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < n; i += nwarps) {
        const int v = A0[i];
        const ripple_update last = ups[feat_last[v]];
        // the last word on the row is either a payload row or the vertex's deletion (zeros)
        const float* src = last.op == RIPPLE_OP_SET_FEATURE ? feat + (size_t)last.v * d0 : nullptr;
        float cn = 1.f, co = 1.f;
        if (src_norm) {
            cn = coef_deg(deg_out[v]);
            co = deg_out_old[v] >= 0 ? coef_deg(deg_out_old[v]) : cn;
        }
        for (int k = lane_id(); k < ld; k += 32) {
            float x = (src && k < d0) ? src[k] : 0.f;
            if (D) {
                float o = H0[(size_t)v * ld + k];
                D[(size_t)i * ld + k] = keep_old ? o : cn * x - co * o;
            }
            H0[(size_t)v * ld + k] = x;
        }
    }
}

void feature_rows(Ctx* c, int n) {
    if (n <= 0) return;
    RP_LAUNCH(c, k_feature_rows, std::min(div_up(n, 8), c->n_sm * 8), 256, 0, c->ctl, c->ups_dev, c->feat_dev,
              c->d[0], c->A[0], c->feat_last, (int)c->src_norm, c->side[0].deg, c->deg_out_old, c->H[0],
              c->ld[0], c->pre[1] ? (float*)nullptr : c->D[0], (int)(rp_monotonic(c->agg) || c->attention));
}

// ---------------------------------------------------------------------------------------------
// senders whose row did not change but whose source coefficient did: D_u = (c_new - c_old) h_u
// ---------------------------------------------------------------------------------------------
__global__ void k_extra_senders(Ctl* ctl, int l, const Rec* __restrict__ rec, int32_t* senders,
                                int32_t* posmap, const int32_t* __restrict__ deg_out,
                                const float* __restrict__ H, int ld, float* D) {
    pdl_enter();
    if (ctl->abort) return;
    const int n = ctl->n_rec;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = warp; r < n; r += nwarps) {
        const Rec x = rec[r];
        if (!x.rep[0] || x.silent) continue;   // one record per distinct source (a no-compute copy names a remote one)
        if (posmap[x.u] >= 0) continue;    // already a sender: its delta came from the row update
        int idx = 0;
        if (lane_id() == 0) idx = atomicAdd(&ctl->nC[l], 1);
        idx = __shfl_sync(FULL, idx, 0);
        const float dc = coef_deg(deg_out[x.u]) - coef_deg(x.deg_out_old);
        if (D)
            for (int k = lane_id(); k < ld; k += 32) D[(size_t)idx * ld + k] = dc * H[(size_t)x.u * ld + k];
        if (lane_id() == 0) { senders[idx] = x.u; posmap[x.u] = idx; }
    }
}

void extra_sender_rows(Ctx* c, int l, int n) {
    RP_LAUNCH(c, k_extra_senders, std::min(div_up(n, 8), c->n_sm * 8), 256, 0, c->ctl, l, c->rec,
              c->Clist[l & 1], c->posmap, c->side[0].deg, c->H[l], c->ld[l], c->pre[l + 1] ? (float*)nullptr : c->D[l & 1]);
}

}  // namespace rp
