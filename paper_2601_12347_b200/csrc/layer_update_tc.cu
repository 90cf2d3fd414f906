// Tensor-core form of the affected-row layer update for sm_100a: tcgen05.mma (kind::tf32) with
// the accumulator tile in tensor memory.
//
// One persistent CTA per SM takes tiles of 128 affected rows x one group of at most 128 output columns.  The product is
// formed transposed, weights times rows: the 128 lanes of the accumulator are output columns and its R columns are
// affected rows, so that a warp reading it back holds 32 consecutive columns of one row per register -- whole lines
// of the row's embedding, cached projection and delta, with no turn through shared memory.
//
// Per 32-float K chunk the loader warps gather the rows by vertex id with asynchronous copies straight into shared
// memory, in the K-major 128-byte-swizzle layout the tensor core reads.  The tensor core takes the upper 19 bits of an
// fp32 entry x (its tf32 part, hi); the loaders read the landed pieces back and store lo = x - hi, exact in fp32, as a
// second operand.  The transposed weights lie in global memory already split, swizzled and cut into chunks, so that a
// chunk is one bulk copy.  One thread issues, per 8-float K step, the weights' hi times [hi | lo] of the rows (256 columns)
// and the weights' lo times the rows' hi: all but the product of the two low parts (2^-22 relative).  The small products
// gather in accumulator columns of their own and meet the large ones in the epilogue: the tensor core rounds every
// addition towards zero, and of a sum of 96 terms (K = 256) only 32 are then added at full size.
// Error against fp64, 2-norm, 116 to 256 columns alike: 2.1e-7 at K = 32, 3.6e-7 at 100, 7e-7 at 256, 1.5e-6 at 602; GIN's
// two products of 256 x 256 1.3e-6 (one accumulator for all of it: 6.8e-7, 1.2e-6, 2.4e-6, 5e-6; 4.4e-6; fp32 sums on SIMT: 1.1e-7,
// 1.8e-7, 2.9e-7, 4.4e-7; 3.5e-7).  With tc_mode = TC_TF32 only hi * hi is issued (plain TF32, 2^-10).  Row factors (sink
// normalisation, GIN's self factor) are applied to the finished sums.
// Accumulators are double-buffered in tensor memory: the epilogue warps finish a tile (bias / cached terms /
// activation / delta / commit) while the next tile's main loop is already running.
//
// What bounds it and why it is cut this way.  Each of the three pipelines -- gather and split, products, epilogue -- needs
// about a microsecond per step whatever the bandwidth, so they overlap and each is kept free of chains: sixteen loader
// warps with three stages of rows where the weights stream, eight with two where they stay, one warp that does nothing but
// issue (its operands in uniform registers), one that fetches weights, eight epilogue warps whose loads travel ahead and
// whose stores are predicated.  The weights of a group stay in shared memory for the life of the CTA while they fit
// (K <= 128: 128 KB); beyond that they stream from L2 with every chunk.  Groups of one row tile run on neighbouring CTAs
// at the same time and find each other's rows in L2.
// Measured on 600 K rows (self and aggregate product of a layer, K = 100, 256 columns each: 1.18 -> 0.67 ms; GIN's two
// products of 256 x 256: 2.02 -> 0.97 ms).
//
// Every wait is bounded: if an mbarrier does not complete within the spin limit the CTA records
// RIPPLE_ERR_TIMEOUT in the control block, waits (again bounded) for its own copies and products in flight, frees its
// tensor memory and returns.
#include "layer_update.cuh"

#include <algorithm>
#include <cstring>
#include <vector>

namespace rp {

constexpr int TC_COLS = 128;     // output columns per group (= TMEM lanes)
constexpr int TC_KC = 32;        // floats per K chunk: one 128-byte swizzle row
constexpr int TC_TILE = 128;     // affected rows per tile
// Loader threads: sixteen warps where the weights stream, eight where they stay (whose epilogue, with a cached projection
// to read for every row, needs the registers more).
__host__ __device__ constexpr int tc_loaders(bool resident, bool pieces) { return pieces ? 128 : resident ? 256 : 512; }
constexpr int TC_EPI_WARPS = 8;  // two per tensor-memory lane quarter, half of the tile's rows each
__host__ __device__ constexpr int tc_threads(bool resident, bool pieces) { return tc_loaders(resident, pieces) + 32 * TC_EPI_WARPS + 64; }   // and the warps that issue and that fetch the weights
constexpr int TC_W_HALF = TC_COLS * 128;         // one half (hi or lo) of a chunk of weights
constexpr int TC_W_BYTES = 2 * TC_W_HALF;
constexpr int TC_RESIDENT_CHUNKS = 4;            // weights of up to this many chunks stay in shared memory
// What fits into 227 KB: stages of rows ([hi | lo], 32 KB each), weights, and the epilogue's rows in flight (32 KB).
constexpr int TC_W_STAGES = 3;                   // stages of weights that stream
__host__ __device__ constexpr int tc_stages(bool resident) { return resident ? 2 : 3; }
constexpr int TC_AHEAD = 2;                      // blocks of 16 rows an epilogue warp reads ahead
constexpr uint32_t TC_SPIN_LIMIT = 1u << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// true once the phase with the given parity has completed; gives up after `limit` polls
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t limit) {
    const uint32_t addr = smem_u32(bar);
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// a predicated store: as a branch of its own per row the epilogue's sixteen stores took 110 cycles each
__device__ __forceinline__ void tc_store_if(bool on, float* to, float x) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p st.global.f32 [%0], %1;\n\t}" ::"l"(to), "f"(x), "r"((int)on) : "memory");
}

// true in one lane of the (converged) warp
__device__ __forceinline__ bool tc_elect() {
    uint32_t one;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
    return one != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;             // leading byte offset (not used by swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;   // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;             // descriptor version
    d |= (uint64_t)2 << 61;             // SWIZZLE_128B
    return d;
}

__device__ __forceinline__ void tc_mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

__device__ __forceinline__ void tc_mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar)) : "memory");
}

// instruction descriptor: fp32 accumulate, tf32 x tf32 (type 2) or bf16 x bf16 (type 1), both K-major, N = rows, M = 128
__host__ __device__ constexpr uint32_t tc_idesc(int rows, uint32_t type = 2) {
    return (1u << 4) | (type << 7) | (type << 10) | ((uint32_t)(rows >> 3) << 17) | ((uint32_t)(TC_COLS >> 4) << 24);
}

// byte offset of 16-byte chunk c (0..7) of row r inside a K-major SWIZZLE_128B tile
__host__ __device__ __forceinline__ uint32_t tc_swz(int r, int c) {
    return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + (((c ^ r) & 7) << 4));
}

// what the tensor core reads of x
__device__ __forceinline__ float tf32_seen(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

__device__ __forceinline__ float4 tc_lds(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void tc_sts(uint32_t a, float4 v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

__device__ __forceinline__ void tc_sts2(uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

// x0 and x1 (in the upper half) as two parts in bf16, cut and rounded; both leave what the part lacks, exact in fp32.  (The
// first part is cut: rounded, entries near the largest would become infinite.)
__device__ __forceinline__ uint32_t bf16_left(float& x0, float& x1, uint32_t part) {
    x0 -= __uint_as_float(part << 16);
    x1 -= __uint_as_float(part & 0xffff0000u);
    return part;
}
__device__ __forceinline__ uint32_t bf16_cut(float& x0, float& x1) {
    uint32_t d;
    asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(x1), "f"(x0));
    return bf16_left(x0, x1, d);
}
__device__ __forceinline__ uint32_t bf16_round(float& x0, float& x1) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(x1), "f"(x0));
    return bf16_left(x0, x1, d);
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// one chunk of weights: a single bulk copy that completes on the barrier
__device__ __forceinline__ void tc_copy_weights(void* dst, const float* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tc_load16(uint32_t (&x)[16], uint32_t taddr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]),
          "=r"(x[7]), "=r"(x[8]), "=r"(x[9]), "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]),
          "=r"(x[14]), "=r"(x[15])
        : "r"(taddr) : "memory");
}

__device__ __forceinline__ void tc_load32(uint32_t (&x)[32], uint32_t taddr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]), "=r"(x[8]),
          "=r"(x[9]), "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]), "=r"(x[14]), "=r"(x[15]), "=r"(x[16]),
          "=r"(x[17]), "=r"(x[18]), "=r"(x[19]), "=r"(x[20]), "=r"(x[21]), "=r"(x[22]), "=r"(x[23]), "=r"(x[24]),
          "=r"(x[25]), "=r"(x[26]), "=r"(x[27]), "=r"(x[28]), "=r"(x[29]), "=r"(x[30]), "=r"(x[31])
        : "r"(taddr) : "memory");
}

// own[k] without an index register
template <int N, typename T>
__device__ __forceinline__ T tc_pick(const T (&own)[N], int k) {
    T o = own[0];
#pragma unroll
    for (int j = 1; j < N; ++j) o = k == j ? own[j] : o;
    return o;
}

// Barriers (all waits bounded):
//   full_x[s]      8 or 16 arrivals (one per loader warp, after its stores)          -> MMA warp may read the rows
//   full_w[s]      bytes of the weights' copy                                         -> ... and the weights
//   empty[s]       tcgen05.commit of the MMAs that read stage s                      -> both may be refilled
//   acc_full[b]    tcgen05.commit after the last MMA of a tile into buffer b         -> epilogue may read
//   acc_empty[b]   8 arrivals (one per epilogue warp, accumulators read)             -> MMA warp may overwrite
// The step counter runs on across tiles, so the loads of the next tile start while the last MMAs of this one are
// still in flight.
// RESIDENT: the weights stay in shared memory; else they stream.
// SUM: the row operand is alpha h + scale S (GIN), two rows per entry.
// PIECES: narrow outputs, whose products are fp32 sums on SIMT and no less exact here, dense rows or sparse ones (see
// tc_weights_build).  Rows and weights are cut into three parts in bf16, 8 bits each: all 24 bits of an entry.  One product
// is large, that of the first parts, 16 bits wide, so that what the tensor core's rounding towards zero takes of a sum of
// them is small; its accumulator is handed over with every chunk and the chunks meet in the epilogue's registers, in fp32.
// The seven small products (all but that of the third parts, 2^-33 relative) gather over the whole tile.  In a stage, a
// row's 128 bytes hold the first part and the second, the other half of the stage the third and 64 bytes of nothing.
// Lanes 0..63 are the columns of the first problem, lanes 64..127 those of the second, which reads the same rows.  (The
// epilogue's 64 sums per thread leave registers for four loader warps.)
// Measured: 2.4 M rows, K = 256, two products of 48 columns 1.31 -> 1.23 ms (fp32 sums 3.43).  Bound by the chain loaders, products,
// epilogue with two accumulators between them: hand-overs every 16 entries 1.43 ms; the loaders' stores without bank
// conflicts nothing.
template <bool RESIDENT, bool SUM, bool PIECES>
__global__ void __launch_bounds__(tc_threads(RESIDENT, PIECES), 1)
k_update_rows_tc(Ctl* ctl, const __grid_constant__ UpdPair pair) {
    constexpr int TC_LOADERS = tc_loaders(RESIDENT, PIECES);
    constexpr int TILE = TC_TILE, RSTEP = TC_LOADERS / 8, ITS = TILE / RSTEP;
    constexpr int X_HALF = TILE * 128, X_BYTES = 2 * X_HALF, NH = tc_stages(RESIDENT);
    constexpr int W_SLOTS = RESIDENT ? TC_RESIDENT_CHUNKS : TC_W_STAGES;
    // Tensor-memory columns: two accumulators of [hi hi | corrections]; with PIECES two of the former, two of the latter.
    constexpr int BUF = PIECES ? TILE : 2 * TILE;
    pdl_enter();
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_x[NH], full_w[W_SLOTS], empty[NH], acc_full[2], acc_empty[2], drained;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_fail;

    if (ctl->abort) return;
    // This CTA's column group: those of the first problem, then those of the second.
    const int g0 = pair.p[0].tc_groups, G = g0 + (!PIECES && pair.n > 1 ? pair.p[1].tc_groups : 0);
    const int my_g = (int)blockIdx.x % G, member = (int)blockIdx.x / G, members = ((int)gridDim.x - my_g + G - 1) / G;
    const UpdParams& p = pair.p[my_g < g0 ? 0 : 1];
    const int grp = my_g < g0 ? my_g : my_g - g0;
    // (what the issuing warp's control flow depends on is broadcast: its operands stay in uniform registers only if the
    // compiler can see that the warp runs as one; otherwise every MMA instruction costs 90 cycles to issue)
    const int n = __shfl_sync(FULL, upd_rows(p), 0);
    if (!upd_use_tc(p, n)) return;
    const int row_tiles = (n + TILE - 1) / TILE;
    if (member >= row_tiles) return;   // before any allocation

    // the diagnostic that withholds a completion also shortens the waits, so that they run out in milliseconds
    const uint32_t spin_limit = p.tc_withhold ? (1u << 16) : TC_SPIN_LIMIT;
    const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
    const bool x3 = p.tc_mode == TC_TF32X3;
    const int nchunks = p.tc_chunks, K = p.K;
    const float* weights = p.tc_w + (size_t)grp * nchunks * (TC_W_BYTES / 4);
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* x_ring = smem;                                      // stages of rows: [as they come | their remainders]
    uint8_t* w_ring = smem + (size_t)NH * X_BYTES;               // stages of [hi | lo] weights, or all chunks of them
    constexpr uint32_t tmem_cols = 4 * TILE;

    if (tid == 0) {
        for (int s = 0; s < NH; ++s) { mbar_init(&full_x[s], TC_LOADERS / 32); mbar_init(&empty[s], 1); }
        for (int s = 0; s < W_SLOTS; ++s) mbar_init(&full_w[s], 1);
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], TC_EPI_WARPS); }
        mbar_init(&drained, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;

    const int my_tiles = (row_tiles - member + members - 1) / members;
    const int total_steps = my_tiles * nchunks;
    auto tile_row = [&](int lt) { return (member + lt * members) * TILE; };

    if (warp < TC_LOADERS / 32) {
        // ---------------- row gathers ----------------
        // thread: piece c of the rows rb + RSTEP it of every chunk.  A chunk travels as asynchronous copies straight into
        // its stage of the high operand, NH - 1 chunks ahead; when it has landed, the thread that asked for a piece reads
        // it back, takes what the tensor core will not see of it -- it reads the upper 19 bits of an entry -- and stores
        // that as the low operand; with PIECES the three parts take the place of the piece and of its neighbours' in the row.  (Row pieces held in registers across the barrier waits took 1.9 us per chunk, most
        // of it one warp's chain of dependent instructions.)
        const int c = tid & 7, rb = tid >> 3;
        const bool from_s = p.a_mode == A_AGG || SUM;
        const float* const base = (from_s ? p.S : p.Hprev) + c * 4;
        const int ldr = from_s ? p.ld_s : p.ld_h, ldh = p.ld_h;
        const int32_t* const list = p.a_mode == A_DENSE ? nullptr : p.list;
        const uint32_t x_mine = smem_u32(x_ring) + tc_swz(rb, c);
        int rows_next[ITS];           // rows of the tile after the one being requested
        auto ids = [&](int lt) {
#pragma unroll
            for (int it = 0; it < ITS; ++it) {
                const int i = tile_row(lt) + rb + RSTEP * it;
                const int j = lt < my_tiles && i < n ? i : 0;   // (rows beyond the last are multiplied and dropped)
                rows_next[it] = list ? list[j] : j;
            }
        };
        const float *ptr[ITS], *ptr_h[SUM ? ITS : 1];
        float sc_next[SUM ? ITS : 1], sc_req[SUM ? ITS : 1];   // row factors of the tile being requested, and after it
        auto aim = [&]() {
#pragma unroll
            for (int it = 0; it < ITS; ++it) {
                const size_t r = (size_t)rows_next[it];
                ptr[it] = base + r * ldr;
                if constexpr (SUM) {
                    ptr_h[it] = p.Hprev + c * 4 + r * ldh;
                    sc_req[it] = sc_next[it];
                }
            }
        };
        auto scales = [&]() {
            if constexpr (SUM) {
#pragma unroll
                for (int it = 0; it < ITS; ++it) sc_next[it] = upd_row_scale(p, rows_next[it]);
            }
        };
        ids(0);
        scales();
        aim();
        ids(1);
        scales();
        int lt_l = 0, k_l = 0, s_l = 0;   // tile, K offset and stage of the next chunk to request
        // beyond K (and beyond the last chunk) zeros are written and nothing is read
        auto request = [&](bool live) {
            const uint32_t bytes = live && k_l + c * 4 < K ? 16u : 0u;
            const int off = bytes ? k_l : 0;
#pragma unroll
            for (int it = 0; it < ITS; ++it) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                             ::"r"(x_mine + (uint32_t)(s_l * X_BYTES + it * (RSTEP * 128))), "l"(ptr[it] + off), "r"(bytes) : "memory");
                if constexpr (SUM)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                                 ::"r"(x_mine + (uint32_t)(s_l * X_BYTES + X_HALF + it * (RSTEP * 128))), "l"(ptr_h[it] + off), "r"(bytes) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (++s_l == NH) s_l = 0;
            k_l += TC_KC;
            if (k_l >= K) {
                k_l = 0;
                ++lt_l;
                aim();
                ids(lt_l + 1);
                scales();
            }
        };
        // (SUM: the factors of the chunk being converted belong to an earlier request: kept per stage)
        float sc_ring[SUM ? NH : 1][SUM ? ITS : 1];
        auto keep = [&](int slot) {
            if constexpr (SUM) {
#pragma unroll
                for (int it = 0; it < ITS; ++it)
#pragma unroll
                    for (int d = 0; d < NH; ++d) if (d == slot) sc_ring[d][it] = sc_req[it];
            }
        };
        const float alpha = p.alpha;
#pragma unroll
        for (int d = 0; d < NH - 1; ++d) { keep(d); request(d < total_steps); }
        int s = 0, s_prev = NH - 1;
        uint32_t ph_prev = 1;         // phase of the stage that the step before used (a fresh barrier counts as completed)
        bool ok = true;
        for (int g = 0; g < total_steps && ok; ++g) {
            asm volatile("cp.async.wait_group %0;" ::"n"(NH - 2) : "memory");
            const uint32_t hi = x_mine + (uint32_t)(s * X_BYTES), lo = hi + X_HALF;
            if (x3 || SUM) {
                float4 x[ITS];
#pragma unroll
                for (int it = 0; it < ITS; ++it) x[it] = tc_lds(hi + it * (RSTEP * 128));
                if constexpr (PIECES) {
                    const uint32_t to = hi - tc_swz(rb, c) + tc_swz(rb, c >> 1) + 8 * (c & 1);
                    __syncwarp();   // a row's pieces, with eight lanes of this warp, have been read
#pragma unroll
                    for (int it = 0; it < ITS; ++it) {
                        const uint32_t at = to + it * (RSTEP * 128);
                        float4& e = x[it];
                        uint32_t lower = bf16_cut(e.x, e.y), upper = bf16_cut(e.z, e.w);
                        tc_sts2(at, lower, upper);
                        lower = bf16_round(e.x, e.y), upper = bf16_round(e.z, e.w);
                        tc_sts2(at ^ 64, lower, upper);
                        lower = bf16_round(e.x, e.y), upper = bf16_round(e.z, e.w);
                        tc_sts2(at + X_HALF, lower, upper);
                    }
                } else {
                if constexpr (SUM) {
#pragma unroll
                    for (int it = 0; it < ITS; ++it) {
                        const float4 h = tc_lds(lo + it * (RSTEP * 128));
                        float f = sc_ring[0][it];
#pragma unroll
                        for (int d = 1; d < NH; ++d) f = d == s ? sc_ring[d][it] : f;
                        x[it] = make_float4(f * x[it].x + alpha * h.x, f * x[it].y + alpha * h.y, f * x[it].z + alpha * h.z, f * x[it].w + alpha * h.w);
                        tc_sts(hi + it * (RSTEP * 128), x[it]);
                    }
                }
#pragma unroll
                for (int it = 0; it < ITS; ++it)
                    tc_sts(lo + it * (RSTEP * 128), make_float4(x[it].x - tf32_seen(x[it].x), x[it].y - tf32_seen(x[it].y),
                                                                x[it].z - tf32_seen(x[it].z), x[it].w - tf32_seen(x[it].w)));
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&full_x[s]);
            // the stage that the step before used takes the chunk NH - 1 steps ahead
            ok = mbar_wait_bounded(&empty[s_prev], ph_prev, spin_limit);
            keep(s_prev);
            request(g + NH - 1 < total_steps);
            if (g > 0 && s_prev == NH - 1) ph_prev ^= 1;
            if (g == 0) ph_prev = 0;
            s_prev = s;
            if (++s == NH) s = 0;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (!ok) s_fail = 1;
    } else if (warp < TC_LOADERS / 32 + TC_EPI_WARPS) {
        // ---------------- epilogue ----------------
        // A warp's index modulo 4 fixes the tensor-memory lanes it may read: output columns 32 q .. 32 q + 31 of the
        // group, one per lane; the two warps of a quarter take half of the tile's rows each, BLK rows at a time.
        constexpr int BLK = 16, HALF = TILE / 2, OWN = HALF / 32;
        const int q = warp & 3, half = (warp - TC_LOADERS / 32) >> 2;
        const int col0 = PIECES ? 32 * (q & 1) : grp * TC_COLS + 32 * q;   // the first of this warp's columns
        const UpdParams& p = PIECES && q >= 2 ? pair.p[1] : pair.p[my_g < g0 ? 0 : 1];
        int lc = col0 + lane;                     // this lane's column
        const bool col_ok = lc < p.n_cols && (!PIECES || q < 2 || pair.n > 1);
        if (!col_ok) lc = 0;
        float* const hout = p.Hout + lc;
        float* const dout = p.epi_mode == EPI_COMMIT && p.Dout ? p.Dout + lc : nullptr;
        const float bias = p.bias ? p.bias[lc] : 0.f;
        const int ldo = p.ld_o;
        const uint32_t ld_bytes = 4u * (uint32_t)ldo;
        const bool relu = p.act == RIPPLE_ACT_RELU, keep_old = p.dout_old != 0;
        const bool any_z = p.addend2 != nullptr, any_old = upd_needs_old(p);
        const bool plus_s = p.addend || p.addend_rw, temp = p.epi_mode == EPI_TEMP;
        const bool coefs = p.src_norm && any_old;
        const bool scaled = p.a_mode == A_AGG || plus_s;
        const float alpha = p.a_mode == A_SELF ? p.alpha : 1.0f;
        const bool warp_busy = __any_sync(FULL, col_ok);
        // the row that is read ahead: the cached projection or the row's previous value (both have the output's width)
        const bool fetching = any_z || any_old;
        int v_own[OWN], v_next[OWN];        // rows of this tile and the next, 32 per register
        float sc_own[OWN], sc_next[OWN];
        auto ids = [&](int lt) {
#pragma unroll
            for (int k = 0; k < OWN; ++k) {
                const int i = tile_row(lt) + HALF * half + 32 * k + lane;
                const bool in = lt < my_tiles && i < n;
                v_next[k] = in ? (p.list ? p.list[i] : i) : 0;
                sc_next[k] = 1.0f;
                if (scaled && in) sc_next[k] = upd_row_scale(p, v_next[k]);
            }
        };
        // Rows are worked on in blocks.  What is read ahead of a block was requested DEPTH blocks before, across the end of
        // the tile too, as asynchronous copies into shared memory, 16 bytes per lane and four rows per instruction:
        // loads into registers were waited for at the next barrier wait, whatever their distance to the first use.
        constexpr int DEPTH = TC_AHEAD, BLOCKS = HALF / BLK;
        float* const zbuf = reinterpret_cast<float*>(w_ring + (size_t)W_SLOTS * TC_W_BYTES) + (warp - TC_LOADERS / 32) * (DEPTH * BLK * 32);
        // the piece of the row that this lane copies: four columns
        const int pc = col0 + 4 * (lane & 7);
        const float* const piece = (any_z ? p.addend2 : p.Hout) + (pc < p.n_cols ? pc : 0);
        auto fetch = [&](int slot, int v_src, int at) {
#pragma unroll
            for (int i = 0; i < BLK / 4; ++i) {
                const int r = 4 * i + (lane >> 3), v = __shfl_sync(FULL, v_src, at + r);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             ::"r"(smem_u32(zbuf + slot * (BLK * 32) + r * 32 + 4 * (lane & 7))), "l"(piece + (size_t)v * ldo) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        ids(0);
        if (fetching && warp_busy) {
#pragma unroll
            for (int d = 0; d < DEPTH; ++d) fetch(d, tc_pick<OWN>(v_next, d * BLK / 32), (d * BLK) & 31);
        }
        bool ok = true;
        int sg = 0;                         // accumulators handed over so far: one per tile, with PIECES one per chunk
        for (int lt = 0; lt < my_tiles && ok; ++lt) {
            const int r0 = tile_row(lt) + HALF * half;
#pragma unroll
            for (int k = 0; k < OWN; ++k) {
                v_own[k] = v_next[k];
                sc_own[k] = sc_next[k];
            }
            ids(lt + 1);
            auto take = [&](float (&h)[BLK], int blk, int buf) {   // BLK rows of the accumulator, its small products added
                const uint32_t t_mine = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * BUF + HALF * half + blk * BLK);
                uint32_t x[BLK];
                tc_load16(x, t_mine);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int r = 0; r < BLK; ++r) h[r] = __uint_as_float(x[r]);
                if (x3) {
                    tc_load16(x, t_mine + (uint32_t)TILE);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int r = 0; r < BLK; ++r) h[r] += __uint_as_float(x[r]);
                }
            };
            auto block = [&](int blk, float (&h)[BLK]) {
                const int at = (blk * BLK) & 31, i0 = r0 + blk * BLK;
                const int v_src = tc_pick<OWN>(v_own, blk * BLK / 32);
                const float s_src = tc_pick<OWN>(sc_own, blk * BLK / 32);
                if (plus_s) {   // (transformed aggregates with a self term of their own: GIN layers that narrow)
#pragma unroll 1
                    for (int r = 0; r < BLK; ++r) {
                        const int v = __shfl_sync(FULL, v_src, at + r);
                        const float sc = __shfl_sync(FULL, s_src, at + r);
                        float acc = 0.f;
#pragma unroll
                        for (int j = 0; j < BLK; ++j) acc = j == r ? h[j] : acc;
                        if (i0 + r >= n || !col_ok) continue;
                        const size_t row = (size_t)v * ldo, sa = (size_t)v * p.ld_add + lc;
                        float t = p.addend_rw ? p.addend_rw[sa] : p.addend[sa];
                        if (p.addend_rw) {
                            t += p.addend_delta[sa];
                            p.addend_rw[sa] = t;
                            p.addend_delta[sa] = 0.f;
                        }
                        float y = (p.a_mode == A_AGG ? sc : alpha) * acc + bias + sc * t;
                        if (any_z) y += p.addend2[row + lc];
                        if (relu) y = fmaxf(y, 0.f);
                        if (temp) { hout[(size_t)(i0 + r) * ldo] = y; continue; }
                        if (dout) {
                            const float o = hout[row];
                            float cn = 1.f, co = 1.f;
                            if (p.src_norm) {
                                const int dold = p.deg_out_old[v];
                                cn = coef_deg(p.deg_out[v]);
                                co = dold >= 0 ? coef_deg(dold) : cn;
                            }
                            dout[(size_t)(i0 + r) * ldo] = keep_old ? o : cn * y - co * o;
                        }
                        hout[row] = y;
                    }
                    return;
                }
                if (scaled) {
#pragma unroll
                    for (int r = 0; r < BLK; ++r) h[r] = __shfl_sync(FULL, s_src, at + r) * h[r] + bias;
                } else {
#pragma unroll
                    for (int r = 0; r < BLK; ++r) h[r] = alpha * h[r] + bias;
                }
                const float* const z = zbuf + (blk % DEPTH) * (BLK * 32) + lane;
                if (fetching) {
                    asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH - 1) : "memory");
                    __syncwarp();
                }
                if (any_z) {
#pragma unroll
                    for (int r = 0; r < BLK; ++r) h[r] += z[32 * r];
                }
                if (relu) {
#pragma unroll
                    for (int r = 0; r < BLK; ++r) h[r] = fmaxf(h[r], 0.f);
                }
                if (any_old) {
                    const int live = col_ok && dout ? n - i0 : 0;
                    float* to = dout + (size_t)i0 * ldo;
                    if (any_z) {   // both a cached projection and the row's previous value: that one is asked for here
                        float cn = 1.f, co = 1.f;   // source coefficients now and before the batch, one row per lane
                        if (coefs) {
                            const int d_old = p.deg_out_old[v_src];
                            cn = coef_deg(p.deg_out[v_src]);
                            co = d_old >= 0 ? coef_deg(d_old) : cn;
                        }
#pragma unroll
                        for (int r0_ = 0; r0_ < BLK; r0_ += 4) {
                            float o[4];
#pragma unroll
                            for (int r = 0; r < 4; ++r) o[r] = hout[(size_t)__shfl_sync(FULL, v_src, at + r0_ + r) * ldo];
#pragma unroll
                            for (int r = 0; r < 4; ++r, to += ldo) {
                                const float d = __shfl_sync(FULL, cn, at + r0_ + r) * h[r0_ + r] - __shfl_sync(FULL, co, at + r0_ + r) * o[r];
                                tc_store_if(r0_ + r < live, to, keep_old ? o[r] : d);
                            }
                        }
                    } else if (coefs) {
                        const int d_old = p.deg_out_old[v_src];
                        const float cn = coef_deg(p.deg_out[v_src]), co = d_old >= 0 ? coef_deg(d_old) : cn;
#pragma unroll
                        for (int r = 0; r < BLK; ++r, to += ldo)
                            tc_store_if(r < live, to, __shfl_sync(FULL, cn, at + r) * h[r] - __shfl_sync(FULL, co, at + r) * z[32 * r]);
                    } else {
#pragma unroll
                        for (int r = 0; r < BLK; ++r, to += ldo) tc_store_if(r < live, to, keep_old ? z[32 * r] : h[r] - z[32 * r]);
                    }
                }
                if (fetching) {
                    const int nb = blk + DEPTH;
                    __syncwarp();
                    fetch(blk % DEPTH, nb < BLOCKS ? tc_pick<OWN>(v_own, nb * BLK / 32) : tc_pick<OWN>(v_next, (nb - BLOCKS) * BLK / 32), (nb * BLK) & 31);
                }
                const int live = col_ok ? n - i0 : 0;
                uint32_t v[BLK];
#pragma unroll
                for (int r = 0; r < BLK; ++r) v[r] = (uint32_t)__shfl_sync(FULL, v_src, at + r);
                if (temp) {
#pragma unroll
                    for (int r = 0; r < BLK; ++r) v[r] = (uint32_t)(i0 + r);
                }
#pragma unroll
                for (int r = 0; r < BLK; ++r)
                    tc_store_if(r < live, reinterpret_cast<float*>(reinterpret_cast<char*>(hout) + (uint64_t)v[r] * ld_bytes), h[r]);
            };
            const int parts = PIECES ? nchunks : 1;
            float sum[PIECES ? BLOCKS : 1][BLK];
            for (int part = 0; part < parts; ++part, ++sg) {
                const int b = sg & 1;
                ok = mbar_wait_bounded(&acc_full[b], (sg >> 1) & 1, spin_limit);
                if (!ok) { s_fail = 1; break; }
                tc_fence_after();
                if (warp_busy) {
                    if constexpr (PIECES) {
                        const uint32_t t_row = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(HALF * half);
                        if (part == 0) {
#pragma unroll
                            for (int r = 0; r < HALF; ++r) sum[r / BLK][r % BLK] = 0.f;
                        }
                        auto add = [&](uint32_t from, bool small) {   // (an infinite entry has no parts: its small products are NaN)
#pragma unroll
                            for (int r0_ = 0; r0_ < HALF; r0_ += 32) {
                                uint32_t x[32];
                                tc_load32(x, from + (uint32_t)r0_);
                                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                                for (int r = 0; r < 32; ++r) {
                                    float& h = sum[(r0_ + r) / BLK][(r0_ + r) % BLK];
                                    if (!small || fabsf(h) < INFINITY) h += __uint_as_float(x[r]);
                                }
                            }
                        };
                        add(t_row + (uint32_t)(b * BUF), false);
                        if (part == parts - 1) add(t_row + (uint32_t)(2 * TILE + (lt & 1) * TILE), true);
                    } else {
#pragma unroll 1
                        for (int blk = 0; blk < BLOCKS; ++blk) {
                            float h[BLK];
                            take(h, blk, b);
                            block(blk, h);
                        }
                    }
                }
                tc_fence_before();   // accumulators consumed: the MMA warp may overwrite them after this arrival
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[b]);
            }
            if constexpr (PIECES) {
                if (ok && warp_busy) {
#pragma unroll
                    for (int blk = 0; blk < BLOCKS; ++blk) block(blk, sum[blk]);
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    } else if (warp == TC_LOADERS / 32 + TC_EPI_WARPS) {
        // ---------------- MMA issue ----------------
        const bool lead = tc_elect();
        constexpr uint32_t idesc = tc_idesc(TILE), idesc_wide = tc_idesc(2 * TILE);
        const uint64_t dx0 = tc_smem_desc(smem_u32(x_ring)), dw0 = tc_smem_desc(smem_u32(w_ring));
        const bool withhold = p.tc_withhold != 0;
        int s = 0, sw = 0;
        uint32_t ph = 0, phw = 0;              // ring slots and phases of this step
        bool ok = true;
        int sg = 0;                            // accumulators begun so far
        for (int lt = 0; lt < my_tiles; ++lt) {
            uint32_t d_addr = 0, d_corr = 0;
            int left = K, b = 0;
            for (int kc = 0; kc < nchunks; ++kc, left -= TC_KC) {
                auto begin = [&]() {
                    // the epilogue must have drained this accumulator buffer (the one before the last)
                    b = sg & 1;
                    const int ub = sg >> 1;
                    ++sg;
                    if (ub > 0) ok = __all_sync(FULL, mbar_wait_bounded(&acc_empty[b], (ub - 1) & 1, spin_limit));
                    if (!ok) return;
                    tc_fence_after();
                    d_addr = tmem_base + (uint32_t)(b * BUF);
                    // (a tile's small products may go where the tile before the last had them: its last chunk has been drained)
                    d_corr = PIECES ? tmem_base + (uint32_t)(2 * TILE + (lt & 1) * TILE) : d_addr + TILE;
                };
                if (PIECES || kc == 0) begin();
                if (!ok) break;
                if (RESIDENT) sw = kc;
                bool there = true;
                if (!RESIDENT || lt == 0) there = mbar_wait_bounded(&full_w[sw], phw, spin_limit);
                there = there && mbar_wait_bounded(&full_x[s], ph, spin_limit);
                ok = __all_sync(FULL, there);
                if (!ok) break;
                // The loaders' stores become visible to the tensor core's async proxy here, on the reader's side of the
                // barrier: in the loaders the fence would wait for their row gathers in flight as well.
                fence_async_smem();
                tc_fence_after();
                const uint64_t xh = dx0 + (uint64_t)((uint32_t)s * (X_BYTES >> 4));
                const uint64_t wh = dw0 + (uint64_t)((uint32_t)sw * (TC_W_BYTES >> 4)), wl = wh + (TC_W_HALF >> 4);
                const bool last = PIECES || kc == nchunks - 1;   // of what this accumulator takes
                if (lead) {
                    if constexpr (PIECES) {
                        constexpr uint32_t bf16 = tc_idesc(TILE, 1);
#pragma unroll
                        for (int j = 0; j < TC_KC / 16; ++j) {     // one MMA K step = 16 entries = 32 bytes
                            if (16 * j < left) {
                                const uint64_t x1 = xh + 2 * j, x2 = x1 + 4, x_3 = x1 + (X_HALF >> 4);
                                const uint64_t w1 = wh + 2 * j, w2 = w1 + 4, w3 = wl + 2 * j;
                                tc_mma_bf16(d_addr, w1, x1, bf16, j != 0);
                                tc_mma_bf16(d_corr, w1, x2, bf16, (kc | j) != 0);
                                tc_mma_bf16(d_corr, w2, x1, bf16, 1u);
                                tc_mma_bf16(d_corr, w2, x2, bf16, 1u);
                                tc_mma_bf16(d_corr, w1, x_3, bf16, 1u);
                                tc_mma_bf16(d_corr, w3, x1, bf16, 1u);
                                tc_mma_bf16(d_corr, w2, x_3, bf16, 1u);
                                tc_mma_bf16(d_corr, w3, x2, bf16, 1u);
                            }
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < TC_KC / 8; ++j) {     // one MMA K step = 8 floats = 32 bytes
                            if (8 * j < left) {
                                tc_mma_tf32(d_addr, wh + 2 * j, xh + 2 * j, x3 ? idesc_wide : idesc, (kc | j) != 0);
                                if (x3) tc_mma_tf32(d_corr, wl + 2 * j, xh + 2 * j, idesc, 1u);
                            }
                        }
                    }
                    tc_commit(&empty[s]);
                    // (diagnostic: with tc_withhold the first tile is never reported finished, so that
                    // the epilogue's bounded wait runs out and the status path can be exercised)
                    if (last && !(withhold && lt == 0)) tc_commit(&acc_full[b]);
                }
                __syncwarp();
                if (++s == NH) { s = 0; ph ^= 1; }
                if (!RESIDENT && ++sw == TC_W_STAGES) { sw = 0; phw ^= 1; }
            }
            if (!ok) break;
        }
        // No product of this CTA may be in flight when it frees its tensor memory, however the other roles end: an epilogue
        // that gave up waiting leaves while this warp still issues.  (In a pass that ends well the epilogue waits for the
        // same products: nothing is lost by it.)
        if (lead) {
            if (!ok) s_fail = 1;
            tc_commit(&drained);
            mbar_wait_bounded(&drained, 0, TC_SPIN_LIMIT);
        }
    } else {
        // ---------------- weights: bulk copies, one thread ----------------
        if (lane == 0) {
            const int slots = RESIDENT ? nchunks : TC_W_STAGES, all = RESIDENT ? nchunks : total_steps;
            int kc = 0, sw = 0, s = 0, c = 0;
            uint32_t ph = 0;
            for (; c < all; ++c) {
                if (c >= slots) {   // the step whose weights lie there must have been multiplied: step c - slots
                    if (!mbar_wait_bounded(&empty[s], ph, spin_limit)) { s_fail = 1; break; }
                    if (++s == NH) { s = 0; ph ^= 1; }
                }
                tc_copy_weights(w_ring + (size_t)sw * TC_W_BYTES, weights + (size_t)kc * (TC_W_BYTES / 4), TC_W_BYTES, &full_w[sw]);
                if (++kc == nchunks) kc = 0;
                if (++sw == slots) sw = 0;
            }
            // no copy of this CTA may be in flight when it leaves: the latest into each slot (usually long there)
            for (int k = 0; k < min(c, slots); ++k) {
                const int latest = c - 1 - k;
                mbar_wait_bounded(&full_w[latest % slots], (uint32_t)(latest / slots) & 1, TC_SPIN_LIMIT);
            }
        }
    }

    __syncwarp();
    if (s_fail && lane == 0) {
        atomicCAS(&ctl->err, 0, (int)RIPPLE_ERR_TIMEOUT);
        ctl->abort = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
}

static size_t tc_smem_bytes(bool resident) {
    return (size_t)tc_stages(resident) * TC_TILE * 256 + (size_t)(resident ? TC_RESIDENT_CHUNKS : TC_W_STAGES) * TC_W_BYTES +
           (size_t)TC_EPI_WARPS * TC_AHEAD * 16 * 128 + 1024;
}

void launch_update_tc(Ctx* c, const UpdPair& pair, bool pieces) {
    const bool resident = pair.p[0].tc_chunks <= TC_RESIDENT_CHUNKS, sum = pair.p[0].a_mode == A_SUM;
    // one persistent CTA per SM: operands and weights fill its shared memory
#define TC_GO(RES, SUM, PIECES) RP_LAUNCH(c, (k_update_rows_tc<RES, SUM, PIECES>), c->n_sm, tc_threads(RES, PIECES), tc_smem_bytes(RES), c->ctl, pair)
    if (pieces) TC_GO(false, false, true);
    else if (resident && sum) TC_GO(true, true, false);
    else if (resident) TC_GO(true, false, false);
    else if (sum) TC_GO(false, true, false);
    else TC_GO(false, false, false);
#undef TC_GO
}

void tc_prepare() {
#define TC_SET(RES, SUM, PIECES) cudaFuncSetAttribute(k_update_rows_tc<RES, SUM, PIECES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes(RES))
    TC_SET(true, true, false);
    TC_SET(true, false, false);
    TC_SET(false, true, false);
    TC_SET(false, false, false);
    TC_SET(false, false, true);
#undef TC_SET
}

// The weights (row-major K x ldw) as the kernel copies them: per column group and K chunk, the group's 128 columns as rows
// of 32 K entries, first rounded to tf32, then the remainders (likewise rounded), in the swizzled layout of the operand;
// for the form in pieces as three parts in bf16, laid out as the rows' are.
//
// Which outputs have them, and from how many rows the form is taken (RP_TC_MIN_ROWS), is a line of precision.  The tf32 form
// is the faster one from 512 rows on (whole-graph pass of one layer, K = 256, 256 columns: 512 rows 39 us, fp32 sums 46;
// 1024: 39 / 52; 32 768: 94 / 321), but two to three times less exact than fp32 sums (see the top of the file).  Outputs of
// 113 to 256 columns over 1024 and more rows have always been split products, and less exact ones than these; all others
// were fp32 sums and lose nothing: up to 64 columns the form in pieces takes them.  Its error against fp64, 2-norm, and that
// of the fp32 sum, by the entries of a row that are not zero (N(0, 1); K = 256 and 602, 5 to 64 columns alike; neighbouring
// entries or scattered ones): 1 entry 2.5e-8 / 2.5e-8, 2 2.6e-8 / 3.1e-8, 4 2.6e-8 / 4.0e-8, 16 3.3e-8 / 7.4e-8, 64 5.1e-8 / 1.4e-7,
// all of 256 7.4e-8 / 2.9e-7, of 602 1.0e-7 / 4.4e-7; rectified rows 6.2e-8 / 2.1e-7 and 8.8e-8 / 3.0e-7.
// One of 40 columns over 80 K rows: 89 us, fp32 sums 125.
// W2: a second matrix over the same rows, for the form in pieces.
cudaError_t tc_weights_build(TcW* out, const float* W, int K, int ldw, const float* W2) {
    *out = TcW{};
    const bool pieces = ldw <= RP_TC_PIECES_MAX_COLS && K >= RP_TC_PIECES_MIN_K;
    if (K <= 0 || !(pieces || (!W2 && ldw >= RP_TC_MIN_COLS && ldw <= RP_TC_MAX_COLS))) return cudaSuccess;
    out->pieces = pieces;
    auto round_tf32 = [](float v) {
        uint32_t bits;
        memcpy(&bits, &v, 4);
        bits = (bits + 0x1000u) & 0xffffe000u;
        memcpy(&v, &bits, 4);
        return v;
    };
    auto bf16_part = [](float& left, bool round) {   // (as bf16_cut and bf16_round)
        uint32_t bits;
        memcpy(&bits, &left, 4);
        if (round) bits += 0x7fffu + (bits >> 16 & 1u);
        bits &= 0xffff0000u;
        float part;
        memcpy(&part, &bits, 4);
        left -= part;
        return (uint16_t)(bits >> 16);
    };
    out->groups = (ldw + TC_COLS - 1) / TC_COLS;
    out->chunks = (K + TC_KC - 1) / TC_KC;
    const size_t block = TC_W_BYTES / 4;
    std::vector<float> pack(block * out->chunks * out->groups, 0.f);
    for (int m = 0; m < (W2 ? 2 : 1); ++m)
        for (int k = 0; k < K; ++k)
            for (int j = 0; j < ldw; ++j) {
                const float x = (m ? W2 : W)[(size_t)k * ldw + j], h = round_tf32(x);
                const int col = j + m * (TC_COLS / 2);
                const int g = col / TC_COLS, r = col - g * TC_COLS, kc = k / TC_KC, kk = k - kc * TC_KC;
                float* blk = pack.data() + ((size_t)g * out->chunks + kc) * block;
                if (pieces) {
                    uint16_t* const to = reinterpret_cast<uint16_t*>(blk);
                    const uint32_t first = tc_swz(r, kk >> 3) / 2 + (kk & 7);
                    float left = x;
                    to[first] = bf16_part(left, false);
                    to[first ^ 32] = bf16_part(left, true);
                    to[TC_W_HALF / 2 + first] = bf16_part(left, true);
                    continue;
                }
                const uint32_t at = tc_swz(r, kk >> 2) / 4 + (kk & 3);
                blk[at] = h;
                blk[TC_W_HALF / 4 + at] = round_tf32(x - h);
            }
    cudaError_t e = cudaMalloc(&out->w, sizeof(float) * pack.size());
    if (!e) e = cudaMemcpy(out->w, pack.data(), sizeof(float) * pack.size(), cudaMemcpyHostToDevice);
    return e;
}

}  // namespace rp
