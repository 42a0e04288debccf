// bf16 GEMM on the 5th-generation tensor core (tcgen05), fed by TMA.
//
//   C[M][N] = epilogue(A[M][K] @ Wt[N][K]^T), fp32 accumulation in TMEM.
//
// Tilings, picked by gemm_tc_bn:
//   pair   (BN = 256) a cluster of two CTAs works on one 256 x 256 tile with
//          tcgen05.mma.cta_group::2: each CTA loads its 128 rows of A and
//          half of B's 256 rows, 32 KB per 64-deep k step where a CTA of its
//          own with a 128 x 256 tile loads 48 KB -- the operand feed from L2
//          bounds the main loop, so a third fewer bytes per MMA is what the
//          pair is for (and six ring stages fit instead of four);
//   wide   (BN = 256, WIDE) one CTA per 128 x 256 tile, four ring stages, where
//          the row count leaves the pairs a ragged last round;
//   single (BN = 128, 64) one CTA per 128 x BN tile, for GEMMs with too few
//          256 x 256 tiles to fill the pairs.  With few tiles a k step takes
//          the MMA warp's chain of instructions (some 340 cycles) at either
//          width: 64-wide tiles spread the epilogue over twice the CTAs (840 x
//          512 x 512 5.2 us 128 wide, 4.6 64 wide).
// Persistent: the CTAs (pairs) walk the output tiles in grouped super-rows
// (tile_at).  Warp roles (320 threads per CTA):
//   warp 0         : TMA producer, STAGES-deep ring of (A 128x64, B 128x64)
//                    tiles in 128B-swizzled shared memory, continuous across
//                    output tiles; in a pair both CTAs' bytes are counted on
//                    the leader's full barriers;
//   warp 1         : allocates TMEM (two accumulators) and issues
//                    tcgen05.mma (K=16; 4 per 64-wide k-tile) into the free
//                    accumulator from a converged warp; in a pair the
//                    leader's alone, its commits arriving in both CTAs;
//   warps 2..9     : epilogue, two warps per TMEM lane quadrant, half of the
//                    columns each, in 32 x 32 blocks: thread = row, the
//                    block's residual operands arrive in shared memory by
//                    TMA, the fused epilogue (bias / GELU / gated residual /
//                    residual cache / RoPE) runs in registers, and the bf16
//                    block leaves by a TMA store from a 64B-swizzled staging
//                    buffer.  The accumulator is released (to the leader)
//                    after its last TMEM read, so the epilogue of tile i
//                    overlaps the main loop of tile i + 1.
// The skip flag of the block lets the whole recompute path early-exit when
// the gate chose reuse (Eq. 4), so decisions never return to the host.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <unordered_map>

#include "xc_kernels.cuh"
#include "xc_ptx.cuh"

namespace xc {

constexpr int GEMM_BM = 128;
constexpr int GEMM_BK = 64;
constexpr int GEMM_THREADS = 320;              // producer warp, MMA warp, 8 epilogue warps
constexpr int GEMM_SMEM_LIMIT = 232448;        // dynamic shared memory per CTA on this part
constexpr int EPI_BLOCK_BYTES = 32 * 32 * 2;   // one 32 x 32 bf16 block

// Staging ring of an epilogue warp: SLOTS slots of one 32 x 32 block (residual
// cache: two, out / r_hat), used in block order across output tiles.  The
// residual operands of a block land in its slot AHEAD blocks before they are
// needed, the output replaces them in place (a lane touches its own row
// only), and a slot is loaded or written again once its store has been read.
template <int EPI, bool DEEP, bool WIDE>
struct EpiRing {
    static constexpr bool RES = EPI == EPI_RESID_GATE || EPI == EPI_RESID_CACHE;
    static constexpr bool CACHE = EPI == EPI_RESID_CACHE;
    // Two slots leave the main loop six ring stages, four (DEEP) five; a gated
    // residual with a short K gains more from loading two blocks ahead.  Two /
    // four slots measured: 8064 x 1536 x 512 13.3 / 14.4 us, 12960 x 8960 x
    // 1536 + GELU 187 / 190; gated 6000 x 4096 x 512 28.0 / 25.9, gated 4000
    // x 256 x 6976 23.9 / 26.6.  A wide tile's residual cache has room for one
    // (loaded when its block begins) beside four main-loop stages: one slot and
    // four stages / two and three at 2356 x 2048 x 3392 24.0 / 28.6
    static constexpr int SLOTS = DEEP ? 4 : WIDE && CACHE ? 1 : 2;
    static constexpr int AHEAD = SLOTS / 2;
    static constexpr int SLOT_BYTES = (CACHE ? 2 : 1) * EPI_BLOCK_BYTES;
};

template <int BN, int EPI, bool DEEP, bool WIDE>
struct GemmTile {
    static constexpr bool PAIR = BN == 256 && !WIDE;   // two CTAs per tile
    static constexpr int BM = PAIR ? 2 * GEMM_BM : GEMM_BM;
    static constexpr int A_BYTES = GEMM_BM * GEMM_BK * 2;
    static constexpr int B_BYTES = (PAIR ? 128 : BN) * GEMM_BK * 2;   // pair: this CTA's half of B's rows
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int EPI_BYTES = 8 * EpiRing<EPI, DEEP, WIDE>::SLOTS * EpiRing<EPI, DEEP, WIDE>::SLOT_BYTES;
    static constexpr int VEC_BYTES = 8 * 64 * 4;       // bias and gate of a warp's block
    static constexpr int BAR_BYTES = VEC_BYTES + 512;
    static constexpr int FIT = (GEMM_SMEM_LIMIT - BAR_BYTES - EPI_BYTES) / STAGE_BYTES;
    static constexpr int STAGES = FIT > 8 ? 8 : FIT;
    static constexpr int OFF_EPI = STAGES * STAGE_BYTES;                // 1024-aligned
    static constexpr int OFF_VEC = OFF_EPI + EPI_BYTES;
    static constexpr int BAR_OFFSET = OFF_VEC + VEC_BYTES;
    static constexpr int SMEM_BYTES = OFF_VEC + BAR_BYTES;
    static constexpr int TMEM_COLS = 2 * BN;                             // double-buffered accumulator
    static constexpr int EPI_WARPS = PAIR ? 16 : 8;    // that release an accumulator
    static_assert(STAGES >= 3, "main-loop ring too shallow");
    static_assert(SMEM_BYTES <= GEMM_SMEM_LIMIT, "shared memory");
    static_assert(!PAIR || 2 * SMEM_BYTES > GEMM_SMEM_LIMIT, "one pair CTA per SM (pair_count)");
};

// Tensor maps of the epilogue (32 x 32 bf16 boxes, 64-byte swizzle):
// out[0..2] = q, k, v for the QKV epilogue, out[0] otherwise.
struct EpiMaps {
    CUtensorMap out[3];
    CUtensorMap rhat, resid, xin;
};

// Byte offset of 16-byte chunk k (0..3) of row r in a 64B-swizzled 32 x 32
// bf16 block (the layout TMA reads and writes with CU_TENSOR_MAP_SWIZZLE_64B).
__device__ __forceinline__ uint32_t sw64(int r, int k) { return (uint32_t)(r * 64 + ((k ^ ((r >> 1) & 3)) << 4)); }

// (a, b) += (x, y), (a, b) = (x a + r, y b + s): packed fp32 pairs
__device__ __forceinline__ void add2(float &a, float &b, float x, float y) {
    const float2 t = __fadd2_rn(make_float2(a, b), make_float2(x, y));
    a = t.x;
    b = t.y;
}
__device__ __forceinline__ void fma2(float &a, float &b, float x, float y, float r, float s) {
    const float2 t = __ffma2_rn(make_float2(x, y), make_float2(a, b), make_float2(r, s));
    a = t.x;
    b = t.y;
}
// gelu_tanh of two values with the hardware tanh, packed: its relative error of
// some 2^-11 is below the bf16 rounding of the output (2^-9)
__device__ __forceinline__ void gelu_tanh_approx2(float &a, float &b) {
    const float k0 = 0.7978845608028654f;
    const float2 x = make_float2(a, b);
    const float2 c = __fmul2_rn(make_float2(0.044715f, 0.044715f), x), x2 = __fmul2_rn(x, x);
    const float2 u = __fmul2_rn(make_float2(k0, k0), __ffma2_rn(c, x2, x));
    float2 t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t.x) : "f"(u.x));
    asm("tanh.approx.f32 %0, %1;" : "=f"(t.y) : "f"(u.y));
    const float2 hx = __fmul2_rn(make_float2(0.5f, 0.5f), x);
    const float2 y = __ffma2_rn(hx, t, hx);
    a = y.x;
    b = y.y;
}

// 32 bf16 of row r from a swizzled block -> float
__device__ __forceinline__ void read_row32(const uint8_t *blk, int r, float (&v)[32]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint4 u = *reinterpret_cast<const uint4 *>(blk + sw64(r, k));
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 t = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[j]));
            v[8 * k + 2 * j] = t.x;
            v[8 * k + 2 * j + 1] = t.y;
        }
    }
}
// float -> 32 bf16 (round to nearest) into row r of a swizzled block
__device__ __forceinline__ void write_row32(uint8_t *blk, int r, const float (&v)[32]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[8 * k + 2 * j], v[8 * k + 2 * j + 1]);
            w[j] = *reinterpret_cast<uint32_t *>(&h);
        }
        *reinterpret_cast<uint4 *>(blk + sw64(r, k)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Persistent tile order: tile t -> (m block, n block).  Tiles go in
// super-rows of 16 x 128 rows with m varying fastest inside a
// super-row, so the tiles in flight at one time (one per SM or pair) share
// the super-row's row blocks of A and a few column blocks of B -- an
// L2-resident working set -- instead of all of B streaming through L2 for
// every row of m blocks (row-major order re-read B from DRAM once per 2-3
// m-block rows on the large-N projections).
// Pairs: tiles from n_full on (the remainder of the last round, when it would
// leave more than half of the pairs idle) are cut into two 256 x 128 halves,
// items n_full, n_full + 1, ... of the walk: such a round loads 24 KB instead
// of 32 per k step and costs about 0.6 of a full one.
struct TileWalk {
    int tiles_m, tiles_n, n_full, n_items;
};
struct Tile {
    int m0, n0, w;                                   // first row, first column, columns
};
template <int BM, int BN>
__device__ __forceinline__ Tile tile_at(const TileWalk &tw, int item) {
    constexpr int GROUP_M = 16 * GEMM_BM / BM;
    Tile r{0, 0, BN};
    int t = item, sub = 0;
    if (BN == 256 && item >= tw.n_full) {
        t = tw.n_full + ((item - tw.n_full) >> 1);
        sub = (item - tw.n_full) & 1;
        r.w = 128;
    }
    const int per = GROUP_M * tw.tiles_n;
    const int grp = t / per;
    const int first = grp * GROUP_M;
    const int gm = min(GROUP_M, tw.tiles_m - first);
    const int loc = t - grp * per;
    r.m0 = (first + loc % gm) * BM;
    r.n0 = (loc / gm) * BN + sub * 128;
    return r;
}

template <int BN, int EPI, bool DEEP, bool WIDE>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ WeightMaps tmB,
                   const __grid_constant__ EpiMaps em, const EpiParams ep, const int K, const TileWalk tw,
                   const uint8_t *__restrict__ skip_flag, int *err) {
    using G = GemmTile<BN, EPI, DEEP, WIDE>;
    if (threadIdx.x == 0) {                           // kernel parameters: nothing a predecessor writes
        prefetch_tmap(&tmA);
        prefetch_tmap(WIDE ? &tmB.box256 : BN == 64 ? &tmB.box64 : &tmB.box128);
    }
    pdl_wait();
    if (skip_flag != nullptr && *skip_flag == XC_DEC_SKIP) return;
    // 1024-byte aligned (128B swizzle atoms): the declared alignment holds for
    // the window's base; nothing runs if it did not
    extern __shared__ __align__(1024) uint8_t smem[];
    if ((smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) atomicOr(err, ERR_BAD_LAUNCH);
        return;
    }
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + G::BAR_OFFSET);
    uint64_t *empty = full + G::STAGES;
    uint64_t *acc_full = empty + G::STAGES;    // [2]
    uint64_t *acc_empty = acc_full + 2;        // [2]
    uint64_t *ld_bar = acc_empty + 2;          // [8][SLOTS] residual operands of an epilogue warp's slot landed
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(ld_bar + 8 * EpiRing<EPI, DEEP, WIDE>::SLOTS);
    // pair: stages that the leader's and the peer's producer loaded, and that
    // the MMA warp has seen land; each written to both CTAs by its owner
    int *stages = reinterpret_cast<int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto publish = [&](int i, int v) {
        if (lane == 0)
            for (uint32_t r = 0; r < 2; ++r) st_cluster(map_to_cta(stages + i, r), v);
    };
    const int KT = K / GEMM_BK;
    constexpr bool PAIR = G::PAIR;
    // worker = CTA or CTA pair; rank 0 of a pair leads (issues its MMAs)
    const uint32_t rank = PAIR ? cluster_ctarank() : 0;
    const int worker = PAIR ? blockIdx.x >> 1 : blockIdx.x, n_workers = PAIR ? gridDim.x >> 1 : gridDim.x;
    const int row_off = PAIR ? (int)rank * GEMM_BM : 0;      // this CTA's rows of the tile

    if (threadIdx.x == 0) {
        for (int s = 0; s < G::STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], G::EPI_WARPS);
        }
        for (int w = 0; w < 8 * EpiRing<EPI, DEEP, WIDE>::SLOTS; ++w) mbar_init(&ld_bar[w], 1);
        mbar_fence_init();
    }
    if (warp == 1) {
        if constexpr (PAIR) tmem_alloc_pair(tmem_slot, G::TMEM_COLS);
        else tmem_alloc(tmem_slot, G::TMEM_COLS);
    }
    tc_fence_before();
    if constexpr (PAIR) cluster_sync_all();           // the peer's barriers are initialised too
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // The whole warp runs the loop (converged), one elected lane issues.
        int it = 0;
        bool ok = true;
        for (int item = worker; ok && item < tw.n_items; item += n_workers) {
            const Tile t = tile_at<G::BM, BN>(tw, item);
            const int m0 = t.m0 + row_off, n0 = PAIR ? t.n0 + (int)rank * (t.w / 2) : t.n0;
            const int b_rows = PAIR ? t.w / 2 : BN;           // of B
            const CUtensorMap *tb = WIDE ? &tmB.box256 : b_rows == 128 ? &tmB.box128 : &tmB.box64;
            const uint32_t bytes = (uint32_t)G::A_BYTES + (uint32_t)b_rows * (GEMM_BK * 2);
            for (int kt = 0; kt < KT; ++kt, ++it) {
                const int s = it % G::STAGES;
                const bool r = mbar_wait(&empty[s], ((it / G::STAGES) & 1) ^ 1, err, ERR_WAIT_PRODUCER);
                if (!__all_sync(0xffffffffu, r)) {
                    ok = false;
                    break;
                }
                uint8_t *sa = smem + s * G::STAGE_BYTES;
                if constexpr (PAIR)
                    tma_stage_pair_warp(&full[s], map_to_cta(&full[s], 0), rank == 0, 2 * bytes, sa, &tmA, m0,
                                        sa + G::A_BYTES, tb, n0, kt * GEMM_BK);
                else
                    tma_stage_warp(&full[s], bytes, sa, &tmA, m0, sa + G::A_BYTES, tb, n0, kt * GEMM_BK);
            }
        }
        // Drain: every copy this warp started has landed before exit (pairs: at
        // the end, from the counts of both).
        if constexpr (PAIR) {
            publish(rank, it);
        } else {
            for (int j = it - G::STAGES < 0 ? 0 : it - G::STAGES; j < it; ++j)
                mbar_wait(&full[j % G::STAGES], (j / G::STAGES) & 1, err, ERR_WAIT_PRODUCER);
        }
    } else if (warp == 1) {
        // MMA issue: the whole warp runs the loop (converged) and one elected
        // lane issues each tcgen05 instruction, so issue keeps pace while the
        // epilogue warps of the same sub-partitions are busy.
        if (rank == 0) {
            auto wait = [&](uint64_t *b, uint32_t parity) {
                const bool r = mbar_wait(b, parity, err, ERR_WAIT_MMA);
                return __all_sync(0xffffffffu, r);
            };
            // start-address field += offset >> 4 (shared addresses < 256 KB: no carry)
            const uint64_t d0 = sdesc_sw128(smem_u32(smem), 16, 1024);
            // Where few CTAs share the chip this loop's own chain of
            // instructions bounds a k step, whatever the tile's width and the
            // ring's depth.  So stage and parity are counted, not divided out of a
            // step number, and the next stage is looked at before the MMAs of this
            // one: 128 x 512 x 13824 42.0 -> 35.6 us, 486 x 1024 x 5888 19.8 -> 17.0,
            // 684 x 2816 x 4928 17.6 -> 15.6.  Not where the data is not there yet
            // when looked at: wide tiles wait for their 48 KB a step (2356 x 2048 x
            // 13824 87.8 us without, 89.5 with), and up to five steps are all in
            // the ring's first turn (7251 x 768 x 128 5.75 and 5.79, 584 x 7168 x
            // 320 6.34 and 6.40, 447 x 3072 x 384 4.49 and 4.46).  Two loops,
            // because a test of K inside one cost all of the gain.
            auto issue_tiles = [&](auto look) {
                int local = 0, s = 0, turns = 0;
                uint32_t ph = 0;
                bool ok = true, ready = false;
                for (int item = worker; ok && item < tw.n_items; item += n_workers, ++local) {
                    const int buf = local & 1;
                    const uint32_t use = (uint32_t)(local >> 1);
                    const uint32_t idesc = BN == 256 && item >= tw.n_full ? idesc_bf16(G::BM, 128, false, false)
                                                                          : idesc_bf16(G::BM, BN, false, false);
                    if (!wait(&acc_empty[buf], (use & 1) ^ 1)) break;
                    tc_fence_after();
                    const uint32_t acc = tmem + buf * BN;
                    for (int kt = 0; kt < KT; ++kt) {
                        if (!ready && !wait(&full[s], ph)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t da = d0 + (uint64_t)((s * G::STAGE_BYTES) >> 4);
                        const uint64_t db = da + (uint64_t)(G::A_BYTES >> 4);
                        uint64_t *const used = &empty[s];
                        if (++s == G::STAGES) {
                            s = 0;
                            ph ^= 1;
                            ++turns;
                        }
                        // (on every step: it says whether the next one need not wait)
                        if constexpr (decltype(look)::value) ready = __all_sync(0xffffffffu, mbar_test(&full[s], ph));
#pragma unroll
                        for (int k = 0; k < GEMM_BK / 16; ++k) {
                            if constexpr (PAIR) tc_mma_pair_warp(acc, da + 2 * k, db + 2 * k, idesc, (kt | k) != 0 ? 1u : 0u);
                            else tc_mma_warp(acc, da + 2 * k, db + 2 * k, idesc, (kt | k) != 0 ? 1u : 0u);
                        }
                        if constexpr (PAIR) tc_commit_pair_warp(used);
                        else tc_commit_warp(used);
                    }
                    if constexpr (PAIR) tc_commit_pair_warp(&acc_full[buf]);
                    else tc_commit_warp(&acc_full[buf]);
                }
                if constexpr (PAIR) publish(2, turns * G::STAGES + s);
            };
            if (WIDE || KT <= 5) issue_tiles(std::false_type{});
            else issue_tiles(std::true_type{});
        }
    } else {
        // ---------------------------------------------------------- epilogue (warps 2..9)
        // Warp ew = warp - 2 owns TMEM lane quadrant q (rows q*32 .. q*32+31 of
        // the tile; thread = row) and column half `half`, in 32-column blocks.
        using E = EpiRing<EPI, DEEP, WIDE>;
        const int ew = warp - 2;
        const int q = warp & 3;
        const int half = ew >> 2;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        uint8_t *eb = smem + G::OFF_EPI + ew * E::SLOTS * E::SLOT_BYTES;
        float *vec = reinterpret_cast<float *>(smem + G::OFF_VEC) + ew * 64;     // bias [32], gate [32]
        uint64_t *lb = ld_bar + ew * E::SLOTS;
        const bool has_rhat = E::CACHE && ep.rhat != nullptr;
        const int roff = row_off + q * 32;
        int n = 0, n_ld = 0;                             // blocks done, residual loads issued
        auto load_res = [&](int m, int col) {            // lane 0: residual operands of block n_ld
            if constexpr (E::RES) {
                uint8_t *s = eb + (n_ld % E::SLOTS) * E::SLOT_BYTES;
                uint64_t *b = &lb[n_ld % E::SLOTS];
                mbar_expect_tx(b, (uint32_t)EPI_BLOCK_BYTES * (has_rhat ? 2u : 1u));
                tma_load_2d(s, &em.resid, b, col, m);
                if (has_rhat) tma_load_2d(s + EPI_BLOCK_BYTES, &em.xin, b, col, m);
            }
        };
        bool ok = true;
        Tile nt{0, 0, BN};                               // the next tile
        if (worker < tw.n_items) {
            nt = tile_at<G::BM, BN>(tw, worker);
            if constexpr (E::RES)
                for (; n_ld < E::AHEAD; ++n_ld)
                    if (lane == 0) load_res(nt.m0 + roff, nt.n0 + half * (nt.w / 2) + 32 * n_ld);
        }
        int local = 0;
        for (int item = worker; ok && item < tw.n_items; item += n_workers, ++local) {
            const int buf = local & 1;
            const uint32_t use = (uint32_t)(local >> 1);
            const int coff = half * (nt.w / 2), n_blk = nt.w / 64;   // this warp's columns, 32 at a time
            const int m0 = nt.m0 + roff, c0 = nt.n0 + coff;
            const bool more = item + n_workers < tw.n_items;
            if (more) nt = tile_at<G::BM, BN>(tw, item + n_workers);
            const int row = m0 + lane;
            // RoPE position of this thread's row (camera, frame, h, w), once per tile
            int pos0 = 0, pos1 = 0, pos2 = 0, pos3 = 0;
            if constexpr (EPI == EPI_QKV_ROPE) {
                const int4 tp = token_pos(ep, row);
                pos0 = tp.x;
                pos1 = tp.y;
                pos2 = tp.z;
                pos3 = tp.w;
            }
            // bias (and gate) of a block's columns: one value per lane, fetched
            // a block ahead, read back by every lane from shared memory
            float b_next = ep.bias[c0 + lane];
            float g_next = 0.0f;
            if constexpr (E::RES) g_next = ep.gate[c0 + lane];
            ok = mbar_wait(&acc_full[buf], use & 1, err, ERR_WAIT_EPI);
            __syncwarp();
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            tc_fence_after();
#pragma unroll 1
            for (int j = 0; j < n_blk; ++j, ++n) {
                const int col = c0 + 32 * j;
                uint8_t *s_out = eb + (n % E::SLOTS) * E::SLOT_BYTES;
                vec[lane] = b_next;
                if constexpr (E::RES) vec[32 + lane] = g_next;
                if (j + 1 < n_blk) {
                    b_next = ep.bias[col + 32 + lane];
                    if constexpr (E::RES) g_next = ep.gate[col + 32 + lane];
                }
                if constexpr (E::RES) {
                    // operands of block n + AHEAD, into the slot whose last
                    // store (block n + AHEAD - SLOTS) has been read
                    const int ja = j + E::AHEAD;
                    if (ja < n_blk || more) {
                        if (lane == 0) {
                            bulk_wait_read<E::SLOTS - E::AHEAD - 1>();
                            if (ja < n_blk) load_res(m0, c0 + 32 * ja);
                            else load_res(nt.m0 + roff, nt.n0 + half * (nt.w / 2) + 32 * (ja - n_blk));
                        }
                        ++n_ld;
                    }
                } else {
                    if (lane == 0) bulk_wait_read<E::SLOTS - 1>();     // the slot's last store (block n - SLOTS) has been read
                }
                float v[32];
                tmem_ld32_sync(tq + buf * BN + coff + 32 * j, v);
                if (j == n_blk - 1) tc_fence_before();
                __syncwarp();
                // last TMEM read of this tile: hand the accumulator back
                if (j == n_blk - 1 && lane == 0) {
                    if constexpr (PAIR) mbar_arrive_cluster(map_to_cta(&acc_empty[buf], 0));
                    else mbar_arrive(&acc_empty[buf]);
                }
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const float4 b4 = *reinterpret_cast<const float4 *>(vec + i);
                    add2(v[i], v[i + 1], b4.x, b4.y);
                    add2(v[i + 2], v[i + 3], b4.z, b4.w);
                }
                float xi[32];
                if constexpr (E::RES) {
                    ok = mbar_wait(&lb[n % E::SLOTS], (n / E::SLOTS) & 1, err, ERR_WAIT_EPI);
                    __syncwarp();
                    if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                    float r[32];
                    read_row32(s_out, lane, r);
                    if constexpr (E::CACHE)
                        if (has_rhat) read_row32(s_out + EPI_BLOCK_BYTES, lane, xi);
#pragma unroll
                    for (int i = 0; i < 32; i += 4) {
                        const float4 g4 = *reinterpret_cast<const float4 *>(vec + 32 + i);
                        fma2(v[i], v[i + 1], g4.x, g4.y, r[i], r[i + 1]);
                        fma2(v[i + 2], v[i + 3], g4.z, g4.w, r[i + 2], r[i + 3]);
                    }
                }
                if constexpr (EPI == EPI_GELU) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) gelu_tanh_approx2(v[i], v[i + 1]);
                }
                int part = 0, cl = col;
                if constexpr (EPI == EPI_QKV_ROPE) {
                    part = col / ep.d;
                    cl = col - part * ep.d;
                    if (part < 2 && row < ep.M) {
                        const int pair0 = (cl % ep.head_dim) >> 1;
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const int pr = pair0 + k;
                            const int ax = ep.rope_axis[pr];
                            const int pa = ax == 0 ? pos0 : (ax == 1 ? pos1 : (ax == 2 ? pos2 : pos3));
                            const float2 t = ep.rope_cs[ep.rope_off[pr] + pa];
                            const float x0 = v[2 * k], x1 = v[2 * k + 1];
                            v[2 * k] = x0 * t.x - x1 * t.y;
                            v[2 * k + 1] = x0 * t.y + x1 * t.x;
                        }
                    }
                }
                write_row32(s_out, lane, v);
                if constexpr (E::CACHE) {
                    if (has_rhat) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = round_to<bf16>(v[i]) - xi[i];
                        write_row32(s_out + EPI_BLOCK_BYTES, lane, v);
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&em.out[part], s_out, cl, m0);
                    if constexpr (E::CACHE)
                        if (has_rhat) tma_store_2d(&em.rhat, s_out + EPI_BLOCK_BYTES, col, m0);
                    bulk_commit();
                }
            }
        }
        // residual loads still in flight when a wait ran out
        if constexpr (E::RES) {
            if (!ok && lane == 0)
                for (int k = n_ld - E::SLOTS < 0 ? 0 : n_ld - E::SLOTS; k < n_ld; ++k)
                    mbar_wait(&lb[k % E::SLOTS], (k / E::SLOTS) & 1, err, ERR_WAIT_EPI);
        }
        // every TMA store of this warp has completed before the CTA exits
        if (lane == 0) bulk_wait_all();
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) {
        cluster_sync_all();                           // no MMA, commit or arrival of the pair still to come
        // Where a wait ran out, stages are left that no MMA has waited for, and
        // one CTA may have loaded some that the other has not.  The leader makes
        // up their count, so that their phases complete when the copies in flight
        // land, and waits for them; the peer leaves after it.
        const int n0 = stages[0], n1 = stages[1], seen = stages[2];
        if (n0 != seen || n1 != seen) {
            if (rank == 0 && threadIdx.x == 0) {
                for (int j = seen; j < max(n0, n1); ++j) {
                    const Tile t = tile_at<G::BM, BN>(tw, worker + j / KT * n_workers);
                    const uint32_t bytes = (uint32_t)G::A_BYTES + (uint32_t)(t.w / 2) * (GEMM_BK * 2);
                    uint64_t *b = &full[j % G::STAGES];
                    if (j >= n1) mbar_complete_tx(b, bytes);       // expected of the peer
                    if (j >= n0) mbar_expect_tx(b, bytes);         // the peer's alone
                    mbar_wait(b, (j / G::STAGES) & 1, err, ERR_WAIT_PRODUCER);
                }
            }
            __syncthreads();
            cluster_sync_all();
        }
    }
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem, G::TMEM_COLS);
        else tmem_dealloc(tmem, G::TMEM_COLS);
    }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static std::atomic<EncodeTiledFn> known{nullptr};
    EncodeTiledFn fn = known.load(std::memory_order_relaxed);
    if (fn == nullptr) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        known.store(fn, std::memory_order_relaxed);
    }
    return fn;
}

// 2-D bf16 tensor map over a row-major [rows][cols] matrix, zero fill outside
// it.  The driver call needs a current context, which a host thread that has
// made no runtime call that works on the device does not have: it gets the
// device's primary one, as such a runtime call would give it.
static bool make_tmap(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows,
                      uint32_t box_cols, CUtensorMapSwizzle swizzle) {
    EncodeTiledFn fn = encode_fn();
    if (fn == nullptr) return false;
    if ((reinterpret_cast<uintptr_t>(base) & 15) != 0 || (cols * 2) % 16 != 0) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t estr[2] = {1, 1};
    auto encode = [&] {
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode();
    if (r == CUDA_ERROR_INVALID_CONTEXT || r == CUDA_ERROR_NOT_INITIALIZED) {
        int dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = encode();
    }
    return r == CUDA_SUCCESS;
}
// Box [box_rows][64], 128-byte swizzle (operands).
bool make_tmap_bf16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    return make_tmap(m, base, rows, cols, box_rows, 64, CU_TENSOR_MAP_SWIZZLE_128B);
}
// Box [32][32], 64-byte swizzle (epilogue blocks).
static bool make_tmap_epi(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols) {
    return cols % 32 == 0 && make_tmap(m, base, rows, cols, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
}

// Encoded epilogue maps, looked up by (base, rows, cols): the chunk step
// reuses the same activation buffers on every pass, so encoding happens once
// per buffer.
namespace {
struct MapKey {
    const void *base;
    uint64_t rows, cols;
    bool operator==(const MapKey &o) const { return base == o.base && rows == o.rows && cols == o.cols; }
};
struct MapKeyHash {
    size_t operator()(const MapKey &k) const {
        return std::hash<const void *>()(k.base) ^ (size_t)(k.rows * 0x9E3779B97F4A7C15ull) ^ (size_t)(k.cols << 17);
    }
};
std::mutex g_map_mu;
std::unordered_map<MapKey, CUtensorMap, MapKeyHash> g_maps;
}  // namespace

static bool epi_map(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols) {
    if (base == nullptr) {                         // unused slot: any valid map
        memset(m, 0, sizeof(*m));
        return true;
    }
    std::lock_guard<std::mutex> lk(g_map_mu);
    const MapKey key{base, rows, cols};
    auto it = g_maps.find(key);
    if (it != g_maps.end()) {
        *m = it->second;
        return true;
    }
    if (g_maps.size() > 4096) g_maps.clear();
    if (!make_tmap_epi(m, base, rows, cols)) return false;
    g_maps.emplace(key, *m);
    return true;
}

template <int EPI>
static bool build_epi_maps(EpiMaps &em, const EpiParams &ep) {
    memset(&em, 0, sizeof(em));
    if constexpr (EPI == EPI_QKV_ROPE) {
        return epi_map(&em.out[0], ep.out, ep.M, ep.d) && epi_map(&em.out[1], ep.out_k, ep.M, ep.d) &&
               epi_map(&em.out[2], ep.out_v, ep.M, ep.d);
    } else {
        bool ok = epi_map(&em.out[0], ep.out, ep.M, ep.N);
        if constexpr (EPI == EPI_RESID_GATE || EPI == EPI_RESID_CACHE) ok = ok && epi_map(&em.resid, ep.resid, ep.M, ep.N);
        if constexpr (EPI == EPI_RESID_CACHE) {
            if (ep.rhat != nullptr)
                ok = ok && epi_map(&em.rhat, ep.rhat, ep.M, ep.N) && epi_map(&em.xin, ep.xin, ep.M, ep.N);
        }
        return ok;
    }
}

// CTA pairs resident at once (both CTAs of a pair sit on neighbouring SMs); the
// same for every pair kernel, whose shared memory leaves room for one CTA on an
// SM.  The tiling rule and the launch walk with the same count.
static int pair_count() {
    static PerDevice known;
    return known.get([] {
        using G = GemmTile<256, EPI_BIAS, false, false>;
        auto kern = gemm_tc_kernel<256, EPI_BIAS, false, false>;
        static PerDevice smem_done;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * (sm_count() / 2));
        cfg.blockDim = dim3(GEMM_THREADS);
        cfg.dynamicSmemBytes = G::SMEM_BYTES;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int k = 0;
        if (allow_smem(smem_done, kern, G::SMEM_BYTES) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&k, kern, &cfg) != cudaSuccess || k < 1) {
            cudaGetLastError();
            k = sm_count() / 2;
        }
        return k < 1 ? 1 : k;
    });
}

// Walk of a pair grid over 256 x 256 tiles: a remainder of at most half of
// the pairs is cut into halves.
static TileWalk pair_walk(int M, int N, int workers) {
    TileWalk tw;
    tw.tiles_m = (M + 255) / 256;
    tw.tiles_n = N / 256;
    const int n = tw.tiles_m * tw.tiles_n, rem = n % workers;
    tw.n_full = 2 * rem <= workers ? n - rem : n;
    tw.n_items = tw.n_full + 2 * (n - tw.n_full);
    return tw;
}

// Output tiling for an M x N x K GEMM: 256 (CTA pairs), GEMM_WIDE, 128 or 64
// (single CTAs).  Half the pairs' worth of 256 x 256 tiles and fewer are one
// round of single tiles, 64 wide while those find an SM each.  Beyond, the cost
// in SM cycles of the persistent rounds: a 64-deep k step takes about 555
// cycles on a full pair tile, 340 on a half one, 640 on a wide single tile, 450
// on a 128-wide one with every SM busy (bound by the operand feed); no round is
// shorter than its epilogue, the last one's is added, and setting up a pair
// takes some 1500 more, 3500 where a few row blocks make most of B a tile's
// own.  Wide tiles are for row counts that leave the pairs a ragged round.
// Measured, pair / wide / 128-wide: gated residual 2356 x 2048 x 3392 30.7 /
// 20.5 / 24.4 us, 1900 x 2560 x 6144 52.3 / 37.3 / 40.5, 500 x 9728 x 1536 13.4
// / 12.3 / 13.7, 4800 x 4096 x 2048 47.6 / 52.8 / 60.1, 12960 x 5120 x 5120 363 /
// 411 / 453, 9728 x 512 x 512 8.6 / 7.8 / 7.7; residual cache 2356 x 2048 x 3392
// 33.2 / 24.0 / 27.1, x 1024 16.6 / 13.3 / 12.6, 7200 x 2560 x 1024 40.5 / 43.7 /
// 48.7; 239 x 12032 x 3712 22.0 / - / 27.7.
int gemm_tc_bn(int epi, int M, int N, int K) {
    const long n_sm = sm_count(), pairs = pair_count();
    const long tm = (M + 127) / 128, t128 = tm * (N / 128), r128 = (t128 + n_sm - 1) / n_sm;
    if (2 * t128 <= n_sm) return 64;
    if (N % 256 != 0) return 128;
    const TileWalk tw = pair_walk(M, N, (int)pairs);
    if (tw.n_full == 0) return 128;
    const long r_full = (tw.n_full + pairs - 1) / pairs, r_half = tw.n_items > tw.n_full ? 1 : 0;
    const long r_wide = (tm * (N / 256) + n_sm - 1) / n_sm;
    const long kt = K / GEMM_BK;
    const long e_full = epi == EPI_RESID_CACHE ? 12000 : 4500, e_half = epi == EPI_RESID_CACHE ? 6000 : 2500;
    const long pair = r_full * std::max(kt * 555, e_full) + r_half * std::max(kt * 340, e_half) +
                      (r_half ? e_half : e_full) + (tw.tiles_m <= 4 ? 3500 : 1500);
    const long e_wide = epi == EPI_RESID_CACHE ? 14000 : 4500;
    const long wide = r_wide * std::max(kt * 640, e_wide) + e_wide;
    const long narrow = r128 * std::max(kt * 450, e_half) + e_half;
    if (wide < pair && 20 * wide < 19 * narrow) return GEMM_WIDE;
    return pair <= narrow ? 256 : 128;
}

static TileWalk tile_walk(int bn, int M, int N) {
    if (bn == 256) return pair_walk(M, N, pair_count());
    TileWalk tw;
    tw.tiles_m = (M + GEMM_BM - 1) / GEMM_BM;
    tw.tiles_n = N / (bn == GEMM_WIDE ? 256 : bn);
    tw.n_full = tw.n_items = tw.tiles_m * tw.tiles_n;
    return tw;
}
void gemm_tc_tiles(int bn, int M, int N, int *full, int *half) {
    const TileWalk tw = tile_walk(bn, M, N);
    *full = tw.n_full;
    *half = tw.n_items - tw.n_full;
}

template <int EPI, int BN, bool DEEP = false, bool WIDE = false>
static cudaError_t launch_tc(const CUtensorMap &ta, const WeightMaps &tb, const EpiParams &ep, int K,
                             const uint8_t *skip, int *err, cudaStream_t st) {
    using G = GemmTile<BN, EPI, DEEP, WIDE>;
    auto kern = gemm_tc_kernel<BN, EPI, DEEP, WIDE>;
    EpiMaps em;
    if (!build_epi_maps<EPI>(em, ep)) return cudaErrorInvalidValue;
    static PerDevice smem_done;
    const cudaError_t e = allow_smem(smem_done, kern, G::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    int workers = G::PAIR ? pair_count() : sm_count();
    const TileWalk tw = tile_walk(WIDE ? GEMM_WIDE : BN, ep.M, ep.N);
    if (tw.n_items < workers) workers = tw.n_items;
    return launch_pdl_cluster(kern, G::PAIR ? 2 : 1, dim3(G::PAIR ? 2 * workers : workers), dim3(GEMM_THREADS), G::SMEM_BYTES, st,
                              ta, tb, em, ep, K, tw, skip, err);
}

template <int BN, bool WIDE = false>
static cudaError_t gemm_tc_bn_(int epi, const CUtensorMap &ta, const WeightMaps &tb, const EpiParams &ep, int K,
                               const uint8_t *skip, int *err, cudaStream_t st) {
    switch (epi) {
        case EPI_BIAS: return launch_tc<EPI_BIAS, BN, false, WIDE>(ta, tb, ep, K, skip, err, st);
        case EPI_GELU: return launch_tc<EPI_GELU, BN, false, WIDE>(ta, tb, ep, K, skip, err, st);
        case EPI_RESID_GATE:
            if constexpr (BN == 64 || WIDE) return launch_tc<EPI_RESID_GATE, BN, false, WIDE>(ta, tb, ep, K, skip, err, st);
            else return K < 1536 ? launch_tc<EPI_RESID_GATE, BN, true>(ta, tb, ep, K, skip, err, st)
                                 : launch_tc<EPI_RESID_GATE, BN>(ta, tb, ep, K, skip, err, st);
        case EPI_RESID_CACHE: return launch_tc<EPI_RESID_CACHE, BN, false, WIDE>(ta, tb, ep, K, skip, err, st);
        case EPI_QKV_ROPE: return launch_tc<EPI_QKV_ROPE, BN, false, WIDE>(ta, tb, ep, K, skip, err, st);
        default: return cudaErrorInvalidValue;
    }
}

// Entry used by the chunk step and xc_op_linear / xc_op_qkv_rope (bf16 only).
// `ta` covers A [M][K] (boxes of 128 rows), `tb` Wt [N][K]; bn =
// gemm_tc_bn(epi, M, N, K); N a multiple of the tile's width, K % 64 == 0.
cudaError_t gemm_tc(int epi, int bn, const CUtensorMap &ta, const WeightMaps &tb, const EpiParams &ep, int K,
                    const uint8_t *skip, int *err, cudaStream_t st) {
    if (bn == GEMM_WIDE) return gemm_tc_bn_<256, true>(epi, ta, tb, ep, K, skip, err, st);
    if (bn == 256) return gemm_tc_bn_<256>(epi, ta, tb, ep, K, skip, err, st);
    if (bn == 128) return gemm_tc_bn_<128>(epi, ta, tb, ep, K, skip, err, st);
    if (bn == 64) return gemm_tc_bn_<64>(epi, ta, tb, ep, K, skip, err, st);
    return cudaErrorInvalidValue;
}

}  // namespace xc
