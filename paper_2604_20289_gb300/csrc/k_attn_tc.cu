// Flash attention on the tcgen05 tensor core (bf16 in, fp32 softmax / accumulate).
//
//   o = softmax(q k^T / sqrt(hd)) v   per head, no mask inside the window:
//   the current chunk's queries see every resident key of the rolling KV
//   cache (past chunks' clean K/V plus the current chunk's own K/V).
//
// One CTA = two 128-query tiles (Q0, Q1) of one head, 352 threads:
//   warps 0..3  softmax WG 0 (tile Q0), thread = query row = TMEM lane;
//   warps 4..7  softmax WG 1 (tile Q1);
//   warp 8      TMA producer: Q0/Q1 once, then 128-key K and V tiles through
//               a STAGES-deep ring (separate K and V barriers);
//   warp 9      TMEM allocation; MMA issue (hd 64: tile Q0; hd 128: both);
//   warp 10     hd 64: MMA issue for tile Q1 (MMA warps run converged, one
//               elected lane issuing each instruction).
// TMEM: S0 [0,128), S1 [128,256), O0 [256, 256+hd), O1 after it.  P (bf16)
// goes back into TMEM and feeds tcgen05.mma as the A operand straight from
// tensor memory (no shared-memory round trip); V is read MN-major from its
// [keys][hd] tile.
//   hd = 64 : P0 / P1 have their own 64 columns ([384,448), [448,512)), so
//             S_{j+1} is issued as soon as the softmax has READ S_j and runs on
//             the tensor core while the softmax computes P_j.
//   hd = 128: TMEM is full (S0 S1 O0 O1 = 512 columns); P_i overwrites S_i and
//             S_{j+1} waits until P_j V has been issued; the two tiles
//             ping-pong so the tensor core still has the other tile's work.
// At head_dim 64 the two softmax warps of each SM sub-partition (one per
// tile) take turns on the MUFU-bound exponential phase.
// Online softmax in the exp2 domain with lazy rescaling: a row's O and sum
// are rescaled only when its running max grows by more than 8 (hd 64), or
// when a tile's row sum passes 2^15 under the max in use (hd 128).  Score
// scaling and row sums use packed fp32 pairs (FFMA2 / FADD2).  Keys beyond
// n_keys (ragged last tile) are masked to -inf; their K/V rows are finite
// (zero-initialised ring, TMA zero fill).
#include <algorithm>

#include "xc_ptx.cuh"

namespace xc {

template <int HD>
struct AttnTile {
    static constexpr int BQ = 128, BKV = 128, QT = 2;
    static constexpr int NR = HD / 64;                 // 64-wide swizzle regions per row
    static constexpr int REGION = 128 * 128;           // [128 rows][64 bf16]
    static constexpr int Q_BYTES = NR * REGION;        // one 128-row Q tile
    static constexpr int KV_BYTES = NR * REGION;       // one 128-key K or V tile
    static constexpr int STAGES = HD == 64 ? 4 : 2;
    static constexpr int OFF_K = QT * Q_BYTES;
    static constexpr int OFF_V = OFF_K + STAGES * KV_BYTES;
    static constexpr int OFF_O = OFF_V + STAGES * KV_BYTES;    // output staging, 4 KB per softmax warp
    static constexpr int OFF_BAR = OFF_O + 8 * 4096;
    static constexpr int SMEM_BYTES = OFF_BAR + 512 + 1024;
    static constexpr int TMEM_COLS = 512;
    static constexpr int THREADS = 352;            // 8 softmax, 1 TMA, 2 MMA warps
    static constexpr bool SEP_P = HD == 64;            // P has its own TMEM columns
    static constexpr int ISSUERS = SEP_P ? 2 : 1;      // MMA-issuing warps (9, 10)
    __host__ __device__ static constexpr int S_COL(int i) { return 128 * i; }
    __host__ __device__ static constexpr int O_COL(int i) { return 256 + HD * i; }
    __host__ __device__ static constexpr int P_COL(int i) { return SEP_P ? 256 + 2 * HD + 64 * i : 128 * i; }
    static constexpr float LAZY = 8.0f;                // hd 64: rescale threshold (log2 units)
    // hd 128: limit of a tile's row sum, that of 128 keys 2^LAZY above the max in
    // use, so that O and l have the same range at both head dims: n_kt tiles of
    // values below 2^112 / n_kt stay finite
    static constexpr float RAISE = 32768.0f;
};

__device__ __forceinline__ uint8_t *align1024_a(uint8_t *p) {
    const uint32_t s = smem_u32(p);
    return p + ((1024u - (s & 1023u)) & 1023u);
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// Max of a 128-column score row: 16 independent chains of three-input max over
// columns 0..111, the last 16 columns, then a tree.
__device__ __forceinline__ float row_max(const float (&s)[128]) {
    float mx[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) mx[k] = s[k];
#pragma unroll
    for (int c = 16; c < 112; c += 32) {
#pragma unroll
        for (int k = 0; k < 16; ++k) mx[k] = fmax3(mx[k], s[c + k], s[c + 16 + k]);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) mx[k] = fmaxf(mx[k], s[112 + k]);
#pragma unroll
    for (int k = 0; k < 5; ++k) mx[k] = fmax3(mx[k], mx[k + 5], mx[k + 10]);
    return fmax3(fmax3(mx[0], mx[1], mx[2]), fmax3(mx[3], mx[4], mx[15]), mx[0]);
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Probabilities 2^(s * sl2 - m) of the 32 scores of quarter qt, packed to bf16
// pairs and stored to TMEM; their sums go to rs0, rs1.
__device__ __forceinline__ void exp_quarter(const float (&s)[128], int qt, float sl2, float m, uint32_t tP,
                                            float2 &rs0, float2 &rs1) {
    const float2 sc2 = make_float2(sl2, sl2), nm2 = make_float2(-m, -m);
    uint32_t w[16];
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
        const int c = 32 * qt + 2 * k;
        const float2 a = __ffma2_rn(make_float2(s[c], s[c + 1]), sc2, nm2);
        const float2 b = __ffma2_rn(make_float2(s[c + 2], s[c + 3]), sc2, nm2);
        const float2 pa = make_float2(ex2_approx(a.x), ex2_approx(a.y));
        const float2 pb = make_float2(ex2_approx(b.x), ex2_approx(b.y));
        rs0 = __fadd2_rn(rs0, pa);
        rs1 = __fadd2_rn(rs1, pb);
        __nv_bfloat162 h0 = __floats2bfloat162_rn(pa.x, pa.y);
        __nv_bfloat162 h1 = __floats2bfloat162_rn(pb.x, pb.y);
        w[k] = *reinterpret_cast<uint32_t *>(&h0);
        w[k + 1] = *reinterpret_cast<uint32_t *>(&h1);
    }
    tmem_st16u_sync(tP + 16 * qt, w);
}

// Work split.  A unit is (head, pair of 128-query tiles), u = head * n_qblk +
// qblk, with n_kt key tiles, walked by G CTAs (one per SM) in one of three
// orders:
//  * contiguous (ORDER_CONTIGUOUS): the (unit, key tile) iteration space, T =
//    n_units * n_kt, is cut into the contiguous shares [c T / G,
//    (c + 1) T / G).  A unit cut by the boundary between CTAs c - 1 and c is
//    finished by both as an unnormalised partial O with its running max m
//    and sum l (a flash-decoding partial, slot (boundary c, head / tail)),
//    and attn_combine_kernel merges the two.  Every share is at least one
//    unit, so a unit is cut at most once.  The units in flight span every
//    head, so each unit streams its head's K / V from DRAM once the heads'
//    K / V exceed L2.
//  * waves (ORDER_WAVE): CTA c runs the whole units c, c + G, ..., W of
//    them and one more if c < R -- the CTAs running at one time share a few
//    heads and each K / V tile comes from DRAM once per wave -- and, where
//    T2 > 0 (then R = 0), the key tiles of the remaining units, T2 of them,
//    are split evenly: CTA c takes [c T2 / G, (c + 1) T2 / G), at most one
//    unit's worth, touching at most two units (its pieces W and W + 1,
//    partial slots 2 c and 2 c + 1), merged per remaining unit by
//    attn_combine_kernel.  With fewer units than SMs W = 0: every unit is
//    such a remaining one.
//  * clusters (ORDER_CLUSTER): as waves with W = 0 and every unit cut evenly
//    over the CTAs of one thread-block cluster, which leave their partials in
//    their shared memory and merge them there -- no second launch and no
//    partials through global memory.
// Each role walks the CTA's key tiles with a cursor (TileCursor): tile
// counter g, unit u and its key tile k; in the wave order also the piece
// index p and the unit step du.
struct AttnSplit {
    long long T;          // contiguous: total iterations
    long long T2;         // waves: key tiles of the remaining units, split evenly
    int n_kt, n_qblk, G, W, R;
    __host__ __device__ long long begin(int c) const { return T * c / G; }
    __host__ __device__ long long begin2(int c) const { return T2 * c / G; }
};
struct TileCursor {
    int g, u, k;          // tile counter, unit, key tile of the unit
    int p, du;            // waves: piece index, unit step (G over the waves, 1 in the remainder)
};
// Waves: pieces W and W + 1 of CTA c (its share of the remaining units) --
// first key tile of piece W, end key tiles of both (0: no such piece), and
// the unit of piece W.
struct RemSeg {
    int k0, k1a, k1b, u;
};
__device__ __forceinline__ RemSeg rem_seg(const AttnSplit &sp, int c) {
    const int nkt = sp.n_kt;
    RemSeg r{0, 0, 0, 0};
    const long long b = sp.begin2(c), e = sp.begin2(c + 1);
    if (b == e) return r;
    const long long ub = b / nkt, bnd = (ub + 1) * nkt;
    r.u = sp.W * sp.G + (int)ub;
    r.k0 = (int)(b - ub * nkt);
    r.k1a = (int)(e < bnd ? e - ub * nkt : nkt);
    r.k1b = (int)(e > bnd ? e - bnd : 0);
    return r;
}

// Partials: slot sl's O as 4 KB blocks [softmax warp 0..7][32-column group][32
// rows][32 fp32], the 16-byte chunks of a row permuted by its row number (so
// that a lane writes its row to shared memory without bank conflicts and the
// block leaves as one bulk copy).
__host__ __device__ constexpr size_t partial_block(int slot, int warp, int grp, int hd) {
    return ((size_t)(slot * 8 + warp) * (hd / 32) + grp) * 1024;
}

__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)),
                 "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}

// Work orders of attn_tc_kernel (see AttnSplit).
enum { ORDER_CONTIGUOUS = 0, ORDER_WAVE = 1, ORDER_CLUSTER = 2 };

template <int HD, int ORDER>
__global__ void __launch_bounds__(352, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO, const int Lq,
                   const int n_keys, const AttnSplit sp, float *__restrict__ ws_o, float2 *__restrict__ ws_ml,
                   const uint8_t *__restrict__ skip_flag, int *err, bf16 *__restrict__ o, const int d) {
    constexpr bool WAVE = ORDER != ORDER_CONTIGUOUS, CLUSTER = ORDER == ORDER_CLUSTER;
    pdl_wait();
    using A = AttnTile<HD>;
    if (skip_flag != nullptr && *skip_flag == XC_DEC_SKIP) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = align1024_a(smem_raw);
    uint8_t *sQ = smem;
    uint8_t *sK = smem + A::OFF_K;
    uint8_t *sV = smem + A::OFF_V;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + A::OFF_BAR);
    uint64_t *q_full = bar;                    // Q of piece p landed (phase p)
    uint64_t *q_empty = bar + 1;               // every S MMA of piece p done (phase p)
    uint64_t *k_full = bar + 2;
    uint64_t *k_empty = k_full + A::STAGES;
    uint64_t *v_full = k_empty + A::STAGES;
    uint64_t *v_empty = v_full + A::STAGES;
    uint64_t *s_full = v_empty + A::STAGES;    // [2] S_i computed
    uint64_t *s_cons = s_full + 2;             // [2] S_i read by its softmax WG (hd 64)
    uint64_t *p_full = s_cons + 2;             // [2] P_i written, O_i corrected
    uint64_t *pv_done = p_full + 2;            // [2] P_i V done (hd 64: every tile; hd 128: last of a piece)
    uint64_t *o_free = pv_done + 2;            // [2] O_i of piece p read out (phase p)
    uint64_t *turn = o_free + 2;               // [2][4] exponential-phase hand-off per (WG, quadrant)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(turn + 8);
    uint64_t *all_pv = turn + 9;               // clusters: every P V of the CTA done (its K / V ring is free)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkt = sp.n_kt;
    const int cta = blockIdx.x;
    long long it0 = 0;
    int n_t;                                       // key tiles of this CTA (>= 1)
    const int n_whole = sp.W + (cta < sp.R ? 1 : 0);   // waves: whole units of this CTA
    if constexpr (WAVE) {
        n_t = n_whole * nkt + (int)(sp.begin2(cta + 1) - sp.begin2(cta));
    } else {
        it0 = sp.begin(cta);
        n_t = (int)(sp.begin(cta + 1) - it0);
    }
    const int u0 = (int)(it0 / nkt);
    // Waves: this CTA's remainder pieces (registers of the cursor roles),
    // and the tile at which its remainder begins.  The cursor steps like the
    // contiguous one -- next unit after a unit's last key tile -- with a jump
    // to the remainder at tile gw, so the per-tile tests stay the same.
    RemSeg rem{0, 0, 0, 0};
    if constexpr (WAVE) rem = rem_seg(sp, cta);
    const int gw = WAVE ? n_whole * nkt : -1;
    TileCursor c0{0, u0, (int)(it0 % nkt), 0, 1};
    if constexpr (WAVE) c0 = n_whole > 0 ? TileCursor{0, cta, 0, 0, sp.G} : TileCursor{0, rem.u, rem.k0, 0, 1};
    auto piece_of = [&](const TileCursor &c) {    // index of the cursor's piece in this CTA
        if constexpr (WAVE) return c.p;
        else return c.u - u0;
    };
    auto first_of = [&](const TileCursor &c) {
        if constexpr (WAVE) return c.k == 0 || c.g == gw;
        else return c.g == 0 || c.k == 0;
    };
    auto last_of = [&](const TileCursor &c) { return c.g == n_t - 1 || c.k == nkt - 1; };
    auto next = [&](TileCursor &c) {
        ++c.g;
        if (++c.k == nkt) {
            c.k = 0;
            if constexpr (WAVE) {
                c.u += c.du;
                ++c.p;
            } else {
                ++c.u;
            }
        }
        if constexpr (WAVE) {
            if (c.g == gw) {
                c.u = rem.u;
                c.k = rem.k0;
                c.du = 1;
                c.p = sp.W;
            }
        }
    };

    if (threadIdx.x == 0) {
        mbar_init(q_full, 1);
        mbar_init(q_empty, A::ISSUERS);
        if constexpr (CLUSTER) mbar_init(all_pv, 256);
        for (int s = 0; s < A::STAGES; ++s) {
            mbar_init(&k_full[s], 1);
            mbar_init(&k_empty[s], A::ISSUERS);   // freed by every MMA warp
            mbar_init(&v_full[s], 1);
            mbar_init(&v_empty[s], A::ISSUERS);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_full[i], 1);
            mbar_init(&s_cons[i], 128);
            mbar_init(&p_full[i], 128);
            mbar_init(&pv_done[i], 1);
            mbar_init(&o_free[i], 128);
            for (int qd = 0; qd < 4; ++qd) mbar_init(&turn[4 * i + qd], 1);
        }
        mbar_fence_init();
    }
    if (warp == 9) tmem_alloc(tmem_slot, A::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 8) {
        // ------------------------------------------------------ TMA producer
        if (lane == 0) {
            int q_loads = 0, k_issued = 0, v_issued = 0;
            int h = 0;
            for (TileCursor c = c0; c.g < n_t; next(c)) {
                const int g = c.g;
                if (first_of(c)) {
                    const int u = c.u;
                    h = u / sp.n_qblk;
                    const int q0 = (u % sp.n_qblk) * (A::QT * A::BQ);
                    // the previous piece's Q stays until its last S MMA is done
                    if (q_loads > 0 && !mbar_wait(q_empty, (q_loads - 1) & 1, err, ERR_WAIT_PRODUCER)) break;
                    mbar_expect_tx(q_full, A::QT * A::Q_BYTES);
                    for (int i = 0; i < A::QT; ++i)
                        for (int r = 0; r < A::NR; ++r)
                            tma_load_2d(sQ + i * A::Q_BYTES + r * A::REGION, &tmQ, q_full, h * HD + 64 * r,
                                        q0 + i * A::BQ);
                    ++q_loads;
                }
                const int st = g % A::STAGES, kt = c.k;
                const uint32_t ph = ((g / A::STAGES) & 1) ^ 1;
                if (!mbar_wait(&k_empty[st], ph, err, ERR_WAIT_PRODUCER)) break;
                mbar_expect_tx(&k_full[st], A::KV_BYTES);
                for (int r = 0; r < A::NR; ++r)
                    tma_load_2d(sK + st * A::KV_BYTES + r * A::REGION, &tmK, &k_full[st], h * HD + 64 * r,
                                kt * A::BKV);
                k_issued = g + 1;
                if (!mbar_wait(&v_empty[st], ph, err, ERR_WAIT_PRODUCER)) break;
                mbar_expect_tx(&v_full[st], A::KV_BYTES);
                for (int r = 0; r < A::NR; ++r)
                    tma_load_2d(sV + st * A::KV_BYTES + r * A::REGION, &tmV, &v_full[st], h * HD + 64 * r,
                                kt * A::BKV);
                v_issued = g + 1;
            }
            // Drain: every copy this thread started has landed before exit.
            if (q_loads > 0) mbar_wait(q_full, (q_loads - 1) & 1, err, ERR_WAIT_PRODUCER);
            for (int g = k_issued - A::STAGES < 0 ? 0 : k_issued - A::STAGES; g < k_issued; ++g)
                mbar_wait(&k_full[g % A::STAGES], (g / A::STAGES) & 1, err, ERR_WAIT_PRODUCER);
            for (int g = v_issued - A::STAGES < 0 ? 0 : v_issued - A::STAGES; g < v_issued; ++g)
                mbar_wait(&v_full[g % A::STAGES], (g / A::STAGES) & 1, err, ERR_WAIT_PRODUCER);
        }
    } else if (warp >= 9) {
        // ------------------------------------------------------ MMA issue
        // hd 64: warp 9 issues every MMA of Q tile 0, warp 10 those of tile 1,
        // so the issue work is spread over two SM sub-partitions and neither
        // tile waits on the other's softmax.  hd 128: warp 9 alone.  The
        // whole warp runs the loop (converged); one elected lane issues each
        // tcgen05 instruction.
        if (warp == 9 || A::ISSUERS == 2) {
            constexpr uint32_t idesc_s = idesc_bf16(128, 128, false, false);
            constexpr uint32_t idesc_o = idesc_bf16(128, HD, false, true);
            // Descriptors are built once; each MMA adds a constant to the
            // start-address field (addresses stay below 256 KB, so the
            // 14-bit field never carries).
            const uint64_t dQ0 = sdesc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t dK0 = sdesc_sw128(smem_u32(sK), 16, 1024);
            const uint64_t dV0 = sdesc_sw128(smem_u32(sV), A::REGION, 1024);
            auto issue_s = [&](int i, int g) {        // S_i = Q_i K_g^T
                const uint64_t dq = dQ0 + (uint64_t)((i * A::Q_BYTES) >> 4);
                const uint64_t dk = dK0 + (uint64_t)(((g % A::STAGES) * A::KV_BYTES) >> 4);
#pragma unroll
                for (int ks = 0; ks < HD / 16; ++ks) {
                    const uint32_t off = ((ks >> 2) * A::REGION + (ks & 3) * 32) >> 4;
                    tc_mma_warp(tmem + A::S_COL(i), dq + off, dk + off, idesc_s, ks > 0 ? 1u : 0u);
                }
                tc_commit_warp(&s_full[i]);
            };
            auto issue_pv = [&](int i, const TileCursor &c) {   // O_i (+)= P_i V_g, P_i in TMEM
                const uint64_t dv = dV0 + (uint64_t)(((c.g % A::STAGES) * A::KV_BYTES) >> 4);
                const bool fresh = first_of(c);        // first tile of a piece: O_i = P_i V_g
#pragma unroll
                for (int ks = 0; ks < A::BKV / 16; ++ks)
                    tc_mma_tmem_a_warp(tmem + A::O_COL(i), tmem + A::P_COL(i) + 8 * ks, dv + ((ks * 16 * 128) >> 4),
                                       idesc_o, (!fresh || ks > 0) ? 1u : 0u);
            };
            auto wait = [&](uint64_t *b, int parity) -> bool {
                const bool r = mbar_wait(b, parity & 1, err, ERR_WAIT_MMA);
                return __all_sync(0xffffffffu, r) != 0;
            };
            // S of tile g needs its piece's Q (and, after a piece's last S,
            // the producer may replace Q); P V of the first tile of a piece
            // overwrites O, so it waits until the softmax has read O out.
            auto s_ready = [&](const TileCursor &c) -> bool {
                if (first_of(c) && !wait(q_full, piece_of(c))) return false;
                return wait(&k_full[c.g % A::STAGES], c.g / A::STAGES);
            };
            auto pv_ready = [&](int i, const TileCursor &c) -> bool {
                if (first_of(c) && piece_of(c) > 0 && !wait(&o_free[i], piece_of(c) - 1)) return false;
                return wait(&p_full[i], c.g) && wait(&v_full[c.g % A::STAGES], c.g / A::STAGES);
            };
            if constexpr (A::SEP_P) {
                // hd 64: S_i(g+1) is issued once the softmax has read S_i(g) (P
                // has its own columns), then P_i V_g once P_i is ready.
                const int i = warp - 9;
                bool ok = s_ready(c0);
                if (ok) {
                    tc_fence_after();
                    issue_s(i, 0);
                    tc_commit_warp(&k_empty[0]);
                    if (last_of(c0)) tc_commit_warp(q_empty);
                }
                TileCursor cs = c0;                    // next S tile is cs + 1
                for (TileCursor c = c0; ok && c.g < n_t; next(c)) {
                    const int g = c.g;
                    if (g + 1 < n_t) {
                        next(cs);
                        if (!(wait(&s_cons[i], g) && s_ready(cs))) break;
                        tc_fence_after();
                        issue_s(i, g + 1);
                        tc_commit_warp(&k_empty[(g + 1) % A::STAGES]);
                        if (last_of(cs)) tc_commit_warp(q_empty);
                    }
                    if (!pv_ready(i, c)) break;
                    tc_fence_after();
                    issue_pv(i, c);
                    tc_commit_warp(&pv_done[i]);
                    tc_commit_warp(&v_empty[g % A::STAGES]);
                }
            } else {
                // hd 128: one warp issues P0V(g), S0(g+1), P1V(g), S1(g+1) -- the
                // order in which the warpgroups finish their turns; P_i
                // overwrites S_i, so S_i(g+1) follows P_i V_g.
                bool ok = s_ready(c0);
                if (ok) {
                    tc_fence_after();
                    issue_s(0, 0);
                    issue_s(1, 0);
                    tc_commit_warp(&k_empty[0]);
                    if (last_of(c0)) tc_commit_warp(q_empty);
                }
                TileCursor cs = c0;                    // next S tile is cs + 1
                for (TileCursor c = c0; ok && c.g < n_t; next(c)) {
                    const int g = c.g;
                    const bool more = g + 1 < n_t;
                    if (more) next(cs);
                    if (!pv_ready(0, c)) break;
                    tc_fence_after();
                    issue_pv(0, c);
                    if (last_of(c)) tc_commit_warp(&pv_done[0]);
                    if (more) {
                        if (!s_ready(cs)) break;
                        tc_fence_after();
                        issue_s(0, g + 1);
                    }
                    if (!pv_ready(1, c)) break;
                    tc_fence_after();
                    issue_pv(1, c);
                    tc_commit_warp(&v_empty[g % A::STAGES]);
                    if (last_of(c)) tc_commit_warp(&pv_done[1]);
                    if (more) {
                        issue_s(1, g + 1);
                        tc_commit_warp(&k_empty[(g + 1) % A::STAGES]);
                        if (last_of(cs)) tc_commit_warp(q_empty);
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ softmax
        const int wg = warp >> 2;                          // tile of this warpgroup
        const int q = warp & 3;                            // TMEM lane quadrant
        const int r_tile = wg * A::BQ + q * 32 + lane;     // row within the unit (0..255)
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);
        const uint32_t tS = tl + A::S_COL(wg);
        const uint32_t tP = tl + A::P_COL(wg);
        const uint32_t tO = tl + A::O_COL(wg);
        const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;
        const int tail = n_keys - (nkt - 1) * A::BKV;      // valid keys in the last tile
        // One key tile g (key tile kt of its unit): S_i -> running max m,
        // P_i = 2^(S_i sl2 - m) into TMEM, running sum l.  false: a wait ran out.
        auto tile = [&](int g, int kt, bool fresh, float &m, float &l) -> bool {
            bool ok = mbar_wait(&s_full[wg], g & 1, err, ERR_WAIT_SOFTMAX);
            __syncwarp();
            if (!__all_sync(0xffffffffu, ok)) return false;
            tc_fence_after();
            float s[128];
            tmem_ld128_sync(tS, s);
            if constexpr (A::SEP_P) {
                tc_fence_before();
                mbar_arrive(&s_cons[wg]);
            }
            if (kt == nkt - 1 && tail < A::BKV) {
#pragma unroll
                for (int c = 0; c < 128; ++c)
                    if (c >= tail) s[c] = -INFINITY;
            }
            // O_i (this thread's row of it, in TMEM) times alpha; the whole warp
            auto scale_o = [&](float alpha) {
#pragma unroll 1
                for (int c = 0; c < HD / 16; ++c) {
                    float t[16];
                    tmem_ld16_sync(tO + 16 * c, t);
#pragma unroll
                    for (int i = 0; i < 16; ++i) t[i] *= alpha;
                    tmem_st16_sync(tO + 16 * c, t);
                }
            };
            float2 rs0 = make_float2(0.f, 0.f), rs1 = make_float2(0.f, 0.f);
            if constexpr (!A::SEP_P) {
                // hd 128.  m is the row max of the piece's first tile; a later
                // tile takes it as it is, without a max of its own: bf16 and
                // fp32 share their exponent range, so scores above m cost no
                // precision while the sums stay small.  The tile's row sum
                // tells: past RAISE (or not a number) the row's m is raised to
                // its max, O and l are rescaled, and the tile is done again
                // from the scores still in registers.  (The commit behind
                // s_full covers P V of tile g - 1, so O_i is stable.)  With a
                // max for every tile / without: 12960 x 38880 x 40 heads 6.30
                // / 6.20 ms, 12 heads 1.84 / 1.81 ms; at hd 64, where the
                // other tile's exponentials hide the max, 0.494 / 0.555 ms.
                // (P V issued from the first two or three quarters while the
                // softmax computes the rest: 1.94 to 2.01 ms at 12 heads.)
                bool fix = fresh;
                float2 rs;
                for (int pass = 0;; ++pass) {
                    if (__any_sync(0xffffffffu, fix)) {
                        const float m_new = fmaxf(m, row_max(s) * sl2);
                        const float alpha = fix && !fresh ? ex2_approx(m - m_new) : 1.0f;
                        if (fix) m = m_new;
                        if (!fresh) {
                            l *= alpha;
                            scale_o(alpha);
                        }
                    }
                    rs0 = rs1 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int qt = 0; qt < 4; ++qt) exp_quarter(s, qt, sl2, m, tP, rs0, rs1);
                    rs = __fadd2_rn(rs0, rs1);
                    fix = !(rs.x + rs.y <= A::RAISE);
                    if (pass > 0 || !__any_sync(0xffffffffu, fix)) break;
                }
                l += rs.x + rs.y;
                tc_fence_before();
                mbar_arrive(&p_full[wg]);
                return true;
            }
            const float m_new = row_max(s) * sl2;
            if (fresh) m = m_new;
            const bool grow = !fresh && m_new > m + A::LAZY;
            const float alpha = grow ? ex2_approx(m - m_new) : 1.0f;
            if (grow) m = m_new;
            // P_i buffer free and O_i stable once P V of the previous tile is done
            if (g >= 1) {
                ok = mbar_wait(&pv_done[wg], (g - 1) & 1, err, ERR_WAIT_SOFTMAX);
                __syncwarp();
                if (!__all_sync(0xffffffffu, ok)) return false;
                tc_fence_after();
            }
            if (__any_sync(0xffffffffu, grow)) scale_o(alpha);
            // The two warps of each SM sub-partition (quadrant q of WG 0 and
            // of WG 1) take turns on the exponential phase, which is bound
            // by the sub-partition's MUFU: WG 0 does tile g, then WG 1 tile
            // g, then WG 0 tile g + 1 ... so that one warp's exponentials
            // overlap the other's loads, max and MMA waits.  The hand-off is
            // per quadrant, so a slower sub-partition does not hold up the
            // others.
            // (hd 128 takes no turns: its exponential phase is a smaller share of
            // a key tile's work)
            if (wg == 1 || g > 0) {
                ok = mbar_wait(&turn[4 * wg + q], (wg == 1 ? g : g - 1) & 1, err, ERR_WAIT_SOFTMAX);
                __syncwarp();
                if (!__all_sync(0xffffffffu, ok)) return false;
            }
            // probabilities and row sum in four 32-key quarters
#pragma unroll
            for (int qt = 0; qt < 4; ++qt) exp_quarter(s, qt, sl2, m, tP, rs0, rs1);
            const float2 rs = __fadd2_rn(rs0, rs1);
            l = l * alpha + (rs.x + rs.y);
            tc_fence_before();
            mbar_arrive(&p_full[wg]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&turn[4 * (wg ^ 1) + q]);
            return true;
        };
        // End of a piece (its last tile g, unit u, piece p of this CTA): O_i
        // complete -> output (whole unit) or partial.
        auto end_piece = [&](int g, int u, int p, bool head_part, bool cut_front, float m, float l) -> bool {
            const bool ok = mbar_wait(&pv_done[wg], (A::SEP_P ? g : p) & 1, err, ERR_WAIT_SOFTMAX);
            __syncwarp();
            if (!__all_sync(0xffffffffu, ok)) return false;
            tc_fence_after();
            if constexpr (CLUSTER) {
                // unnormalised O and (m, l) stay in shared memory, O in the K / V
                // ring once both Q tiles' last P V has read it
                mbar_arrive(all_pv);
                const bool done = mbar_wait(all_pv, 0, err, ERR_WAIT_SOFTMAX);
                __syncwarp();
                if (!__all_sync(0xffffffffu, done)) return false;
#pragma unroll 1
                for (int c = 0; c < HD / 32; ++c) {
                    float t[32];
                    tmem_ld32_sync(tO + 32 * c, t);
                    uint8_t *blk = sK + partial_block(0, warp, c, HD) * sizeof(float) + lane * 128;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        *reinterpret_cast<float4 *>(blk + ((k ^ (lane & 7)) << 4)) =
                            make_float4(t[4 * k], t[4 * k + 1], t[4 * k + 2], t[4 * k + 3]);
                }
                reinterpret_cast<float2 *>(smem + A::OFF_O)[r_tile] = make_float2(m, l);
                return true;
            }
            // through this warp's 4 KB of shared memory: a thread's own row
            // stores to global memory touch 32 lines per instruction and took
            // 5 us of a 256-query piece at hd 128
            const int h = u / sp.n_qblk;
            const int row0 = (u % sp.n_qblk) * (A::QT * A::BQ) + wg * A::BQ + q * 32;   // this warp's first row
            uint8_t *so = smem + A::OFF_O + warp * 4096 + lane * 128;
            const int sw = lane & 7;
            auto buffer_free = [&]() {                 // the last block's store has read it
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
            };
            if (!head_part && !cut_front) {
                const float inv = 1.0f / l;
#pragma unroll 1
                for (int c = 0; c < HD / 64; ++c) {
                    float t[64];
                    tmem_ld64_sync(tO + 64 * c, t);
                    buffer_free();
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            __nv_bfloat162 b2 = __floats2bfloat162_rn(t[8 * k + 2 * e] * inv, t[8 * k + 2 * e + 1] * inv);
                            w[e] = *reinterpret_cast<uint32_t *>(&b2);
                        }
                        *reinterpret_cast<uint4 *>(so + ((k ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && row0 < Lq) {      // rows past Lq are clipped
                        tma_store_2d(&tmO, smem + A::OFF_O + warp * 4096, h * HD + 64 * c, row0);
                        bulk_commit();
                    }
                }
            } else {
                const int slot = WAVE ? 2 * cta + (p - sp.W)                       // remainder piece 0 / 1
                                      : (head_part ? 2 * (cta + 1) : 2 * cta + 1);   // boundary c + 1 head / c tail
#pragma unroll 1
                for (int c = 0; c < HD / 32; ++c) {
                    float t[32];
                    tmem_ld32_sync(tO + 32 * c, t);
                    buffer_free();
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        *reinterpret_cast<float4 *>(so + ((k ^ sw) << 4)) =
                            make_float4(t[4 * k], t[4 * k + 1], t[4 * k + 2], t[4 * k + 3]);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        bulk_store(ws_o + partial_block(slot, warp, c, HD), smem + A::OFF_O + warp * 4096, 4096);
                        bulk_commit();
                    }
                }
                ws_ml[(size_t)slot * (A::QT * A::BQ) + r_tile] = make_float2(m, l);
            }
            tc_fence_before();
            mbar_arrive(&o_free[wg]);
            return true;
        };
        bool ok = true;
        TileCursor cur = c0;
        while (ok && cur.g < n_t) {
            const bool cut_front = cur.k != 0;     // the piece's unit began in another CTA
            float m = -INFINITY, l = 0.0f;
            bool fresh = true;
            for (;;) {
                ok = tile(cur.g, cur.k, fresh, m, l);
                if (!ok) break;
                fresh = false;
                if (last_of(cur)) break;
                next(cur);
            }
            if (!ok) break;
            ok = end_piece(cur.g, cur.u, piece_of(cur), cur.k != nkt - 1, cut_front, m, l);
            next(cur);
        }
        // every store of this warp has completed before the CTA exits
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CLUSTER) {
        // The cluster's partials: a warp takes 16 rows x 32 columns at a time,
        // first the weights 2^(m_p - m) / l of its rows, then the weighted sum,
        // a lane 4 columns of every fourth row.
        cluster_sync_all();
        const int n_cta = (int)cluster_nctarank(), rank = (int)cluster_ctarank();
        if (warp < 8) {
            const int u = c0.u, h = u / sp.n_qblk;
            float *wgt = reinterpret_cast<float *>(smem + A::OFF_O + 4096) + warp * 256;      // [16 CTAs][16 rows]
            const int lr = lane >> 3, ch = lane & 7;
            for (int b = rank * 8 + warp; b < 16 * (HD / 32); b += 8 * n_cta) {
                const int r16 = (b & 15) * 16, grp = b >> 4;
                const int row0 = (u % sp.n_qblk) * (A::QT * A::BQ) + r16;
                if (row0 >= Lq) continue;
                const float2 *ml = reinterpret_cast<const float2 *>(smem + A::OFF_O) + r16 + (lane & 15);
                float mm = -INFINITY, l = 0.0f;
                for (int p = lane >> 4; p < n_cta; p += 2) mm = fmaxf(mm, ld_cluster2(map_to_cta(ml, p)).x);
                mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, 16));
                for (int p = lane >> 4; p < n_cta; p += 2) {
                    const float2 t = ld_cluster2(map_to_cta(ml, p));
                    const float w = exp2f(t.x - mm);
                    l = fmaf(t.y, w, l);
                    wgt[p * 16 + (lane & 15)] = w;
                }
                l += __shfl_xor_sync(0xffffffffu, l, 16);
                const float inv = 1.0f / l;
                for (int p = lane >> 4; p < n_cta; p += 2) wgt[p * 16 + (lane & 15)] *= inv;
                __syncwarp();
                const uint8_t *blk = sK + partial_block(0, r16 >> 5, grp, HD) * sizeof(float) + (r16 & 31) * 128 + ch * 16;
                float4 acc[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
                for (int p = 0; p < n_cta; ++p) {
                    const uint32_t src = map_to_cta(blk, p);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 x = ld_cluster4(src + (lr + 4 * i) * 128);
                        const float w = wgt[p * 16 + lr + 4 * i];
                        acc[i].x = fmaf(x.x, w, acc[i].x);
                        acc[i].y = fmaf(x.y, w, acc[i].y);
                        acc[i].z = fmaf(x.z, w, acc[i].z);
                        acc[i].w = fmaf(x.w, w, acc[i].w);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = lr + 4 * i;
                    if (row0 + r >= Lq) break;
                    __nv_bfloat162 lo = __floats2bfloat162_rn(acc[i].x, acc[i].y);
                    __nv_bfloat162 hi = __floats2bfloat162_rn(acc[i].z, acc[i].w);
                    uint2 pk;
                    pk.x = *reinterpret_cast<uint32_t *>(&lo);
                    pk.y = *reinterpret_cast<uint32_t *>(&hi);
                    *reinterpret_cast<uint2 *>(o + (size_t)(row0 + r) * d + h * HD + 32 * grp +
                                               4 * (ch ^ (r & 7))) = pk;
                }
                __syncwarp();
            }
        }
        cluster_sync_all();                            // no CTA leaves while another reads its partials
    }
    if (warp == 9) {
        tc_fence_after();
        tmem_dealloc(tmem, A::TMEM_COLS);
    }
}

// Merges the partials of the units cut between CTAs (see AttnSplit): m =
// max_p m_p, O = sum of O_p 2^(m_p - m) / sum of l_p 2^(m_p - m).  Contiguous
// order: grid.x = CTA boundaries, two partials (head and tail) of the unit
// the boundary cuts.  Waves: grid.x = remaining units, the partials of the
// CTAs whose pieces touch it, in CTA order (at most G / units + 2).  grid.y
// picks 32 of the head's columns, grid.z 32 of the unit's 256 query rows, 16
// per warp.  The threads first find the partials' slots (one each: the share
// bounds take 64-bit divisions, which one thread walking them alone spent
// longer on than on the data), then every warp the weights 2^(m_p - m) / l of
// its rows, and then it runs over the partials with four in flight, a lane
// taking 4 columns of every fourth row (a load reads 512 contiguous bytes).
// 19 partials of 8 units, hd 128: 35 us with one thread per row.
constexpr int COMBINE_ROWS = 32, COMBINE_COLS = 32;
template <int HD, bool WAVE>
__global__ void __launch_bounds__(64)
    attn_combine_kernel(bf16 *__restrict__ o, const int Lq, const int d, const AttnSplit sp, const int max_part,
                        const float *__restrict__ ws_o, const float2 *__restrict__ ws_ml,
                        const uint8_t *__restrict__ skip_flag) {
    pdl_wait();
    if (skip_flag != nullptr && *skip_flag == XC_DEC_SKIP) return;
    extern __shared__ int comb_smem[];                 // slots [max_part], weights [2 warps][max_part][16]
    int *slots = comb_smem;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *wgt = reinterpret_cast<float *>(comb_smem + max_part) + warp * max_part * 16;
    int u, n;
    if constexpr (WAVE) {
        const int rr = blockIdx.x;                     // remaining unit
        const long long ub = (long long)rr * sp.n_kt, ue = ub + sp.n_kt;
        u = sp.W * sp.G + rr;
        int c0 = (int)(ub * sp.G / sp.T2);             // begin2(c0) <= ub: the first CTA that can touch the unit
        if (sp.begin2(c0 + 1) <= ub) ++c0;
        // CTAs c0 .. c0 + n - 1 touch it; slot 2 c (its first piece) or 2 c + 1
        n = 0;
        for (int base = c0; base < sp.G; base += 64) {
            const int c = base + threadIdx.x;
            const long long b = sp.begin2(c), e = sp.begin2(c + 1);
            const bool touch = c < sp.G && b < ue;
            const int k = c - c0;
            if (touch && k < max_part) slots[k] = e > b ? 2 * c + (b >= ub ? 0 : 1) : -1;
            const int hit = __syncthreads_count(touch);
            n += hit;
            if (hit < 64) break;
        }
        n = min(n, max_part);
        if (n == 1) return;                            // one CTA ran the whole unit and wrote it
    } else {
        const int b = blockIdx.x + 1;                  // boundary between CTAs b-1 and b
        const long long it = sp.begin(b);
        if (it % sp.n_kt == 0) return;                 // the boundary falls between units
        u = (int)(it / sp.n_kt);
        n = 2;
        if (threadIdx.x < 2) slots[threadIdx.x] = 2 * b + threadIdx.x;         // head, tail
        __syncthreads();
    }
    const int h = u / sp.n_qblk;
    const int r16 = blockIdx.z * COMBINE_ROWS + warp * 16;                     // the warp's first row of the unit
    const int row0 = (u % sp.n_qblk) * 256 + r16;
    if (row0 >= Lq) return;
    {   // weights: lane -> row lane % 16, every second partial
        const float2 *ml = ws_ml + r16 + (lane & 15);
        float m = -INFINITY, l = 0.0f;
#pragma unroll 4
        for (int p = lane >> 4; p < n; p += 2)
            if (slots[p] >= 0) m = fmaxf(m, ml[(size_t)slots[p] * 256].x);
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
#pragma unroll 4
        for (int p = lane >> 4; p < n; p += 2) {
            float w = 0.0f;
            if (slots[p] >= 0) {
                const float2 t = ml[(size_t)slots[p] * 256];
                w = exp2f(t.x - m);
                l = fmaf(t.y, w, l);
            }
            wgt[p * 16 + (lane & 15)] = w;
        }
        l += __shfl_xor_sync(0xffffffffu, l, 16);
        const float inv = 1.0f / l;
        for (int p = lane >> 4; p < n; p += 2) wgt[p * 16 + (lane & 15)] *= inv;
        __syncwarp();
    }
    constexpr int NR = 4;                              // rows of a lane: lr, lr + 4, ...
    const int lr = lane >> 3, ch = lane & 7;
    const int w8 = r16 >> 5, b16 = r16 & 31;           // softmax warp that wrote the rows, row of its block
    float4 acc[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int p = 0; p < n; ++p) {
        const int sl = slots[p];
        if (sl < 0) continue;
        const float4 *src = reinterpret_cast<const float4 *>(ws_o + partial_block(sl, w8, blockIdx.y, HD));
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const float4 x = src[(b16 + lr + 4 * i) * 8 + ch];                 // chunk ch ^ (row & 7) of its row
            const float w = wgt[p * 16 + lr + 4 * i];
            acc[i].x = fmaf(x.x, w, acc[i].x);
            acc[i].y = fmaf(x.y, w, acc[i].y);
            acc[i].z = fmaf(x.z, w, acc[i].z);
            acc[i].w = fmaf(x.w, w, acc[i].w);
        }
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const int r = lr + 4 * i;
        if (row0 + r >= Lq) break;
        __nv_bfloat162 lo = __floats2bfloat162_rn(acc[i].x, acc[i].y);
        __nv_bfloat162 hi = __floats2bfloat162_rn(acc[i].z, acc[i].w);
        uint2 pk;
        pk.x = *reinterpret_cast<uint32_t *>(&lo);
        pk.y = *reinterpret_cast<uint32_t *>(&hi);
        *reinterpret_cast<uint2 *>(o + (size_t)(row0 + r) * d + h * HD + blockIdx.y * COMBINE_COLS +
                                   4 * (ch ^ ((b16 + r) & 7))) = pk;
    }
}

bool make_tmap_bf16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows);

size_t attn_workspace_bytes(int head_dim) {
    const size_t slots = 2 * ((size_t)sm_count() + 1);
    return slots * 256 * ((size_t)head_dim * sizeof(float) + sizeof(float2));
}

template <int HD, int ORDER>
static cudaError_t attn_attr() {
    static PerDevice done;
    return allow_smem(done, attn_tc_kernel<HD, ORDER>, AttnTile<HD>::SMEM_BYTES);
}

// Clusters of `size` attention CTAs (one per SM) that are resident at once.
template <int HD>
static int attn_clusters(int size) {
    static PerDevice known[9];
    return known[size].get([size] {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(size * (sm_count() / size)));
        cfg.blockDim = dim3(AttnTile<HD>::THREADS);
        cfg.dynamicSmemBytes = AttnTile<HD>::SMEM_BYTES;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (attn_attr<HD, ORDER_CLUSTER>() != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel<HD, ORDER_CLUSTER>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        return n > 0 ? n : -1;
    });
}

template <int HD, int ORDER>
static cudaError_t launch_attn_(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv,
                                const CUtensorMap &to, bf16 *o, int Lq, int n_keys, int d, const AttnSplit &sp,
                                int cluster, int n_combine, void *ws, const uint8_t *skip, int *err, int *n_launched,
                                cudaStream_t st) {
    using A = AttnTile<HD>;
    constexpr bool WAVE = ORDER != ORDER_CONTIGUOUS;
    cudaError_t e = attn_attr<HD, ORDER>();
    if (e != cudaSuccess) return e;
    const int n_sm = sm_count();
    float *ws_o = n_combine > 0 ? reinterpret_cast<float *>(ws) : nullptr;
    float2 *ws_ml = n_combine > 0 ? reinterpret_cast<float2 *>(ws_o + 2 * ((size_t)n_sm + 1) * 256 * HD) : nullptr;
    e = launch_pdl_cluster(attn_tc_kernel<HD, ORDER>, (unsigned)cluster, dim3(sp.G), dim3(A::THREADS), A::SMEM_BYTES, st,
                           tq, tk, tv, to, Lq, n_keys, sp, ws_o, ws_ml, skip, err, o, d);
    if (e != cudaSuccess) return e;
    if (n_launched) *n_launched = 1;
    if (n_combine > 0) {
        const int max_part = WAVE ? std::min(sp.G, sp.G / n_combine + 2) : 2;
        e = launch_pdl(attn_combine_kernel<HD, WAVE>, dim3(n_combine, HD / COMBINE_COLS, 256 / COMBINE_ROWS), dim3(64),
                       (size_t)max_part * 33 * sizeof(float), st, o, Lq, d, sp, max_part,
                       static_cast<const float *>(ws_o), static_cast<const float2 *>(ws_ml), skip);
        if (n_launched) *n_launched = 2;
    }
    return e;
}

// What a launch runs: an order, its split, the CTAs of a cluster and what the
// merge launch has to merge (0: no such launch).
struct AttnPlan {
    int order, cluster, n_combine;
    AttnSplit sp;
};

// Work order (see AttnSplit).  Cutting units balances the SMs at the price of
// partials and their merge.  Both sides are compared in key tiles (1.2 us at hd
// 64, 1.6 at hd 128): whole units take the longest CTA's tiles, a cut the tiles
// of a CTA's share and the time of its merge, fitted to 450 shapes measured both
// ways (98 to 12960 queries, 3 to 48 key tiles, 2 to 2040 units; the choice
// costs at most 3 % of the better one).
//  * Fewer units than SMs: every unit is split over the same number of CTAs,
//    so that no CTA touches two units: in clusters, which merge in rounds of 8
//    warps per CTA over the unit's 16-row blocks and read a partial of every
//    CTA in each (200 x 590 x 12 heads of 64: 10.1 us whole, 12.4 in clusters of
//    3; 98 x 974 x 12 13.2 whole, 10.5 in clusters of 4), or merged through
//    global memory (1000 x 718 x 12 of 128 14.6 whole, 16.0 by 3; 300 x 974 x 6
//    17.1 whole, 14.6 by 4; 1000 x 10000 x 2 118 and 27).
//  * More than half as many units as SMs: over all SMs, a CTA touching two
//    units (512 x 1614 x 40 of 64 19.5 whole, 20.9 cut; 512 x 2510 x 40 27.3 and
//    25.3; 1000 x 2560 x 24 of 128 34.6 and 37.3, 512 x 3278 x 40 43.4 and 38.2).
//  * Waves with the remaining units split when there are many waves (W >= 8)
//    and the K / V of all heads exceed L2 -- measured at the 14B shape (40
//    heads x 20 MB of K / V, W = 13): 40.7 -> 1.2 GB of DRAM traffic per
//    launch at the same attention time, the GPU's power then allowing a
//    higher clock under its cap (1500 -> 1965 MHz, 0.766 -> 0.801 chunks/s).
//  * Else contiguous shares (at the 1.3B shape, W = 4, the waves were 4 %
//    slower per launch): 4000 x 718 x 12 of 64 20.3 whole, 21.5 cut; 4000 x 1230 x
//    12 29.2 and 27.0; 12960 x 718 x 12 of 128 56.9 and 60.8, 4000 x 1408 x 12 39.6
//    and 37.5.
template <int HD>
static AttnPlan attn_plan(int Lq, int n_keys, int n_heads, bool can_cut) {
    using A = AttnTile<HD>;
    AttnPlan pl{ORDER_WAVE, 1, 0, {}};
    AttnSplit &sp = pl.sp;
    sp.n_kt = (n_keys + A::BKV - 1) / A::BKV;
    sp.n_qblk = (Lq + A::QT * A::BQ - 1) / (A::QT * A::BQ);
    const int n_units = sp.n_qblk * n_heads;
    const int n_sm = sm_count();
    sp.T = (long long)n_units * sp.n_kt;
    sp.T2 = 0;
    sp.G = n_units < n_sm ? n_units : n_sm;
    sp.W = n_units / sp.G;
    sp.R = n_units - sp.W * sp.G;
    const double whole = (double)(sp.W + (sp.R > 0 ? 1 : 0)) * sp.n_kt, even = (double)sp.T / n_sm;
    // (one whole unit per CTA: contiguous shares of n_kt tiles, whose cursor is
    // the cheaper one: 98 x 2048 x 100 of 64 22.2 us, 22.4 as a wave)
    if (n_units <= n_sm) pl.order = ORDER_CONTIGUOUS;
    if (!can_cut || whole <= even) return pl;
    if (n_units < n_sm) {
        // One cluster of up to 8 CTAs per unit, as many as can all be resident
        // at once, while a CTA has at most 8 key tiles: beyond, more CTAs per
        // unit gain more than their merge through global memory costs (1000 x
        // 10000 x 2 heads of 128: 26.7 us by 16, 27.4 in clusters of 8).  At
        // hd 128, with twice the partials, clusters of 3 and 4 lost: 840 x
        // 2520 by 10 heads 22.8 -> 23.8 us, 8 heads 19.9 -> 20.2, 6 heads
        // (clusters of 6) 20.4 -> 19.5; at hd 64 by 10 heads 18.8 -> 18.4, 6
        // heads 17.4 -> 14.6, 4 heads 16.4 -> 14.3.
        constexpr int CL_MIN = HD == 64 ? 2 : 6;
        const int most = std::min(n_sm / n_units, (sp.n_kt + 1) / 2);    // CTAs of a unit, each two tiles
        int cl = std::min(8, most);
        while (cl >= CL_MIN && n_units > attn_clusters<HD>(cl)) --cl;
        // CTAs per unit otherwise: a key tile takes a CTA about 1.2 us and a
        // partial the merge about 0.4, so some sqrt(3 n_kt) of them are best (300
        // x 30000 x 1 head of 128: 76 / 59 / 40 per unit 66 / 53 / 43 us; 474 x
        // 8116 x 2 heads of 64: 32 / 16 / 11 30 / 21.8 / 21.3)
        int per = 1;
        while (per * per < 3 * sp.n_kt) ++per;
        per = std::min(per, most);
        double cut;
        bool in_cluster = false;
        if (cl >= CL_MIN && sp.n_kt <= 8 * cl) {
            const int blocks = (std::min(Lq, A::QT * A::BQ) + 15) / 16 * (HD / 32), rounds = (blocks + 8 * cl - 1) / (8 * cl);
            cut = (sp.n_kt + cl - 1) / cl + (HD == 64 ? 2.5 + 0.4 * rounds * cl : 3.4 + 0.27 * rounds * cl);
            in_cluster = true;
        } else if (per >= 2) {
            cut = (sp.n_kt + per - 1) / per + 2.8 + 0.4 * per + 0.02 * n_units;
        } else {
            cut = even + (HD == 64 ? 8.0 : 10.5);
        }
        if (whole <= cut) return pl;
        pl.order = in_cluster ? ORDER_CLUSTER : ORDER_WAVE;
        pl.cluster = in_cluster ? cl : 1;
        pl.n_combine = in_cluster ? 0 : n_units;
        sp.G = in_cluster ? n_units * cl : per >= 2 ? n_units * per : n_sm;
        sp.W = sp.R = 0;
        sp.T2 = sp.T;
        return pl;
    }
    if (whole <= even + (HD == 64 ? 5.0 : 7.0)) return pl;
    const double kv_bytes = 2.0 * n_keys * (double)(n_heads * HD) * sizeof(bf16);
    if (sp.W >= 8 && kv_bytes > 128.0 * 1024 * 1024) {
        pl.n_combine = sp.R;
        sp.T2 = (long long)sp.R * sp.n_kt;
        sp.R = 0;
        return pl;
    }
    pl.order = ORDER_CONTIGUOUS;
    pl.n_combine = sp.G - 1;
    return pl;
}

template <int HD>
static cudaError_t launch_attn(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv,
                               const CUtensorMap &to, bf16 *o, int Lq, int n_keys, int n_heads, int d, void *ws,
                               size_t ws_bytes, const uint8_t *skip, int *err, int *n_launched, cudaStream_t st) {
    // (partials leave by bulk copies: 16-byte aligned)
    const bool can_cut = ws != nullptr && ws_bytes >= attn_workspace_bytes(HD) &&
                         (reinterpret_cast<uintptr_t>(ws) & 15) == 0;
    const AttnPlan pl = attn_plan<HD>(Lq, n_keys, n_heads, can_cut);
    auto run = [&](auto launch) {
        return launch(tq, tk, tv, to, o, Lq, n_keys, d, pl.sp, pl.cluster, pl.n_combine, ws, skip, err, n_launched, st);
    };
    if (pl.order == ORDER_CLUSTER) return run(launch_attn_<HD, ORDER_CLUSTER>);
    if (pl.order == ORDER_CONTIGUOUS) return run(launch_attn_<HD, ORDER_CONTIGUOUS>);
    return run(launch_attn_<HD, ORDER_WAVE>);
}

int attn_tc_plan(int head_dim, int Lq, int n_keys, int n_heads, bool can_cut, int plan[4]) {
    const AttnPlan pl = head_dim == 64 ? attn_plan<64>(Lq, n_keys, n_heads, can_cut)
                                       : attn_plan<128>(Lq, n_keys, n_heads, can_cut);
    plan[0] = pl.sp.G;
    plan[1] = pl.cluster;
    plan[2] = pl.n_combine;
    plan[3] = pl.sp.W;
    return pl.order;
}

// q [Lq][d], k / v maps over [>= n_keys][d] (boxes of 128 rows), o [Lq][d] and
// its map (boxes of 32 rows); hd in {64, 128}.  ws: attn_workspace_bytes(hd)
// bytes, 16-byte aligned, let units be cut between CTAs (nullptr, smaller or
// not aligned: whole units only).
cudaError_t attn_tc(int head_dim, const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv,
                    const CUtensorMap &to, bf16 *o, int Lq, int n_keys, int n_heads, int d, void *ws, size_t ws_bytes,
                    const uint8_t *skip, int *err, int *n_launched, cudaStream_t st) {
    if (n_keys < 1 || Lq < 1) return cudaErrorInvalidValue;
    if (head_dim == 64)
        return launch_attn<64>(tq, tk, tv, to, o, Lq, n_keys, n_heads, d, ws, ws_bytes, skip, err, n_launched, st);
    if (head_dim == 128)
        return launch_attn<128>(tq, tk, tv, to, o, Lq, n_keys, n_heads, d, ws, ws_bytes, skip, err, n_launched, st);
    return cudaErrorInvalidValue;
}

}  // namespace xc
