// fp32 path of the recompute kernels (fp32 models only).  The fp32 bound
// max|err| <= 1e-4 * RMS rules out TF32 tensor cores, so these run on the
// CUDA cores with fp32 FMA; the shapes that use them are small, and latency
// (how much of the chip a launch reaches, how long its serial chain is)
// bounds them before the FMA rate does.
#include "xc_common.cuh"

namespace xc {

// ------------------------------------------------------------------ GEMM
// C[M][N] = epilogue(A[M][K] @ Wt[N][K]^T), both operands K-major.  Every
// thread owns a 4 x 4 block of outputs.
constexpr int SG_THREADS = 256;

// Four consecutive k of one row (0 past K).  VEC: rows and base 16-byte
// aligned (K % 4 == 0), one 16-byte load; otherwise single loads.
template <bool VEC>
__device__ __forceinline__ float4 load_k4(const float *__restrict__ row, int k, int K) {
    if constexpr (VEC) {
        return k < K ? *reinterpret_cast<const float4 *>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        return make_float4(k < K ? row[k] : 0.f, k + 1 < K ? row[k + 1] : 0.f, k + 2 < K ? row[k + 2] : 0.f,
                           k + 3 < K ? row[k + 3] : 0.f);
    }
}
__device__ __forceinline__ void fma_k4(float &acc, const float4 &a, const float4 &w) {
    acc = fmaf(a.x, w.x, acc);
    acc = fmaf(a.y, w.y, acc);
    acc = fmaf(a.z, w.z, acc);
    acc = fmaf(a.w, w.w, acc);
}

// Few outputs: 16 x 16 tile per CTA, K split over 16 groups of 16 threads
// (group g takes the 4-wide k runs g, g + 16, ...), operands straight from
// global memory into registers -- eight 16-byte loads in flight per thread,
// no staging, one barrier -- and the groups' partial sums added in group
// order through shared memory.  Bound by the latency of one load and one
// barrier: K = 64 is a single step.  Measured (call to call, host included)
// against one thread per 16 outputs walking K alone: 64 x 192 x 64 30.7 ->
// 8.8 us, 512 x 256 x 1024 560 -> 27 us.
template <int EPI, bool VEC>
__global__ void __launch_bounds__(SG_THREADS)
    gemm_simt_small(const EpiParams ep, const float *__restrict__ A, const float *__restrict__ Wt, const int K,
                    const uint8_t *__restrict__ skip_flag) {
    pdl_wait();
    pdl_release();
    if (skip_flag != nullptr && *skip_flag == XC_DEC_SKIP) return;
    __shared__ __align__(16) float part[16][16][16];          // [group][row][column]
    const int tid = threadIdx.x;
    const int g = tid >> 4, r4 = (tid >> 2) & 3, c4 = tid & 3;
    const int nt = ep.N / 16;
    const int m0 = (blockIdx.x / nt) * 16, n0 = (blockIdx.x % nt) * 16;
    const int row0 = m0 + 4 * r4, col0 = n0 + 4 * c4;
    const float *ar[4], *wr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        ar[i] = A + (size_t)min(row0 + i, ep.M - 1) * K;      // rows past M: a copy of the last, not stored
        wr[i] = Wt + (size_t)(col0 + i) * K;                  // N % 16 == 0
    }
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
#pragma unroll 2
    for (int k = 4 * g; k < K; k += 64) {
        float4 a[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            a[i] = load_k4<VEC>(ar[i], k, K);
            w[i] = load_k4<VEC>(wr[i], k, K);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) fma_k4(acc[i][j], a[i], w[j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4 *>(&part[g][4 * r4 + i][4 * c4]) =
            make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    __syncthreads();
    if (tid < 64) {                                           // one run of 4 columns per thread
        const int r = tid >> 2, c = 4 * (tid & 3);
        float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const float4 t = *reinterpret_cast<const float4 *>(&part[q][r][c]);
            v[0] += t.x;
            v[1] += t.y;
            v[2] += t.z;
            v[3] += t.w;
        }
        epilogue_run<EPI>(ep, m0 + r, n0 + c, v);
    }
}

// Many outputs: 64 x 64 tile per CTA, k steps of 16 through a double-buffered
// shared-memory stage (transposed to [k][row], so a k step of a thread is one
// 16-byte read of each operand for 16 FMA), the next step's global loads in
// flight during the current one.
constexpr int SG_TILE = 64, SG_BK = 16, SG_LD = SG_TILE + 4;
template <int EPI, bool VEC>
__global__ void __launch_bounds__(SG_THREADS)
    gemm_simt_tile(const EpiParams ep, const float *__restrict__ A, const float *__restrict__ Wt, const int K,
                   const uint8_t *__restrict__ skip_flag) {
    pdl_wait();
    pdl_release();
    if (skip_flag != nullptr && *skip_flag == XC_DEC_SKIP) return;
    __shared__ __align__(16) float as[2][SG_BK][SG_LD], ws[2][SG_BK][SG_LD];
    const int tid = threadIdx.x;
    const int nt = (ep.N + SG_TILE - 1) / SG_TILE;
    const int m0 = (blockIdx.x / nt) * SG_TILE, n0 = (blockIdx.x % nt) * SG_TILE;
    // staging: thread -> row tid / 4 of each operand, k run 4 (tid % 4);
    // rows past M or N read the last one (never stored)
    const int sr = tid >> 2, sk = 4 * (tid & 3);
    const float *ar = A + (size_t)min(m0 + sr, ep.M - 1) * K;
    const float *wr = Wt + (size_t)min(n0 + sr, ep.N - 1) * K;
    const int r4 = 4 * (tid >> 4), c4 = 4 * (tid & 15);
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    float4 an = load_k4<VEC>(ar, sk, K), wn = load_k4<VEC>(wr, sk, K);
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += SG_BK, buf ^= 1) {
        as[buf][sk][sr] = an.x;
        as[buf][sk + 1][sr] = an.y;
        as[buf][sk + 2][sr] = an.z;
        as[buf][sk + 3][sr] = an.w;
        ws[buf][sk][sr] = wn.x;
        ws[buf][sk + 1][sr] = wn.y;
        ws[buf][sk + 2][sr] = wn.z;
        ws[buf][sk + 3][sr] = wn.w;
        __syncthreads();
        if (k0 + SG_BK < K) {
            an = load_k4<VEC>(ar, k0 + SG_BK + sk, K);
            wn = load_k4<VEC>(wr, k0 + SG_BK + sk, K);
        }
#pragma unroll
        for (int k = 0; k < SG_BK; ++k) {
            const float4 a = *reinterpret_cast<const float4 *>(&as[buf][k][r4]);
            const float4 w = *reinterpret_cast<const float4 *>(&ws[buf][k][c4]);
            const float av[4] = {a.x, a.y, a.z, a.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], wv[j], acc[i][j]);
        }
        // one barrier per step: buffer `buf` is rewritten two steps later,
        // after the next step's barrier has seen every thread past its reads
    }
    if (n0 + c4 < ep.N) {
#pragma unroll
        for (int i = 0; i < 4; ++i) epilogue_run<EPI>(ep, m0 + r4 + i, n0 + c4, acc[i]);
    }
}

template <int EPI, bool VEC>
static cudaError_t gemm_simt_vec(const EpiParams &ep, const float *A, const float *Wt, int K, const uint8_t *skip,
                                 cudaStream_t st) {
    // 64 x 64 tiles reuse operands 4 times as often but reach 1 / 16 of the
    // CTAs and do not split K.  Both measured: 32 tiles (512 x 256 x 1024)
    // 46.8 us against 27.1 for the 16 x 16 ones, 56 tiles (840 x 256 x 256)
    // 12.9 against 12.8, 128 tiles (1024 x 512 x 512) 24.4 against 49.6; the
    // line is at 3/8 of the SMs
    const long tiles = (long)((ep.M + SG_TILE - 1) / SG_TILE) * ((ep.N + SG_TILE - 1) / SG_TILE);
    if (8 * tiles >= 3L * sm_count())
        return launch_pdl(gemm_simt_tile<EPI, VEC>, dim3((unsigned)tiles), dim3(SG_THREADS), 0, st, ep, A, Wt, K, skip);
    return launch_pdl(gemm_simt_small<EPI, VEC>, dim3((unsigned)((ep.M + 15) / 16 * (ep.N / 16))), dim3(SG_THREADS), 0,
                      st, ep, A, Wt, K, skip);
}

template <int EPI>
static cudaError_t gemm_simt_epi(const EpiParams &ep, const float *A, const float *Wt, int K, const uint8_t *skip,
                                 cudaStream_t st) {
    const bool vec = K % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0 && (reinterpret_cast<uintptr_t>(Wt) & 15) == 0;
    return vec ? gemm_simt_vec<EPI, true>(ep, A, Wt, K, skip, st) : gemm_simt_vec<EPI, false>(ep, A, Wt, K, skip, st);
}

cudaError_t gemm_simt(int epi, const EpiParams &ep, const float *A, const float *Wt, int K, const uint8_t *skip,
                      cudaStream_t st) {
    switch (epi) {
        case EPI_BIAS: return gemm_simt_epi<EPI_BIAS>(ep, A, Wt, K, skip, st);
        case EPI_GELU: return gemm_simt_epi<EPI_GELU>(ep, A, Wt, K, skip, st);
        case EPI_RESID_GATE: return gemm_simt_epi<EPI_RESID_GATE>(ep, A, Wt, K, skip, st);
        case EPI_RESID_CACHE: return gemm_simt_epi<EPI_RESID_CACHE>(ep, A, Wt, K, skip, st);
        case EPI_QKV_ROPE: return gemm_simt_epi<EPI_QKV_ROPE>(ep, A, Wt, K, skip, st);
        default: return cudaErrorInvalidValue;
    }
}

// ------------------------------------------------------------- attention
// o = softmax(q k^T / sqrt(hd)) v, online softmax in fp32.  CTA = 16 queries
// of one head, NW warps that share the keys: warp w takes the 32-key tiles
// w, w + NW, ... with its own running max, sum and unnormalised output, and
// the warps' results are merged in warp order at the end.  Within a tile a
// lane owns one key for the scores (its row of k in registers, the queries
// broadcast from shared memory) and then hd / 32 output dims (half the
// queries at hd 16) for P V, the probabilities passing through shared memory.
// One thread per (query, head), the layout before this one, put 256 threads
// on the chip at 64 tokens x 4 heads, each walking every key serially: 64
// queries x 192 keys x 4 heads x 16 86.7 -> 9.9 us (call to call), 1024 x
// 3072 x 8 x 64 7.09 -> 0.51 ms (12.7 TFLOP/s: issue-bound by the broadcast
// reads of queries and probabilities).
constexpr int SA_Q = 16, SA_K = 32;
template <int HD, int NW>
struct SaSmem {
    float q[SA_Q][HD];
    union {
        float p[NW][SA_K][SA_Q + 4];                 // probabilities of a warp's tile
        float o[NW][SA_Q][HD];                       // unnormalised outputs, for the merge
    };
    float m[NW][SA_Q], l[NW][SA_Q];
};

template <int HD, int NW, bool VEC>
__global__ void __launch_bounds__(NW * 32)
    attn_simt_f32(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                  float *__restrict__ o, const int Lq, const int n_keys, const int H,
                  const uint8_t *__restrict__ skip_flag) {
    pdl_wait();
    pdl_release();
    if (skip_flag != nullptr && *skip_flag == XC_DEC_SKIP) return;
    constexpr int DPL = HD >= 32 ? HD / 32 : 1;      // output dims per lane
    constexpr int QPL = HD >= 32 ? SA_Q : SA_Q / 2;  // queries per lane in P V
    __shared__ __align__(16) SaSmem<HD, NW> sm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_qt = (Lq + SA_Q - 1) / SA_Q;
    const int h = blockIdx.x / n_qt, q0 = (blockIdx.x % n_qt) * SA_Q;
    const int d = H * HD;
    const float scale = 1.0f / sqrtf((float)HD);
    for (int i = tid; i < SA_Q * HD; i += NW * 32) {
        const int r = i / HD, c = i % HD;
        sm.q[r][c] = q0 + r < Lq ? q[(size_t)(q0 + r) * d + h * HD + c] * scale : 0.0f;
    }
    __syncthreads();
    const int od = HD >= 32 ? lane * DPL : lane % HD;            // first output dim
    const int oq = HD >= 32 ? 0 : (lane / HD) * QPL;             // first query of P V
    float m[SA_Q], l[SA_Q], acc[QPL][DPL];
#pragma unroll
    for (int i = 0; i < SA_Q; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.0f;
    }
#pragma unroll
    for (int i = 0; i < QPL; ++i)
#pragma unroll
        for (int e = 0; e < DPL; ++e) acc[i][e] = 0.0f;
    const int n_kt = (n_keys + SA_K - 1) / SA_K;
    for (int kt = warp; kt < n_kt; kt += NW) {
        const int key = kt * SA_K + lane;
        const float *kr = k + (size_t)min(key, n_keys - 1) * d + h * HD;
        float s[SA_Q];
#pragma unroll
        for (int i = 0; i < SA_Q; ++i) s[i] = 0.0f;
#pragma unroll
        for (int c = 0; c < HD; c += 4) {
            const float4 kv = load_k4<VEC>(kr, c, HD);
#pragma unroll
            for (int i = 0; i < SA_Q; ++i) {
                const float4 qv = *reinterpret_cast<const float4 *>(&sm.q[i][c]);
                s[i] = fmaf(qv.x, kv.x, s[i]);
                s[i] = fmaf(qv.y, kv.y, s[i]);
                s[i] = fmaf(qv.z, kv.z, s[i]);
                s[i] = fmaf(qv.w, kv.w, s[i]);
            }
        }
        float alpha[SA_Q];
#pragma unroll
        for (int i = 0; i < SA_Q; ++i) {
            float mx = key < n_keys ? s[i] : -INFINITY;
#pragma unroll
            for (int w = 16; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
            // (a tile of -inf scores keeps m = -inf: no inf - inf)
            mx = fmaxf(mx, m[i]);
            alpha[i] = mx == m[i] ? 1.0f : expf(m[i] - mx);
            m[i] = mx;
            s[i] = key < n_keys && s[i] != -INFINITY ? expf(s[i] - mx) : 0.0f;
            l[i] = l[i] * alpha[i] + s[i];
        }
#pragma unroll
        for (int i = 0; i < QPL; ++i)
#pragma unroll
            for (int e = 0; e < DPL; ++e) acc[i][e] *= HD >= 32 ? alpha[i] : (lane < HD ? alpha[i] : alpha[i + SA_Q - QPL]);
#pragma unroll
        for (int i = 0; i < SA_Q; i += 4)
            *reinterpret_cast<float4 *>(&sm.p[warp][lane][i]) = make_float4(s[i], s[i + 1], s[i + 2], s[i + 3]);
        __syncwarp();
        const float *vb = v + (size_t)(kt * SA_K) * d + h * HD + od;
        const int nk = min(SA_K, n_keys - kt * SA_K);
#pragma unroll 4
        for (int j = 0; j < nk; ++j) {
            float vv[DPL];
            if constexpr (VEC && DPL == 2) {
                const float2 t = *reinterpret_cast<const float2 *>(vb + (size_t)j * d);
                vv[0] = t.x;
                vv[1] = t.y;
            } else {
#pragma unroll
                for (int e = 0; e < DPL; ++e) vv[e] = vb[(size_t)j * d + e];
            }
#pragma unroll
            for (int i = 0; i < QPL; i += 4) {
                const float4 p = *reinterpret_cast<const float4 *>(&sm.p[warp][j][oq + i]);
                const float pv[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                for (int t = 0; t < 4; ++t)
#pragma unroll
                    for (int e = 0; e < DPL; ++e) acc[i + t][e] = fmaf(pv[t], vv[e], acc[i + t][e]);
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < SA_Q; ++i)
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], w);
    __syncthreads();                                 // every warp is done with sm.p (sm.o shares its space)
#pragma unroll
    for (int i = 0; i < QPL; ++i)
#pragma unroll
        for (int e = 0; e < DPL; ++e) sm.o[warp][oq + i][od + e] = acc[i][e];
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < SA_Q; ++i) {
            sm.m[warp][i] = m[i];
            sm.l[warp][i] = l[i];
        }
    }
    __syncthreads();
    // merge the warps in warp order; a warp without a tile has m = -inf, weight 0
    for (int i = tid; i < SA_Q * HD; i += NW * 32) {
        const int r = i / HD, c = i % HD;
        if (q0 + r >= Lq) continue;
        float mm = sm.m[0][r];
#pragma unroll
        for (int w = 1; w < NW; ++w) mm = fmaxf(mm, sm.m[w][r]);
        float den = 0.0f, num = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float f = expf(sm.m[w][r] - mm);
            den = fmaf(sm.l[w][r], f, den);
            num = fmaf(sm.o[w][r][c], f, num);
        }
        o[(size_t)(q0 + r) * d + h * HD + c] = num / den;
    }
}

template <int HD, bool VEC>
static cudaError_t attn_simt_vec(const float *q, const float *k, const float *v, float *o, int Lq, int n_keys, int H,
                                 const uint8_t *skip, cudaStream_t st) {
    const long n = (long)((Lq + SA_Q - 1) / SA_Q) * H;
    // eight warps over the keys while all CTAs are resident at once (their
    // registers: one CTA per SM at hd 64, two below), four beyond.  Both
    // measured, eight / four warps: 300 x 2000 x 4 x 32 (76 CTAs) 53 / 91
    // us, 1024 x 3072 x 2 x 64 (128) 115 / 183, 640 x 640 x 4 x 64 (160) 57 / 50
    if (n > (HD >= 64 ? 1L : 2L) * sm_count())
        return launch_pdl(attn_simt_f32<HD, 4, VEC>, dim3((unsigned)n), dim3(128), 0, st, q, k, v, o, Lq, n_keys, H, skip);
    return launch_pdl(attn_simt_f32<HD, 8, VEC>, dim3((unsigned)n), dim3(256), 0, st, q, k, v, o, Lq, n_keys, H, skip);
}
template <int HD>
static cudaError_t attn_simt_hd(const float *q, const float *k, const float *v, float *o, int Lq, int n_keys, int H,
                                const uint8_t *skip, cudaStream_t st) {
    // k and v rows are multiples of 16 floats apart: 16-byte loads when the bases allow them
    const bool vec = ((reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v)) & 15) == 0;
    return vec ? attn_simt_vec<HD, true>(q, k, v, o, Lq, n_keys, H, skip, st)
               : attn_simt_vec<HD, false>(q, k, v, o, Lq, n_keys, H, skip, st);
}

cudaError_t attn_simt(int head_dim, const float *q, const float *k, const float *v, float *o, int Lq, int n_keys,
                      int H, const uint8_t *skip, cudaStream_t st) {
    switch (head_dim) {
        case 16: return attn_simt_hd<16>(q, k, v, o, Lq, n_keys, H, skip, st);
        case 32: return attn_simt_hd<32>(q, k, v, o, Lq, n_keys, H, skip, st);
        case 64: return attn_simt_hd<64>(q, k, v, o, Lq, n_keys, H, skip, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace xc
