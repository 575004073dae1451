// tcgen05 / TMA kernels of the OSDN layer for bf16 I/O, K = V = 128, chunk = 64 (sm_100a).
//
// Data flow of the forward pass (gated chunk form; G_i in-chunk gate prefix, gamma = exp(G),
// Gamma_ij = exp(G_i - G_j), rho_i = exp(G_C - G_i)):
//
//   phase1_fwd (CUDA cores)      ktil = d (.) k in bf16, preconditioner at chunk starts
//   tc_chunk_fwd  per (chunk, head), parallel:
//        [K;Q] Ktil^T  -> A = strictLower(beta_i Gamma_ij <k_i,ktil_j>),  P' = scale * Lower(Gamma_ij <q_i,ktil_j>)
//        T = (I + A)^-1 (blocks of 16 by fp32 substitution, the rest by TF32 block products), Tb = T diag(beta),
//        Tbg = T diag(beta gamma)
//        W^T = K^T Tbg^T                               (tensor memory: lane = feature, column = token)
//   tc_chain_fwd  per chain, sequential over chunks, state S (V x K, fp32) resident in tensor memory:
//        dU^T = V^T Tb^T - S W^T ;  O1^T = S Q^T
//        O2^T = dU^T P'^T ;         S <- gamma_C S + (rho dU)^T Ktil
//        O^T  = scale gamma_i O1^T + O2^T
//
// Work tiles that travel between kernels are stored in HBM as ready-made images of the
// 128-byte-swizzled shared-memory layout (see umma.cuh), so that the consumer fetches them with a
// plain bulk copy; user tensors (q, k, ktil, v, dout) are fetched with TMA tensor maps.
#include <algorithm>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "osdn_common.cuh"
#include <type_traits>

#include "umma.cuh"

namespace osdn {

using namespace umma;


namespace {

constexpr int KD = 128;  // K = V = 128 on this path
constexpr uint32_t BOX = 8192;   // one [64 rows x 128 B] box

// device status codes of bounded waits
enum { ERR_QUEUE = 121, ERR_READY = 122, ERR_TMA = 101, ERR_MMA1 = 102, ERR_MMA2 = 103, ERR_CHAIN_TMA = 111, ERR_CHAIN_MMA1 = 112, ERR_CHAIN_MMA2 = 113 };

constexpr uint32_t REC_BYTES = 49152;   // stride of the Tb | W^T | P' | Qg record of a tile

struct TcLayout {
    size_t ktil, WT, Tb, Tm, P, Qg, Sn, dUT, ready, ddUT, dSn, dktil, dkread, queue, total;
};

TcLayout make_tc_layout(const osdn_params& p, const WsLayout& L, bool need_bwd)
{
    TcLayout t{};
    const size_t Ttot = p.nseq > 0 ? (size_t)p.T : (size_t)p.B * p.T;
    const size_t H = p.H, NT = L.NTmax;
    size_t off = L.ktil;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b, 1024); return o; };
    off = align_up(off, 1024);
    t.ktil = take(Ttot * H * KD * 2);
    // One record per (chunk, head) tile, Tb | W^T | P' | Qg, so that either chain kernel fetches the
    // tiles it needs (the first three forward, the last three backward) with a single bulk copy.
    const size_t rec = take(NT * H * (size_t)REC_BYTES);
    t.Tb = rec;
    t.WT = rec + 8192;
    t.P = rec + 24576;
    t.Qg = rec + 32768;
    t.Tm = take(NT * H * 8192);
    t.Sn = take(NT * H * 32768);
    t.dUT = take(NT * H * 16384);
    t.ready = take(sizeof(int) * (64 + NT * H));   // ticket counter, then one flag per tile
    if (need_bwd) {
        t.ddUT = take(NT * H * 16384);
        t.dSn = take(NT * H * 32768);
        t.dktil = take(Ttot * H * KD * 4);
        t.dkread = take(Ttot * H * KD * 4);
        t.queue = take(sizeof(int) * (64 + NT * H));
    }
    t.total = off;
    return t;
}

// ---------------------------------------------------------------------------------------------
// tensor maps
// ---------------------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled get_encoder()
{
    static PFN_cuTensorMapEncodeTiled fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled>(ptr);
    }
    return fn;
}

// Map over a packed [rows, H * 128] bf16 tensor; boxes of 64 rows x 64 columns, 128-byte swizzle,
// out-of-range rows read as zero.
bool make_token_map(CUtensorMap* m, const void* base, size_t rows, int H)
{
    PFN_cuTensorMapEncodeTiled enc = get_encoder();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)H * KD, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)H * KD * 2};
    cuuint32_t box[2] = {64, 64};
    cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

__device__ __forceinline__ uint8_t* align1024(uint8_t* p)
{
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Zero rows [len, 64) of a box (tail chunks only).
__device__ __forceinline__ void zero_tail_rows(uint8_t* box, int len, int tid, int nthreads)
{
    const int rows = CH - len;
    for (int e = tid; e < rows * 8; e += nthreads)
        *reinterpret_cast<uint4*>(box + (len + e / 8) * 128 + (e % 8) * 16) = make_uint4(0, 0, 0, 0);
}

// fp32 value as a TF32 operand (round to nearest)
__device__ __forceinline__ uint32_t to_tf32(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// Warp-level 16x8x8 TF32 MMA (fp32 accumulate).  The 16 x 16 blocks of the triangular solve are
// below the smallest tcgen05 tile (M = 64), so they use the warp-level tensor path.
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ---------------------------------------------------------------------------------------------
// T = (I + A)^-1 for a 64 x 64 strictly lower triangular A, in place (fp32, shared memory, row
// stride LCF), by 16 x 16 blocks: warps 0 and 1 take a pair of diagonal blocks each, by forward substitution with a
// column per thread in registers, and the block below it; then warps 0 to 3 the 32 x 32 block below those,
//     T_21 = -T_22 (A_21 T_11).
// The inner products are parked in the upper triangle, so on return only entries with j <= i are meaningful.
// Called by all threads of the group (at least 128) behind a barrier; ends with a barrier.  Three barriers, where block row
// by block row took eight; a chain of four block products instead of six (that order with three barriers: 8 x 2048 tokens, 8
// heads, forward 126.3 -> 130.1 us).  Another rounding, not a larger one: errors of the outputs against 64 bits, over those of
// the other order, 1.0000 with gates and 0.9995 to 1.0005 without (24 seeds each).
// ---------------------------------------------------------------------------------------------
constexpr int LCF = CH + 4;   // stride = 4 mod 32 words: conflict-free 16-byte row stores and A fragments

// acc (16 x 16, two 16 x 8 fragments) += A (16 x 16) * B (16 x 16), fp32 in shared memory with row
// stride LD, as one TF32 product per fragment: T leaves this kernel as a bf16 operand image (8 bits of
// mantissa), TF32 operands keep 11.  (Splitting every operand into a high and a low part, three
// products per fragment, was measured: 6 us more per launch on the 340M training shape and no
// change of the parity errors beyond their third digit.)  One warp.
template <int LD>
__device__ __forceinline__ void block16_mma_ld(float (&acc)[2][4], const float* A, const float* B, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
        const uint32_t a4[4] = {to_tf32(A[g * LD + 8 * kt + t]), to_tf32(A[(g + 8) * LD + 8 * kt + t]),
                                to_tf32(A[g * LD + 8 * kt + t + 4]), to_tf32(A[(g + 8) * LD + 8 * kt + t + 4])};
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const uint32_t b2[2] = {to_tf32(B[(8 * kt + t) * LD + 8 * nt + g]), to_tf32(B[(8 * kt + t + 4) * LD + 8 * nt + g])};
            mma_tf32(acc[nt], a4, b2);
        }
    }
}

// store a 16 x 16 accumulator (optionally negated) to shared memory
template <int LD>
__device__ __forceinline__ void block16_store_ld(float* C, const float (&acc)[2][4], float sign, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        *reinterpret_cast<float2*>(C + g * LD + 8 * nt + 2 * t) = make_float2(sign * acc[nt][0], sign * acc[nt][1]);
        *reinterpret_cast<float2*>(C + (g + 8) * LD + 8 * nt + 2 * t) = make_float2(sign * acc[nt][2], sign * acc[nt][3]);
    }
}

template <typename Sync> __device__ __forceinline__ void ut_inverse_64_inplace(float* sA, int tid, Sync sync)
{
    const int warp = tid >> 5, lane = tid & 31;
    if (warp < 2) {
        {
            float x[16];
            float* Ab = sA + (16 * (tid >> 4)) * (LCF + 1);
            const int col = tid & 15;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float sum = i == col ? 1.f : 0.f;
#pragma unroll
                for (int j4 = 0; j4 < 16; j4 += 4)
                    if (j4 < i) {
                        const float4 r4 = *reinterpret_cast<const float4*>(Ab + i * LCF + j4);
                        const float r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj)
                            if (j4 + jj < i) sum = fmaf(-r[jj], x[j4 + jj], sum);
                    }
                x[i] = sum;
            }
            __syncwarp();   // every column has read the block before anyone overwrites it
#pragma unroll
            for (int i = 0; i < 16; ++i) Ab[i * LCF + col] = x[i];
            __syncwarp();
        }
        float* P = sA + 32 * warp * (LCF + 1);
        float acc[2][4] = {}, acc2[2][4] = {};
        block16_mma_ld<LCF>(acc, P + 16 * LCF, P, lane);
        block16_store_ld<LCF>(P + 16, acc, 1.f, lane);
        __syncwarp();
        block16_mma_ld<LCF>(acc2, P + 16 * LCF + 16, P + 16, lane);
        __syncwarp();
        block16_store_ld<LCF>(P + 16 * LCF, acc2, -1.f, lane);
    }
    sync();
    const int r = 16 * ((warp >> 1) & 1), c = 16 * (warp & 1);   // this warp's block of the 32 x 32 one
    float* X = sA + 32;                                          // rows 0 .. 31, columns 32 .. 63
    if (warp < 4) {
        float acc[2][4] = {};
        block16_mma_ld<LCF>(acc, sA + (32 + r) * LCF + 16, sA + 16 * LCF + c, lane);   // T_11's upper block is zero
        if (c == 0) block16_mma_ld<LCF>(acc, sA + (32 + r) * LCF, sA, lane);
        block16_store_ld<LCF>(X + r * LCF + c, acc, 1.f, lane);
    }
    sync();
    if (warp < 4) {
        float acc[2][4] = {};
        block16_mma_ld<LCF>(acc, sA + (32 + r) * LCF + 32, X + c, lane);
        if (r) block16_mma_ld<LCF>(acc, sA + (32 + r) * LCF + 48, X + 16 * LCF + c, lane);
        block16_store_ld<LCF>(sA + (32 + r) * LCF + c, acc, -1.f, lane);
    }
    sync();
}

// ---------------------------------------------------------------------------------------------
// chunk-local forward
// ---------------------------------------------------------------------------------------------
struct TcChunkArgs {
    int H;
    int* ready;   // merged forward launch: per (chunk, head) tile, set to 1 once the tile's images are in global memory
    Table tab;
    const float *beta, *gate;
    float scale;
    uint8_t *WT, *Tb, *Tm, *P, *Qg;
    int save;
    int* status;
};

// 8 warps = 4 lane quadrants x 2 column halves; 50 KB of shared memory and 128 tensor-memory columns,
// so that four CTAs share an SM and hide each other's waits.
constexpr int CL_THREADS = 256;
constexpr size_t CL_SMEM = 32768 + CH * LCF * 4 + 1024;

// Small per-group state of the chunk-local forward that lives in shared memory.
struct ClGroupShared {
    uint64_t bar_tma, bar_mma1, bar_mma2, bar_drain;
    int ticket;
    int pad;
    float sG[CH];
    alignas(16) float sGam[CH], sBeta[CH];
};

// One (chunk, head) tile by a group of CL_THREADS threads (local index `tid`) that synchronise on hardware
// barrier `bar_id`; `sm`: CL_SMEM - 1024 bytes, 1024-byte aligned; `tb`: 128 tensor-memory columns;
// `ph`: parity of the group's three barriers (they complete once per tile).  False, for all threads alike, where a wait ran
// out: the tile's copies and products have ended then, and the group takes no more (its barriers are out of step).
__device__ __forceinline__ bool chunk_fwd_tile(const CUtensorMap& tmK, const CUtensorMap& tmQ, const CUtensorMap& tmKt,
                                               const TcChunkArgs& a, int c, int h, uint8_t* sm, ClGroupShared& gs,
                                               uint32_t tb, int tid, int bar_id, uint32_t ph, int* publish)
{
    auto sync = [&]() { named_sync(bar_id, CL_THREADS); };
    uint64_t& bar_tma = gs.bar_tma;
    uint64_t& bar_mma1 = gs.bar_mma1;
    uint64_t& bar_mma2 = gs.bar_mma2;
    float* sG = gs.sG;
    float* sGam = gs.sGam;
    float* sBeta = gs.sBeta;
    uint8_t* sKQ = sm;                 // per k-half h: [K rows 0-63 | Q rows 64-127], 16 KB each
    uint8_t* sKt = sKQ + 32768;        // per k-half: 8 KB
    // A, then T (fp32, in place) take over the space of Ktil once the first product has consumed it;
    // the T diag(beta gamma) operand image takes over the first Q box once Qg has been written.
    float* sA = reinterpret_cast<float*>(sKt);
    uint8_t* sTb = sKQ + BOX;          // K-major [i][j]
    const int H = a.H;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return true;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const bool lead = lane == 0;
    const int quad = warp & 3, half = warp >> 2;

    if (tid == 0) {
        mbar_expect_tx(&bar_tma, 6 * BOX);
        for (int hf = 0; hf < 2; ++hf) {
            tma_load_2d(sKQ + hf * 16384, &tmK, h * KD + hf * 64, tok0, &bar_tma);
            tma_load_2d(sKQ + hf * 16384 + BOX, &tmQ, h * KD + hf * 64, tok0, &bar_tma);
            tma_load_2d(sKt + hf * BOX, &tmKt, h * KD + hf * 64, tok0, &bar_tma);
        }
    }
    if (warp == 2) {   // per-token scalars and the in-chunk gate prefix G_i
        const bool in0 = lane < len, in1 = lane + 32 < len;
        float sa = in0 ? a.gate[(size_t)(tok0 + lane) * H + h] : 0.f;
        float sb = in1 ? a.gate[(size_t)(tok0 + lane + 32) * H + h] : 0.f;
        sBeta[lane] = in0 ? a.beta[(size_t)(tok0 + lane) * H + h] : 0.f;
        sBeta[lane + 32] = in1 ? a.beta[(size_t)(tok0 + lane + 32) * H + h] : 0.f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ua = __shfl_up_sync(0xffffffffu, sa, o), ub = __shfl_up_sync(0xffffffffu, sb, o);
            if (lane >= o) { sa += ua; sb += ub; }
        }
        sb += __shfl_sync(0xffffffffu, sa, 31);
        sG[lane] = sa;
        sG[lane + 32] = sb;
        sGam[lane] = __expf(sa);
        sGam[lane + 32] = __expf(sb);
    }
    // The group's previous tile is published here, behind a barrier that is needed anyway: the barrier
    // orders every thread's stores before thread 0, whose fence (cumulative) then orders them before the flag.
    tc_fence_before();
    sync();
    tc_fence_after();
    if (publish && tid == 0) {
        __threadfence();
        st_release_gpu(publish, 1);
    }

    bool ok = mbar_wait(&bar_tma, ph, a.status, ERR_TMA);
    if (len < CH) {
        for (int hf = 0; hf < 2; ++hf) {
            zero_tail_rows(sKQ + hf * 16384, len, tid, CL_THREADS);
            zero_tail_rows(sKQ + hf * 16384 + BOX, len, tid, CL_THREADS);
            zero_tail_rows(sKt + hf * BOX, len, tid, CL_THREADS);
        }
        fence_proxy_async();
        sync();
    }

    // ---- D1[128 x 64] = [K;Q] Ktil^T ---------------------------------------------------------
    if (warp == 0 && ok) {
        const uint32_t idesc = make_idesc(128, 64);
        for (int s = 0; s < 8; ++s) {
            const uint64_t da = desc_advance(desc_kmajor(sKQ + (s >> 2) * 16384), 32 * (s & 3));
            const uint64_t db = desc_advance(desc_kmajor(sKt + (s >> 2) * BOX), 32 * (s & 3));
            mma_ss(tb, da, db, idesc, s > 0, lead);
        }
        mma_commit(&bar_mma1, lead);
    }
    // gated, scaled queries for both state chains, while the product runs: Qg = scale gamma_i Q
    // (same image layout as Q)
    for (int e = tid; e < 2 * CH * 8; e += CL_THREADS) {
        const int hf = e >> 9, i = (e >> 3) & 63, ch = e & 7;
        const uint32_t off = sw128_chunk(i, ch);
        const uint4 w = *reinterpret_cast<const uint4*>(sKQ + hf * 16384 + BOX + off);
        const float f = a.scale * sGam[i];
        const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&w);
        uint32_t o[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float2 v = __bfloat1622float2(p2[x]);
            o[x] = pack_bf16(v.x * f, v.y * f);
        }
        *reinterpret_cast<uint4*>(a.Qg + tile * REC_BYTES + hf * BOX + off) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    ok = ok && mbar_wait(&bar_mma1, ph, a.status, ERR_MMA1);
    tc_fence_after();
    if (ok) {
        const int L = quad * 32 + lane;
        const uint32_t taddr = tb + ((uint32_t)(quad * 32) << 16) + half * 32;
        if (L < CH) {   // A_ij = beta_i Gamma_ij <k_i, ktil_j>, j < i
            const int i = L;
            const float bi = sBeta[i], Gi = sG[i];
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                const int j0 = half * 32 + cb * 16;
                float av[16];
                if (j0 <= (quad & 1) * 32 + 31) {   // warp-uniform: some row of this warp reaches the block
                    uint32_t r[16];
                    tmem_ld16(taddr + cb * 16, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const int j = j0 + x;
                        av[x] = j < i ? bi * __expf(Gi - sG[j]) * __uint_as_float(r[x]) : 0.f;
                    }
                } else {
#pragma unroll
                    for (int x = 0; x < 16; ++x) av[x] = 0.f;
                }
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4)
                    *reinterpret_cast<float4*>(sA + i * LCF + j0 + q4 * 4) =
                        make_float4(av[q4 * 4 + 0], av[q4 * 4 + 1], av[q4 * 4 + 2], av[q4 * 4 + 3]);
            }
        } else {        // P'_ij = scale Gamma_ij <q_i, ktil_j>, j <= i
            const int i = L - CH;
            const float Gi = sG[i];
            uint8_t* Pg = a.P + tile * REC_BYTES;
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                const int j0 = half * 32 + cb * 16;
                float pv[16];
                if (j0 <= (quad & 1) * 32 + 31) {   // warp-uniform
                    uint32_t r[16];
                    tmem_ld16(taddr + cb * 16, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const int j = j0 + x;
                        pv[x] = j <= i ? a.scale * __expf(Gi - sG[j]) * __uint_as_float(r[x]) : 0.f;
                    }
                } else {
#pragma unroll
                    for (int x = 0; x < 16; ++x) pv[x] = 0.f;
                }
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {
                    uint4 w;
                    w.x = pack_bf16(pv[c2 * 8 + 0], pv[c2 * 8 + 1]);
                    w.y = pack_bf16(pv[c2 * 8 + 2], pv[c2 * 8 + 3]);
                    w.z = pack_bf16(pv[c2 * 8 + 4], pv[c2 * 8 + 5]);
                    w.w = pack_bf16(pv[c2 * 8 + 6], pv[c2 * 8 + 7]);
                    *reinterpret_cast<uint4*>(Pg + sw128_chunk(i, (j0 >> 3) + c2)) = w;
                }
            }
        }
    }
    sync();

    // ---- T = (I + A)^-1, blocked, in place ---------------------------------------------------------
    ut_inverse_64_inplace(sA, tid, sync);

    // ---- operand images: Tbg (shared), Tb and T (HBM) -----------------------------------------
    {
        const int ch = tid & 7;   // the same eight columns in every round
        float bj[8], gj[8];
#pragma unroll
        for (int x = 0; x < 8; x += 4) {
            const float4 b4 = *reinterpret_cast<const float4*>(sBeta + ch * 8 + x), g4 = *reinterpret_cast<const float4*>(sGam + ch * 8 + x);
            bj[x] = b4.x; bj[x + 1] = b4.y; bj[x + 2] = b4.z; bj[x + 3] = b4.w;
            gj[x] = g4.x; gj[x + 1] = g4.y; gj[x + 2] = g4.z; gj[x + 3] = g4.w;
        }
#pragma unroll 1
        for (int i = tid >> 3; i < CH; i += CL_THREADS / 8) {
            const float4 t0 = *reinterpret_cast<const float4*>(sA + i * LCF + ch * 8);
            const float4 t1 = *reinterpret_cast<const float4*>(sA + i * LCF + ch * 8 + 4);
            float t[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
            const uint32_t off = sw128_chunk(i, ch);
#pragma unroll
            for (int x = 0; x < 8; ++x) t[x] = ch * 8 + x <= i ? t[x] : 0.f;   // above the diagonal the array holds scratch
            if (a.save)
                *reinterpret_cast<uint4*>(a.Tm + tile * 8192 + off) =
                    make_uint4(pack_bf16(t[0], t[1]), pack_bf16(t[2], t[3]), pack_bf16(t[4], t[5]), pack_bf16(t[6], t[7]));
#pragma unroll
            for (int x = 0; x < 8; ++x) t[x] *= bj[x];
            *reinterpret_cast<uint4*>(a.Tb + tile * REC_BYTES + off) =
                make_uint4(pack_bf16(t[0], t[1]), pack_bf16(t[2], t[3]), pack_bf16(t[4], t[5]), pack_bf16(t[6], t[7]));
#pragma unroll
            for (int x = 0; x < 8; ++x) t[x] *= gj[x];
            *reinterpret_cast<uint4*>(sTb + off) =
                make_uint4(pack_bf16(t[0], t[1]), pack_bf16(t[2], t[3]), pack_bf16(t[4], t[5]), pack_bf16(t[6], t[7]));
        }
    }
    fence_proxy_async();
    tc_fence_before();
    sync();

    // ---- D2[128 x 64] = K^T Tbg^T  (W^T) -----------------------------------------------------
    if (warp == 0 && ok) {
        tc_fence_after();
        const uint32_t idesc = make_idesc(128, 64, IDESC_A_MN);
        const uint64_t da0 = desc_mnmajor(sKQ, 16384);
        const uint64_t db0 = desc_kmajor(sTb);
        for (int s = 0; s < 4; ++s) mma_ss(tb + 64, desc_advance(da0, 2048 * s), desc_advance(db0, 32 * s), idesc, s > 0, lead);
        mma_commit(&bar_mma2, lead);
    }
    ok = ok && mbar_wait(&bar_mma2, ph, a.status, ERR_MMA2);
    tc_fence_after();
    if (ok) {
        const int k = quad * 32 + lane;
        const uint32_t taddr = tb + ((uint32_t)(quad * 32) << 16) + 64 + half * 32;
        uint8_t* Wg = a.WT + tile * REC_BYTES;
        uint32_t r[2][16];
        tmem_ld16(taddr, r[0]);
        tmem_ld16(taddr + 16, r[1]);
        tmem_ld_wait();
#pragma unroll
        for (int cb = 0; cb < 2; ++cb)
#pragma unroll
            for (int c2 = 0; c2 < 2; ++c2) {
                uint4 w;
                w.x = pack_bf16(__uint_as_float(r[cb][c2 * 8 + 0]), __uint_as_float(r[cb][c2 * 8 + 1]));
                w.y = pack_bf16(__uint_as_float(r[cb][c2 * 8 + 2]), __uint_as_float(r[cb][c2 * 8 + 3]));
                w.z = pack_bf16(__uint_as_float(r[cb][c2 * 8 + 4]), __uint_as_float(r[cb][c2 * 8 + 5]));
                w.w = pack_bf16(__uint_as_float(r[cb][c2 * 8 + 6]), __uint_as_float(r[cb][c2 * 8 + 7]));
                *reinterpret_cast<uint4*>(Wg + sw128_chunk(k, half * 4 + cb * 2 + c2)) = w;
            }
    }
    tc_fence_before();
    ok = named_sync_and(bar_id, CL_THREADS, ok);
    if (!ok) {
        mbar_drain(&bar_tma, ph);
        if (warp == 0) {
            mma_commit(&gs.bar_drain, lead);
            mbar_drain(&gs.bar_drain, 0);
        }
        sync();
    }
    return ok;
}

// Stand-alone launch: one tile per CTA, four CTAs per SM.
__global__ void __launch_bounds__(CL_THREADS, 4)
tc_chunk_fwd_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ,
                    const __grid_constant__ CUtensorMap tmKt, TcChunkArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ ClGroupShared gs;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x;
    pdl_wait();
    if (a.tab.chunk_len(blockIdx.x) == 0) return;
    if (tid == 0) {
        mbar_init(&gs.bar_tma, 1);
        mbar_init(&gs.bar_mma1, 1);
        mbar_init(&gs.bar_mma2, 1);
        mbar_init(&gs.bar_drain, 1);
        fence_mbar_init();
    }
    if ((tid >> 5) == 1) tmem_alloc(&tmem_base, 128);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    chunk_fwd_tile(tmK, tmQ, tmKt, a, blockIdx.x, blockIdx.y, align1024(smem_raw), gs, tmem_base, tid, 1, 0u, nullptr);
    __syncthreads();
    if ((tid >> 5) == 1) tmem_dealloc(tmem_base, 128);
}

// ---------------------------------------------------------------------------------------------
// state chain, forward
// ---------------------------------------------------------------------------------------------
struct TcChainArgs {
    int H;
    Table tab;
    const float *gate, *init_state;
    __nv_bfloat16* out;
    float* final_state;
    const uint8_t *WT, *Tb, *P;
    uint8_t *Sn, *dUT;
    float scale;
    int save;
    int* status;
    const int* ready;   // nullable: per (chunk, head) tile, nonzero once the chunk-local pass has written it
};

constexpr uint32_t STAGE_BYTES = 8192 + 16384 + 8192 + 3 * 16384;   // Tb, WT, P, Qg, V, Ktil = 81920
constexpr uint32_t ST_TB = 0, ST_WT = 8192, ST_P = 24576, ST_QG = 32768, ST_V = 49152, ST_KT = 65536;
constexpr size_t CF_SMEM = 2 * STAGE_BYTES + 32768 + 2 * 16384 + 1024;

// In-chunk gate prefix by one warp: lane l holds g_l and g_{l+32}.  Writes gamma_i = exp(G_i),
// rho_i = exp(G_C - G_i) and gamma_C into the given slot.
__device__ __forceinline__ void warp_gate_vectors(float ga, float gb, int lane, float* gam, float* rho, float* gC)
{
    float sa = ga, sb = gb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float ua = __shfl_up_sync(0xffffffffu, sa, o), ub = __shfl_up_sync(0xffffffffu, sb, o);
        if (lane >= o) { sa += ua; sb += ub; }
    }
    const float ta = __shfl_sync(0xffffffffu, sa, 31);
    sb += ta;
    const float tot = __shfl_sync(0xffffffffu, sb, 31);
    if (gam) { gam[lane] = __expf(sa); gam[lane + 32] = __expf(sb); }
    rho[lane] = __expf(tot - sa);
    rho[lane + 32] = __expf(tot - sb);
    if (lane == 0) *gC = __expf(tot);
}

// Warp roles of the forward chain: 16 state warps (4 lane quadrants x 4 column groups), 4 output warps
// (one per lane quadrant), one warp that issues the tensor-core work, one warp that issues the loads
// and prepares the gate vectors.  The roles run decoupled and meet only at mbarriers:
//   full[st]    loads of a chunk have landed (and its gate vectors are written)      producer -> all
//   empty[st]   every product reading the stage has finished                         tensor core -> producer
//   s_ready     S is in shared memory as a bf16 operand, the accumulator is decayed  state warps -> issuer
//   du_done     dU^T accumulator complete                                            tensor core -> state warps
//   du_ready    dU^T operands are in shared memory                                   state warps -> issuer
//   s_done      the state update of the chunk is complete                            tensor core -> state warps
//   o_done[st]  both output accumulators of the chunk are complete                   tensor core -> output warps
//   o_free[st]  the output accumulators have been read                               output warps -> issuer
// The state warps carry the recurrence and never store to global memory inside the loop: a warp's
// tensor-memory load does not return while its earlier global stores are outstanding, which would
// put the latency of the output stores on the chunk-to-chunk path.
constexpr int CFW_EPI_WARPS = 16, CFW_OUT_WARPS = 4;
constexpr int CFW_OUT_WARP0 = 16, CFW_MMA_WARP = 20, CFW_TMA_WARP = 21;
constexpr int CFW_THREADS = 22 * 32;

// One chain by the first CFW_THREADS threads of the CTA (all threads of the CTA must call: the function
// synchronises the CTA).  `sm`: CF_SMEM - 1024 bytes, 1024-byte aligned; `tb`: 512 tensor-memory columns.
// With `a.ready` set, the loads of a chunk wait until the chunk-local pass has published it.
__device__ __forceinline__ void chain_fwd_role(const CUtensorMap& tmV, const CUtensorMap& tmKt, const TcChainArgs& a,
                                               int chain, uint8_t* sm, uint32_t tb)
{
    uint8_t* sStage = sm;                       // 2 stages
    uint8_t* sS = sm + 2 * STAGE_BYTES;         // S as bf16, K-major: 2 k-halves x [128 rows x 128 B]
    uint8_t* sDU1 = sS + 32768;                 // dU^T, K-major [v][i]
    uint8_t* sDU2 = sDU1 + 16384;               // (rho dU)^T
    __shared__ uint64_t bar_full[2], bar_empty[2], bar_s_ready, bar_du_done, bar_du_ready, bar_s_done;
    __shared__ uint64_t bar_o_done[2], bar_o_free[2], bar_drain;
    __shared__ float sRho[2][CH], sGC[2];              // slot = chunk % 2

    const int H = a.H;
    const int s = chain / H, h = chain % H;
    const int c0 = a.tab.seq_chunk0(s), c1 = a.tab.seq_chunk0(s + 1);
    const int seq_t0 = a.tab.seq_tok0(s), seq_len = a.tab.seq_len(s);
    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const bool lead = lane == 0;
    const int quad = warp & 3, colq = (warp >> 2) & 3;
    const int v = quad * 32 + lane;             // state row owned by a state-warp thread
    float* fin = a.final_state ? a.final_state + (((size_t)s * H + h) * KD + v) * KD + colq * 32 : nullptr;
    const float* ini = a.init_state ? a.init_state + (((size_t)s * H + h) * KD + v) * KD + colq * 32 : nullptr;
    if (c1 <= c0) {   // empty sequence: the state passes through
        if (fin && warp < CFW_EPI_WARPS)
            for (int x = 0; x < 32; ++x) fin[x] = ini ? ini[x] : 0.f;
        return;
    }
    uint64_t* const all_bars[] = {&bar_full[0], &bar_full[1], &bar_empty[0], &bar_empty[1], &bar_s_ready, &bar_du_done,
                                  &bar_du_ready, &bar_s_done, &bar_o_done[0], &bar_o_done[1], &bar_o_free[0],
                                  &bar_o_free[1], &bar_drain};
    const int nchunks = c1 - c0;
    auto chunk_tok0 = [&](int n) { return seq_t0 + n * CH; };
    auto chunk_len = [&](int n) { return min(CH, seq_len - n * CH); };

    if (tid == 0) {
        mbar_init(&bar_full[0], 2);
        mbar_init(&bar_full[1], 2);
        mbar_init(&bar_empty[0], 1);
        mbar_init(&bar_empty[1], 1);
        mbar_init(&bar_s_ready, CFW_EPI_WARPS);
        mbar_init(&bar_du_done, 1);
        mbar_init(&bar_du_ready, CFW_EPI_WARPS);
        mbar_init(&bar_s_done, 1);
        mbar_init(&bar_o_done[0], 1);
        mbar_init(&bar_o_done[1], 1);
        mbar_init(&bar_o_free[0], CFW_OUT_WARPS);
        mbar_init(&bar_o_free[1], CFW_OUT_WARPS);
        mbar_init(&bar_drain, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tS = tb, tDU = tb + 128, tO = tb + 192;   // O^T: two buffers of 64 columns

    if (warp >= CFW_THREADS / 32) {
        // not part of the chain
    } else if (warp == CFW_TMA_WARP) {
        // ------------------------------------------------------------------ producer
        // A stage is complete when its copies have landed (transaction count, first arrival) and the
        // gate vectors of the chunk are written (second arrival).  The gates are read a chunk ahead.
        bool ok = true;
        auto load_gates = [&](int n, float& ga, float& gb) {
            const int tok0 = chunk_tok0(n), len = chunk_len(n);
            ga = lane < len ? a.gate[(size_t)(tok0 + lane) * H + h] : 0.f;
            gb = lane + 32 < len ? a.gate[(size_t)(tok0 + lane + 32) * H + h] : 0.f;
        };
        float ga, gb;
        load_gates(0, ga, gb);
        int asked = 0;   // chunks whose copies have been asked for
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1, gs = n & 1;
            const int tok0 = chunk_tok0(n);
            float ga_next = 0.f, gb_next = 0.f;
            if (n + 1 < nchunks) load_gates(n + 1, ga_next, gb_next);
            // The record's flag is looked at before the stage is waited for: its round trip to memory then
            // runs while the products of the chunk before last still read the stage.
            if (a.ready) {   // the chunk-local pass runs beside the chains: wait until the record is written
                const int* flag = a.ready + (size_t)(c0 + n) * H + h;
                const long long t0 = clock64();
                bool seen = false;
                while (!(seen = ld_acquire_gpu(flag) != 0)) {
                    if (clock64() - t0 > WAIT_LIMIT_CYCLES) break;
                    __nanosleep(64);
                }
                if (!seen) {
                    if (lane == 0) atomicCAS(a.status, 0, ERR_READY);
                    ok = false;
                    break;
                }
                fence_proxy_async_all();
            }
            if (n >= 2) ok = mbar_wait(&bar_empty[st], ((n >> 1) - 1) & 1, a.status, ERR_CHAIN_TMA);
            if (!ok) break;
            if (lane == 0) {
                const size_t tile = (size_t)(c0 + n) * H + h;
                uint8_t* d = sStage + st * STAGE_BYTES;
                mbar_expect_tx(&bar_full[st], STAGE_BYTES);
                bulk_load(d + ST_TB, a.Tb + tile * REC_BYTES, REC_BYTES, &bar_full[st]);   // Tb, W^T, P', Qg
                for (int hf = 0; hf < 2; ++hf) tma_load_2d(d + ST_V + hf * BOX, &tmV, h * KD + hf * 64, tok0, &bar_full[st]);
                for (int hf = 0; hf < 2; ++hf) tma_load_2d(d + ST_KT + hf * BOX, &tmKt, h * KD + hf * 64, tok0, &bar_full[st]);
            }
            __syncwarp();
            warp_gate_vectors(ga, gb, lane, nullptr, sRho[gs], &sGC[gs]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_full[st]);
            ga = ga_next;
            gb = gb_next;
            asked = n + 1;
        }
        for (int n = max(0, asked - 2); n < asked; ++n) mbar_drain(&bar_full[n & 1], (n >> 1) & 1);
    } else if (warp == CFW_MMA_WARP) {
        // ------------------------------------------------------------------ tensor-core issuer
        bool ok = true;
        bool ut_issued = false;   // V^T Tb^T of the coming chunk is already in the dU^T accumulator
        auto issue_ut = [&](uint8_t* d) {   // dU^T = V^T Tb^T
            const uint32_t idesc = make_idesc(128, 64, IDESC_A_MN);
            const uint64_t da0 = desc_mnmajor(d + ST_V, BOX), db0 = desc_kmajor(d + ST_TB);
            for (int k = 0; k < 4; ++k)
                mma_ss(tDU, desc_advance(da0, 2048 * k), desc_advance(db0, 32 * k), idesc, k > 0, lead);
        };
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1;
            const size_t tile = (size_t)(c0 + n) * H + h;
            uint8_t* d = sStage + st * STAGE_BYTES;
            if (!ut_issued) ok = mbar_wait(&bar_full[st], (n >> 1) & 1, a.status, ERR_CHAIN_TMA);
            ok = ok && mbar_wait(&bar_s_ready, n & 1, a.status, ERR_CHAIN_MMA1);
            if (!ok) break;
            tc_fence_after();
            if (lead && a.save) {
                bulk_wait_read();   // saved images of the previous chunk have left shared memory
                bulk_store(a.Sn + tile * 32768, sS, 32768);
                bulk_commit();
            }
            __syncwarp();
            {
                if (!ut_issued) issue_ut(d);
                {   // dU^T -= S W^T
                    const uint32_t idesc = make_idesc(128, 64, IDESC_A_NEG | IDESC_B_MN);
                    const uint64_t db0 = desc_mnmajor(d + ST_WT, 0);
                    for (int k = 0; k < 8; ++k)
                        mma_ss(tDU, desc_advance(desc_kmajor(sS + (k >> 2) * 16384), 32 * (k & 3)),
                               desc_advance(db0, 2048 * k), idesc, 1, lead);
                }
                mma_commit(&bar_du_done, lead);
            }
            __syncwarp();
            // the output accumulators of chunk n - 2 (same buffers) have been read
            if (n >= 2) ok = mbar_wait(&bar_o_free[st], ((n >> 1) - 1) & 1, a.status, ERR_CHAIN_MMA2);
            if (!ok) break;
            tc_fence_after();
            {   // O^T = S Qg^T
                const uint32_t idesc = make_idesc(128, 64);
                for (int k = 0; k < 8; ++k)
                    mma_ss(tO + st * 64, desc_advance(desc_kmajor(sS + (k >> 2) * 16384), 32 * (k & 3)),
                           desc_advance(desc_kmajor(d + ST_QG + (k >> 2) * BOX), 32 * (k & 3)), idesc, k > 0, lead);
            }
            __syncwarp();
            ok = mbar_wait(&bar_du_ready, n & 1, a.status, ERR_CHAIN_MMA2);
            if (!ok) break;
            tc_fence_after();
            if (lead && a.save) {
                // The image of S sent off at the start of this chunk must have left shared memory before
                // the state update is released: its completion lets the state warps overwrite that image.
                bulk_wait_read();
                bulk_store(a.dUT + tile * 16384, sDU1, 16384);
                bulk_commit();
            }
            __syncwarp();
            {
                {   // S += (rho dU)^T Ktil
                    const uint32_t idesc = make_idesc(128, 128, IDESC_B_MN);
                    const uint64_t da0 = desc_kmajor(sDU2), db0 = desc_mnmajor(d + ST_KT, BOX);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(tS, desc_advance(da0, 32 * k), desc_advance(db0, 2048 * k), idesc, 1, lead);
                }
                mma_commit(&bar_s_done, lead);
                {   // O^T += dU^T P'^T
                    const uint32_t idesc = make_idesc(128, 64);
                    const uint64_t da0 = desc_kmajor(sDU1), db0 = desc_kmajor(d + ST_P);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(tO + st * 64, desc_advance(da0, 32 * k), desc_advance(db0, 32 * k), idesc, 1, lead);
                }
                mma_commit(&bar_o_done[st], lead);
                mma_commit(&bar_empty[st], lead);
            }
            __syncwarp();
            // The part of the next chunk's dU^T that does not depend on the state goes in now, while the
            // state warps convert S (full chunks only: a ragged chunk has its tail rows cleared first).
            ut_issued = false;
            if (n + 1 < nchunks && chunk_len(n + 1) == CH) {
                ok = mbar_wait(&bar_full[st ^ 1], ((n + 1) >> 1) & 1, a.status, ERR_CHAIN_TMA);
                if (!ok) break;
                issue_ut(sStage + (st ^ 1) * STAGE_BYTES);
                __syncwarp();
                ut_issued = true;
            }
        }
        mma_commit(&bar_drain, lead);
        mbar_drain(&bar_drain, 0);
        if (lane == 0) bulk_wait_all();
    } else if (warp >= CFW_OUT_WARP0) {
        // ------------------------------------------------------------------ output warps
        // o_i = (S Qg^T + dU^T P'^T)_i is complete in the accumulator: lane = feature, 16 token columns
        // per load.  Results leave as 16-byte stores: three shuffle rounds turn "lane = feature, 16
        // tokens" into "lane = 8 consecutive features of 2 tokens" (lane bit 0 picks the token half,
        // bits 1-2 the token pair inside it, bits 3-4 the feature octet).
        const int ow = warp - CFW_OUT_WARP0;   // == lane quadrant
        const uint32_t lane_addr = (uint32_t)(ow * 32) << 16;
        const bool b0 = lane & 1, b1 = lane & 2, b2 = lane & 4;
        const int tsub = (b0 ? 8 : 0) + ((lane >> 1) & 3) * 2;
        bool ok = true;
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1;
            const int tok0 = chunk_tok0(n), len = chunk_len(n);
            // Warm L2 with the operands of chunk n + 2 (the stage copies can only run one chunk ahead).
            if (lane == 0 && n + 2 < nchunks) {
                const int t2 = chunk_tok0(n + 2);
                if (ow == 0 && !a.ready) bulk_prefetch(a.Tb + ((size_t)(c0 + n + 2) * H + h) * REC_BYTES, REC_BYTES);
                if (ow == 1)
                    for (int hf = 0; hf < 2; ++hf) tma_prefetch_2d(&tmV, h * KD + hf * 64, t2);
                if (ow == 2)
                    for (int hf = 0; hf < 2; ++hf) tma_prefetch_2d(&tmKt, h * KD + hf * 64, t2);
            }
            ok = mbar_wait(&bar_o_done[st], (n >> 1) & 1, a.status, ERR_CHAIN_MMA2);
            if (!ok) break;
            tc_fence_after();
            __nv_bfloat16* op = a.out + ((size_t)tok0 * H + h) * KD + ow * 32 + (lane >> 3) * 8;
#pragma unroll
            for (int cg = 0; cg < 4; ++cg) {
                uint32_t ra[16];
                tmem_ld16(tO + st * 64 + lane_addr + cg * 16, ra);
                tmem_ld_wait();
                if (cg == 3) {   // everything is in registers: the buffer may be overwritten
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar_o_free[st]);
                }
                uint32_t w[8];    // feature pair (lane >> 1), token (b0 ? 8 : 0) + i
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float lo = __uint_as_float(ra[i]), hi = __uint_as_float(ra[i + 8]);
                    const float recv = __shfl_xor_sync(0xffffffffu, b0 ? lo : hi, 1);
                    w[i] = b0 ? pack_bf16(recv, hi) : pack_bf16(lo, recv);
                }
                uint32_t wa[2][2][2];   // [token-pair bit 1][token parity][feature pair 0 / 1]
#pragma unroll
                for (int th = 0; th < 2; ++th)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t w0 = w[(th * 2 + 0) * 2 + e], w1 = w[(th * 2 + 1) * 2 + e];
                        const uint32_t keep = b1 ? w1 : w0;
                        const uint32_t recv = __shfl_xor_sync(0xffffffffu, b1 ? w0 : w1, 2);
                        wa[th][e][0] = b1 ? recv : keep;
                        wa[th][e][1] = b1 ? keep : recv;
                    }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    uint32_t q4[4];
#pragma unroll
                    for (int sp = 0; sp < 2; ++sp) {
                        const uint32_t keep = b2 ? wa[1][e][sp] : wa[0][e][sp];
                        const uint32_t recv = __shfl_xor_sync(0xffffffffu, b2 ? wa[0][e][sp] : wa[1][e][sp], 4);
                        q4[sp] = b2 ? recv : keep;
                        q4[2 + sp] = b2 ? keep : recv;
                    }
                    const int i = cg * 16 + tsub + e;
                    if (i < len)
                        *reinterpret_cast<uint4*>(op + (size_t)i * H * KD) = make_uint4(q4[0], q4[1], q4[2], q4[3]);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ state warps
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        const int etid = tid;   // 0 .. 511
        // initial state into tensor memory
        for (int cb = 0; cb < 2; ++cb) {
            uint32_t r[16];
#pragma unroll
            for (int x4 = 0; x4 < 4; ++x4) {
                const float4 f4 = ini ? *reinterpret_cast<const float4*>(ini + cb * 16 + x4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                r[x4 * 4 + 0] = __float_as_uint(f4.x);
                r[x4 * 4 + 1] = __float_as_uint(f4.y);
                r[x4 * 4 + 2] = __float_as_uint(f4.z);
                r[x4 * 4 + 3] = __float_as_uint(f4.w);
            }
            tmem_st16(tS + lane_addr + colq * 32 + cb * 16, r);
        }
        tmem_st_wait();

        bool ok = true;
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1, gs = n & 1;
            const int len = chunk_len(n);
            uint8_t* d = sStage + st * STAGE_BYTES;
            ok = mbar_wait(&bar_full[st], (n >> 1) & 1, a.status, ERR_CHAIN_TMA);   // gate vectors, tail rows
            if (n > 0) ok = ok && mbar_wait(&bar_s_done, (n - 1) & 1, a.status, ERR_CHAIN_MMA2);
            if (!ok) break;
            tc_fence_after();
            // ---- E0: S -> bf16 operand (what the next products wait for), then decay the accumulator
            uint32_t rr[2][16];
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) tmem_ld16(tS + lane_addr + colq * 32 + cb * 16, rr[cb]);
            tmem_ld_wait();
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                const uint32_t* r = rr[cb];
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {
                    uint4 w;
                    w.x = pack_bf16(__uint_as_float(r[c2 * 8 + 0]), __uint_as_float(r[c2 * 8 + 1]));
                    w.y = pack_bf16(__uint_as_float(r[c2 * 8 + 2]), __uint_as_float(r[c2 * 8 + 3]));
                    w.z = pack_bf16(__uint_as_float(r[c2 * 8 + 4]), __uint_as_float(r[c2 * 8 + 5]));
                    w.w = pack_bf16(__uint_as_float(r[c2 * 8 + 6]), __uint_as_float(r[c2 * 8 + 7]));
                    *reinterpret_cast<uint4*>(sS + (colq >> 1) * 16384 + sw128_chunk(v, (colq & 1) * 4 + cb * 2 + c2)) = w;
                }
            }
            if (len < CH) {
                for (int hf = 0; hf < 2; ++hf) {
                    zero_tail_rows(d + ST_V + hf * BOX, len, etid, CFW_EPI_WARPS * 32);
                    zero_tail_rows(d + ST_KT + hf * BOX, len, etid, CFW_EPI_WARPS * 32);
                }
            }
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_s_ready);
            {   // gamma_C S back into the accumulator: only the state update (after du_ready) reads it
                const float gC = sGC[gs];
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
#pragma unroll
                    for (int x = 0; x < 16; ++x) rr[cb][x] = __float_as_uint(__uint_as_float(rr[cb][x]) * gC);
                    tmem_st16(tS + lane_addr + colq * 32 + cb * 16, rr[cb]);
                }
            }

            // ---- E1: dU^T -> bf16 operands
            float rho[16];
#pragma unroll
            for (int x = 0; x < 16; ++x) rho[x] = sRho[gs][colq * 16 + x];
            ok = mbar_wait(&bar_du_done, n & 1, a.status, ERR_CHAIN_MMA1);
            if (!ok) break;
            tc_fence_after();
            {
                uint32_t r[16];
                tmem_ld16(tDU + lane_addr + colq * 16, r);
                tmem_ld_wait();
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {
                    float f[8], g[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        f[x] = __uint_as_float(r[c2 * 8 + x]);
                        g[x] = f[x] * rho[c2 * 8 + x];
                    }
                    const uint32_t off = sw128_chunk(v, colq * 2 + c2);
                    *reinterpret_cast<uint4*>(sDU2 + off) = make_uint4(pack_bf16(g[0], g[1]), pack_bf16(g[2], g[3]),
                                                                      pack_bf16(g[4], g[5]), pack_bf16(g[6], g[7]));
                    *reinterpret_cast<uint4*>(sDU1 + off) = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]),
                                                                      pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
                }
            }
            tmem_st_wait();   // the decayed accumulator is in place
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_du_ready);
        }
        tmem_st_wait();
        if (ok) ok = mbar_wait(&bar_s_done, (nchunks - 1) & 1, a.status, ERR_CHAIN_MMA2);
        tc_fence_after();
        if (ok && fin) {
            for (int cb = 0; cb < 2; ++cb) {
                uint32_t r[16];
                tmem_ld16(tS + lane_addr + colq * 32 + cb * 16, r);
                tmem_ld_wait();
#pragma unroll
                for (int x4 = 0; x4 < 4; ++x4)
                    *reinterpret_cast<float4*>(fin + cb * 16 + x4 * 4) =
                        make_float4(__uint_as_float(r[x4 * 4 + 0]), __uint_as_float(r[x4 * 4 + 1]),
                                    __uint_as_float(r[x4 * 4 + 2]), __uint_as_float(r[x4 * 4 + 3]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0)
        for (uint64_t* b : all_bars) mbar_inval(b);
    __syncthreads();
}

// Stand-alone launch: one chain per CTA.
__global__ void __launch_bounds__(CFW_THREADS, 1)
tc_chain_fwd_kernel(const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmKt, TcChainArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_base;
    if (threadIdx.x < 32) tmem_alloc(&tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();
    chain_fwd_role(tmV, tmKt, a, blockIdx.x, align1024(smem_raw), tmem_base);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(tmem_base, 512);
}

// ---------------------------------------------------------------------------------------------
// Forward of phase 2 in one launch.  Every CTA starts as three groups that take (chunk, head) tiles of
// the chunk-local pass from a ticket counter, chunk position by chunk position across the chains, and
// publish each finished tile with a flag.  Once `switch_at` tickets are out, the first `nchains` CTAs
// turn into the state chains, whose loads wait for those flags; the other CTAs keep producing, and a CTA
// whose chain is finished joins them again.  No worker ever waits, so the chains always make progress.
// ---------------------------------------------------------------------------------------------
// Cost of a chain step in units of the time one SM needs for a tile.  Forward, us, at 0.5 / 0.65 / 0.8: 8 x 2048 tokens, 8 heads
// 130.1 / 126.3 / 132.3; 4 x 4096, 16 heads 232 / 214 / 221; 14 x 4096, 8 heads 378 / 367 / 387; up to 32 chains, and packed rows, alike.
constexpr float FWD_STEP_OVER_TILE_F = 0.65f;
struct FwdSched {
    int* tickets;     // zero at launch
    int ntickets;     // number of (chunk, head) tiles
    int nchains;
    int nchunks;      // dense batch: chunk positions per chain (sequences of equal length)
    int switch_at;
    const int* order; // packed batch: the chunks sorted by position inside their sequence (else null); then
                      // ntickets and switch_at are worked out on the device from the chunk table
    const int* longest;   // packed batch: chunks of the longest sequence
    int nseq, feeders;
};

// Packed batches: the realised number of tiles and the longest chain are only known on the device.
__device__ __forceinline__ void fwd_sched_resolve(FwdSched& sc, const Table& tab, int H)
{
    if (!sc.order) return;
    sc.ntickets = tab.seq_chunk0(sc.nseq) * H;
    const float fed = (float)sc.feeders * (float)(*sc.longest) * FWD_STEP_OVER_TILE_F;
    sc.switch_at = max(0, sc.ntickets - (int)fed);
}
// Worker groups per CTA: four (1024 threads, 64 registers: the chain role loses about a tenth of its speed)
// when the chunk-local tiles are the larger part of the work, three (768 threads, 80 registers) when the
// longest chain is.  Forward, us, with three / four: 2048 tokens, 8 heads, 1 sequence 93.6 / 102, 4 sequences 107 / 116,
// 8 sequences 130 / 126; 4 x 4096, 16 heads 231 / 214; 131072 tokens in 8 packed sequences 1107 / 1235.
constexpr uint32_t FWD_GROUP_SMEM = (uint32_t)CL_SMEM - 1024;
static_assert(4 * FWD_GROUP_SMEM + 4 * sizeof(ClGroupShared) <= CF_SMEM - 1024, "worker groups fit");
static_assert(3 * CL_THREADS >= CFW_THREADS, "the chain fits into the CTA");

template <int FWD_GROUPS>
__device__ __forceinline__ void chunk_fwd_workers(const CUtensorMap& tmK, const CUtensorMap& tmQ,
                                                  const CUtensorMap& tmKt, const TcChunkArgs& cl, const FwdSched& sc,
                                                  int limit, uint8_t* sm, uint32_t tb)
{
    const int tid = threadIdx.x, g = tid / CL_THREADS, ltid = tid % CL_THREADS;
    ClGroupShared& gs = reinterpret_cast<ClGroupShared*>(sm + FWD_GROUPS * FWD_GROUP_SMEM)[g];
    auto gsync = [&]() { named_sync(1 + g, CL_THREADS); };
    if (ltid == 0) {
        mbar_init(&gs.bar_tma, 1);
        mbar_init(&gs.bar_mma1, 1);
        mbar_init(&gs.bar_mma2, 1);
        mbar_init(&gs.bar_drain, 1);
        fence_mbar_init();
    }
    gsync();
    // Tickets are drawn one tile ahead by a thread that leads nothing else, and looked at only when the tile in
    // progress is done: nobody waits for the atomic.  A ticket that has been drawn is always worked off before the group
    // stops; it stops drawing when the tickets out, by its own last one and the groups at work, reach the limit.
    constexpr int DRAWER = CL_THREADS - 32;
    const int ahead = (int)gridDim.x * FWD_GROUPS;
    uint32_t ph = 0;
    int* publish = nullptr;   // flag of the tile the group finished last
    int next = -1;
    if (ltid == DRAWER && *reinterpret_cast<volatile int*>(sc.tickets) < limit) next = atomicAdd(sc.tickets, 1);
    while (true) {
        if (ltid == DRAWER) gs.ticket = next < sc.ntickets ? next : -1;
        gsync();
        const int t = gs.ticket;
        if (t < 0) break;
        if (ltid == DRAWER) {
            next = -1;
            if (t + ahead < limit || limit >= sc.ntickets) next = atomicAdd(sc.tickets, 1);
        }
        int c, h;
        if (sc.order) {   // packed batch: position-major order from the sorted list, heads innermost
            const int j = t / cl.H;
            h = t - j * cl.H;
            c = sc.order[j];
        } else {
            const int n = t / sc.nchains, chain = t - n * sc.nchains;
            const int s = chain / cl.H;
            h = chain - s * cl.H;
            c = s * sc.nchunks + n;
        }
        if (!chunk_fwd_tile(tmK, tmQ, tmKt, cl, c, h, sm + g * FWD_GROUP_SMEM, gs, tb + g * 128, ltid, 1 + g, ph, publish)) {
            publish = nullptr;   // the chains that need the tile, and tickets drawn and not worked off, give up in their turn
            break;
        }
        publish = cl.ready + (size_t)c * cl.H + h;
        ph ^= 1;
    }
    if (publish) {
        gsync();
        if (ltid == 0) {
            __threadfence();
            st_release_gpu(publish, 1);
        }
    }
    gsync();
    if (ltid == 0) {
        mbar_inval(&gs.bar_tma);
        mbar_inval(&gs.bar_mma1);
        mbar_inval(&gs.bar_mma2);
        mbar_inval(&gs.bar_drain);
    }
    __syncthreads();
}

template <int FWD_GROUPS>
__global__ void __launch_bounds__(FWD_GROUPS * CL_THREADS, 1)
tc_fwd_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ,
              const __grid_constant__ CUtensorMap tmKt, const __grid_constant__ CUtensorMap tmV, TcChunkArgs cl,
              TcChainArgs ch, FwdSched sched)
{
    FwdSched sc = sched;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = align1024(smem_raw);
    __shared__ uint32_t tmem_base;
    if (threadIdx.x < 32) tmem_alloc(&tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = tmem_base;
    pdl_wait();
    fwd_sched_resolve(sc, cl.tab, cl.H);
    const bool chain_cta = (int)blockIdx.x < sc.nchains;
    // packed batch: a chain starts when the tickets reach its own first tile (short sequences start late)
    if (chain_cta && sc.order) sc.switch_at = max(sc.switch_at, cl.tab.seq_first_[blockIdx.x / cl.H] * cl.H);
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {   // one copy of the worker code: it has to stay in the instruction cache
        chunk_fwd_workers<FWD_GROUPS>(tmK, tmQ, tmKt, cl, sc, chain_cta && pass == 0 ? sc.switch_at : sc.ntickets, sm, tb);
        if (!chain_cta || pass == 1) break;
        chain_fwd_role(tmV, tmKt, ch, blockIdx.x, sm, tb);
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(tb, 512);
}

// ---------------------------------------------------------------------------------------------
// state chain, backward (reverse over chunks); dS (V x K, fp32) resident in tensor memory
//   ddU^T = dO^T P' + rho_i (dS Ktil^T) ;   dS <- gamma_C dS + dO^T Qg - ddU^T W
// ---------------------------------------------------------------------------------------------
struct TcChainBwdArgs {
    int H;
    Table tab;
    const float *gate, *dfinal_state;
    float* dinit_state;
    const uint8_t *WT, *P, *Qg;
    uint8_t *dSn, *ddUT;
    int* status;
};

constexpr uint32_t BS_DO = 0, BS_KT = 16384, BS_WT = 32768, BS_P = 49152, BS_QG = 57344;
constexpr uint32_t BSTAGE_BYTES = 73728;
constexpr size_t CB_SMEM = 2 * BSTAGE_BYTES + 32768 + 16384 + 1024;

// Warp roles as in the forward chain: 16 state warps (4 lane quadrants x 4 column groups), one warp
// issuing the tensor-core work, one producer warp.  Barriers:
//   full[st]   copies of a chunk have landed and its gate vectors are written          producer -> all
//   empty[st]  every product reading the stage has finished                           tensor core -> producer
//   s_ready    dS is in shared memory as a bf16 operand, the accumulator is decayed    state warps -> issuer
//   a_done     both parts of ddU^T are complete                                        tensor core -> state warps
//   a_ready    ddU^T is in shared memory as a bf16 operand                             state warps -> issuer
//   s_done     the cotangent update of the chunk is complete                           tensor core -> state warps
constexpr int CBK_EPI_WARPS = 16, CBK_MMA_WARP = 16, CBK_TMA_WARP = 17;
constexpr int CBK_THREADS = 18 * 32;

// Queue of (chunk, head) tiles between the backward chains (producers) and the chunk-local backward
// (consumers) inside one kernel: slot i holds tile + 1 once the i-th finished tile has been published
// (0 = not yet); consumers draw tickets from `head`.  The whole array is cleared before the launch.
struct TileQueue {
    int* slots;
    unsigned *head, *tail;
    // Publishes `count` tiles first, first + stride, ... (one fence and one counter update for all).
    __device__ __forceinline__ void push(int first, int stride, int count) const
    {
        if (count <= 0) return;
        fence_proxy_async_all();   // the tiles' images were written through the async proxy
        __threadfence();
        const unsigned slot = atomicAdd(tail, (unsigned)count);
        for (int i = 0; i < count; ++i) *reinterpret_cast<volatile int*>(slots + slot + i) = first + i * stride + 1;
    }
};

// One chain (sequence, head) of the backward state recurrence, by all CBK_THREADS threads of the CTA.
// `tb`: 256 free tensor-memory columns.  Every (chunk, head) tile whose cotangent images have reached
// global memory is appended to the tile queue `tq`, in the order the chains produce them.
__device__ __forceinline__ void chain_bwd_role(const CUtensorMap& tmDO, const CUtensorMap& tmKt, const TcChainBwdArgs& a,
                                               int chain, uint8_t* sm, uint32_t tb, const TileQueue& tq)
{
    uint8_t* sStage = sm;
    uint8_t* sdS = sm + 2 * BSTAGE_BYTES;       // dS as bf16, K-major, 2 k-halves x [128 x 128 B]
    uint8_t* sddU = sdS + 32768;                // ddU^T, K-major [v][i]
    __shared__ uint64_t bar_full[2], bar_empty[2], bar_s_ready, bar_a_done, bar_a_ready, bar_s_done, bar_drain;
    __shared__ float sRho[2][CH], sGC[2];

    const int H = a.H;
    const int s = chain / H, h = chain % H;
    const int c0 = a.tab.seq_chunk0(s), c1 = a.tab.seq_chunk0(s + 1);
    const int seq_t0 = a.tab.seq_tok0(s), seq_len = a.tab.seq_len(s);
    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const bool lead = lane == 0;
    const int quad = warp & 3, colq = (warp >> 2) & 3;
    const int v = quad * 32 + lane;
    float* dini = a.dinit_state ? a.dinit_state + (((size_t)s * H + h) * KD + v) * KD + colq * 32 : nullptr;
    const float* dfin = a.dfinal_state ? a.dfinal_state + (((size_t)s * H + h) * KD + v) * KD + colq * 32 : nullptr;
    if (c1 <= c0) {
        if (dini && warp < CBK_EPI_WARPS)
            for (int x = 0; x < 32; ++x) dini[x] = dfin ? dfin[x] : 0.f;
        return;
    }
    const int nchunks = c1 - c0;
    // step n of the reverse walk handles chunk c1 - 1 - n of the sequence
    auto chunk_rel = [&](int n) { return nchunks - 1 - n; };
    auto chunk_tok0 = [&](int n) { return seq_t0 + chunk_rel(n) * CH; };
    auto chunk_len = [&](int n) { return min(CH, seq_len - chunk_rel(n) * CH); };
    auto chunk_tile = [&](int n) { return (size_t)(c0 + chunk_rel(n)) * H + h; };

    if (tid == 0) {
        mbar_init(&bar_full[0], 2);
        mbar_init(&bar_full[1], 2);
        mbar_init(&bar_empty[0], 1);
        mbar_init(&bar_empty[1], 1);
        mbar_init(&bar_s_ready, CBK_EPI_WARPS);
        mbar_init(&bar_a_done, 1);
        mbar_init(&bar_a_ready, CBK_EPI_WARPS);
        mbar_init(&bar_s_done, 1);
        mbar_init(&bar_drain, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tS = tb, tA1 = tb + 128, tA2 = tb + 192;

    if (warp == CBK_TMA_WARP) {
        // ------------------------------------------------------------------ producer
        bool ok = true;
        auto load_gates = [&](int n, float& ga, float& gb) {
            const int tok0 = chunk_tok0(n), len = chunk_len(n);
            ga = lane < len ? a.gate[(size_t)(tok0 + lane) * H + h] : 0.f;
            gb = lane + 32 < len ? a.gate[(size_t)(tok0 + lane + 32) * H + h] : 0.f;
        };
        float ga, gb;
        load_gates(0, ga, gb);
        int asked = 0;   // chunks whose copies have been asked for
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1;
            float ga_next = 0.f, gb_next = 0.f;
            if (n + 1 < nchunks) load_gates(n + 1, ga_next, gb_next);
            if (n >= 2) ok = mbar_wait(&bar_empty[st], ((n >> 1) - 1) & 1, a.status, ERR_CHAIN_TMA);
            if (!ok) break;
            if (lane == 0) {
                const int tok0 = chunk_tok0(n);
                uint8_t* d = sStage + st * BSTAGE_BYTES;
                mbar_expect_tx(&bar_full[st], BSTAGE_BYTES);
                bulk_load(d + BS_WT, a.WT + chunk_tile(n) * REC_BYTES, 40960, &bar_full[st]);   // W^T, P', Qg
                for (int hf = 0; hf < 2; ++hf) tma_load_2d(d + BS_DO + hf * BOX, &tmDO, h * KD + hf * 64, tok0, &bar_full[st]);
                for (int hf = 0; hf < 2; ++hf) tma_load_2d(d + BS_KT + hf * BOX, &tmKt, h * KD + hf * 64, tok0, &bar_full[st]);
            }
            __syncwarp();
            warp_gate_vectors(ga, gb, lane, nullptr, sRho[st], &sGC[st]);
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bar_full[st]);
                // warm L2 two chunks ahead: the stage copies can only run one chunk ahead
                if (n + 2 < nchunks) {
                    const int t2 = chunk_tok0(n + 2);
                    bulk_prefetch(a.WT + chunk_tile(n + 2) * REC_BYTES, 40960);
                    for (int hf = 0; hf < 2; ++hf) {
                        tma_prefetch_2d(&tmDO, h * KD + hf * 64, t2);
                        tma_prefetch_2d(&tmKt, h * KD + hf * 64, t2);
                    }
                }
            }
            ga = ga_next;
            gb = gb_next;
            asked = n + 1;
        }
        for (int n = max(0, asked - 2); n < asked; ++n) mbar_drain(&bar_full[n & 1], (n >> 1) & 1);
    } else if (warp == CBK_MMA_WARP) {
        // ------------------------------------------------------------------ tensor-core issuer
        bool ok = true;
        bool a1_issued = false;   // dO^T P' of the coming chunk is already in its accumulator
        int next_pub = 1, interval = 1, published = 0;   // publication of finished tiles (lane 0)
        auto issue_a1 = [&](uint8_t* d) {   // acc1 = dO^T P'
            const uint32_t idesc = make_idesc(128, 64, IDESC_A_MN | IDESC_B_MN);
            const uint64_t da0 = desc_mnmajor(d + BS_DO, BOX), db0 = desc_mnmajor(d + BS_P, 0);
            for (int k = 0; k < 4; ++k)
                mma_ss(tA1, desc_advance(da0, 2048 * k), desc_advance(db0, 2048 * k), idesc, k > 0, lead);
        };
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1;
            const size_t tile = chunk_tile(n);
            uint8_t* d = sStage + st * BSTAGE_BYTES;
            if (!a1_issued) ok = mbar_wait(&bar_full[st], (n >> 1) & 1, a.status, ERR_CHAIN_TMA);
            ok = ok && mbar_wait(&bar_s_ready, n & 1, a.status, ERR_CHAIN_MMA1);
            if (!ok) break;
            tc_fence_after();
            if (lead) {
                bulk_wait_read();   // the ddU^T image of the previous chunk has left shared memory
                bulk_store(a.dSn + tile * 32768, sdS, 32768);   // cotangent at the end of this chunk
                bulk_commit();
            }
            __syncwarp();
            {
                if (!a1_issued) issue_a1(d);
                {   // acc2 = dS Ktil^T
                    const uint32_t idesc = make_idesc(128, 64);
                    for (int k = 0; k < 8; ++k)
                        mma_ss(tA2, desc_advance(desc_kmajor(sdS + (k >> 2) * 16384), 32 * (k & 3)),
                               desc_advance(desc_kmajor(d + BS_KT + (k >> 2) * BOX), 32 * (k & 3)), idesc, k > 0, lead);
                }
                mma_commit(&bar_a_done, lead);
                {   // dS += dO^T Qg (the accumulator has been decayed before s_ready)
                    const uint32_t idesc = make_idesc(128, 128, IDESC_A_MN | IDESC_B_MN);
                    const uint64_t da0 = desc_mnmajor(d + BS_DO, BOX), db0 = desc_mnmajor(d + BS_QG, BOX);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(tS, desc_advance(da0, 2048 * k), desc_advance(db0, 2048 * k), idesc, 1, lead);
                }
            }
            __syncwarp();
            ok = mbar_wait(&bar_a_ready, n & 1, a.status, ERR_CHAIN_MMA2);
            if (!ok) break;
            tc_fence_after();
            if (lead) {
                // The dS image sent off above must have left shared memory before the update is
                // released: its completion lets the state warps overwrite that image.
                bulk_wait_read();
                bulk_store(a.ddUT + tile * 16384, sddU, 16384);
                bulk_commit();
            }
            __syncwarp();
            {
                {   // dS -= ddU^T W
                    const uint32_t idesc = make_idesc(128, 128, IDESC_A_NEG);
                    const uint64_t da0 = desc_kmajor(sddU), db0 = desc_kmajor(d + BS_WT);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(tS, desc_advance(da0, 32 * k), desc_advance(db0, 32 * k), idesc, 1, lead);
                }
                mma_commit(&bar_s_done, lead);
                mma_commit(&bar_empty[st], lead);
            }
            __syncwarp();
            // the state-independent part of the next chunk's ddU^T, while the state warps convert dS
            a1_issued = false;
            if (n + 1 < nchunks && chunk_len(n + 1) == CH) {
                ok = mbar_wait(&bar_full[st ^ 1], ((n + 1) >> 1) & 1, a.status, ERR_CHAIN_TMA);
                if (!ok) break;
                issue_a1(sStage + (st ^ 1) * BSTAGE_BYTES);
                __syncwarp();
                a1_issued = true;
            }
            // Finished tiles go to the chunk-local workers in batches: a publication costs the issuing
            // thread a fence and a round trip to memory, and the workers consume far more slowly than the
            // chains produce, so the batches grow (1, 2, 4, ... up to 16 steps).  Only tiles whose two
            // bulk groups were committed at least a whole step ago are included: waiting for this
            // chunk's own stores would put their round trip on the chunk-to-chunk path.
            if (lane == 0 && n >= next_pub) {
                bulk_wait_all_but<2>();
                tq.push((int)chunk_tile(n - 1), H, n - published);   // steps published .. n - 1 (tile ids rise by H per step back)
                published = n;
                interval = min(2 * interval, 16);
                next_pub = n + interval;
            }
            __syncwarp();
        }
        if (lane == 0) {
            bulk_wait_all();
            if (ok) tq.push((int)chunk_tile(nchunks - 1), H, nchunks - published);
        }
        __syncwarp();
        mma_commit(&bar_drain, lead);   // (behind the push: the last tiles are waited for)
        mbar_drain(&bar_drain, 0);
    } else {
        // ------------------------------------------------------------------ state warps
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        for (int cb = 0; cb < 2; ++cb) {
            uint32_t r[16];
#pragma unroll
            for (int x4 = 0; x4 < 4; ++x4) {
                const float4 f4 = dfin ? *reinterpret_cast<const float4*>(dfin + cb * 16 + x4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                r[x4 * 4 + 0] = __float_as_uint(f4.x);
                r[x4 * 4 + 1] = __float_as_uint(f4.y);
                r[x4 * 4 + 2] = __float_as_uint(f4.z);
                r[x4 * 4 + 3] = __float_as_uint(f4.w);
            }
            tmem_st16(tS + lane_addr + colq * 32 + cb * 16, r);
        }
        tmem_st_wait();

        bool ok = true;
        for (int n = 0; n < nchunks && ok; ++n) {
            const int st = n & 1;
            const int len = chunk_len(n);
            uint8_t* d = sStage + st * BSTAGE_BYTES;
            ok = mbar_wait(&bar_full[st], (n >> 1) & 1, a.status, ERR_CHAIN_TMA);   // gate vectors, tail rows
            if (n > 0) ok = ok && mbar_wait(&bar_s_done, (n - 1) & 1, a.status, ERR_CHAIN_MMA2);
            if (!ok) break;
            tc_fence_after();
            // ---- E0: dS (cotangent at the chunk end) -> bf16 operand; decay the accumulator
            {
                const float gC = sGC[st];
                uint32_t rr[2][16];
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) tmem_ld16(tS + lane_addr + colq * 32 + cb * 16, rr[cb]);
                tmem_ld_wait();
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    uint32_t* r = rr[cb];
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {
                        uint4 w;
                        w.x = pack_bf16(__uint_as_float(r[c2 * 8 + 0]), __uint_as_float(r[c2 * 8 + 1]));
                        w.y = pack_bf16(__uint_as_float(r[c2 * 8 + 2]), __uint_as_float(r[c2 * 8 + 3]));
                        w.z = pack_bf16(__uint_as_float(r[c2 * 8 + 4]), __uint_as_float(r[c2 * 8 + 5]));
                        w.w = pack_bf16(__uint_as_float(r[c2 * 8 + 6]), __uint_as_float(r[c2 * 8 + 7]));
                        *reinterpret_cast<uint4*>(sdS + (colq >> 1) * 16384 + sw128_chunk(v, (colq & 1) * 4 + cb * 2 + c2)) = w;
                    }
#pragma unroll
                    for (int x = 0; x < 16; ++x) r[x] = __float_as_uint(__uint_as_float(r[x]) * gC);
                    tmem_st16(tS + lane_addr + colq * 32 + cb * 16, r);
                }
                tmem_st_wait();
            }
            if (len < CH) {
                for (int hf = 0; hf < 2; ++hf) {
                    zero_tail_rows(d + BS_DO + hf * BOX, len, tid, CBK_EPI_WARPS * 32);
                    zero_tail_rows(d + BS_KT + hf * BOX, len, tid, CBK_EPI_WARPS * 32);
                }
            }
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_s_ready);

            // ---- E1: ddU^T = acc1 + rho_i acc2 -> bf16 operand
            float rho[16];
#pragma unroll
            for (int x = 0; x < 16; ++x) rho[x] = sRho[st][colq * 16 + x];
            ok = mbar_wait(&bar_a_done, n & 1, a.status, ERR_CHAIN_MMA1);
            if (!ok) break;
            tc_fence_after();
            {
                uint32_t r1[16], r2[16];
                tmem_ld16(tA1 + lane_addr + colq * 16, r1);
                tmem_ld16(tA2 + lane_addr + colq * 16, r2);
                tmem_ld_wait();
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {
                    float f[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        f[x] = __uint_as_float(r1[c2 * 8 + x]) + rho[c2 * 8 + x] * __uint_as_float(r2[c2 * 8 + x]);
                    *reinterpret_cast<uint4*>(sddU + sw128_chunk(v, colq * 2 + c2)) =
                        make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
                }
            }
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_a_ready);
        }
        if (ok) ok = mbar_wait(&bar_s_done, (nchunks - 1) & 1, a.status, ERR_CHAIN_MMA2);
        tc_fence_after();
        if (ok && dini) {
            for (int cb = 0; cb < 2; ++cb) {
                uint32_t r[16];
                tmem_ld16(tS + lane_addr + colq * 32 + cb * 16, r);
                tmem_ld_wait();
#pragma unroll
                for (int x4 = 0; x4 < 4; ++x4)
                    *reinterpret_cast<float4*>(dini + cb * 16 + x4 * 4) =
                        make_float4(__uint_as_float(r[x4 * 4 + 0]), __uint_as_float(r[x4 * 4 + 1]),
                                    __uint_as_float(r[x4 * 4 + 2]), __uint_as_float(r[x4 * 4 + 3]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {   // the barrier words are initialised again for the CTA's next chain
        mbar_inval(&bar_full[0]); mbar_inval(&bar_full[1]); mbar_inval(&bar_empty[0]); mbar_inval(&bar_empty[1]);
        mbar_inval(&bar_s_ready); mbar_inval(&bar_a_done); mbar_inval(&bar_a_ready); mbar_inval(&bar_s_done);
        mbar_inval(&bar_drain);
    }
    __syncthreads();
    tc_fence_after();
}

// ---------------------------------------------------------------------------------------------
// chunk-local backward.  Feature-major ("transposed") accumulators: lane = feature, column = token.
// With dU = T R, R = diag(beta) (V - gamma K S^T):  dL/dR = T^T ddU =: dVb, dL/dA = -strictLower(dVb dU^T).
//   phase A : dVb^T = ddU^T T ; dP' = dO dU^T ; dQ1^T = S^T dO^T ; dKtr^T = dS^T dU
//             (reads only what the chain kernels and the caller wrote: issued ahead)
//   phase B : dA = -strictLower(dVb dU^T) ; dKb^T = -S^T dVb^T ; dq2^T = Ktil^T M1^T ; dktil^T = Q^T M1
//             (M1 = scale Gamma (.) lower(dP'))
//             R0 = K Ktil^T                                   (issued ahead)
//   phase C : dktil^T += K^T M2 ; dkr^T = Ktil^T M2^T       (M2 = diag(beta) (dA (.) Gamma))
//   final   : dq = scale gamma dQ1 + dq2 ; dv = beta dVb ; dktil += rho dKtr ; dk_read = beta gamma dKb + dkr ;
//             dbeta = <dVb, v> + <gamma dKb, k> + sum_j (dA Gamma R0)_ij ; dgate from the products of the gradients with their inputs
// ---------------------------------------------------------------------------------------------
struct TcChunkBwdArgs {
    int H, nseq;
    Table tab;
    const float *beta, *gate;
    float scale, d_min;
    const uint8_t *Tm, *Sn, *dSn, *dUT, *ddUT;
    const unsigned* skipw;
    __nv_bfloat16 *dq, *dk, *dv;
    float *dbeta, *dgate, *dktil, *dkread;
    int* status;
};

constexpr int CBW_WARPS = 16, CBW_THREADS = CBW_WARPS * 32, CBW_MMA_WARP = 16, CBW_PROD_WARP = 17;
static_assert((CBW_PROD_WARP + 1) * 32 == CBK_THREADS, "the chunk-local role takes every warp of the CTA");
constexpr uint32_t R_Q = 0, R_K = 16384, R_KT = 32768, R_V = 49152, R_DO = 65536, R_DU = 81920, R_DDU = 98304,
                   R_T = 114688, R_S = 122880, R_DS = 155648, R_M2 = 188416, R_M1 = 204800;
constexpr uint32_t R_DVB = R_DDU;   // the dVb^T image replaces ddU, which only the first product reads
// Output tiles over dead space: dq over v, dv over dO, dk over the images of phase C.
constexpr uint32_t ST_DQ = R_V, ST_DV = R_DO, ST_DK = R_M2;
constexpr size_t CBW_SMEM = R_M1 + 8192 + 1024;

// The chunk-local backward of the tiles drawn from the queue, by all CBK_THREADS threads of the CTA: sixteen epilogue warps
// (4 lane quadrants x 4 groups of 16 columns), one warp that issues the products, one that talks to the tile queue, copies
// tiles in and out and finishes the per-token sums.  `tb`: 512 tensor-memory columns.  The roles meet at mbarriers only, each
// completed once per tile (vec: one of the two):
//   vec[2] per-token scalars and the tile's coordinates are in shared memory               producer -> all
//   c, s, tok, v   copies: ddU T dO dU | S dS | q k ktil | v                               producer -> issuer, epilogue
//   mma[0..3]      dVb, dP' | dA (and dQ1, dKtr, R0) | dKb, dq2, first half of dktil | phase C  tensor core -> epilogue
//   e_a    images of M1 and dVb written                                                    epilogue -> issuer
//   e_d    images of M2 written, dv staged, <dS, S> formed                                 epilogue -> issuer, producer
//   e_f    everything of the tile is read; dq, dk staged, partial sums written             epilogue -> issuer, producer
// and in a tile of fewer than 64 tokens
//   zero   the rows beyond it are cleared                                                  epilogue -> issuer, epilogue
//   rows   dq, dk, dv are staged                                                           epilogue -> epilogue
// A wait that runs out ends its warp's loop and no other's: what a warp waits for between two tiles has to be an mbarrier,
// whose wait is bounded. (A hardware barrier would wait for the warps that have left.)
// A copy of the next tile is requested as soon as the space that it lands in is dead, the next tile's first products run
// under this tile's last epilogue.
// What bounds it: with three dependent phases (five when dL/dT was formed from dW K^T and ddU V^T and carried through
// T^T . T^T) the tile's copies, 184 KB in and 48 KB out.  Epilogues read the accumulators in the fragment layout of ldmatrix:
// two packed instructions move what sixteen 2-byte accesses of a lane-per-feature layout did, and eight sums of a token pair
// over the warp's features take seven shuffles.
__device__ __forceinline__ void chunk_bwd_role(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmKt,
                                               const CUtensorMap& tmV, const CUtensorMap& tmDO, const CUtensorMap& tmDQ,
                                               const CUtensorMap& tmDK, const CUtensorMap& tmDV, const TcChunkBwdArgs& a,
                                               uint8_t* sm, uint32_t tb, const TileQueue& tq)
{
    __shared__ uint64_t bar_vec[2], bar_c, bar_s, bar_tok, bar_v, bar_zero, bar_rows, bar_mma[4], bar_ea, bar_ed, bar_ef, bar_drain;
    __shared__ int sInfo[2][4];                            // tile (-1: no more), first token, length, head
    __shared__ unsigned sSkipW[2][2];
    __shared__ __align__(16) float sVec[2][4][CH];         // G_i, gamma_i = exp(G_i), rho_i = exp(G_C - G_i), beta_i
    __shared__ float sSum[2][4][2][CH];                    // per quadrant of features: gate and beta terms of every token
    __shared__ float sRow[2][4][CH];                       // per group of columns: the scores' share of a row's beta gradient
    __shared__ float sRed[2][CBW_WARPS];

    const int H = a.H;
    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const bool lead = lane == 0;
    if (tid == 0) {
        for (uint64_t* b : {&bar_vec[0], &bar_vec[1], &bar_c, &bar_s, &bar_tok, &bar_v, &bar_mma[0], &bar_mma[1], &bar_mma[2], &bar_mma[3], &bar_drain}) mbar_init(b, 1);
        for (uint64_t* b : {&bar_zero, &bar_rows, &bar_ea, &bar_ed, &bar_ef}) mbar_init(b, CBW_WARPS);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // tensor memory columns (64 each); dA takes the place of dP', dkr that of R0
    const uint32_t cDP = tb, cDQ1 = tb + 64, cDKTR = tb + 128, cDVB = tb + 192;
    const uint32_t cR0 = tb + 256, cDKB = tb + 320, cDQ2 = tb + 384, cDKT = tb + 448, cDA = cDP, cDKR = cR0;

    if (warp == CBW_PROD_WARP) {
        // ------------------------------------------------------------------ producer
        const int total = a.tab.seq_chunk0(a.nseq) * H;   // realised (chunk, head) tiles
        struct Tile { int t, h, tok0, len; };
        auto resolve = [&](int v) {   // v = slot value (tile + 1)
            Tile x{v - 1, 0, 0, 0};
            const int c = x.t / H;
            x.h = x.t - c * H;
            x.tok0 = a.tab.chunk_tok0(c);
            x.len = a.tab.chunk_len(c);
            fence_proxy_async_all();   // the tile's images are read through the async proxy
            return x;
        };
        auto draw = [&]() {
            unsigned t = 0;
            if (lane == 0) t = atomicAdd(tq.head, 1u);
            return t;   // lane 0 only: broadcast where it is used, long after the atomic
        };
        // slot of a ticket: 0 where the chains have not published it yet
        auto look = [&](unsigned ticket) { return ld_acquire_gpu(tq.slots + ticket); };
        auto look_blocking = [&](unsigned ticket) {
            int v = look(ticket);
            const long long t0 = clock64();
            while (!v) {
                if (clock64() - t0 > WAIT_LIMIT_CYCLES || *reinterpret_cast<volatile int*>(a.status) != 0) {
                    if (lane == 0) atomicCAS(a.status, 0, ERR_QUEUE);
                    break;
                }
                __nanosleep(64);
                v = look(ticket);
            }
            return __shfl_sync(0xffffffffu, v, 0);
        };
        auto load_tok = [&](const CUtensorMap& m, uint32_t region, const Tile& x, uint64_t* bar) {
            for (int hf = 0; hf < 2; ++hf) tma_load_2d(sm + region + hf * BOX, &m, x.h * KD + hf * 64, x.tok0, bar);
        };
        auto store_tok = [&](const CUtensorMap& m, uint32_t region, const Tile& x) {
            for (int hf = 0; hf < 2; ++hf) tma_store_2d(&m, x.h * KD + hf * 64, x.tok0, sm + region + hf * BOX);
        };
        auto load_t_ds = [&](const Tile& x) {
            mbar_announce_tx(&bar_c, 8192);
            bulk_load(sm + R_T, a.Tm + (size_t)x.t * 8192, 8192, &bar_c);
            mbar_announce_tx(&bar_s, 32768);
            bulk_load(sm + R_DS, a.dSn + (size_t)x.t * 32768, 32768, &bar_s);
        };
        auto load_u_s = [&](const Tile& x) {
            mbar_announce_tx(&bar_c, 32768);
            mbar_expect_tx(&bar_s, 32768);
            bulk_load(sm + R_DDU, a.ddUT + (size_t)x.t * 16384, 16384, &bar_c);
            bulk_load(sm + R_DU, a.dUT + (size_t)x.t * 16384, 16384, &bar_c);
            bulk_load(sm + R_S, a.Sn + (size_t)x.t * 32768, 32768, &bar_s);
        };
        auto load_do = [&](const Tile& x) {
            mbar_expect_tx(&bar_c, 2 * BOX);
            load_tok(tmDO, R_DO, x, &bar_c);
        };
        auto load_kkq = [&](const Tile& x) {
            mbar_expect_tx(&bar_tok, 6 * BOX);
            load_tok(tmK, R_K, x, &bar_tok);
            load_tok(tmKt, R_KT, x, &bar_tok);
            load_tok(tmQ, R_Q, x, &bar_tok);
        };
        auto load_v = [&](const Tile& x) {
            mbar_expect_tx(&bar_v, 2 * BOX);
            load_tok(tmV, R_V, x, &bar_v);
        };
        // The next tile's operands on their way into L2 while this one is worked on: most of them were written by the
        // forward pass and come from HBM.
        auto warm = [&](const Tile& x) {
            bulk_prefetch(a.Tm + (size_t)x.t * 8192, 8192);
            bulk_prefetch(a.dSn + (size_t)x.t * 32768, 32768);
            bulk_prefetch(a.dUT + (size_t)x.t * 16384, 16384);
            bulk_prefetch(a.Sn + (size_t)x.t * 32768, 32768);
            bulk_prefetch(a.ddUT + (size_t)x.t * 16384, 16384);
            for (int hf = 0; hf < 2; ++hf) {
                const int c = x.h * KD + hf * 64;
                tma_prefetch_2d(&tmDO, c, x.tok0);
                tma_prefetch_2d(&tmK, c, x.tok0);
                tma_prefetch_2d(&tmKt, c, x.tok0);
                tma_prefetch_2d(&tmQ, c, x.tok0);
                tma_prefetch_2d(&tmV, c, x.tok0);
            }
        };
        struct Scal { float ga, gb, ba, bb; unsigned w; };
        auto fetch = [&](const Tile& x) {   // lane: tokens l and l + 32; tokens beyond the chunk read as zero
            Scal y;
            const bool in0 = lane < x.len, in1 = lane + 32 < x.len;
            const size_t th = (size_t)(x.tok0 + lane) * H + x.h, th1 = th + (size_t)32 * H;
            y.ga = in0 ? a.gate[th] : 0.f;
            y.gb = in1 ? a.gate[th1] : 0.f;
            y.ba = in0 ? a.beta[th] : 0.f;
            y.bb = in1 ? a.beta[th1] : 0.f;
            y.w = lane < 2 ? a.skipw[(size_t)x.t * 2 + lane] : 0u;
            return y;
        };
        auto publish = [&](const Tile& x, const Scal& y, int buf) {   // x.t < 0: no more tiles
            if (x.t >= 0) {
                float sa = y.ga, sb = y.gb;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float ua = __shfl_up_sync(0xffffffffu, sa, o), ub = __shfl_up_sync(0xffffffffu, sb, o);
                    if (lane >= o) { sa += ua; sb += ub; }
                }
                sb += __shfl_sync(0xffffffffu, sa, 31);
                const float tot = __shfl_sync(0xffffffffu, sb, 31);
                float(*v)[CH] = sVec[buf];
                v[0][lane] = sa;
                v[0][lane + 32] = sb;
                v[1][lane] = __expf(sa);
                v[1][lane + 32] = __expf(sb);
                v[2][lane] = __expf(tot - sa);
                v[2][lane + 32] = __expf(tot - sb);
                v[3][lane] = y.ba;
                v[3][lane + 32] = y.bb;
                if (lane < 2) sSkipW[buf][lane] = y.w;
            }
            if (lane == 0) {
                sInfo[buf][0] = x.t;
                sInfo[buf][1] = x.tok0;
                sInfo[buf][2] = x.len;
                sInfo[buf][3] = x.h;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_vec[buf]);
        };
        // dgate_j is the suffix sum of the per-token terms (the in-chunk prefix G_i collects every g_j with j <= i); the
        // chunk-level term goes to the last token
        auto finish_sums = [&](const Tile& x, int buf) {
            float s[2], b[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = lane + 32 * u;
                s[u] = (sSum[buf][0][0][j] + sSum[buf][1][0][j]) + (sSum[buf][2][0][j] + sSum[buf][3][0][j]);
                b[u] = (sSum[buf][0][1][j] + sSum[buf][1][1][j]) + (sSum[buf][2][1][j] + sSum[buf][3][1][j]) +
                       ((sRow[buf][0][j] + sRow[buf][1][j]) + (sRow[buf][2][j] + sRow[buf][3][j]));
            }
            float tot = lane < CBW_WARPS ? sRed[buf][lane] : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
            if (lane == 31) s[1] += tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float u0 = __shfl_down_sync(0xffffffffu, s[0], o), u1 = __shfl_down_sync(0xffffffffu, s[1], o);
                if (lane + o < 32) { s[0] += u0; s[1] += u1; }
            }
            s[0] += __shfl_sync(0xffffffffu, s[1], 0);
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (lane + 32 * u < x.len) {
                    const size_t th = (size_t)(x.tok0 + lane + 32 * u) * H + x.h;
                    a.dgate[th] = s[u];
                    a.dbeta[th] = b[u];
                }
        };

        // copies asked for: those of the tiles before `newest`, and of this one T and dS (1), ddU, dU and S (2), dO (3),
        // k, ktil and q (4), v (5)
        int newest = -1, asked = 0;
        Tile cur{-1, 0, 0, 0};
        unsigned ticket = __shfl_sync(0xffffffffu, draw(), 0), after = draw();
        if (ticket < (unsigned)total) {
            const int v = look_blocking(ticket);
            if (v) cur = resolve(v);
        }
        Scal sc{};
        if (cur.t >= 0) {
            if (lane == 0) {
                load_t_ds(cur);
                load_u_s(cur);
                load_do(cur);
                load_kkq(cur);
                load_v(cur);
            }
            __syncwarp();
            newest = 0;
            asked = 5;
            sc = fetch(cur);
        }
        publish(cur, sc, 0);
        for (uint32_t it = 0; cur.t >= 0; ++it) {
            const uint32_t ph = it & 1;
            const bool full = cur.len == CH;
            // the next tile, if the chains have published it already (asked again behind this tile if not)
            ticket = __shfl_sync(0xffffffffu, after, 0);
            const bool more = ticket < (unsigned)total;
            if (more) after = draw();
            Tile next{-1, 0, 0, 0};
            int v = more ? __shfl_sync(0xffffffffu, look(ticket), 0) : 0;
            const bool known = v != 0;
            if (known) {
                next = resolve(v);
                if (lane == 0) warm(next);
                __syncwarp();
                sc = fetch(next);
            }
            if (known || !more) publish(next, sc, (int)(ph ^ 1u));
            if (!mbar_wait(&bar_ed, ph, a.status, ERR_MMA2)) break;
            // dA is formed, hence dVb, dP', dQ1 and dKtr too: T and dS are dead
            if (lane == 0) {
                if (full) {
                    store_tok(tmDV, ST_DV, cur);
                    bulk_commit();
                }
                if (known) load_t_ds(next);
            }
            __syncwarp();
            if (known) {
                newest = (int)it + 1;
                asked = 1;
            }
            if (!mbar_wait(&bar_mma[2], ph, a.status, ERR_MMA2)) break;
            if (lane == 0) {
                if (known) load_u_s(next);   // S, dU and the dVb image (in the space of ddU) are dead
                if (full) {
                    bulk_wait_read();
                    if (known) load_do(next);
                }
            }
            __syncwarp();
            if (known) asked = full ? 3 : 2;
            if (!mbar_wait(&bar_ef, ph, a.status, ERR_MMA2)) break;
            if (lane == 0) {
                if (full) {
                    store_tok(tmDQ, ST_DQ, cur);
                    store_tok(tmDK, ST_DK, cur);
                    bulk_commit();
                }
                if (known) {
                    if (!full) load_do(next);
                    load_kkq(next);
                }
            }
            __syncwarp();
            if (known) asked = 4;
            finish_sums(cur, (int)ph);
            if (lane == 0 && full) bulk_wait_read();   // v lands where dq was staged, the next M2 images where dk was
            __syncwarp();
            if (known) {
                if (lane == 0) load_v(next);
            } else if (more) {
                v = look_blocking(ticket);
                if (!v) break;
                next = resolve(v);
                if (lane == 0) {
                    load_t_ds(next);
                    load_u_s(next);
                    load_do(next);
                    load_kkq(next);
                    load_v(next);
                }
                __syncwarp();
                newest = (int)it + 1;
                sc = fetch(next);
                publish(next, sc, (int)(ph ^ 1u));
            }
            __syncwarp();
            if (newest == (int)it + 1) asked = 5;
            cur = next;
        }
        // Whatever ended the loop, the copies asked for land before the memory is given up.  (A phase that was only announced
        // in part gets its arrival here.)
        if (newest >= 0) {
            if (lane == 0) {
                if (asked < 2) mbar_arrive(&bar_s);
                if (asked < 3) mbar_arrive(&bar_c);
            }
            mbar_drain(&bar_c, newest & 1);
            mbar_drain(&bar_s, newest & 1);
            const int tok = asked < 4 ? newest - 1 : newest, vv = asked < 5 ? newest - 1 : newest;
            if (tok >= 0) mbar_drain(&bar_tok, tok & 1);
            if (vv >= 0) mbar_drain(&bar_v, vv & 1);
        }
        if (lane == 0) bulk_wait_all();
        __syncwarp();
    } else if (warp == CBW_MMA_WARP) {
        // ------------------------------------------------------------------ tensor-core issuer
        uint32_t ragged = 0;
        for (uint32_t it = 0;; ++it) {
            const uint32_t ph = it & 1;
            if (!mbar_wait(&bar_vec[ph], (it >> 1) & 1, a.status, ERR_TMA) || sInfo[ph][0] < 0) break;
            if (!mbar_wait(&bar_c, ph, a.status, ERR_TMA)) break;
            if (sInfo[ph][2] < CH && !mbar_wait(&bar_zero, ragged++ & 1, a.status, ERR_TMA)) break;
            tc_fence_after();
            {   // phase A, first part
                {   // dVb^T[v][j] = sum_i ddU^T[v][i] T[i][j]
                    const uint64_t da0 = desc_kmajor(sm + R_DDU), db0 = desc_mnmajor(sm + R_T, 0);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(cDVB, desc_advance(da0, 32 * k), desc_advance(db0, 2048 * k), make_idesc(128, 64, IDESC_B_MN), k > 0, lead);
                }
                {   // dP'[i][j] = sum_v dO[i][v] dU[j][v]                                      (M = 64)
                    const uint64_t db0 = desc_mnmajor(sm + R_DU, 0);
                    for (int k = 0; k < 8; ++k)
                        mma_ss(cDP, desc_advance(desc_kmajor(sm + R_DO + (k >> 2) * BOX), 32 * (k & 3)),
                               desc_advance(db0, 2048 * k), make_idesc(64, 64, IDESC_B_MN), k > 0, lead);
                }
                mma_commit(&bar_mma[0], lead);
            }
            __syncwarp();
            if (!mbar_wait(&bar_s, ph, a.status, ERR_TMA)) break;
            if (it > 0 && !mbar_wait(&bar_ef, ph ^ 1u, a.status, ERR_MMA1)) break;   // the previous dQ1 and dKtr have been read
            tc_fence_after();
            {   // phase A, second part: only the later epilogues read it
                const uint64_t das = desc_mnmajor(sm + R_S, 16384), dads = desc_mnmajor(sm + R_DS, 16384), dbu = desc_mnmajor(sm + R_DU, 0);
                for (int k = 0; k < 8; ++k)   // dQ1^T[k][i] = sum_v S[v][k] dO[i][v]
                    mma_ss(cDQ1, desc_advance(das, 2048 * k), desc_advance(desc_kmajor(sm + R_DO + (k >> 2) * BOX), 32 * (k & 3)),
                           make_idesc(128, 64, IDESC_A_MN), k > 0, lead);
                for (int k = 0; k < 8; ++k)   // dKtr^T[k][j] = sum_v dS[v][k] dU[j][v]
                    mma_ss(cDKTR, desc_advance(dads, 2048 * k), desc_advance(dbu, 2048 * k),
                           make_idesc(128, 64, IDESC_A_MN | IDESC_B_MN), k > 0, lead);
            }
            __syncwarp();
            if (!mbar_wait(&bar_tok, ph, a.status, ERR_TMA)) break;
#pragma unroll 1   // (a tile's code is long: unrolled, the 340M step 299.2 instead of 298.0 us, ungated 894.3 instead of 893.6)
            for (int k = 0; k < 8; ++k)   // R0[i][j] = sum_c K[i][c] Ktil[j][c]                           (M = 64)
                mma_ss(cR0, desc_advance(desc_kmajor(sm + R_K + (k >> 2) * BOX), 32 * (k & 3)),
                       desc_advance(desc_kmajor(sm + R_KT + (k >> 2) * BOX), 32 * (k & 3)), make_idesc(64, 64), k > 0, lead);
            __syncwarp();
            if (!mbar_wait(&bar_ea, ph, a.status, ERR_MMA1)) break;
            tc_fence_after();
            {   // phase B
                const uint64_t dbv = desc_mnmajor(sm + R_DVB, 0);
                {   // dA[a][b] = sum_v dVb[a][v] dU[b][v] (its negative, its strictly lower part)     (M = 64)
                    const uint64_t dbu = desc_mnmajor(sm + R_DU, 0);
                    for (int k = 0; k < 8; ++k)
                        mma_ss(cDA, desc_advance(dbv, 2048 * k), desc_advance(dbu, 2048 * k),
                               make_idesc(64, 64, IDESC_A_MN | IDESC_B_MN), k > 0, lead);
                }
                mma_commit(&bar_mma[1], lead);
                {   // dKb^T[k][j] = -sum_v S[v][k] dVb[j][v]
                    const uint64_t das = desc_mnmajor(sm + R_S, 16384);
                    for (int k = 0; k < 8; ++k)
                        mma_ss(cDKB, desc_advance(das, 2048 * k), desc_advance(dbv, 2048 * k),
                               make_idesc(128, 64, IDESC_A_MN | IDESC_B_MN | IDESC_A_NEG), k > 0, lead);
                }
                {   // dq2^T[k][i] = sum_j Ktil[j][k] M1[i][j] ;  dktil^T[k][j] = sum_i Q[i][k] M1[i][j]
                    const uint64_t da0 = desc_mnmajor(sm + R_KT, BOX), da1 = desc_mnmajor(sm + R_Q, BOX);
                    const uint64_t dbk = desc_kmajor(sm + R_M1), dbm = desc_mnmajor(sm + R_M1, 0);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(cDQ2, desc_advance(da0, 2048 * k), desc_advance(dbk, 32 * k), make_idesc(128, 64, IDESC_A_MN), k > 0, lead);
                    for (int k = 0; k < 4; ++k)
                        mma_ss(cDKT, desc_advance(da1, 2048 * k), desc_advance(dbm, 2048 * k),
                               make_idesc(128, 64, IDESC_A_MN | IDESC_B_MN), k > 0, lead);
                }
                mma_commit(&bar_mma[2], lead);
            }
            __syncwarp();
            if (!mbar_wait(&bar_ed, ph, a.status, ERR_MMA2)) break;
            tc_fence_after();
            {   // phase C: dktil^T += K^T M2 ; dkr^T[k][i] = sum_j Ktil[j][k] M2[i][j]
                const uint64_t da0 = desc_mnmajor(sm + R_K, BOX), da1 = desc_mnmajor(sm + R_KT, BOX);
                const uint64_t dbm = desc_mnmajor(sm + R_M2, 0), dbk = desc_kmajor(sm + R_M2);
                for (int k = 0; k < 4; ++k)
                    mma_ss(cDKT, desc_advance(da0, 2048 * k), desc_advance(dbm, 2048 * k),
                           make_idesc(128, 64, IDESC_A_MN | IDESC_B_MN), 1, lead);
                for (int k = 0; k < 4; ++k)
                    mma_ss(cDKR, desc_advance(da1, 2048 * k), desc_advance(dbk, 32 * k), make_idesc(128, 64, IDESC_A_MN), k > 0, lead);
                mma_commit(&bar_mma[3], lead);
            }
            __syncwarp();
        }
        mma_commit(&bar_drain, lead);
        mbar_drain(&bar_drain, 0);
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const int quad = warp & 3, colq = warp >> 2;      // lane quadrant (32 features or 16 rows), group of 16 columns
        const int lr = lane >> 2, lc = 2 * (lane & 3);    // fragment row and first column
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        const uint32_t s0 = smem_u32(sm);
        // addresses of the 8 x 8 matrices (half = lane / 16, octet of columns = lane / 8 % 2) that this lane provides:
        const int half = lane >> 4, oct = (lane >> 3) & 1, mr = lane & 7;
        const uint32_t offI = sw128_chunk(quad * 16 + half * 8 + mr, colq * 2 + oct);          // 64 x 64 image
        const uint32_t offF = sw128_chunk(quad * 32 + half * 8 + mr, colq * 2 + oct);          // feature-major image
        const uint32_t offT = (uint32_t)(quad >> 1) * BOX + sw128_chunk(colq * 16 + oct * 8 + mr, (quad & 1) * 4 + half);   // token tile; second sixteen features: ^ 32
        const int i0 = quad * 16 + lr, j0 = colq * 16 + lc;   // row (and i0 + 8) of 64-row accumulators; columns j0, j0 + 1, j0 + 8, j0 + 9
        uint32_t ragged = 0;
        for (uint32_t it = 0;; ++it) {
            const uint32_t ph = it & 1;
            if (!mbar_wait(&bar_vec[ph], (it >> 1) & 1, a.status, ERR_TMA)) break;
            const int tile = sInfo[ph][0], tok0 = sInfo[ph][1], len = sInfo[ph][2], h = sInfo[ph][3];
            if (tile < 0) break;
            const unsigned long long sk = (unsigned long long)sSkipW[ph][0] | ((unsigned long long)sSkipW[ph][1] << 32);
            const float *sG = sVec[ph][0], *sGam = sVec[ph][1], *sRho = sVec[ph][2], *sBeta = sVec[ph][3];
            if (len < CH) {   // rows beyond the sequence belong to another one
                if (!mbar_wait(&bar_c, ph, a.status, ERR_TMA) || !mbar_wait(&bar_tok, ph, a.status, ERR_TMA) ||
                    !mbar_wait(&bar_v, ph, a.status, ERR_TMA))
                    break;
                for (const uint32_t reg : {R_DO, R_Q, R_K, R_KT, R_V})
                    for (int hf = 0; hf < 2; ++hf) zero_tail_rows(sm + reg + hf * BOX, len, tid, CBW_THREADS);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar_zero);
                if (!mbar_wait(&bar_zero, ragged & 1, a.status, ERR_TMA)) break;
            }
            // ---- M1 = scale Gamma (.) lower(dP') and dVb^T as operands
            float gam[8], dvb[2][8];   // Gamma_ij = exp(G_i - G_j), j <= i (else 0); index 4 octet + 2 (row half) + column parity
            {
                const float Gi[2] = {sG[i0], sG[i0 + 8]};
                float Gj[2][2];
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const float2 g2 = *reinterpret_cast<const float2*>(sG + j0 + 8 * o);
                    Gj[o][0] = g2.x;
                    Gj[o][1] = g2.y;
                }
#pragma unroll
                for (int o = 0; o < 2; ++o)
#pragma unroll
                    for (int rh = 0; rh < 2; ++rh)
#pragma unroll
                        for (int e = 0; e < 2; ++e)
                            gam[4 * o + 2 * rh + e] = j0 + 8 * o + e <= i0 + 8 * rh ? __expf(Gi[rh] - Gj[o][e]) : 0.f;
            }
            if (!mbar_wait(&bar_mma[0], ph, a.status, ERR_MMA1)) break;
            tc_fence_after();
            {
                uint32_t r[8];
                tmem_ld_frag16(cDP + lane_addr + colq * 16, r);
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
                    tmem_ld_frag16(cDVB + lane_addr + ((uint32_t)(16 * hf) << 16) + colq * 16, reinterpret_cast<uint32_t*>(dvb[hf]));
                tmem_ld_wait();
                uint32_t m[4];
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    m[x] = pack_bf16(a.scale * gam[2 * x] * __uint_as_float(r[2 * x]), a.scale * gam[2 * x + 1] * __uint_as_float(r[2 * x + 1]));
                stmatrix_x4(s0 + R_M1 + offI, m[0], m[2], m[1], m[3]);
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    uint32_t p[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) p[x] = pack_bf16(dvb[hf][2 * x], dvb[hf][2 * x + 1]);
                    stmatrix_x4(s0 + R_DVB + offF + hf * 2048, p[0], p[2], p[1], p[3]);
                }
            }
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ea);

            // ---- while dA is formed: dv = beta dVb (stored once dQ1 has read dO) and dVb's share of the beta gradient, <dS, S>
            uint32_t wv[2][4];
            float gv[4] = {}, bv[4];   // per-token terms of this thread's features: tokens j0, j0 + 1, j0 + 8, j0 + 9
            float bj[4];
            {
                const float2 b0 = *reinterpret_cast<const float2*>(sBeta + j0), b1 = *reinterpret_cast<const float2*>(sBeta + j0 + 8);
                bj[0] = b0.x; bj[1] = b0.y; bj[2] = b1.x; bj[3] = b1.y;
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) bv[x] = 0.f;
            if (!mbar_wait(&bar_v, ph, a.status, ERR_TMA)) break;
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                uint32_t vr[4];   // matrices (half, octet): fragment index 2 octet + half <-> register 2 half + octet
                ldmatrix_x4_trans(s0 + R_V + (offT ^ (32u * hf)), vr);
#pragma unroll
                for (int o = 0; o < 2; ++o)
#pragma unroll
                    for (int rh = 0; rh < 2; ++rh) {
                        const float x0 = dvb[hf][4 * o + 2 * rh], x1 = dvb[hf][4 * o + 2 * rh + 1];
                        const uint32_t vw = vr[2 * rh + o];
                        bv[2 * o] = fmaf(x0, bf16_lo(vw), bv[2 * o]);
                        bv[2 * o + 1] = fmaf(x1, bf16_hi(vw), bv[2 * o + 1]);
                        wv[hf][2 * rh + o] = pack_bf16(bj[2 * o] * x0, bj[2 * o + 1] * x1);
                    }
            }
            float part;
            if (!mbar_wait(&bar_s, ph, a.status, ERR_TMA)) break;
            {   // rows 8 warp .. of both images: the diagonals of 8 x 8 products are the rows' inner products
                float c[4] = {};
                const uint32_t row = (uint32_t)(warp * 8 + mr);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t off = (uint32_t)(q >> 1) * 16384 + sw128_chunk(row, (uint32_t)((q & 1) * 4) + (uint32_t)(lane >> 3));
                    uint32_t x[4], y[4];
                    ldmatrix_x4(s0 + R_DS + off, x);
                    ldmatrix_x4(s0 + R_S + off, y);
                    mma_bf16(c, x[0], 0u, x[1], 0u, y[0], y[1]);
                    mma_bf16(c, x[2], 0u, x[3], 0u, y[2], y[3]);
                }
                part = (lr >> 1) == (lane & 3) ? ((lr & 1) ? c[1] : c[0]) : 0.f;
            }

            // ---- dA = -strictLower -> M2 = beta_i dA Gamma
            float rw[2] = {};   // rows' sums of dA Gamma R0, from the accumulators (as <dkr, k>, through dkr's operand, they would be rounded to bf16)
            if (!mbar_wait(&bar_mma[1], ph, a.status, ERR_MMA2)) break;
            tc_fence_after();
            {
                uint32_t r[8], r0[8];
                tmem_ld_frag16(cDA + lane_addr + colq * 16, r);
                tmem_ld_frag16(cR0 + lane_addr + colq * 16, r0);
                const float bi[2] = {sBeta[i0], sBeta[i0 + 8]};
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
                    stmatrix_x4_trans(s0 + ST_DV + (offT ^ (32u * hf)), wv[hf][0], wv[hf][1], wv[hf][2], wv[hf][3]);
                tmem_ld_wait();
                uint32_t m[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {   // x = 2 octet + row half
                    const int o = x >> 1, rh = x & 1;
                    float u[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        u[e] = j0 + 8 * o + e < i0 + 8 * rh ? -__uint_as_float(r[2 * x + e]) * gam[2 * x + e] : 0.f;
                        rw[rh] = fmaf(u[e], __uint_as_float(r0[2 * x + e]), rw[rh]);
                    }
                    m[x] = pack_bf16(bi[rh] * u[0], bi[rh] * u[1]);
                }
                stmatrix_x4(s0 + R_M2 + offI, m[0], m[2], m[1], m[3]);
            }
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ed);

            // ---- while phase C runs: the row sums' four lanes together; dq = scale gamma dQ1 + dq2, staged over v
            {
                const bool up = lane & 1;
                float y = (up ? rw[1] : rw[0]) + __shfl_xor_sync(0xffffffffu, up ? rw[0] : rw[1], 1);
                y += __shfl_xor_sync(0xffffffffu, y, 2);
                if (!(lane & 2)) sRow[ph][colq][i0 + (up ? 8 : 0)] = y;
            }
            float gj[4];
            {
                const float2 g0 = *reinterpret_cast<const float2*>(sGam + j0), g1 = *reinterpret_cast<const float2*>(sGam + j0 + 8);
                gj[0] = g0.x; gj[1] = g0.y; gj[2] = g1.x; gj[3] = g1.y;
            }
            // (the products have waited for q, k and ktil, but only a wait of its own makes a copy visible to a thread)
            if (!mbar_wait(&bar_tok, ph, a.status, ERR_TMA) || !mbar_wait(&bar_mma[2], ph, a.status, ERR_MMA2)) break;
            tc_fence_after();
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const uint32_t ad = lane_addr + ((uint32_t)(16 * hf) << 16) + colq * 16;
                uint32_t r1[8], r2[8], qr[4], w[4];
                tmem_ld_frag16(cDQ1 + ad, r1);
                tmem_ld_frag16(cDQ2 + ad, r2);
                ldmatrix_x4_trans(s0 + R_Q + (offT ^ (32u * hf)), qr);
                tmem_ld_wait();
#pragma unroll
                for (int o = 0; o < 2; ++o)
#pragma unroll
                    for (int rh = 0; rh < 2; ++rh) {
                        const int x = 4 * o + 2 * rh;
                        const float d0 = a.scale * gj[2 * o] * __uint_as_float(r1[x]) + __uint_as_float(r2[x]);
                        const float d1 = a.scale * gj[2 * o + 1] * __uint_as_float(r1[x + 1]) + __uint_as_float(r2[x + 1]);
                        gv[2 * o] = fmaf(d0, bf16_lo(qr[2 * rh + o]), gv[2 * o]);
                        gv[2 * o + 1] = fmaf(d1, bf16_hi(qr[2 * rh + o]), gv[2 * o + 1]);
                        w[2 * rh + o] = pack_bf16(d0, d1);
                    }
                stmatrix_x4_trans(s0 + ST_DQ + (offT ^ (32u * hf)), w[0], w[1], w[2], w[3]);
            }

            // ---- dk = dk_read + d_min dL/dktil; the fp32 parts only where the preconditioner's reverse pass reads them
            float rj[4];
            {
                const float2 r0 = *reinterpret_cast<const float2*>(sRho + j0), r1 = *reinterpret_cast<const float2*>(sRho + j0 + 8);
                rj[0] = r0.x; rj[1] = r0.y; rj[2] = r1.x; rj[3] = r1.y;
            }
            const unsigned long long in = len == CH ? ~0ull : (1ull << len) - 1;
            const uint32_t want_kr = (uint32_t)((~sk & in) >> (colq * 16)) & 0xffffu;                       // step really taken
            const uint32_t want_kt = (uint32_t)(((~sk | (~sk << 1) | 1ull) & in) >> (colq * 16)) & 0xffffu;   // ... or a restart behind it
            float rsum = 0.f;
            if (!mbar_wait(&bar_mma[3], ph, a.status, ERR_MMA2)) break;
            tc_fence_after();
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const uint32_t ad = lane_addr + ((uint32_t)(16 * hf) << 16) + colq * 16;
                uint32_t rt[8], rd[8], rb[8], rk[8], kr[4], ktr[4], w[4];
                tmem_ld_frag16(cDKTR + ad, rt);
                tmem_ld_frag16(cDKT + ad, rd);
                tmem_ld_frag16(cDKB + ad, rb);
                tmem_ld_frag16(cDKR + ad, rk);
                ldmatrix_x4_trans(s0 + R_K + (offT ^ (32u * hf)), kr);
                ldmatrix_x4_trans(s0 + R_KT + (offT ^ (32u * hf)), ktr);
                tmem_ld_wait();
                float dkr[8], dkt[8];
#pragma unroll
                for (int o = 0; o < 2; ++o)
#pragma unroll
                    for (int rh = 0; rh < 2; ++rh) {
                        const uint32_t kw = kr[2 * rh + o], tw = ktr[2 * rh + o];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int x = 4 * o + 2 * rh + e, j = 2 * o + e;
                            const float kv = e ? bf16_hi(kw) : bf16_lo(kw), ktv = e ? bf16_hi(tw) : bf16_lo(tw);
                            const float dktr = rj[j] * __uint_as_float(rt[x]);
                            dkt[x] = dktr + __uint_as_float(rd[x]);
                            const float u = gj[j] * __uint_as_float(rb[x]);
                            dkr[x] = fmaf(bj[j], u, __uint_as_float(rk[x]));
                            gv[j] += dkr[x] * kv - dkt[x] * ktv;
                            bv[j] = fmaf(u, kv, bv[j]);
                            rsum = fmaf(dktr, ktv, rsum);
                        }
                        const int x = 4 * o + 2 * rh;
                        w[2 * rh + o] = pack_bf16(fmaf(a.d_min, dkt[x], dkr[x]), fmaf(a.d_min, dkt[x + 1], dkr[x + 1]));
                    }
                stmatrix_x4_trans(s0 + ST_DK + (offT ^ (32u * hf)), w[0], w[1], w[2], w[3]);
                if (want_kt) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int bit = lc + 8 * (j >> 1) + (j & 1);
                        const size_t g = ((size_t)(tok0 + colq * 16 + bit) * H + h) * KD + quad * 32 + hf * 16 + lr;
                        const int x = 4 * (j >> 1) + (j & 1);
                        if ((want_kt >> bit) & 1u) {
                            a.dktil[g] = dkt[x];
                            a.dktil[g + 8] = dkt[x + 2];
                        }
                        if ((want_kr >> bit) & 1u) {
                            a.dkread[g] = dkr[x];
                            a.dkread[g + 8] = dkr[x + 2];
                        }
                    }
                }
            }
            {   // per-token sums over the warp's 32 features: lane bit 4 picks the set, bits 3 and 2 the token of the four
                float x[8] = {gv[0], gv[1], gv[2], gv[3], bv[0], bv[1], bv[2], bv[3]};
#pragma unroll
                for (int st = 4; st > 0; st >>= 1) {
                    const bool up = (lane & (4 * st)) != 0;
#pragma unroll
                    for (int y = 0; y < st; ++y) {
                        const float send = up ? x[y] : x[y + st], keep = up ? x[y + st] : x[y];
                        x[y] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * st);
                    }
                }
                sSum[ph][quad][lane >> 4][j0 + 8 * ((lane >> 3) & 1) + ((lane >> 2) & 1)] = x[0];
                const float y = warp_sum(fmaf(sGam[CH - 1], part, rsum));   // gamma_C <dS, S> and the writes' decay to the chunk's end
                if (lane == 0) sRed[ph][warp] = y;
            }
            fence_proxy_async();
            tc_fence_before();
            if (len < CH) {   // a ragged chunk leaves row by row, once every warp has staged its part
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar_rows);
                if (!mbar_wait(&bar_rows, ragged++ & 1, a.status, ERR_MMA2)) break;
                for (int e = tid; e < len * 16; e += CBW_THREADS) {
                    const int j = e >> 4, ch = e & 15;
                    const size_t g = ((size_t)(tok0 + j) * H + h) * KD + ch * 8;
                    const uint32_t off = (uint32_t)(ch >> 3) * BOX + sw128_chunk(j, ch & 7);
                    *reinterpret_cast<uint4*>(a.dq + g) = *reinterpret_cast<const uint4*>(sm + ST_DQ + off);
                    *reinterpret_cast<uint4*>(a.dv + g) = *reinterpret_cast<const uint4*>(sm + ST_DV + off);
                    if ((sk >> j) & 1ull) *reinterpret_cast<uint4*>(a.dk + g) = *reinterpret_cast<const uint4*>(sm + ST_DK + off);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ef);
        }
    }
    tc_fence_before();
    __syncthreads();
}

// Backward of the layer's second phase in one launch.  CTA b first walks the chains b, b + grid, ...
// (reverse state recurrence), each of which publishes its finished tiles; then every CTA processes
// chunk-local tiles from the queue until none is left.  CTAs beyond the number of chains start on the
// queue at once, so the SMs the chains leave idle work on the tiles the chains have already finished.
// Nothing in a chain waits for a consumer, and a consumer waits (within a bound) only for tiles whose
// chain is running or has run: lower block indices are dispatched first.
__global__ void __launch_bounds__(CBK_THREADS, 1)
tc_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
              const __grid_constant__ CUtensorMap tmKt, const __grid_constant__ CUtensorMap tmV,
              const __grid_constant__ CUtensorMap tmDO, const __grid_constant__ CUtensorMap tmDQ,
              const __grid_constant__ CUtensorMap tmDK, const __grid_constant__ CUtensorMap tmDV,
              TcChainBwdArgs ca, TcChunkBwdArgs cb, TileQueue tq, int nchains)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = align1024(smem_raw);
    __shared__ uint32_t tmem_base;
    const int warp = threadIdx.x >> 5;
    if (warp == 0) tmem_alloc(&tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = tmem_base;
    pdl_release();
    pdl_wait();
    for (int chain = (int)blockIdx.x; chain < nchains; chain += (int)gridDim.x)
        chain_bwd_role(tmDO, tmKt, ca, chain, sm, tb, tq);
    chunk_bwd_role(tmQ, tmK, tmKt, tmV, tmDO, tmDQ, tmDK, tmDV, cb, sm, tb, tq);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tb, 512);
}

// Exercises the bounded wait by itself: one warp waits on a barrier that nothing ever arrives on.  The
// wait gives up after `limit_cycles`, records `code` in the status word and the kernel returns.
__global__ void wait_timeout_selftest_kernel(int* status, long long limit_cycles, int code)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    mbar_wait(&bar, 0, status, code, limit_cycles);
}

template <typename F> bool set_smem(F* kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

}  // namespace

// Merged forward launch: SMs that must be left over to feed the chains.
constexpr int FWD_MIN_FEEDERS = 32;
constexpr double FWD_STEP_OVER_TILE = FWD_STEP_OVER_TILE_F;

int launch_wait_timeout_selftest(int* status, long long limit_cycles, int code, cudaStream_t st)
{
    wait_timeout_selftest_kernel<<<1, 32, 0, st>>>(status, limit_cycles, code);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

bool tc_supported(const osdn_params& p)
{
    return p.io_dtype == OSDN_BF16 && p.K == KD && p.V == KD && get_encoder() != nullptr;
}

int tc_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, bool save,
               cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    const TcLayout t = make_tc_layout(p, L, save);
    if (t.total > L.total) return -1;
    Table tab = carve_table(ws, L);
    const int S = L.S, H = p.H;
    const size_t Ttot = p.nseq > 0 ? (size_t)p.T : (size_t)p.B * p.T;
    int* status = reinterpret_cast<int*>(w + L.status);
    int launches = 0;

    // phase 1 on CUDA cores: bf16 write keys, chunk-start preconditioners
    // and the control regions that have to start at zero: the forward's tickets and flags, the backward's tile queue
    // (which the backward clears again behind itself)
    const int region = 64 + L.NTmax * H;
    ClearList clear{};
    clear.p[0] = reinterpret_cast<int*>(w + t.ready);
    clear.n[0] = region;
    if (save) {
        clear.p[1] = reinterpret_cast<int*>(w + t.queue);
        clear.n[1] = region;
    }
    const int n1 = phase1_forward(p, hy, L, ws, a, w + t.ktil, true, save, clear, st);
    if (n1 < 0) return -1;
    launches += n1;

    CUtensorMap tmK, tmQ, tmKt, tmV;
    if (!make_token_map(&tmK, a.k, Ttot, H) || !make_token_map(&tmQ, a.q, Ttot, H) ||
        !make_token_map(&tmKt, w + t.ktil, Ttot, H) || !make_token_map(&tmV, a.v, Ttot, H))
        return -1;
    TcChunkArgs ca{};
    ca.H = H; ca.tab = tab; ca.beta = a.beta; ca.gate = a.gate; ca.scale = hy.scale;
    ca.WT = reinterpret_cast<uint8_t*>(w + t.WT); ca.Tb = reinterpret_cast<uint8_t*>(w + t.Tb);
    ca.Tm = reinterpret_cast<uint8_t*>(w + t.Tm); ca.P = reinterpret_cast<uint8_t*>(w + t.P);
    ca.Qg = reinterpret_cast<uint8_t*>(w + t.Qg); ca.save = save ? 1 : 0; ca.status = status;
    TcChainArgs ch{};
    ch.H = H; ch.tab = tab; ch.gate = a.gate; ch.init_state = a.init_state;
    ch.out = static_cast<__nv_bfloat16*>(a.out); ch.final_state = a.final_state;
    ch.WT = reinterpret_cast<uint8_t*>(w + t.WT); ch.Tb = reinterpret_cast<uint8_t*>(w + t.Tb);
    ch.P = reinterpret_cast<uint8_t*>(w + t.P); ch.Sn = reinterpret_cast<uint8_t*>(w + t.Sn);
    ch.dUT = reinterpret_cast<uint8_t*>(w + t.dUT); ch.scale = hy.scale; ch.save = save ? 1 : 0;
    ch.status = status;
    // One launch for both passes when enough SMs are left over to feed the chains.  The order of the tiles is arithmetic in
    // a dense batch and comes from the chunk table in a packed one.
    const int grid = num_sms(), nchains = S * H;
    const int nchunks = p.nseq > 0 ? 0 : (p.T + CH - 1) / CH;
    if (nchains + FWD_MIN_FEEDERS <= grid) {
        FwdSched sc{};
        sc.tickets = reinterpret_cast<int*>(w + t.ready);
        sc.nchains = nchains;
        sc.nchunks = nchunks;
        sc.ntickets = nchunks * nchains;
        sc.nseq = S;
        sc.feeders = grid - nchains;
        // The chains start once the feeders alone can keep up with them to the end: a chain step costs
        // about FWD_STEP_OVER_TILE of the time one SM needs for a tile.
        const double fed = (double)(grid - nchains) * nchunks * FWD_STEP_OVER_TILE;
        sc.switch_at = (int)std::max(0.0, (double)sc.ntickets - fed);
        if (p.nseq > 0) {   // both are worked out on the device from the chunk table
            sc.order = tab.order_;
            sc.longest = tab.pos_;
        }
        ca.ready = sc.tickets + 64;
        ch.ready = sc.tickets + 64;
        // Three worker groups when the longest chain outweighs the tiles (packed batches: their longest
        // sequence is not known here, and a long tail is what packing produces), four otherwise.
        const bool chain_bound = p.nseq > 0 || (double)nchunks * 2.3 > 1.5 * (double)sc.ntickets * 5.5 / grid;
        stage_mark(st, "tc_fwd");
        if (chain_bound) {
            if (!set_smem(tc_fwd_kernel<3>, CF_SMEM)) return -1;
            if (!launch_after(tc_fwd_kernel<3>, grid, 3 * CL_THREADS, CF_SMEM, st, tmK, tmQ, tmKt, tmV, ca, ch, sc)) return -1;
        } else {
            if (!set_smem(tc_fwd_kernel<4>, CF_SMEM)) return -1;
            if (!launch_after(tc_fwd_kernel<4>, grid, 4 * CL_THREADS, CF_SMEM, st, tmK, tmQ, tmKt, tmV, ca, ch, sc)) return -1;
        }
        ++launches;
    } else {
        if (!set_smem(tc_chunk_fwd_kernel, CL_SMEM)) return -1;
        stage_mark(st, "tc_chunk_fwd");
        if (!launch_after(tc_chunk_fwd_kernel, dim3(L.NTmax, H), CL_THREADS, CL_SMEM, st, tmK, tmQ, tmKt, ca)) return -1;
        ++launches;
        if (!set_smem(tc_chain_fwd_kernel, CF_SMEM)) return -1;
        stage_mark(st, "tc_chain_fwd");
        if (!launch_after(tc_chain_fwd_kernel, S * H, CFW_THREADS, CF_SMEM, st, tmV, tmKt, ch)) return -1;
        ++launches;
    }
    stage_end(st);
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

bool tc_backward_supported(const osdn_params& p) { return tc_supported(p); }

int tc_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    const TcLayout t = make_tc_layout(p, L, true);
    if (t.total > L.total) return -1;
    Table tab = carve_table(ws, L);
    const int S = L.S, H = p.H;
    const size_t Ttot = p.nseq > 0 ? (size_t)p.T : (size_t)p.B * p.T;
    int* status = reinterpret_cast<int*>(w + L.status);
    int launches = 0;
    auto U8 = [&](size_t off) { return reinterpret_cast<uint8_t*>(w + off); };
    CUtensorMap tmK, tmQ, tmKt, tmV, tmDO;
    if (!make_token_map(&tmK, a.k, Ttot, H) || !make_token_map(&tmQ, a.q, Ttot, H) ||
        !make_token_map(&tmKt, w + t.ktil, Ttot, H) || !make_token_map(&tmV, a.v, Ttot, H) ||
        !make_token_map(&tmDO, a.dout, Ttot, H))
        return -1;
    {
        TcChainBwdArgs ch{};
        ch.H = H; ch.tab = tab; ch.gate = a.gate; ch.dfinal_state = a.dfinal_state; ch.dinit_state = a.dinit_state;
        ch.WT = U8(t.WT); ch.P = U8(t.P); ch.Qg = U8(t.Qg); ch.dSn = U8(t.dSn); ch.ddUT = U8(t.ddUT);
        ch.status = status;
        TcChunkBwdArgs cb{};
        cb.H = H; cb.nseq = S; cb.tab = tab; cb.beta = a.beta; cb.gate = a.gate; cb.scale = hy.scale; cb.d_min = hy.d_min;
        cb.Tm = U8(t.Tm); cb.Sn = U8(t.Sn); cb.dSn = U8(t.dSn); cb.dUT = U8(t.dUT); cb.ddUT = U8(t.ddUT);
        cb.skipw = carve_p1(ws, L).skipw;
        cb.dq = static_cast<__nv_bfloat16*>(a.dq); cb.dk = static_cast<__nv_bfloat16*>(a.dk);
        cb.dv = static_cast<__nv_bfloat16*>(a.dv); cb.dbeta = a.dbeta; cb.dgate = a.dgate;
        cb.dktil = reinterpret_cast<float*>(w + t.dktil); cb.dkread = reinterpret_cast<float*>(w + t.dkread);
        cb.status = status;
        CUtensorMap tmDQ, tmDK, tmDV;
        if (!make_token_map(&tmDQ, a.dq, Ttot, H) || !make_token_map(&tmDK, a.dk, Ttot, H) ||
            !make_token_map(&tmDV, a.dv, Ttot, H))
            return -1;
        // tile queue between the chains and the chunk-local workers: two counters, then one slot per tile
        // (zero: cleared by the forward that saved the residuals, and again behind each backward)
        TileQueue tq{};
        tq.head = reinterpret_cast<unsigned*>(w + t.queue);
        tq.tail = tq.head + 32;
        tq.slots = reinterpret_cast<int*>(w + t.queue) + 64;
        const size_t smem = std::max(CB_SMEM, CBW_SMEM);
        if (!set_smem(tc_bwd_kernel, smem)) return -1;
        stage_mark(st, "tc_bwd");
        if (!launch_after(tc_bwd_kernel, num_sms(), CBK_THREADS, smem, st, tmQ, tmK, tmKt, tmV, tmDO, tmDQ, tmDK, tmDV, ch, cb, tq, S * H)) return -1;
        ++launches;
    }
    ClearList clear{};
    clear.p[0] = reinterpret_cast<int*>(w + t.queue);
    clear.n[0] = 64 + L.NTmax * H;
    const int n1 = phase1_backward(p, hy, L, ws, a, reinterpret_cast<float*>(w + t.dktil),
                                   reinterpret_cast<float*>(w + t.dkread), false, clear, st);
    if (n1 < 0) return -1;
    launches += n1;
    stage_end(st);
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

}  // namespace osdn

