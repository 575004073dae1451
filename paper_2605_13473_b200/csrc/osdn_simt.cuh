// Phase 2 of the layer on CUDA cores in fp32, chunk by chunk, for a scalar gate (osdn_simt.cu) and for one gate
// per key channel (osdn_kda.cu).  Everything that crosses a chunk boundary is written in pre-gated operands, so
// that the chains and the output do not know which gate it is:
//   Ktr = rho (.) ktil   (rho_i = exp(G_C - G_i), what a write still counts for at the chunk's end)
//   Qg  = gamma (.) q    (gamma_i = exp(G_i));   gC = exp(G_C), one value per key channel
// (with a scalar gate Qg is not written: its readers scale q by gamma, and gC is gamma's last value)
//   W = T diag(beta) (gamma (.) K),  U = T diag(beta) V,  P_ij = sum_c q_ic ktil_jc exp(G_ic - G_jc)
//   dU = U - W S^T,  S+ = S diag(gC) + dU^T Ktr,  O = scale (Qg S^T + P dU)
// G is the inclusive prefix of the log-gates inside the chunk.
//
// With a channel gate the factors exp(G_ic - G_jc) sit inside the contraction.  Where every |G_C| of the chunk is at
// most SAFE_RANGE they are split over the operands, exp(G_ic) and exp(-G_jc), both far inside the fp32 range, and the
// scores are plain products.  A chunk with stronger gates forms the differences pair by pair.  A factor's relative error
// is the absolute error of its exponent, and a prefix of -30 in one float is off by 1e-6 (one of -10000, behind a gate
// that forgets everything, by 5e-4): the prefix is kept as a sum of two floats.
#pragma once

#include "osdn_common.cuh"
#include "umma.cuh"

namespace osdn {
namespace {

// ---------------------------------------------------------------------------------------
// Register-tile product.  A group of 256 threads forms a 64 x (16 TN) result; a thread owns the rows
// 4 tm .. 4 tm + 3 (tm = its half-warp: rows of a warp are 8 consecutive ones) and TN columns.  Operands are
// fetched four values at a time through functors:
//   a(m, k)  -> A[m][k .. k+3]            (contraction index contiguous)
//   at(k, m) -> A^T[k][m .. m+3]          (row index contiguous)
//   b(k, n)  -> B[k][n .. n+3]            columns of a thread: 4 tn + 64 c + 0..3
//   bt(n, k) -> B^T[n][k .. k+3]          columns of a thread: tn + 16 j   (lanes read neighbouring rows)
// Per four steps of the contraction: 8 vector loads, 64 (TN = 4) or 128 (TN = 8) FMAs per thread, so the
// product runs at the FMA rate.
// ---------------------------------------------------------------------------------------
struct Lane {
    int tm, tn;   // half-warp index inside the group, lane inside the half-warp
};
__device__ __forceinline__ int row_of(const Lane& l, int i) { return l.tm * 4 + i; }
template <bool BT> __device__ __forceinline__ int col_of(const Lane& l, int j)
{
    return BT ? l.tn + 16 * j : l.tn * 4 + (j & 3) + 64 * (j >> 2);
}
__device__ __forceinline__ float comp(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

template <bool AT, bool BT, int TN, class A, class B>
__device__ __forceinline__ void tile_mm(float (&acc)[4][TN], int k0, int k1, const Lane& l, A a, B b)
{
#pragma unroll 2
    for (int k = k0; k < k1; k += 4) {
        float4 av[4], bv[TN];
#pragma unroll
        for (int i = 0; i < 4; ++i) av[i] = AT ? a(k + i, l.tm * 4) : a(l.tm * 4 + i, k);
        if constexpr (BT) {
#pragma unroll
            for (int j = 0; j < TN; ++j) bv[j] = b(l.tn + 16 * j, k);
        } else {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int c = 0; c < TN / 4; ++c) bv[c * 4 + kk] = b(k + kk, l.tn * 4 + 64 * c);
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float x = AT ? comp(av[kk], i) : comp(av[i], kk);
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    acc[i][j] = fmaf(x, BT ? comp(bv[j], kk) : comp(bv[(j >> 2) * 4 + kk], j & 3), acc[i][j]);
            }
    }
}
template <int TN> __device__ __forceinline__ void zero(float (&acc)[4][TN])
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
}
// Sum over the half-warp (the lanes that share a row).
__device__ __forceinline__ float half_sum(float x)
{
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p)
{
    const uint2 w = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, float4 v)
{
    __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    uint2 w;
    w.x = *reinterpret_cast<uint32_t*>(&a);
    w.y = *reinterpret_cast<uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = w;
}
__device__ __forceinline__ float4 operator*(float s, const float4& v) { return make_float4(s * v.x, s * v.y, s * v.z, s * v.w); }

// A tile of token rows of a packed [T,H,D] tensor: rows at or beyond len read as zero.
template <typename T, int D> struct Rows {
    const T* p;      // token tok0, head h
    size_t ld;       // H * D
    int len;
    __device__ __forceinline__ float4 operator()(int i, int c) const
    {
        return i < len ? ld4(p + (size_t)i * ld + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
};
template <typename T, int D> __device__ __forceinline__ Rows<T, D> rows_of(const void* p, int tok0, int len, int H, int h)
{
    return {static_cast<const T*>(p) + ((size_t)tok0 * H + h) * D, (size_t)H * D, len};
}

// In-chunk gate prefix and the factors derived from it: one warp scans (lane l holds tokens l and l + 32).
struct GateVecs {
    float G[CH], gam[CH], rho[CH], beta[CH];
};
__device__ __forceinline__ void load_gates(GateVecs& gv, const float* __restrict__ gate,
                                           const float* __restrict__ beta, int tok0, int len, int H, int h)
{
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        float a = l < len ? gate[(size_t)(tok0 + l) * H + h] : 0.f;
        float b = l + 32 < len ? gate[(size_t)(tok0 + l + 32) * H + h] : 0.f;
        gv.beta[l] = l < len ? beta[(size_t)(tok0 + l) * H + h] : 0.f;
        gv.beta[l + 32] = l + 32 < len ? beta[(size_t)(tok0 + l + 32) * H + h] : 0.f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
            if (l >= o) { a += ua; b += ub; }
        }
        b += __shfl_sync(0xffffffffu, a, 31);
        const float tot = __shfl_sync(0xffffffffu, b, 31);
        gv.G[l] = a;
        gv.G[l + 32] = b;
        gv.gam[l] = expf(a);
        gv.gam[l + 32] = expf(b);
        gv.rho[l] = expf(tot - a);
        gv.rho[l + 32] = expf(tot - b);
    }
}

// 16 bytes on their way into shared memory, zeros where !in (nothing is read then); both addresses 16-byte aligned.
__device__ __forceinline__ void copy16(float* dst, const float* src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(umma::smem_u32(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
// Rows of N floats, contiguous in global memory, into rows of LD floats.
template <int N, int LD, int NT> __device__ __forceinline__ void copy_rows(float* dst, const float* src, int rows)
{
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * N / 4; e += NT) copy16(dst + e / (N / 4) * LD + e % (N / 4) * 4, src + e * 4, true);
}
// An fp32 token tile like load_tile's, asynchronously.
template <int D, int LD, int NT> __device__ __forceinline__ void copy_tile(float* dst, const float* src, int tok0, int len, int H, int h)
{
    const float* p = src + ((size_t)tok0 * H + h) * D;
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * D / 4; e += NT) {
        const int i = e / (D / 4), c = e % (D / 4) * 4;
        copy16(dst + i * LD + c, p + (size_t)(i < len ? i : 0) * H * D + c, i < len);
    }
}
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// the copies asked for so far are a group; all groups but the newest have landed
__device__ __forceinline__ void copies_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void older_copies_landed() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Load a [64 x D] token tile into shared memory (rows beyond len are zero), 16 bytes at a time.
template <typename T, int D, int NT>
__device__ __forceinline__ void load_tile(float* dst, int ld, const T* __restrict__ src, int tok0, int len,
                                          int H, int h)
{
    const Rows<T, D> r = rows_of<T, D>(src, tok0, len, H, h);
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * D / 4; e += NT) {
        const int i = e / (D / 4), c = e % (D / 4) * 4;
        st4(dst + i * ld + c, r(i, c));
    }
}

// T = (I + A)^-1 in fp32 for A strictly lower triangular, 64 x 64, row stride LC; 512 threads.  The four
// 16 x 16 diagonal blocks by substitution (a thread per column, the column in registers), then the blocks
// below them by T21 = -T22 (A21 T11), 16 and then 32 wide.  tmp: 32 x 32 floats.
constexpr int LC = CH + 4;
__device__ __forceinline__ void ut_inverse_64(const float* sA, float* sT, float* tmp)
{
    const int tid = threadIdx.x;
    if (tid < 64) {
        const int blk = tid >> 4, c = tid & 15;
        const float* Ab = sA + blk * 16 * (LC + 1);
        float x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float sum = 0.f;
#pragma unroll
            for (int j4 = 0; j4 < 16; j4 += 4)
                if (j4 < i) {
                    const float4 r = ld4(Ab + i * LC + j4);
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj)
                        if (j4 + jj < i) sum = fmaf(comp(r, jj), x[j4 + jj], sum);
                }
            x[i] = (i == c ? 1.f : 0.f) - sum;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) sT[(blk * 16 + i) * LC + blk * 16 + c] = x[i];
    }
    for (int e = tid; e < CH * CH; e += 512) {   // above the diagonal blocks: zero
        const int i = e / CH, j = e % CH;
        if (j / 16 > i / 16) sT[i * LC + j] = 0.f;
    }
    __syncthreads();
    {
        const int pr = tid >> 8, i = (tid >> 4) & 15, j = tid & 15, r0 = 32 * pr + 16, c0 = 32 * pr;
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) m = fmaf(sA[(r0 + i) * LC + c0 + k], sT[(c0 + k) * LC + c0 + j], m);
        tmp[tid] = m;
        __syncthreads();
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) t = fmaf(sT[(r0 + i) * LC + r0 + k], tmp[pr * 256 + k * 16 + j], t);
        sT[(r0 + i) * LC + c0 + j] = -t;
    }
    __syncthreads();
    {
        const int i = tid >> 4, j = (tid & 15) * 2;
        float m0 = 0.f, m1 = 0.f;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const float av = sA[(32 + i) * LC + k];
            const float2 tv = *reinterpret_cast<const float2*>(sT + k * LC + j);
            m0 = fmaf(av, tv.x, m0);
            m1 = fmaf(av, tv.y, m1);
        }
        *reinterpret_cast<float2*>(tmp + i * 32 + j) = make_float2(m0, m1);
        __syncthreads();
        float t0 = 0.f, t1 = 0.f;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const float tt = sT[(32 + i) * LC + 32 + k];
            const float2 mv = *reinterpret_cast<const float2*>(tmp + k * 32 + j);
            t0 = fmaf(tt, mv.x, t0);
            t1 = fmaf(tt, mv.y, t1);
        }
        *reinterpret_cast<float2*>(sT + (32 + i) * LC + j) = make_float2(-t0, -t1);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------
// arguments of the tile-parallel passes
// ---------------------------------------------------------------------------------------
// One CTA per (chunk, head): chunks along x, heads along y and, beyond what a grid's y takes, z.
constexpr int GRID_Y = 65535;
inline dim3 tile_grid(int chunks, int H) { return dim3(chunks, H < GRID_Y ? H : GRID_Y, (H + GRID_Y - 1) / GRID_Y); }
__device__ __forceinline__ int tile_head() { return blockIdx.z * GRID_Y + blockIdx.y; }

constexpr float SAFE_RANGE = 30.f;
constexpr int CL_NT = 512;   // two groups of 256 threads, each with its own product between two barriers

struct ChunkArgs {
    int H;
    Table tab;
    const void *q, *k, *v;
    const float *beta, *gate;        // gate: [T,H], channel gate [T,H,K]
    const float* ktil;
    float *Tm, *P, *R, *W, *U;       // R: the Gram with its gate factors, A without beta.  Tm, R: null without a backward
    float *gam;                      // scalar gate only
    float *Ktr, *Qg, *gC, *G;        // Qg, gC: channel gate only.  G: channel gate only, [tile][2][64][K], the prefix's high and low parts
    // output pass, backward
    void* out;
    const void* dout;
    const float *Sn, *dU;
    float *ddU, *dSn, *dktil, *dkread;
    void *dq, *dv;
    float *dbeta, *dgate;
    Hyper hy;
};

__device__ __forceinline__ float4 exp4(const float4& v) { return make_float4(expf(v.x), expf(v.y), expf(v.z), expf(v.w)); }
// exp of a sum h + l with |l| a rounding of h
__device__ __forceinline__ float exp_sum(float h, float l)
{
    const float e = expf(h);
    return fmaf(e, l, e);
}
__device__ __forceinline__ float4 exp_sum(const float4& h, const float4& l) { return make_float4(exp_sum(h.x, l.x), exp_sum(h.y, l.y), exp_sum(h.z, l.z), exp_sum(h.w, l.w)); }
// x + y into x, the rounding of the sum into e
__device__ __forceinline__ void add_exact(float& x, float& e, float y)
{
    const float s = x + y, b = s - x;
    e += (x - (s - b)) + (y - b);
    x = s;
}
// exp((ah + al) - (bh + bl))
__device__ __forceinline__ float exp_diff(float ah, float al, float bh, float bl)
{
    float e = al - bl;
    add_exact(ah, e, -bh);
    return exp_sum(ah, e);
}
__device__ __forceinline__ float4 exp_diff(const float4& ah, const float4& al, const float4& bh, const float4& bl)
{
    return make_float4(exp_diff(ah.x, al.x, bh.x, bl.x), exp_diff(ah.y, al.y, bh.y, bl.y), exp_diff(ah.z, al.z, bh.z, bl.z), exp_diff(ah.w, al.w, bh.w, bl.w));
}
__device__ __forceinline__ float4 operator*(const float4& a, const float4& b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
__device__ __forceinline__ float4 operator-(const float4& a, const float4& b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ float4 operator+(const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 neg_part(const float4& v) { return make_float4(fminf(v.x, 0.f), fminf(v.y, 0.f), fminf(v.z, 0.f), fminf(v.w, 0.f)); }
template <int TN> __device__ __forceinline__ float4 quad(const float (&x)[TN], int c) { return make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]); }
template <int TN> __device__ __forceinline__ void set_quad(float (&x)[TN], int c, const float4& v) { x[c] = v.x; x[c + 1] = v.y; x[c + 2] = v.z; x[c + 3] = v.w; }

// Strong channel gates: acc[i][n] += sum_j c(m, j) b(j, n) exp(G_mn - G_jn) over j <= m, or with REV exp(G_jn - G_mn)
// over j >= m.  c is zero on the other side of the diagonal, where the exponent is clamped.  g, gl: the prefix's parts.
template <bool REV, int TN, class C, class B, class GG, class GL>
__device__ __forceinline__ void pair_mm(float (&acc)[4][TN], int j0, int j1, const Lane& l, C c, B b, GG g, GL gl)
{
#pragma unroll
    for (int cc = 0; cc < TN; cc += 4) {
        const int n = col_of<false>(l, cc);
        float4 gm[4], lm[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            gm[i] = g(row_of(l, i), n);
            lm[i] = gl(row_of(l, i), n);
        }
        for (int j = j0; j < j1; ++j) {
            const float4 bj = b(j, n), gj = g(j, n), lj = gl(j, n);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 e = c(row_of(l, i), j) * (bj * exp4(neg_part(REV ? (gj - gm[i]) + (lj - lm[i]) : (gm[i] - gj) + (lm[i] - lj))));
                set_quad(acc[i], cc, make_float4(acc[i][cc] + e.x, acc[i][cc + 1] + e.y, acc[i][cc + 2] + e.z, acc[i][cc + 3] + e.w));
            }
        }
    }
}

// A gate below this is a factor of zero in fp32 whatever its value (exp(-104) is less than half of the smallest number),
// and taken as this the prefix stays finite.
constexpr float GATE_FLOOR = -104.f;

// In-chunk prefix of the channel gates in shared memory, [64][LD], over the rows, as high parts in x and low parts in lo;
// the threads cut the rows into segments.  tot: [2][CL_NT / K][K] scratch.
template <int K, int LD> __device__ __forceinline__ void gate_prefix(float* x, float* lo, float* tot)
{
    constexpr int SEG = CL_NT / K, ROWS = CH / SEG;
    const int c = threadIdx.x % K, s = threadIdx.x / K;
    auto gate = [&](int r) {
        const float g = x[(s * ROWS + r) * LD + c];
        return g < GATE_FLOOR ? GATE_FLOOR : g;
    };
    float h = 0.f, l = 0.f;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) add_exact(h, l, gate(r));
    tot[s * K + c] = h;
    tot[(SEG + s) * K + c] = l;
    __syncthreads();
    h = l = 0.f;
#pragma unroll
    for (int o = 0; o < SEG; ++o)
        if (o < s) {
            add_exact(h, l, tot[o * K + c]);
            l += tot[(SEG + o) * K + c];
        }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        add_exact(h, l, gate(r));
        const float g = h + l;
        x[(s * ROWS + r) * LD + c] = g;
        lo[(s * ROWS + r) * LD + c] = (h - g) + l;
    }
    __syncthreads();
}

// Inclusive sums of the columns of x, [64][LD], down the rows (REV: up), in place.  tot: [CL_NT / K][K] scratch.
template <int K, int LD, bool REV> __device__ __forceinline__ void column_scan(float* x, float* tot)
{
    constexpr int SEG = CL_NT / K, ROWS = CH / SEG;
    const int c = threadIdx.x % K, s = threadIdx.x / K;
    float acc = 0.f;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int i = s * ROWS + (REV ? ROWS - 1 - r : r);
        acc += x[i * LD + c];
        x[i * LD + c] = acc;
    }
    tot[s * K + c] = acc;
    __syncthreads();
    float off = 0.f;
#pragma unroll
    for (int o = 0; o < SEG; ++o)
        if (REV ? o > s : o < s) off += tot[o * K + c];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) x[(s * ROWS + r) * LD + c] += off;
    __syncthreads();
}

template <typename T, int K, int V, bool CG> struct LocalFwd {
    static constexpr int LD = K + 4;
    static constexpr size_t SMEM = sizeof(float) * ((CG ? 5 : 3) * CH * LD + 2 * CH * LC);
    // scalar gate at K = V = 64: two CTAs per SM
    static constexpr int MIN_CTAS = !CG && K + V == 128 ? 2 : 1;
};

// Chunk-local forward: A, T = (I + A)^-1, W, U, P and the gated operands.  Bound by its FMAs.
template <typename T, int K, int V, bool CG>
__global__ void __launch_bounds__(CL_NT, LocalFwd<T, K, V, CG>::MIN_CTAS) chunk_local_fwd_kernel(ChunkArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    constexpr int LD = K + 4, TK = K / 16, TV = V / 16;
    float* sK = sm;                   // k; channel gate: gamma (.) k
    float* sKt = sK + CH * LD;        // ktil; channel gate, safe: ktil exp(-G)
    float* sQ = sKt + CH * LD;        // q; channel gate: gamma (.) q
    float* sT = sQ + CH * LD;
    float* sA = sT + CH * LC;
    float* sG = sA + CH * LC;         // channel gate only: the prefix's high and low parts
    float* sL = sG + CH * LD;
    __shared__ GateVecs gv;
    __shared__ float tmp[32 * 32];

    const int c = blockIdx.x, h = tile_head(), H = a.H;
    if (h >= H) return;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const int grp = threadIdx.x >> 8;
    const Lane l{(int)(threadIdx.x & 255) >> 4, (int)threadIdx.x & 15};

    copy_tile<K, LD, CL_NT>(sKt, a.ktil, tok0, len, H, h);   // on their way while k and q are converted
    if constexpr (CG) copy_tile<K, LD, CL_NT>(sG, a.gate, tok0, len, H, h);
    load_tile<T, K, CL_NT>(sK, LD, static_cast<const T*>(a.k), tok0, len, H, h);
    load_tile<T, K, CL_NT>(sQ, LD, static_cast<const T*>(a.q), tok0, len, H, h);
    copies_landed();
    bool safe = true;
    if constexpr (CG) {
        if (threadIdx.x < CH) gv.beta[threadIdx.x] = threadIdx.x < len ? a.beta[(size_t)(tok0 + threadIdx.x) * H + h] : 0.f;
        __syncthreads();
        gate_prefix<K, LD>(sG, sL, tmp);
        safe = __syncthreads_and(threadIdx.x >= K || fabsf(sG[(CH - 1) * LD + (threadIdx.x & (K - 1))]) <= SAFE_RANGE);
        if (threadIdx.x < K) a.gC[tile * K + threadIdx.x] = exp_sum(sG[(CH - 1) * LD + threadIdx.x], sL[(CH - 1) * LD + threadIdx.x]);
    } else {
        load_gates(gv, a.gate, a.beta, tok0, len, H, h);
        __syncthreads();
        if (threadIdx.x < CH) a.gam[tile * CH + threadIdx.x] = gv.gam[threadIdx.x];
    }
    for (int e = threadIdx.x; e < CH * K / 4; e += CL_NT) {
        const int i = e / (K / 4), n = e % (K / 4) * 4;
        const size_t g = tile * CH * K + e * 4;
        const float4 kt = ld4(sKt + i * LD + n);
        if constexpr (CG) {
            const float4 q = ld4(sQ + i * LD + n);
            const float4 G = ld4(sG + i * LD + n), gl = ld4(sL + i * LD + n), eg = exp_sum(G, gl), qg = eg * q;
            if (a.G) {
                st4(a.G + tile * 2 * CH * K + e * 4, G);
                st4(a.G + (tile * 2 + 1) * CH * K + e * 4, gl);
            }
            st4(a.Qg + g, qg);
            st4(a.Ktr + g, exp_diff(ld4(sG + (CH - 1) * LD + n), ld4(sL + (CH - 1) * LD + n), G, gl) * kt);
            st4(sQ + i * LD + n, qg);
            st4(sK + i * LD + n, eg * ld4(sK + i * LD + n));
            if (safe) st4(sKt + i * LD + n, exp_sum(-1.f * G, -1.f * gl) * kt);
        } else {
            st4(a.Ktr + g, gv.rho[i] * kt);
        }
    }
    __syncthreads();

    // R_ij = 1[j<i] <k_i, ktil_j>_gated, A = beta_i R   (group 0)   and   P_ij = 1[j<=i] <q_i, ktil_j>_gated
    {
        float acc[4][4];
        zero(acc);
        if (!CG || safe) {
            const float* X = grp == 0 ? sK : sQ;
            tile_mm<false, true, 4>(acc, 0, K, l, [&](int m, int k) { return ld4(X + m * LD + k); },
                                    [&](int n, int k) { return ld4(sKt + n * LD + k); });
        } else {
            const Rows<T, K> x = rows_of<T, K>(grp == 0 ? a.k : a.q, tok0, len, H, h);
            for (int k = 0; k < K; k += 4) {
                float4 kt[4], gn[4], ln[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    kt[j] = ld4(sKt + col_of<true>(l, j) * LD + k);
                    gn[j] = ld4(sG + col_of<true>(l, j) * LD + k);
                    ln[j] = ld4(sL + col_of<true>(l, j) * LD + k);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 xm = x(row_of(l, i), k), gm = ld4(sG + row_of(l, i) * LD + k), lm = ld4(sL + row_of(l, i) * LD + k);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 p = (xm * kt[j]) * exp4(neg_part((gm - gn[j]) + (lm - ln[j])));
                        acc[i][j] += (p.x + p.y) + (p.z + p.w);
                    }
                }
            }
        }
        float* out = (grp == 0 ? a.R : a.P) + tile * CH * CH;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = row_of(l, i), n = col_of<true>(l, j);
                float g = n < m || (n == m && grp == 1) ? acc[i][j] : 0.f;
                if constexpr (!CG) g *= expf(fminf(gv.G[m] - gv.G[n], 0.f));
                if (grp == 1 || a.R) out[m * CH + n] = g;
                if (grp == 0) sA[m * LC + n] = gv.beta[m] * g;
            }
    }
    __syncthreads();
    // v takes q's place while the first 64 threads substitute (read where it is, inside the product, it held the tile up for
    // 20000 of 64000 cycles at K = V = 128)
    if constexpr (V <= K) {
        const Rows<T, V> v = rows_of<T, V>(a.v, tok0, len, H, h);
        if (threadIdx.x >= 64)
#pragma unroll 4
            for (int e = threadIdx.x - 64; e < CH * V / 4; e += CL_NT - 64) st4(sQ + e / (V / 4) * LD + e % (V / 4) * 4, v(e / (V / 4), e % (V / 4) * 4));
    }
    ut_inverse_64(sA, sT, tmp);
    if (a.Tm) {
        float* Tg = a.Tm + tile * CH * CH;
        for (int e = threadIdx.x; e < CH * CH / 4; e += CL_NT) st4(Tg + e * 4, ld4(sT + (e / 16) * LC + (e % 16) * 4));
    }

    // W = T diag(beta) (gamma K) ; U = T diag(beta) V.  T is lower triangular: rows of a warp end at 8 w + 8.
    const int jend = (l.tm & ~1) * 4 + 8;
    if (grp == 0) {
        float acc[4][TK];
        zero(acc);
        tile_mm<false, false, TK>(acc, 0, jend, l, [&](int m, int j) { return ld4(sT + m * LC + j); },
                                  [&](int j, int n) { return (CG ? gv.beta[j] : gv.beta[j] * gv.gam[j]) * ld4(sK + j * LD + n); });
        float* Wg = a.W + tile * CH * K;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TK; cc += 4) st4(Wg + row_of(l, i) * K + col_of<false>(l, cc), quad(acc[i], cc));
    } else {
        float acc[4][TV];
        zero(acc);
        const Rows<T, V> v = rows_of<T, V>(a.v, tok0, len, H, h);
        tile_mm<false, false, TV>(acc, 0, jend, l, [&](int m, int j) { return ld4(sT + m * LC + j); },
                                  [&](int j, int n) {
                                    if constexpr (V <= K) return gv.beta[j] * ld4(sQ + j * LD + n);
                                    else return gv.beta[j] * v(j, n);
                                });
        float* Ug = a.U + tile * CH * V;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TV; cc += 4) st4(Ug + row_of(l, i) * V + col_of<false>(l, cc), quad(acc[i], cc));
    }
}

// O = scale (Qg S_n^T + P dU), one tile per CTA once the chain has left S_n and dU: the output is off the
// sequential path.
template <int K, int V> constexpr size_t output_smem() { return sizeof(float) * ((CH + V) * (K + 4) + CH * LC); }
// gamma (.) q of a tile into shared memory.
template <typename T, int K, bool CG, int LD, int NT> __device__ __forceinline__ void load_gated_q(float* dst, const ChunkArgs& a, size_t tile, int tok0, int len, int h)
{
    const Rows<T, K> q = rows_of<T, K>(a.q, tok0, len, a.H, h);
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * K / 4; e += NT) {
        const int i = e / (K / 4), n = e % (K / 4) * 4;
        if constexpr (CG) st4(dst + i * LD + n, ld4(a.Qg + tile * CH * K + e * 4));
        else st4(dst + i * LD + n, a.gam[tile * CH + i] * q(i, n));
    }
}

template <typename T, int K, int V, bool CG>
__global__ void __launch_bounds__(256) output_kernel(ChunkArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    constexpr int TV = V / 16, LD = K + 4, NT = 256;
    float* sQ = sm;                  // [64][LD]
    float* sS = sQ + CH * LD;        // [V][LD], S_n; then dU [64][V]
    float* sP = sS + V * LD;         // [64][LC]
    const int c = blockIdx.x, h = tile_head(), H = a.H;
    if (h >= H) return;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const Lane l{(int)threadIdx.x >> 4, (int)threadIdx.x & 15};
    const float* S = a.Sn + tile * V * K;
    const float* P = a.P + tile * CH * CH;
    const float* dU = a.dU + tile * CH * V;
#pragma unroll 8
    for (int e = threadIdx.x; e < V * K / 4; e += NT) st4(sS + e / (K / 4) * LD + e % (K / 4) * 4, ld4(S + e * 4));
    load_gated_q<T, K, CG, LD, NT>(sQ, a, tile, tok0, len, h);
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * CH / 4; e += NT) st4(sP + e / 16 * LC + e % 16 * 4, ld4(P + e * 4));
    float4 u[CH * V / 4 / NT];
#pragma unroll
    for (int x = 0; x < CH * V / 4 / NT; ++x) u[x] = ld4(dU + (threadIdx.x + x * NT) * 4);
    __syncthreads();
    float acc[4][TV];
    zero(acc);
    tile_mm<false, true, TV>(acc, 0, K, l, [&](int m, int k) { return ld4(sQ + m * LD + k); }, [&](int n, int k) { return ld4(sS + n * LD + k); });
    __syncthreads();
    float* sU = sS;
#pragma unroll
    for (int x = 0; x < CH * V / 4 / NT; ++x) st4(sU + (threadIdx.x + x * NT) * 4, u[x]);
    __syncthreads();
    const int jend = (l.tm & ~1) * 4 + 8;
    for (int j4 = 0; j4 < jend; j4 += 4) {   // columns tn + 16 n as above: scalar reads of dU
        float4 pv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) pv[i] = ld4(sP + row_of(l, i) * LC + j4);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
#pragma unroll
            for (int n = 0; n < TV; ++n) {
                const float x = sU[(j4 + jj) * V + l.tn + 16 * n];
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][n] = fmaf(comp(pv[i], jj), x, acc[i][n]);
            }
    }
    T* o = static_cast<T*>(a.out);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = row_of(l, i);
        if (m < len)
#pragma unroll
            for (int n = 0; n < TV; ++n) stf(o + ((size_t)(tok0 + m) * H + h) * V + l.tn + 16 * n, a.hy.scale * acc[i][n]);
    }
}

// What the reverse chain's step does not need the state cotangent for, tile-parallel:
//   ddU0 = scale P^T dO  (into ddU)   and   G0 = scale dO^T Qg  (into dSn, which the chain then overwrites)
template <int K, int V> constexpr size_t pre_bwd_smem() { return sizeof(float) * (CH * CH + CH * V + CH * K); }
template <typename T, int K, int V, bool CG>
__global__ void __launch_bounds__(256) pre_bwd_kernel(ChunkArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    constexpr int TV = V / 16, TK = K / 16, NT = 256;
    float* sP = sm;
    float* sO = sP + CH * CH;   // [64][V]
    float* sQ = sO + CH * V;    // [64][K]
    const int c = blockIdx.x, h = tile_head(), H = a.H;
    if (h >= H) return;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const Lane l{(int)threadIdx.x >> 4, (int)threadIdx.x & 15};
    const float* P = a.P + tile * CH * CH;
    const float s = a.hy.scale;
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * CH / 4; e += NT) st4(sP + e * 4, ld4(P + e * 4));
    load_gated_q<T, K, CG, K, NT>(sQ, a, tile, tok0, len, h);
    load_tile<T, V, NT>(sO, V, static_cast<const T*>(a.dout), tok0, len, H, h);
    __syncthreads();
    {
        float acc[4][TV];
        zero(acc);
        // P is lower triangular: row i of P^T starts at column i
        tile_mm<true, false, TV>(acc, (l.tm & ~1) * 4, CH, l, [&](int j, int m) { return ld4(sP + j * CH + m); },
                                 [&](int j, int n) { return ld4(sO + j * V + n); });
        float* o = a.ddU + tile * CH * V;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TV; cc += 4) st4(o + row_of(l, i) * V + col_of<false>(l, cc), s * quad(acc[i], cc));
    }
    float* g0 = a.dSn + tile * V * K;
#pragma unroll
    for (int v0 = 0; v0 < V; v0 += 64) {
        float acc[4][TK];
        zero(acc);
        tile_mm<true, false, TK>(acc, 0, CH, l, [&](int j, int m) { return ld4(sO + j * V + v0 + m); },
                                 [&](int j, int n) { return ld4(sQ + j * K + n); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TK; cc += 4) st4(g0 + (v0 + row_of(l, i)) * K + col_of<false>(l, cc), s * quad(acc[i], cc));
    }
}

// ---------------------------------------------------------------------------------------
// State chains.  Forward and backward are the same recurrence over pre-gated tiles,
//   D = D0 -+ X S^T ;   S <- S diag(gC) + G0 +- D^T Y
//   forward   X = W,   Y = Ktr, D0 = U,    G0 = 0,                  chunks ascending  (D = dU,  S = state)
//   backward  X = Ktr, Y = W,   D0 = ddU0, G0 = scale dO^T Qg,      chunks descending (D = ddU, S = its cotangent)
// and rows of S do not interact, so a chain is cut into slices of rows, one CTA each.  A tile's X and Y rows
// arrive by asynchronous copies, one chunk ahead.
// ---------------------------------------------------------------------------------------
struct ChainArgs {
    int H;
    Table tab;
    const float *X, *Y, *D0, *G0, *S0;        // G0, S0 nullable
    const float *gC, *gam;                    // decay of a chunk: per channel (channel gate), or gam's last value
    float *D, *Sall, *Sfin;                   // Sall: S before every chunk of the walk; Sfin nullable
    int* status;
};
constexpr int CODE_SIMT_RING = 141;

// X and Y of a tile, rows padded to K + 4 floats.
template <int K> struct Stage {
    float X[CH * (K + 4)], Y[CH * (K + 4)];
};
// One group of 16-byte copies by all threads.  Narrow slices take this form: with one bulk copy per row, four warps issue 32
// each, one after the other, in the middle of a step that is short (4 x 1000 tokens, 4 heads, K = V = 64: a chain 38.9 -> 28.8
// us, forward and backward 196 -> 178).
template <int K, int NT> __device__ __forceinline__ void fetch_group(Stage<K>& g, const ChainArgs& a, size_t tile, bool any)
{
    if (any) {
        copy_rows<K, K + 4, NT>(g.X, a.X + tile * CH * K, CH);
        copy_rows<K, K + 4, NT>(g.Y, a.Y + tile * CH * K, CH);
    }
    copies_group();
}
// One bulk copy per row by the first 128 threads.  Wide slices take this form: their step hides the issue (channel gate, 8 x 2048
// tokens, 8 heads, reverse chain: 336 us against 358 with the copies above; forward chains equal).
template <int K> __device__ __forceinline__ void fetch_stage(Stage<K>& g, const ChainArgs& a, size_t tile, uint64_t* bar)
{
    if (threadIdx.x == 0) umma::mbar_expect_tx(bar, 2 * CH * K * 4);
    __syncwarp();
    if (threadIdx.x < 2 * CH) {
        // a copy's bytes may be counted before they are expected: the count is signed, and the phase cannot end
        // while the one arrival (with the expected bytes) is missing
        const int i = threadIdx.x & (CH - 1);
        const float* src = (threadIdx.x < CH ? a.X : a.Y) + (tile * CH + i) * K;
        umma::bulk_load((threadIdx.x < CH ? g.X : g.Y) + i * (K + 4), src, K * 4, bar);
    }
}

struct ChainWalk {   // the chunks of one chain in the order of the walk
    int first, n, step;
    __device__ __forceinline__ int at(int j) const { return first + j * step; }
};
template <bool BWD> __device__ __forceinline__ ChainWalk walk_of(const Table& tab, int sq)
{
    const int c0 = tab.seq_chunk0(sq), c1 = tab.seq_chunk0(sq + 1);
    return {BWD ? c1 - 1 : c0, c1 - c0, BWD ? -1 : 1};
}

template <int N> __device__ __forceinline__ void ldn(float (&x)[N], const float* p)
{
    if constexpr (N == 4) set_quad(x, 0, ld4(p));
    else {
        const float2 v = *reinterpret_cast<const float2*>(p);
        x[0] = v.x; x[1] = v.y;
    }
}
template <int N> __device__ __forceinline__ void stn(float* p, const float (&x)[N])
{
    if constexpr (N == 4) st4(p, quad(x, 0));
    else *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
}

// ---- slices of 8 rows: for few chains, where a step's latency counts.  Eight warps split the contraction of
// both products, every lane holds a 4 x 4 tile, the partial sums meet in shared memory.
constexpr int VS = 8, CNT = 256;

// acc[i][v] += sum over this warp's k of X[i][k] S[v][k]   (rows i = li + 16 ii, v = 4 lv + vv)
template <int K, int LD>
__device__ __forceinline__ void slice_dot(float (&acc)[4][4], const float* X, const float* Y, int warp, int li, int lv)
{
    constexpr int KW = K / 8;
#pragma unroll
    for (int k = 0; k < KW; k += 4) {
        float4 x[4], y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = ld4(X + (li + 16 * i) * LD + warp * KW + k);
#pragma unroll
        for (int v = 0; v < 4; ++v) y[v] = ld4(Y + (lv * 4 + v) * LD + warp * KW + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[i][v] = fmaf(comp(x[i], kk), comp(y[v], kk), acc[i][v]);
    }
}
// acc[v][kk] += sum over tokens i0 .. i0 + ni - 1 of D[i][v] Y[i][k + kk]   (v = 4 lv + vv)
template <int LD>
__device__ __forceinline__ void slice_outer(float (&acc)[4][4], const float* Y, const float* D, int i0, int ni, int k)
{
#pragma unroll 8
    for (int i = i0; i < i0 + ni; ++i) {
        const float4 y = ld4(Y + i * LD + k), d = ld4(D + i * VS);
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) acc[v][kk] = fmaf(comp(d, v), comp(y, kk), acc[v][kk]);
    }
}

template <int K> struct NarrowShared {
    static constexpr int LD = K + 4, CW = K / 64, GROUPS = 8 / CW;   // a warp takes 64 columns and 64 / GROUPS tokens
    Stage<K> stage[2];
    float S[VS * LD];
    float part[8 * CH * VS];     // dot: [8][64][VS]; outer: [GROUPS][VS][K] (the same size)
    float D[CH * VS];
};

template <int K, int V, bool BWD, bool CG>
__global__ void __launch_bounds__(CNT) chain_narrow_kernel(ChainArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    using Sh = NarrowShared<K>;
    constexpr int LD = Sh::LD, CW = Sh::CW, G = Sh::GROUPS, NI = CH / G, PER = VS * K / CNT;   // state values per thread
    Sh& s = *reinterpret_cast<Sh*>(sm);
    const int chain = blockIdx.x, H = a.H;
    const int sq = chain / H, h = chain % H, v0 = blockIdx.y * VS;
    const ChainWalk w = walk_of<BWD>(a.tab, sq);
    const int t = threadIdx.x, warp = t >> 5, li = t & 15, lv = (t >> 4) & 1;
    const size_t srow = (((size_t)sq * H + h) * V + v0) * K;
    const int oi = t / (VS / 2), ov = t % (VS / 2) * 2;       // outputs of the first product's summing pass
    const int sv = t * PER / K, sk = t * PER % K;             // this thread's values of S
    auto tile_of = [&](int j) { return (size_t)w.at(j) * H + h; };

    float S[PER] = {};
    if (a.S0) ldn(S, a.S0 + srow + t * PER);
    auto ld2 = [](const float* p) { return *reinterpret_cast<const float2*>(p); };
    auto d0_of = [&](int j) { return j < w.n ? ld2(a.D0 + (tile_of(j) * CH + oi) * V + v0 + ov) : make_float2(0.f, 0.f); };
    fetch_group<K, CNT>(s.stage[0], a, tile_of(0), w.n > 0);
    float2 d0 = d0_of(0);
    for (int j = 0; j < w.n; ++j) {
        const size_t tile = tile_of(j);
        const Stage<K>& g = s.stage[j & 1];
        float g0[PER] = {}, gc[PER];
        if constexpr (BWD) ldn(g0, a.G0 + (tile * V + v0) * K + t * PER);
        if constexpr (CG) ldn(gc, a.gC + tile * K + sk);
        else {
            const float g1 = a.gam[tile * CH + CH - 1];
#pragma unroll
            for (int x = 0; x < PER; ++x) gc[x] = g1;
        }
        stn(s.S + sv * LD + sk, S);
        fetch_group<K, CNT>(s.stage[(j + 1) & 1], a, tile_of(j + 1), j + 1 < w.n);
        older_copies_landed();
        __syncthreads();
        stn(a.Sall + (tile * V + v0) * K + t * PER, S);   // (backward: the place this thread took G0 from)
        {
            float acc[4][4];
            zero(acc);
            slice_dot<K, LD>(acc, g.X, s.S, warp, li, lv);
#pragma unroll
            for (int i = 0; i < 4; ++i) st4(s.part + (warp * CH + li + 16 * i) * VS + lv * 4, quad(acc[i], 0));
        }
        __syncthreads();
        {
            float2 d = d0;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const float2 p = ld2(s.part + x * CH * VS + t * 2);
                d = BWD ? make_float2(d.x + p.x, d.y + p.y) : make_float2(d.x - p.x, d.y - p.y);
            }
            *reinterpret_cast<float2*>(a.D + (tile * CH + oi) * V + v0 + ov) = d;
            *reinterpret_cast<float2*>(s.D + t * 2) = BWD ? make_float2(-d.x, -d.y) : d;
            d0 = d0_of(j + 1);
        }
        __syncthreads();
        {
            float acc[4][4];
            zero(acc);
            const int grp = warp / CW, k = warp % CW * 64 + li * 4;
            slice_outer<LD>(acc, g.Y, s.D + lv * 4, grp * NI, NI, k);
#pragma unroll
            for (int v = 0; v < 4; ++v) st4(s.part + (grp * VS + lv * 4 + v) * K + k, quad(acc[v], 0));
        }
        __syncthreads();
#pragma unroll
        for (int x = 0; x < PER; ++x) {
            float p = g0[x];
#pragma unroll
            for (int y = 0; y < G; ++y) p += s.part[y * VS * K + t * PER + x];
            S[x] = fmaf(gc[x], S[x], p);
        }
        // part is read here and written again two barriers on; the stage and s.S were last read before the
        // barrier above
    }
    if (a.Sfin) stn(a.Sfin + srow + t * PER, S);
}

// ---- slices of 64 rows: for many chains, where the FMAs count.  One 4 x 4 thread tile per product; K / 64 groups of
// 256 threads split the contraction of the first product and the columns of the second.
constexpr int WS = 64;
template <int K> struct WideShared {
    static constexpr int LD = K + 4, LW = WS + 4, G = K / 64;
    Stage<K> stage[2];
    float S[WS * LD];
    float part[G][CH * LW];      // first product's partial sums, then D in part[0]
    uint64_t full[2];
};

template <int K, int V, bool BWD, bool CG>
__global__ void __launch_bounds__(K / 64 * 256) chain_wide_kernel(ChainArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    using Sh = WideShared<K>;
    constexpr int LD = Sh::LD, LW = Sh::LW, G = Sh::G, NT = G * 256;
    Sh& s = *reinterpret_cast<Sh*>(sm);
    const int chain = blockIdx.x, H = a.H;
    const int sq = chain / H, h = chain % H, v0 = blockIdx.y * WS;
    const ChainWalk w = walk_of<BWD>(a.tab, sq);
    const int t = threadIdx.x, grp = t >> 8;
    const Lane l{(t & 255) >> 4, t & 15};
    const size_t srow = (((size_t)sq * H + h) * V + v0) * K;
    auto tile_of = [&](int j) { return (size_t)w.at(j) * H + h; };
    const int k_own = grp * 64 + l.tn * 4;   // columns of S this thread advances, rows 4 tm + i

    if (t == 0) {
        umma::mbar_init(&s.full[0], 1);
        umma::mbar_init(&s.full[1], 1);
        umma::fence_mbar_init();
    }
    for (int e = t * 4; e < WS * K; e += NT * 4)
        st4(s.S + e / K * LD + e % K, a.S0 ? ld4(a.S0 + srow + e) : make_float4(0.f, 0.f, 0.f, 0.f));
    __syncthreads();
    if (w.n > 0) fetch_stage<K>(s.stage[0], a, tile_of(0), &s.full[0]);
    for (int j = 0; j < w.n; ++j) {
        const size_t tile = tile_of(j);
        const Stage<K>& g = s.stage[j & 1];
        const float* D0 = a.D0 + tile * CH * V + v0;
        float* sn = a.Sall + (tile * V + v0) * K;
        if (j + 1 < w.n) fetch_stage<K>(s.stage[(j + 1) & 1], a, tile_of(j + 1), &s.full[(j + 1) & 1]);
        float4 g0[4], d0[CH * WS / 4 / NT];
        float4 gc;
        if constexpr (CG) gc = ld4(a.gC + tile * K + k_own);
        else gc.x = gc.y = gc.z = gc.w = a.gam[tile * CH + CH - 1];
        if constexpr (BWD)
#pragma unroll
            for (int i = 0; i < 4; ++i) g0[i] = ld4(a.G0 + (tile * V + v0 + l.tm * 4 + i) * K + k_own);
#pragma unroll
        for (int x = 0; x < CH * WS / 4 / NT; ++x) {
            const int e = (t + x * NT) * 4;
            d0[x] = ld4(D0 + (size_t)(e / WS) * V + e % WS);
        }
        const bool ok = umma::mbar_wait(&s.full[j & 1], (j >> 1) & 1, a.status, CODE_SIMT_RING);
        if (!__syncthreads_and(ok)) {   // give up, once the copies in flight have landed
            for (int x = j; x <= j + 1 && x < w.n; ++x) umma::mbar_drain(&s.full[x & 1], (x >> 1) & 1);
            break;
        }
        // S is complete and G0 has been read
        for (int e = t * 4; e < WS * K; e += NT * 4) st4(sn + e, ld4(s.S + e / K * LD + e % K));
        {
            float acc[4][4];
            zero(acc);
            tile_mm<false, true, 4>(acc, grp * 64, grp * 64 + 64, l, [&](int m, int k) { return ld4(g.X + m * LD + k); },
                                    [&](int n, int k) { return ld4(s.S + n * LD + k); });
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) s.part[grp][row_of(l, i) * LW + col_of<true>(l, jj)] = acc[i][jj];
        }
        __syncthreads();
#pragma unroll
        for (int x = 0; x < CH * WS / 4 / NT; ++x) {
            const int e = (t + x * NT) * 4, o = e / WS * LW + e % WS;
            float4 d = d0[x];
#pragma unroll
            for (int y = 0; y < G; ++y) {
                const float4 p = ld4(s.part[y] + o);
                d = BWD ? make_float4(d.x + p.x, d.y + p.y, d.z + p.z, d.w + p.w) : d - p;
            }
            st4(a.D + tile * CH * V + (size_t)(e / WS) * V + v0 + e % WS, d);
            st4(s.part[0] + o, BWD ? -1.f * d : d);
        }
        __syncthreads();
        {
            float acc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if constexpr (BWD) set_quad(acc[i], 0, g0[i]);
                else set_quad(acc[i], 0, make_float4(0.f, 0.f, 0.f, 0.f));
            tile_mm<true, false, 4>(acc, 0, CH, l, [&](int k, int m) { return ld4(s.part[0] + k * LW + m); },
                                    [&](int k, int n) { return ld4(g.Y + k * LD + grp * 64 + n); });
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float* S = s.S + (l.tm * 4 + i) * LD + k_own;
                const float4 o = gc * ld4(S);
                st4(S, make_float4(acc[i][0] + o.x, acc[i][1] + o.y, acc[i][2] + o.z, acc[i][3] + o.w));
            }
        }
        __syncthreads();   // the stage may be filled again
    }
    if (a.Sfin)
        for (int e = t * 4; e < WS * K; e += NT * 4) st4(a.Sfin + srow + e, ld4(s.S + e / K * LD + e % K));
}

// ---------------------------------------------------------------------------------------
// chunk-local backward: gradients through P, the state-advance factors, the solve, A, gates.
//
// With dU = T R, R = diag(beta) (V - gamma (.) K S^T):  dVb = T^T ddU is R's gradient, dA = -strictLower(dVb dU^T) the
// scores', and dKb = -dVb S the read keys' share of R.  (Gradients of W, U and T, and T^T dT T^T, are never formed: a fifth
// fewer FMAs than that way, and one phase fewer.)  Ten products per tile in three phases; in each the two groups of 256
// threads form different ones.  Bound by the FMAs and the shared-memory pipe.  k, ktil, q (gated as in the forward), dU, dVb, T
// and the 64 x 64 intermediates sit in shared memory; S, dS, ddU, v and dO are read where they are, by rows that a half-warp
// shares or by whole lines.
//
// The gate gradient needs no sums of its own over the score matrices: with
//   E_i = dq_i (.) q_i + dk_read_i (.) k_i - dktil_i (.) ktil_i     (phase-2 gradients)
// dG_i = E_i + 1[i = last] (sum_j dKtr_j (.) Ktr_j + gC (.) sum_v dS (.) S), summed over the channels, and the gate's
// gradient is its suffix sum inside the chunk.
// With a gate per channel that sum is taken apart, since behind strong gates it is small against terms that cancel in it: a
// token's product with itself (the diagonal of P), which is in dq (.) q and in dktil (.) ktil, is left out of both; and what
// the chunk's end takes from the writes, sum over j < i of dKtr_j (.) Ktr_j, is a prefix sum instead of the total less a
// suffix.
// ---------------------------------------------------------------------------------------
template <int K, int V> constexpr size_t local_bwd_smem() { return sizeof(float) * (3 * CH * (K + 4) + CH * ((K > V ? K : V) + 4) + 4 * CH * LC); }
template <typename T, int K, int V, bool CG>
__global__ void __launch_bounds__(CL_NT) chunk_local_bwd_kernel(ChunkArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    constexpr int LD = K + 4, LU = V + 4, TK = K / 16, TV = V / 16, PARTS = CL_NT / K;
    float* sK = sm;                 // as in the forward: channel gate gamma (.) k
    float* sKt = sK + CH * LD;      //                    safe: ktil exp(-G)
    float* sQ = sKt + CH * LD;      //                    gamma (.) q
    float* sW = sQ + CH * LD;       // dVb [64][LU]; channel gate, at the end: dq (.) q + dk (.) k [64][LD]
    float* sX = sW + CH * (K > V ? LD : LU);   // [64][LC] dA * beta_i * gates; before that, and the space behind it, dU [64][LU]
    float* sT = sX + 2 * CH * LC;   // T.  Channel gate, at the end, with the space before it: dktil (.) ktil
    float* sDP = sT + CH * LC;      // dP * gates
    float* sU = sX;
    __shared__ GateVecs gv;
    __shared__ float sB[3][CH], sE[3][CH];   // channel gate: sE[0] the diagonal of dP
    __shared__ __align__(16) float sRed[PARTS][K], sR[8][K];   // column sums of dS (.) S and of dKtr (.) Ktr

    const int c = blockIdx.x, h = tile_head(), H = a.H;
    if (h >= H) return;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const float scale = a.hy.scale;
    const int grp = threadIdx.x >> 8;
    const Lane l{(int)(threadIdx.x & 255) >> 4, (int)threadIdx.x & 15};
    const int m_hi = (l.tm & ~1) * 4 + 8, m_lo = m_hi - 8;   // rows of this warp: [m_lo, m_hi)

    const Rows<T, K> qr = rows_of<T, K>(a.q, tok0, len, H, h), kr = rows_of<T, K>(a.k, tok0, len, H, h);
    const Rows<T, V> vr = rows_of<T, V>(a.v, tok0, len, H, h), dor = rows_of<T, V>(a.dout, tok0, len, H, h);
    const float* Sg = a.Sn + tile * V * K;
    const float* dSg = a.dSn + tile * V * K;
    const float* dUg = a.dU + tile * CH * V;
    const float* ddUg = a.ddU + tile * CH * V;
    const float* Gg = CG ? a.G + tile * 2 * CH * K : nullptr;
    auto G4 = [&](int i, int n) { return ld4(Gg + i * K + n); };
    auto L4 = [&](int i, int n) { return ld4(Gg + (CH + i) * K + n); };
    auto expG = [&](int i, int n) { return exp_sum(G4(i, n), L4(i, n)); };
    auto expmG = [&](int i, int n) { return exp_sum(-1.f * G4(i, n), -1.f * L4(i, n)); };

    bool safe = true;
    if constexpr (CG) safe = __syncthreads_and(threadIdx.x >= K || fabsf(Gg[(CH - 1) * K + (threadIdx.x & (K - 1))]) <= SAFE_RANGE);
    // what is needed as it is comes asynchronously, under the gate factors
    copy_rows<CH, LC, CL_NT>(sT, a.Tm + tile * CH * CH, CH);
    copy_rows<V, LU, CL_NT>(sU, dUg, CH);
    if constexpr (CG) copy_rows<K, LD, CL_NT>(sQ, a.Qg + tile * CH * K, CH);
#pragma unroll 2
    for (int e = threadIdx.x; e < CH * K / 4; e += CL_NT) {
        const int i = e / (K / 4), n = e % (K / 4) * 4;
        const Rows<float, K> ktr = rows_of<float, K>(a.ktil, tok0, len, H, h);
        float4 k = kr(i, n), kt = ktr(i, n);
        if constexpr (CG) {
            k = expG(i, n) * k;
            if (safe) kt = expmG(i, n) * kt;
        } else {
            st4(sQ + i * LD + n, qr(i, n));
        }
        st4(sK + i * LD + n, k);
        st4(sKt + i * LD + n, kt);
    }
    if constexpr (CG) {
        if (threadIdx.x < CH) gv.beta[threadIdx.x] = threadIdx.x < len ? a.beta[(size_t)(tok0 + threadIdx.x) * H + h] : 0.f;
    } else {
        load_gates(gv, a.gate, a.beta, tok0, len, H, h);
    }
    {
        const int n = threadIdx.x % K, part = threadIdx.x / K;
        float s = 0.f;
#pragma unroll 16
        for (int v = part; v < V; v += PARTS) s = fmaf(Sg[v * K + n], dSg[v * K + n], s);
        sRed[part][n] = s;
    }
    copies_landed();
    __syncthreads();

    // row sums <x_i, y_i> of a 4 x TN tile, written by one lane per row
    auto row_dots = [&](auto& acc, auto ld, float* dst) {
        constexpr int TN = sizeof(acc[0]) / 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float s = 0.f;
#pragma unroll
            for (int cc = 0; cc < TN; cc += 4) {
                const float4 y = ld(row_of(l, i), col_of<false>(l, cc));
                s = fmaf(acc[i][cc], y.x, fmaf(acc[i][cc + 1], y.y, fmaf(acc[i][cc + 2], y.z, fmaf(acc[i][cc + 3], y.w, s))));
            }
            s = half_sum(s);
            if (l.tn == 0) dst[row_of(l, i)] = s;
        }
    };
    auto store_rows = [&](auto& acc, auto* base, int D) {   // rows of this tile that exist, at [token, head, :]
        constexpr int TN = sizeof(acc[0]) / 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (row_of(l, i) < len)
#pragma unroll
                for (int cc = 0; cc < TN; cc += 4)
                    st4(base + ((size_t)(tok0 + row_of(l, i)) * H + h) * D + col_of<false>(l, cc), quad(acc[i], cc));
    };
    auto scale_rows = [&](auto& acc, auto f) {   // f(m, n): a factor per element (four at a time)
        constexpr int TN = sizeof(acc[0]) / 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TN; cc += 4) set_quad(acc[i], cc, f(row_of(l, i), col_of<false>(l, cc)) * quad(acc[i], cc));
    };
    auto splat = [](float x) { return make_float4(x, x, x, x); };
    // channel gate: x (.) y of a tile, plus z, into dst [64][LD]
    auto put_products = [&](auto& acc, auto ld, float* dst, auto z) {
        constexpr int TN = sizeof(acc[0]) / 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TN; cc += 4) {
                const int m = row_of(l, i), n = col_of<false>(l, cc);
                const float4 p = quad(acc[i], cc) * ld(m, n), o = z(m, n);
                st4(dst + m * LD + n, make_float4(p.x + o.x, p.y + o.y, p.z + o.z, p.w + o.w));
            }
    };
    // channel gate: the diagonal of dP times x
    auto add_diag = [&](auto& acc, auto ld) {
        constexpr int TN = sizeof(acc[0]) / 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TN; cc += 4) set_quad(acc[i], cc, quad(acc[i], cc) + sE[0][row_of(l, i)] * ld(row_of(l, i), col_of<false>(l, cc)));
    };
    auto ldK = [&](int m, int n) { return ld4(sK + m * LD + n); };
    auto ldKt = [&](int m, int n) { return ld4(sKt + m * LD + n); };
    auto ldQ = [&](int m, int n) { return ld4(sQ + m * LD + n); };

    // (1) dVb = T^T ddU ; dv = beta dVb                     |  dP * gates = 1[j<=i] scale dO dU^T
    if (grp == 0) {
        float acc[4][TV];
        zero(acc);
        tile_mm<true, false, TV>(acc, m_lo, CH, l, [&](int k, int m) { return ld4(sT + k * LC + m); }, [&](int k, int n) { return ld4(ddUg + k * V + n); });
        row_dots(acc, vr, sB[1]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TV; cc += 4) st4(sW + row_of(l, i) * LU + col_of<false>(l, cc), quad(acc[i], cc));
        scale_rows(acc, [&](int m, int) { return splat(gv.beta[m]); });
        store_rows(acc, static_cast<T*>(a.dv), V);
    } else {
        float acc[4][4];
        zero(acc);
        tile_mm<false, true, 4>(acc, 0, V, l, [&](int m, int k) { return dor(m, k); }, [&](int n, int k) { return ld4(sU + n * LU + k); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = row_of(l, i), n = col_of<true>(l, j);
                float x = n <= m ? scale * acc[i][j] : 0.f;
                if constexpr (!CG) x *= expf(fminf(gv.G[m] - gv.G[n], 0.f));
                else if (n == m) {
                    sE[0][m] = x;
                    x = 0.f;
                }
                sDP[m * LC + n] = x;
            }
    }
    __syncthreads();

    float keep[4][TK];   // group 0: dk of the read key; group 1: dktil
    zero(keep);
    // (2) dq = gamma (scale dO S) + dP ktil (gated)         |  dA = -strictLower(dVb dU^T), dbeta_i += dA_ij R_ij
    if (grp == 0) {
        float acc[4][TK];
        zero(acc);
        tile_mm<false, false, TK>(acc, 0, V, l, [&](int m, int k) { return scale * dor(m, k); }, [&](int k, int n) { return ld4(Sg + k * K + n); });
        auto dP = [&](int m, int k) { return ld4(sDP + m * LC + k); };
        if constexpr (!CG) {
            scale_rows(acc, [&](int m, int) { return splat(gv.gam[m]); });
            tile_mm<false, false, TK>(acc, 0, m_hi, l, dP, ldKt);
            row_dots(acc, ldQ, sE[0]);
        } else {
            auto products = [&](auto ld) {   // dq (.) q waits in dgate, for the same thread
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (row_of(l, i) < len)
#pragma unroll
                        for (int cc = 0; cc < TK; cc += 4)
                            st4(a.dgate + ((size_t)(tok0 + row_of(l, i)) * H + h) * K + col_of<false>(l, cc),
                                quad(acc[i], cc) * ld(row_of(l, i), col_of<false>(l, cc)));
            };
            if (safe) {
                tile_mm<false, false, TK>(acc, 0, m_hi, l, dP, ldKt);
                products(ldQ);
                add_diag(acc, ldKt);
                scale_rows(acc, expG);
            } else {
                scale_rows(acc, expG);
                pair_mm<false, TK>(acc, 0, m_hi, l, [&](int m, int j) { return sDP[m * LC + j]; }, ldKt, G4, L4);
                products(qr);
                add_diag(acc, ldKt);
            }
        }
        store_rows(acc, static_cast<T*>(a.dq), K);
        // dKb = -dVb S (dk grows from it)                   |  dKtr = dU dS (dktil grows from it)
        tile_mm<false, false, TK>(keep, 0, V, l, [&](int m, int k) { return ld4(sW + m * LU + k); }, [&](int k, int n) { return ld4(Sg + k * K + n); });
        scale_rows(keep, [&](int m, int) { return splat(CG ? -1.f : -gv.gam[m]); });
        row_dots(keep, ldK, sB[0]);
        scale_rows(keep, [&](int m, int) { return splat(gv.beta[m]); });
    } else {
        {
            float acc[4][4];
            zero(acc);
            tile_mm<false, true, 4>(acc, 0, V, l, [&](int m, int k) { return ld4(sW + m * LU + k); }, [&](int n, int k) { return ld4(sU + n * LU + k); });
            asm volatile("bar.sync 1, 256;" ::: "memory");   // dU, whose space X takes, has been read
            const float* Rg = a.R + tile * CH * CH;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int m = row_of(l, i);
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int n = col_of<true>(l, j);
                    float da = n < m ? -acc[i][j] : 0.f;
                    s = fmaf(da, Rg[m * CH + n], s);
                    if constexpr (!CG) da *= expf(fminf(gv.G[m] - gv.G[n], 0.f));
                    sX[m * LC + n] = da * gv.beta[m];
                }
                s = half_sum(s);
                if (l.tn == 0) sB[2][m] = s;
            }
        }
        tile_mm<false, false, TK>(keep, 0, V, l, [&](int m, int k) { return ld4(dUg + m * V + k); }, [&](int k, int n) { return ld4(dSg + k * K + n); });
        // towards dktil: rho (.) dKtr; channel gate, safe: gC (.) dKtr, the common factor exp(-G) follows at the end
        if constexpr (!CG) scale_rows(keep, [&](int m, int) { return splat(gv.rho[m]); });
        else if (safe) scale_rows(keep, [&](int, int n) { return expG(CH - 1, n); });
        else scale_rows(keep, [&](int m, int n) { return exp_diff(G4(CH - 1, n), L4(CH - 1, n), G4(m, n), L4(m, n)); });
        if constexpr (!CG) {
            float col[TK];
#pragma unroll
            for (int j = 0; j < TK; ++j) col[j] = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int cc = 0; cc < TK; cc += 4) {
                    const float4 p = quad(keep[i], cc) * ldKt(row_of(l, i), col_of<false>(l, cc));
                    col[cc] += p.x; col[cc + 1] += p.y; col[cc + 2] += p.z; col[cc + 3] += p.w;
                }
#pragma unroll
            for (int j = 0; j < TK; ++j) col[j] += __shfl_xor_sync(0xffffffffu, col[j], 16);
            if (!(threadIdx.x & 16))
#pragma unroll
                for (int cc = 0; cc < TK; cc += 4) st4(&sR[(threadIdx.x >> 5) & 7][col_of<false>(l, cc)], quad(col, cc));
        } else {   // waits in dktil, for the same thread
            store_rows(keep, a.dktil, K);
            zero(keep);
        }
        auto dPt = [&](int k, int m) { return ld4(sDP + k * LC + m); };
        if (!CG || safe) tile_mm<true, false, TK>(keep, m_lo, CH, l, dPt, ldQ);
        else pair_mm<true, TK>(keep, m_lo, CH, l, [&](int m, int j) { return sDP[j * LC + m]; }, qr, G4, L4);
    }
    __syncthreads();

    // (3) dk (read side) = beta gamma dKb + X ktil (gated)   |  dktil = dKtr part + dP^T q + X^T k (gated)
    float* sE2 = sT - CH * LC;   // channel gate: dktil (.) ktil, over the rest of dU and T
    if (grp == 0) {
        auto X = [&](int m, int k) { return ld4(sX + m * LC + k); };
        if constexpr (!CG) {
            tile_mm<false, false, TK>(keep, 0, m_hi, l, X, ldKt);
            row_dots(keep, ldK, sE[1]);
        } else {
            const Rows<float, K> eq = rows_of<float, K>(a.dgate, tok0, len, H, h);
            auto put = [&](auto ld) { put_products(keep, ld, sW, eq); };
            if (safe) {
                tile_mm<false, false, TK>(keep, 0, m_hi, l, X, ldKt);
                put(ldK);
                scale_rows(keep, expG);
            } else {
                scale_rows(keep, expG);
                pair_mm<false, TK>(keep, 0, m_hi, l, [&](int m, int j) { return sX[m * LC + j]; }, ldKt, G4, L4);
                put(kr);
            }
        }
        store_rows(keep, a.dkread, K);
    } else {
        if (!CG || safe) tile_mm<true, false, TK>(keep, m_lo, CH, l, [&](int k, int m) { return ld4(sX + k * LC + m); }, ldK);
        else pair_mm<true, TK>(keep, m_lo, CH, l, [&](int m, int j) { return sX[j * LC + m]; }, kr, G4, L4);
        if constexpr (!CG) {
            row_dots(keep, ldKt, sE[2]);
        } else {
            const Rows<float, K> part = rows_of<float, K>(a.dktil, tok0, len, H, h);   // (rows beyond len: dU is zero there)
            put_products(keep, ldKt, sE2, [](int, int) { return make_float4(0.f, 0.f, 0.f, 0.f); });
            if (safe) add_diag(keep, ldQ);
            else add_diag(keep, qr);
            asm volatile("bar.sync 1, 256;" ::: "memory");   // gamma (.) q has been read: its place takes dKtr (.) Ktr
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int cc = 0; cc < TK; cc += 4) {
                    const int m = row_of(l, i), n = col_of<false>(l, cc);
                    const float4 x = part(m, n);
                    st4(sQ + m * LD + n, x * ldKt(m, n));
                    set_quad(keep[i], cc, quad(keep[i], cc) + x);
                }
            if (safe) scale_rows(keep, expmG);
        }
        store_rows(keep, a.dktil, K);
    }
    __syncthreads();

    // gate gradients: suffix sums of dG inside the chunk; dbeta
    if constexpr (!CG) {
        if (threadIdx.x < 32) {   // one warp, lane l holds tokens l and l + 32
            const int i = threadIdx.x;
            float x = sE[0][i] + sE[1][i] - sE[2][i], y = sE[0][i + 32] + sE[1][i + 32] - sE[2][i + 32];
            float rs = 0.f, tot = 0.f;
            for (int n = i; n < K; n += 32) {
#pragma unroll
                for (int p = 0; p < 8; ++p) rs += sR[p][n];
#pragma unroll
                for (int p = 0; p < PARTS; ++p) tot += sRed[p][n];
            }
            rs = warp_sum(rs);
            tot = warp_sum(tot);
            if (i == 31) y += rs + gv.gam[CH - 1] * tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float ux = __shfl_down_sync(0xffffffffu, x, o), uy = __shfl_down_sync(0xffffffffu, y, o);
                if (i + o < 32) { x += ux; y += uy; }
            }
            x += __shfl_sync(0xffffffffu, y, 0);
            const size_t th = (size_t)(tok0 + i) * H + h;
            if (i < len) a.dgate[th] = x;
            if (i + 32 < len) a.dgate[th + (size_t)32 * H] = y;
        }
    } else {
        for (int e = threadIdx.x; e < CH * K / 4; e += CL_NT) {
            const int i = e / (K / 4), n = e % (K / 4) * 4;
            st4(sW + i * LD + n, ld4(sW + i * LD + n) - ld4(sE2 + i * LD + n));
        }
        __syncthreads();
        column_scan<K, LD, true>(sW, sK);
        column_scan<K, LD, false>(sQ, sK);
        for (int e = threadIdx.x; e < len * (K / 4); e += CL_NT) {
            const int i = e / (K / 4), n = e % (K / 4) * 4;
            float4 tot = make_float4(0.f, 0.f, 0.f, 0.f), x = ld4(sW + i * LD + n);
#pragma unroll
            for (int p = 0; p < PARTS; ++p) tot = tot + ld4(&sRed[p][n]);
            if (i > 0) x = x + ld4(sQ + (i - 1) * LD + n);
            st4(a.dgate + ((size_t)(tok0 + i) * H + h) * K + n, x + ld4(a.gC + tile * K + n) * tot);
        }
    }
    if (threadIdx.x >= 64 && threadIdx.x < 64 + CH) {
        const int i = threadIdx.x - 64;
        if (i < len) a.dbeta[(size_t)(tok0 + i) * H + h] = sB[0][i] + sB[1][i] + sB[2][i];
    }
}

// ---------------------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------------------
template <typename F> bool set_smem(F* kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

// Narrow or wide slices: whichever walk is expected to end first.  What decides is how many waves of CTAs each cut makes; a
// wave of wide slices (eight times the rows) takes as long as WIDE_STEP waves of narrow ones.  Measured, 512 tokens, forward
// chain, microseconds for 1, 2, 3, 4, 5 waves of narrow slices against one of wide ones: K = 64 25 (18 with one CTA to an SM),
// 45, 64, 82 against 53; K = 128 25, 43, 59, 78, 96 against 86 (channel gate, reverse chain 27, -, 64, 84, 104 against 88).
template <int K> constexpr int WIDE_STEP_TENTHS = K == 64 ? 25 : 40;
template <int K, int V, bool BWD, bool CG> int launch_chain(const ChainArgs& ch, int chains, cudaStream_t st)
{
    const int SLOTS = num_sms() * (K == 64 ? 2 : 1);   // CTAs of either kind that fit an SM: by their shared memory
    const long narrow = ((long)chains * (V / VS) + SLOTS - 1) / SLOTS, wide = ((long)chains * (V / WS) + SLOTS - 1) / SLOTS;
    stage_mark(st, BWD ? "chain_bwd" : "chain_fwd");
    if (narrow * 10 <= wide * WIDE_STEP_TENTHS<K>) {
        if (!set_smem(chain_narrow_kernel<K, V, BWD, CG>, sizeof(NarrowShared<K>))) return -1;
        if (!launch_after(chain_narrow_kernel<K, V, BWD, CG>, dim3(chains, V / VS), CNT, sizeof(NarrowShared<K>), st, ch)) return -1;
    } else {
        if (!set_smem(chain_wide_kernel<K, V, BWD, CG>, sizeof(WideShared<K>))) return -1;
        if (!launch_after(chain_wide_kernel<K, V, BWD, CG>, dim3(chains, V / WS), K / 64 * 256, sizeof(WideShared<K>), st, ch)) return -1;
    }
    return 1;
}

inline ChunkArgs chunk_args(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, float* G)
{
    char* w = static_cast<char*>(ws);
    auto F = [&](size_t off) { return off ? reinterpret_cast<float*>(w + off) : nullptr; };   // (none of these regions is the first)
    ChunkArgs c{};
    c.H = p.H; c.tab = carve_table(ws, L); c.q = a.q; c.k = a.k; c.v = a.v; c.beta = a.beta; c.gate = a.gate;
    c.ktil = F(L.ktil); c.Tm = F(L.Tm); c.P = F(L.P); c.R = F(L.R); c.W = F(L.W); c.U = F(L.dU);
    c.Ktr = F(L.Ktr); c.Qg = F(L.Qg); c.gC = F(L.gC); c.gam = F(L.gam); c.G = G; c.Sn = F(L.Sn); c.dU = F(L.dU); c.hy = hy;
    return c;
}

// Phase 2 forward behind phase 1 (fp32 write keys in L.ktil); returns the number of launches or -1.
template <typename T, int K, int V, bool CG>
int chunk_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, float* G, cudaStream_t st)
{
    ChunkArgs c = chunk_args(p, hy, L, ws, a, G);
    c.out = a.out;
    const dim3 tiles = tile_grid(L.NTmax, p.H);
    using LF = LocalFwd<T, K, V, CG>;
    if (!set_smem(chunk_local_fwd_kernel<T, K, V, CG>, LF::SMEM)) return -1;
    stage_mark(st, "chunk_local_fwd");
    if (!launch_after(chunk_local_fwd_kernel<T, K, V, CG>, tiles, CL_NT, LF::SMEM, st, c)) return -1;
    ChainArgs ch{};
    ch.H = p.H; ch.tab = c.tab; ch.X = c.W; ch.Y = c.Ktr; ch.D0 = c.U; ch.gC = c.gC; ch.gam = c.gam; ch.S0 = a.init_state;
    ch.D = const_cast<float*>(c.dU); ch.Sall = const_cast<float*>(c.Sn); ch.Sfin = a.final_state;
    ch.status = reinterpret_cast<int*>(static_cast<char*>(ws) + L.status);
    if (launch_chain<K, V, false, CG>(ch, L.S * p.H, st) < 0) return -1;
    if (!set_smem(output_kernel<T, K, V, CG>, output_smem<K, V>())) return -1;
    stage_mark(st, "chunk_output");
    if (!launch_after(output_kernel<T, K, V, CG>, tiles, 256, output_smem<K, V>(), st, c)) return -1;
    return cudaGetLastError() == cudaSuccess ? 3 : -1;
}

// Phase 2 backward; leaves the fp32 gradients of the read keys and the write keys for phase 1.
template <typename T, int K, int V, bool CG>
int chunk_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, float* G, cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    auto F = [&](size_t off) { return reinterpret_cast<float*>(w + off); };
    ChunkArgs c = chunk_args(p, hy, L, ws, a, G);
    c.dout = a.dout; c.ddU = F(L.ddU); c.dSn = F(L.dSn); c.dktil = F(L.dktil); c.dkread = F(L.dkread);
    c.dq = a.dq; c.dv = a.dv; c.dbeta = a.dbeta; c.dgate = a.dgate;
    const dim3 tiles = tile_grid(L.NTmax, p.H);
    if (!set_smem(pre_bwd_kernel<T, K, V, CG>, pre_bwd_smem<K, V>())) return -1;
    stage_mark(st, "chunk_pre_bwd");
    if (!launch_after(pre_bwd_kernel<T, K, V, CG>, tiles, 256, pre_bwd_smem<K, V>(), st, c)) return -1;
    ChainArgs ch{};
    ch.H = p.H; ch.tab = c.tab; ch.X = c.Ktr; ch.Y = c.W; ch.D0 = c.ddU; ch.G0 = c.dSn; ch.gC = c.gC; ch.gam = c.gam; ch.S0 = a.dfinal_state;
    ch.D = c.ddU; ch.Sall = c.dSn; ch.Sfin = a.dinit_state;
    ch.status = reinterpret_cast<int*>(w + L.status);
    if (launch_chain<K, V, true, CG>(ch, L.S * p.H, st) < 0) return -1;
    if (!set_smem(chunk_local_bwd_kernel<T, K, V, CG>, local_bwd_smem<K, V>())) return -1;
    stage_mark(st, "chunk_local_bwd");
    if (!launch_after(chunk_local_bwd_kernel<T, K, V, CG>, tiles, CL_NT, local_bwd_smem<K, V>(), st, c)) return -1;
    return cudaGetLastError() == cudaSuccess ? 3 : -1;
}

// FN<T, K, V>(...) for the problem's types and sizes.
#define OSDN_DISPATCH(FN, ...)                                                              \
    do {                                                                                    \
        if (p.io_dtype == OSDN_FP32) {                                                      \
            if (p.K == 64 && p.V == 64) return FN<float, 64, 64>(__VA_ARGS__);              \
            if (p.K == 128 && p.V == 128) return FN<float, 128, 128>(__VA_ARGS__);          \
            if (p.K == 64 && p.V == 128) return FN<float, 64, 128>(__VA_ARGS__);            \
            if (p.K == 128 && p.V == 64) return FN<float, 128, 64>(__VA_ARGS__);            \
        } else {                                                                            \
            if (p.K == 64 && p.V == 64) return FN<__nv_bfloat16, 64, 64>(__VA_ARGS__);      \
            if (p.K == 128 && p.V == 128) return FN<__nv_bfloat16, 128, 128>(__VA_ARGS__);  \
            if (p.K == 64 && p.V == 128) return FN<__nv_bfloat16, 64, 128>(__VA_ARGS__);    \
            if (p.K == 128 && p.V == 64) return FN<__nv_bfloat16, 128, 64>(__VA_ARGS__);    \
        }                                                                                   \
        return -1;                                                                          \
    } while (0)

}  // namespace
}  // namespace osdn
