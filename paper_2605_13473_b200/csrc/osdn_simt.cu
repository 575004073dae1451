// CUDA-core (fp32 FMA) kernels of the OSDN layer.
//
// This family is the fp32 mode of the library (fp32 I/O needs better than TF32 accuracy)
// and the reference-quality path for bf16 I/O when OSDN_FLAG_FORCE_SIMT is set.  Every
// step of the chunkwise algorithm runs here in fp32:
//
//   phase1_fwd      Algorithm 1 with APF and the box projection, one warp per chain
//   chunk_local_fwd decay-ratio Gram A, UT inverse T, W = T diag(beta gamma) K,
//                   U = T diag(beta) V, local scores P           (gated chunk form)
//   chain_fwd       dU = U - W S^T ; S <- gamma_C S + dU^T (rho Ktil)   (state recurrence)
//   output          O = scale[(gamma Q) S^T + P dU]
//   ddu0, chain_bwd reverse state chain: ddU (its part without dS first), dS
//   chunk_local_bwd all chunk-local gradients (through P, W, U, T, A and the gate prefix)
//   phase1_bwd      reverse sweep over the projected affine recurrence (Section 3.5)
//
// Notation follows the paper: G_i in-chunk inclusive prefix of the log gate,
// gamma_i = exp(G_i), Gamma_ij = exp(G_i - G_j), rho_i = exp(G_C - G_i).
#include "osdn_common.cuh"

namespace osdn {

namespace {

// ---------------------------------------------------------------------------------------
// chunk table
// ---------------------------------------------------------------------------------------
// One CTA.  Chunk counts per sequence are scanned 256 sequences at a time; every chunk then finds
// its sequence by bisection over the chunk offsets (kept in shared memory while they fit).
constexpr int TBL_THREADS = 256, TBL_SMEM_SEQ = 2048;

// The offsets live on the device, so the host cannot check them: a sequence is clamped into the packed
// token range [0, T_total] (every later access stays inside the user tensors whatever cu_seqlens
// holds), and a violated contract (cu[0] != 0, a decreasing pair, cu[S] != T_total) is reported through
// the device status word.
__device__ __forceinline__ void clamped_sequence(const int* __restrict__ cu, int s, int T_total, int& t0, int& len, bool& bad)
{
    const int a = cu[s], b = cu[s + 1];
    bad = b < a || a < 0 || b > T_total;
    t0 = min(max(a, 0), T_total);
    len = min(max(b, t0), T_total) - t0;
}

__global__ void __launch_bounds__(TBL_THREADS)
build_table_kernel(int S, int T_dense, const int* __restrict__ cu, int NTmax, Table t, int* status)
{
    __shared__ int s_c0[TBL_SMEM_SEQ + 1];
    __shared__ int s_scan[TBL_THREADS];
    __shared__ int s_carry;
    const int tid = threadIdx.x;
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < S; base += TBL_THREADS) {
        const int s = base + tid;
        int t0 = 0, len = 0;
        if (s < S) {
            if (cu) {   // packed batch: T_dense is the packed token count
                bool bad;
                clamped_sequence(cu, s, T_dense, t0, len, bad);
                if (s == 0 && cu[0] != 0) bad = true;
                if (s == S - 1 && cu[S] != T_dense) bad = true;
                if (bad && status) atomicCAS(status, 0, OSDN_DEVICE_BAD_CU_SEQLENS);
            } else {
                t0 = s * T_dense;
                len = T_dense;
            }
        }
        const int nc = (len + CH - 1) / CH;
        s_scan[tid] = nc;
        __syncthreads();
        for (int o = 1; o < TBL_THREADS; o <<= 1) {   // inclusive scan
            const int v = tid >= o ? s_scan[tid - o] : 0;
            __syncthreads();
            s_scan[tid] += v;
            __syncthreads();
        }
        const int carry = s_carry;
        if (s < S) {
            const int c = min(carry + s_scan[tid] - nc, NTmax);
            t.seq_tok0_[s] = t0;
            t.seq_len_[s] = len;
            t.seq_chunk0_[s] = c;
            if (s <= TBL_SMEM_SEQ) s_c0[s] = c;
        }
        __syncthreads();
        if (tid == TBL_THREADS - 1) s_carry = carry + s_scan[tid];
        __syncthreads();
    }
    const int total = min(s_carry, NTmax);
    if (tid == 0) {
        t.seq_chunk0_[S] = total;
        if (S <= TBL_SMEM_SEQ) s_c0[S] = total;
    }
    __syncthreads();
    const bool in_smem = S <= TBL_SMEM_SEQ;
    for (int j = tid; j < NTmax; j += TBL_THREADS) {
        if (j >= total) {
            t.chunk_tok0_[j] = 0;
            t.chunk_len_[j] = 0;
            t.chunk_seq_[j] = 0;
            continue;
        }
        int lo = 0, hi = S - 1;   // last sequence whose first chunk is <= j (empty sequences share an offset)
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            const int c = in_smem ? s_c0[mid] : t.seq_chunk0_[mid];
            if (c <= j) lo = mid;
            else hi = mid - 1;
        }
        const int s = lo;
        const int c0 = in_smem ? s_c0[s] : t.seq_chunk0_[s];
        int t0 = s * T_dense, len = T_dense;
        if (cu) {
            bool bad;
            clamped_sequence(cu, s, T_dense, t0, len, bad);
        }
        const int rem = len - (j - c0) * CH;
        t.chunk_tok0_[j] = t0 + (j - c0) * CH;
        t.chunk_len_[j] = rem < CH ? rem : CH;
        t.chunk_seq_[j] = s;
    }
    // The chunks sorted by the step at which their chain needs them when every chain is to END at the same
    // time: chunk n of a sequence of nc chunks has the key longest - nc + n, so a short sequence starts
    // late and the longest ones are served first (a counting sort; the order among chunks of equal key
    // is whatever the atomics give).  pos_: [0] longest sequence in chunks, [2 + key] number of chunks
    // with that key, then its running offset, [2 + NTmax + 1 + key] fill counter.
    int* cnt = t.pos_ + 2;
    int* fill = t.pos_ + 3 + NTmax;
    for (int j = tid; j <= NTmax; j += TBL_THREADS) {
        cnt[j] = 0;
        if (j < NTmax) fill[j] = 0;
    }
    if (tid == 0) t.pos_[0] = 0;
    __syncthreads();
    for (int s = tid; s < S; s += TBL_THREADS) atomicMax(&t.pos_[0], t.seq_chunk0_[s + 1] - t.seq_chunk0_[s]);
    __syncthreads();
    const int maxn = t.pos_[0];
    auto key_of = [&](int j) {
        const int s = t.chunk_seq_[j];
        const int c0 = in_smem ? s_c0[s] : t.seq_chunk0_[s], c1 = in_smem ? s_c0[s + 1] : t.seq_chunk0_[s + 1];
        return maxn - (c1 - c0) + (j - c0);
    };
    for (int j = tid; j < total; j += TBL_THREADS) atomicAdd(&cnt[key_of(j)], 1);
    __syncthreads();
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < maxn; base += TBL_THREADS) {   // exclusive scan of the counts, in place
        const int n = base + tid;
        const int v = n < maxn ? cnt[n] : 0;
        s_scan[tid] = v;
        __syncthreads();
        for (int o = 1; o < TBL_THREADS; o <<= 1) {
            const int u = tid >= o ? s_scan[tid - o] : 0;
            __syncthreads();
            s_scan[tid] += u;
            __syncthreads();
        }
        const int carry = s_carry;
        if (n < maxn) cnt[n] = carry + s_scan[tid] - v;
        __syncthreads();
        if (tid == TBL_THREADS - 1) s_carry = carry + s_scan[tid];
        __syncthreads();
    }
    for (int j = tid; j < total; j += TBL_THREADS) {
        const int n = key_of(j);
        t.order_[cnt[n] + atomicAdd(&fill[n], 1)] = j;
    }
    for (int s = tid; s < S; s += TBL_THREADS) {
        const int nc = t.seq_chunk0_[s + 1] - t.seq_chunk0_[s];
        t.seq_first_[s] = nc > 0 ? cnt[maxn - nc] : 0;
    }
}

__device__ __forceinline__ float warp_sum(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

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
// chunk-local forward: A, T = (I + A)^-1, W, U, P
// ---------------------------------------------------------------------------------------
struct ChunkArgs {
    int H;
    Table tab;
    const void *q, *k, *v;
    const float *beta, *gate;
    const float* ktil;
    float *Tm, *P, *W, *U, *gvec;   // gvec: [tile][2][64] rho, gamma
    // output pass, backward
    void* out;
    const void* dout;
    const float *Sn, *dSn, *dU;
    float *ddU, *dktil, *dkread;
    void *dq, *dv;
    float *dbeta, *dgate;
    Hyper hy;
};

constexpr int CL_NT = 512;   // two groups of 256 threads, each with its own product between two barriers

// Bound by its FMAs (five products of 64 x 64 x K per tile); two CTAs per SM at K = 64.
template <typename T, int K, int V>
__global__ void __launch_bounds__(CL_NT, K + V == 128 ? 2 : 1) chunk_local_fwd_kernel(ChunkArgs a)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int LD = K + 4, TK = K / 16, TV = V / 16;
    float* sK = sm;
    float* sKt = sK + CH * LD;
    float* sQ = sKt + CH * LD;
    float* sT = sQ + CH * LD;
    float* sA = sT + CH * LC;
    __shared__ GateVecs gv;
    __shared__ float tmp[32 * 32];

    const int c = blockIdx.x, h = blockIdx.y, H = a.H;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const int grp = threadIdx.x >> 8;
    const Lane l{(int)(threadIdx.x & 255) >> 4, (int)threadIdx.x & 15};

    load_tile<T, K, CL_NT>(sK, LD, static_cast<const T*>(a.k), tok0, len, H, h);
    load_tile<float, K, CL_NT>(sKt, LD, a.ktil, tok0, len, H, h);
    load_tile<T, K, CL_NT>(sQ, LD, static_cast<const T*>(a.q), tok0, len, H, h);
    load_gates(gv, a.gate, a.beta, tok0, len, H, h);
    __syncthreads();
    if (threadIdx.x < 2 * CH) a.gvec[tile * 2 * CH + threadIdx.x] = threadIdx.x < CH ? gv.rho[threadIdx.x] : gv.gam[threadIdx.x - CH];

    // A_ij = 1[j<i] beta_i Gamma_ij <k_i, ktil_j>   and   P_ij = 1[j<=i] Gamma_ij <q_i, ktil_j>
    {
        float acc[4][4];
        zero(acc);
        const float* X = grp == 0 ? sK : sQ;
        tile_mm<false, true, 4>(acc, 0, K, l, [&](int m, int k) { return ld4(X + m * LD + k); },
                                [&](int n, int k) { return ld4(sKt + n * LD + k); });
        float* Pg = a.P + tile * CH * CH;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = row_of(l, i), n = col_of<true>(l, j);
                const float g = n <= m ? expf(gv.G[m] - gv.G[n]) * acc[i][j] : 0.f;
                if (grp == 0) sA[m * LC + n] = n < m ? gv.beta[m] * g : 0.f;
                else Pg[m * CH + n] = g;
            }
    }
    __syncthreads();
    ut_inverse_64(sA, sT, tmp);
    float* Tg = a.Tm + tile * CH * CH;
    for (int e = threadIdx.x; e < CH * CH / 4; e += CL_NT) st4(Tg + e * 4, ld4(sT + (e / 16) * LC + (e % 16) * 4));

    // W = T diag(beta gamma) K ; U = T diag(beta) V.  T is lower triangular: rows of a warp end at 8 w + 8.
    const int jend = (l.tm & ~1) * 4 + 8;
    if (grp == 0) {
        float acc[4][TK];
        zero(acc);
        tile_mm<false, false, TK>(acc, 0, jend, l, [&](int m, int j) { return ld4(sT + m * LC + j); },
                                  [&](int j, int n) { return (gv.beta[j] * gv.gam[j]) * ld4(sK + j * LD + n); });
        float* Wg = a.W + tile * CH * K;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TK; cc += 4)
                st4(Wg + row_of(l, i) * K + col_of<false>(l, cc), make_float4(acc[i][cc], acc[i][cc + 1], acc[i][cc + 2], acc[i][cc + 3]));
    } else {
        float acc[4][TV];
        zero(acc);
        const Rows<T, V> v = rows_of<T, V>(a.v, tok0, len, H, h);
        tile_mm<false, false, TV>(acc, 0, jend, l, [&](int m, int j) { return ld4(sT + m * LC + j); },
                                  [&](int j, int n) { return gv.beta[j] * v(j, n); });
        float* Ug = a.U + tile * CH * V;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TV; cc += 4)
                st4(Ug + row_of(l, i) * V + col_of<false>(l, cc), make_float4(acc[i][cc], acc[i][cc + 1], acc[i][cc + 2], acc[i][cc + 3]));
    }
}

// ---------------------------------------------------------------------------------------
// O = scale [ (gamma Q) S_n^T + P dU ], one tile per CTA once the chain has left S_n and dU: the output is
// off the sequential path.
// ---------------------------------------------------------------------------------------
template <typename T, int K, int V>
__global__ void __launch_bounds__(256) output_kernel(ChunkArgs a)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int TV = V / 16, LD = K + 4, NT = 256;
    float* sQ = sm;                  // [64][LD]
    float* sS = sQ + CH * LD;        // [V][LD], S_n; then dU [64][V]
    float* sP = sS + V * LD;         // [64][LC]
    const int c = blockIdx.x, h = blockIdx.y, H = a.H;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const Lane l{(int)threadIdx.x >> 4, (int)threadIdx.x & 15};
    const float* S = a.Sn + tile * V * K;
    const float* P = a.P + tile * CH * CH;
    const float* dU = a.dU + tile * CH * V;
    load_tile<T, K, NT>(sQ, LD, static_cast<const T*>(a.q), tok0, len, H, h);
#pragma unroll 8
    for (int e = threadIdx.x; e < V * K / 4; e += NT) st4(sS + e / (K / 4) * LD + e % (K / 4) * 4, ld4(S + e * 4));
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * CH / 4; e += NT) st4(sP + e / 16 * LC + e % 16 * 4, ld4(P + e * 4));
    float4 u[CH * V / 4 / NT];
#pragma unroll
    for (int x = 0; x < CH * V / 4 / NT; ++x) u[x] = ld4(dU + (threadIdx.x + x * NT) * 4);
    __syncthreads();
    float acc[4][TV];
    zero(acc);
    tile_mm<false, true, TV>(acc, 0, K, l, [&](int m, int k) { return ld4(sQ + m * LD + k); }, [&](int n, int k) { return ld4(sS + n * LD + k); });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float g = a.gvec[tile * 2 * CH + CH + row_of(l, i)];
#pragma unroll
        for (int j = 0; j < TV; ++j) acc[i][j] *= g;
    }
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

// ---------------------------------------------------------------------------------------
// State chain.  One CTA of eight warps per (chain, slice of VS = 8 state rows); only what the recurrence
// needs runs here:
//   forward   dU = U - W S^T ;                          S  <- gamma_C S + dU^T (rho Ktil)
//   backward  ddU = ddU0 + (rho Ktil) dS^T ;            dS <- gamma_C dS + scale dO^T (gamma Q) - ddU^T W
// (O and ddU0 = scale P^T dO are tile-parallel passes of their own.)  A step is two products of a 64-row
// operand with the slice, bound by latency: the warps split the contraction, every lane holds a 4 x 4
// tile, the partial sums meet in shared memory.  The next chunk's operands arrive by cp.async meanwhile.
// Narrow slices because the work is a chain of dependent steps: 32 rows and one pass over all rows per
// thread took 16 us a chunk, 8 rows split this way take under 1 us.
// ---------------------------------------------------------------------------------------
struct ChainArgs {
    int S, H;
    Table tab;
    const void* q;
    const float *ktil, *W, *U, *gvec, *init_state;
    float *final_state, *Sn, *dU;
    // backward
    const void* dout;
    const float* dfinal_state;
    float *ddU, *dSn, *dinit_state;
    Hyper hy;
};
constexpr int VS = 8, CNT = 256;

__device__ __forceinline__ void cpa16(void* dst, const void* src, bool in)
{
    const int n = in ? 16 : 0;   // 0: the destination is filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 64 rows of D elements into rows of LD elements; row i at src + i * stride, rows >= len zero
template <typename T, int D, int LD>
__device__ __forceinline__ void cpa_rows(T* dst, const T* src, size_t stride, int len)
{
    constexpr int PER = D * sizeof(T) / 16, EL = 16 / sizeof(T);
    for (int e = threadIdx.x; e < CH * PER; e += CNT) {
        const int i = e / PER, c = e % PER * EL;
        cpa16(dst + i * LD + c, src + (size_t)(i < len ? i : 0) * stride + c, i < len);
    }
}

// part[i][v] += sum over this warp's k of X[i][k] s_i Y[v][k]   (rows i = li + 16 ii, v = 4 lv + vv)
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
// acc[c][v][kk] += sum over this warp's tokens of D[i][v] X[i][k]   (v = 4 lv + vv, k = 64 c + 4 li + kk).  A warp
// takes 64 columns and a share of the tokens, so that the partial sums of K = 128 take no more room than those of 64.
template <typename T, int K, int LD>
__device__ __forceinline__ void slice_outer(float (&acc)[4][4], const T* X, const float* D, int i0, int ni, int k)
{
#pragma unroll 8
    for (int i = i0; i < i0 + ni; ++i) {
        const float4 x = ld4(X + i * LD + k), d = ld4(D + i * VS);
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) acc[v][kk] = fmaf(comp(d, v), comp(x, kk), acc[v][kk]);
    }
}

template <int K> struct ChainShared {
    static constexpr int LD = K + 4, CW = K / 64, GROUPS = 8 / CW;   // column halves, token groups
    float S[VS * LD];
    float part[8 * CH * VS];     // dot: [8][64][VS]; outer: [GROUPS][VS][K] (the same size)
    float D[CH * VS];            // rho dU, or ddU negated
};
template <int K> struct FwdStage {
    float W[CH * (K + 4)], Kt[CH * (K + 4)], U[CH * VS], rho[CH], gam[CH];
};
template <typename T, int K> struct BwdStage {
    float W[CH * (K + 4)], Kt[CH * (K + 4)], rho[CH], gam[CH];
    T Q[CH * (K + 4 * (4 / sizeof(T)))];
    T dO[CH * VS];
};

// sum of the dot product's partial tiles for the outputs 2 t, 2 t + 1 of [64][VS]
__device__ __forceinline__ float2 sum_dot(const float* part)
{
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const float2 p = *reinterpret_cast<const float2*>(part + w * CH * VS + threadIdx.x * 2);
        s.x += p.x;
        s.y += p.y;
    }
    return s;
}
// S <- gC S + partial tiles of the outer product
template <int K> __device__ __forceinline__ void advance_state(ChainShared<K>& s, float gC)
{
    constexpr int LD = K + 4, G = ChainShared<K>::GROUPS;
#pragma unroll
    for (int e = threadIdx.x * 2; e < VS * K; e += CNT * 2) {
        const int v = e / K, k = e % K;
        float2 t = make_float2(0.f, 0.f);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float2 p = *reinterpret_cast<const float2*>(s.part + g * VS * K + e);
            t.x += p.x;
            t.y += p.y;
        }
        float2* S = reinterpret_cast<float2*>(s.S + v * LD + k);
        const float2 o = *S;
        *S = make_float2(fmaf(gC, o.x, t.x), fmaf(gC, o.y, t.y));
    }
}
template <int K> __device__ __forceinline__ void load_state(ChainShared<K>& s, const float* src)
{
    for (int e = threadIdx.x; e < VS * K; e += CNT) s.S[(e / K) * (K + 4) + e % K] = src ? src[e] : 0.f;
}
template <int K> __device__ __forceinline__ void store_state(const ChainShared<K>& s, float* dst)
{
    for (int e = threadIdx.x * 4; e < VS * K; e += CNT * 4) st4(dst + e, ld4(s.S + (e / K) * (K + 4) + e % K));
}

template <int K, int V>
__global__ void __launch_bounds__(CNT) chain_fwd_kernel(ChainArgs a)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int LD = K + 4, CW = ChainShared<K>::CW, NI = CH / ChainShared<K>::GROUPS;
    ChainShared<K>& s = *reinterpret_cast<ChainShared<K>*>(sm);
    FwdStage<K>* stage = reinterpret_cast<FwdStage<K>*>(sm + sizeof(ChainShared<K>) / 4);
    const int chain = blockIdx.x, H = a.H;
    const int sq = chain / H, h = chain % H, v0 = blockIdx.y * VS;
    const int c0 = a.tab.seq_chunk0(sq), c1 = a.tab.seq_chunk0(sq + 1);
    const int seq_t0 = a.tab.seq_tok0(sq), seq_len = a.tab.seq_len(sq);
    const int t = threadIdx.x, warp = t >> 5, li = t & 15, lv = (t >> 4) & 1;
    const size_t srow = (((size_t)sq * H + h) * V + v0) * K;

    auto fetch = [&](int c) {
        if (c < c1) {
            FwdStage<K>& g = stage[(c - c0) & 1];
            const size_t tile = (size_t)c * H + h;
            const int n0 = (c - c0) * CH;
            cpa_rows<float, K, LD>(g.W, a.W + tile * CH * K, K, CH);
            cpa_rows<float, K, LD>(g.Kt, a.ktil + ((size_t)(seq_t0 + n0) * H + h) * K, (size_t)H * K, seq_len - n0);
            cpa_rows<float, VS, VS>(g.U, a.U + tile * CH * V + v0, V, CH);
            if (t < 32) cpa16(g.rho + t * 4, a.gvec + tile * 2 * CH + t * 4, true);   // rho, then gamma
        }
        cpa_commit();
    };
    load_state<K>(s, a.init_state ? a.init_state + srow : nullptr);
    fetch(c0);
    for (int c = c0; c < c1; ++c) {
        const size_t tile = (size_t)c * H + h;
        fetch(c + 1);
        cpa_wait<1>();
        __syncthreads();   // the chunk has landed, S is complete
        const FwdStage<K>& g = stage[(c - c0) & 1];
        {
            float acc[4][4];
            zero(acc);
            slice_dot<K, LD>(acc, g.W, s.S, warp, li, lv);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                st4(s.part + (warp * CH + li + 16 * i) * VS + lv * 4, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
        }
        store_state<K>(s, a.Sn + (tile * V + v0) * K);
        __syncthreads();
        {
            const float2 d = sum_dot(s.part), u = *reinterpret_cast<const float2*>(g.U + t * 2);
            const int i = t / (VS / 2), v = t % (VS / 2) * 2;
            const float2 du = make_float2(u.x - d.x, u.y - d.y);
            *reinterpret_cast<float2*>(a.dU + tile * CH * V + (size_t)i * V + v0 + v) = du;
            const float r = g.rho[i];
            *reinterpret_cast<float2*>(s.D + t * 2) = make_float2(r * du.x, r * du.y);
        }
        __syncthreads();
        {
            float acc[4][4];
            zero(acc);
            const int half = warp % CW, grp = warp / CW, k = half * 64 + li * 4;
            slice_outer<float, K, LD>(acc, g.Kt, s.D + lv * 4, grp * NI, NI, k);
#pragma unroll
            for (int v = 0; v < 4; ++v)
                st4(s.part + (grp * VS + lv * 4 + v) * K + k, make_float4(acc[v][0], acc[v][1], acc[v][2], acc[v][3]));
        }
        __syncthreads();
        advance_state<K>(s, g.gam[CH - 1]);
        __syncthreads();   // nobody reads the stage any more: it may be filled again
    }
    if (a.final_state) {
        __syncthreads();
        store_state<K>(s, a.final_state + srow);
    }
}

template <typename T, int K, int V>
__global__ void __launch_bounds__(CNT) chain_bwd_kernel(ChainArgs a)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int LD = K + 4, LQ = K + 4 * (4 / sizeof(T)), CW = ChainShared<K>::CW, NI = CH / ChainShared<K>::GROUPS;
    ChainShared<K>& s = *reinterpret_cast<ChainShared<K>*>(sm);
    BwdStage<T, K>* stage = reinterpret_cast<BwdStage<T, K>*>(sm + sizeof(ChainShared<K>) / 4);
    __shared__ __align__(16) float sE[sizeof(T) == 4 ? 4 : CH * VS];   // scale gamma_i dO (fp32: in place of dO)
    const int chain = blockIdx.x, H = a.H;
    const int sq = chain / H, h = chain % H, v0 = blockIdx.y * VS;
    const int c0 = a.tab.seq_chunk0(sq), c1 = a.tab.seq_chunk0(sq + 1);
    const int seq_t0 = a.tab.seq_tok0(sq), seq_len = a.tab.seq_len(sq);
    const int t = threadIdx.x, warp = t >> 5, li = t & 15, lv = (t >> 4) & 1;
    const size_t srow = (((size_t)sq * H + h) * V + v0) * K;
    const int oi = t / (VS / 2), ov = t % (VS / 2) * 2;   // the two outputs of the summing passes

    auto fetch = [&](int c) {
        if (c >= c0) {
            BwdStage<T, K>& g = stage[(c - c0) & 1];
            const size_t tile = (size_t)c * H + h;
            const int n0 = (c - c0) * CH, len = seq_len - n0;
            const size_t tok = (size_t)(seq_t0 + n0) * H + h;
            cpa_rows<float, K, LD>(g.W, a.W + tile * CH * K, K, CH);
            cpa_rows<float, K, LD>(g.Kt, a.ktil + tok * K, (size_t)H * K, len);
            cpa_rows<T, K, LQ>(g.Q, static_cast<const T*>(a.q) + tok * K, (size_t)H * K, len);
            cpa_rows<T, VS, VS>(g.dO, static_cast<const T*>(a.dout) + tok * V + v0, (size_t)H * V, len);
            if (t < 32) cpa16(g.rho + t * 4, a.gvec + tile * 2 * CH + t * 4, true);
        }
        cpa_commit();
    };
    auto ddu0_of = [&](int c) {   // ddU0, left in the ddU region by the pass before, a chunk ahead
        return c >= c0 ? *reinterpret_cast<const float2*>(a.ddU + ((size_t)c * H + h) * CH * V + (size_t)oi * V + v0 + ov) : make_float2(0.f, 0.f);
    };
    load_state<K>(s, a.dfinal_state ? a.dfinal_state + srow : nullptr);
    fetch(c1 - 1);
    float2 ddu0 = ddu0_of(c1 - 1);
    for (int c = c1 - 1; c >= c0; --c) {
        const size_t tile = (size_t)c * H + h;
        fetch(c - 1);
        cpa_wait<1>();
        __syncthreads();
        BwdStage<T, K>& g = stage[(c - c0) & 1];
        float* E = sizeof(T) == 4 ? reinterpret_cast<float*>(g.dO) : sE;
        {
            float acc[4][4];
            zero(acc);
            slice_dot<K, LD>(acc, g.Kt, s.S, warp, li, lv);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                st4(s.part + (warp * CH + li + 16 * i) * VS + lv * 4, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
        }
        store_state<K>(s, a.dSn + (tile * V + v0) * K);
        {
            const float f = a.hy.scale * g.gam[oi];
            *reinterpret_cast<float2*>(E + t * 2) = make_float2(f * ldf(g.dO + t * 2), f * ldf(g.dO + t * 2 + 1));
        }
        __syncthreads();
        {
            const float2 d = sum_dot(s.part);
            const float r = g.rho[oi];
            const float2 x = make_float2(fmaf(r, d.x, ddu0.x), fmaf(r, d.y, ddu0.y));
            *reinterpret_cast<float2*>(a.ddU + tile * CH * V + (size_t)oi * V + v0 + ov) = x;
            *reinterpret_cast<float2*>(s.D + t * 2) = make_float2(-x.x, -x.y);
            ddu0 = ddu0_of(c - 1);
        }
        __syncthreads();
        {
            float acc[4][4];
            zero(acc);
            const int half = warp % CW, grp = warp / CW, k = half * 64 + li * 4;
            slice_outer<T, K, LQ>(acc, g.Q, E + lv * 4, grp * NI, NI, k);
            slice_outer<float, K, LD>(acc, g.W, s.D + lv * 4, grp * NI, NI, k);
#pragma unroll
            for (int v = 0; v < 4; ++v)
                st4(s.part + (grp * VS + lv * 4 + v) * K + k, make_float4(acc[v][0], acc[v][1], acc[v][2], acc[v][3]));
        }
        __syncthreads();
        advance_state<K>(s, g.gam[CH - 1]);
        __syncthreads();
    }
    if (a.dinit_state) {
        __syncthreads();
        store_state<K>(s, a.dinit_state + srow);
    }
}

// ddU0 = scale P^T dO: what the reverse chain's step does not need the state cotangent for, tile-parallel.
template <typename T, int V>
__global__ void __launch_bounds__(256) ddu0_kernel(ChunkArgs a)
{
    constexpr int TV = V / 16;
    const int c = blockIdx.x, h = blockIdx.y, H = a.H;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const Lane l{(int)threadIdx.x >> 4, (int)threadIdx.x & 15};
    __shared__ __align__(16) float sP[CH * CH];
    extern __shared__ __align__(16) float sO[];   // [64][V]
    const float* P = a.P + tile * CH * CH;
#pragma unroll
    for (int e = threadIdx.x; e < CH * CH / 4; e += 256) st4(sP + e * 4, ld4(P + e * 4));
    load_tile<T, V, 256>(sO, V, static_cast<const T*>(a.dout), tok0, len, H, h);
    __syncthreads();
    float acc[4][TV];
    zero(acc);
    // P is lower triangular: row i of P^T starts at column i
    tile_mm<true, false, TV>(acc, (l.tm & ~1) * 4, CH, l, [&](int j, int m) { return ld4(sP + j * CH + m); },
                             [&](int j, int n) { return ld4(sO + j * V + n); });
    float* o = a.ddU + tile * CH * V;
    const float s = a.hy.scale;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int cc = 0; cc < TV; cc += 4)
            st4(o + row_of(l, i) * V + col_of<false>(l, cc), s * make_float4(acc[i][cc], acc[i][cc + 1], acc[i][cc + 2], acc[i][cc + 3]));
}

// ---------------------------------------------------------------------------------------
// chunk-local backward: gradients through P, the state-advance factors, W, U, T, A, gates.
//
// Fifteen products per tile, six phases; in each the two groups of 256 threads form different products.
// Bound by the FMAs.  k, ktil, q, T and the 64 x 64 intermediates sit in shared memory; S, dS, dU, ddU, v and
// dO are read where they are (a tile of each fits the first-level cache).  With thread tiles fed by scalar
// shared-memory reads and one shared-memory atomic per element of the row sums the kernel took 412 us for 256
// tiles of K = V = 64.  The gate gradient needs no sums of its own over the score matrices: with
// E_i = <dq_i, q_i> + <dk_read_i, k_i> - <dktil_i, ktil_i> (phase-2 gradients),
//   dG_i = E_i + 1[i = last] (sum_j rho_j <(dU dS)_j, ktil_j> + gamma_C <dS, S>).
// ---------------------------------------------------------------------------------------
template <typename T, int K, int V>
__global__ void __launch_bounds__(CL_NT) chunk_local_bwd_kernel(ChunkArgs a)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int LD = K + 4, TK = K / 16, TV = V / 16;
    float* sK = sm;
    float* sKt = sK + CH * LD;
    float* sQ = sKt + CH * LD;
    float* sW = sQ + CH * LD;       // dW
    float* sT = sW + CH * LD;       // [64][LC]
    float* sX = sT + CH * LC;       // dT, the raw Gram, then dA * beta_i * Gamma_ij
    float* sY = sX + CH * LC;       // T^T dT
    float* sDP = sY + CH * LC;      // dP * Gamma
    __shared__ GateVecs gv;
    __shared__ float sB[3][CH], sE[3][CH], sR[CH], sRed[CL_NT / 32];

    const int c = blockIdx.x, h = blockIdx.y, H = a.H;
    const int len = a.tab.chunk_len(c);
    if (len == 0) return;
    const int tok0 = a.tab.chunk_tok0(c);
    const size_t tile = (size_t)c * H + h;
    const float scale = a.hy.scale;
    const int grp = threadIdx.x >> 8;
    const Lane l{(int)(threadIdx.x & 255) >> 4, (int)threadIdx.x & 15};
    const int m_hi = (l.tm & ~1) * 4 + 8, m_lo = m_hi - 8;   // rows of this warp: [m_lo, m_hi)

    const Rows<T, V> vr = rows_of<T, V>(a.v, tok0, len, H, h), dor = rows_of<T, V>(a.dout, tok0, len, H, h);
    const float* Sg = a.Sn + tile * V * K;
    const float* dSg = a.dSn + tile * V * K;
    const float* dUg = a.dU + tile * CH * V;
    const float* ddUg = a.ddU + tile * CH * V;

    load_tile<T, K, CL_NT>(sK, LD, static_cast<const T*>(a.k), tok0, len, H, h);
    load_tile<float, K, CL_NT>(sKt, LD, a.ktil, tok0, len, H, h);
    load_tile<T, K, CL_NT>(sQ, LD, static_cast<const T*>(a.q), tok0, len, H, h);
    for (int e = threadIdx.x; e < CH * CH / 4; e += CL_NT) st4(sT + (e / 16) * LC + (e % 16) * 4, ld4(a.Tm + tile * CH * CH + e * 4));
    // dU, then v, are read by rows that differ between lanes: staged in the place of X and Y until those are written
    constexpr int LU = V + 4;
    float* sU = sX;
#pragma unroll 4
    for (int e = threadIdx.x; e < CH * V / 4; e += CL_NT) st4(sU + e / (V / 4) * LU + e % (V / 4) * 4, ld4(dUg + e * 4));
    if (V == 64) load_tile<T, V, CL_NT>(sY, LU, static_cast<const T*>(a.v), tok0, len, H, h);
    load_gates(gv, a.gate, a.beta, tok0, len, H, h);
    {   // <dS, S>_F (for the gradient of the chunk-level decay gamma_C)
        float part = 0.f;
        for (int e = threadIdx.x * 4; e < V * K; e += CL_NT * 4) {
            const float4 x = ld4(Sg + e), y = ld4(dSg + e);
            part += x.x * y.x + x.y * y.y + (x.z * y.z + x.w * y.w);
        }
        part = warp_sum(part);
        if ((threadIdx.x & 31) == 0) sRed[threadIdx.x >> 5] = part;
    }
    __syncthreads();

    // (1) dP * Gamma = 1[j<=i] Gamma_ij scale dO dU^T      |  dW = -ddU S
    if (grp == 0) {
        float acc[4][4];
        zero(acc);
        tile_mm<false, true, 4>(acc, 0, V, l, [&](int m, int k) { return dor(m, k); }, [&](int n, int k) { return ld4(sU + n * LU + k); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int m = row_of(l, i), n = col_of<true>(l, j);
                sDP[m * LC + n] = n <= m ? scale * acc[i][j] * expf(gv.G[m] - gv.G[n]) : 0.f;
            }
    } else {
        float acc[4][TK];
        zero(acc);
        tile_mm<false, false, TK>(acc, 0, V, l, [&](int m, int k) { return ld4(ddUg + m * V + k); }, [&](int k, int n) { return ld4(Sg + k * K + n); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int cc = 0; cc < TK; cc += 4)
                st4(sW + row_of(l, i) * LD + col_of<false>(l, cc), -1.f * make_float4(acc[i][cc], acc[i][cc + 1], acc[i][cc + 2], acc[i][cc + 3]));
    }
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
                    st4(base + ((size_t)(tok0 + row_of(l, i)) * H + h) * D + col_of<false>(l, cc),
                        make_float4(acc[i][cc], acc[i][cc + 1], acc[i][cc + 2], acc[i][cc + 3]));
    };

    // (2) dq = gamma_i scale dO S + (dP Gamma) Ktil         |  dT = dW (beta gamma K)^T + ddU (beta V)^T
    if (grp == 0) {
        float acc[4][TK];
        zero(acc);
        tile_mm<false, false, TK>(acc, 0, V, l, [&](int m, int k) { return dor(m, k); }, [&](int k, int n) { return ld4(Sg + k * K + n); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TK; ++j) acc[i][j] *= scale * gv.gam[row_of(l, i)];
        tile_mm<false, false, TK>(acc, 0, m_hi, l, [&](int m, int k) { return ld4(sDP + m * LC + k); }, [&](int k, int n) { return ld4(sKt + k * LD + n); });
        store_rows(acc, static_cast<T*>(a.dq), K);
        row_dots(acc, [&](int m, int n) { return ld4(sQ + m * LD + n); }, sE[0]);
    } else {
        const float* sV = V == 64 ? sY : sX;
        if constexpr (V == 128) {   // no room for both before: v takes the place of dU now (this group alone)
            const int t = threadIdx.x & 255;
#pragma unroll 4
            for (int e = t; e < CH * V / 4; e += 256) st4(sX + e / (V / 4) * LU + e % (V / 4) * 4, vr(e / (V / 4), e % (V / 4) * 4));
            asm volatile("bar.sync 1, 256;" ::: "memory");
        }
        float acc[4][4];
        zero(acc);
        tile_mm<false, true, 4>(acc, 0, K, l, [&](int m, int k) { return ld4(sW + m * LD + k); }, [&](int n, int k) { return ld4(sK + n * LD + k); });
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i][j] *= gv.gam[col_of<true>(l, j)];
        tile_mm<false, true, 4>(acc, 0, V, l, [&](int m, int k) { return ld4(ddUg + m * V + k); }, [&](int n, int k) { return ld4(sV + n * LU + k); });
        if constexpr (V == 128) asm volatile("bar.sync 1, 256;" ::: "memory");   // v has been read
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sX[row_of(l, i) * LC + col_of<true>(l, j)] = gv.beta[col_of<true>(l, j)] * acc[i][j];
    }
    __syncthreads();

    // (3) dKb = T^T dW, dVb = T^T ddU (kept by group 0: dk grows from dKb)   |  T^T dT ; rho_j dU dS (kept by group 1)
    float keep[4][TK];   // group 0: dk of the read key; group 1: d ktil
    zero(keep);
    if (grp == 0) {
        tile_mm<true, false, TK>(keep, m_lo, CH, l, [&](int k, int m) { return ld4(sT + k * LC + m); }, [&](int k, int n) { return ld4(sW + k * LD + n); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TK; ++j) keep[i][j] *= gv.gam[row_of(l, i)];
        row_dots(keep, [&](int m, int n) { return ld4(sK + m * LD + n); }, sB[0]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TK; ++j) keep[i][j] *= gv.beta[row_of(l, i)];
        float acc[4][TV];
        zero(acc);
        tile_mm<true, false, TV>(acc, m_lo, CH, l, [&](int k, int m) { return ld4(sT + k * LC + m); }, [&](int k, int n) { return ld4(ddUg + k * V + n); });
        row_dots(acc, [&](int m, int n) { return vr(m, n); }, sB[1]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TV; ++j) acc[i][j] *= gv.beta[row_of(l, i)];
        store_rows(acc, static_cast<T*>(a.dv), V);
    } else {
        float acc[4][4];
        zero(acc);
        tile_mm<true, false, 4>(acc, m_lo, CH, l, [&](int k, int m) { return ld4(sT + k * LC + m); }, [&](int k, int n) { return ld4(sX + k * LC + n); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
            st4(sY + row_of(l, i) * LC + col_of<false>(l, 0), make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
        tile_mm<false, false, TK>(keep, 0, V, l, [&](int m, int k) { return ld4(dUg + m * V + k); }, [&](int k, int n) { return ld4(dSg + k * K + n); });
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TK; ++j) keep[i][j] *= gv.rho[row_of(l, i)];
        row_dots(keep, [&](int m, int n) { return ld4(sKt + m * LD + n); }, sR);
    }
    __syncthreads();

    // (4) dA = -strictLower(T^T dT T^T)                      |  the raw Gram once more: dbeta_i += dA_ij Gamma_ij <k_i, ktil_j>
    {
        float acc[4][4];
        zero(acc);
        if (grp == 0) {   // column n of T^T ends at n
            tile_mm<false, true, 4>(acc, 0, CH, l, [&](int m, int k) { return ld4(sY + m * LC + k); }, [&](int n, int k) { return ld4(sT + n * LC + k); });
        } else {
            tile_mm<false, true, 4>(acc, 0, K, l, [&](int m, int k) { return ld4(sK + m * LD + k); }, [&](int n, int k) { return ld4(sKt + n * LD + k); });
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) sX[row_of(l, i) * LC + col_of<true>(l, j)] = acc[i][j];
        }
        __syncthreads();
        if (grp == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int m = row_of(l, i);
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int n = col_of<true>(l, j);
                    const float da = n < m ? -acc[i][j] * expf(gv.G[m] - gv.G[n]) : 0.f;
                    float* x = sX + m * LC + n;
                    s = fmaf(da, *x, s);
                    *x = da * gv.beta[m];
                }
                s = half_sum(s);
                if (l.tn == 0) sB[2][m] = s;
            }
        }
    }
    __syncthreads();

    // (5) dk (read side) = beta gamma dKb + X Ktil           |  dktil = rho dU dS + (dP Gamma)^T Q + X^T K
    if (grp == 0) {
        tile_mm<false, false, TK>(keep, 0, m_hi, l, [&](int m, int k) { return ld4(sX + m * LC + k); }, [&](int k, int n) { return ld4(sKt + k * LD + n); });
        store_rows(keep, a.dkread, K);
        row_dots(keep, [&](int m, int n) { return ld4(sK + m * LD + n); }, sE[1]);
    } else {
        tile_mm<true, false, TK>(keep, m_lo, CH, l, [&](int k, int m) { return ld4(sDP + k * LC + m); }, [&](int k, int n) { return ld4(sQ + k * LD + n); });
        tile_mm<true, false, TK>(keep, m_lo, CH, l, [&](int k, int m) { return ld4(sX + k * LC + m); }, [&](int k, int n) { return ld4(sK + k * LD + n); });
        store_rows(keep, a.dktil, K);
        row_dots(keep, [&](int m, int n) { return ld4(sKt + m * LD + n); }, sE[2]);
    }
    __syncthreads();

    // (6) gate gradients: reverse in-chunk prefix of dG (one warp, lane l holds tokens l and l + 32); dbeta
    if (threadIdx.x < 32) {
        const int i = threadIdx.x;
        float x = sE[0][i] + sE[1][i] - sE[2][i], y = sE[0][i + 32] + sE[1][i + 32] - sE[2][i + 32];
        const float rsum = warp_sum(sR[i] + sR[i + 32]);
        const float tot = warp_sum(i < CL_NT / 32 ? sRed[i] : 0.f);
        if (i == 31) y += rsum + gv.gam[CH - 1] * tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ux = __shfl_down_sync(0xffffffffu, x, o), uy = __shfl_down_sync(0xffffffffu, y, o);
            if (i + o < 32) { x += ux; y += uy; }
        }
        x += __shfl_sync(0xffffffffu, y, 0);
        const size_t th = (size_t)(tok0 + i) * H + h;
        if (i < len) a.dgate[th] = x;
        if (i + 32 < len) a.dgate[th + (size_t)32 * H] = y;
    } else if (threadIdx.x >= 64 && threadIdx.x < 64 + CH) {
        const int i = threadIdx.x - 64;
        if (i < len) a.dbeta[(size_t)(tok0 + i) * H + h] = sB[0][i] + sB[1][i] + sB[2][i];
    }
}

template <typename F> bool set_smem(F* kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

template <typename T, int K, int V>
int fwd_impl(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
             bool save, cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    Table tab = carve_table(ws, L);
    int launches = 0;
    const int S = L.S, H = p.H;
    {
        const int n1 = phase1_forward(p, hy, L, ws, a, w + L.ktil, false, save, st);
        if (n1 < 0) return -1;
        launches += n1;
    }
    auto F = [&](size_t off) { return reinterpret_cast<float*>(w + off); };
    ChunkArgs ca{};
    ca.H = H; ca.tab = tab; ca.q = a.q; ca.k = a.k; ca.v = a.v; ca.beta = a.beta; ca.gate = a.gate;
    ca.ktil = F(L.ktil); ca.Tm = F(L.Tm); ca.P = F(L.P); ca.W = F(L.W); ca.U = F(L.U); ca.gvec = F(L.gvec);
    ca.Sn = F(L.Sn); ca.dU = F(L.dU); ca.out = a.out; ca.hy = hy;
    {
        const size_t smem = sizeof(float) * (3 * CH * (K + 4) + 2 * CH * LC);
        if (!set_smem(chunk_local_fwd_kernel<T, K, V>, smem)) return -1;
        stage_mark(st, "simt_chunk_local_fwd");
        chunk_local_fwd_kernel<T, K, V><<<dim3(L.NTmax, H), CL_NT, smem, st>>>(ca);
        ++launches;
    }
    {
        ChainArgs ch{};
        ch.S = S; ch.H = H; ch.tab = tab; ch.ktil = F(L.ktil); ch.W = F(L.W); ch.U = F(L.U); ch.gvec = F(L.gvec);
        ch.init_state = a.init_state; ch.final_state = a.final_state; ch.Sn = F(L.Sn); ch.dU = F(L.dU); ch.hy = hy;
        const size_t smem = sizeof(ChainShared<K>) + 2 * sizeof(FwdStage<K>);
        if (!set_smem(chain_fwd_kernel<K, V>, smem)) return -1;
        stage_mark(st, "simt_chain_fwd");
        chain_fwd_kernel<K, V><<<dim3(S * H, V / VS), CNT, smem, st>>>(ch);
        ++launches;
    }
    const size_t smem_out = sizeof(float) * ((CH + V) * (K + 4) + CH * LC);
    if (!set_smem(output_kernel<T, K, V>, smem_out)) return -1;
    stage_mark(st, "simt_output");
    output_kernel<T, K, V><<<dim3(L.NTmax, H), 256, smem_out, st>>>(ca);
    ++launches;
    stage_end(st);
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

template <typename T, int K, int V>
int bwd_impl(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
             cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    Table tab = carve_table(ws, L);
    int launches = 0;
    const int S = L.S, H = p.H;
    auto F = [&](size_t off) { return reinterpret_cast<float*>(w + off); };
    ChunkArgs ca{};
    ca.H = H; ca.tab = tab; ca.q = a.q; ca.k = a.k; ca.v = a.v; ca.beta = a.beta; ca.gate = a.gate;
    ca.ktil = F(L.ktil); ca.Tm = F(L.Tm); ca.P = F(L.P);
    ca.dout = a.dout; ca.Sn = F(L.Sn); ca.dSn = F(L.dSn); ca.dU = F(L.dU); ca.ddU = F(L.ddU);
    ca.dktil = F(L.dktil); ca.dkread = F(L.dkread);
    ca.dq = a.dq; ca.dv = a.dv; ca.dbeta = a.dbeta; ca.dgate = a.dgate; ca.hy = hy;
    stage_mark(st, "simt_ddu0");
    ddu0_kernel<T, V><<<dim3(L.NTmax, H), 256, CH * V * sizeof(float), st>>>(ca);
    ++launches;
    {
        ChainArgs ch{};
        ch.S = S; ch.H = H; ch.tab = tab; ch.q = a.q; ch.ktil = F(L.ktil); ch.W = F(L.W); ch.gvec = F(L.gvec);
        ch.dout = a.dout; ch.dfinal_state = a.dfinal_state; ch.ddU = F(L.ddU); ch.dSn = F(L.dSn);
        ch.dinit_state = a.dinit_state; ch.hy = hy;
        const size_t smem = sizeof(ChainShared<K>) + 2 * sizeof(BwdStage<T, K>);
        if (!set_smem(chain_bwd_kernel<T, K, V>, smem)) return -1;
        stage_mark(st, "simt_chain_bwd");
        chain_bwd_kernel<T, K, V><<<dim3(S * H, V / VS), CNT, smem, st>>>(ch);
        ++launches;
    }
    {
        const size_t smem = sizeof(float) * (4 * CH * (K + 4) + 4 * CH * LC);
        if (!set_smem(chunk_local_bwd_kernel<T, K, V>, smem)) return -1;
        stage_mark(st, "simt_chunk_local_bwd");
        chunk_local_bwd_kernel<T, K, V><<<dim3(L.NTmax, H), CL_NT, smem, st>>>(ca);
        ++launches;
    }
    {
        const int n1 = phase1_backward(p, hy, L, ws, a, F(L.dktil), F(L.dkread), true, st);
        if (n1 < 0) return -1;
        launches += n1;
    }
    stage_end(st);
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

}  // namespace

int launch_build_table(const osdn_params& p, const WsLayout& L, void* ws, cudaStream_t st)
{
    Table tab = carve_table(ws, L);
    if (L.dense_T) return 0;   // dense batch: the table is arithmetic, nothing to build
    stage_mark(st, "build_table");
    build_table_kernel<<<1, TBL_THREADS, 0, st>>>(L.S, p.T, p.cu_seqlens, L.NTmax, tab,
                                                  reinterpret_cast<int*>(static_cast<char*>(ws) + L.status));
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

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

int simt_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                 bool save, cudaStream_t st)
{
    OSDN_DISPATCH(fwd_impl, p, hy, L, ws, a, save, st);
}

int simt_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                  cudaStream_t st)
{
    OSDN_DISPATCH(bwd_impl, p, hy, L, ws, a, st);
}

}  // namespace osdn
