// Recurrent (decode) step of the layer: the gate, the preconditioner update and the rank-1
// delta-rule write for a few tokens in one launch, on a state and a preconditioner that live in the
// caller's cache (the paper's "Single-token recurrence kernel for OSGDN", for q_len <= 64).
//
//   alpha_t = exp(g_t)
//   ktil_t  = d_t (.) k_t                               (write key from the PRE-update d)
//   d_{t+1} = clip(rho_t d_t + c_t k_t^2)                c_t = eta b_t (1 - b_t <d_t, k_t^2>) / max(|k_t|^2, eps)
//             (rho_t a scalar, or one retention per coordinate in the vector-retention mode)
//   S_t     = alpha_t S_{t-1} + beta_t (v_t - alpha_t S_{t-1} k_t) ktil_t^T ,   o_t = scale S_t q_t
//
// exactly the recurrence the chunk path evaluates chunk by chunk, so that a prefill with osdn_fwd
// followed by osdn_decode_step continues the same sequence.
//
// The work is bound by reading and writing the state once (V x K fp32 per chain).  Rows of S are independent; lane l of a
// warp owns the R = K / 32 consecutive columns R l .. R l + R - 1 of its rows (one vector access per row), the rows stay
// in registers over all tokens of the call, and every CTA repeats the preconditioner update for its own use.  Two shapes:
//   few chains     V / 16 CTAs of 4 warps x 4 rows per chain: a call of a few sequences is bound by latency and is spread
//                  over the chip.  They form one thread-block cluster: the preconditioner is updated in place, so the
//                  CTA that stores the advanced vector may do so only once every CTA of the chain has read the old one;
//                  a cluster barrier (releasing arrival after the read, acquiring wait before the store) gives exactly
//                  that order.
//   many chains    one CTA of 8 warps per chain (see launch_one): no cluster to schedule, the preconditioner
//                  update once per chain instead of eight times, a row's two sums share their shuffles with fifteen
//                  other rows'.
// Calls of several tokens stage the tokens' rows through shared memory, eight tokens at a time and one block ahead
// (fetched one token ahead, a token cost a trip to memory).
#include "osdn_common.cuh"

namespace osdn {

namespace {

constexpr int DEC_TB = 8;        // tokens of a staged block

struct DecArgs {
    int B, L, H;
    const void *q, *k, *v;
    const float *beta, *gate, *log_ret;
    float *state, *precond;
    void* out;
    Hyper hy;
};

// Two floats in one 64-bit register: the packed multiply and multiply-add issue once for both.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float x, float y)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpack2(F2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

__device__ __forceinline__ void dec_cp16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void dec_cp4(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

template <typename T, int K, int VB, bool VEC> struct alignas(16) DecBlock {
    T k[DEC_TB][K], q[DEC_TB][K], v[DEC_TB][VB];
    float beta[DEC_TB], gate[DEC_TB], lr[DEC_TB];
    alignas(16) float lrv[VEC ? DEC_TB : 1][VEC ? K : 1];
};

// RW rows per warp, WARPS warps per CTA.  VEC: vector retention (one log-retention per coordinate, log_ret [B,T,H,K]).
// MULTI: the call has several tokens per sequence.
template <typename T, int K, int V, bool VEC, int RW, int WARPS, bool MULTI> __device__ __forceinline__ void decode_body(const DecArgs& a)
{
    constexpr int R = K / 32, VB = RW * WARPS, SLICES = V / VB, NT = WARPS * 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chain = blockIdx.x / SLICES, slice = blockIdx.x % SLICES;
    const int b = chain / a.H, h = chain % a.H;
    const int vb0 = slice * VB, vw = warp * RW, row = lane % RW;   // the CTA's first row, the warp's first of these, this lane's
    const Hyper hy = a.hy;
    const T* qp = static_cast<const T*>(a.q);
    const T* kp = static_cast<const T*>(a.k);
    const T* vp = static_cast<const T*>(a.v);
    T* op = static_cast<T*>(a.out);
    auto th_of = [&](int t) { return ((size_t)b * a.L + t) * a.H + h; };

    float d[R];
    F2 S[RW][R / 2];
    float* srow = a.state + ((size_t)chain * V + vb0 + vw) * K;
    load_row<R>(a.precond + (size_t)chain * K, lane, d);
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        float x[R];
        load_row<R>(srow + (size_t)r * K, lane, x);
#pragma unroll
        for (int j = 0; j < R / 2; ++j) S[r][j] = pack2(x[2 * j], x[2 * j + 1]);
    }
    // v: of this lane's row; lrv: the log-retention vector (VEC)
    auto step = [&](int t, const float (&k1)[R], const float (&q1)[R], float v, float beta, float gate, float lr, const float (&lrv)[VEC ? R : 1]) {
        const float alpha = expf(gate);
        const float rho1 = hy.apf_mode == 0 ? 1.0f : (hy.apf_mode == 1 ? alpha : expf(lr));
        // preconditioner step
        float kap[R], ktil[R], sumk = 0.f, al = 0.f;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            kap[j] = k1[j] * k1[j];
            sumk += kap[j];
            al = fmaf(d[j], kap[j], al);
            ktil[j] = d[j] * k1[j];
        }
        sumk = warp_sum(sumk);
        al = warp_sum(al);
        const float n = fmaxf(sumk, hy.eps);
        const float bb = hy.beta_aware ? beta : 1.0f;
        const float c = hy.eta * bb * (1.0f - bb * al) / n;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            float rho = rho1;
            if constexpr (VEC) rho = expf(lrv[j]);
            float x = fmaf(c, kap[j], rho * d[j]);
            if (hy.clamp) x = fminf(fmaxf(x, hy.d_min), hy.d_max);
            d[j] = x;
        }
        // rank-1 write and read-out
        F2 k2[R / 2], q2[R / 2], t2[R / 2];
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            k2[j] = pack2(k1[2 * j], k1[2 * j + 1]);
            q2[j] = pack2(q1[2 * j], q1[2 * j + 1]);
            t2[j] = pack2(ktil[2 * j], ktil[2 * j + 1]);
        }
        auto dots = [&](const F2 (&x)[R / 2]) {   // lane l: row l % RW
            float p[RW];
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                F2 s = mul2(S[r][0], x[0]);
#pragma unroll
                for (int j = 1; j < R / 2; ++j) s = fma2(S[r][j], x[j], s);
                const float2 u = unpack2(s);
                p[r] = u.x + u.y;
            }
            return transpose_sum(p, lane);
        };
        const float rv = beta * (v - alpha * dots(k2));
        const F2 alpha2 = pack2(alpha, alpha);
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const float x = __shfl_sync(0xffffffffu, rv, r);
            const F2 x2 = pack2(x, x);
#pragma unroll
            for (int j = 0; j < R / 2; ++j) S[r][j] = fma2(alpha2, S[r][j], mul2(x2, t2[j]));
        }
        const float o = dots(q2);
        // The chain's preconditioner has been read (the sums above hold it): this slice's arrival releases that read to
        // the slice that overwrites it behind the wait.  The state rows have come back by now too and nothing has been stored yet.
        if constexpr (SLICES > 1)
            if (t == 0) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (lane < RW) stf(op + th_of(t) * V + vb0 + vw + lane, hy.scale * o);
    };

    if constexpr (!MULTI) {
        const size_t th = th_of(0);
        float k1[R], q1[R], lrv[VEC ? R : 1];
        load_row<R>(kp + th * K, lane, k1);
        load_row<R>(qp + th * K, lane, q1);
        if constexpr (VEC) load_row<R>(a.log_ret + th * K, lane, lrv);
        step(0, k1, q1, ldf(vp + th * V + vb0 + vw + row), a.beta[th], a.gate[th], hy.apf_mode == 2 ? a.log_ret[th] : 0.f, lrv);
    } else {
        __shared__ DecBlock<T, K, VB, VEC> blk[2];
        auto stage = [&](int t0) {
            DecBlock<T, K, VB, VEC>& B = blk[(t0 / DEC_TB) & 1];
            const int n = min(DEC_TB, a.L - t0);
            constexpr int PK = K * (int)sizeof(T) / 16, PV = VB * (int)sizeof(T) / 16, PL = VEC ? K / 4 : 0, PER = 2 * PK + PV + PL, EL = 16 / (int)sizeof(T);
            for (int e = threadIdx.x; e < n * PER; e += NT) {
                const int j = e / PER, p = e % PER;
                const size_t th = th_of(t0 + j);
                if (p < PK) dec_cp16(&B.k[j][p * EL], kp + th * K + p * EL);
                else if (p < 2 * PK) dec_cp16(&B.q[j][(p - PK) * EL], qp + th * K + (p - PK) * EL);
                else if (p < 2 * PK + PV) dec_cp16(&B.v[j][(p - 2 * PK) * EL], vp + th * V + vb0 + (p - 2 * PK) * EL);
                else dec_cp16(&B.lrv[VEC ? j : 0][VEC ? (p - 2 * PK - PV) * 4 : 0], a.log_ret + th * K + (p - 2 * PK - PV) * 4);
            }
            if ((int)threadIdx.x < n) {
                const size_t th = th_of(t0 + threadIdx.x);
                dec_cp4(&B.beta[threadIdx.x], a.beta + th);
                dec_cp4(&B.gate[threadIdx.x], a.gate + th);
                if (hy.apf_mode == 2) dec_cp4(&B.lr[threadIdx.x], a.log_ret + th);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        stage(0);
        for (int t0 = 0; t0 < a.L; t0 += DEC_TB) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();   // the block is there for everybody, and everybody is done with the one before
            if (t0 + DEC_TB < a.L) stage(t0 + DEC_TB);
            const DecBlock<T, K, VB, VEC>& B = blk[(t0 / DEC_TB) & 1];
            const int n = min(DEC_TB, a.L - t0);
            for (int j = 0; j < n; ++j) {
                float k1[R], q1[R], lrv[VEC ? R : 1];
                load_row<R>(B.k[j], lane, k1);
                load_row<R>(B.q[j], lane, q1);
                if constexpr (VEC) load_row<R>(B.lrv[VEC ? j : 0], lane, lrv);
                step(t0 + j, k1, q1, ldf(&B.v[j][vw + row]), B.beta[j], B.gate[j], hy.apf_mode == 2 ? B.lr[j] : 0.f, lrv);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        float x[R];
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            const float2 u = unpack2(S[r][j]);
            x[2 * j] = u.x;
            x[2 * j + 1] = u.y;
        }
        store_row<R>(srow + (size_t)r * K, lane, x);
    }
    // every warp (of every slice) of the chain has read the old preconditioner before it is overwritten
    if constexpr (SLICES > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
    if (slice == 0 && warp == 0) store_row<R>(a.precond + (size_t)chain * K, lane, d);
}

constexpr int FEW_RW = 4, FEW_WARPS = 4, MANY_WARPS = 8;

template <typename T, int K, int V, bool VEC, bool MULTI>
__global__ void __cluster_dims__(V / (FEW_RW * FEW_WARPS), 1, 1) __launch_bounds__(FEW_WARPS * 32) decode_few_kernel(DecArgs a)
{
    pdl_wait();
    decode_body<T, K, V, VEC, FEW_RW, FEW_WARPS, MULTI>(a);
}
template <typename T, int K, int V, bool VEC, bool MULTI>
__global__ void __launch_bounds__(MANY_WARPS * 32, 2) decode_many_kernel(DecArgs a)
{
    pdl_wait();
    decode_body<T, K, V, VEC, V / MANY_WARPS, MANY_WARPS, MULTI>(a);
}

// From about two chains to three SMs on a CTA per chain is the faster one: it has no slices to wait for one another.  Measured
// in a graph, K = V = 128, slices against a CTA per chain, us: one token 64 chains 2.65 / 3.02, 96 chains 3.02 / 3.10, 104
// chains 3.12 / 3.12, 112 chains 3.29 / 3.18, 144 chains 4.62 / 3.40; 7 tokens 64 chains 7.1 / 8.9, 104 chains 9.0 / 9.0, 112
// chains 12.5 / 9.0.  Slices for every call against these rules (plain launches): 4096 chains 106.5 -> 84.0 us, 1110 chains x 7
// tokens fp32 98 -> 52 us, 512 chains x 16 tokens 103 -> 52 us.
constexpr unsigned MANY_CHAINS = 104;
template <typename T, int K, int V, bool VEC> bool launch_one(unsigned chains, const DecArgs& a, cudaStream_t st)
{
    constexpr unsigned SLICES = V / (FEW_RW * FEW_WARPS);
    // Programmatic dependents: the launch of a call runs under the kernel before it in the stream, whose results it waits for
    // before its first access (one sequence, 8 chains, in a graph 2.28 -> 1.98 us, back to back from the host 4.1 -> 3.1; 4096
    // chains 83.9 -> 81.2 back to back).  No early release: the next call's CTAs would come in on the SMs that this one leaves
    // idle, several to an SM (K = V = 128, 104 chains x 16 tokens 16.7 -> 26.3 us, 64 chains, K = V = 64, 9.7 -> 16.5).
    if (chains >= MANY_CHAINS)
        return launch_after(a.L > 1 ? decode_many_kernel<T, K, V, VEC, true> : decode_many_kernel<T, K, V, VEC, false>, chains, MANY_WARPS * 32, 0, st, a);
    return launch_after(a.L > 1 ? decode_few_kernel<T, K, V, VEC, true> : decode_few_kernel<T, K, V, VEC, false>, chains * SLICES, FEW_WARPS * 32, 0, st, a);
}

template <typename T> int launch_typed(const osdn_params& p, const DecArgs& a, cudaStream_t st)
{
    const unsigned chains = (unsigned)p.B * (unsigned)p.H;
    bool ok;
    if (a.hy.apf_mode == 3) {
        if (p.K == 128 && p.V == 128) ok = launch_one<T, 128, 128, true>(chains, a, st);
        else if (p.K == 128 && p.V == 64) ok = launch_one<T, 128, 64, true>(chains, a, st);
        else if (p.K == 64 && p.V == 128) ok = launch_one<T, 64, 128, true>(chains, a, st);
        else ok = launch_one<T, 64, 64, true>(chains, a, st);
    } else {
        if (p.K == 128 && p.V == 128) ok = launch_one<T, 128, 128, false>(chains, a, st);
        else if (p.K == 128 && p.V == 64) ok = launch_one<T, 128, 64, false>(chains, a, st);
        else if (p.K == 64 && p.V == 128) ok = launch_one<T, 64, 128, false>(chains, a, st);
        else ok = launch_one<T, 64, 64, false>(chains, a, st);
    }
    return ok ? 1 : -1;
}

}  // namespace

int decode_step(const osdn_params& p, const Hyper& hy, const void* q, const void* k, const void* v,
                const float* beta, const float* gate, const float* log_ret, float* state, float* precond,
                void* out, cudaStream_t st)
{
    DecArgs a{};
    a.B = p.B; a.L = p.T; a.H = p.H;
    a.q = q; a.k = k; a.v = v; a.beta = beta; a.gate = gate; a.log_ret = log_ret;
    a.state = state; a.precond = precond; a.out = out; a.hy = hy;
    stage_mark(st, "decode_step");
    const int n = p.io_dtype == OSDN_FP32 ? launch_typed<float>(p, a, st) : launch_typed<__nv_bfloat16>(p, a, st);
    stage_end(st);
    return n;
}

}  // namespace osdn
