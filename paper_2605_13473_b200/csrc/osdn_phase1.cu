// Phase 1 of the layer: the online preconditioner sweep (Algorithm 1 with APF and the box
// projection) and its reverse sweep (Section 3.5), on CUDA cores in fp32.
//
// The sweep is a length-L sequential chain per (sequence, head).  Two observations keep it off
// the critical path without changing what is computed:
//
//  * Everything of a step that does not depend on d (k^2, its sum, the retention) is evaluated for
//    all tokens in parallel first (phase1_spec).
//  * Once every coordinate of d sits on the lower face of the box, the step for token t maps
//    d_min*1 to d_min*1 again iff every pre-projection value rho_t d_min + c_t k_t^2 is below d_min,
//    a condition that involves token t alone.  phase1_spec evaluates that step for every token
//    ("flag" bit), eight lanes per token; from the face the step has a closed form.  The sequential kernel
//    (phase1_seq) then only walks tokens where d is not on the face or the flag is clear; flagged
//    tokens entered on the face are skipped (their write key d_min*k was already emitted, their
//    projection mask is all zero).  On the benchmark distributions with the retention aliased to
//    the gate this removes almost every token from the chain; on inputs where d really moves it
//    degenerates to the plain sequential scan.
//
// For the backward pass the forward records, per processed token, d_t and the projection mask,
// and per chunk which tokens were skipped.  A skipped token has an all-zero mask, so the reverse
// recurrence restarts there: lambda_t = k_t (.) dL/dktil_t, dk_t = dk_read_t + d_min dL/dktil_t.
#include <type_traits>

#include "osdn_common.cuh"
#include "umma.cuh"

namespace osdn {

namespace {

// Asynchronous copies into shared memory; their completion is counted per committed group, first in first out.
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16_zfill(void* smem, const void* gmem, bool in)   // zeros where !in
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The coordinate the recurrence runs in, y = (d - lo) / w.  With c' = c / w a step is
//   y' = project(rho y + (c' k^2 + (rho - 1) lo / w)),   c' = e' - a2 <y, k^2>,   e' = (e - a2 lo sum k^2) / w.
//   P1_SAT    a box of ordinary width above zero: lo = d_min, w = d_max - d_min; the projection is the saturation of a
//             multiply-add.  d - d_min is at most d there, so that a rounding of y is none larger than one of d.
//   P1_PLAIN  everything else: no projection; a box that is open, without width, or of a width that 1 / w could not take
//             (w = 1); a negative lower edge, below which d - d_min would be larger than d and cost its last bits (lo = 0).
// Where lo = d_min the lower face is y = 0.  Core, finishing warps and the walk use the same functions, hence the same
// values.
enum P1Mode { P1_SAT, P1_PLAIN };
struct P1Coord {           // made by the host: in the kernels these are constants, not registers and a division
    float lo, w, iw, k0;   // k0 = lo / w
    P1Mode mode;
    bool face;             // y = 0 is the lower face, tokens may be skipped there
};
inline P1Coord p1_coord(const Hyper& hy)
{
    const bool face = hy.clamp && hy.d_min >= 0.f && hy.d_min <= 1e30f;
    const float width = hy.d_max - hy.d_min;
    const P1Mode mode = face && width >= 1e-12f && width <= 1e12f ? P1_SAT : P1_PLAIN;
    const float lo = face ? hy.d_min : 0.f, w = mode == P1_SAT ? width : 1.0f, iw = 1.0f / w;
    return {lo, w, iw, lo * iw, mode, face};
}

// the stand-alone preconditioner update (no workspace)
struct P1Args {
    int S, H, T_dense;
    const int* cu;
    const void* k;
    const float *beta, *retsrc, *d0;
    void* ktil;
    float* d_final;
    float* ratio;      // nullable: residual ratio q_t per token-head
    float* log_sum;    // nullable: sum_t log q_t per chain
    Hyper hy;
    P1Coord q;
};

// ---------------------------------------------------------------------------------------------
// forward: parallel speculative pass, then the sequential pass over what is left
// ---------------------------------------------------------------------------------------------
struct P1Fwd {
    int S, H, NT;
    Table tab;
    const void* k;
    const float *beta, *retsrc, *d0;
    void* ktil;          // [T,H,K] float or bf16
    float* d_final;      // nullable
    P1Regions r;
    int save;
    Hyper hy;
    P1Coord q;
    int* status;         // device status word (bounded waits of the rings report here)
    ClearList clear;
};

__device__ __forceinline__ void clear_regions(const ClearList& c)
{
    const int at = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
#pragma unroll
    for (int r = 0; r < 3; ++r)
        for (int i = at; i < c.n[r]; i += step) c.p[r][i] = 0;
}

// Eight consecutive values of a row as floats (one 16-byte load for bf16, two for fp32).
__device__ __forceinline__ void load8(const float* p, float (&x)[8])
{
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&x)[8])
{
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 f = __bfloat1622float2(h[q]);
        x[2 * q] = f.x;
        x[2 * q + 1] = f.y;
    }
}
__device__ __forceinline__ void store8(float* p, const float (&x)[8])
{
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4*>(p + 4) = make_float4(x[4], x[5], x[6], x[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&x)[8])
{
    uint4 v;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(x[2 * q], x[2 * q + 1]);
    *reinterpret_cast<uint4*>(p) = v;
}

// One warp per (chunk, head, 32-token half), eight lanes per token (four tokens at a time): a row is
// read in full 128-byte lines and the sums need three shuffle rounds.  The step is taken from
// d = d_min 1: then <d, k^2> = d_min sum k^2, and since x_r = rho d_min + c k_r^2 is monotone in k_r^2
// for a fixed c, "every x_r below d_min" is decided by the largest (c >= 0) or smallest (c < 0) k_r^2.
// With a vector retention (VEC) rho differs per coordinate and every x_r is formed.
template <typename TI, typename TO, int K, bool VEC>
__global__ void __launch_bounds__(128) phase1_spec_kernel(P1Fwd a)
{
    constexpr int NV = K / 64;   // 8-value vectors per lane
    const int lane = threadIdx.x & 31;
    const int grp = lane >> 3, l8 = lane & 7;
    const long w = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long tile = w >> 1;
    const int half = (int)(w & 1);
    pdl_release();
    pdl_wait();
    clear_regions(a.clear);
    if (tile >= (long)a.NT * a.H) return;
    const int c = (int)(tile / a.H), h = (int)(tile % a.H);
    const int len = a.tab.chunk_len(c), tok0 = a.tab.chunk_tok0(c);
    const Hyper hy = a.hy;
    const TI* kbase = static_cast<const TI*>(a.k);
    TO* tbase = static_cast<TO*>(a.ktil);
    unsigned word = 0;
    // Four iterations' rows and scalars are on their way before the first one is worked on: a warp's time is a few trips to
    // memory, not its arithmetic (two at a time: 20 us at 8 x 2048 tokens, 8 heads, 10.5 us at a single sequence).
    constexpr int AHEAD = 4, PIECES = 8 * (int)sizeof(TI) / 16;
#pragma unroll 1
    for (int it0 = 0; it0 < 8; it0 += AHEAD) {
        uint4 raw[AHEAD][NV][PIECES];
        float rets[AHEAD], betas[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const int i = half * 32 + (it0 + u) * 4 + grp;
            const bool in = i < len;
            const size_t th = (size_t)(tok0 + (in ? i : 0)) * a.H + h;
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int x = 0; x < PIECES; ++x)
                    raw[u][v][x] = reinterpret_cast<const uint4*>(kbase + th * K + v * 64 + l8 * 8)[x];
            rets[u] = (!VEC && in && hy.apf_mode != 0) ? a.retsrc[th] : 0.f;
            betas[u] = (in && hy.beta_aware) ? a.beta[th] : 1.0f;
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const int it = it0 + u;
            const int i = half * 32 + it * 4 + grp;
            const bool in = i < len;
            const size_t th = (size_t)(tok0 + (in ? i : 0)) * a.H + h;
            float x[NV][8];
#pragma unroll
            for (int v = 0; v < NV; ++v) load8(reinterpret_cast<const TI*>(raw[u][v]), x[v]);
            const float ret = rets[u], b = betas[u];
            float sumk = 0.f, kmax = 0.f, kmin = 3.0e38f;
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float kap = x[v][e] * x[v][e];
                    sumk += kap;
                    kmax = fmaxf(kmax, kap);
                    kmin = fminf(kmin, kap);
                }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                sumk += __shfl_xor_sync(0xffffffffu, sumk, o);
                kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
                kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
            }
            const float n = fmaxf(sumk, hy.eps);
            const float rho = hy.apf_mode == 0 ? 1.0f : expf(ret);
            bool low = false;
            if (hy.clamp) {
                const float al = hy.d_min * sumk;
                const float cc = hy.eta * b * (1.0f - b * al) / n;
                if constexpr (VEC) {
                    bool below = true;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        float lr[8];
                        load8(a.retsrc + th * K + v * 64 + l8 * 8, lr);
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            below = below && fmaf(cc, x[v][e] * x[v][e], expf(lr[e]) * hy.d_min) < hy.d_min;
                    }
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) below = __shfl_xor_sync(0xffffffffu, (int)below, o) && below;
                    low = in && below;
                } else {
                    const float xtop = fmaf(cc, cc >= 0.f ? kmax : kmin, rho * hy.d_min);
                    low = in && xtop < hy.d_min;
                }
            }
            if (in && l8 == 0) {
                a.r.sumk[th] = sumk;
                a.r.kmax[th] = kmax;
                a.r.rho[th] = rho;
            }
            if (low) {   // the write key of a token entered on the face: d_min k
#pragma unroll
                for (int v = 0; v < NV; ++v) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[v][e] *= hy.d_min;
                    store8(tbase + th * K + v * 64 + l8 * 8, x[v]);
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, low);
            word |= ((bal & 1u) | ((bal >> 7) & 2u) | ((bal >> 14) & 4u) | ((bal >> 21) & 8u)) << (it * 4);
        }
    }
    if (lane == 0) {
        a.r.flags[tile * 2 + half] = word;
        if (a.save) a.r.skipw[tile * 2 + half] = word;   // what the sequential pass skips, if it does not say otherwise
    }
}

__device__ __forceinline__ void prefetch_l2(const void* p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
// ---------------------------------------------------------------------------------------------
// The sequential pass, forward.  What it processes are lists of tokens of one chain: a dense run where d is off the
// lower face, otherwise the unflagged tokens with a few tokens behind each (what lies between is skipped, provided that
// d is back on the face there).  Walking such a list token by token is bound by the latency of the warp-wide sum
// <d_t, k_t^2> in the middle of every step (five shuffle rounds of 30 cycles each, or an integer reduction of 75 with its
// conversions; a multiply-add takes 5).  So the step scalars c_t of a block of PB tokens are solved for together:
//
//   guess c for the block; run d through the block with these c (one multiply-add per token and coordinate on the
//   dependent path); form all PB sums at once; c_t = e_t - a2_t <d_t, k_t^2>; repeat until c does not change.
//
// c_t depends on d_t, hence on the c of earlier tokens only: after m rounds the first m tokens are exact whatever the
// input, so it ends; and the dependence is weak (a change of c_s moves c_t by eta beta^2 <k_s^2, k_t^2>, and
// <k_s^2, k_t^2> is about 1/128 for unit keys): measured 1.2 rounds at a step size of 0.003, 3.4 at 0.3.
// A round's c is taken when the d it leads to are unchanged: |change of c_t| max k_t^2 at most 2^-26 of the smallest d
// the box allows (a quarter of its rounding unit), or a unit in the last place of c_t.
// In isolation a block of 32 tokens takes 630 + 660 cycles a round with a coordinate per lane (in the kernel, two a lane,
// 3470 cycles at 3.3 rounds), against 109 cycles a token for one warp with one integer reduction per token.
//
// Warps of a chain's CTA: K / 64 core warps, two that fetch keys and scalars (blocks in turn), four that finish (with more
// chains than SMs one of each; they repeat a block's steps from its c, the same operations in the same order, and write ktil_t = d_t (.) k_t, d_t and the
// mask words).  Blocks go round a ring of buffers; the roles meet at mbarriers (full: fetch -> core and finish, done:
// core -> finish, free: finish -> fetch).  Warp 0 decides between two lists and walks short ones alone.
// ---------------------------------------------------------------------------------------------
constexpr int PB = 32;
constexpr int P1_ERR_PIPE = 131;
constexpr long long P1_WAIT_LIMIT = 4000000000ll;   // about two seconds
constexpr int LIST_MAX = 256;                       // entries of a sparse list
constexpr int WALK = 16;                            // tokens of a first dense run
constexpr int SCAN_CHUNKS = 128;                    // chunks whose words warp 0 reads at a time

// A block's way round the ring (fetch, core, finish) takes about six times what the core needs for it, hence that many
// helpers and a deep ring: with four buffers and two finishing warps the core waited for half of the time.
// The forward's core warps own two coordinates a lane and have a scheduler each, 0 and 1; the helpers sit on schedulers
// 2 and 3 (warp numbers modulo four), the warps in between leave at once.  Beside helpers on its own scheduler a core of
// four warps took 4700 cycles for a block instead of 2900.
template <int K, bool MANY> struct FwdPipe {
    static constexpr int CORE = K / 64, FETCH0 = 2, FETCH = 2, FINISH0 = 4, FINISH = 4, THREADS = 384, ACTIVE = (CORE + FETCH + FINISH) * 32;
    static constexpr int CTAS = 1, RING_BYTES = 216 * 1024;
    // the role number of a hardware warp: core 0 .., fetch 2, 3, finish 4 .. 7; -1: idle
    __device__ static __forceinline__ int role(int warp)
    {
        const int sched = warp & 3, row = warp >> 2;
        return sched < 2 ? (row == 0 && warp < CORE ? warp : -1) : row * 2 + sched;
    }
};
// More chains than SMs: one fetching and one finishing warp and a short ring, so that three chains share an SM (one to an
// SM, they queue for it: the moving stand-alone update of 1024 tokens, 74 us for 64 chains, took 203 us for 300 and now
// takes 118; the forward's pass 265 -> 160 us).
template <int K> struct FwdPipe<K, true> {
    static constexpr int CORE = K / 64, FETCH0 = CORE, FETCH = 1, FINISH0 = CORE + 1, FINISH = 1, THREADS = (CORE + 2) * 32, ACTIVE = THREADS;
    static constexpr int CTAS = 3, RING_BYTES = 72 * 1024;
    __device__ static __forceinline__ int role(int warp) { return warp; }
};
template <int K> struct Pipe {
    static constexpr int CORE = K / 32, FETCH0 = CORE, FETCH = 2, FINISH0 = CORE + FETCH, FINISH = 4, WARPS = FINISH0 + FINISH, THREADS = WARPS * 32;
};
constexpr int RING_MAX = 8;
// Buffers of the given size that fit `room` bytes: RING_MAX or half of it, or any number with one helper of each kind.  The
// depth is a multiple of the numbers of fetching and of finishing warps, so that all uses of a buffer are the same warps'
// and follow one another in order (a wait tells a barrier's phases apart by their parity only).
constexpr int ring_depth(size_t bytes, size_t room, int helpers)
{
    if (helpers == 1) return bytes * 4 <= room ? 4 : (int)(room / bytes);
    return bytes * RING_MAX <= room ? RING_MAX : RING_MAX / 2;
}

// Bounded: gives up after P1_WAIT_LIMIT cycles, records the error and returns false.  The whole warp calls; the vote at
// the end brings its lanes together again (lanes that leave the loop in different turns would otherwise run what
// follows one after the other).
__device__ __forceinline__ bool p1_mbar_wait(uint64_t* b, uint32_t parity, int* status)
{
    const uint32_t addr = (uint32_t)__cvta_generic_to_shared(b);
    uint32_t ok = 0;
    const long long t0 = clock64();
    while (!ok) {
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok)
                     : "r"(addr), "r"(parity)
                     : "memory");
        if (!ok && clock64() - t0 > P1_WAIT_LIMIT) break;
    }
    if (!ok && status) atomicCAS(status, 0, P1_ERR_PIPE);
    return __all_sync(0xffffffffu, ok != 0);
}
template <int NT> __device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(NT) : "memory"); }
// The barrier with a vote: whether `pred` held everywhere, so that the warps go on, or give up, together.
template <int NT> __device__ __forceinline__ bool bar_sync_and(int id, bool pred)
{
    uint32_t r;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; barrier.cta.red.and.pred q, %2, %3, p; selp.u32 %0, 1, 0, q; }"
                 : "=r"(r) : "r"((uint32_t)pred), "r"(id), "n"(NT) : "memory");
    return r != 0;
}
__device__ __forceinline__ bool bit_of(unsigned m, int j) { return (m >> j) & 1u; }

struct PipeBars {
    uint64_t full[RING_MAX], done[RING_MAX], free_[RING_MAX];
};
__device__ __forceinline__ void init_bars(PipeBars& bars, int n, int core_warps)
{
    for (int i = 0; i < n; ++i) {
        umma::mbar_init(&bars.full[i], 1);
        umma::mbar_init(&bars.done[i], core_warps);
        umma::mbar_init(&bars.free_[i], 1);
    }
}

template <typename TI, int K, bool VEC> struct PipeBuf {
    TI k[PB][K];                            // as it sits in memory; rows beyond the list are zero
    float y0[K];                            // core: y on entry to the block
    float raw[4][PB];                       // sum k^2, max k^2, retention, beta as they sit in memory
    float rho[PB], off[PB];                 // retention (0 behind a jump: y is 0 there), (retention - 1) d_min / w
    float4 scal[PB];                        // e', a2, max k^2, sum k^2
    float2 res[PB];                         // core: c', <y, k^2>
    unsigned jump;                          // bit j: the token before this one was skipped, d enters on the face
    int n;                                  // core: tokens of the block that stand
    alignas(16) float rv[VEC ? PB : 1][VEC ? K : 1];   // vector retention: l_t, then (core) exp(l_t)
};
template <typename TI, int K, bool VEC, bool MANY> struct PipeShared {
    using P = FwdPipe<K, MANY>;
    static constexpr int CW = P::CORE, PN = ring_depth(sizeof(PipeBuf<TI, K, VEC>), P::RING_BYTES, P::FINISH);
    static_assert(PN >= 2 && PN % P::FETCH == 0 && PN % P::FINISH == 0, "a buffer belongs to one fetching and one finishing warp");
    PipeBuf<TI, K, VEC> buf[PN];
    float y[K];                             // between two lists
    float c[CW][PB];                        // a core warp's c' of the round
    float part[2][CW][PB];                  // the core warps' shares of the sums, by round parity
    unsigned bad[CW];                       // jumps that d enters off the face
    unsigned long long words[SCAN_CHUNKS];
    uint16_t list[LIST_MAX];
    int cmd_tok, cmd_n, cmd_dense;          // first token (a list's offsets count from it), entries; none: finished
    int stop;                               // entries that stand
    PipeBars bars;
};

__device__ __forceinline__ float p1_y(float d, const P1Coord& q) { return __fmul_rn(d - q.lo, q.iw); }
__device__ __forceinline__ float p1_d(float y, const P1Coord& q) { return fmaf(q.w, y, q.lo); }
__device__ __forceinline__ float p1_off(float rho, const P1Coord& q) { return fmaf(rho, q.k0, -q.k0); }
__device__ __forceinline__ float p1_raw(float y, float kap, float c, float rho, float off) { return fmaf(rho, y, fmaf(c, kap, off)); }
template <P1Mode M> __device__ __forceinline__ float p1_project(float x, const Hyper& hy, const P1Coord& q)
{
    if (M == P1_SAT) return __saturatef(x);
    if (!hy.clamp) return x;
    return q.face ? fminf(fmaxf(x, 0.f), hy.d_max - hy.d_min) : fminf(fmaxf(x, hy.d_min), hy.d_max);
}
// e', a2, max k^2, sum k^2 of a token
__device__ __forceinline__ float4 p1_scalars(float sumk, float kmax, float beta, const Hyper& hy, const P1Coord& q)
{
    const float b = hy.beta_aware ? beta : 1.0f;
    const float e = hy.eta * b / fmaxf(sumk, hy.eps), a2 = e * b;
    return make_float4(fmaf(-a2 * q.lo, sumk, e) * q.iw, a2, kmax, sumk);
}

__device__ __forceinline__ float2 load2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 load2(const __nv_bfloat16* p) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p)); }

// One block by the core warps: y of this lane's coordinates goes through it (slots beyond its n tokens leave y alone).
// r: <y, k^2> / sum k^2 of the latest token, the start of the next guess; rounds: all rounds so far.  Returns the tokens
// that stand: n, or those before the first jump that d enters off the face (y is then its value there).
template <typename TI, int K, bool VEC, bool MANY, P1Mode M>
__device__ __forceinline__ int core_block(PipeShared<TI, K, VEC, MANY>& sh, PipeBuf<TI, K, VEC>& B, int n, float2& y, float& r, uint32_t& rounds,
                                          const Hyper& hy, const P1Coord& q, int warp, int lane)
{
    constexpr int CW = FwdPipe<K, MANY>::CORE;
    const int i = warp * 64 + lane * 2;   // this lane's coordinates: i, i + 1
    float ka[PB], kb[PB];
#pragma unroll
    for (int j = 0; j < PB; ++j) {
        const float2 k = load2(&B.k[j][i]);
        ka[j] = __fmul_rn(k.x, k.x);
        kb[j] = __fmul_rn(k.y, k.y);
    }
    auto retention = [&](int j) -> float2& { return *reinterpret_cast<float2*>(&B.rv[VEC ? j : 0][VEC ? i : 0]); };
    if constexpr (VEC) {
#pragma unroll 4
        for (int j = 0; j < PB; ++j) {
            float2& v = retention(j);
            v = j < n ? make_float2(expf(v.x), expf(v.y)) : make_float2(1.f, 1.f);
        }
    }
    *reinterpret_cast<float2*>(B.y0 + i) = y;
    const unsigned jump = B.jump;
    const float4 sc = B.scal[lane];   // lane j: token j
    const bool jumped = bit_of(jump, lane);
    const float tol = hy.clamp ? 1.4901161e-8f * fmaxf(hy.d_min, 0.f) * q.iw : 0.f;
    float c = jumped ? sc.x : fmaf(-sc.y, sc.w * r, sc.x), sum = 0.f;
    float2 z = y;
    // a step of both coordinates; keep: 0 behind a jump (then the scalar retention is 0 already)
    auto step = [&](float2 v, float kx, float ky, float cj, float rho, float off, int j) {
        float rx = rho, ry = rho, ox = off, oy = off;
        if constexpr (VEC) {   // (rho: 0 behind a jump, else 1)
            const float2 x = retention(j);
            ox = p1_off(x.x, q);
            oy = p1_off(x.y, q);
            rx *= x.x;
            ry *= x.y;
        }
        return make_float2(p1_project<M>(p1_raw(v.x, kx, cj, rx, ox), hy, q), p1_project<M>(p1_raw(v.y, ky, cj, ry, oy), hy, q));
    };
    for (int round = 0; round <= PB; ++round) {   // (round PB + 1 could change nothing)
        const uint32_t par = rounds++ & 1;
        sh.c[warp][lane] = c;
        __syncwarp();
        float p[PB];
        z = y;
#pragma unroll
        for (int j = 0; j < PB; j += 4) {
            const float4 c4 = *reinterpret_cast<const float4*>(&sh.c[warp][j]), r4 = *reinterpret_cast<const float4*>(B.rho + j);
            const float4 o4 = *reinterpret_cast<const float4*>(B.off + j);
            const float cv[4] = {c4.x, c4.y, c4.z, c4.w}, rv[4] = {r4.x, r4.y, r4.z, r4.w}, ov[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                p[j + u] = fmaf(z.x, ka[j + u], z.y * kb[j + u]);
                z = step(z, ka[j + u], kb[j + u], cv[u], rv[u], ov[u], j + u);
            }
        }
        sum = transpose_sum(p, lane);
        if constexpr (CW > 1) {
            float(*part)[PB] = sh.part[par];
            part[warp][lane] = sum;
            bar_sync<CW * 32>(3);
            sum = part[0][lane];
#pragma unroll
            for (int x = 1; x < CW; ++x) sum += part[x][lane];
        }
        if (jumped) sum = 0.f;
        const float cn = fmaf(-sc.y, sum, sc.x);
        const float dc = fabsf(cn - c);
        // the same values in every core warp, so they all leave in the same round
        if (__all_sync(0xffffffffu, dc * sc.z <= tol || dc <= 1.1920929e-7f * fabsf(cn) || lane >= n)) break;
        c = cn;
    }
    int stand = n;
    if (jump) {   // was d on the face at the jumps?
        auto to = [&](int end, unsigned& off_face) {
            float2 v = y;
#pragma unroll 4
            for (int j = 0; j < end; ++j) {
                if (bit_of(jump, j) && (v.x != 0.f || v.y != 0.f)) off_face |= 1u << j;
                const float2 k = load2(&B.k[j][i]);
                v = step(v, __fmul_rn(k.x, k.x), __fmul_rn(k.y, k.y), sh.c[warp][j], B.rho[j], B.off[j], j);
            }
            return v;
        };
        unsigned bad = 0;
        to(n, bad);
        bad = __reduce_or_sync(0xffffffffu, bad);
        if constexpr (CW > 1) {
            if (lane == 0) sh.bad[warp] = bad;
            bar_sync<CW * 32>(3);
#pragma unroll
            for (int x = 0; x < CW; ++x) bad |= sh.bad[x];
        }
        if (bad) {
            stand = __ffs((int)bad) - 1;
            unsigned none = 0;
            z = to(stand, none);
        }
    }
    y = z;
    if (warp == 0) {
        B.res[lane] = make_float2(c, sum);
        if (lane == 0) B.n = stand;
    }
    r = __shfl_sync(0xffffffffu, sum / fmaxf(sc.w, 1e-30f), n - 1);
    return stand;
}
template <typename TI, int K, bool VEC, bool MANY>
__device__ __forceinline__ int core_block(PipeShared<TI, K, VEC, MANY>& sh, PipeBuf<TI, K, VEC>& B, int n, float2& y, float& r, uint32_t& rounds,
                                          const Hyper& hy, const P1Coord& q, int warp, int lane)
{
    if (q.mode == P1_SAT) return core_block<TI, K, VEC, MANY, P1_SAT>(sh, B, n, y, r, rounds, hy, q, warp, lane);
    return core_block<TI, K, VEC, MANY, P1_PLAIN>(sh, B, n, y, r, rounds, hy, q, warp, lane);
}

// Rows of D elements on their way into a buffer; lane j of the warp holds the number of row j in the source (NO_ROW: the
// row is filled with zeros).
constexpr uint32_t NO_ROW = ~0u;
template <typename T, int D> __device__ __forceinline__ void fetch_rows(T* dst, const T* src, uint32_t mine, int rows, int lane)
{
    constexpr int PIECES = D * (int)sizeof(T) / 16, EL = 16 / (int)sizeof(T), STEP = 32 / PIECES;
    static_assert(PIECES <= 32, "a row is one or a part of a warp-wide copy");
    const int c = lane % PIECES * EL;
#pragma unroll 8
    for (int j = lane / PIECES; j < (rows + STEP - 1) / STEP * STEP; j += STEP) {
        const uint32_t row = __shfl_sync(0xffffffffu, mine, j);
        cp_async16_zfill(dst + j * D + c, src + (row == NO_ROW ? 0 : (size_t)row * D) + c, row != NO_ROW);
    }
}

// A finishing warp's work on a block: out(j, d_t, k_t, bits) for its n tokens; bit r of `bits`: the projection passed
// gradient for coordinate R lane + r (inside the box, faces included).
template <typename TI, int K, bool VEC, P1Mode M, typename OUT>
__device__ __forceinline__ void finish_block(const PipeBuf<TI, K, VEC>& B, int n, const Hyper& hy, const P1Coord& q, int lane, OUT out)
{
    constexpr int R = K / 32;
    const unsigned jump = B.jump;
    float y[R];
    load_row<R>(B.y0, lane, y);
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        float kk[R], d[R], rho[R], off[R];
        load_row<R>(B.k[j], lane, kk);
        const float c = B.res[j].x;
        if constexpr (VEC) {
            load_row<R>(B.rv[VEC ? j : 0], lane, rho);
#pragma unroll
            for (int r = 0; r < R; ++r) off[r] = p1_off(rho[r], q);
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                rho[r] = B.rho[j];
                off[r] = B.off[j];
            }
        }
        const float keep = bit_of(jump, j) ? 0.f : 1.f;
        unsigned bits = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float v = y[r] * keep;
            d[r] = p1_d(v, q);
            const float x = p1_raw(v, __fmul_rn(kk[r], kk[r]), c, rho[r], off[r]);
            y[r] = p1_project<M>(x, hy, q);
            bits |= y[r] == x ? (1u << r) : 0u;
        }
        out(j, d, kk, bits);
    }
}
template <typename TI, int K, bool VEC, typename OUT>
__device__ __forceinline__ void finish_block(const PipeBuf<TI, K, VEC>& B, int n, const Hyper& hy, const P1Coord& q, int lane, OUT out)
{
    if (q.mode == P1_SAT) finish_block<TI, K, VEC, P1_SAT>(B, n, hy, q, lane, out);
    else finish_block<TI, K, VEC, P1_PLAIN>(B, n, hy, q, lane, out);
}

// The list in sh through the ring, all roles.  y travels through sh.y; guess and rounds belong to the core warps.
template <typename TI, typename TO, int K, bool VEC, bool MANY>
__device__ __forceinline__ bool run_list(const P1Fwd& a, int h, PipeShared<TI, K, VEC, MANY>& sh, float& guess, uint32_t& rounds, uint32_t& uses,
                                         int warp, int lane)
{
    constexpr int R = K / 32;
    using P = FwdPipe<K, MANY>;
    constexpr int PN = PipeShared<TI, K, VEC, MANY>::PN;
    const int H = a.H;
    const Hyper hy = a.hy;
    const P1Coord& q = a.q;
    const int tok0 = sh.cmd_tok, total = sh.cmd_n;
    const bool dense = sh.cmd_dense != 0;
    const int nblk = (total + PB - 1) / PB;
    bool ok = true;
    // block b uses buffer (base + b) % PN; its barriers complete once per use: parity of the use count
    const uint32_t base = uses;
    auto tok_of = [&](int idx) { return tok0 + (dense ? idx : (int)sh.list[idx] & 0x7fff); };
    auto len_of = [&](int b) { return min(PB, total - b * PB); };
    auto th_of = [&](int b) { return lane < len_of(b) ? (uint32_t)(tok_of(b * PB + lane) * H + h) : NO_ROW; };   // lane j: token j
    if (warp < P::CORE) {
        float2 y = load2(sh.y + warp * 64 + lane * 2);
        int stop = total;
        bool dead = false;   // d left the list: what follows in it is dropped
        for (int b = 0; b < nblk; ++b) {
            const int bi = (base + b) % PN;
            ok = bar_sync_and<P::CORE * 32>(3, p1_mbar_wait(&sh.bars.full[bi], ((base + b) / PN) & 1, a.status));
            if (!ok) break;
            PipeBuf<TI, K, VEC>& B = sh.buf[bi];
            if (!dead) {
                const int n = len_of(b), stand = core_block<TI, K, VEC, MANY>(sh, B, n, y, guess, rounds, hy, q, warp, lane);
                if (stand < n) {
                    dead = true;
                    stop = b * PB + stand;
                }
            } else if (warp == 0 && lane == 0) {
                B.n = 0;
            }
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.done[bi]);
        }
        *reinterpret_cast<float2*>(sh.y + warp * 64 + lane * 2) = y;
        if (warp == 0 && lane == 0) sh.stop = ok ? stop : 0;
    } else if (warp < P::FINISH0) {
        // the warps take the blocks in turn
        auto start = [&](int b) {
            const uint32_t use = base + b;
            const int bi = use % PN;
            if (use >= PN) ok = p1_mbar_wait(&sh.bars.free_[bi], ((use / PN) - 1) & 1, a.status);
            if (!ok) return;
            PipeBuf<TI, K, VEC>& B = sh.buf[bi];
            const uint32_t th = th_of(b);
            fetch_rows<TI, K>(&B.k[0][0], static_cast<const TI*>(a.k), th, PB, lane);
            if constexpr (VEC) fetch_rows<float, K>(&B.rv[0][0], a.retsrc, th, PB, lane);
            if (th != NO_ROW) {
                cp_async4(&B.raw[0][lane], a.r.sumk + th);
                cp_async4(&B.raw[1][lane], a.r.kmax + th);
                cp_async4(&B.raw[2][lane], a.r.rho + th);
                cp_async4(&B.raw[3][lane], a.beta + th);
            }
            cp_async_commit();
        };
        auto complete = [&](int b) {   // the step's scalars from the raw ones
            const int bi = (base + b) % PN;
            PipeBuf<TI, K, VEC>& B = sh.buf[bi];
            const int n = len_of(b), idx = b * PB + lane;
            float4 sc = make_float4(0.f, 0.f, 0.f, 0.f);   // an empty slot: c' = 0, k^2 = 0, rho = 1
            float rho = 1.f;
            bool jump = false;
            if (lane < n) {
                sc = p1_scalars(B.raw[0][lane], B.raw[1][lane], B.raw[3][lane], hy, q);
                rho = B.raw[2][lane];
                jump = !dense && idx > 0 && tok_of(idx) != tok_of(idx - 1) + 1;
            }
            const unsigned jumps = __ballot_sync(0xffffffffu, jump);
            B.scal[lane] = sc;
            B.off[lane] = p1_off(rho, q);
            B.rho[lane] = jump ? 0.f : VEC ? 1.f : rho;
            if (lane == 0) B.jump = jumps;
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.full[bi]);
        };
        int b = (int)((warp - P::FETCH0 - base) & (P::FETCH - 1));
        if (b < nblk) start(b);
        for (; b < nblk && ok; b += P::FETCH) {
            cp_async_wait<0>();
            __syncwarp();
            complete(b);
            if (b + P::FETCH < nblk) start(b + P::FETCH);
        }
        cp_async_wait<0>();
    } else {
        TO* kt = static_cast<TO*>(a.ktil);
        for (int b = (int)((warp - P::FINISH0 - base) & (P::FINISH - 1)); b < nblk; b += P::FINISH) {
            const int bi = (base + b) % PN;
            ok = p1_mbar_wait(&sh.bars.done[bi], ((base + b) / PN) & 1, a.status);
            if (!ok) break;
            const PipeBuf<TI, K, VEC>& B = sh.buf[bi];
            const int n = B.n;
            const uint32_t mine = th_of(b);
            finish_block<TI, K, VEC>(B, n, hy, q, lane, [&](int j, const float (&d)[R], const float (&kk)[R], unsigned bits) {
                const size_t th = __shfl_sync(0xffffffffu, mine, j);
                float wk[R];
#pragma unroll
                for (int r = 0; r < R; ++r) wk[r] = d[r] * kk[r];
                store_row<R>(kt + th * K, lane, wk);
                if (a.save) {
                    store_row<R>(a.r.dtraj + th * K, lane, d);
                    a.r.pmask[th * 32 + lane] = bits;
                }
            });
            if (a.save && lane < n) a.r.al[mine] = fmaf(q.w, B.res[lane].y, q.lo * B.scal[lane].w);
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.free_[bi]);
        }
    }
    uses = base + nblk;
    return ok;
}

// A list of at most PB entries by warp 0 alone, token by token (a few tokens are done before a ring would be full, and
// the code is short).  An entry marked with bit 15 is skipped when d enters it on the face.  Returns the entries
// that stand (fewer than n where d is off the face at a jump); sets the bits of the processed tokens in `proc`.
template <typename TI, typename TO, int K, bool VEC, bool MANY>
__device__ __forceinline__ int walk_list(const P1Fwd& a, int h, PipeShared<TI, K, VEC, MANY>& sh, int tok0, int n, bool& face, unsigned long long& proc, int lane)
{
    constexpr int R = K / 32;
    const int H = a.H;
    const Hyper hy = a.hy;
    const P1Coord& q = a.q;
    // the projection as minimum and maximum in every mode: the same values, and no choice per token on the walk's path
    const bool clip = hy.clamp;
    const float bottom = q.face ? 0.f : hy.d_min, top = q.mode == P1_SAT ? 1.0f : q.face ? hy.d_max - hy.d_min : hy.d_max;
    PipeBuf<TI, K, VEC>& B = sh.buf[0];
    const uint32_t mine = lane < n ? (uint32_t)((tok0 + ((int)sh.list[lane] & 0x7fff)) * H + h) : NO_ROW;
    fetch_rows<TI, K>(&B.k[0][0], static_cast<const TI*>(a.k), mine, n, lane);
    if constexpr (VEC) fetch_rows<float, K>(&B.rv[0][0], a.retsrc, mine, n, lane);
    cp_async_commit();
    if (lane < n) {
        const float rho = a.r.rho[mine];
        B.scal[lane] = p1_scalars(a.r.sumk[mine], a.r.kmax[mine], a.beta[mine], hy, q);
        B.rho[lane] = rho;
        B.off[lane] = p1_off(rho, q);
    }
    float y[R];
    load_row<R>(sh.y, lane, y);
    cp_async_wait<0>();
    __syncwarp();
    int prev = -1, j = 0;
#pragma unroll 1
    for (; j < n; ++j) {
        const int e = sh.list[j], at = e & 0x7fff;
        if (face && (e & 0x8000)) continue;
        if (!face && prev >= 0 && at != prev + 1) break;
        prev = at;
        const size_t th = (size_t)(tok0 + at) * H + h;
        const float4 sc = B.scal[j];
        float kk[R], rho[R], off[R], d[R], wk[R], s = 0.f;
        load_row<R>(B.k[j], lane, kk);
        if constexpr (VEC) {
            load_row<R>(B.rv[VEC ? j : 0], lane, rho);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                rho[r] = expf(rho[r]);
                off[r] = p1_off(rho[r], q);
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                rho[r] = B.rho[j];
                off[r] = B.off[j];
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) s = fmaf(y[r], __fmul_rn(kk[r], kk[r]), s);
        s = warp_sum(s);
        const float c = fmaf(-sc.y, s, sc.x);
        unsigned bits = 0;
        bool on = q.face;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            d[r] = p1_d(y[r], q);
            wk[r] = d[r] * kk[r];
            const float x = p1_raw(y[r], __fmul_rn(kk[r], kk[r]), c, rho[r], off[r]);
            y[r] = clip ? fminf(fmaxf(x, bottom), top) : x;
            bits |= y[r] == x ? (1u << r) : 0u;
            on = on && y[r] == 0.f;
        }
        store_row<R>(static_cast<TO*>(a.ktil) + th * K, lane, wk);
        if (a.save) {
            store_row<R>(a.r.dtraj + th * K, lane, d);
            a.r.pmask[th * 32 + lane] = bits;
            if (lane == 0) a.r.al[th] = fmaf(q.w, s, q.lo * sc.w);
        }
        if (lane == at >> 6) proc |= 1ull << (at & 63);
        face = __all_sync(0xffffffffu, on);
    }
    store_row<R>(sh.y, lane, y);
    __syncwarp();
    return j;
}

// The tokens of 32 chunks from bit `pos` on, for the lane that holds chunk `lane`.
__device__ __forceinline__ unsigned long long from_bit(int pos, int lane)
{
    const int rel = pos - 64 * lane;
    return rel <= 0 ? ~0ull : rel >= 64 ? 0ull : ~0ull << rel;
}
__device__ __forceinline__ unsigned long long valid_bits(int len) { return len >= 64 ? ~0ull : len <= 0 ? 0ull : (1ull << len) - 1ull; }

// Set bits of the lanes' words, in order, into a list of at most `most` offsets (those that are set in `mark` too with
// bit 15); returns how many there were.
__device__ __forceinline__ int write_list(uint16_t* list, unsigned long long w, unsigned long long mark, int most, int lane)
{
    const int mine = __popcll(w);
    int end = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += u;
    }
    for (int at = end - mine; w && at < most; ++at) {
        const int t = __ffsll((long long)w) - 1;
        w &= w - 1;
        list[at] = (uint16_t)((64 * lane + t) | (int)((mark >> t) & 1ull) << 15);
    }
    __syncwarp();
    return __shfl_sync(0xffffffffu, end, 31);
}

// The words of SCAN_CHUNKS chunks from c on, complemented (set: unflagged, or processed) and cut to the sequence, into
// shared memory, four loads in flight per lane (one group of 32 at a time made a long sequence wait for memory once per 2048
// tokens).  Chunks [c0, c1); word of chunk c + x at words[x].
__device__ __forceinline__ void scan_words(unsigned long long* words, const unsigned* src, int c, int c0, int c1, int seq_len, int H, int h, int lane)
{
    uint2 w[SCAN_CHUNKS / 32];
#pragma unroll
    for (int g = 0; g < SCAN_CHUNKS / 32; ++g) {
        const int x = c + g * 32 + lane;
        w[g] = x < c1 ? *reinterpret_cast<const uint2*>(src + ((size_t)x * H + h) * 2) : make_uint2(~0u, ~0u);
    }
#pragma unroll
    for (int g = 0; g < SCAN_CHUNKS / 32; ++g)
        words[g * 32 + lane] = ~((unsigned long long)w[g].x | (unsigned long long)w[g].y << 32) & valid_bits(seq_len - (c + g * 32 + lane - c0) * CH);
    __syncwarp();
}

// Which tokens are processed, decided by warp 0.
//   on the face   the next unflagged tokens with `follow` tokens behind each, at most LIST_MAX; d is expected back on
//                 the face where the list jumps (where it is not, the list ends there, and the chain's later lists
//                 take more tokens behind each)
//   off the face  every token, WALK at first, then 128 and twice as many each time d is still off at the end
// What is not listed is skipped: its write key d_min k is there already and its projection mask is all zero.
// Lists of up to PB entries are walked, unless they are dense and mostly unflagged (d will not be back soon).
template <typename TI, typename TO, int K, bool VEC, bool MANY> struct ListPlan {
    const P1Fwd& a;
    PipeShared<TI, K, VEC, MANY>& sh;
    const int h, lane, c0, c1, seq_t0, seq_len;
    // the group of 32 chunks in hand: unflagged and processed tokens (a chunk per lane), tokens, first token, next one
    int cbase, base = 0, glen = 0, pos = 0;
    unsigned long long unf = 0ull, proc = 0ull, cand = 0ull;
    int follow = 3, run = WALK;
    bool face, listed = false, touched = false;

    __device__ __forceinline__ ListPlan(const P1Fwd& a_, PipeShared<TI, K, VEC, MANY>& sh_, int s, int h_, int lane_)
        : a(a_), sh(sh_), h(h_), lane(lane_), c0(a_.tab.seq_chunk0(s)), c1(a_.tab.seq_chunk0(s + 1)), seq_t0(a_.tab.seq_tok0(s)),
          seq_len(a_.tab.seq_len(s)), cbase(c0 - 32)
    {
        face = on_face();
    }
    __device__ __forceinline__ bool on_face() const
    {
        constexpr int R = K / 32;
        float y[R];
        load_row<R>(sh.y, lane, y);
        bool on = a.q.face;
#pragma unroll
        for (int r = 0; r < R; ++r) on = on && y[r] == 0.f;
        return __all_sync(0xffffffffu, on) != 0;
    }
    __device__ __forceinline__ bool next_group()
    {
        if (cbase >= c0 && a.save && cbase + lane < c1 && (unf ^ proc) != 0ull) {   // (the parallel pass left the flags there)
            const unsigned long long skipped = valid_bits(glen - 64 * lane) & ~proc;
            *reinterpret_cast<uint2*>(a.r.skipw + ((size_t)(cbase + lane) * a.H + h) * 2) =
                make_uint2((unsigned)(skipped & 0xffffffffull), (unsigned)(skipped >> 32));
        }
        cbase += 32;
        if (cbase >= c1) return false;
        const int at = (cbase - c0) % SCAN_CHUNKS;
        if (at == 0) scan_words(sh.words, a.r.flags, cbase, c0, c1, seq_len, a.H, h, lane);
        base = (cbase - c0) * CH;
        glen = min(32 * CH, seq_len - base);
        unf = sh.words[at + lane];
        proc = 0ull;
        pos = 0;
        return true;
    }
    // Leaves the next list for run_list in sh; cmd_n 0: the chain is finished (cmd_dense: anything was processed).
    __device__ __forceinline__ void next()
    {
        if (sh.cmd_n != 0) {   // the list before has been worked off
            const int stop = sh.stop, n = sh.cmd_n;
            face = on_face();
            if (listed) {
                if (stop) pos = ((int)sh.list[stop - 1] & 0x7fff) + 1;
                proc |= cand & ~from_bit(pos, lane);
                if (stop < n) follow = min(2 * follow + 1, 15);
                run = WALK;
            } else {
                pos += stop;
                proc |= cand;
                run = face ? WALK : min(max(2 * run, 4 * PB), 32 * CH);
            }
            if (stop == 0) {   // a wait ran out
                pos = glen;
                cbase = c1;
            }
        }
        while (true) {
            if (pos >= glen) {
                if (next_group()) continue;
                __syncwarp();
                if (lane == 0) {
                    sh.cmd_n = 0;
                    sh.cmd_dense = touched;
                }
                return;
            }
            const unsigned long long valid = valid_bits(glen - 64 * lane);
            int n;
            bool walk;
            listed = face;
            if (face) {
                const unsigned long long my = unf & from_bit(pos, lane);
                if (!__any_sync(0xffffffffu, my != 0ull)) {   // the rest of the group is skipped
                    pos = glen;
                    continue;
                }
                cand = my;
                for (int f = 0; f < follow; ++f) {
                    unsigned long long up = __shfl_up_sync(0xffffffffu, cand, 1) >> 63;
                    if (lane == 0) up = 0ull;
                    cand = my | (cand << 1) | up;
                }
                cand &= valid;
                n = write_list(sh.list, cand, ~unf, LIST_MAX, lane);
                walk = n <= PB;
                n = min(n, LIST_MAX);
            } else {
                n = min(glen - pos, run);
                cand = from_bit(pos, lane) & ~from_bit(pos + n, lane) & valid;
                walk = run == WALK && __reduce_add_sync(0xffffffffu, __popcll(unf & cand)) * 2 < n;
                if (walk) write_list(sh.list, cand, ~unf, LIST_MAX, lane);
            }
            touched = true;
            if (walk) {
                const int stop = walk_list<TI, TO, K, VEC, MANY>(a, h, sh, seq_t0 + base, n, face, proc, lane);
                pos = ((int)sh.list[stop - 1] & 0x7fff) + 1;
                run = face || listed ? WALK : 4 * PB;
                continue;
            }
            __syncwarp();
            if (lane == 0) {
                sh.cmd_tok = seq_t0 + base + (listed ? 0 : pos);
                sh.cmd_n = n;
                sh.cmd_dense = !listed;
            }
            return;
        }
    }
};

// One chain per CTA.
template <typename TI, typename TO, int K, bool VEC, bool MANY>
__global__ void __launch_bounds__(FwdPipe<K, MANY>::THREADS, FwdPipe<K, MANY>::CTAS) phase1_seq_kernel(P1Fwd a)
{
    using P = FwdPipe<K, MANY>;
    extern __shared__ __align__(16) uint8_t p1_dyn[];
    PipeShared<TI, K, VEC, MANY>& sh = *reinterpret_cast<PipeShared<TI, K, VEC, MANY>*>(p1_dyn);
    const int lane = threadIdx.x & 31, warp = P::role(threadIdx.x >> 5);
    const int chain = blockIdx.x;
    const int s = chain / a.H, h = chain % a.H, H = a.H;
    const P1Coord& q = a.q;
    const int coord = threadIdx.x;   // (the first K threads)
    if (threadIdx.x == 0) {
        init_bars(sh.bars, PipeShared<TI, K, VEC, MANY>::PN, P::CORE);
        sh.cmd_n = 0;
    }
    pdl_wait();   // no early release: see pdl_release
    float d_in = 1.0f, guess = 0.f;
    if (coord < K) {
        if (a.d0) d_in = a.d0[((size_t)s * H + h) * K + coord];
        sh.y[coord] = p1_y(d_in, q);
    }
    uint32_t rounds = 0, uses = 0;
    __syncthreads();
    if (warp >= 0) {
    ListPlan<TI, TO, K, VEC, MANY> plan(a, sh, s, h, lane);
    while (true) {   // warp 0 announces a list, all work it off (one call site: the warps share the code)
        if (warp == 0) plan.next();
        bar_sync<P::ACTIVE>(1);
        if (sh.cmd_n == 0) break;
        run_list<TI, TO, K, VEC, MANY>(a, h, sh, guess, rounds, uses, warp, lane);
        bar_sync<P::ACTIVE>(2);
    }
    }
    __syncthreads();
    if (a.d_final && coord < K) a.d_final[((size_t)s * H + h) * K + coord] = sh.cmd_dense ? p1_d(sh.y[coord], q) : d_in;
}

// The stand-alone sweep processes every token: the whole sequence is one list (see above).  The fetching warps also
// form the normalisers here (there is no parallel pass before this kernel; max k^2, which only the rounds' tolerance
// needs, is taken as sum k^2); the finishing ones form the write keys and the residual ratios.
template <typename TI, typename TO, int K, bool VEC, bool MANY>
__global__ void __launch_bounds__(FwdPipe<K, MANY>::THREADS, FwdPipe<K, MANY>::CTAS) phase1_stream_kernel(P1Args a)
{
    constexpr int R = K / 32;
    using P = FwdPipe<K, MANY>;
    constexpr int PN = PipeShared<TI, K, VEC, MANY>::PN;
    extern __shared__ __align__(16) uint8_t p1_dyn[];
    PipeShared<TI, K, VEC, MANY>& sh = *reinterpret_cast<PipeShared<TI, K, VEC, MANY>*>(p1_dyn);
    __shared__ float log_part[P::FINISH];
    const int lane = threadIdx.x & 31, warp = P::role(threadIdx.x >> 5);
    const int chain = blockIdx.x;
    const int s = chain / a.H, h = chain % a.H, H = a.H;
    pdl_wait();
    // packed batch: T_dense is the packed token count; a malformed offset pair is clamped into it
    const int t0 = a.cu ? min(max(a.cu[s], 0), a.T_dense) : s * a.T_dense;
    const int len = a.cu ? min(max(a.cu[s + 1], t0), a.T_dense) - t0 : a.T_dense;
    const Hyper hy = a.hy;
    const P1Coord& q = a.q;
    if (threadIdx.x == 0) init_bars(sh.bars, PN, P::CORE);
    __syncthreads();
    const int nblk = (len + PB - 1) / PB;
    const bool scalar_ret = !VEC && hy.apf_mode != 0;
    bool ok = true;
    float lsum = 0.f;
    auto len_of = [&](int b) { return min(PB, len - b * PB); };
    auto th_of = [&](int b) { return lane < len_of(b) ? (uint32_t)((t0 + b * PB + lane) * H + h) : NO_ROW; };   // lane j: token j
    if (warp < 0) {
        // idle
    } else if (warp < P::CORE) {
        const size_t at = ((size_t)s * H + h) * K + warp * 64 + lane * 2;
        const float2 d0 = a.d0 ? load2(a.d0 + at) : make_float2(1.0f, 1.0f);
        float2 y = make_float2(p1_y(d0.x, q), p1_y(d0.y, q));
        float guess = 0.f;
        uint32_t rounds = 0;
        for (int b = 0; b < nblk; ++b) {
            ok = bar_sync_and<P::CORE * 32>(3, p1_mbar_wait(&sh.bars.full[b % PN], (b / PN) & 1, nullptr));
            if (!ok) break;
            core_block<TI, K, VEC, MANY>(sh, sh.buf[b % PN], len_of(b), y, guess, rounds, hy, q, warp, lane);
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.done[b % PN]);
        }
        if (a.d_final && ok) *reinterpret_cast<float2*>(a.d_final + at) = nblk > 0 ? make_float2(p1_d(y.x, q), p1_d(y.y, q)) : d0;
    } else if (warp < P::FINISH0) {
        auto start = [&](int b) {
            if (b >= PN) ok = p1_mbar_wait(&sh.bars.free_[b % PN], ((b / PN) - 1) & 1, nullptr);
            if (!ok) return;
            PipeBuf<TI, K, VEC>& B = sh.buf[b % PN];
            const uint32_t th = th_of(b);
            fetch_rows<TI, K>(&B.k[0][0], static_cast<const TI*>(a.k), th, PB, lane);
            if constexpr (VEC) fetch_rows<float, K>(&B.rv[0][0], a.retsrc, th, PB, lane);
            if (th != NO_ROW) {
                cp_async4(&B.raw[3][lane], a.beta + th);
                if (scalar_ret) cp_async4(&B.raw[2][lane], a.retsrc + th);
            }
            cp_async_commit();
        };
        int b = warp - P::FETCH0;
        if (b < nblk) start(b);
        for (; b < nblk && ok; b += P::FETCH) {
            cp_async_wait<0>();
            __syncwarp();
            PipeBuf<TI, K, VEC>& B = sh.buf[b % PN];
            float x[PB];
#pragma unroll
            for (int j = 0; j < PB; ++j) {
                float kk[R];
                load_row<R>(B.k[j], lane, kk);
                x[j] = 0.f;
#pragma unroll
                for (int r = 0; r < R; ++r) x[j] = fmaf(kk[r], kk[r], x[j]);
            }
            const float sumk = transpose_sum(x, lane);
            float4 sc = make_float4(0.f, 0.f, 0.f, 0.f);
            float rho = 1.f;
            if (lane < len_of(b)) {
                sc = p1_scalars(sumk, sumk, B.raw[3][lane], hy, q);
                if (scalar_ret) rho = expf(B.raw[2][lane]);
            }
            B.scal[lane] = sc;
            B.rho[lane] = rho;
            B.off[lane] = p1_off(rho, q);
            if (lane == 0) B.jump = 0u;
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.full[b % PN]);
            if (b + P::FETCH < nblk) start(b + P::FETCH);
        }
        cp_async_wait<0>();
    } else {
        TO* kt = static_cast<TO*>(a.ktil);
        for (int b = warp - P::FINISH0; b < nblk; b += P::FINISH) {
            ok = p1_mbar_wait(&sh.bars.done[b % PN], (b / PN) & 1, nullptr);
            if (!ok) break;
            const PipeBuf<TI, K, VEC>& B = sh.buf[b % PN];
            const int n = len_of(b);
            const uint32_t mine = th_of(b);
            if (kt)
                finish_block<TI, K, VEC>(B, n, hy, q, lane, [&](int j, const float (&d)[R], const float (&kk)[R], unsigned) {
                    const size_t th = __shfl_sync(0xffffffffu, mine, j);
                    float wk[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) wk[r] = d[r] * kk[r];
                    store_row<R>(kt + th * K, lane, wk);
                });
            if (a.ratio || a.log_sum) {
                // residual ratio of the write of a token (token-local theorem): the loss |S k - v|^2 after the
                // write over the loss before it is (1 - beta <d_t, k^2>)^2, with the write strength beta itself
                // (whether or not the step of d is beta-aware) and the d the write key was formed with
                float lq = 0.f;
                if (lane < n) {
                    const float fac = 1.0f - B.raw[3][lane] * fmaf(q.w, B.res[lane].y, q.lo * B.scal[lane].w);
                    const float qt = fac * fac;
                    if (a.ratio) a.ratio[mine] = qt;
                    lq = logf(fmaxf(qt, 1.17549435e-38f));
                }
                lsum += warp_sum(lq);
            }
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.free_[b % PN]);
        }
    }
    if (a.log_sum) {   // the finishing warps' shares, always in the same order
        if (warp >= P::FINISH0 && lane == 0) log_part[warp - P::FINISH0] = lsum;
        __syncthreads();
        if (threadIdx.x == 0) {
            float sum = log_part[0];
#pragma unroll
            for (int x = 1; x < P::FINISH; ++x) sum += log_part[x];
            a.log_sum[(size_t)s * H + h] = sum;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------------------------
struct P1Bwd {
    int S, H, NT;
    Table tab;
    const void* k;
    const float *beta, *dktil, *dkread, *dprecond_out;
    const float* log_ret;   // [T,H,K], vector retention only
    void* dk;
    float *dbeta, *dgate, *dlog_ret, *dprecond_in;
    P1Regions r;
    Hyper hy;
    int* status;
    ClearList clear;
};

// skipped tokens: dk = dk_read + d_min dL/dktil (one warp per (chunk, head, 32-token half))
template <typename T, int K>
__global__ void __launch_bounds__(128) phase1_bwd_bulk_kernel(P1Bwd a)
{
    constexpr int R = K / 32;
    pdl_release();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const long w = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long tile = w >> 1;
    const int half = (int)(w & 1);
    if (tile >= (long)a.NT * a.H) return;
    const int c = (int)(tile / a.H), h = (int)(tile % a.H);
    const int len = a.tab.chunk_len(c), tok0 = a.tab.chunk_tok0(c);
    const unsigned word = a.r.skipw[tile * 2 + half] & (unsigned)(len - half * 32 >= 32 ? ~0u : len > half * 32 ? (1u << (len - half * 32)) - 1u : 0u);
    T* dkp = static_cast<T*>(a.dk);
    constexpr int AHEAD = 8;   // rows of eight tokens in flight (one at a time: 18 us for 4000 tokens, 4 heads of 64)
#pragma unroll 1
    for (int j0 = 0; j0 < 32; j0 += AHEAD) {
        if (!((word >> j0) & ((1u << AHEAD) - 1u))) continue;
        float x[AHEAD][R], y[AHEAD][R];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u)
            if ((word >> (j0 + u)) & 1u) {
                const size_t th = (size_t)(tok0 + half * 32 + j0 + u) * a.H + h;
                load_row<R>(a.dkread + th * K, lane, x[u]);
                load_row<R>(a.dktil + th * K, lane, y[u]);
            }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u)
            if ((word >> (j0 + u)) & 1u) {
                const size_t th = (size_t)(tok0 + half * 32 + j0 + u) * a.H + h;
#pragma unroll
                for (int r = 0; r < R; ++r) x[u][r] = fmaf(a.hy.d_min, y[u][r], x[u][r]);
                store_row<R>(dkp + th * K, lane, x[u]);
            }
    }
}

// ---------------------------------------------------------------------------------------------
// The reverse pass over the processed tokens of a chain, last one first:
//   lambda <- mask (.) lambda ;  u = <lambda, k^2> ;  lambda <- rho lambda - a2 u k^2 + k (.) dL/dktil
// (lambda = dL/dd behind the token).  It is the forward pass's problem once more (u_t depends on lambda_t, hence on the u
// of the tokens behind it, by the same weak coupling), linear this time, and is solved the same way: the u of a block of
// PB tokens together, in rounds.  A round's u is taken when lambda is unchanged to its precision: a2 |change of u| max k^2
// at most 2^-24 of the block's largest |u| / n (a weighted mean of |lambda|), or a unit in the last place of u.
// A skipped token's mask is all zero, so lambda restarts there from k (.) dL/dktil: where a processed token's upper
// neighbour was skipped, that neighbour goes into the list as well, with its mask and its step taken as zero, and
// nothing is written for it.  Warps and ring as in the forward pass (the finishing warps form dk and the retention and
// beta gradients and read d_t and dk_read, which the core does not need, from global memory, four tokens ahead).
// In isolation a block of 32 takes 2200 cycles at a step size of 0.003 (two rounds), 3700 at 0.3 (four).
// ---------------------------------------------------------------------------------------------
template <typename T, int K, bool VEC> struct RevBuf {
    T k[PB][K];
    float dkt[PB][K];
    unsigned mask[PB][32];
    float lam0[K];                          // core: lambda on entry to the block
    float raw[5][PB];                       // sum k^2, max k^2, retention, beta, <d_t, k^2> as they sit in memory
    float4 scal[PB];                        // a2, rho, max k^2, 1 / n
    float4 grad[PB];                        // c, factor of the beta gradient, of the normaliser's, u (by the core)
    float rho[PB];
    unsigned restart;                       // bit j: a skipped token, there to restart lambda
    alignas(16) float rv[VEC ? PB : 1][VEC ? K : 1];   // vector retention: l_t, then (core) exp(l_t)
};
template <typename T, int K, bool VEC> struct RevShared {
    static constexpr int CW = K / 32, QN = ring_depth(sizeof(RevBuf<T, K, VEC>), 216 * 1024, Pipe<K>::FINISH);
    static_assert(QN >= 3 && QN % Pipe<K>::FETCH == 0 && QN % Pipe<K>::FINISH == 0, "a buffer belongs to one fetching and one finishing warp");
    RevBuf<T, K, VEC> buf[QN];
    float lam[K];                           // between two lists
    float au[CW][PB];                       // a core warp's -a2 u of the round
    float part[2][CW][PB];
    unsigned long long words[SCAN_CHUNKS];
    uint16_t list[32 * CH + 8];             // bit 15: a restart
    int cmd_tok, cmd_n, live;
    PipeBars bars;
};

// The factors of a processed token: scal and grad (without u).
__device__ __forceinline__ void rev_scalars(float sumk, float kmax, float rho, float beta, float al, const Hyper& hy, float4& sc, float4& gr)
{
    const float b = hy.beta_aware ? beta : 1.0f, rn = 1.0f / fmaxf(sumk, hy.eps);
    const float e = hy.eta * b * rn, a2 = e * b, cc = fmaf(-a2, al, e);
    sc = make_float4(a2, rho, kmax, rn);
    gr = make_float4(cc, hy.eta * (1.0f - 2.0f * b * al) * rn, sumk > hy.eps ? -cc * rn : 0.f, 0.f);
}
__device__ __forceinline__ float rev_step(float lm, float kap, float w, float au, float rho) { return fmaf(rho, lm, fmaf(au, kap, w)); }

template <typename T, int K, bool VEC>
__device__ __forceinline__ void rev_core_block(RevShared<T, K, VEC>& sh, RevBuf<T, K, VEC>& B, int n, float& lam, uint32_t& rounds, int warp, int lane)
{
    constexpr int CW = K / 32, R = K / 32;
    const int i = warp * 32 + lane;
    float kap[PB], w[PB];
    unsigned pass = 0;
#pragma unroll
    for (int j = 0; j < PB; ++j) {
        const float k = ldf(&B.k[j][i]);
        kap[j] = __fmul_rn(k, k);
        w[j] = __fmul_rn(k, B.dkt[j][i]);
        pass |= ((B.mask[j][i / R] >> (i % R)) & 1u) << j;
    }
    pass &= ~B.restart;
    if constexpr (VEC) {
#pragma unroll 4
        for (int j = 0; j < PB; ++j) {
            float& v = B.rv[VEC ? j : 0][VEC ? i : 0];
            v = j < n ? expf(v) : 1.0f;
        }
    }
    B.lam0[i] = lam;
    const float4 sc = B.scal[lane];   // lane j: token j
    float u = 0.f, un = 0.f, l = lam;   // un: the sums of the latest lambda
    for (int round = 0; round <= PB; ++round) {
        const uint32_t par = rounds++ & 1;
        sh.au[warp][lane] = -sc.x * u;
        __syncwarp();
        float p[PB];
        l = lam;
#pragma unroll
        for (int j = 0; j < PB; j += 4) {
            const float4 u4 = *reinterpret_cast<const float4*>(&sh.au[warp][j]), r4 = *reinterpret_cast<const float4*>(B.rho + j);
            const float au[4] = {u4.x, u4.y, u4.z, u4.w}, rs[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float rho = VEC ? B.rv[VEC ? j + x : 0][VEC ? i : 0] : rs[x];
                const float lm = bit_of(pass, j + x) ? l : 0.f;
                p[j + x] = lm * kap[j + x];
                l = rev_step(lm, kap[j + x], w[j + x], au[x], rho);
            }
        }
        const float mine = transpose_sum(p, lane);
        float(*part)[PB] = sh.part[par];
        part[warp][lane] = mine;
        bar_sync<CW * 32>(3);
        un = part[0][lane];
#pragma unroll
        for (int x = 1; x < CW; ++x) un += part[x][lane];
        const float du = fabsf(un - u);
        const float size = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(un) * sc.w)));
        if (__all_sync(0xffffffffu, du * sc.x * sc.z <= 5.9604645e-8f * size || du <= 1.1920929e-7f * fabsf(un) || lane >= n)) break;
        u = un;
    }
    lam = l;
    if (warp == 0) B.grad[lane].w = un;   // (a small a2 lets lambda stand before u does: the gradients need u itself)
}

// What a processed token leaves: dk and, where one per coordinate is asked for, the retention gradient.
template <typename T, int K, bool VEC>
__device__ __forceinline__ void rev_outputs(const P1Bwd& a, size_t th, int lane, const float4& g, float a2, const float (&kk)[K / 32],
                                            const float (&dt)[K / 32], const float (&dkt)[K / 32], const float (&dkr)[K / 32],
                                            const float (&lm)[K / 32], const float (&rv)[K / 32])
{
    constexpr int R = K / 32;
    const float da = -a2 * g.w, dn = g.z * g.w;
    if constexpr (VEC) {   // r_i lambda_i d_i
        if (a.dlog_ret) {
            float dl[R];
#pragma unroll
            for (int r = 0; r < R; ++r) dl[r] = rv[r] * lm[r] * dt[r];
            store_row<R>(a.dlog_ret + th * K, lane, dl);
        }
    }
    float out[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float dkap = g.x * lm[r] + da * dt[r] + dn;
        out[r] = dkr[r] + dt[r] * dkt[r] + 2.0f * kk[r] * dkap;
    }
    store_row<R>(static_cast<T*>(a.dk) + th * K, lane, out);
}
// The per-token scalar gradients, added on top of what the chunk-local backward wrote (as reductions without a return
// value, so that nobody waits for memory); dr = <lambda, d_t>.
__device__ __forceinline__ void rev_scalar_grads(const P1Bwd& a, size_t th, const float4& g, float rho, float dr)
{
    if (a.hy.beta_aware) atomicAdd(&a.dbeta[th], g.y * g.w);
    if (a.hy.apf_mode == 1) atomicAdd(&a.dgate[th], rho * dr);
    if (a.hy.apf_mode == 2 && a.dlog_ret) a.dlog_ret[th] = rho * dr;
}

template <typename T, int K, bool VEC>
__device__ __forceinline__ bool run_rev_list(const P1Bwd& a, int h, RevShared<T, K, VEC>& sh, uint32_t& rounds, uint32_t& uses, int warp, int lane)
{
    constexpr int R = K / 32;
    using P = Pipe<K>;
    constexpr int QN = RevShared<T, K, VEC>::QN;
    const int H = a.H;
    const int tok0 = sh.cmd_tok, total = sh.cmd_n;
    const int nblk = (total + PB - 1) / PB;
    bool ok = true;
    const uint32_t base = uses;
    auto entry = [&](int idx) { return (int)sh.list[total - 1 - idx]; };   // from the last token on
    auto len_of = [&](int b) { return min(PB, total - b * PB); };
    auto th_of = [&](int b) {   // lane j: token j
        return lane < len_of(b) ? (uint32_t)((tok0 + (entry(b * PB + lane) & 0x7fff)) * H + h) : NO_ROW;
    };
    if (warp < P::CORE) {
        float lam = sh.lam[warp * 32 + lane];
        for (int b = 0; b < nblk; ++b) {
            const int bi = (base + b) % QN;
            ok = bar_sync_and<P::CORE * 32>(3, p1_mbar_wait(&sh.bars.full[bi], ((base + b) / QN) & 1, a.status));
            if (!ok) break;
            rev_core_block<T, K, VEC>(sh, sh.buf[bi], len_of(b), lam, rounds, warp, lane);
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.done[bi]);
        }
        sh.lam[warp * 32 + lane] = lam;
    } else if (warp < P::FINISH0) {
        auto start = [&](int b) {
            const uint32_t use = base + b;
            const int bi = use % QN;
            if (use >= QN) ok = p1_mbar_wait(&sh.bars.free_[bi], ((use / QN) - 1) & 1, a.status);
            if (!ok) return;
            RevBuf<T, K, VEC>& B = sh.buf[bi];
            const uint32_t th = th_of(b);
            fetch_rows<T, K>(&B.k[0][0], static_cast<const T*>(a.k), th, PB, lane);
            fetch_rows<float, K>(&B.dkt[0][0], a.dktil, th, PB, lane);
            fetch_rows<unsigned, 32>(&B.mask[0][0], a.r.pmask, th, PB, lane);
            if constexpr (VEC) fetch_rows<float, K>(&B.rv[0][0], a.log_ret, th, PB, lane);
            if (th != NO_ROW) {
                cp_async4(&B.raw[0][lane], a.r.sumk + th);
                cp_async4(&B.raw[1][lane], a.r.kmax + th);
                cp_async4(&B.raw[2][lane], a.r.rho + th);
                cp_async4(&B.raw[3][lane], a.beta + th);
                cp_async4(&B.raw[4][lane], a.r.al + th);
                for (int o = 0; o < K * 4; o += 128) {   // what the finishing warps will read
                    prefetch_l2(reinterpret_cast<const char*>(a.r.dtraj + (size_t)th * K) + o);
                    prefetch_l2(reinterpret_cast<const char*>(a.dkread + (size_t)th * K) + o);
                }
            }
            cp_async_commit();
        };
        auto complete = [&](int b) {
            const int bi = (base + b) % QN;
            RevBuf<T, K, VEC>& B = sh.buf[bi];
            const int n = len_of(b);
            // an empty slot has to leave lambda alone: mask all ones, rho = 1 (k = 0)
            float4 sc = make_float4(0.f, 1.f, 0.f, 0.f), gr = make_float4(0.f, 0.f, 0.f, 0.f);
            bool skipped = false;
            if (lane < n) {
                skipped = (entry(b * PB + lane) & 0x8000) != 0;
                if (!skipped) rev_scalars(B.raw[0][lane], B.raw[1][lane], B.raw[2][lane], B.raw[3][lane], B.raw[4][lane], a.hy, sc, gr);
            }
            const unsigned restarts = __ballot_sync(0xffffffffu, skipped);
            B.scal[lane] = sc;
            B.grad[lane] = gr;
            B.rho[lane] = sc.y;
            if (lane == 0) B.restart = restarts;
            for (int j = n; j < PB; ++j) B.mask[j][lane] = 0xffffffffu;
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.full[bi]);
        };
        int b = (int)((warp - P::FETCH0 + base) & 1);
        if (b < nblk) start(b);
        for (; b < nblk && ok; b += 2) {
            cp_async_wait<0>();
            __syncwarp();
            complete(b);
            if (b + 2 < nblk) start(b + 2);
        }
        cp_async_wait<0>();
    } else {
        for (int b = (int)((warp - P::FINISH0 - base) & (P::FINISH - 1)); b < nblk; b += P::FINISH) {
            const int bi = (base + b) % QN;
            const RevBuf<T, K, VEC>& B = sh.buf[bi];
            const int n = len_of(b);
            const uint32_t mine = th_of(b);
            struct Ahead {
                float dt[4][R], dkr[4][R];
            } even, odd;
            auto load = [&](int j0, Ahead& x) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const size_t th = __shfl_sync(0xffffffffu, mine, min(j0 + j, n - 1));
                    load_row<R>(a.r.dtraj + th * K, lane, x.dt[j]);
                    load_row<R>(a.dkread + th * K, lane, x.dkr[j]);
                }
            };
            load(0, even);
            ok = p1_mbar_wait(&sh.bars.done[bi], ((base + b) / QN) & 1, a.status);
            if (!ok) break;
            const unsigned restart = B.restart;
            float lam[R];
            load_row<R>(B.lam0, lane, lam);
            auto work = [&](int j0, const Ahead& x) {
                float drv[4];
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int j = j0 + jj;
                    float kk[R], dkt[R], lm[R], rv[R];
                    load_row<R>(B.k[j], lane, kk);
                    load_row<R>(B.dkt[j], lane, dkt);
                    const unsigned mw = bit_of(restart, j) ? 0u : B.mask[j][lane];
                    const float4 sc = B.scal[j], g = B.grad[j];
                    if constexpr (VEC) load_row<R>(B.rv[VEC ? j : 0], lane, rv);
                    else {
#pragma unroll
                        for (int r = 0; r < R; ++r) rv[r] = sc.y;
                    }
                    drv[jj] = 0.f;
                    const float au = -sc.x * g.w;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        lm[r] = bit_of(mw, r) ? lam[r] : 0.f;
                        drv[jj] = fmaf(lm[r], x.dt[jj][r], drv[jj]);
                        lam[r] = rev_step(lm[r], __fmul_rn(kk[r], kk[r]), __fmul_rn(kk[r], dkt[r]), au, rv[r]);
                    }
                    const size_t th = __shfl_sync(0xffffffffu, mine, j);
                    if (j < n && !bit_of(restart, j)) rev_outputs<T, K, VEC>(a, th, lane, g, sc.x, kk, x.dt[jj], dkt, x.dkr[jj], lm, rv);
                }
                const float dr = transpose_sum(drv, lane);   // lane j: token j0 + j
                const int j = (j0 + lane) & (PB - 1);
                const size_t th = __shfl_sync(0xffffffffu, mine, j);
                if (lane < 4 && j < n && !bit_of(restart, j)) rev_scalar_grads(a, th, B.grad[j], B.scal[j].y, dr);
            };
#pragma unroll 1
            for (int j0 = 0; j0 < n; j0 += 8) {
                load(j0 + 4, odd);
                work(j0, even);
                load(j0 + 8, even);
                if (j0 + 4 < n) work(j0 + 4, odd);
            }
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&sh.bars.free_[bi]);
        }
    }
    uses = base + nblk;
    return ok;
}

// A list of at most PB entries by warp 0 alone, token by token.
template <typename T, int K, bool VEC>
__device__ __forceinline__ void walk_rev_list(const P1Bwd& a, int h, RevShared<T, K, VEC>& sh, int tok0, int n, int lane)
{
    constexpr int R = K / 32;
    const int H = a.H;
    RevBuf<T, K, VEC>& B = sh.buf[0];
    const uint32_t mine = lane < n ? (uint32_t)((tok0 + ((int)sh.list[n - 1 - lane] & 0x7fff)) * H + h) : NO_ROW;
    fetch_rows<T, K>(&B.k[0][0], static_cast<const T*>(a.k), mine, n, lane);
    fetch_rows<float, K>(&B.dkt[0][0], a.dktil, mine, n, lane);
    fetch_rows<unsigned, 32>(&B.mask[0][0], a.r.pmask, mine, n, lane);
    fetch_rows<float, K>(&sh.buf[1].dkt[0][0], a.r.dtraj, mine, n, lane);
    fetch_rows<float, K>(&sh.buf[2].dkt[0][0], a.dkread, mine, n, lane);
    if constexpr (VEC) fetch_rows<float, K>(&B.rv[0][0], a.log_ret, mine, n, lane);
    cp_async_commit();
    if (lane < n) {
        float4 sc, gr;
        rev_scalars(a.r.sumk[mine], a.r.kmax[mine], a.r.rho[mine], a.beta[mine], a.r.al[mine], a.hy, sc, gr);
        B.scal[lane] = sc;
        B.grad[lane] = gr;
    }
    float lam[R];
    load_row<R>(sh.lam, lane, lam);
    cp_async_wait<0>();
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const float4 sc = B.scal[j];
        float4 g = B.grad[j];
        float kk[R], dkt[R], dt[R], dkr[R], lm[R], rv[R], u = 0.f, dr = 0.f;
        load_row<R>(B.k[j], lane, kk);
        load_row<R>(B.dkt[j], lane, dkt);
        if (sh.list[n - 1 - j] & 0x8000) {   // a restart
#pragma unroll
            for (int r = 0; r < R; ++r) lam[r] = kk[r] * dkt[r];
            continue;
        }
        load_row<R>(sh.buf[1].dkt[j], lane, dt);
        load_row<R>(sh.buf[2].dkt[j], lane, dkr);
        if constexpr (VEC) {
            load_row<R>(B.rv[VEC ? j : 0], lane, rv);
#pragma unroll
            for (int r = 0; r < R; ++r) rv[r] = expf(rv[r]);
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) rv[r] = sc.y;
        }
        const unsigned mw = B.mask[j][lane];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            lm[r] = bit_of(mw, r) ? lam[r] : 0.f;
            u = fmaf(lm[r], kk[r] * kk[r], u);
            dr = fmaf(lm[r], dt[r], dr);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            u += __shfl_xor_sync(0xffffffffu, u, o);
            dr += __shfl_xor_sync(0xffffffffu, dr, o);
        }
        g.w = u;
        const float au = -sc.x * u;
#pragma unroll
        for (int r = 0; r < R; ++r) lam[r] = rev_step(lm[r], kk[r] * kk[r], kk[r] * dkt[r], au, rv[r]);
        const size_t th = __shfl_sync(0xffffffffu, mine, j);
        rev_outputs<T, K, VEC>(a, th, lane, g, sc.x, kk, dt, dkt, dkr, lm, rv);
        if (lane == 0) rev_scalar_grads(a, th, g, sc.y, dr);
    }
    store_row<R>(sh.lam, lane, lam);
    __syncwarp();
}

// Skip words are taken 32 chunks at a time, the last ones first, and their processed tokens (with the restarts
// between them) are one list.  Warp 0 walks short lists itself.
template <typename T, int K, bool VEC> struct RevPlan {
    const P1Bwd& a;
    RevShared<T, K, VEC>& sh;
    const int h, lane, c0, c1, seq_t0, seq_len;
    int g, scanned = -1;
    bool live = true;   // the token above the group was processed (at the end: the sequence's first one): lambda holds

    __device__ __forceinline__ RevPlan(const P1Bwd& a_, RevShared<T, K, VEC>& sh_, int s, int h_, int lane_)
        : a(a_), sh(sh_), h(h_), lane(lane_), c0(a_.tab.seq_chunk0(s)), c1(a_.tab.seq_chunk0(s + 1)), seq_t0(a_.tab.seq_tok0(s)),
          seq_len(a_.tab.seq_len(s)), g(c1 > c0 ? (c1 - c0 - 1) >> 5 : -1)
    {
    }
    __device__ __forceinline__ void next()
    {
        for (; g >= 0; --g) {
            const int top = g * 32 / SCAN_CHUNKS;
            if (top != scanned) scan_words(sh.words, a.r.skipw, c0 + top * SCAN_CHUNKS, c0, c1, seq_len, a.H, h, lane);
            scanned = top;
            const int base = g * 32 * CH, glen = min(32 * CH, seq_len - base);
            const unsigned long long valid = valid_bits(glen - 64 * lane), proc = sh.words[g * 32 % SCAN_CHUNKS + lane];
            unsigned long long up = __shfl_up_sync(0xffffffffu, proc, 1) >> 63;
            if (lane == 0) up = 0ull;
            const unsigned long long restart = ((proc << 1) | up) & ~proc & valid;
            const bool above = live;
            const unsigned long long last = __shfl_sync(0xffffffffu, proc, (glen - 1) / CH);
            live = (__shfl_sync(0xffffffffu, proc, 0) & 1ull) != 0ull;
            if (!__any_sync(0xffffffffu, proc != 0ull)) continue;
            int n = write_list(sh.list, proc | restart, restart, 32 * CH, lane);
            if (((last >> ((glen - 1) % CH)) & 1ull) && !above) {   // (the sequence goes on above: `above` starts out true)
                if (lane == 0) sh.list[n] = (uint16_t)(glen | 0x8000);
                __syncwarp();
                ++n;
            }
            if (n <= PB) {
                walk_rev_list<T, K, VEC>(a, h, sh, seq_t0 + base, n, lane);
                continue;
            }
            if (lane == 0) {
                sh.cmd_tok = seq_t0 + base;
                sh.cmd_n = n;
            }
            --g;
            return;
        }
        if (lane == 0) {
            sh.cmd_n = 0;
            sh.live = live;
        }
    }
};

// One chain per CTA.
template <typename T, int K, bool VEC>
__global__ void __launch_bounds__(Pipe<K>::THREADS, 1) phase1_bwd_seq_kernel(P1Bwd a)
{
    using P = Pipe<K>;
    extern __shared__ __align__(16) uint8_t p1_dyn[];
    RevShared<T, K, VEC>& sh = *reinterpret_cast<RevShared<T, K, VEC>*>(p1_dyn);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chain = blockIdx.x;
    const int s = chain / a.H, h = chain % a.H, H = a.H;
    const int coord = warp * 32 + lane;   // core warps
    const size_t mine = ((size_t)s * H + h) * K + coord;
    if (threadIdx.x == 0) init_bars(sh.bars, RevShared<T, K, VEC>::QN, P::CORE);
    pdl_wait();   // no early release: the next call's parallel pass would crowd on the SMs that this one leaves idle (8 x 2048 tokens: + 5 us)
    clear_regions(a.clear);
    if (warp < P::CORE) sh.lam[coord] = a.dprecond_out ? a.dprecond_out[mine] : 0.f;
    uint32_t rounds = 0, uses = 0;
    __syncthreads();
    RevPlan<T, K, VEC> plan(a, sh, s, h, lane);
    while (true) {
        if (warp == 0) plan.next();
        bar_sync<P::THREADS>(1);
        if (sh.cmd_n == 0) break;
        if (!run_rev_list<T, K, VEC>(a, h, sh, rounds, uses, warp, lane)) plan.g = -1;
        bar_sync<P::THREADS>(2);
    }
    if (a.dprecond_in && warp < P::CORE) {
        float lam = sh.lam[coord];
        if (!sh.live) {   // the first token was skipped: lambda restarts there
            const size_t th = (size_t)a.tab.seq_tok0(s) * H + h;
            lam = ldf(static_cast<const T*>(a.k) + th * K + coord) * a.dktil[th * K + coord];
        }
        a.dprecond_in[mine] = lam;
    }
}

// The kernel variant for a number of chains; launch(VEC, MANY) gets the two as types.  The line is where the chains no longer
// have an SM each (stand-alone update, 1024 moving tokens: 144 chains 74 us one to an SM; 160 chains 136 us that way, 95 us
// sharing).
template <typename F> bool p1_variant(bool vec, unsigned chains, F launch)
{
    const bool many = chains > (unsigned)num_sms();
    if (vec) return many ? launch(std::true_type(), std::true_type()) : launch(std::true_type(), std::false_type());
    return many ? launch(std::false_type(), std::true_type()) : launch(std::false_type(), std::false_type());
}

template <typename TI, typename TO, int K>
int fwd_launch(const P1Fwd& a, cudaStream_t st)
{
    const long warps = (long)a.NT * a.H * 2;
    const unsigned gspec = (unsigned)((warps + 3) / 4);
    stage_mark(st, "phase1_spec");
    if (!launch_after(a.hy.apf_mode == 3 ? phase1_spec_kernel<TI, TO, K, true> : phase1_spec_kernel<TI, TO, K, false>, gspec, 128, 0, st, a)) return -1;
    stage_mark(st, "phase1_seq");
    const unsigned chains = (unsigned)(a.S * a.H);
    const bool okl = p1_variant(a.hy.apf_mode == 3, chains, [&](auto vec, auto many) {
        constexpr bool VEC = decltype(vec)::value, MANY = decltype(many)::value;
        constexpr size_t smem = sizeof(PipeShared<TI, K, VEC, MANY>);
        const auto kernel = phase1_seq_kernel<TI, TO, K, VEC, MANY>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
        return launch_after(kernel, chains, FwdPipe<K, MANY>::THREADS, smem, st, a);
    });
    if (!okl) return -1;
    return cudaGetLastError() == cudaSuccess ? 2 : -1;
}

template <typename T, int K>
int bwd_launch(const P1Bwd& a, bool bulk, cudaStream_t st)
{
    int n = 0;
    if (bulk) {
        const long warps = (long)a.NT * a.H * 2;
        stage_mark(st, "phase1_bwd_bulk");
        if (!launch_after(phase1_bwd_bulk_kernel<T, K>, (unsigned)((warps + 3) / 4), 128, 0, st, a)) return -1;
        ++n;
    }
    stage_mark(st, "phase1_bwd_seq");
    const unsigned chains = (unsigned)(a.S * a.H);
    auto launch_seq = [&](auto kernel, size_t smem) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
        return launch_after(kernel, chains, Pipe<K>::THREADS, smem, st, a);
    };
    if (!(a.hy.apf_mode == 3 ? launch_seq(phase1_bwd_seq_kernel<T, K, true>, sizeof(RevShared<T, K, true>))
                             : launch_seq(phase1_bwd_seq_kernel<T, K, false>, sizeof(RevShared<T, K, false>))))
        return -1;
    ++n;
    return cudaGetLastError() == cudaSuccess ? n : -1;
}

}  // namespace

int phase1_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                   void* ktil, bool ktil_bf16, bool save, const ClearList& clear, cudaStream_t st)
{
    P1Fwd f{};
    f.S = L.S; f.H = p.H; f.NT = L.NTmax; f.tab = carve_table(ws, L);
    f.k = a.k; f.beta = a.beta; f.retsrc = p.apf_mode >= 2 ? a.log_ret : a.gate; f.d0 = a.precond_in;
    f.ktil = ktil; f.d_final = a.precond_out; f.r = carve_p1(ws, L); f.save = save ? 1 : 0; f.hy = hy; f.q = p1_coord(hy);
    f.status = reinterpret_cast<int*>(static_cast<char*>(ws) + L.status);
    f.clear = clear;
    if (L.dense_T) {   // (a packed batch's table kernel has cleared it)
        f.clear.p[2] = f.status;
        f.clear.n[2] = 1;
    }
    if (p.io_dtype == OSDN_FP32) {
        if (ktil_bf16) return -1;
        return p.K == 64 ? fwd_launch<float, float, 64>(f, st) : fwd_launch<float, float, 128>(f, st);
    }
    if (ktil_bf16) return p.K == 128 ? fwd_launch<__nv_bfloat16, __nv_bfloat16, 128>(f, st) : -1;   // (the tensor-core family)
    return p.K == 64 ? fwd_launch<__nv_bfloat16, float, 64>(f, st) : fwd_launch<__nv_bfloat16, float, 128>(f, st);
}

int phase1_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                    const float* dktil, const float* dkread, bool bulk, const ClearList& clear, cudaStream_t st)
{
    P1Bwd b{};
    b.S = L.S; b.H = p.H; b.NT = L.NTmax; b.tab = carve_table(ws, L);
    b.k = a.k; b.beta = a.beta; b.dktil = dktil; b.dkread = dkread; b.dprecond_out = a.dprecond_out;
    b.dk = a.dk; b.dbeta = a.dbeta; b.dgate = a.dgate; b.dlog_ret = a.dlog_ret; b.dprecond_in = a.dprecond_in;
    b.r = carve_p1(ws, L); b.hy = hy; b.log_ret = a.log_ret;
    b.status = reinterpret_cast<int*>(static_cast<char*>(ws) + L.status);
    b.clear = clear;
    // retention gradients are written for processed tokens only; a skipped token (projection mask all
    // zero) has none
    if (p.apf_mode >= 2 && a.dlog_ret) {
        const size_t Ttot = p.nseq > 0 ? (size_t)p.T : (size_t)p.B * p.T;
        const size_t nb = Ttot * p.H * (p.apf_mode == 3 ? (size_t)p.K : 1) * sizeof(float);
        if (cudaMemsetAsync(a.dlog_ret, 0, nb, st) != cudaSuccess) return -1;
    }
    if (p.io_dtype == OSDN_FP32)
        return p.K == 64 ? bwd_launch<float, 64>(b, bulk, st) : bwd_launch<float, 128>(b, bulk, st);
    return p.K == 64 ? bwd_launch<__nv_bfloat16, 64>(b, bulk, st) : bwd_launch<__nv_bfloat16, 128>(b, bulk, st);
}

int phase1_update(const osdn_params& p, const Hyper& hy, const void* k, const float* beta, const float* retsrc,
                  const float* precond_in, void* ktil_out, float* precond_out, float* ratio_out,
                  float* log_sum_out, cudaStream_t st)
{
    P1Args pa{};
    pa.S = p.nseq > 0 ? p.nseq : p.B;
    pa.H = p.H; pa.T_dense = p.T; pa.cu = p.nseq > 0 ? p.cu_seqlens : nullptr;
    pa.k = k; pa.beta = beta; pa.retsrc = retsrc; pa.d0 = precond_in; pa.ktil = ktil_out;
    pa.d_final = precond_out; pa.ratio = ratio_out; pa.log_sum = log_sum_out; pa.hy = hy; pa.q = p1_coord(hy);
    const unsigned chains = (unsigned)(pa.S * pa.H);
    stage_mark(st, "phase1_stream");
    auto typed = [&](auto t, auto kk) {
        using T = decltype(t);
        constexpr int K = decltype(kk)::value;
        return p1_variant(hy.apf_mode == 3, chains, [&](auto vec, auto many) {
            constexpr bool VEC = decltype(vec)::value, MANY = decltype(many)::value;
            constexpr size_t smem = sizeof(PipeShared<T, K, VEC, MANY>);
            const auto kernel = phase1_stream_kernel<T, T, K, VEC, MANY>;
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
            return launch_after(kernel, chains, FwdPipe<K, MANY>::THREADS, smem, st, pa);
        });
    };
    using K64 = std::integral_constant<int, 64>;
    using K128 = std::integral_constant<int, 128>;
    const bool ok = p.io_dtype == OSDN_FP32 ? (p.K == 64 ? typed(float(), K64()) : typed(float(), K128()))
                                            : (p.K == 64 ? typed(__nv_bfloat16(), K64()) : typed(__nv_bfloat16(), K128()));
    if (!ok) return -1;
    stage_end(st);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace osdn
