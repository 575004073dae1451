// CUDA-core (fp32 FMA) kernels of the OSDN layer.
//
// This family is the fp32 mode of the library (fp32 I/O needs better than TF32 accuracy)
// and the reference-quality path for bf16 I/O when OSDN_FLAG_FORCE_SIMT is set.  Every
// step of the chunkwise algorithm runs in fp32; phase 2 is in osdn_simt.cuh:
//
//   chunk_local_fwd decay-ratio Gram A, UT inverse T, W, U, local scores P  (gated chunk form)
//   chain_fwd       dU = U - W S^T ; S <- gamma_C S + dU^T (rho Ktil)   (state recurrence)
//   output          O = scale[(gamma Q) S^T + P dU]
//   pre_bwd, chain_bwd  reverse state chain: ddU and dS (their parts that need no dS first)
//   chunk_local_bwd all chunk-local gradients (through P, the state's advance, the right side of the solve, A and the gate prefix)
//
// This file also builds the chunk table of packed batches.
#include "osdn_simt.cuh"

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
    pdl_wait();
    if (tid == 0) {
        s_carry = 0;
        if (status) *status = 0;
    }
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

template <typename T, int K, int V>
int forward_typed(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, bool save, cudaStream_t st)
{
    const int n1 = phase1_forward(p, hy, L, ws, a, static_cast<char*>(ws) + L.ktil, false, save, ClearList{}, st);
    if (n1 < 0) return -1;
    const int n2 = chunk_forward<T, K, V, false>(p, hy, L, ws, a, nullptr, st);
    stage_end(st);
    return n2 < 0 ? -1 : n1 + n2;
}

template <typename T, int K, int V>
int backward_typed(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    const int n2 = chunk_backward<T, K, V, false>(p, hy, L, ws, a, nullptr, st);
    if (n2 < 0) return -1;
    const int n1 = phase1_backward(p, hy, L, ws, a, reinterpret_cast<float*>(w + L.dktil), reinterpret_cast<float*>(w + L.dkread), true, ClearList{}, st);
    stage_end(st);
    return n1 < 0 ? -1 : n1 + n2;
}

}  // namespace

int launch_build_table(const osdn_params& p, const WsLayout& L, void* ws, cudaStream_t st)
{
    Table tab = carve_table(ws, L);
    if (L.dense_T) return 0;   // dense batch: the table is arithmetic, nothing to build
    stage_mark(st, "build_table");
    return launch_after(build_table_kernel, 1, TBL_THREADS, 0, st, L.S, p.T, p.cu_seqlens, L.NTmax, tab, reinterpret_cast<int*>(static_cast<char*>(ws) + L.status)) ? 1 : -1;
}

int simt_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                 bool save, cudaStream_t st)
{
    OSDN_DISPATCH(forward_typed, p, hy, L, ws, a, save, st);
}

int simt_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                  cudaStream_t st)
{
    OSDN_DISPATCH(backward_typed, p, hy, L, ws, a, st);
}

}  // namespace osdn
