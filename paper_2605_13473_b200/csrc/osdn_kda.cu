// Online-scaled delta rule with a channel gate (the OSKDA backbone extension: Kimi Delta Attention with
// Online Scaling).  The scalar gate exp(g_t) of the layer becomes one gate per key channel,
//     Sbar = S_{t-1} Diag(alpha_t),  u = v_t - Sbar k_t,  S_t = Sbar + beta_t u ktil_t^T,  o_t = scale S_t q_t,
// with the state kept V x K as everywhere in this library (the paper's K x V state is its transpose).
// Phase 1 (preconditioner, write keys, their adjoint) is the layer's own and is reused unchanged; phase 2 is the
// chunk form of the appendix in fp32 on CUDA cores (osdn_simt.cuh), which the scalar-gate fp32 layer shares.  A
// token-by-token walk of the state rows, bound by the instructions of two warp-wide dot products per row and token
// (and, backward, by three walks over every chunk), took 1.7 ms forward and 7.3 ms backward at 8 x 2048 tokens,
// 8 heads of 128.
#include "osdn_simt.cuh"

namespace osdn {

// The in-chunk gate prefix of every tile (high and low parts), which the backward reads again.
size_t kda_extra_bytes(const osdn_params& p, const WsLayout& L, bool need_bwd)
{
    return need_bwd ? align_up((size_t)L.NTmax * p.H * 2 * CH * p.K * 4, 256) : 0;
}

namespace {
float* prefix_region(const WsLayout& L, void* ws)
{
    return reinterpret_cast<float*>(static_cast<char*>(ws) + align_up(L.total, 256));
}
template <typename T, int K, int V>
int forward_typed(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, bool save, cudaStream_t st)
{
    return chunk_forward<T, K, V, true>(p, hy, L, ws, a, save ? prefix_region(L, ws) : nullptr, st);
}
template <typename T, int K, int V>
int backward_typed(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, cudaStream_t st)
{
    return chunk_backward<T, K, V, true>(p, hy, L, ws, a, prefix_region(L, ws), st);
}
int phase2_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, bool save, cudaStream_t st)
{
    OSDN_DISPATCH(forward_typed, p, hy, L, ws, a, save, st);
}
int phase2_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, cudaStream_t st)
{
    OSDN_DISPATCH(backward_typed, p, hy, L, ws, a, st);
}
}  // namespace

int kda_forward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a, bool save,
                cudaStream_t st)
{
    const int n0 = launch_build_table(p, L, ws, st);
    if (n0 < 0) return -1;
    const int n1 = phase1_forward(p, hy, L, ws, a, static_cast<char*>(ws) + L.ktil, false, save, ClearList{}, st);
    if (n1 < 0) return -1;
    const int n2 = phase2_forward(p, hy, L, ws, a, save, st);
    stage_end(st);
    return n2 < 0 ? -1 : n0 + n1 + n2;
}

int kda_backward(const osdn_params& p, const Hyper& hy, const WsLayout& L, void* ws, const Pointers& a,
                 cudaStream_t st)
{
    char* w = static_cast<char*>(ws);
    const int n2 = phase2_backward(p, hy, L, ws, a, st);
    if (n2 < 0) return -1;
    // phase-1 adjoint: dk = dk(read key) + d_t (.) d ktil + preconditioner terms; adds its share to d beta
    const int n1 = phase1_backward(p, hy, L, ws, a, reinterpret_cast<float*>(w + L.dktil), reinterpret_cast<float*>(w + L.dkread), true, ClearList{}, st);
    stage_end(st);
    return n1 < 0 ? -1 : n1 + n2;
}

}  // namespace osdn
