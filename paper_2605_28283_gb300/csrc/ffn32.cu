// Routing of any number of tokens on the CUDA cores (both storage types), and
// the fp32 layer for more tokens than one fused decode launch takes.
//
// fp32 has no tensor-core form that keeps 32 bits, and the fp32 shapes are
// small (the tiny ReLU model: 2 MB of weights), so what bounds a call is
// launches and latency, not bytes: three launches for any token count, each
// with enough independent warps to fill the chip.  Slices of 8 tokens through
// the fused decode kernel took 8 x 28 us at 64 tokens, and the router ran on
// one CTA (29 us): 142 us a call, 12 us now in a graph (23 us issued eagerly).
// Up to 8 tokens the fused kernel's one launch is kept (8 tokens: 13 us against
// 11 us in a graph, but a third of the launches).
//
//   route   a CTA per token (or four): logits, then the selection
//   gate/up a warp per (8 weight rows, group of tokens): coalesced float4 loads
//           along K, every row against every token of the group in registers,
//           one butterfly for all 32 or 64 sums; groups without a token that
//           selected the expert are skipped
//   down    the same over the experts that the group selected
#include "pp_common.cuh"
#include "pp_kernels.h"
#include "pp_launch.h"
#include "pp_select.cuh"

namespace pp {
namespace {

// TB tokens per CTA of 8 warps.  Warp w takes experts w, w + 8, ...; a lane
// every 32nd 16-byte chunk of K.  Bound: L2 latency for few tokens (TB = 1);
// above kRouteOneMax tokens the W_r reads of the CTAs would bound it, and four
// tokens share them.
constexpr int kRouteOneMax = 608;

template <typename TW, int TB>
__global__ void __launch_bounds__(256)
    route_tokens_kernel(const TW* __restrict__ x, int T, int d, const TW* __restrict__ Wr, int E, float p, int rule,
                        int gate, int32_t* ids, int32_t* counts, float* gates, float* logits, uint32_t* bits,
                        float* gexp, unsigned* status) {
    using EL = Elem<TW>;
    constexpr int kEl = EL::kPer16B;
    __shared__ float lg[TB][kMaxExperts];
    __shared__ __align__(16) SelScratch sc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t0 = blockIdx.x * TB, n = min(TB, T - t0);
    const int nchunk = d / kEl;
    pdl_wait();
    pdl_launch_dependents();
    for (int e = warp; e < E; e += 8) {
        const uint4* w = reinterpret_cast<const uint4*>(Wr + (size_t)e * d);
        float acc[TB];
#pragma unroll
        for (int i = 0; i < TB; i++) acc[i] = 0.0f;
#pragma unroll 2
        for (int c = lane; c < nchunk; c += 32) {
            float wf[kEl];
            EL::unpack(w[c], wf);
#pragma unroll
            for (int i = 0; i < TB; i++) {
                if (TB > 1 && i >= n) break;
                float xf[kEl];
                EL::unpack(reinterpret_cast<const uint4*>(x + (size_t)(t0 + i) * d)[c], xf);
#pragma unroll
                for (int q = 0; q < kEl; q++) acc[i] = fmaf(wf[q], xf[q], acc[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < TB; i++) {
            acc[i] = warp_sum(acc[i]);
            if (lane == 0) lg[i][e] = acc[i];
        }
    }
    __syncthreads();
    for (int i = 0; i < n; i++) {
        const size_t row = (size_t)(t0 + i) * E;
        const SelOut o{ids ? ids + row : nullptr, counts ? counts + t0 + i : nullptr, gates ? gates + row : nullptr,
                       logits ? logits + row : nullptr, bits ? bits + (size_t)(t0 + i) * 8 : nullptr, gexp + row};
        select_token_cta([&](int j) { return lg[i][j]; }, E, p, rule, gate, sc, o, status);
        if (TB > 1) __syncthreads();  // the scratch is reused by the next token
    }
}

// Sum over the warp of N values per lane, N a power of two of 32 or more:
// afterwards lane l holds the totals of values l * (N / 32) + i in v[i].
template <int N>
PP_DEVINL void warp_transpose_sum(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int n = N / 2;
#pragma unroll
    for (int m = 16; m > 0; m >>= 1, n >>= 1) {
#pragma unroll
        for (int i = 0; i < N / 2; i++) {
            if (i >= n) break;
            const bool hi = (lane & m) != 0;
            const float keep = hi ? v[i + n] : v[i], send = hi ? v[i] : v[i + n];
            v[i] = keep + __shfl_xor_sync(kFull, send, m);
        }
    }
}

constexpr int kRows = 8;     // weight rows of a warp
constexpr int kWarps32 = 4;  // warps of a CTA, on consecutive row blocks

// h[t][e][n] = act(.) * gate weight for the tokens of group blockIdx.y (TG
// tokens) that selected expert e; rows of a gated expert: 4 gate rows, then
// the same neurons' 4 up rows.
template <int TG>
__global__ void __launch_bounds__(kWarps32 * 32)
    gu32_kernel(const float* __restrict__ x, int T, int d, int E, int act, const float* __restrict__ Wg,
                const float* __restrict__ Wu, const float* __restrict__ gexp, float* __restrict__ h) {
    pdl_wait();
    pdl_launch_dependents();
    const bool gated = act == PP_ACT_SWIGLU;
    const int lane = threadIdx.x & 31, blk = blockIdx.x * kWarps32 + (threadIdx.x >> 5);
    const int npw = gated ? kRows / 2 : kRows;  // neurons of a warp
    const int n0 = blk * npw;
    if (n0 >= E * kDExpert) return;
    const int e = n0 / kDExpert, t0 = blockIdx.y * TG;
    const float gl = lane < TG && t0 + lane < T ? gexp[(size_t)(t0 + lane) * E + e] : 0.0f;
    if (__ballot_sync(kFull, gl != 0.0f) == 0u) return;  // no token of the group selected the expert
    float acc[kRows * TG];
#pragma unroll
    for (int i = 0; i < kRows * TG; i++) acc[i] = 0.0f;
    const float* wrow[kRows];
#pragma unroll
    for (int r = 0; r < kRows; r++)
        wrow[r] = (gated && r < kRows / 2 ? Wg : Wu) + (size_t)(n0 + (gated ? r % (kRows / 2) : r)) * d;
    for (int k = lane * 4; k < d; k += 128) {
        float4 xv[TG];
#pragma unroll
        for (int i = 0; i < TG; i++) xv[i] = *reinterpret_cast<const float4*>(x + (size_t)min(t0 + i, T - 1) * d + k);
#pragma unroll
        for (int r = 0; r < kRows; r++) {
            const float4 w = *reinterpret_cast<const float4*>(wrow[r] + k);
#pragma unroll
            for (int i = 0; i < TG; i++) {
                float& s = acc[i * kRows + r];
                s = fmaf(w.x, xv[i].x, s);
                s = fmaf(w.y, xv[i].y, s);
                s = fmaf(w.z, xv[i].z, s);
                s = fmaf(w.w, xv[i].w, s);
            }
        }
    }
    warp_transpose_sum(acc);
    // value v = token * kRows + row is in lane v / (TG / 4), slot v % (TG / 4)
    constexpr int kPer = kRows * TG / 32;
#pragma unroll
    for (int i = 0; i < kPer; i++) {
        const int v = lane * kPer + i, tg = v / kRows, r = v % kRows;
        const float g = __shfl_sync(kFull, gl, tg);
        float other = 0.0f;  // the up sum of a gate row
        if (gated) other = __shfl_down_sync(kFull, acc[i], (kRows / 2) / kPer);
        const int t = t0 + tg;
        if (g == 0.0f || (gated && r >= kRows / 2)) continue;
        h[((size_t)t * E) * kDExpert + n0 + r] = (gated ? act_h(act, other, acc[i]) : act_h(act, acc[i], 0.0f)) * g;
    }
}

// y[t][row] = sum over the group's experts of h . W_down, two experts a step
// (one per half warp); a token that did not select an expert contributes 0.
template <int TG>
__global__ void __launch_bounds__(kWarps32 * 32)
    down32_kernel(const float* __restrict__ h, int T, int d, int E, const float* __restrict__ Wd,
                  const float* __restrict__ gexp, float* __restrict__ y) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ int ul[kMaxExperts];       // experts that a token of the group selected, ascending
    __shared__ unsigned um[kMaxExperts];  // which tokens did
    __shared__ int nU;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t0 = blockIdx.y * TG;
    if (warp == 0) {
        int base = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + lane;
            unsigned m = 0u;
#pragma unroll
            for (int i = 0; i < TG; i++)
                m |= (e < E && t0 + i < T && gexp[(size_t)(t0 + i) * E + e] != 0.0f ? 1u : 0u) << i;
            const unsigned any = __ballot_sync(kFull, m != 0u);
            if (m) {
                const int pos = base + __popc(any & ((1u << lane) - 1u));
                ul[pos] = e;
                um[pos] = m;
            }
            base += __popc(any);
        }
        if (lane == 0) nU = base;
    }
    __syncthreads();
    const int row0 = (blockIdx.x * kWarps32 + warp) * kRows;
    if (row0 >= d) return;
    const int n = nU, half = lane >> 4, c = (lane & 15) * 4;
    const size_t ld = (size_t)E * kDExpert;
    float acc[kRows * TG];
#pragma unroll
    for (int i = 0; i < kRows * TG; i++) acc[i] = 0.0f;
    for (int u = half; u < n; u += 2) {
        const int col = ul[u] * kDExpert + c;
        const unsigned m = um[u];
        float4 hv[TG];
#pragma unroll
        for (int i = 0; i < TG; i++)
            hv[i] = (m >> i) & 1u ? *reinterpret_cast<const float4*>(h + (size_t)(t0 + i) * ld + col)
                                  : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int r = 0; r < kRows; r++) {
            const float4 w = *reinterpret_cast<const float4*>(Wd + (size_t)min(row0 + r, d - 1) * ld + col);
#pragma unroll
            for (int i = 0; i < TG; i++) {
                float& s = acc[i * kRows + r];
                if (!((m >> i) & 1u)) continue;  // (also keeps a non-finite weight from the token)
                s = fmaf(w.x, hv[i].x, s);
                s = fmaf(w.y, hv[i].y, s);
                s = fmaf(w.z, hv[i].z, s);
                s = fmaf(w.w, hv[i].w, s);
            }
        }
    }
    warp_transpose_sum(acc);
    constexpr int kPer = kRows * TG / 32;
#pragma unroll
    for (int i = 0; i < kPer; i++) {
        const int v = lane * kPer + i, t = t0 + v / kRows, row = row0 + v % kRows;
        if (t < T && row < d) y[(size_t)t * d + row] = acc[i];
    }
}

template <int TG>
cudaError_t ffn32_groups(const Ffn32Args& a, cudaStream_t st) {
    const bool gated = a.act == PP_ACT_SWIGLU;
    const int gblk = a.E * kDExpert / (gated ? kRows / 2 : kRows), dblk = (a.d + kRows - 1) / kRows, ng = (a.T + TG - 1) / TG;
    PP_LAUNCH(gu32_kernel<TG>, dim3((gblk + kWarps32 - 1) / kWarps32, ng), dim3(kWarps32 * 32), 0, st, a.x, a.T, a.d, a.E,
              a.act, a.Wg, a.Wu, a.gexp, a.h);
    PP_LAUNCH(down32_kernel<TG>, dim3((dblk + kWarps32 - 1) / kWarps32, ng), dim3(kWarps32 * 32), 0, st, a.h, a.T, a.d,
              a.E, a.Wd, a.gexp, a.y);
    return cudaGetLastError();
}

template <typename TW>
cudaError_t route_typed(const RouteArgs& a, cudaStream_t st) {
    const TW* x = static_cast<const TW*>(a.x);
    const TW* Wr = static_cast<const TW*>(a.Wr);
    if (a.T <= kRouteOneMax)
        PP_LAUNCH((route_tokens_kernel<TW, 1>), dim3(a.T), dim3(256), 0, st, x, a.T, a.d, Wr, a.E, a.p, a.rule, a.gate,
                  a.ids, a.counts, a.gates, a.logits, a.bits, a.gexp, a.status);
    else
        PP_LAUNCH((route_tokens_kernel<TW, 4>), dim3((a.T + 3) / 4), dim3(256), 0, st, x, a.T, a.d, Wr, a.E, a.p, a.rule,
                  a.gate, a.ids, a.counts, a.gates, a.logits, a.bits, a.gexp, a.status);
    return cudaGetLastError();
}

}  // namespace

cudaError_t route_tokens(int dtype, const RouteArgs& a, cudaStream_t st) {
    return dtype == PP_BF16 ? route_typed<__nv_bfloat16>(a, st) : route_typed<float>(a, st);
}

// Groups of 4 tokens keep the warps many and the skipped work large; above 256
// tokens there are warps enough, and groups of 8 halve the weight reads.
cudaError_t ffn32(const Ffn32Args& a, cudaStream_t st) {
    return a.T <= 256 ? ffn32_groups<4>(a, st) : ffn32_groups<8>(a, st);
}

}  // namespace pp
