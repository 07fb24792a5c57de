// Batched path for a few to a few hundred tokens (bf16, 5 to kUnionMaxT
// tokens): one cooperative launch, one CTA per SM, for the whole layer, with
// the FFN evaluated over the union of the batch's selected experts.
//
// At these sizes the weights are the traffic (a 64-token Llama-3-8B call reads
// 287 MB of selected expert blocks and 0.5 MB of x), so the tokens are the N
// operand of both GEMMs for every expert of the union, with no token
// permutation: a token that did not select an expert gets a zero activation.
// The tensor work that this adds is idle capacity (N <= 256 columns per 128
// weight rows), and in exchange there is no dispatch, no per-assignment output
// row and no combine:
//
//   router   (token tile, K split) partial logits on tcgen05, as
//            router_gemm_kernel computes them
//   select   a CTA per token
//   gate/up  the union's neurons are cut into units of 16 weight rows (8 gate
//            + 8 up rows, or 16 up rows of a non-gated FFN) and every CTA takes
//            the same number of consecutive units, whatever expert they belong
//            to, in one pass over K with x streamed beside them
//   down     the (128-row tile of W_down, expert) pairs are dealt to the CTAs
//            in equal consecutive runs; a CTA accumulates a tile's experts in
//            TMEM (fp32) and writes one partial tile per run
//   reduce   y = the tile's partials in CTA order (deterministic)
//
// Up to 5 tokens the activations go through the down projection as three bf16
// terms each (all 24 bits of the fp32 value), in columns that the MMA's 16 have
// to spare; beyond, rounded to bf16.
//
// A grid barrier separates the phases (about 1.5 us, against 4-5 us for a
// launch boundary with 200 KB CTAs, which cannot overlap their predecessors),
// and the first W_down tiles of a CTA are in flight while it waits for the
// others' activations.
// Per layer of the 8B shape, against six kernels over 16-row items of whole
// experts: 8 tokens 52 -> 39 us, 64 tokens 88 -> 75; GPT-2-medium, 16 tokens,
// 28 -> 25.
//// The FFN phases are in pp_union.cuh.
#include "pp_common.cuh"
#include "pp_kernels.h"
#include "pp_launch.h"
#include "pp_select.cuh"
#include "pp_tc.cuh"
#include "pp_union.cuh"

namespace pp {
namespace {

constexpr int kRouterStages = 4;
constexpr int kUnionSmem = 218 * 1024;  // dynamic: the ring of the phase that runs, aligned to 1 KB

struct UnionArgs {
    UnionFfn f;
    CUtensorMap map_rx, map_wr;  // router: x in 128-row boxes, W_r in rn-row boxes
    int rn, kpb, nsplit, mt, gate, rule, do_route;
    float p;
    float* part;            // router partials [nsplit][T][E]
    int32_t *ids, *counts;  // selection outputs (NULL: not wanted)
    float *gates, *logits;
    uint32_t* bits;
    float* gexp;
};

struct RouterShared {
    uint64_t full[kRouterStages], empty[kRouterStages], done;
    uint32_t um[8];  // the union's bits
};

// Partial logits of (token tile, K split, group of rn experts): the chunks of a
// split in the order of router_gemm_kernel, so a logit's sum is the same.  The
// expert groups make 112 CTAs of what would be 16 (d = 4096, E = 224): a CTA's
// loads, MMAs (N = 32) and stores are a seventh (64 tokens: 6.1 -> 3.2 us).
// Before the previous kernel on the stream has completed, the W_r tiles are only
// prefetched into L2 (where that kernel's writes arrive too): it may be the one
// that writes W_r.
PP_DEVINL void router_phase(const UnionArgs& a, RouterShared& sh, unsigned char* smem, uint32_t tmem) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ngrp = (a.f.E + a.rn - 1) / a.rn, tasks = a.mt * a.nsplit * ngrp, rstage = kTileW + a.rn * 128;
    uint32_t round = 0;
    int it0 = 0;  // chunks of this CTA's earlier rounds
    for (int b = blockIdx.x; b < tasks; b += gridDim.x, round++) {
        const int e0 = (b % ngrp) * a.rn, m0 = (b / ngrp % a.mt) * 128, split = b / ngrp / a.mt;
        const int k0 = split * a.kpb, n = min(a.f.nk, k0 + a.kpb) - k0;
        if (round == 0) {
            if (warp < kRouterStages && lane == 0)
                for (int i = warp; i < n; i += kRouterStages) tma_prefetch_2d(&a.map_wr, (k0 + i) * 64, e0);
            pdl_wait();
            pdl_launch_dependents();
        }
        // warp w < 4 loads into stage w: chunk i of all the CTA's chunks is in stage i % 4
        if (warp < kRouterStages && lane == 0) {
            unsigned char* st = smem + (size_t)warp * rstage;
            for (int i = (warp - it0) & (kRouterStages - 1); i < n; i += kRouterStages) {
                const int q = (it0 + i) / kRouterStages;
                if (q > 0) mbar_wait(&sh.empty[warp], (uint32_t)(q - 1) & 1u, a.f.status, a.f.lim);
                mbar_arrive_expect_tx(&sh.full[warp], (uint32_t)rstage);
                tma_load_2d(st + kTileW, &a.map_wr, (k0 + i) * 64, e0, &sh.full[warp]);
                tma_load_2d(st, &a.map_rx, (k0 + i) * 64, m0, &sh.full[warp]);
            }
        }
        if (warp == kMmaWarp && lane == 0) {
            const uint32_t idesc = idesc_bf16_m128(a.rn);
            for (int i = 0; i < n; i++) {
                const int s = (it0 + i) & (kRouterStages - 1);
                mbar_wait(&sh.full[s], (uint32_t)((it0 + i) / kRouterStages) & 1u, a.f.status, a.f.lim);
                tc_fence_after();
                unsigned char* st = smem + (size_t)s * rstage;
                umma_k64(tmem, st, st + kTileW, idesc, i > 0);
                umma_commit(&sh.empty[s]);
            }
            umma_commit(&sh.done);
        }
        __syncwarp();
        it0 += n;
        // epilogue: lane = token row of TMEM lanes 32 * warp ..
        const int r0 = m0 + 32 * warp, t = r0 + lane;
        if (warp < kProd && r0 < a.f.T) {
            mbar_wait(&sh.done, round & 1u, a.f.status, a.f.lim);
            tc_fence_after();
            for (int c = e0; c < min(e0 + a.rn, a.f.E); c += 32) {
                uint32_t r[32];
                tmem_ld32(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(c - e0), r);
                tmem_ld_wait();
                if (t >= a.f.T) continue;
                float* row = a.part + ((size_t)split * a.f.T + t) * a.f.E + c;
                if ((a.f.E & 3) == 0) {
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        if (c + i < a.f.E) *reinterpret_cast<uint4*>(row + i) = make_uint4(r[i], r[i + 1], r[i + 2], r[i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; i++)
                        if (c + i < a.f.E) row[i] = __uint_as_float(r[i]);
                }
            }
            tc_fence_before();
        }
        __syncthreads();  // the accumulator is free for the next round
        tc_fence_after();
    }
    if (round == 0) {  // no task
        pdl_wait();
        pdl_launch_dependents();
    }
}

// Selection of tokens b, b + G, ... from the summed partial logits.
PP_DEVINL void select_phase(const UnionArgs& a, unsigned char* smem) {
    SelScratch& s = *reinterpret_cast<SelScratch*>(smem);
    for (int t = blockIdx.x; t < a.f.T; t += gridDim.x) {
        const size_t row = (size_t)t * a.f.E;
        auto logit = [&](int e) {  // partials added in split order, eight loads in flight
            const float* q = a.part + row + e;
            const size_t stride = (size_t)a.f.T * a.f.E;
            float v = 0.0f;
            int i = 0;
            for (; i + 8 <= a.nsplit; i += 8) {
                float r[8];
#pragma unroll
                for (int k = 0; k < 8; k++) r[k] = __ldcg(q + (size_t)(i + k) * stride);
#pragma unroll
                for (int k = 0; k < 8; k++) v += r[k];
            }
            for (; i < a.nsplit; i++) v += __ldcg(q + (size_t)i * stride);
            return v;
        };
        const SelOut o{a.ids ? a.ids + row : nullptr, a.counts ? a.counts + t : nullptr, a.gates ? a.gates + row : nullptr,
                       a.logits ? a.logits + row : nullptr, a.bits + (size_t)t * 8, a.gexp + row};
        select_token_cta(logit, a.f.E, a.p, a.rule, a.gate, s, o, a.f.status);
        __syncthreads();  // the scratch is reused by the next token
    }
}
__global__ void __launch_bounds__(kUnionThreads, 1) union_layer_kernel(const __grid_constant__ UnionArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ UnionShared<kUnionMaxT> sh;
    __shared__ RouterShared rs;
    const int tid = threadIdx.x;
    const int T = a.f.T, E = a.f.E;
    if (tid == 0) {
        for (int i = 0; i < kRouterStages; i++) {
            mbar_init(&rs.full[i], 1);
            mbar_init(&rs.empty[i], 1);
        }
        mbar_init(&rs.done, 1);
    }
    if (tid < 8) rs.um[tid] = 0u;
    const uint32_t cols = union_cols(a.f, a.rn), tmem = union_begin(a.f, sh, cols);
    if (a.do_route) {
        router_phase(a, rs, smem, tmem);
        if (tid == 32 * kHWarp) sh.bar_target = grid_bar_base(a.f.bar);
        grid_sync(a.f, sh);
        tc_fence_after();
        select_phase(a, smem);
        grid_sync(a.f, sh);
    } else {
        pdl_wait();
        pdl_launch_dependents();
        if (tid == 0) sh.bar_target = grid_bar_base(a.f.bar);
    }
    // the union of the tokens' experts, ascending
    uint32_t own = 0u;
    for (int t = tid >> 3; t < T; t += kUnionThreads / 8) own |= __ldcg(a.bits + (size_t)t * 8 + (tid & 7));
    if (own) atomicOr(&rs.um[tid & 7], own);
    __syncthreads();
    int nU = 0;
    {
        const int e = tid;
        uint32_t before = 0u;
#pragma unroll
        for (int w = 0; w < 8; w++) {
            // experts past E (a selection that is not this call's, after an error) are dropped
            const uint32_t m = 32 * w + 32 <= E ? rs.um[w] : 32 * w < E ? rs.um[w] & ((1u << (E & 31)) - 1u) : 0u;
            nU += __popc(m);
            if (w < (e >> 5)) before += __popc(m);
            if (w == (e >> 5)) {
                before += __popc(m & ((1u << (e & 31)) - 1u));
                if ((m >> (e & 31)) & 1u) sh.ul[before] = e;
            }
        }
    }
    __syncthreads();
    auto gate = [gexp = a.gexp, E](int t, int e) { return __ldcg(gexp + (size_t)t * E + e); };
    gu_phase<kUnionSmem - 1024>(a.f, sh, gate, smem, tmem, nU);
    down_phase<kUnionSmem - 1024>(a.f, sh, gate, smem, tmem, nU);
    union_end(tmem, cols);
}

int pad16(int T) { return (T + 15) / 16 * 16; }

}  // namespace

size_t union_part_floats(int T, int d) {
    // [CTAs][slots][T][128] for any grid of up to kUnionMaxGrid CTAs (slots below)
    const size_t ntile = (size_t)(d + 127) / 128, rows = 3 * (size_t)kUnionMaxGrid + ntile;
    return rows * 128 * (size_t)std::min(std::max(T, 16), kUnionMaxT);
}

bool union_ffn_args(const GroupedArgs& g, int grid, UnionFfn* a) {
    const bool gated = g.act == PP_ACT_SWIGLU;
    const uint64_t rows = (uint64_t)g.E * kDExpert;
    a->T = g.T;
    a->E = g.E;
    a->d = g.d;
    a->N = pad16(g.T);
    a->terms = 3 * g.T <= 16 ? 3 : 1;  // the terms fit the MMA's 16 columns
    a->nk = g.plan.nk;
    a->ntile = (g.d + 127) / 128;
    // tiles that a run can touch: ceil(pairs / CTAs) consecutive pairs, or 3
    // pairs where there are fewer than kMinRun pairs per CTA
    a->slots = std::max(a->ntile / grid + 2, 3);
    a->act = g.act;
    a->H = g.H;
    a->dpart = g.dpart;
    a->Wd = static_cast<const __nv_bfloat16*>(g.Wd);
    a->y = static_cast<__nv_bfloat16*>(g.y);
    a->bar = g.bar;
    a->status = g.status;
    a->lim = g.timeout_ns;
    const uint32_t box = gated ? 8 : 16;
    return encode_2d(&a->map_x, g.x, g.d, g.T, 64, a->N) && encode_2d(&a->map_wu, g.Wu, g.d, rows, 64, box) &&
           encode_2d(&a->map_wg, gated ? g.Wg : g.Wu, g.d, rows, 64, box) &&
           encode_2d(&a->map_h, g.H, rows, (uint64_t)a->terms * g.T, 64, a->N) &&
           encode_2d(&a->map_wd, g.Wd, rows, g.d, 64, 128, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

// A stream may own fewer SMs than the device has (a green context): the grid
// then shrinks until it is resident at once (each CTA takes more units and runs).
cudaError_t union_layer(const GroupedArgs& g, bool do_route, int sms, cudaStream_t st) {
    cudaError_t e = set_smem(union_layer_kernel, kUnionSmem);
    if (e != cudaSuccess) return e;
    for (int grid = std::min(sms, kUnionMaxGrid);; grid = (grid + 1) / 2) {
        UnionArgs a;
        std::memset(&a, 0, sizeof a);
        if (!union_ffn_args(g, grid, &a.f)) return cudaErrorInvalidValue;
        a.mt = (g.T + 127) / 128;
        a.kpb = g.plan.kpb;
        a.nsplit = g.plan.nsplit;
        // experts of a router task: 32, or 64 where the tasks of 32 would not fit one round
        a.rn = a.mt * a.nsplit * ((g.E + 31) / 32) <= grid ? 32 : 64;
        a.gate = g.gate;
        a.rule = g.rule;
        a.do_route = do_route ? 1 : 0;
        a.p = g.p;
        a.part = g.part;
        a.ids = do_route ? g.ids : nullptr;
        a.counts = do_route ? g.counts : nullptr;
        a.gates = do_route ? g.gates : nullptr;
        a.logits = do_route ? g.logits_out : nullptr;
        a.bits = g.bits;
        a.gexp = g.gexp;
        if (do_route && (!encode_2d(&a.map_rx, g.x, g.d, g.T, 64, 128) || !encode_2d(&a.map_wr, g.Wr, g.d, g.E, 64, a.rn)))
            return cudaErrorInvalidValue;
        e = launch_coop(union_layer_kernel, dim3(grid), dim3(kUnionThreads), kUnionSmem, st, a);
        if (e != cudaErrorCooperativeLaunchTooLarge || grid == 1) return e;
        (void)cudaGetLastError();
    }
}

}  // namespace pp
