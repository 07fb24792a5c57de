// Tensor-core (tcgen05) path for prompts and prefill (bf16, more than
// kUnionMaxT tokens), and the stand-alone routing of the batched path.
//
//   router GEMM   logits = X W_r^T (Eq. routing_logits), split over K; the
//                 selection kernel sums the K-split partials in fixed order
//   selection     a warp per token; an activated (token, expert) pair takes
//                 the next slot of the expert's token list
//   grouped G/U   per work item (expert e, <= 128 of its tokens):
//                 D[128 x (64|128)] = X_gathered * [W_gate_e ; W_up_e]^T on
//                 tcgen05 (TMA gather4 for the token rows), then
//                 h = act(gate, up) * gate weight (Eq. ffn, Eq. moe_output),
//                 stored bf16, one row per pair, experts in ascending order
//   grouped down  per (work item, 128-row tile of W_down):
//                 D[128 rows x tokens] = W_down[tile, e-block] * H_item^T
//                 (K = 64); each pair's output row is stored bf16
//   combine       y[t] = sum over t's experts, in ascending expert order, of
//                 its pairs' rows (fp32 accumulation, deterministic)
//   An expert whose rows do not all fit the row buffer (only near-dense
//   selections have one) adds them into an fp32 accumulator instead, which the
//   gate/up kernel clears when the call's pairs exceed the capacity and the
//   combine step adds.
//   (Nothing is expected of it before the call: its place depends on the
//   call's token count, so calls of other lengths write over it.)
//
// A slot is given out by an atomic, so the order of an expert's tokens varies
// between calls; no pair's value depends on it (a row of a GEMM tile does not
// depend on its place, the combine step goes by expert, and all of an expert's
// pairs are rounded alike: to bf16 in the row buffer, or not at all in the
// accumulator).  What is free is the order of the fp32 additions into that
// accumulator, so a token with several such experts may differ in the last bit.
// All waits are bounded (PP_ERR_TIMEOUT).
#include "pp_common.cuh"
#include "pp_kernels.h"
#include "pp_launch.h"
#include "pp_select.cuh"
#include "pp_tc.cuh"

namespace pp {

constexpr int kTcThreads = 192;
constexpr int kTileBytesA = 128 * 128;  // 128 rows x 64 bf16


// ====================================================================== router
// Grid (m-tiles, splits).  CTA (m, s): D[128 tokens x NE] over K chunks
// [s*kpb, min((s+1)*kpb, nk)), one at least (grouped_plan); partial logits to
// part[s][t][e].
template <int NE>
__global__ void __launch_bounds__(kTcThreads, 1)
    router_gemm_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_wr,
                       int T, int E, int nk, int kpb, float* part, int* cnt, unsigned* status,
                       uint64_t lim) {
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    if (cnt && blockIdx.x == 0 && blockIdx.y == 0)  // the selection fills the lists
        for (int e = threadIdx.x; e < E; e += blockDim.x) cnt[e] = 0;
    constexpr int kStages = 4;
    constexpr int kTileB = NE * 128;
    constexpr int kStage = kTileBytesA + kTileB;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[kStages], empty[kStages], tfull;
    __shared__ uint32_t taddr_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * 128, split = blockIdx.y;
    const int k0 = split * kpb, k1 = min(nk, k0 + kpb);
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; i++) {
            mbar_init(&full[i], 2);
            mbar_init(&empty[i], 1);
        }
        mbar_init(&tfull, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(&taddr_s, NE <= 128 ? 128 : 256);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = taddr_s;

    // the W_r and x tiles are issued by two warps (a TMA instruction costs its
    // warp 24 ns plus 1.3 ns per row: 224 + 128 rows a stage by one took 450 ns)
    if ((warp == 0 || warp == 2) && lane == 0) {
        for (int kc = k0, it = 0; kc < k1; kc++, it++) {
            const int s = it % kStages;
            if (it >= kStages) mbar_wait(&empty[s], (uint32_t)((it / kStages) - 1) & 1u, status, lim);
            unsigned char* st = smem + (size_t)s * kStage;
            mbar_arrive_expect_tx(&full[s], warp == 0 ? kTileB : kTileBytesA);
            if (warp == 0)
                tma_load_2d(st + kTileBytesA, &map_wr, kc * 64, 0, &full[s]);
            else
                tma_load_2d(st, &map_x, kc * 64, m0, &full[s]);
        }
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16_m128(NE);
        for (int kc = k0, it = 0; kc < k1; kc++, it++) {
            const int s = it % kStages;
            mbar_wait(&full[s], (uint32_t)(it / kStages) & 1u, status, lim);
            tc_fence_after();
            unsigned char* st = smem + (size_t)s * kStage;
            umma_k64(tmem, st, st + kTileBytesA, idesc, it > 0);
            umma_commit(&empty[s]);
        }
        umma_commit(&tfull);
    }
    __syncwarp();
    if (warp >= 2) {
        // lane = token row 32 q + lane; a lane stores its row's 32 logits in
        // 16-byte pieces where rows are 16-byte aligned
        const int q = warp & 3, t = m0 + 32 * q + lane;
        mbar_wait(&tfull, 0, status, lim);
        tc_fence_after();
        float* row = part + ((size_t)split * T + t) * E;
#pragma unroll 1
        for (int c = 0; c < (m0 + 32 * q < T ? E : 0); c += 32) {
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c, r);
            tmem_ld_wait();
            if (t >= T) continue;
            if ((E & 3) == 0) {
#pragma unroll
                for (int i = 0; i < 32; i += 4)
                    if (c + i < E)
                        *reinterpret_cast<uint4*>(row + c + i) = make_uint4(r[i], r[i + 1], r[i + 2], r[i + 3]);
            } else {
#pragma unroll
                for (int i = 0; i < 32; i++)
                    if (c + i < E) row[c + i] = __uint_as_float(r[i]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, NE <= 128 ? 128 : 256);
}

// ================================================================= selection
// Selection from K-split partial logits (summed in split order): one CTA per
// token up to kCtaSelectMaxTokens tokens (latency), one warp per token beyond.
constexpr int kCtaSelectMaxTokens = 256;

// Logit = sum over s of part[s * stride + off], added in split order; the
// loads go out 8 at a time instead of one dependent round trip each.
PP_DEVINL float sum_partials(const float* __restrict__ part, int nsplit, size_t stride, size_t off) {
    float v = 0.0f;
    int s = 0;
    for (; s + 8 <= nsplit; s += 8) {
        float q[8];
#pragma unroll
        for (int i = 0; i < 8; i++) q[i] = __ldg(part + (size_t)(s + i) * stride + off);
#pragma unroll
        for (int i = 0; i < 8; i++) v += q[i];
    }
    for (; s < nsplit; s++) v += __ldg(part + (size_t)s * stride + off);
    return v;
}

// Per-expert lists of the activated pairs: cnt[e] tokens ltok[e * T + slot]
// with gate weights lgate[e * T + slot]; slot_of[t * E + e] = slot.
struct Lists {
    int* cnt;
    int* ltok;
    float* lgate;
    int* slot_of;
};

PP_DEVINL void list_add(const Lists& l, int T, int E, int t, int e, float gv) {
    const int s = atomicAdd(&l.cnt[e], 1);
    l.ltok[(size_t)e * T + s] = t;
    l.lgate[(size_t)e * T + s] = gv;
    l.slot_of[(size_t)t * E + e] = s;
}

// Selection of one token by a warp, lane l holding logits l, l + 32, ...: the
// experts are taken in descending order one by one (two warp reductions each)
// until the rule stops, with the exact fixed-point masses of group_mass_cut, so
// the decisions are the same.  An activated expert costs about 110 cycles and
// nothing is sorted that is not activated: one CTA per token took 46 us for
// 8192 tokens of 216 experts (6 activated each), this 20 us (under ncu).  ids and gates
// (together), counts, logits_out may be NULL; so may bits with the lists.
template <int S>
__global__ void __launch_bounds__(256)
    select_warp_kernel(const float* __restrict__ part, int nsplit, int T, int E, float p, int rule, int gate, int32_t* ids,
                       int32_t* counts, float* gates, float* logits_out, uint32_t* bits, Lists lists, unsigned* status) {
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= T) return;
    const size_t row = (size_t)t * E;
    float g[S];
    uint32_t D[S], U[S];
    bool fin = true;
    uint32_t dmin = 0xffffffffu;
    const size_t stride = (size_t)T * E;
#pragma unroll
    for (int s = 0; s < S; s++) g[s] = 0.0f;
#pragma unroll 4
    for (int sp = 0; sp < nsplit; sp++) {  // partials added in split order, all slots' loads in flight
        const float* q = part + sp * stride + row + lane;
#pragma unroll
        for (int s = 0; s < S; s++)
            if (lane + 32 * s < E) g[s] += __ldg(q + 32 * s);
    }
#pragma unroll
    for (int s = 0; s < S; s++) {
        const int j = lane + 32 * s;
        D[s] = 0xffffffffu;  // no finite logit has this key
        if (j < E) {
            if (logits_out) logits_out[row + j] = g[s];
            fin = fin && isfinite(g[s]);
            D[s] = desc_key(g[s]);
            dmin = min(dmin, D[s]);
        }
    }
    fin = __all_sync(kFull, fin);
    if (!fin && lane == 0) record_status(status, PP_ERR_NONFINITE);
    const float m = desc_key_logit(__reduce_min_sync(kFull, dmin));
    const bool mass_cut = (rule == PP_SEL_MIN_PREFIX || rule == PP_SEL_PAPER) && p < 1.0f;
    unsigned long long z = 0ull;
#pragma unroll
    for (int s = 0; s < S; s++) {
        U[s] = mass_cut && lane + 32 * s < E ? __float2uint_rn(expf(g[s] - m) * 2147483648.0f) : 0u;
        z += U[s];
    }
    long long thr = -1;
    if (mass_cut) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(kFull, z, o);
        thr = prefix_threshold(p, z);
    }
    const int kmax = !fin ? 0 : rule == PP_SEL_TOPK ? min(E, (int)p) : E;
    unsigned long long A = 0ull;  // mass ahead of rank r
    int r = 0, my_e = 0;          // lane l keeps rank 32 i + l until it is written
    float my_g = 0.0f;
    auto flush = [&](int base, int n) {
        if (lane < n) {
            const float gv = gate == PP_GATE_NONE ? 1.0f : sigmoidf_(my_g);
            if (ids) {
                ids[row + base + lane] = my_e;
                gates[row + base + lane] = gv;
            }
            if (bits) list_add(lists, T, E, t, my_e, gv);
        }
    };
    while (r < kmax) {
        uint32_t bd = 0xffffffffu, bu = 0u;
        int bs = 0;
        float bg = 0.0f;
#pragma unroll
        for (int s = 0; s < S; s++)
            if (D[s] < bd) {  // the lowest index of equal keys
                bd = D[s];
                bs = s;
                bu = U[s];
                bg = g[s];
            }
        const uint32_t wd = __reduce_min_sync(kFull, bd);
        const unsigned wj = __reduce_min_sync(kFull, bd == wd ? (unsigned)(bs * 32 + lane) : 0xffffffffu);
        const int owner = (int)(wj & 31u);
        const uint32_t u = __shfl_sync(kFull, bu, owner);
        const float gv = __shfl_sync(kFull, bg, owner);
        if (mass_cut) {
            const unsigned long long mass = rule == PP_SEL_PAPER ? A + u : A;
            if (!(A == 0ull || (thr >= 0 && mass <= (unsigned long long)thr))) break;
            A += u;
        } else if (rule == PP_SEL_LTE && !(gv >= p)) {
            break;
        }
        if (lane == (r & 31)) {
            my_e = (int)wj;
            my_g = gv;
        }
#pragma unroll
        for (int s = 0; s < S; s++)
            if (lane == owner && s == bs) D[s] = 0xffffffffu;
        r++;
        if ((r & 31) == 0) flush(r - 32, 32);
    }
    flush(r & ~31, r & 31);
    if (ids)
        for (int i = r + lane; i < E; i += 32) {
            ids[row + i] = -1;
            gates[row + i] = 0.0f;
        }
    if (counts && lane == 0) counts[t] = r;
    if (bits) {
#pragma unroll
        for (int s = 0; s < 8; s++) {  // expert lane + 32 s is bit `lane` of word s
            bool on = false;
            if (s < S) on = fin && lane + 32 * s < E && D[s < S ? s : 0] == 0xffffffffu;
            const unsigned v = __ballot_sync(kFull, on);
            if (lane == s) bits[(size_t)t * 8 + s] = v;
        }
    }
}

// One CTA per token.
__global__ void __launch_bounds__(256) select_part_cta_kernel(const float* __restrict__ part, int nsplit, int T,
                                                              int E, float p, int rule, int gate, int32_t* ids,
                                                              int32_t* counts, float* gates, float* logits_out,
                                                              unsigned* status) {
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    __shared__ __align__(16) SelScratch sc;
    const int t = blockIdx.x;
    const size_t row = (size_t)t * E;
    const SelOut o{ids + row, counts + t, gates + row, logits_out ? logits_out + row : nullptr, nullptr, nullptr};
    select_token_cta([&](int j) { return sum_partials(part, nsplit, (size_t)T * E, row + j); }, E, p, rule, gate, sc, o,
                     status);
}

// ================================================================== dispatch
// bits[t][w]: bit (e % 32) of word e / 32 set when token t activated e;
// gexp[t][e]: gexp_entry of that assignment's gate weight (gates of a repeated
// id add up), +0 where e is not activated.  Invalid ids and counts are recorded
// and skipped.
__global__ void __launch_bounds__(256) dispatch_bits_kernel(const int32_t* __restrict__ ids,
                                                            const int32_t* __restrict__ counts,
                                                            const float* __restrict__ gates, int T, int E,
                                                            uint32_t* bits, float* gexp, int* cnt,
                                                            unsigned* status) {
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    if (cnt && blockIdx.x == 0)  // lengths of the lists that dispatch_list_kernel fills
        for (int e = threadIdx.x; e < E; e += blockDim.x) cnt[e] = 0;
    // one warp per token: coalesced row writes
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= T) return;
    float* grow = gexp + (size_t)t * E;
    for (int e = lane; e < E; e += 32) grow[e] = 0.0f;
    int k = counts[t];
    if (k < 0 || k > E) {
        if (lane == 0) record_status(status, PP_ERR_INVALID_ARG);
        k = k < 0 ? 0 : E;
    }
    __syncwarp();
    uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    // entries in rank order, one lane each; repeated ids add their gates in
    // rank order (the lanes of a round take turns on a repeated id)
    for (int r0 = 0; r0 < k; r0 += 32) {
        const int r = r0 + lane;
        int e = r < k ? ids[(size_t)t * E + r] : -1;
        if (r < k && (e < 0 || e >= E)) {
            record_status(status, PP_ERR_INVALID_ARG);
            e = -1;
        }
        const float gv = e >= 0 ? gates[(size_t)t * E + r] : 0.0f;
        if (e >= 0) w[e >> 5] |= 1u << (e & 31);
        for (int l = 0; l < 32; l++) {
            const int el = __shfl_sync(kFull, e, l);
            const float gl = __shfl_sync(kFull, gv, l);
            if (el >= 0 && lane == (el & 31)) grow[el] += gl;
            __syncwarp();
        }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        uint32_t v = w[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(kFull, v, o);
        if (lane == i) bits[(size_t)t * 8 + i] = v;
        // (the entries that this lane has summed)
        if ((v >> lane) & 1u && grow[32 * i + lane] == 0.0f) grow[32 * i + lane] = gexp_entry(0.0f);
    }
}

// The lists from bits and gexp (a selection given by the caller): a warp per
// token, lane l the experts l, l + 32, ...
__global__ void __launch_bounds__(256) dispatch_list_kernel(const uint32_t* __restrict__ bits,
                                                            const float* __restrict__ gexp, int T, int E, Lists lists) {
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, t = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t >= T) return;
    for (int e = lane; e < E; e += 32)
        if ((bits[(size_t)t * 8 + (e >> 5)] >> (e & 31)) & 1u) list_add(lists, T, E, t, e, gexp[(size_t)t * E + e]);
}

// Work items of a call, formed by each CTA from the list lengths: expert e's
// tokens are cut into items of 128; off = first row of the expert in H and Y.
struct Item {
    int e, m0, cnt, a0;  // expert, first slot, tokens (<= 128), first row
};

struct ItemTable {
    int off[kMaxExperts + 1], ib[kMaxExperts + 1];
    int longest;  // tokens of the longest item

    // Warp 0 of the CTA builds the table (8 experts per lane); a barrier follows.
    PP_DEVINL void build(const int* __restrict__ cnt, int E) {
        if (threadIdx.x >= 32) return;
        const int lane = threadIdx.x;
        int c[8], cs = 0, ms = 0, cm = 0;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int e = lane * 8 + q;
            c[q] = e < E ? cnt[e] : 0;
            cm = max(cm, min(c[q], 128));
            cs += c[q];
            ms += (c[q] + 127) / 128;
        }
        int ci = cs, mi = ms;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int cv = __shfl_up_sync(kFull, ci, o), mv = __shfl_up_sync(kFull, mi, o);
            if (lane >= o) {
                ci += cv;
                mi += mv;
            }
        }
        int co = ci - cs, mo = mi - ms;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            off[lane * 8 + q] = co;
            ib[lane * 8 + q] = mo;
            co += c[q];
            mo += (c[q] + 127) / 128;
        }
        cm = __reduce_max_sync(kFull, cm);
        if (lane == 31) {
            longest = cm;
            off[kMaxExperts] = co;
            ib[kMaxExperts] = mo;
        }
    }
    PP_DEVINL int n_items() const { return ib[kMaxExperts]; }
    PP_DEVINL int n_pairs() const { return off[kMaxExperts]; }
    // whether expert e's rows end past the row buffer
    PP_DEVINL bool spills(int e, long long ycap) const { return off[e + 1] > ycap; }
    PP_DEVINL Item item(int wi) const {
        int lo = 0, hi = kMaxExperts;  // ib[lo] <= wi < ib[hi]
#pragma unroll 1
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (ib[mid] <= wi) lo = mid; else hi = mid;
        }
        const int m0 = (wi - ib[lo]) * 128;
        return Item{lo, m0, min(128, off[lo + 1] - off[lo] - m0), off[lo] + m0};
    }
};

// =============================================================== grouped G/U
// Persistent over tasks: a work item, or half of its neurons where whole items
// would leave the last round nearly empty.  A = the item's token rows (TMA
// gather4, live rows only), B = the expert's gate and up rows, K-chunks of 64.
//
// What bounds it: the SM's TMA and L2 path, about 1 ns per 128-byte row (256
// rows of a full chunk), if enough warps issue and enough stages are in flight
// (a stage's round trip is about 1.4 us: the ring holds as many stages as the
// longest item's rows leave room for, 16 at most; six fixed stages took 330 ns
// per chunk of a 12-token item's half).  Under ncu: 8192 tokens of the 13B shape
// 170 -> 100 us, 2048 tokens 93 -> 76, 333 tokens of the 7B shape 61 -> 57: a gather4 costs its warp about
// 30 ns, so eight producer warps take 4 of a chunk's 32 gathers each (one
// gather thread per row with cp.async, three stages in flight, took 400-580 ns
// per chunk).  An MMA thread needs 55-64 cycles per MMA and about 300 for a
// stage's wait and commit, so two MMA warps take the stages in turn, each with
// its own accumulators (added in the epilogue); the ring is even, so that a
// slot is always the same MMA warp's.  Two accumulator sets let the epilogue
// of one task overlap the MMAs of the next.  An MMA reads 128 token rows; those
// past the item's are whatever the ring holds, and so are their sums, which are
// never stored.
constexpr int kGuProd = 8, kGuMma = 2, kGuEpi = 4;  // warps
constexpr int kGuThreads = (kGuProd + kGuMma + kGuEpi) * 32;
constexpr int kGuStages = 16;  // at most
constexpr size_t kGuRing = 206 * 1024, kGuSlack = kTileBytesA;  // ring, and the rows that the last MMA reads past it
constexpr int kGuBox = 32;  // weight rows of a TMA box

__global__ void __launch_bounds__(kGuThreads, 1)
    gu_gemm_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_wg,
                   const __grid_constant__ CUtensorMap map_wu, const int* __restrict__ cnt, const int* __restrict__ ltok,
                   const float* __restrict__ lgate, int* offsets, int T, int E, int d, int nk, int act, __nv_bfloat16* H,
                   long long ycap, float* yacc, unsigned* status, uint64_t lim) {
    const bool gated = act == PP_ACT_SWIGLU;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[kGuStages], empty[kGuStages], tfull[2], tempty[2];
    __shared__ uint32_t taddr_s;
    __shared__ ItemTable tab;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kGuStages; i++) {
            mbar_init(&full[i], kGuProd);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&tfull[i], kGuMma);
            mbar_init(&tempty[i], kGuEpi);
        }
        fence_mbar_init();
    }
    if (warp == kGuProd) {
        tmem_alloc(&taddr_s, 512);  // 2 sets x 2 MMA warps x 128 columns
        tmem_relinquish();
    }
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    tab.build(cnt, E);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = taddr_s;
    if (blockIdx.x == 0)
        for (int e = threadIdx.x; e <= E; e += kGuThreads) offsets[e] = tab.off[e];
    // whole items, or halves where they shorten the longest CTA (a half costs
    // about 0.6 of an item: its tokens are gathered again)
    const int n_items = tab.n_items(), G = gridDim.x;
    const int split = ((2 * n_items + G - 1) / G) * 6 < ((n_items + G - 1) / G) * 10 ? 2 : 1;
    const int nb = 64 / split, n_tasks = n_items * split;  // neurons of a task
    const int brows = gated ? 2 * nb : nb;
    const int bbytes = brows * 128, stage = bbytes + ((tab.longest + 7) & ~7) * 128;
    const int nst = min(kGuStages, (int)kGuRing / stage) & ~1;

    if (warp < kGuProd) {
        int it_s = 0;
        uint32_t it_ph = 0;
        bool primed = false;
        for (int v = blockIdx.x; v < n_tasks; v += G) {
            const Item w = tab.item(v / split);
            const int n0 = (v % split) * nb;
            // lane l < 4: rows 4 (warp + 8 l) .. + 3 (past the count: the last row)
            const int grp = warp + kGuProd * lane, ng = (w.cnt + 3) >> 2;
            const bool gather = lane < 4 && grp < ng;
            int r[4] = {0, 0, 0, 0};
            if (gather)
#pragma unroll
                for (int i = 0; i < 4; i++) r[i] = ltok[(size_t)w.e * T + w.m0 + min(4 * grp + i, w.cnt - 1)];
            // box `warp` of the weight rows goes out from lane 4
            const bool box = lane == 4 && warp * kGuBox < brows;
            const bool up = !gated || warp * kGuBox >= nb;
            const int brow = w.e * 64 + n0 + (up && gated ? warp * kGuBox - nb : warp * kGuBox);
            const uint32_t bytes =
                (uint32_t)(__popc(__ballot_sync(kFull, gather)) * 512 + (warp * kGuBox < brows ? kGuBox * 128 : 0));
            for (int kc = 0; kc < nk; kc++) {
                if (lane == 0) {
                    if (primed) mbar_wait(&empty[it_s], it_ph ^ 1u, status, lim);
                    mbar_arrive_expect_tx(&full[it_s], bytes);
                }
                __syncwarp();
                unsigned char* st = smem + (size_t)it_s * stage;
                if (gather) tma_gather4(st + bbytes + grp * 512, &map_x, kc * 64, r[0], r[1], r[2], r[3], &full[it_s]);
                if (box)
                    tma_load_2d(st + warp * kGuBox * 128, up ? &map_wu : &map_wg, kc * 64, brow, &full[it_s]);
                if (++it_s == nst) {
                    it_s = 0;
                    it_ph ^= 1u;
                    primed = true;
                }
            }
        }
    } else if (warp < kGuProd + kGuMma) {
        if (lane == 0) {
            const int m = warp - kGuProd;
            const uint32_t idesc = idesc_bf16_m128(brows);
            int it = 0, s = 0, acc = 0;
            uint32_t ph = 0;
            for (int v = blockIdx.x; v < n_tasks; v += G, acc++) {
                const int a = acc & 1;
                if (acc >= 2) mbar_wait(&tempty[a], (uint32_t)((acc >> 1) - 1) & 1u, status, lim);
                tc_fence_after();
                bool fresh = true;
                for (int kc = 0; kc < nk; kc++, it++) {
                    if ((it & 1) == m) {
                        mbar_wait(&full[s], ph, status, lim);
                        tc_fence_after();
                        unsigned char* st = smem + (size_t)s * stage;
                        umma_k64(tmem + (uint32_t)(a * 256 + m * 128), st + bbytes, st, idesc, !fresh);
                        umma_commit(&empty[s]);
                        fresh = false;
                    }
                    if (++s == nst) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                umma_commit(&tfull[a]);
            }
        }
        __syncwarp();
    } else {
        const int q = warp & 3;
        const int row = 32 * q + lane;
        // some pairs go past the row buffer: their accumulator starts at zero
        // (before the first sums are there; d is a multiple of 8)
        if (tab.n_pairs() > ycap) {
            float4* z = reinterpret_cast<float4*>(yacc);
            const size_t n = (size_t)T * d / 4, step = (size_t)G * kGuEpi * 32;
            for (size_t i = (size_t)blockIdx.x * kGuEpi * 32 + row; i < n; i += step) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        int acc = 0, it = 0;
        for (int v = blockIdx.x; v < n_tasks; v += G, acc++, it += nk) {
            const Item w = tab.item(v / split);
            const int n0 = (v % split) * nb;
            const int a = acc & 1;
            const bool live = row < w.cnt;
            const float gw = live ? lgate[(size_t)w.e * T + w.m0 + row] : 0.0f;
            mbar_wait(&tfull[a], (uint32_t)(acc >> 1) & 1u, status, lim);
            tc_fence_after();
            if (32 * q < w.cnt) {
                // a single chunk is in the accumulator of the MMA warp that took it
                const uint32_t b0 = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(a * 256);
                const bool both = nk > 1;
                const uint32_t base = both ? b0 : b0 + (uint32_t)((it & 1) * 128);
                auto sums = [&](int c, uint32_t (&r)[16]) {
                    tmem_ld16(base + (uint32_t)c, r);
                    if (both) {
                        uint32_t o[16];
                        tmem_ld16(b0 + (uint32_t)(128 + c), o);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; i++) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(o[i]));
                    } else {
                        tmem_ld_wait();
                    }
                };
                for (int c = 0; c < nb; c += 16) {
                    uint32_t u[16];
                    float h[16];
                    sums(gated ? nb + c : c, u);
                    if (gated) {
                        uint32_t g[16];
                        sums(c, g);
#pragma unroll
                        for (int i = 0; i < 16; i++) h[i] = act_h(PP_ACT_SWIGLU, __uint_as_float(u[i]), __uint_as_float(g[i])) * gw;
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; i++) h[i] = act_h(act, __uint_as_float(u[i]), 0.0f) * gw;
                    }
                    if (live) {
                        uint4* dst = reinterpret_cast<uint4*>(H + (size_t)(w.a0 + row) * 64 + n0 + c);
#pragma unroll
                        for (int k = 0; k < 2; k++)
                            dst[k] = make_uint4(pack_bf16x2(h[8 * k], h[8 * k + 1]), pack_bf16x2(h[8 * k + 2], h[8 * k + 3]),
                                                pack_bf16x2(h[8 * k + 4], h[8 * k + 5]), pack_bf16x2(h[8 * k + 6], h[8 * k + 7]));
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[a]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kGuProd) tmem_dealloc(tmem, 512);
}

// ============================================================== grouped down
// (128-row tile of W_down, work item) pairs, tile by tile, dealt to the CTAs in
// equal consecutive runs: D[128 rows x N] = W_down[tile, expert] * H_item^T,
// N = the item's tokens padded to 16.  Weights are the M operand, so a tile's
// epilogue costs by the tokens that there are and every warp has rows to store;
// with tokens as M, one warp held all 12 tokens of a short prompt's item (45 us
// at 333 tokens of the 7B shape for 90 MB of weights).  Tile by tile, a CTA
// reads the 128-byte column blocks of consecutive experts, neighbours in a row
// of W_down, and an expert's items share its block in L2.  Bound: HBM (W_down
// and the rows of Y).  A pair's round trip (MMA, commit, TMEM load) is about
// 1 us: four accumulators, released as soon as they are in registers.  The
// 32-token groups of a pair are transposed through shared memory and leave as
// one 256-byte bulk copy per token (4-byte stores, 64 bytes to a row, took
// 1.6-2.2 us per pair: 94 us at 2048 tokens of the 13B shape).  333 tokens of
// the 7B shape: 45 -> 31 us.
constexpr int kDnEpi = 8;  // epilogue warps: two sets of four (TMEM lane quarters), on alternating 32 tokens or pairs
constexpr int kDnThreads = (2 + kDnEpi) * 32;
constexpr int kDnStages = 12, kDnAcc = 4;
constexpr int kDnBox = 32;               // H rows of a TMA box
constexpr int kDnPitch = 128 * 2 + 16;   // staged token row
constexpr int kDnStageOut = 32 * kDnPitch;
constexpr size_t kDnRing = 172 * 1024;   // followed by 2 staging areas per set of epilogue warps
constexpr int kDrStages = 4, kDrTileB = 256 * 128;  // tokens as the M operand: the W_down ring

// Position in the pairs of a call: item `it` of tile rt is work item `sub` of
// expert e.
struct DownPos {
    const ItemTable& tab;
    int rt, it, e, sub;
    PP_DEVINL DownPos(const ItemTable& t, long long p) : tab(t) {
        const int n = t.n_items();
        rt = (int)(p / n);
        it = (int)(p - (long long)rt * n);
        const Item w = t.item(it);
        e = w.e;
        sub = w.m0 / 128;
    }
    PP_DEVINL int a0() const { return tab.off[e] + 128 * sub; }
    PP_DEVINL int count() const { return min(128, tab.off[e + 1] - a0()); }
    PP_DEVINL void next() {
        if (++it == tab.n_items()) {
            it = 0;
            rt++;
            e = 0;
            sub = 0;
        } else if (++sub < tab.ib[e + 1] - tab.ib[e]) {
            return;
        } else {
            e++;
            sub = 0;
        }
        while (tab.ib[e + 1] == tab.ib[e]) e++;  // (n_items > 0)
    }
};

struct DownShared {
    ItemTable tab;
    uint32_t taddr;
    uint64_t full[kDnStages], empty[kDnStages], tfull[kDnAcc], tempty[kDnAcc];    // down_tiles
    uint64_t rfull[kDrStages], rempty[kDrStages], rtfull[2], rtempty[2], afull, aempty;  // down_rows
};

PP_DEVINL void down_tiles(const CUtensorMap& map_h, const CUtensorMap& map_wd, DownShared& sh, unsigned char* smem,
                          uint32_t tmem, const int* __restrict__ ltok, int T, int d, __nv_bfloat16* Y, long long ycap,
                          float* yacc, unsigned* status, uint64_t lim) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nrt = (d + 127) / 128;
    const ItemTable& tab = sh.tab;
    uint64_t *full = sh.full, *empty = sh.empty, *tfull = sh.tfull, *tempty = sh.tempty;
    const long long P = (long long)tab.n_items() * nrt;
    const long long p0 = P * blockIdx.x / gridDim.x;
    const int n = (int)(P * (blockIdx.x + 1) / gridDim.x - p0);
    // H tiles in boxes of kDnBox rows, as many as the longest item needs
    const int nbox = (tab.longest + kDnBox - 1) / kDnBox, stage = kTileBytesA + nbox * kDnBox * 128;
    const int nst = min(kDnStages, (int)kDnRing / stage);

    if (n > 0 && warp == 0) {
        if (lane == 0) {
            DownPos w(tab, p0);
            int s = 0;
            uint32_t ph = 0;
            for (int i = 0; i < n; i++) {
                if (i >= nst) mbar_wait(&empty[s], ph ^ 1u, status, lim);
                mbar_arrive_expect_tx(&full[s], (uint32_t)stage);
                unsigned char* st = smem + (size_t)s * stage;
                tma_load_2d(st, &map_wd, w.e * 64, w.rt * 128, &full[s]);
                for (int b = 0; b < nbox; b++)
                    tma_load_2d(st + kTileBytesA + b * kDnBox * 128, &map_h, 0, w.a0() + b * kDnBox, &full[s]);
                if (++s == nst) {
                    s = 0;
                    ph ^= 1u;
                }
                if (i + 1 < n) w.next();
            }
        }
        __syncwarp();
    } else if (n > 0 && warp == 1) {
        if (lane == 0) {
            DownPos w(tab, p0);
            int s = 0, a = 0;
            uint32_t ph = 0, aph = 0;
            for (int i = 0; i < n; i++) {
                if (i >= kDnAcc) mbar_wait(&tempty[a], aph ^ 1u, status, lim);
                mbar_wait(&full[s], ph, status, lim);
                tc_fence_after();
                unsigned char* st = smem + (size_t)s * stage;
                umma_k64(tmem + (uint32_t)(a * 128), st, st + kTileBytesA, idesc_bf16_m128((w.count() + 15) & ~15), false);
                umma_commit(&empty[s]);
                umma_commit(&tfull[a]);
                if (++s == nst) {
                    s = 0;
                    ph ^= 1u;
                }
                if (++a == kDnAcc) {
                    a = 0;
                    aph ^= 1u;
                }
                if (i + 1 < n) w.next();
            }
        }
        __syncwarp();
    } else if (n > 0) {
        const int q = warp & 3, set = (warp - 2) >> 2;
        unsigned char* out_s = smem + kDnRing + (size_t)set * 2 * kDnStageOut;
        DownPos w(tab, p0);
        int a = 0, buf = 0;
        uint32_t aph = 0;
        for (int i = 0; i < n; i++) {
            const int m = w.count(), a0 = w.a0();
            const bool spill = tab.spills(w.e, ycap);  // the expert's rows go to yacc
            mbar_wait(&tfull[a], aph, status, lim);
            tc_fence_after();
            const int row = w.rt * 128 + 32 * q + lane;  // output element
            const uint32_t rbytes = (uint32_t)min(128, d - w.rt * 128) * 2u;
            // items of one group: the sets take the pairs in turn
            const int c0 = m > 32 ? 32 * set : set == (i & 1) ? 0 : m;
            if (c0 >= m) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[a]);
            }
            for (int c = c0; c < m; c += 64) {
                uint32_t v[32];
                tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(a * 128 + c), v);
                tmem_ld_wait();
                if (c + 64 >= m) {  // the accumulator is in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[a]);
                }
                if (!spill) {
                    // this thread's copies out of the buffer, two groups ago, have been read
                    bulk_wait_read<1>();
                    named_bar_sync(1 + set, 128);
                    unsigned char* sb = out_s + buf * kDnStageOut;
                    __nv_bfloat16* col = reinterpret_cast<__nv_bfloat16*>(sb) + 32 * q + lane;
#pragma unroll
                    for (int k = 0; k < 32; k++) {
                        if ((k & 7) == 0 && c + k >= m) break;
                        col[(size_t)k * (kDnPitch / 2)] = __float2bfloat16_rn(__uint_as_float(v[k]));
                    }
                    fence_proxy_async_smem();
                    named_bar_sync(1 + set, 128);
                    // warp q sends tokens q, q + 4, ... of the group
                    const int t = 4 * lane + q;
                    if (lane < 8 && c + t < m)
                        bulk_s2g(Y + (size_t)(a0 + c + t) * d + w.rt * 128, sb + t * kDnPitch, rbytes);
                    bulk_commit();
                    buf ^= 1;
                } else if (row < d) {
#pragma unroll
                    for (int k = 0; k < 32; k++) {
                        const int t = c + k;
                        if (t >= m) break;
                        atomicAdd(&yacc[(size_t)ltok[(size_t)w.e * T + 128 * w.sub + t] * d + row], __uint_as_float(v[k]));
                    }
                }
            }
            if (++a == kDnAcc) {
                a = 0;
                aph ^= 1u;
            }
            if (i + 1 < n) w.next();
        }
        bulk_wait_all();  // the stores are done before the CTA's shared memory goes away
        __syncwarp();
    }
}

// Tokens as the M operand.  Persistent over work items: an item's H tile is
// loaded once and the 256-wide slices of d stream through the B ring.  Two
// 256-column TMEM accumulators overlap the stores of one slice with the next
// slice's MMAs.  Warp 0 loads, 1 issues the MMAs, 2-5 store.
PP_DEVINL void down_rows(const CUtensorMap& map_h, const CUtensorMap& map_wd, const CUtensorMap& map_y, DownShared& sh,
                         unsigned char* smem, uint32_t tmem, const int* __restrict__ ltok, int T, int d,
                         __nv_bfloat16* Y, long long ycap, float* yacc, unsigned* status, uint64_t lim) {
    constexpr int kStages = kDrStages;
    constexpr int kTileB = kDrTileB;
    unsigned char* tileA = smem;
    unsigned char* ringB = smem + kTileBytesA;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, njt = (d + 255) / 256;
    const ItemTable& tab = sh.tab;
    uint64_t *full = sh.rfull, *empty = sh.rempty, *tfull = sh.rtfull, *tempty = sh.rtempty;
    const int n_items = tab.n_items();

    if (warp == 0) {
        if (lane == 0) {
            int it = 0, ii = 0;
            for (int v = blockIdx.x; v < n_items; v += gridDim.x, ii++) {
                const Item w = tab.item(v);
                if (ii >= 1) mbar_wait(&sh.aempty, (uint32_t)(ii - 1) & 1u, status, lim);
                mbar_arrive_expect_tx(&sh.afull, kTileBytesA);
                tma_load_2d(tileA, &map_h, 0, w.a0, &sh.afull);
                for (int jt = 0; jt < njt; jt++, it++) {
                    const int s = it % kStages;
                    if (it >= kStages) mbar_wait(&empty[s], (uint32_t)((it / kStages) - 1) & 1u, status, lim);
                    mbar_arrive_expect_tx(&full[s], kTileB);
                    tma_load_2d(ringB + (size_t)s * kTileB, &map_wd, w.e * 64, jt * 256, &full[s]);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16_m128(256);
            int it = 0, acc = 0, ii = 0;
            for (int v = blockIdx.x; v < n_items; v += gridDim.x, ii++) {
                mbar_wait(&sh.afull, (uint32_t)ii & 1u, status, lim);
                for (int jt = 0; jt < njt; jt++, it++, acc++) {
                    const int a = acc & 1;
                    if (acc >= 2) mbar_wait(&tempty[a], (uint32_t)((acc >> 1) - 1) & 1u, status, lim);
                    const int s = it % kStages;
                    mbar_wait(&full[s], (uint32_t)(it / kStages) & 1u, status, lim);
                    tc_fence_after();
                    umma_k64(tmem + (uint32_t)(a * 256), tileA, ringB + (size_t)s * kTileB, idesc, false);
                    umma_commit(&empty[s]);
                    umma_commit(&tfull[a]);
                }
                umma_commit(&sh.aempty);
            }
        }
        __syncwarp();
    } else if (warp < 6) {
        const int q = warp & 3;
        const int row = 32 * q + lane;
        // this warp's staging area for bulk stores: four 64-column boxes of
        // its 32 rows in the 128-byte swizzle (conflict-free row writes)
        unsigned char* stage = smem + kTileBytesA + (size_t)kStages * kTileB + (size_t)q * 16384;
        int acc = 0;
        for (int v = blockIdx.x; v < n_items; v += gridDim.x) {
            const Item w = tab.item(v);
            const bool live = row < w.cnt;
            const bool group_live = 32 * q < w.cnt;  // any live row in this warp's 32 rows
            const bool spill = tab.spills(w.e, ycap);  // the expert's rows go to yacc
            // all 32 rows live: the group's rows go out as 2-D bulk stores
            const bool group_full = 32 * q + 32 <= w.cnt && !spill;
            const long long arow = (long long)w.a0 + row;
            const bool in_buf = live && !spill;
            const int tok = live && !in_buf ? ltok[(size_t)w.e * T + w.m0 + row] : -1;
            float* yrow = tok >= 0 ? yacc + (size_t)tok * d : nullptr;
            __nv_bfloat16* Yrow = in_buf ? Y + (size_t)arow * d : nullptr;
            for (int jt = 0; jt < njt; jt++, acc++) {
                const int a = acc & 1;
                mbar_wait(&tfull[a], (uint32_t)(acc >> 1) & 1u, status, lim);
                tc_fence_after();
                const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(a * 256);
                if (group_full) {
                    // two halves of 128 columns; a half's two boxes are rewritten
                    // only after the store that last used them has read them
#pragma unroll 1
                    for (int h = 0; h < 2; h++) {
                        if (lane == 0) bulk_wait_read<1>();
                        __syncwarp();
#pragma unroll 1
                        for (int c = 128 * h; c < 128 * h + 128; c += 32) {
                            uint32_t r[32];
                            tmem_ld32(base + (uint32_t)c, r);
                            tmem_ld_wait();
#pragma unroll
                            for (int vv = 0; vv < 4; vv++) {
                                const int j = (c >> 3) + vv;  // 16-byte chunk of the 256 columns
                                const uint32_t off = (uint32_t)(j >> 3) * 4096u + (uint32_t)lane * 128u +
                                                     ((((uint32_t)j & 7u) ^ ((uint32_t)lane & 7u)) << 4);
                                *reinterpret_cast<uint4*>(stage + off) = make_uint4(
                                    pack_bf16x2(__uint_as_float(r[8 * vv]), __uint_as_float(r[8 * vv + 1])),
                                    pack_bf16x2(__uint_as_float(r[8 * vv + 2]), __uint_as_float(r[8 * vv + 3])),
                                    pack_bf16x2(__uint_as_float(r[8 * vv + 4]), __uint_as_float(r[8 * vv + 5])),
                                    pack_bf16x2(__uint_as_float(r[8 * vv + 6]), __uint_as_float(r[8 * vv + 7])));
                            }
                        }
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            for (int b = 2 * h; b < 2 * h + 2; b++)
                                if (jt * 256 + b * 64 < d)
                                    tma_store_2d(&map_y, stage + b * 4096, jt * 256 + b * 64, w.a0 + 32 * q);
                            bulk_commit();
                        }
                    }
                }
#pragma unroll 1
                for (int c = 0; c < (group_live && !group_full ? 256 : 0); c += 32) {
                    uint32_t r[32];
                    tmem_ld32(base + (uint32_t)c, r);
                    tmem_ld_wait();
                    const int j0 = jt * 256 + c;
                    if (Yrow) {
#pragma unroll
                        for (int v = 0; v < 4; v++)
                            if (j0 + 8 * v < d)
                                *reinterpret_cast<uint4*>(Yrow + j0 + 8 * v) = make_uint4(
                                    pack_bf16x2(__uint_as_float(r[8 * v]), __uint_as_float(r[8 * v + 1])),
                                    pack_bf16x2(__uint_as_float(r[8 * v + 2]), __uint_as_float(r[8 * v + 3])),
                                    pack_bf16x2(__uint_as_float(r[8 * v + 4]), __uint_as_float(r[8 * v + 5])),
                                    pack_bf16x2(__uint_as_float(r[8 * v + 6]), __uint_as_float(r[8 * v + 7])));
                    } else if (yrow) {
#pragma unroll
                        for (int v = 0; v < 8; v++)
                            if (j0 + 4 * v < d)
                                red_add_v4(yrow + j0 + 4 * v, __uint_as_float(r[4 * v]), __uint_as_float(r[4 * v + 1]),
                                           __uint_as_float(r[4 * v + 2]), __uint_as_float(r[4 * v + 3]));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[a]);
            }
        }
        if (lane == 0) bulk_wait_all();  // the stores are done before the CTA's shared memory goes away
        __syncwarp();
    }
}

// The form goes by the call's tokens per work item and by its items, which only
// the device knows.  With tokens as M an item costs the same however few tokens
// it has, and fewer items than SMs leave SMs idle; with weights as M an item
// costs by its tokens.  Whole layers, us, weights / tokens as M (tokens an item):
//   8B, 300 tokens    (32) 144/146   (48) 165/161   (80) 217/195   (86, 2 items an expert) 392/293
//   13B, 2000 tokens  (28) 156/167   (46) 184/182   (83) 245/225
//   GPT-2-medium, 600 tokens  (47, 64 items) 29/30   (81, 104 items) 40/38
//   d = 4096, 12 experts, 300 tokens  (100, 12 items) 49/67
// By the call's tokens alone (rows above 1024) dense prompts of 257 to 1024
// tokens took up to half as long again: 13B, 1024 tokens, every expert 2577 us,
// 1738 by this rule.
constexpr int kDownRowsMinItem = 48;

__global__ void __launch_bounds__(kDnThreads, 1)
    down_kernel(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_wd,
                const __grid_constant__ CUtensorMap map_h128, const __grid_constant__ CUtensorMap map_wd256,
                const __grid_constant__ CUtensorMap map_y, const int* __restrict__ cnt, const int* __restrict__ ltok, int T,
                int E, int d, __nv_bfloat16* Y, long long ycap, float* yacc, unsigned* status, uint64_t lim) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ DownShared sh;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kDnStages; i++) {
            mbar_init(&sh.full[i], 1);
            mbar_init(&sh.empty[i], 1);
        }
        for (int i = 0; i < kDnAcc; i++) {
            mbar_init(&sh.tfull[i], 1);
            mbar_init(&sh.tempty[i], kDnEpi);
        }
        for (int i = 0; i < kDrStages; i++) {
            mbar_init(&sh.rfull[i], 1);
            mbar_init(&sh.rempty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&sh.rtfull[i], 1);
            mbar_init(&sh.rtempty[i], 4);
        }
        mbar_init(&sh.afull, 1);
        mbar_init(&sh.aempty, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(&sh.taddr, 512);
        tmem_relinquish();
    }
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    sh.tab.build(cnt, E);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.taddr;
    if (sh.tab.n_pairs() >= kDownRowsMinItem * sh.tab.n_items() && 2 * sh.tab.n_items() >= (int)gridDim.x)
        down_rows(map_h128, map_wd256, map_y, sh, smem, tmem, ltok, T, d, Y, ycap, yacc, status, lim);
    else
        down_tiles(map_h, map_wd, sh, smem, tmem, ltok, T, d, Y, ycap, yacc, status, lim);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// =================================================================== combine
// y[t] = the sum of token t's assignment rows Y[pos] in ascending expert
// order, plus yacc[t] when the call's pairs exceed the row buffer.  Grid (T, ceil(d / 1024)): 128 threads of 8 columns each.
// The expert list is built in parallel: 128 experts per round, compacted in
// ascending order with ballots.
__global__ void __launch_bounds__(128) combine_kernel(const uint32_t* __restrict__ bits, const int* __restrict__ slot_of,
                                                      const int* __restrict__ offsets,
                                                      const __nv_bfloat16* __restrict__ Y, long long ycap,
                                                      const float* __restrict__ yacc, int T, int E, int d,
                                                      __nv_bfloat16* y) {
    pdl_wait();  // the previous kernel on the stream has completed (programmatic dependent launch)
    pdl_launch_dependents();
    const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int pos_s[kMaxExperts];
    __shared__ int wn_s[4];
    int n = 0;
    for (int e0 = 0; e0 < E; e0 += 128) {
        const int e = e0 + tid;
        bool on = e < E && ((bits[(size_t)t * 8 + (e >> 5)] >> (e & 31)) & 1u);
        const int pos = on ? offsets[e] + slot_of[(size_t)t * E + e] : 0;
        on = on && offsets[e + 1] <= ycap;
        const unsigned bal = __ballot_sync(kFull, on);
        if (lane == 0) wn_s[warp] = __popc(bal);
        __syncthreads();
        int base = n;
        for (int w = 0; w < warp; w++) base += wn_s[w];
        if (on) pos_s[base + __popc(bal & ((1u << lane) - 1u))] = pos;
        n += wn_s[0] + wn_s[1] + wn_s[2] + wn_s[3];
        __syncthreads();
    }
    const int c = blockIdx.y * 1024 + tid * 8;
    if (c >= d) return;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (offsets[E] > ycap) {
        const float4* ya = reinterpret_cast<const float4*>(yacc + (size_t)t * d + c);
        const float4 a0 = ya[0], a1 = ya[1];
        acc[0] = a0.x; acc[1] = a0.y; acc[2] = a0.z; acc[3] = a0.w;
        acc[4] = a1.x; acc[5] = a1.y; acc[6] = a1.z; acc[7] = a1.w;
    }
    // rows added in ascending expert order; their loads go out 4 at a time
    for (int i0 = 0; i0 < n; i0 += 4) {
        uint4 v4[4];
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (i0 + u < n) v4[u] = *reinterpret_cast<const uint4*>(Y + (size_t)pos_s[i0 + u] * d + c);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (i0 + u >= n) break;
            const uint4 v = v4[u];
            acc[0] += bf16lo(v.x); acc[1] += bf16hi(v.x); acc[2] += bf16lo(v.y); acc[3] += bf16hi(v.y);
            acc[4] += bf16lo(v.z); acc[5] += bf16hi(v.z); acc[6] += bf16lo(v.w); acc[7] += bf16hi(v.w);
        }
    }
    *reinterpret_cast<uint4*>(y + (size_t)t * d + c) =
        make_uint4(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]), pack_bf16x2(acc[4], acc[5]),
                   pack_bf16x2(acc[6], acc[7]));
}

// ====================================================================== host
namespace {

template <int NE>
cudaError_t launch_router(const CUtensorMap& mx, const CUtensorMap& mwr, int T, int E, int nk, int kpb, int nsplit,
                          float* part, int* cnt, unsigned* status, uint64_t lim, cudaStream_t st) {
    const size_t smem = 4 * (size_t)(kTileBytesA + NE * 128) + 1024;
    cudaError_t e = set_smem(router_gemm_kernel<NE>, smem);
    if (e != cudaSuccess) return e;
    PP_LAUNCH(router_gemm_kernel<NE>, dim3((T + 127) / 128, nsplit), dim3(kTcThreads), smem, st, mx, mwr, T, E, nk,
        kpb, part, cnt, status, lim);
    return cudaGetLastError();
}

}  // namespace

GroupedPlan grouped_plan(int T, int d, int E, int sms) {
    GroupedPlan g{};
    g.nk = (d + 63) / 64;  // the last chunk's columns past d are zero-filled by TMA
    // router K splits: at most one wave of CTAs, at least 4 chunks each
    const int mt = (T + 127) / 128;
    const int ns = std::max(1, std::min(sms / mt, std::min(g.nk / 4, 64)));
    g.kpb = (g.nk + ns - 1) / ns;
    g.nsplit = (g.nk + g.kpb - 1) / g.kpb;
    g.nnz_max = (long long)T * E;
    g.ycap = (long long)T * std::min(E, 64);  // assignment rows kept for the combine
    return g;
}

// nsplit(t) is at most the K chunks' limit and at most sms / ceil(t / 128), or 1:
// it falls as t crosses a multiple of 128, so nsplit(t) * t does too, and the
// bound is the largest of either limit's products.
size_t router_part_rows(int T, int d, int sms) {
    const size_t t = (size_t)std::max(T, 1);
    const size_t most = (size_t)std::max(1, std::min((d + 63) / 64 / 4, 64));
    return std::max(t, std::min(t * most, (size_t)sms * 128));
}

cudaError_t grouped_route(const GroupedArgs& a, cudaStream_t st) {
    const GroupedPlan& g = a.plan;
    CUtensorMap mx, mwr;
    const int NE = router_ne(a.E);
    int* cnt = a.bits ? a.cnt : nullptr;  // the FFN's lists
    if (!encode_2d(&mx, a.x, a.d, a.T, 64, 128) || !encode_2d(&mwr, a.Wr, a.d, a.E, 64, NE)) return cudaErrorInvalidValue;
    cudaError_t e;
    switch (NE) {
        case 32: e = launch_router<32>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
        case 64: e = launch_router<64>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
        case 128: e = launch_router<128>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
        case 160: e = launch_router<160>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
        case 192: e = launch_router<192>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
        case 224: e = launch_router<224>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
        default: e = launch_router<256>(mx, mwr, a.T, a.E, g.nk, g.kpb, g.nsplit, a.part, cnt, a.status, a.timeout_ns, st); break;
    }
    if (e != cudaSuccess) return e;
    if (a.T <= kCtaSelectMaxTokens) {  // pp_route: the union kernel makes its own selection
        PP_LAUNCH(select_part_cta_kernel, dim3(a.T), dim3(256), 0, st, a.part, g.nsplit, a.T, a.E, a.p, a.rule, a.gate,
                  a.ids, a.counts, a.gates, a.logits_out, a.status);
        return cudaGetLastError();
    }
    const dim3 grid((a.T + 7) / 8), block(256);
    const Lists lists{a.cnt, a.ltok, a.lgate, a.slot_of};
#define PP_SELECT(S)                                                                                                   \
    PP_LAUNCH(select_warp_kernel<S>, grid, block, 0, st, a.part, g.nsplit, a.T, a.E, a.p, a.rule, a.gate, a.ids, a.counts, \
              a.gates, a.logits_out, a.bits, lists, a.status)
    switch (sel_slots_for(a.E)) {
        case 1: PP_SELECT(1); break;
        case 2: PP_SELECT(2); break;
        case 4: PP_SELECT(4); break;
        default: PP_SELECT(8); break;
    }
#undef PP_SELECT
    return cudaGetLastError();
}

cudaError_t grouped_load_selection(const GroupedArgs& a, cudaStream_t st) {
    const bool lists = a.cnt != nullptr && a.T > kUnionMaxT;
    PP_LAUNCH(dispatch_bits_kernel, dim3((a.T + 7) / 8), dim3(256), 0, st, a.ids, a.counts, a.gates, a.T, a.E, a.bits,
              a.gexp, lists ? a.cnt : nullptr, a.status);
    if (lists)
        PP_LAUNCH(dispatch_list_kernel, dim3((a.T + 7) / 8), dim3(256), 0, st, a.bits, a.gexp, a.T, a.E,
                  Lists{a.cnt, a.ltok, a.lgate, a.slot_of});
    return cudaGetLastError();
}

cudaError_t grouped_ffn(const GroupedArgs& a, int sms, cudaStream_t st) {
    if (a.T <= kUnionMaxT) return union_layer(a, false, sms, st);
    const GroupedPlan& g = a.plan;
    const bool gated = a.act == PP_ACT_SWIGLU;
    const uint64_t rows = (uint64_t)a.E * 64;
    CUtensorMap mx, mwg, mwu, mh, mwd;
    if (!encode_2d(&mx, a.x, a.d, a.T, 64, 1) || !encode_2d(&mwu, a.Wu, a.d, rows, 64, kGuBox) ||
        !encode_2d(&mwg, gated ? a.Wg : a.Wu, a.d, rows, 64, kGuBox) ||
        !encode_2d(&mh, a.H, 64, (uint64_t)g.nnz_max + 128, 64, kDnBox) ||
        !encode_2d(&mwd, a.Wd, rows, a.d, 64, 128, CU_TENSOR_MAP_L2_PROMOTION_L2_128B))
        return cudaErrorInvalidValue;
    // (down: the larger of the two forms' rings and staging areas)
    const size_t gu_smem = kGuRing + kGuSlack + 1024;
    const size_t dn_smem =
        std::max(kDnRing + 4 * kDnStageOut, (size_t)kTileBytesA + kDrStages * (size_t)kDrTileB + 4 * (size_t)16384) + 1024;
    CUtensorMap mh128, mwd256, my;
    if (!encode_2d(&mh128, a.H, 64, (uint64_t)g.nnz_max + 128, 64, 128) ||
        !encode_2d(&mwd256, a.Wd, rows, a.d, 64, 256, CU_TENSOR_MAP_L2_PROMOTION_L2_128B) ||
        !encode_2d(&my, a.Y, a.d, (uint64_t)g.ycap, 64, 32))
        return cudaErrorInvalidValue;
    cudaError_t e;
    if ((e = set_smem(gu_gemm_kernel, gu_smem)) != cudaSuccess || (e = set_smem(down_kernel, dn_smem)) != cudaSuccess)
        return e;
    PP_LAUNCH(gu_gemm_kernel, dim3(sms), dim3(kGuThreads), gu_smem, st, mx, mwg, mwu, a.cnt, a.ltok, a.lgate, a.offsets, a.T,
              a.E, a.d, g.nk, a.act, a.H, g.ycap, a.yacc, a.status, a.timeout_ns);
    PP_LAUNCH(down_kernel, dim3(sms), dim3(kDnThreads), dn_smem, st, mh, mwd, mh128, mwd256, my, a.cnt, a.ltok, a.T, a.E, a.d,
              a.Y, g.ycap, a.yacc, a.status, a.timeout_ns);
    PP_LAUNCH(combine_kernel, dim3(a.T, (a.d + 1023) / 1024), dim3(128), 0, st, a.bits, a.slot_of, a.offsets, a.Y, g.ycap,
              a.yacc, a.T, a.E, a.d, reinterpret_cast<__nv_bfloat16*>(a.y));
    return cudaGetLastError();
}

}  // namespace pp
