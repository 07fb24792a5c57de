// The FFN over the union of a call's selected experts, for kernels of one CTA
// per SM that have made the selection: gate/up, down projection and the sum of
// its partial tiles (union.cu says how the work is cut and why).  Used by the
// union kernel (union.cu) and, when a call of 2 to 4 tokens selects many
// experts, by the fused decode kernel (decode.cu).
//
// Warps: 0-3 producers of the gate/up ring and epilogues (TMEM lanes
// 32 * warp ..), 4-5 MMA issue, 6 W_down producer, 7 H producer.
#pragma once

#include "pp_common.cuh"
#include "pp_kernels.h"
#include "pp_tc.cuh"

namespace pp {

constexpr int kUnitRows = 16;                 // weight rows of a unit
constexpr int kUnitBytes = kUnitRows * 128;   // per 64-wide K chunk
constexpr int kPassUnits = 16;                // units of one pass: two M = 128 tiles
constexpr int kTileUnits = 128 / kUnitRows;
constexpr int kProd = 4;                      // producer / epilogue warps
constexpr int kMmaWarp = 4;                   // first of the two MMA warps
constexpr int kWdWarp = 6, kHWarp = 7;        // down projection: W_down and H producers
constexpr int kUnionThreads = 256;
constexpr int kMaxStages = 16;
constexpr int kTileW = 128 * 128;             // 128 rows x 64 bf16
// An MMA always reads 128 weight rows, also where the last tile of a gate/up
// pass holds fewer units, so that ring is followed by a tile's worth of slack.
constexpr int kGuSlack = kTileW - kUnitBytes;

PP_DEVINL uint32_t tmem_cols(int n) { return n <= 32 ? 32u : n <= 64 ? 64u : n <= 128 ? 128u : n <= 256 ? 256u : 512u; }

// Ring position: slot and phase parity, advanced without a division.
struct Ring {
    int s = 0;
    uint32_t ph = 0;
    PP_DEVINL void next(int n) {
        if (++s == n) {
            s = 0;
            ph ^= 1u;
        }
    }
};

// The L = tiles * nU (row tile, union expert) pairs of the down projection (at
// most 64 * 256) are cut into runs, one per CTA b < run_count; CTAs past it
// have none.  A run has at least kMinRun pairs: every run ends in a partial
// tile that the reduction reads back.
constexpr int kMinRun = 2;
PP_DEVINL int run_count(int L, int G) { return max(1, min(G, L / kMinRun)); }
PP_DEVINL int run_begin(int L, int b, int R) { return b >= R ? L : L * b / R; }
// The run that holds pair i: run_begin(b) <= i < run_begin(b + 1).
PP_DEVINL int run_of(int L, int i, int R) { return ((i + 1) * R - 1) / L; }

// kRing: bytes of shared memory for a phase's ring.  `gate(t, e)` in the functions
// below is the gate weight of token t for expert e, +0 where the token did not
// select it (a weight of zero is -0).
PP_DEVINL bool selected(float gate) { return __float_as_uint(gate) != 0u; }

template <int MaxT>
struct UnionShared {
    uint64_t full[kMaxStages], empty[kMaxStages], tfull;             // gate/up
    uint64_t dfull[kMaxStages], dempty[kMaxStages], dt[2], de[2];    // down
    unsigned long long bar_target;  // arrivals that complete the last barrier this CTA has joined
    uint32_t taddr;
    int ul[kMaxExperts];  // the union, ascending
    float gw[kPassUnits / 4 + 1][MaxT];  // gate weights of the pass's experts
};

// Every thread of the CTA: what it wrote is visible to every CTA's reads after.
template <int MaxT>
PP_DEVINL void grid_sync(const UnionFfn& a, UnionShared<MaxT>& sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
        grid_arrive(a.bar);
        sh.bar_target += kBarrierSum;
        grid_wait(a.bar, sh.bar_target, a.status, a.lim);
    }
    __syncthreads();
}
// MMA warps of the down projection: two take a run's pairs in turn, each with
// its own two accumulators (added in the epilogue); above 128 tokens the four
// accumulators would not fit the tensor memory.
PP_DEVINL int down_mma(int N) { return N <= 128 ? 2 : 1; }

// Run of this CTA in the down projection.
template <int kRing>
struct DownRun {
    int R, n, tile0, first, stage, nst;
    PP_DEVINL DownRun(const UnionFfn& a, int nU) {
        const int L = a.ntile * nU;
        R = run_count(L, gridDim.x);
        const int i0 = run_begin(L, blockIdx.x, R);
        n = run_begin(L, blockIdx.x + 1, R) - i0;
        tile0 = n > 0 ? i0 / nU : 0;
        first = n > 0 ? i0 % nU : 0;
        stage = kTileW + a.N * 128;
        nst = min(kMaxStages, kRing / stage) & ~1;  // even, as in gu_phase
    }
};

template <int kRing, int MaxT>
PP_DEVINL void load_wd(const UnionFfn& a, UnionShared<MaxT>& sh, unsigned char* smem, const DownRun<kRing>& d, int slot, int u, int tile) {
    mbar_arrive_expect_tx(&sh.dfull[slot], (uint32_t)kTileW);
    tma_load_2d(smem + (size_t)slot * d.stage, &a.map_wd, sh.ul[u] * kDExpert, tile * 128, &sh.dfull[slot]);
}

// The first W_down tiles of the run, one ring's worth (lane 0 of warp kWdWarp).
template <int kRing, int MaxT>
PP_DEVINL void wd_prologue(const UnionFfn& a, UnionShared<MaxT>& sh, unsigned char* smem, int nU) {
    if ((threadIdx.x & 31) == 0) {
        const DownRun<kRing> d(a, nU);
        int u = d.first, tile = d.tile0;
        for (int i = 0; i < min(d.n, d.nst); i++) {
            load_wd(a, sh, smem, d, i, u, tile);
            if (++u == nU) {
                u = 0;
                tile++;
            }
        }
    }
    __syncwarp();
}

// An activation in bf16, or as three bf16 terms (24 bits: the fp32 value) whose
// rows are `next` elements apart.
PP_DEVINL void store_h(__nv_bfloat16* p, float h, int terms, size_t next) {
    const __nv_bfloat16 hi = __float2bfloat16_rn(h);
    *p = hi;
    if (terms == 1) return;
    const float r = isfinite(h) ? h - __bfloat162float(hi) : 0.0f;
    const __nv_bfloat16 mid = __float2bfloat16_rn(r);
    p[next] = mid;
    p[2 * next] = __float2bfloat16_rn(r - __bfloat162float(mid));
}

// Out of line: the epilogue runs once per launch and is bound by instruction
// fetch (unrolled inline, 16 copies of the tanh form took 4.4 us at 16 tokens, 3.6 now).
static __device__ __noinline__ float union_act(int act, float u, float g) { return act_h(act, u, g); }

// h = act(gate, up) * gate weight of the pass's units [base, base + nun), bf16,
// at H[t][union position * 64 + neuron].  Warps w and w + 4 share the TMEM lanes
// 32 (w % 4) .. and take every other 16 tokens.  A token that did not select
// the expert (most do not: 5 % of the pairs at 64 tokens of the 8B shape) costs
// a store of zero and no activation.  `halves`: the sums are those of two
// accumulators.
// UN: how far the loops over the tokens are unrolled.  A column block of 16 that
// is run once is bound by instruction fetch, so it is rolled (8 tokens of the 8B
// shape: 321 -> 313 us for 8 layers); the four blocks of 64 tokens reuse the
// unrolled code (604 against 612 us).
template <int UN, int MaxT>
PP_DEVINL void gu_epilogue(const UnionFfn& a, UnionShared<MaxT>& sh, uint32_t tmem, int base, int nun, int upe, bool halves) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3;
    const int T = a.T, N = a.N, p0 = base / upe;
    const bool gated = upe == 8;
    const size_t ldh = (size_t)a.E * kDExpert;
    for (int m = 0; m * kTileUnits < nun; m++) {
        if (m * kTileUnits + q * 2 >= nun) break;  // no unit in this warp's lanes
        const int ui = m * kTileUnits + q * 2 + (lane >> 4);  // this lane's unit of the pass
        const bool live = ui < nun;
        const int g = base + min(ui, nun - 1), p = g / upe;
        const float* gt = sh.gw[p - p0];
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(m * N);
        // lane -> neuron: rows 0-7 of a gated unit are gate rows, 8-15 the up
        // rows of the same neurons
        __nv_bfloat16* Hn = a.H + (size_t)p * kDExpert + (gated ? (g % upe) * 8 + (lane & 7) : (g % upe) * 16 + (lane & 15));
        for (int c = 16 * (warp >> 2); c < N; c += 32) {
            uint32_t v[16];
            tmem_ld16(ta + (uint32_t)c, v);
            if (halves) {
                uint32_t o[16];
                tmem_ld16(ta + (uint32_t)(N + c), o);
                tmem_ld_wait();
#pragma unroll
                for (int k = 0; k < 16; k++) v[k] = __float_as_uint(__uint_as_float(v[k]) + __uint_as_float(o[k]));
            } else {
                tmem_ld_wait();
            }
            if (gated) {
                // gate lanes finish the even tokens, up lanes the odd ones
                const bool up = (lane & 8) != 0;
#pragma unroll UN
                for (int k = 0; k < 8; k++) {
                    const int t = c + 2 * k + (up ? 1 : 0);
                    const float w = live && t < T ? gt[t] : 0.0f;
                    float h = 0.0f;
                    if (__any_sync(kFull, selected(w))) {
                        const float e0 = __uint_as_float(v[2 * k]), e1 = __uint_as_float(v[2 * k + 1]);
                        const float o = __shfl_xor_sync(kFull, up ? e0 : e1, 8);
                        if (selected(w)) h = union_act(PP_ACT_SWIGLU, up ? e1 : o, up ? o : e0) * w;
                    }
                    if (live && t < T) store_h(Hn + (size_t)t * ldh, h, a.terms, T * ldh);
                }
            } else {
#pragma unroll UN
                for (int k = 0; k < 16; k++) {
                    const int t = c + k;
                    const float w = live && t < T ? gt[t] : 0.0f;
                    const float h = selected(w) ? union_act(a.act, __uint_as_float(v[k]), 0.0f) * w : 0.0f;
                    if (live && t < T) store_h(Hn + (size_t)t * ldh, h, a.terms, T * ldh);
                }
            }
        }
    }
    tc_fence_before();
}

// Gate/up over the union.  Bound: HBM (each selected gate/up row read once).
// A TMA instruction costs a warp about 24 ns plus 1.3 ns per 128-byte line it
// moves, so one warp issuing the 1 KB boxes of the units reaches 26 GB/s on its
// SM and four warps 80 GB/s; an SM's share of HBM is 45 GB/s.  Units of 8
// neurons keep every CTA within one unit of the mean (64 tokens of the 8B
// shape: 1488 units on 152 CTAs, 10 at most against 9.8; whole experts left
// two rounds for 186 experts).
// One thread issues an MMA every 55 cycles at best and spends about 300 more on
// a stage's wait and commit, so a single MMA warp took 250 ns per 64-wide chunk
// (16 us of an 8-token call's 24).  Two warps share the work: one M = 128 tile
// each, or, when every pass fits one tile, every other stage each (the two sums
// are added in the epilogue).
// The unused rows of a pass's last tile hold whatever the ring holds; their
// sums stay in accumulator rows that are never read.
template <int kRing, int MaxT, typename Gate>
PP_DEVINL void gu_phase(const UnionFfn& a, UnionShared<MaxT>& sh, Gate gate, unsigned char* smem, uint32_t tmem, int nU) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = a.T, N = a.N, nk = a.nk;
    const bool gated = a.act == PP_ACT_SWIGLU;
    const int upe = gated ? 8 : 4;  // units of an expert
    const int units = nU * upe, G = gridDim.x;
    const int u0 = units * (int)blockIdx.x / G, u1 = units * ((int)blockIdx.x + 1) / G;
    const int most = min(kPassUnits, (units + G - 1) / G);
    const bool two = most > kTileUnits;  // MMA warp m takes tile m; else every other stage
    // a stage holds one K chunk, or two where at least four stages of two fit
    const int xbytes = N * 128, chunk = xbytes + most * kUnitBytes, avail = kRing - kGuSlack;
    const int cps = avail / (2 * chunk) >= 4 ? 2 : 1;
    // With the stages dealt to two MMA warps in turn, the ring is even: a slot is
    // then always the same warp's, which has seen every earlier phase of its
    // full barrier (a parity wait cannot tell a phase from the one two before).
    const int stage = cps * chunk, fit = min(kMaxStages, avail / stage), nst = two ? fit : fit & ~1;
    const int nks = (nk + cps - 1) / cps;
    if (tid == 0) {
        for (int i = 0; i < kMaxStages; i++) {
            mbar_init(&sh.full[i], kProd);
            mbar_init(&sh.empty[i], two ? 2 : 1);
        }
        mbar_init(&sh.tfull, 2);
        fence_mbar_init();
    }
    fence_proxy_async_smem();  // the ring was ordinary shared memory before
    __syncthreads();
    if (u0 == u1 && warp == kWdWarp) wd_prologue<kRing>(a, sh, smem, nU);
    Ring rp, rm;          // producers' and MMA warps' positions
    bool primed = false;  // the ring has been filled once
    uint32_t pass = 0;
    for (int base = u0; base < u1; base += kPassUnits, pass ^= 1u) {
        const int nun = min(kPassUnits, u1 - base);
        if (warp < kProd) {
            // box i of a stage: 0 = the x tile, then the units' weight rows;
            // box i goes out from lane i / 4 of warp i % 4
            const int i = lane * kProd + warp, per = gated ? 2 : 1;
            const int nbox = 1 + nun * per;
            int row = 0, off = 0;
            const CUtensorMap* map = &a.map_x;
            if (i > 0 && i < nbox) {
                const int g = base + (i - 1) / per, half = (i - 1) % per;
                row = sh.ul[g / upe] * kDExpert + (g % upe) * (kDExpert / upe);
                off = xbytes + (i - 1) * (kUnitBytes / per);
                map = gated && half == 0 ? &a.map_wg : &a.map_wu;
            }
            const int nmine = nbox > warp ? (nbox - warp + kProd - 1) / kProd : 0;  // this warp's boxes
            const uint32_t bytes = (uint32_t)(cps * (warp == 0 ? xbytes + (nmine - 1) * (kUnitBytes / per)
                                                               : nmine * (kUnitBytes / per)));
            for (int ks = 0; ks < nks; ks++) {
                if (lane == 0) {
                    if (primed) mbar_wait(&sh.empty[rp.s], rp.ph ^ 1u, a.status, a.lim);
                    mbar_arrive_expect_tx(&sh.full[rp.s], bytes);
                }
                __syncwarp();
                // (a chunk past the row end is filled with zeros)
                if (i < nbox) {
                    unsigned char* dst = smem + (size_t)rp.s * stage + off;
                    tma_load_2d(dst, map, ks * cps * 64, row, &sh.full[rp.s]);
                    if (cps == 2) tma_load_2d(dst + chunk, map, (ks * 2 + 1) * 64, row, &sh.full[rp.s]);
                }
                rp.next(nst);
                if (rp.s == 0) primed = true;
            }
        } else if (warp < kMmaWarp + 2) {
            const int m = warp - kMmaWarp;
            const uint32_t idesc = idesc_bf16_m128(N), acc = tmem + (uint32_t)(m * N);
            const int a0 = xbytes + (two ? m * kTileW : 0);
            if (lane == 0) {
                for (int ks = 0; ks < nks; ks++) {
                    if (two || (ks & 1) == m) {
                        mbar_wait(&sh.full[rm.s], rm.ph, a.status, a.lim);
                        if (two && m * kTileUnits >= nun) {
                            mbar_arrive(&sh.empty[rm.s]);  // no unit in this tile
                        } else {
                            tc_fence_after();
                            unsigned char* st = smem + (size_t)rm.s * stage;
                            umma_k64(acc, st + a0, st, idesc, ks > (two ? 0 : m));
                            if (cps == 2) umma_k64(acc, st + chunk + a0, st + chunk, idesc, true);
                            umma_commit(&sh.empty[rm.s]);
                        }
                    }
                    rm.next(nst);
                }
                umma_commit(&sh.tfull);
            }
            __syncwarp();
        }
        // gate weights of the pass's experts, while the last stages land
        const int p0 = base / upe, np = (base + nun - 1) / upe - p0 + 1;
        if (warp >= kMmaWarp + 2)
            for (int p = 0; p < np; p++)
                for (int t = tid - 32 * (kMmaWarp + 2); t < T; t += 64) sh.gw[p][t] = gate(t, sh.ul[p0 + p]);
        __syncthreads();
        mbar_wait(&sh.tfull, pass, a.status, a.lim);
        // the ring is free: the first W_down tiles may go out
        if (warp == kWdWarp && base + kPassUnits >= u1) wd_prologue<kRing>(a, sh, smem, nU);
        tc_fence_after();
        if (N == 16)
            gu_epilogue<1>(a, sh, tmem, base, nun, upe, !two && nks > 1);
        else
            gu_epilogue<16>(a, sh, tmem, base, nun, upe, !two && nks > 1);
        if (base + kPassUnits < u1) {  // the accumulators and gw are free for the next pass
            __syncthreads();
            tc_fence_after();
        }
    }
}

// y[t][row] without the experts that token t did not select: a zero activation
// times a non-finite weight is NaN in the union's sums, so a non-finite result
// is formed again from the token's own experts.
template <typename Gate>
__device__ __noinline__ float own_experts_only(const UnionFfn& a, Gate gate, const int* ul, int nU, int t, int row) {
    const size_t ld = (size_t)a.E * kDExpert;
    float s = 0.0f;
    for (int u = 0; u < nU; u++) {
        const int e = ul[u];
        if (!selected(gate(t, e))) continue;
        for (int k = 0; k < kDExpert; k++)
            for (int m = a.terms - 1; m >= 0; m--)
                s = fmaf(__bfloat162float(a.H[(size_t)(m * a.T + t) * ld + u * kDExpert + k]),
                         __bfloat162float(a.Wd[(size_t)row * ld + e * kDExpert + k]), s);
    }
    return s;
}

// Down projection over the union: D[128 rows x N] += W_down[tile, expert]
// . H_expert^T, a tile's experts accumulated in TMEM.  Bound: HBM (each
// selected column block of W_down read once; the 64-column block of a tile is
// one 16 KB box).  A run crosses at most `slots - 1` tile boundaries, so CTA b
// writes its i-th tile's sums to slot i of its partials [slots][T][128]; the
// partials of a tile are then added in CTA order, a warp per (tile, token).
// Only the H producer waits for the other CTAs' activations.
template <int kRing, int MaxT, typename Gate>
PP_DEVINL void down_phase(const UnionFfn& a, UnionShared<MaxT>& sh, Gate gate, unsigned char* smem, uint32_t tmem, int nU) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = a.T, TT = a.terms * T, N = a.N, G = gridDim.x;  // TT columns are used
    const DownRun<kRing> d(a, nU);
    const int mm = down_mma(N);
    const int L = a.ntile * nU, R = d.R, n = d.n, tile0 = d.tile0, first = d.first, stage = d.stage, nst = d.nst;
    __syncthreads();  // this CTA's activations are written
    if (tid == 32 * kHWarp) grid_arrive(a.bar);

    if (warp < kProd) {
        const int nseg = n > 0 ? (first + n - 1) / nU + 1 : 0;
        for (int sg = 0; sg < nseg; sg++) {
            const int acc = sg & 1;
            mbar_wait(&sh.dt[acc], (uint32_t)(sg >> 1) & 1u, a.status, a.lim);
            tc_fence_after();
            float* out = a.dpart + ((size_t)blockIdx.x * a.slots + sg) * TT * 128 + 32 * warp + lane;
            const uint32_t ta = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(acc * mm * N);
            // pairs [s0, s1) of the run; a single pair is in the accumulator of its own MMA warp
            const int s0 = max(0, sg * nU - first), s1 = min(n, (sg + 1) * nU - first);
            const bool both = mm == 2 && s1 - s0 > 1;
            const uint32_t tb = both || mm == 1 ? ta : ta + (uint32_t)((s0 & 1) * N);
            for (int c = 0; c < N; c += 16) {
                uint32_t v[16];
                tmem_ld16(tb + (uint32_t)c, v);
                if (both) {
                    uint32_t o[16];
                    tmem_ld16(ta + (uint32_t)(N + c), o);
                    tmem_ld_wait();
#pragma unroll
                    for (int k = 0; k < 16; k++) v[k] = __float_as_uint(__uint_as_float(v[k]) + __uint_as_float(o[k]));
                } else {
                    tmem_ld_wait();
                }
#pragma unroll
                for (int k = 0; k < 16; k++)
                    if (c + k < TT) out[(size_t)(c + k) * 128] = __uint_as_float(v[k]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.de[acc]);
        }
    } else if (warp < kMmaWarp + mm) {
        if (lane == 0) {
            const int m = warp - kMmaWarp;
            const uint32_t idesc = idesc_bf16_m128(N);
            Ring r;
            int u = first, acc = 0;
            bool fresh = true;  // no pair of this segment yet
            for (int i = 0; i < n; i++) {
                const int c = acc & 1;
                if (acc >= 2 && u == 0) mbar_wait(&sh.de[c], (uint32_t)((acc >> 1) - 1) & 1u, a.status, a.lim);
                if ((i & (mm - 1)) == m) {
                    mbar_wait(&sh.dfull[r.s], r.ph, a.status, a.lim);
                    tc_fence_after();
                    unsigned char* st = smem + (size_t)r.s * stage;
                    umma_k64(tmem + (uint32_t)((c * mm + m) * N), st, st + kTileW, idesc, !fresh);
                    umma_commit(&sh.dempty[r.s]);
                    fresh = false;
                }
                r.next(nst);
                if (++u == nU || i + 1 == n) {
                    umma_commit(&sh.dt[c]);
                    acc++;
                    u = 0;
                    fresh = true;
                }
            }
        }
        __syncwarp();
    } else if (warp == kWdWarp) {
        if (lane == 0) {  // after the first ring's worth (wd_prologue)
            Ring r;
            int i = min(n, nst), u = first + i, tile = tile0;
            for (; u >= nU && nU > 0; u -= nU) tile++;
            for (; i < n; i++) {
                mbar_wait(&sh.dempty[r.s], r.ph, a.status, a.lim);
                load_wd(a, sh, smem, d, r.s, u, tile);
                r.next(nst);
                if (++u == nU) {
                    u = 0;
                    tile++;
                }
            }
        }
        __syncwarp();
    } else if (warp == kHWarp) {
        if (lane == 0) {
            sh.bar_target += kBarrierSum;
            grid_wait(a.bar, sh.bar_target, a.status, a.lim);
            fence_proxy_async_global();  // H was written by ordinary stores
            const int hbytes = N * 128;
            Ring r;
            int u = first;
            for (int i = 0; i < n; i++) {
                if (i >= nst) mbar_wait(&sh.dempty[r.s], r.ph ^ 1u, a.status, a.lim);
                mbar_arrive_expect_tx(&sh.dfull[r.s], (uint32_t)hbytes);
                tma_load_2d(smem + (size_t)r.s * stage + kTileW, &a.map_h, u * kDExpert, 0, &sh.dfull[r.s]);
                r.next(nst);
                if (++u == nU) u = 0;
            }
        }
        __syncwarp();
    }
    grid_sync(a, sh);
    for (int q = blockIdx.x * (kUnionThreads / 32) + warp; q < a.ntile * T; q += G * (kUnionThreads / 32)) {
        const int tile = q / T, t = q - tile * T, row = tile * 128 + lane * 4;
        if (row >= a.d) continue;
        float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (nU > 0) {
            const int j0 = tile * nU, b0 = run_of(L, j0, R), b1 = run_of(L, j0 + nU - 1, R);
            // the first run may have begun in an earlier tile; every other run
            // of the tile begins inside it (slot 0)
            const int slot0 = tile - run_begin(L, b0, R) / nU;
            for (int m = a.terms - 1; m >= 0; m--) {  // the smallest term first
                const float* base = a.dpart + (size_t)(m * T + t) * 128 + lane * 4;
                for (int b = b0; b <= b1; b += 8) {
                    float4 v[8];
#pragma unroll
                    for (int k = 0; k < 8; k++)
                        if (b + k <= b1)
                            v[k] = __ldcg(reinterpret_cast<const float4*>(
                                base + ((size_t)(b + k) * a.slots + (b + k == b0 ? slot0 : 0)) * TT * 128));
#pragma unroll
                    for (int k = 0; k < 8; k++)
                        if (b + k <= b1) {
                            s[0] += v[k].x;
                            s[1] += v[k].y;
                            s[2] += v[k].z;
                            s[3] += v[k].w;
                        }
                }
            }
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (!isfinite(s[k])) s[k] = own_experts_only(a, gate, sh.ul, nU, t, row + k);
        }
        *reinterpret_cast<uint2*>(a.y + (size_t)t * a.d + row) = make_uint2(pack_bf16x2(s[0], s[1]), pack_bf16x2(s[2], s[3]));
    }
}
// Barriers of the down projection and the tensor memory, before gu_phase (which
// sets up its own barriers): the columns, for union_end.  Every thread calls;
// its last barrier also orders what the caller wrote to sh.
template <int MaxT>
PP_DEVINL uint32_t union_begin(const UnionFfn& a, UnionShared<MaxT>& sh, uint32_t cols) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int i = 0; i < kMaxStages; i++) {
            mbar_init(&sh.dfull[i], 2);
            mbar_init(&sh.dempty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&sh.dt[i], down_mma(a.N));
            mbar_init(&sh.de[i], kProd);
        }
        fence_mbar_init();
    }
    if (tid >> 5 == kMmaWarp) {
        tmem_alloc(&sh.taddr, cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    return sh.taddr;
}

PP_DEVINL uint32_t union_cols(const UnionFfn& a, int least) {
    return tmem_cols(max(least, a.N * (down_mma(a.N) > 1 ? 4 : 2)));
}

// After down_phase.
PP_DEVINL void union_end(uint32_t tmem, uint32_t cols) {
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x >> 5 == kMmaWarp) tmem_dealloc(tmem, cols);
}

}  // namespace pp
