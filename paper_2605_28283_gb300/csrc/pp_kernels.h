// Internal launch interfaces of libprunepath (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

#include <cuda_bf16.h>

#include "prunepath.h"

namespace pp {

// ---------------------------------------------------------------- rules
// Whether `rule` is one of the pp_rule values.
inline bool rule_known(int rule) { return rule >= PP_SEL_MIN_PREFIX && rule <= PP_SEL_LTE; }

// The rule parameter p (not NaN) in the form the selection kernels take:
// the mass budget for MIN_PREFIX / PAPER, the count k in [1, E] for TOPK,
// and for LTE the smallest fp32 logit g with sigmoid(g) > p (-inf for
// p <= 0: every logit; +inf for p >= 1: none).
float rule_kernel_param(int rule, float p, int E);

// ---------------------------------------------------------------- decode
struct DecodeArgs {
    CUtensorMap tmap_down;  // W_down [d][d_ff], box {64, R6}; must stay first (64-byte aligned)
    const void* x;
    const void* Wr;
    const void* Wg;
    const void* Wu;
    void* y;
    int32_t* sel_ids;      // route: outputs (CTA 0) or NULL; ffn-only: inputs
    int32_t* sel_counts;
    float* sel_gates;
    float* sel_logits;     // route: optional output
    unsigned long long* tlog;  // [T][E] tagged logits
    unsigned long long* th;    // [|U|][T][64] tagged gate/up activations ([E][8][64] words)
    unsigned* epochs;          // [grid] launch count per CTA (Control.epoch)
    unsigned* status;
    uint64_t timeout_ns;
    int T, d, E;
    int act, gate, rule;
    float p;
    int do_route, do_ffn;
    int R6, NS4, ded6, slots6, hch;
    uint32_t off_x, off_gw, off_mask, off_ulist, off_red, off_red6, off_ring6, off_ring4, off_union;
    // chained step: x = RMSNorm(x_prev + y_prev) * gamma computed in the
    // prologue (a.x is then x_prev); y_prev and gamma staged in the phase-4
    // ring at off_chain (free until phase 4), x written to x_out by CTA 0
    int chain;
    uint32_t off_chain;
    const void* y_prev;
    const void* gamma;
    void* x_out;
    float eps;
    // timeline instantiation only: [grid][kDecodeStamps] global-timer stamps
    unsigned long long* tline;
    int union_min;  // with a UnionFfn: the union kernel's phases do the FFN of this many experts or more
};

// The FFN over the union of a call's selected experts on the tensor cores
// (pp_union.cuh).
struct UnionFfn {
    CUtensorMap map_x, map_wg, map_wu;  // gate/up
    CUtensorMap map_h, map_wd;          // down
    int T, E, d, N, terms, nk, ntile, slots, act;
    __nv_bfloat16* H;  // [terms * T][E * 64]: activations at union position * 64 + neuron
    float* dpart;
    const __nv_bfloat16* Wd;
    __nv_bfloat16* y;
    unsigned long long* bar;
    unsigned* status;
    uint64_t lim;
};

// Phase boundaries recorded by the decode kernel's timeline instantiation,
// per CTA (0 where a CTA skips the phase).
enum DecodeStamp {
    kStEntry = 0,    // first instruction
    kStReleased,     // the preceding grid on the stream has completed
    kStX,            // x (and the launch tag) in shared memory
    kStRouter,       // this CTA's router logits published
    kStSelected,     // every token's selection made (all logits received)
    kStUnion,        // union U of the activated experts formed
    kStIssued4,      // first gate/up row loads issued
    kStPhase4,       // this CTA's gate/up activations published
    kStFirstH,       // warp 0's first activations of phase 6 received
    kStPhase6,       // warp 0's down-projection products done
    kStEnd,          // y written (or the CTA's last phase done)
    kStLogits,       // cumulative-mass cut: every logit of token 0 received (warp 0)
    kStCut,          // cumulative-mass cut: warp 0's part of the count done
    kStCand,         // one-warp cut: candidates of token 0 formed (warp 0)
    kStLanded4,      // warp 0's first gate/up rows landed in shared memory
    kDecodeStamps = 16
};
// SM clock assumed by the timeline stamps between global-timer readings
// (the maximum clock of this GPU, which it runs at under this load)
constexpr long long kStampMHz = 2070;

struct DecodePlanIn {
    int dtype, d, E, TS, grid;
    bool gated;
    size_t smem_limit;
    bool chain = false;  // room for the chained step's y_prev and gamma
};

struct DecodePlan {
    int R6, RPL, NS4, ded6, slots6, hch, threads;
    size_t smem;
    uint32_t off_x, off_gw, off_mask, off_ulist, off_red, off_red6, off_ring6, off_ring4;
    uint32_t off_chain;  // within the phase-4 ring: y_prev [TS][d] then gamma [d]
    uint32_t off_union;  // ring of the union phases: x and everything after it
};

// Part of the per-block shared-memory limit left to the decode kernel's
// static shared memory (selection scratch and counters, 4 KB once padded to
// the 1 KB alignment of the dynamic area).
constexpr size_t kDecodeStaticSmemReserve = 6144;

// The same for the barriers and tables of the union phases, in calls that may
// take them.
constexpr size_t kUnionStaticSmemReserve = 2048;
// Ring of the union phases in the fused decode kernel: what every plan leaves
// after its tables (DecodePlan.off_union).
constexpr int kDecodeUnionRing = 200 * 1024;

bool decode_plan(const DecodePlanIn& in, DecodePlan* out);
// `uni` (NULL: none): the call may do its FFN by the union phases.
cudaError_t decode_launch(const DecodeArgs& a, const DecodePlan& p, int dtype, int TS, int grid,
                          const UnionFfn* uni, cudaStream_t st);
int decode_max_ts(int dtype);

// --------------------------------------------------------- route / select
// Logits and selection of T tokens on the CUDA cores; any output may be NULL
// (ids and gates, and bits and gexp, only together).
struct RouteArgs {
    const void* x;
    const void* Wr;
    int T, d, E, rule, gate;
    float p;
    int32_t* ids;
    int32_t* counts;
    float* gates;
    float* logits;
    uint32_t* bits;
    float* gexp;
    unsigned* status;
};
cudaError_t route_tokens(int dtype, const RouteArgs& a, cudaStream_t st);
// fp32 FFN of T tokens over gexp [T][E] (gate weights, 0: not selected).
struct Ffn32Args {
    const float *x, *Wg, *Wu, *Wd, *gexp;
    float *h, *y;  // h: [T][E * 64] scratch
    int T, d, E, act;
};
constexpr int kFfn32Slice = 1024;  // tokens of a call's scratch; more run in slices
cudaError_t ffn32(const Ffn32Args& a, cudaStream_t st);
cudaError_t select_launch(const float* logits, int T, int E, float p, int rule, int gate,
                          int32_t* ids, int32_t* counts, float* gates, unsigned* status,
                          cudaStream_t st);
cudaError_t stats_launch(const int32_t* counts, int T, int E, uint64_t* acc, cudaStream_t st);
// x[t] = RMSNorm(x_prev[t] + y_prev[t]) * gamma (y_prev, gamma nullable), one CTA per token
cudaError_t rmsnorm_residual_launch(int dtype, const void* x_prev, const void* y_prev, const void* gamma,
                                    float eps, int T, int d, void* x, cudaStream_t st);
int router_stats_blocks(int T);  // parts [blocks][E + 2] floats of router_stats_launch
cudaError_t router_stats_launch(const float* logits, int T, int E, float eps, float* part, double* out,
                                unsigned* status, cudaStream_t st);
cudaError_t wait_timeout_launch(unsigned* flag, unsigned* status, long long timeout_ns,
                                cudaStream_t st);

// ------------------------------------------------- tensor-core grouped path
struct GroupedPlan {
    int nk;          // 64-wide K chunks of d
    int kpb;         // router K chunks per split
    int nsplit;      // router K splits
    long long nnz_max;  // upper bound on (token, expert) assignments
    long long ycap;     // rows of the bf16 assignment-output buffer
};

struct GroupedArgs {
    GroupedPlan plan;
    const void* x;
    const void* Wr;
    const void* Wg;
    const void* Wu;
    const void* Wd;
    void* y;
    int T, d, E, act, gate, rule;
    float p;
    int32_t* ids;
    int32_t* counts;
    float* gates;
    float* logits_out;  // optional final logits
    float* part;        // [nsplit][T][E] router partials
    uint32_t* bits;     // [T][8]
    float* gexp;        // [T][E] gate weight per (token, expert)
    int* slot_of;       // [T][E] slot of the token in the expert's list
    int* cnt;           // [E] list lengths (more than kUnionMaxT tokens)
    int* ltok;          // [E][T] tokens of each expert
    float* lgate;       // [E][T] their gate weights
    int* offsets;       // [E + 1] first row of each expert in H and Y
    __nv_bfloat16* H;   // [nnz_max + 128][64]
    __nv_bfloat16* Y;   // [ycap][d] assignment outputs
    float* yacc;        // [T][d] sums of the pairs past ycap
    float* dpart;       // partial down-projection tiles (union path)
    unsigned long long* bar;  // grid barrier counter (union path)
    unsigned* status;
    uint64_t timeout_ns;
};

// -------------------------------------- union path (up to kUnionMaxT tokens)
// 256 is the most columns an MMA has for the tokens (256 tokens of the 8B shape:
// 125 us per layer against 140 by token lists).
constexpr int kUnionMaxT = 256;
constexpr int kUnionMaxGrid = 152;
size_t union_part_floats(int T, int d);  // of GroupedArgs.dpart

GroupedPlan grouped_plan(int T, int d, int E, int sms);
// Rows of GroupedArgs.part that calls with up to T tokens need: at least
// nsplit(t) * t for every t <= T.
size_t router_part_rows(int T, int d, int sms);
cudaError_t grouped_route(const GroupedArgs& a, cudaStream_t st);
// The FFN over a.bits / a.gexp (the selection as the FFN kernels read it,
// written by grouped_route, or by grouped_load_selection from a.ids, a.counts
// and a.gates).
cudaError_t grouped_load_selection(const GroupedArgs& a, cudaStream_t st);
cudaError_t grouped_ffn(const GroupedArgs& a, int sms, cudaStream_t st);
// The whole layer (do_route), or the FFN alone over a.bits / a.gexp, in one
// cooperative launch; a.T <= kUnionMaxT.  a.ids, a.counts, a.gates may be NULL.
cudaError_t union_layer(const GroupedArgs& a, bool do_route, int sms, cudaStream_t st);
// The FFN part alone, for a kernel of `grid` CTAs (false: no tensor maps).
bool union_ffn_args(const GroupedArgs& g, int grid, UnionFfn* a);
// Columns of the router's MMA for E experts.
inline int router_ne(int E) {
    return E <= 32 ? 32 : E <= 64 ? 64 : E <= 128 ? 128 : E <= 160 ? 160 : E <= 192 ? 192 : E <= 224 ? 224 : 256;
}

// ------------------------------------------------ MoEfication (Sec. 2.2)
// Balanced k-means over the neurons' input weights (host, offline); shapes
// and init already validated.  Returns PP_OK or PP_ERR_HOST.
pp_status moefy_cluster_host(int dtype, const void* Wg, const void* Wu, int dff, int d, int E, const int32_t* init,
                             int max_iter, int32_t* labels, int32_t* perm, int* iters, double* objective);
// perm check + row gather (W_gate, W_up) + column gather (W_down); Wg NULL for non-gated FFNs
cudaError_t moefy_permute_launch(int dtype, const int32_t* perm, const void* Wg, const void* Wu, const void* Wd,
                                 void* Wg_out, void* Wu_out, void* Wd_out, int d, int dff, int sms, unsigned* status,
                                 cudaStream_t st);

// cuTensorMapEncodeTiled through the runtime's driver entry point (nullptr if unavailable)
typedef CUresult (*TensorMapEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                      const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
TensorMapEncodeFn tensor_map_encoder();

inline int sel_slots_for(int E) { return E <= 32 ? 1 : E <= 64 ? 2 : E <= 128 ? 4 : 8; }

}  // namespace pp
