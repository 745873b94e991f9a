// kick_sym.cuh -- what the two arithmetic forms of the symmetric all-pairs
// kick share (kick.cu: FP64, kick_ff.cu: mixed): the work decomposition's
// arguments and the buffered candidate output of the fused pre-check.
#pragma once

#include "common.cuh"

namespace genga {

constexpr int kSymT = 128;                     // bodies per tile
constexpr int kSymMaxP = 6;                    // tiles per super-range, at most

struct SymArgs {
    const double *x, *y, *z, *m;
    const double *irc;          // FP64: 1 / rc per body (inv_rc)
    const float *thr;           // FP64: upper bound of rc^2
    const float4 *body;         // mixed: the bodies as float expansions, by tiles (kick_ff.cu)
    const float2 *ircf;         // mixed: 1 / rc as two floats, padded to whole tiles
    const int *ff_flags;        // mixed: device flags of the inputs (kick_ff.cu)
    const double *tmass;        // mixed: per tile, the bodies' common scaled mass, or 0
    int n, nT, P, nItems;
    int nm;                     // bodies i >= nm are test particles (no pair of two); n: none
    const int2 *items;          // (X, Y) super-tile pairs, X <= Y, in dispatch order
    unsigned *ctr;              // dispatch counter, zero at launch
    double *part;               // FP64 [nS][6][n] (sum, compensation), mixed [nS][3][n] (forces)
    // fused pre-check (PC): candidates i < j with r^2 < max(pc2_i, pc2_j)
    const double *pc2;          // (f_pc rc)^2
    const float *thr_pc;        // FP64: upper bound of pc2 (2^-16 margin)
    const float2 *pcf;          // pc2 as an unevaluated sum of two floats, padded to whole tiles
    uint2 *cand;
    unsigned long long *cand_count;
    unsigned long long cand_cap;
};

constexpr int kSymPcBuf = 128;                 // per-warp candidate buffer (shared memory)

// Far-away stand-in position of the k-th padding body of the last tile:
// distinct for distinct k (no zero separation), massless.
__device__ __forceinline__ double pad_pos(int k) { return 1.0e15 + 1.0e13 * (double)k; }

// Appends a warp's buffered candidates to the global list (one atomic per flush).
__device__ __forceinline__ void sym_pc_flush(const SymArgs &A, const uint2 *buf, int &cnt, int lane) {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0 && cnt) base = atomicAdd(A.cand_count, (unsigned long long)cnt);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int t = lane; t < cnt; t += 32) {
        const unsigned long long idx = base + (unsigned long long)t;
        if (idx < A.cand_cap) A.cand[idx] = buf[t];
    }
    __syncwarp();
    cnt = 0;
}

// One pair's pre-check inside the kick (warp-uniform call).  Lanes with
// `maybe` decide r^2 < max(pc2_i, pc2_j) from the kick's float r^2 (Rh + Rl,
// within rel of r^2) against that pc2 as two floats (pc2 = h + l; rounding to
// nearest is monotone, so the larger pair of floats is the larger pc2): outside
// a band of width `band` around it the sign of (Rh - h) + (Rl - l) decides, on
// the FP32 pipe; inside it (never met in practice) the exact FP64 test of
// precheck_kernel does.  The warp appends its candidates (i < j) to its
// buffer, flushed when it could overflow on the next step.
__device__ __forceinline__ void sym_precheck(const SymArgs &A, uint2 *buf, int &pend, int lane, bool maybe,
                                             int i, int j, float Rh, float Rl, float band) {
    if (!__any_sync(0xffffffffu, maybe)) return;
    bool emit = false;
    if (maybe && i < A.n && j < A.n) {
        const float2 pci = A.pcf[i], pcj = A.pcf[j];
        const float2 P = (pci.x > pcj.x || (pci.x == pcj.x && pci.y >= pcj.y)) ? pci : pcj;
        const float D = (Rh - P.x) + (Rl - P.y);
        const float w = band * P.x;
        if (D < -w) emit = true;
        else if (D > w) emit = false;
        else emit = dist2_rn(A.x[j] - A.x[i], A.y[j] - A.y[i], A.z[j] - A.z[i]) < fmax(A.pc2[i], A.pc2[j]);
    }
    const unsigned ball = __ballot_sync(0xffffffffu, emit);
    if (emit) buf[pend + __popc(ball & ((1u << lane) - 1u))] = make_uint2((unsigned)min(i, j), (unsigned)max(i, j));
    pend += __popc(ball);
    if (pend > kSymPcBuf - 32) sym_pc_flush(A, buf, pend, lane);
}

// kick_ff.cu: the mixed form.
// Bytes of dynamic shared memory of the mixed kernel for super-range P, and the
// resident blocks per SM it reaches with them (0 on error).
size_t sym_ff_smem(int P);
int sym_ff_blocks_per_sm(int P);
// Packs the bodies (float expansions, thresholds) and zeroes the dispatch
// counter and, with pre-check, the candidate count.
constexpr int kFfBoundBlocks = 152;
struct FfPack {
    const double *pos, *m, *rc, *pc2;
    int n, nT;
    float4 *bounds;                   // scratch, kFfBoundBlocks entries
    float4 *body;                     // 4 float4 per body, whole tiles
    float2 *ircf, *pcf;
    double *tmass;                    // per tile
    int *header;                      // flags, the exponents masses and lengths are scaled by
    unsigned *ctr;
    unsigned long long *cand_count;   // NULL: left alone
};
cudaError_t launch_ff_pack(const FfPack &k, cudaStream_t stream, int64_t *launches);
cudaError_t launch_sym_ff(const SymArgs &S, bool precheck, int blocks, cudaStream_t stream);
cudaError_t launch_ff_finalize(const FfPack &k, const double *part, int nslot, int tp_first, int tp_slots, double G,
                               double dt_half, double *vel, double *acc_out, cudaStream_t stream, int64_t *launches);

// 1 / rc: the Newton reciprocal for every rc the FP32 seed can take, an exact
// division for smaller ones, infinite for rc = 0 (so that min(1/rc_i, 1/rc_j) is
// 1 / max(rc_i, rc_j) for any pair).
__device__ __forceinline__ double inv_rc(double rc) {
    if (rc > 1e-30) return rcp_newton(rc);
    return rc > 0.0 ? 1.0 / rc : __longlong_as_double(0x7ff0000000000000ll);
}

}  // namespace genga
