// kick_sym.cuh -- what the two arithmetic forms of the symmetric all-pairs
// kick share (kick.cu: FP64, kick_ff.cu: mixed): the work decomposition's
// arguments and the buffered candidate output of the fused pre-check.
#pragma once

#include "common.cuh"
#include "ff2.cuh"

namespace genga {

constexpr int kSymT = 128;                     // bodies per tile
constexpr int kSymMaxP = 6;                    // tiles per super-range, at most

struct SymArgs {
    const double *x, *y, *z, *m;
    const double *rc;           // critical radii
    const double *irc;          // FP64, symmetric: 1 / rc per body (inv_rc)
    const float *thr;           // FP64: upper bound of rc^2
    const float4 *body;         // mixed: the bodies as float expansions, by tiles (kick_ff.cu)
    const float2 *ircf;         // mixed: 1 / rc as two floats, padded to whole tiles
    const int *ff_header;       // mixed: header of the packed bodies
    const double *tmass;        // mixed: per tile, the bodies' common scaled mass, or 0
    int n, nT, nItems;
    int P;                      // tiles per super-range; tiled kick: steps per chunk
    int nm;                     // bodies i >= nm are test particles (no pair of two); n: none
    const int2 *items;          // (X, Y) super-tile pairs, X <= Y, in dispatch order
    unsigned *ctr;              // dispatch counter, zero at launch
    double *part;               // FP64 [nS][6][n] (sum, compensation), mixed [nS][3][n] (forces)
    // fused pre-check (PC): candidates i < j with r^2 < max(pc2_i, pc2_j)
    const double *pc2;          // (f_pc rc)^2
    const float *thr_pc;        // FP64: upper bound of pc2 (2^-16 margin)
    uint2 *cand;
    unsigned long long *cand_count;
    unsigned long long cand_cap;
};

// Far-away stand-in position of the k-th padding body of the last tile:
// distinct for distinct k (no zero separation), massless.
__device__ __forceinline__ double pad_pos(int k) { return 1.0e15 + 1.0e13 * (double)k; }

// The fused pre-check.  A pair whose float r^2 is below an upper bound of max(pc2_i,
// pc2_j) (2^-16 margin: no candidate is missed) goes to its warp's buffer in
// shared memory, and the whole warp decides a buffer of them at once by the exact
// FP64 test of precheck_kernel.  (Deciding each pair where it is met, from float
// copies of pc2, took 6 ms of the 65,540-body kick's 15: a third of the steps
// meet one, and each waited for its loads.)
constexpr int kSymPcBuf = 128;                 // entries per warp
constexpr int kSymPcFlush = kSymPcBuf - 64;    // decided when more than this are held

// Decides the warp's buffered pairs; the candidates go to the global list (one
// atomic per call).
__device__ __forceinline__ void sym_pc_flush(const SymArgs &A, uint2 *buf, int &cnt, int lane) {
    __syncwarp();
    int kept = 0;
    for (int t0 = 0; t0 < cnt; t0 += 32) {
        const int t = t0 + lane;
        uint2 q = make_uint2(0u, 0u);
        bool emit = false;
        if (t < cnt) {
            q = buf[t];
            const int i = (int)q.x, j = (int)q.y;
            if (i < A.n && j < A.n)
                emit = dist2_rn(A.x[j] - A.x[i], A.y[j] - A.y[i], A.z[j] - A.z[i]) < fmax(A.pc2[i], A.pc2[j]);
        }
        const unsigned ball = __ballot_sync(0xffffffffu, emit);
        __syncwarp();                          // all read their entries before any is overwritten
        if (emit) buf[kept + __popc(ball & ((1u << lane) - 1u))] = make_uint2(min(q.x, q.y), max(q.x, q.y));
        kept += __popc(ball);
    }
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0 && kept) base = atomicAdd(A.cand_count, (unsigned long long)kept);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int t = lane; t < kept; t += 32) {
        const unsigned long long idx = base + (unsigned long long)t;
        if (idx < A.cand_cap) A.cand[idx] = buf[t];
    }
    __syncwarp();
    cnt = 0;
}

// Appends the pairs (i, j) of the lanes with `maybe` (warp-uniform call).
__device__ __forceinline__ void sym_pc_push(uint2 *buf, int &cnt, int lane, bool maybe, int i, int j) {
    const unsigned ball = __ballot_sync(0xffffffffu, maybe);
    if (maybe) buf[cnt + __popc(ball & ((1u << lane) - 1u))] = make_uint2((unsigned)i, (unsigned)j);
    cnt += __popc(ball);
}

// The bodies as float expansions (kick_ff.cu).  A tile of 128 bodies: 7 rows of 64 float4.  Entry g * 32 + l of a row holds
// the bodies l (x, z) and l + 32 (y, w) of group g:
//   0: h_x h_y   1: h_z m_hi   2: m_x m_y   3: m_z m_lo   4: l_x l_y   5: l_z thr_rc
//   6: m_lo2 thr_pc
// (m_hi + m_lo + m_lo2 the scaled mass).  Lengths are in units of 2^-6 S, S = 2^6 > every
// coordinate in them.
constexpr int kFfRow = 64, kFfTile = 7 * kFfRow;
constexpr int kFfScale = 6;
constexpr int kFfTwoMass = 1;                  // flag of the packed bodies, see kick_ff.cu
constexpr int kFfPlain = 0, kFfUniform = 1, kFfGeneral = 2, kFfExact = 3;      // instances of the pair loops
// A body whose coordinates the three floats do not hold has NaN in their place.  Its pairs
// take FP64 -- buffered, 32 at a time, in the tiled kick (mixed, one such body in 4,096: 108
// us against 93; in its own lane: 316), one by one in the symmetric one (16,384: 881
// against 667) --, and with more than one such coordinate per 128 bodies every pair
// takes the instance of FP64 displacements (kFfExact): FP64 kick of 16,384 3.2 ms against
// 2.0 (5.4 for the FP64 symmetric form), mixed kick of 65,540 20.0 against 9.0 (34.9 with
// displacement and sums in FP64).
// So they do where a quarter of the bodies are within 2^-kFfInner of the largest coordinate
// from the star: their pairs would be near ones (r < 2^-20 S), taken one by one.
constexpr int kFfInner = 15;
__device__ __forceinline__ bool ff_exact_pairs(const int *header, int n) {
    return 128ll * header[3] > n || 4ll * header[5] > n;
}
// Bounds of r^2: below, the parts give no displacement in proper order (2^-20 S) or r^-3
// nears the end of the floats' range (kFfExact); above (kFfExact), the same.
constexpr float kFfClose2 = 0x1p-28f, kFfExactClose2 = 0x1p-64f, kFfExactFar2 = 0x1p60f;
// r^2 that stands in for a masked pair's: no bound of a near pair reaches it, so that a
// diagonal tile's steps don't enter the changeover's branch for the body itself (3,001
// bodies whose rc^2 is above 1 in units: 51 us with 1, 41 so).
constexpr float kFfMasked2 = 0x1p56f;
__device__ __forceinline__ f2 f2_lo(const float4 &v) { return f2_make(v.x, v.y); }
__device__ __forceinline__ f2 f2_hi(const float4 &v) { return f2_make(v.z, v.w); }

// kick_ff.cu: the mixed form.
// Bytes of dynamic shared memory of the mixed kernel for super-range P, and the
// resident blocks per SM it reaches with them (0 on error).
size_t sym_ff_smem(int P);
int sym_ff_blocks_per_sm(int P);
// Packs the bodies (float expansions, thresholds) and zeroes the dispatch
// counter and, with pre-check, the candidate count.
constexpr int kFfBoundBlocks = 152;
// Coordinates below 2^-window of their axis' S are not held: their last bits lie below
// the parts.  18: every bit is held (FP64 kick), 25: to 2^-47 (mixed), none: to 2^-72 S,
// enough for a distance (energy).  And how many powers of two S may lie above what nearly
// all bodies reach before a body beyond it is left out: it takes as many from the window.
// (Mixed kick of 16,384 bodies with |z| < 4e-4 and four planets at 0.03: 669 us with 8, 887
// with 4, which leaves the planets out.)
constexpr int kFfWindow64 = 18, kFfWindowMixed = 25, kFfWindowNone = 4096;
constexpr int kFfMargin64 = 4, kFfMarginMixed = 8;
struct FfPack {
    const double *pos, *m, *rc, *pc2;
    int n, nT;
    int window, margin;
    int4 *bounds;                     // scratch, 2 kFfBoundBlocks entries
    float4 *body;                     // whole tiles
    float2 *ircf;
    double *tmass;                    // per tile
    int *header;                      // flags, exponents masses and lengths are scaled by, coordinates not held,
                                      // kFfClose2 (float), inner bodies; 8 ints
    unsigned *ctr;                    // NULL: left alone
    unsigned long long *cand_count;   // NULL: left alone
};
// Makes sure the system's packed-body arrays hold its bodies, and their addresses.
cudaError_t ff_reserve(genga_system *s);
FfPack ff_pack_args(const genga_system *s);
// The same on caller-provided memory: its bytes for n bodies, and the addresses in it.
size_t ff_bytes(int n);
void ff_place(FfPack &k, void *mem, size_t tiles);
cudaError_t launch_ff_pack(const FfPack &k, cudaStream_t stream, int64_t *launches);
cudaError_t launch_sym_ff(const SymArgs &S, bool precheck, int blocks, cudaStream_t stream);     // two launches
// kick_tile.cu: the tiled kick.  Steps (two bodies j) per chunk, chunks, predicted SM
// cycles.  Chunk 0: no plan (max_part, in doubles, holds no partial sums).
struct TilePlan {
    int chunk = 0, nchunk = 0;
    double cycles = 0.0;
};
TilePlan tile_plan(int n, int nm, int num_sms, bool mixed, size_t max_part);
// Partial sums [nchunk][3][n].
cudaError_t launch_tile_kick(const SymArgs &S, int chunk, int nchunk, bool mixed, bool precheck, cudaStream_t stream);

// 1 / rc: the Newton reciprocal for every rc the FP32 seed can take, an exact
// division for smaller ones, infinite for rc = 0 (so that min(1/rc_i, 1/rc_j) is
// 1 / max(rc_i, rc_j) for any pair).
__device__ __forceinline__ double inv_rc(double rc) {
    if (rc > 1e-30) return rcp_newton(rc);
    return rc > 0.0 ? 1.0 / rc : __longlong_as_double(0x7ff0000000000000ll);
}

}  // namespace genga
