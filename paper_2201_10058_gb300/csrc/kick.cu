// kick.cu -- all-pairs changeover kick of Eq. Hb (Appendix A "Kick(dt/2)"):
//   a_i = G sum_{j != i} m_j K(r_ij; rc_ij) (x_j - x_i) / r_ij^3
// and the close-encounter pre-check (Appendix A).
//
// GB300 design.  FP64 runs at 1.68 instructions per clock and SM (measured, 1/74
// of FP32), so the kernels minimise FP64 instructions per interaction.  Layouts:
//   * tiled (kick_tile.cu): every ordered pair, one target per thread against groups
//     of 64 sources in shared memory, a grid of equal blocks; on float expansions
//     of the bodies, 3 FP64 instructions per pair (FP64) or none (mixed);
//   * symmetric: each unordered pair once, its force to both bodies (Newton's
//     third law).  The mixed form (kick_ff.cu) is faster than the tiled one from
//     N ~ 6,000 on (12,000: 0.41 ms against 0.58; 4,096: 0.111 against 0.089) and
//     taken where predicted so; the FP64 form (kick_sym_kernel, below), 21 FP64
//     instructions per unordered pair, only on request (20,011: 7.9 ms against
//     2.9 tiled; 128: 0.106 against 0.028).
// The pre-check rides along in both.  Both write partial sums folded in a fixed
// order (deterministic).  The rare pairs inside rc_ij are found by an FP32 test on
// r^2 against a conservative threshold; only those evaluate the changeover function.
//   * kick_kernel: the tiled form without packed bodies, for the allocation-free
//     entry point where its scratch does not hold them (N > 190,282).
//
// kick_kernel, MIXED: FP64 displacement; r^2 formed as an unevaluated sum of two floats
// from an exact integer split of the displacement (no FP64 work); FP32 rsqrt seed
// y0; one Newton correction from the residual e = 1 - r^2 y0^2 (its leading
// part 1 - u y0 by an FP32 FMA on the exact float product u y0, rounded once:
// the float a double residual would be rounded to; the tails in FP32);
// r^-3 = y0^3 (1 + 1.5 e + 1.875 e^2) = m y0^3 + corr in float-float; FP64
// accumulation of (m y0^3) dx, the corrections corr dx (< 2^-19 of each term)
// summed in float-float and added to the FP64 sums with the partials; 6 FP64
// instructions per ordered pair (3 subtractions, 3 accumulations).  FP64: CUDA's
// double rsqrt (17 FP64 instructions per pair, counted).
#include <algorithm>
#include <queue>
#include <utility>
#include <vector>

#include "kick_sym.cuh"

namespace genga {
namespace {

constexpr int kKickThreads = 128;
// Resident blocks per SM the register allocation must allow (128 threads
// each), chosen by measurement at N = 65,540: mixed 5 (at most 96
// registers), FP64 7 (72).
constexpr int kick_min_blocks(bool mixed) {
    return mixed ? 5 : 7;
}
constexpr int kTile = 256;

struct KickArgs {
    const double *x, *y, *z, *m;
    const double *rc, *pc2;
    const float *thr_rc;        // FP32 upper bound of rc^2
    int n;
    int nm;                     // bodies i >= nm are test particles (nm = n: none)
    int chunk;
    double *part;               // [nchunk][6][n]
    uint2 *cand;
    unsigned long long *cand_count;
    unsigned long long cand_cap;
};

// FP32 value of a positive double, mantissa truncated (never above the input);
// 0 for inputs below 2^-126 (including 0).
__device__ __forceinline__ float r2_to_float_trunc(double r2) {
    unsigned hi = (unsigned)__double2hiint(r2);
    unsigned lo = (unsigned)__double2loint(r2);
    unsigned fb = (hi >= 0x38100000u) ? (((hi - 0x38000000u) << 3) | (lo >> 29)) : 0u;
    return __uint_as_float(fb);
}

template <bool MIXED>
__global__ void __launch_bounds__(kKickThreads, kick_min_blocks(MIXED))
kick_kernel(KickArgs A)
{
    __shared__ double sx[kTile], sy[kTile], sz[kTile], sm[kTile];
    __shared__ double sirc[kTile];            // 1 / rc_j
    __shared__ float2 sircf[MIXED ? kTile : 1]; // MIXED: 1 / rc_j as two floats
    __shared__ float sthr[kTile], smh[kTile], sml[kTile];

    const int n = A.n;
    const int i = blockIdx.x * kKickThreads + threadIdx.x;
    const bool valid = i < n;

    double xi = 1e15, yi = 1e15, zi = 1e15;
    double irci = 0.0;                        // 1 / rc_i (infinite for rc_i = 0)
    float thri = 0.0f;
    float2 ircfi = make_float2(0.0f, 0.0f);
    if (valid) {
        xi = A.x[i]; yi = A.y[i]; zi = A.z[i];
        thri = A.thr_rc[i];
        irci = inv_rc(A.rc[i]);
        if (MIXED) ircfi = ff_of_irc(irci);
    }

    const int jbeg = blockIdx.y * A.chunk;
    const int jend = min(n, jbeg + A.chunk);

    double S0 = 0.0, S1 = 0.0, S2 = 0.0;   // compensated chunk totals
    double C0 = 0.0, C1 = 0.0, C2 = 0.0;

    for (int jt = jbeg; jt < jend; jt += kTile) {
        const int cnt = min(kTile, jend - jt);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += kKickThreads) {
            const int j = jt + k;
            sx[k] = A.x[j]; sy[k] = A.y[j]; sz[k] = A.z[j]; sm[k] = A.m[j];
            sthr[k] = A.thr_rc[j];
            sirc[k] = inv_rc(A.rc[j]);
            if (MIXED) sircf[k] = ff_of_irc(sirc[k]);
            if (MIXED) {     // mass as an unevaluated sum of two floats
                const float mh = __double2float_rn(A.m[j]);
                smh[k] = mh;
                sml[k] = __double2float_rn(A.m[j] - (double)mh);
            }
        }
        __syncthreads();

        double ax = 0.0, ay = 0.0, az = 0.0;
        // MIXED: the small correction terms corr * dx (|corr| < 2^-19 m r^-3) of
        // this tile, summed in float-float (TwoSum) and folded into the FP64
        // sums once per tile
        float cxh = 0.0f, cxl = 0.0f, cyh = 0.0f, cyl = 0.0f, czh = 0.0f, czl = 0.0f;
#pragma unroll 4
        for (int k = 0; k < cnt; k++) {
            const int j = jt + k;
            const double dx = sx[k] - xi;
            const double dy = sy[k] - yi;
            const double dz = sz[k] - zi;
            // r^2: FP64 (FP64 form) or Rh + Rl, two floats (MIXED: float-float
            // square sum of the split displacement, relative error ~2^-46).
            // r2f, used only against thresholds with 2^-16 margins, is a
            // float within 2^-23 of r^2.
            double r2 = 0.0;
            float Rh = 0.0f, Rl = 0.0f, hx = 0.0f, hy = 0.0f, hz = 0.0f;
            float r2f;
            if (MIXED) {
                float lx, ly, lz;
                split_f64(dx, hx, lx);
                split_f64(dy, hy, ly);
                split_f64(dz, hz, lz);
                const float px = hx * hx, py = hy * hy, pz = hz * hz;
                const float pxe = fmaf(hx, hx, -px), pye = fmaf(hy, hy, -py), pze = fmaf(hz, hz, -pz);
                const float s1 = px + py, b1 = s1 - px;
                const float e1 = (px - (s1 - b1)) + (py - b1);
                const float s2 = s1 + pz, b2 = s2 - s1;
                const float e2 = (s1 - (s2 - b2)) + (pz - b2);
                const float cross = 2.0f * fmaf(hx, lx, fmaf(hy, ly, hz * lz));
                const float tail = ((e1 + e2) + (pxe + pye + pze)) + cross;
                Rh = s2 + tail;
                Rl = tail - (Rh - s2);
                r2f = Rh;
            } else {
                r2 = fma(dz, dz, fma(dy, dy, dx * dx));
                r2f = r2_to_float_trunc(r2);
            }
            double mk = sm[k];
            float mh = 0.0f, ml = 0.0f;
            if (MIXED) { mh = smh[k]; ml = sml[k]; }
            // Changeover band (rare): K < 1 needs r < rc_ij.  K is flat (zero slope) at
            // r = rc, so the branch may follow the FP32 bound and K uses the r^2 above.
            // The branch runs on few lanes of a warp while the FP64 pipe charges the
            // whole warp: the FP64 form takes r from the Newton rsqrt and
            // 1/rc_ij = min(1/rc_i, 1/rc_j) staged beforehand (no division); MIXED
            // evaluates K in float-float on the FP32 pipe (below).
            const bool band = r2f < fmaxf(thri, sthr[k]);
            if (band && j == i) {
                mk = 0.0; r2 = 1.0; r2f = 1.0f;              // self term: zero, finite
                Rh = 1.0f; Rl = 0.0f;
                mh = 0.0f; ml = 0.0f;
            }
            if (!MIXED && band && j != i)
                mk = mk * changeover_fast(r2 * rsqrt_newton(r2), fmin(irci, sirc[k]));
            {
                double s;
                if (MIXED) {
                    // FP32 seed y0 ~ r^-1; Newton residual e = 1 - r^2 y0^2 with
                    // r^2 = Rh + Rl and Rh y0 = u + ue (exact float product): 1 - u y0
                    // by one FP32 FMA (the product u y0 is exact inside the FMA, so the
                    // result is 1 - u y0 rounded once to a float, error < 2^-46), the
                    // tails ue y0 + Rl y0^2 (~2^-24) in FP32.
                    // r^-3 = y0^3 (1 - e)^(-3/2) = y0^3 (1 + 1.5 e + 1.875 e^2 + O(e^3)),
                    // |e| < 2^-20.  m y0^3 is formed exactly enough (~2^-46) as a sum of
                    // two floats, the correction in FP32, and the parts meet in one FP64 add.
                    const float y0f = rsqrtf(Rh);
                    const float u = Rh * y0f, ue = fmaf(Rh, y0f, -u);   // Rh y0 = u + ue exactly
                    const float e1 = fmaf(-u, y0f, 1.0f);
                    const float p = y0f * y0f, pe = fmaf(y0f, y0f, -p);
                    const float q = p * y0f;
                    float qe = fmaf(p, y0f, -q);
                    qe = fmaf(pe, y0f, qe);
                    const float ef = e1 - fmaf(ue, y0f, Rl * p);
                    if (band && j != i) {      // K in float-float, the mass scaled by it
                        const float2 cj = sircf[k];
                        const bool ci = ircfi.x < cj.x || (ircfi.x == cj.x && ircfi.y <= cj.y);
                        float Kh, Kl;
                        changeover_ff(u, ue, Rl, y0f, ef, ci ? ircfi.x : cj.x, ci ? ircfi.y : cj.y, Kh, Kl);
                        ff_mul(mh, ml, Kh, Kl);
                    }
                    const float ch = q * mh;
                    float ce = fmaf(q, mh, -ch);
                    ce = fmaf(q, ml, ce);
                    ce = fmaf(qe, mh, ce);
                    const float corr = fmaf(ch, fmaf(1.875f * ef, ef, 1.5f * ef), ce);
                    s = f64_of_f32_any(ch);
                    float_two_sum_acc(cxh, cxl, corr * hx);
                    float_two_sum_acc(cyh, cyl, corr * hy);
                    float_two_sum_acc(czh, czl, corr * hz);
                } else {
                    const double yv = rsqrt(r2);
                    s = (mk * yv) * (yv * yv);
                }
                ax = fma(s, dx, ax);
                ay = fma(s, dy, ay);
                az = fma(s, dz, az);
            }
        }
        if (MIXED) {
            ax += f64_of_f32_any(cxh) + f64_of_f32_any(cxl);
            ay += f64_of_f32_any(cyh) + f64_of_f32_any(cyl);
            az += f64_of_f32_any(czh) + f64_of_f32_any(czl);
        }
        {
            double t, e;
            two_sum(S0, ax, t, e); S0 = t; C0 += e;
            two_sum(S1, ay, t, e); S1 = t; C1 += e;
            two_sum(S2, az, t, e); S2 = t; C2 += e;
        }
    }
    if (valid) {
        double *p = A.part + (size_t)blockIdx.y * 6 * n;
        p[0 * (size_t)n + i] = S0;
        p[1 * (size_t)n + i] = S1;
        p[2 * (size_t)n + i] = S2;
        p[3 * (size_t)n + i] = C0;
        p[4 * (size_t)n + i] = C1;
        p[5 * (size_t)n + i] = C2;
    }
}

// Close-encounter pre-check over the pairs i < j: candidates are the pairs
// with r_ij^2 < (f_pc rc_ij)^2, the exact FP64 test in the defining operation
// order (dist2_rn, no contraction).  Most pairs are decided in FP32 from float
// copies of the positions (round to nearest, |x_f - x| <= 2^-24 |x| per
// component): the float distance r_f differs from r by at most
//   m_ij = sqrt(3) 2^-23 (max|x_i| + max|x_j|)   plus relative rounding,
// so r_f^2 >= ((1 + 2^-20) P + m_ij)^2 (1 + 2^-20) is surely outside and
// r_f^2 < ((1 - 2^-20) P - m_ij)^2 (1 - 2^-20) surely inside (P = f_pc rc_ij
// in FP32); only the band between takes the exact test.  Candidates collect
// in a per-warp shared-memory buffer and go to the global list in batches.
constexpr int kPcThreads = 128;
constexpr int kPcI = 4;                         // targets i per thread
constexpr int kPcTile = 512;

constexpr int kPcWarpBuf = 256;                  // per-warp candidate buffer (shared memory)

// Appends the warp's pending candidates to the global list: one atomic per
// flush reserves the space (a single global counter serialises on its L2
// slice, so it is touched about once per hundred candidates).
__device__ __forceinline__ void precheck_flush(const KickArgs &A, const uint2 *buf, unsigned &cnt,
                                               unsigned lane) {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0 && cnt) base = atomicAdd(A.cand_count, (unsigned long long)cnt);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (unsigned t = lane; t < cnt; t += 32) {
        const unsigned long long idx = base + t;
        if (idx < A.cand_cap) A.cand[idx] = buf[t];
    }
    __syncwarp();
    cnt = 0;
}

__global__ void __launch_bounds__(kPcThreads)
precheck_kernel(KickArgs A, double f_pc)
{
    __shared__ float4 sj[kPcTile];                   // x, y, z, P = f_pc rc (floats)
    __shared__ float sM[kPcTile];
    __shared__ uint2 wbuf[kPcThreads / 32][kPcWarpBuf];
    const int n = A.n;
    const int i0 = blockIdx.x * (kPcThreads * kPcI);
    if (i0 >= A.nm) return;                              // only test-particle rows: no pairs
    const int jbeg = max(blockIdx.y * A.chunk, i0 + 1);
    const int jend = min(n, blockIdx.y * A.chunk + A.chunk);
    if (jbeg >= jend) return;                            // block below the diagonal
    const unsigned lane = threadIdx.x & 31u;
    uint2 *buf = wbuf[threadIdx.x >> 5];
    unsigned pend = 0;                                   // candidates in buf (warp-uniform)
    constexpr float kM = 1.7320509f * 1.1920929e-07f;    // sqrt(3) 2^-23
    constexpr float kUp = 1.0f + 9.5367432e-07f, kDn = 1.0f - 9.5367432e-07f;   // 1 +- 2^-20
    float xf[kPcI], yf[kPcI], zf[kPcI], Pi[kPcI], Mi[kPcI];
    int ii[kPcI];
#pragma unroll
    for (int r = 0; r < kPcI; r++) {
        const int i = i0 + r * kPcThreads + threadIdx.x;
        ii[r] = i;
        xf[r] = yf[r] = zf[r] = 3.0e38f; Pi[r] = 0.0f; Mi[r] = 0.0f;
        if (i < n && i < A.nm) {        // a test-particle row pairs only with j > i: none
            xf[r] = f32_of_f64_rn(A.x[i]); yf[r] = f32_of_f64_rn(A.y[i]); zf[r] = f32_of_f64_rn(A.z[i]);
            Pi[r] = (float)f_pc * f32_of_f64_rn(A.rc[i]);
            Mi[r] = kM * fmaxf(fabsf(xf[r]), fmaxf(fabsf(yf[r]), fabsf(zf[r])));
        }
    }
    for (int jt = jbeg; jt < jend; jt += kPcTile) {
        const int cnt = min(kPcTile, jend - jt);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += kPcThreads) {
            const int j = jt + k;
            const float x = f32_of_f64_rn(A.x[j]), y = f32_of_f64_rn(A.y[j]), z = f32_of_f64_rn(A.z[j]);
            sj[k] = make_float4(x, y, z, (float)f_pc * f32_of_f64_rn(A.rc[j]));
            sM[k] = kM * fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
        }
        __syncthreads();
        for (int k = 0; k < cnt; k++) {
            const int j = jt + k;
            const float4 q = sj[k];
            const float Mj = sM[k];
            bool maybe[kPcI];
            bool any = false;
#pragma unroll
            for (int r = 0; r < kPcI; r++) {
                const float dx = q.x - xf[r], dy = q.y - yf[r], dz = q.z - zf[r];
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                const float to = fmaf(fmaxf(Pi[r], q.w), kUp, Mi[r] + Mj);
                maybe[r] = (j > ii[r]) && (r2 < to * to * kUp);
                any |= maybe[r];
            }
            if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
            for (int r = 0; r < kPcI; r++) {
                bool emit = false;
                if (maybe[r]) {
                    const float dx = q.x - xf[r], dy = q.y - yf[r], dz = q.z - zf[r];
                    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                    const float ti = fmaf(fmaxf(Pi[r], q.w), kDn, -(Mi[r] + Mj));
                    if (ti > 0.0f && r2 < ti * ti * kDn) {
                        emit = true;
                    } else {
                        const int i = ii[r];
                        emit = dist2_rn(A.x[j] - A.x[i], A.y[j] - A.y[i], A.z[j] - A.z[i]) <
                               fmax(A.pc2[i], A.pc2[j]);
                    }
                }
                const unsigned ball = __ballot_sync(0xffffffffu, emit);
                if (emit) buf[pend + __popc(ball & ((1u << lane) - 1u))] = make_uint2((unsigned)ii[r], (unsigned)j);
                pend += __popc(ball);
            }
            if (pend > kPcWarpBuf - 32 * kPcI) precheck_flush(A, buf, pend, lane);
        }
    }
    precheck_flush(A, buf, pend, lane);
}

// ---------------------------------------------------------------------------
// Symmetric kick, FP64 form: each unordered pair {i, j} is evaluated once and its
// force goes to both bodies with opposite signs (Newton's third law): the terms
// m_j K r^-3 (x_j - x_i) of a_i and -m_i K r^-3 (x_j - x_i) of a_j share the
// displacement, r^-3 and K.  21 FP64 instructions per unordered pair (the Newton
// rsqrt of common.cuh instead of CUDA's double rsqrt), 10.5 per ordered pair
// against ~17 of kick_kernel.  The mixed form shares the decomposition, with two
// warps per block and two bodies j per lane (kick_ff.cu).
//
// Work decomposition.  Bodies in tiles of 128 (one per thread of a 4-warp
// block), tiles in super-ranges of P tiles.  A work item is a super-tile pair
// (X, Y), X <= Y: the rows a of X (the i-tile, one body per thread, sums in
// registers) against the tiles b of Y (b >= a when X == Y).  In a tile pair,
// warp w holds i-subtile w (32 bodies, one per lane) and meets the j-subtiles
// q = (w + s) mod 4 in four phases s.  In a phase, lane L at step t pairs its
// i with body (L + t) mod 32 of subtile q, whose running sums ride along the
// lanes (one shuffle per step: every j is handled by one lane at a time); at
// the end of the phase the lanes add them to the item's j sums in shared
// memory -- one warp per subtile per phase, so without conflicts and in a fixed
// order.  A diagonal subtile (q = w, a = b) takes the steps 1..16, step 16 on
// lanes 0..15 only: every pair inside it once, no self pair.
//
// Partial sums.  Every body gets one compensated partial per super-range
// (nS = ceil(nT / P)): item (X, Y) writes its row sums to slot Y of the X
// bodies and its j sums to slot X of the Y bodies; a diagonal item (X, X)
// writes both, added, to slot X as each row completes.  Every (slot, body) is
// written exactly once, and kick_fold_kernel adds the slots as whole numbers, so
// the result is deterministic.
//
// Dispatch.  One persistent block per resident block slot takes items from a
// counter in the host's order (largest first, the diagonal items last); the
// host picks P for each N by list-scheduling the items over the resident
// blocks, with the finalize's cost counted.
// Resident blocks per SM the register allocation must allow (128 threads each).
constexpr int sym_min_blocks(bool pc) { return pc ? 6 : 4; }

// Dynamic shared memory of the FP64 form: the staged j tile (x, y, z, m, 1/rc;
// thr), then the item's j sums (x, y, z).
constexpr size_t sym_smem(int P) {
    return (size_t)kSymT * (5 * sizeof(double) + sizeof(float)) + (size_t)P * kSymT * 3 * sizeof(double);
}

__global__ void kick_pack_kernel(const double *rc, const double *pc2, int n, double *irc, float *thr_pc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    irc[i] = inv_rc(rc[i]);
    // rounded up, then 2^-16 more: any float r^2 within 2^-23 of an r^2 below
    // pc2 is below it
    thr_pc[i] = fmaxf(__double2float_ru(pc2[i]) * 1.0000153f, 1.17549435e-38f);
}

// PC: the close-encounter pre-check of Appendix A fused into the kick: a pair
// whose float r^2 (within 2^-23 of r^2) is below max(thr_pc_i, thr_pc_j) takes
// the exact FP64 test of precheck_kernel (dist2_rn, no contraction): the same
// candidates.
template <bool PC, bool TP>
__global__ void __launch_bounds__(kSymT, sym_min_blocks(PC))
kick_sym_kernel(SymArgs A)
{
    extern __shared__ __align__(16) unsigned char sym_sh[];
    double *sx = reinterpret_cast<double *>(sym_sh);
    double *sy = sx + kSymT, *sz = sy + kSymT, *sm = sz + kSymT, *sirc = sm + kSymT;
    const int PT = A.P * kSymT;
    double *jax = sirc + kSymT;
    double *jay = jax + PT, *jaz = jay + PT;
    float *sthr = reinterpret_cast<float *>(jaz + PT);
    __shared__ int s_item;
    __shared__ float sthp[PC ? kSymT : 1];                // thr_pc of the j tile
    __shared__ uint2 pcb[PC ? kSymT / 32 : 1][PC ? kSymPcBuf : 1];
    int pend = 0;                                         // candidates in this warp's buffer

    const int n = A.n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (;;) {
        __syncthreads();                      // the previous item's shared sums are written out
        if (threadIdx.x == 0) s_item = (int)atomicAdd(A.ctr, 1u);
        __syncthreads();
        const int it = s_item;
        if (it >= A.nItems) break;
        const int2 XY = A.items[it];
        const int a0 = XY.x * A.P, a1 = min(A.nT, a0 + A.P);
        const int b0 = XY.y * A.P, b1 = min(A.nT, b0 + A.P);
        const bool diag = XY.x == XY.y;
        const int nj = (b1 - b0) * kSymT;
        for (int e = threadIdx.x; e < nj; e += kSymT) jax[e] = jay[e] = jaz[e] = 0.0;
        for (int a = a0; a < a1; a++) {
            const int i = a * kSymT + threadIdx.x;
            const bool valid = i < n;
            double xi, yi, zi, mi = 0.0, irci = 0.0;
            float thri = 0.0f, thpi = 0.0f;
            if (valid) {
                xi = A.x[i]; yi = A.y[i]; zi = A.z[i]; mi = A.m[i];
                thri = A.thr[i];
                irci = A.irc[i];
                if (PC) thpi = A.thr_pc[i];
            } else {
                xi = yi = zi = pad_pos(threadIdx.x);
            }
            double ax = 0.0, ay = 0.0, az = 0.0;

            for (int b = diag ? a : b0; b < b1; b++) {
                __syncthreads();              // the tile buffer is free
                {
                    const int k = threadIdx.x, j = b * kSymT + k;
                    if (j < n) {
                        sx[k] = A.x[j]; sy[k] = A.y[j]; sz[k] = A.z[j]; sm[k] = A.m[j];
                        sirc[k] = A.irc[j];
                        sthr[k] = A.thr[j];
                        if (PC) sthp[k] = A.thr_pc[j];
                    } else {
                        sx[k] = sy[k] = sz[k] = pad_pos(k); sm[k] = 0.0;
                        sirc[k] = 0.0;
                        sthr[k] = 0.0f;
                        if (PC) sthp[k] = 0.0f;
                    }
                }
                __syncthreads();
                const bool same = a == b;
                for (int s = 0; s < 4; s++) {
                    const int q = (w + s) & 3;
                    if (!same || q >= w) {
                        const bool dsub = same && q == w;
                        const int t0 = dsub ? 1 : 0, t1 = dsub ? 17 : 32;
                        const int qb = q * 32;
                        // running sums of the j body this lane holds: (lane + t) mod 32 at step t
                        double jx = 0.0, jy = 0.0, jz = 0.0;
#pragma unroll 4
                        for (int t = t0; t < t1; t++) {
                            const int k = qb + ((lane + t) & 31);
                            // no contribution and no candidate: the pair lane - 16 takes in
                            // a diagonal subtile's step 16; TP, a pair of two test particles
                            const bool half = (dsub && t == 16 && lane >= 16) ||
                                              (TP && i >= A.nm && b * kSymT + k >= A.nm);
                            const double dx = sx[k] - xi;
                            const double dy = sy[k] - yi;
                            const double dz = sz[k] - zi;
                            const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
                            const float r2f = r2_to_float_trunc(r2);
                            if (PC) {
                                const bool maybe = !half && r2f < fmaxf(thpi, sthp[k]);
                                if (__any_sync(0xffffffffu, maybe)) {
                                    sym_pc_push(pcb[w], pend, lane, maybe, i, b * kSymT + k);
                                    if (pend > kSymPcFlush) sym_pc_flush(A, pcb[w], pend, lane);
                                }
                            }
                            const double yv = rsqrt_newton(r2);
                            double y3 = (yv * yv) * yv;
                            if (r2f < fmaxf(thri, sthr[k]))
                                y3 *= changeover_fast(r2 * yv, fmin(irci, sirc[k]));
                            const double sj = half ? 0.0 : sm[k] * y3;
                            const double si = half ? 0.0 : mi * y3;
                            ax = fma(sj, dx, ax);
                            ay = fma(sj, dy, ay);
                            az = fma(sj, dz, az);
                            jx = fma(-si, dx, jx);
                            jy = fma(-si, dy, jy);
                            jz = fma(-si, dz, jz);
                            // pass the j sums on: lane L takes over lane L + 1's body
                            const int src = (lane + 1) & 31;
                            jx = __shfl_sync(0xffffffffu, jx, src);
                            jy = __shfl_sync(0xffffffffu, jy, src);
                            jz = __shfl_sync(0xffffffffu, jz, src);
                        }
                        // after the last step's hand-over the lane holds body (lane + t1) mod 32
                        const int e = (b - b0) * kSymT + qb + ((lane + t1) & 31);
                        jax[e] += jx;
                        jay[e] += jy;
                        jaz[e] += jz;
                    }
                    __syncthreads();          // subtile sums handed to the next warp
                }
            }
            // row a done: its sums over the tiles of Y (slot Y), or, in a
            // diagonal item, with the j sums of tile a, now complete (slot X)
            if (valid) {
                double S[3] = {ax, ay, az};
                double C[3] = {0.0, 0.0, 0.0};
                if (diag) {
                    const int e = (a - b0) * kSymT + threadIdx.x;
                    const double J[3] = {jax[e], jay[e], jaz[e]};
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        double t;
                        two_sum(S[c], J[c], t, C[c]);
                        S[c] = t;
                    }
                }
                double *pp = A.part + (size_t)(diag ? XY.x : XY.y) * 6 * n;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    pp[(size_t)c * n + i] = S[c];
                    pp[(size_t)(3 + c) * n + i] = C[c];
                }
            }
        }
        if (!diag) {                          // j sums of the Y tiles: slot X
            double *pp = A.part + (size_t)XY.x * 6 * n;
            for (int e = threadIdx.x; e < nj; e += kSymT) {
                const int j = b0 * kSymT + e;
                if (j >= n) continue;
                const double J[3] = {jax[e], jay[e], jaz[e]};
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    pp[(size_t)c * n + j] = J[c];
                    pp[(size_t)(3 + c) * n + j] = 0.0;
                }
            }
        }
    }
    if (PC) sym_pc_flush(A, pcb[w], pend, lane);
}

// A sum of doubles as a 96-bit whole number of 2^(e - 1075 - kFixLow): exact but for
// the bits below 2^-25 of the last place of the largest term.  ~25 integer
// operations per term instead of TwoSum's four FP64 ones (256 cycles of the pipe).
constexpr int kFixLow = 25;                    // 53 + 25 + 17 bits for the number of terms + sign = 96
struct Fix96 {
    unsigned w0, w1;
    int w2;
    int e;                                     // largest exponent field met
    bool bad;                                  // an infinite or NaN term

    // the sum on the scale of exponent field f >= e
    __device__ __forceinline__ void rescale(int f) {
        const int d = f - e;
        e = f;
        const int s = w2 >> 31;
        if (d >= 32) { w0 = w1; w1 = (unsigned)w2; w2 = s; }
        if (d >= 64) { w0 = w1; w1 = (unsigned)w2; }
        if (d >= 96) w0 = (unsigned)s;
        const int r = d >= 96 ? 31 : d & 31;
        w0 = __funnelshift_r(w0, w1, r);
        w1 = __funnelshift_r(w1, (unsigned)w2, r);
        w2 >>= r;
    }
    // += (x2 x1 x0 ^ s) + (s & 1), s = 0 or all ones
    __device__ __forceinline__ void add_words(unsigned x0, unsigned x1, unsigned x2, unsigned s) {
        unsigned r0, r1, r2;
        asm("{\n\t.reg .u32 c, a, b;\n\tadd.cc.u32 c, %3, %3;\n\taddc.cc.u32 a, %4, %7;\n\taddc.cc.u32 b, %5, %8;\n\t"
            "addc.u32 c, %6, %9;\n\tmov.u32 %0, a;\n\tmov.u32 %1, b;\n\tmov.u32 %2, c;\n\t}"
            : "=r"(r0), "=r"(r1), "=r"(r2)
            : "r"(s), "r"(w0), "r"(w1), "r"((unsigned)w2), "r"(x0 ^ s), "r"(x1 ^ s), "r"(x2 ^ s));
        w0 = r0; w1 = r1; w2 = (int)r2;
    }
    __device__ __forceinline__ void add(double v) {
        const int hi = __double2hiint(v);
        const unsigned lo = (unsigned)__double2loint(v);
        int f = (hi >> 20) & 0x7ff;
        bad = bad || f == 0x7ff;
        const unsigned mh = (hi & 0xfffff) | (f ? 0x100000u : 0u);
        f = max(f, 1);
        if (f > e) rescale(f);
        const int d = min(e - f, 127);
        unsigned x2 = mh >> (32 - kFixLow), x1 = __funnelshift_l(lo, mh, kFixLow), x0 = lo << kFixLow;
        if (d & 32) { x0 = x1; x1 = x2; x2 = 0u; }
        if (d & 64) { x0 = x2; x1 = x2 = 0u; }
        x0 = __funnelshift_r(x0, x1, d);
        x1 = __funnelshift_r(x1, x2, d);
        x2 >>= d & 31;
        add_words(x0, x1, x2, (unsigned)(hi >> 31));
    }
    __device__ __forceinline__ void add(Fix96 o) {
        bad = bad || o.bad;
        if (o.e > e) rescale(o.e);
        if (o.e < e) o.rescale(e);
        add_words(o.w0, o.w1, (unsigned)o.w2, 0u);
    }
    __device__ __forceinline__ double value() const {
        const double t = fma((double)w2, 4294967296.0 * 4294967296.0, fma((double)w1, 4294967296.0, (double)w0));
        return scalbn(t, e - 1075 - kFixLow);
    }
};

// Sums a body's partials, one lane per component in each of the block's warps, scales by G (and from the
// packed units, header) and applies the kick v += dt_half a; optionally stores
// a.  COMP: partials are [6][n], with compensations; otherwise [3][n].  mass: the
// partials are forces (unless the header says kFfTwoMass) -- of the symmetric mixed
// kick.  Bodies from tp_first on have tp_slots partials.
// N = 16,384, 128 slots: 24 us; one thread per component and TwoSum, each load
// waiting for the last sum: 118 us with one thread per body, 64 us per component.
// N = 2,048, 64 slots: 6.7 us.
struct FoldArgs {
    const double *part;
    int nslot, tp_first, tp_slots, n;
    double G;
    const int *header;
    const double *mass;
    double dt_half;
    double *vel, *acc_out;
};
constexpr int kFoldWarps = 4;                  // the slots of 32 bodies are dealt to the warps in turn
template <bool COMP>
__global__ void __launch_bounds__(32 * kFoldWarps) kick_fold_kernel(FoldArgs A) {
    __shared__ Fix96 sh[kFoldWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane, c = blockIdx.y;
    const int nslot = i >= A.n ? 0 : i >= A.tp_first ? A.tp_slots : A.nslot;
    const size_t step = (size_t)(COMP ? 6 : 3) * A.n;
    const double *p = A.part + (size_t)c * A.n + i;
    Fix96 sum = {0u, 0u, 0, 1, false};
    constexpr int B = COMP ? 4 : 8;            // slots whose loads are under way together
    for (int q0 = w; q0 < nslot; q0 += B * kFoldWarps) {
        double v[B], u[B];
#pragma unroll
        for (int b = 0; b < B; b++) {
            const int q = q0 + b * kFoldWarps;
            v[b] = q < nslot ? p[q * step] : 0.0;
            if (COMP) u[b] = q < nslot ? p[q * step + (size_t)3 * A.n] : 0.0;
        }
#pragma unroll
        for (int b = 0; b < B; b++) {
            if (q0 + b * kFoldWarps >= A.nslot) break;
            sum.add(v[b]);
            if (COMP) sum.add(u[b]);
        }
    }
    sh[w][lane] = sum;
    __syncthreads();
    if (w || i >= A.n) return;
#pragma unroll
    for (int k = 1; k < kFoldWarps; k++) sum.add(sh[k][lane]);
    const double t = sum.bad ? __longlong_as_double(0x7ff8000000000000ll) : sum.value();
    double f = A.G;
    if (A.header) {
        f *= scalbn(1.0, A.header[1] - 2 * A.header[2]);
        if (A.mass && !(A.header[0] & kFfTwoMass)) f /= A.mass[i] * scalbn(1.0, -A.header[1]);
    }
    const double a = f * t;
    if (A.acc_out) A.acc_out[(size_t)c * A.n + i] = a;
    if (A.dt_half != 0.0) A.vel[(size_t)c * A.n + i] += A.dt_half * a;
}

cudaError_t launch_fold(const FoldArgs &A, bool comp, cudaStream_t stream) {
    const dim3 grid((A.n + 31) / 32, 3);
    if (comp) kick_fold_kernel<true><<<grid, 32 * kFoldWarps, 0, stream>>>(A);
    else kick_fold_kernel<false><<<grid, 32 * kFoldWarps, 0, stream>>>(A);
    return cudaGetLastError();
}

__global__ void raw_thresholds_kernel(int n, const double *rc, float *thr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    thr[i] = fmaxf(__double2float_ru(__dmul_rn(rc[i], rc[i])) * 1.0000153f, 1.17549435e-38f);
}

void kick_geometry(int n, int num_sms, int *chunk, int *nchunk) {
    // (i-tiles x j-chunks) grid
    const int iblocks = (n + kKickThreads - 1) / kKickThreads;
    const int max_chunks = (n + kTile - 1) / kTile;
    // aim for at least 8 blocks per SM, each at least one tile and at most 16
    int want = (8 * num_sms + iblocks - 1) / iblocks;
    int tiles_per_chunk = (max_chunks + want - 1) / (want > 0 ? want : 1);
    if (tiles_per_chunk > 16) tiles_per_chunk = 16;
    if (tiles_per_chunk < 1) tiles_per_chunk = 1;
    if ((max_chunks + tiles_per_chunk - 1) / tiles_per_chunk > kMaxKickChunks)
        tiles_per_chunk = (max_chunks + kMaxKickChunks - 1) / kMaxKickChunks;
    *chunk = tiles_per_chunk * kTile;
    *nchunk = (n + *chunk - 1) / *chunk;
}

}  // namespace

static KickArgs make_args(genga_system *s) {
    KickArgs A;
    const int64_t n = s->n;
    A.x = s->pos; A.y = s->pos + n; A.z = s->pos + 2 * n; A.m = s->mass;
    A.rc = s->rcl[0].rc; A.pc2 = s->rcl[0].pc2;
    A.thr_rc = s->rcl[0].thr_rc;
    A.n = (int)n;
    A.nm = tp_bound(s);
    A.chunk = s->kick_chunk;
    A.part = s->kick_part;
    A.cand = s->cand;
    A.cand_count = &s->ctr->cand_count;
    A.cand_cap = (unsigned long long)s->cand_cap;
    return A;
}

// Symmetric-kick geometry for the system's N and precision: the super-range P
// (0: the symmetric kick is not used), chosen by list-scheduling the items,
// largest first, over the resident blocks and adding the finalize's cost.
namespace {

struct SymPlan {
    int P = 0, nS = 0, blocks = 0;
    int R = 0;                     // super-ranges holding large bodies (TP); nS otherwise
    std::vector<int2> items;
};

double sym_item_cost(int nT, int P, int X, int Y) {
    const int px = std::min(P, nT - X * P), py = std::min(P, nT - Y * P);
    return X == Y ? 0.5 * px * px : (double)px * py;
}

// Items in dispatch order and the predicted makespan (tile-pair units per
// block), each item also costing `ovh` units of fixed work (its tile loads,
// partial-sum writes and dispatch).  Only rows X < Xmax: with test particles,
// a super-range made only of test particles has no pair left with a later one.
double sym_schedule(int nT, int P, int slots, int Xmax, double ovh, std::vector<int2> *order) {
    const int nS = (nT + P - 1) / P;
    std::vector<std::pair<double, int2>> it;
    it.reserve((size_t)nS * (nS + 1) / 2);
    for (int X = 0; X < std::min(nS, Xmax); X++)
        for (int Y = X; Y < nS; Y++) it.push_back({sym_item_cost(nT, P, X, Y), make_int2(X, Y)});
    std::stable_sort(it.begin(), it.end(), [](const std::pair<double, int2> &u, const std::pair<double, int2> &v) {
        return u.first > v.first;
    });
    std::priority_queue<double, std::vector<double>, std::greater<double>> h;
    for (int k = 0; k < slots; k++) h.push(0.0);
    double ms = 0.0;
    for (const auto &e : it) {
        const double t = h.top() + e.first + ovh;
        h.pop();
        h.push(t);
        ms = std::max(ms, t);
    }
    if (order) {
        order->clear();
        for (const auto &e : it) order->push_back(e.second);
    }
    return ms;
}

template <bool MIXED>
SymPlan sym_plan(int n, int nm, int num_sms, double t_best, int req_P) {
    SymPlan best;
    const int nT = (n + kSymT - 1) / kSymT;
    // SM cycles per unordered pair and per partial slot per body in the fold
    const double c_sym = MIXED ? 1.32 : 12.2, c_fin = MIXED ? 7.0 : 9.7;
    // fixed work per item, in tile pairs (mixed: fits the times over P at N = 16,384,
    // 65,540 and 131,071, all within 3 % of the best)
    const double ovh = MIXED ? 0.05 : 0.0;
    // predicted time in SM cycles: the makespan (tile pairs per block, each block at
    // 1/nb of its SM) plus the fold's slots
    for (int P = req_P > 0 ? req_P : 1; P <= (req_P > 0 ? req_P : kSymMaxP); P++) {
        const int nS = (nT + P - 1) / P;
        if ((double)nS * 6.0 * n * sizeof(double) > 16.0 * (1ull << 30)) continue;   // partial sums
        if ((double)nS * (nS + 1) / 2 > 4.0e6) continue;                                // host schedule
        int nb = 0;
        if (MIXED)
            nb = sym_ff_blocks_per_sm(P);
        else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kick_sym_kernel<false, false>, kSymT,
                                                               sym_smem(P)) != cudaSuccess)
            nb = 0;
        if (nb < 1) continue;
        const int slots = nb * num_sms;
        const int R = (nm + P * kSymT - 1) / (P * kSymT);
        const double ms = sym_schedule(nT, P, slots, R, ovh, nullptr);
        const double t = c_sym * (double)kSymT * kSymT * ms * nb + c_fin * (double)nS * n / num_sms;
        if (t < t_best) {
            t_best = t;
            best.P = P; best.nS = nS; best.blocks = slots; best.R = R;
        }
    }
    if (best.P) sym_schedule(nT, best.P, best.blocks, best.R, ovh, &best.items);
    return best;
}

}  // namespace

constexpr size_t kMaxPart = ((size_t)16 << 30) / sizeof(double);      // partial sums, at most

// Chooses the kick geometry for the current N and precision and makes sure the
// partial-sum and packed-body buffers are large enough.
cudaError_t kick_reserve(genga_system *s) {
    const int n = (int)s->n;
    if (s->kick_chunk == 0) kick_geometry(n, s->num_sms, &s->kick_chunk, &s->kick_nchunk);
    const bool mixed = s->p.precision == GENGA_MIXED;
    const int nm = tp_bound(s);
    GENGA_CUDA_TRY(ff_reserve(s));
    if (s->ksym_n != s->n || s->ksym_prec != s->p.precision || s->ksym_nm != nm) {
        const TilePlan tile = tile_plan(n, nm, s->num_sms, mixed, kMaxPart);
        SymPlan plan;
        // FP64: the tiled kick is the faster one at every N
        if (s->ksym_layout == GENGA_KICK_SYMMETRIC || (s->ksym_layout == GENGA_KICK_AUTO && mixed)) {
            const double t = s->ksym_layout == GENGA_KICK_AUTO ? tile.cycles : 1e300;
            plan = mixed ? sym_plan<true>(n, nm, s->num_sms, t, s->ksym_req_P)
                         : sym_plan<false>(n, nm, s->num_sms, t, s->ksym_req_P);
        }
        if (!plan.P && !tile.chunk) return cudaErrorMemoryAllocation;
        s->ktile_chunk = tile.chunk;
        s->ktile_nchunk = tile.nchunk;
        s->ksym_P = plan.P;
        s->ksym_nS = plan.nS;
        s->ksym_blocks = plan.blocks;
        s->ksym_items = (int)plan.items.size();
        s->ksym_R = plan.R;
        if (plan.P) {
            if ((size_t)s->ksym_items > s->ksym_list_cap) {
                if (s->ksym_list) cudaFree(s->ksym_list);
                s->ksym_list = nullptr;
                s->ksym_list_cap = 0;
                GENGA_CUDA_TRY(cudaMalloc((void **)&s->ksym_list, sizeof(int2) * plan.items.size()));
                s->ksym_list_cap = plan.items.size();
            }
            if (!plan.items.empty())
                GENGA_CUDA_TRY(cudaMemcpy(s->ksym_list, plan.items.data(), sizeof(int2) * plan.items.size(),
                                          cudaMemcpyHostToDevice));
            if (!s->ksym_ctr) GENGA_CUDA_TRY(cudaMalloc((void **)&s->ksym_ctr, sizeof(unsigned)));
            if (!mixed && (size_t)n > s->ksym_body_cap) {
                for (void *q : {(void *)s->ksym_irc, (void *)s->ksym_thrpc})
                    if (q) cudaFree(q);
                s->ksym_irc = nullptr; s->ksym_thrpc = nullptr;
                s->ksym_body_cap = 0;
                GENGA_CUDA_TRY(cudaMalloc((void **)&s->ksym_irc, sizeof(double) * (size_t)n));
                GENGA_CUDA_TRY(cudaMalloc((void **)&s->ksym_thrpc, sizeof(float) * (size_t)n));
                s->ksym_body_cap = (size_t)n;
            }
        }
        s->ksym_n = s->n;
        s->ksym_prec = s->p.precision;
        s->ksym_nm = nm;
    }
    const size_t need = (size_t)(s->ksym_P ? s->ksym_nS : s->ktile_nchunk) * (s->ksym_P && !mixed ? 6 : 3) * (size_t)n;
    if (need > s->kick_part_cap) {
        if (s->kick_part) cudaFree(s->kick_part);
        s->kick_part = nullptr;
        s->kick_part_cap = 0;
        GENGA_CUDA_TRY(cudaMalloc((void **)&s->kick_part, sizeof(double) * need));
        s->kick_part_cap = need;
    }
    return cudaSuccess;
}

cudaError_t launch_kick(genga_system *s, double dt_half, bool precheck, double *acc_out) {
    const int n = (int)s->n;
    GENGA_CUDA_TRY(kick_reserve(s));
    const bool mixed = s->p.precision == GENGA_MIXED, sym = s->ksym_P > 0;
    // the pre-check, if asked for, rides along
    SymArgs S;
    S.x = s->pos; S.y = s->pos + n; S.z = s->pos + 2 * (size_t)n; S.m = s->mass;
    S.rc = s->rcl[0].rc; S.irc = s->ksym_irc; S.thr = s->rcl[0].thr_rc; S.thr_pc = s->ksym_thrpc;
    S.n = n; S.nT = (n + kSymT - 1) / kSymT; S.P = s->ksym_P; S.nItems = s->ksym_items;
    S.nm = tp_bound(s);
    S.items = s->ksym_list; S.ctr = s->ksym_ctr; S.part = s->kick_part;
    S.pc2 = s->rcl[0].pc2;
    S.cand = s->cand; S.cand_count = &s->ctr->cand_count; S.cand_cap = (unsigned long long)s->cand_cap;
    FfPack ff = ff_pack_args(s);
    S.body = ff.body; S.ircf = ff.ircf; S.ff_header = ff.header; S.tmass = ff.tmass;
    const bool tp = S.nm < n;
    FoldArgs F;
    F.part = s->kick_part; F.nslot = sym ? s->ksym_nS : s->ktile_nchunk; F.tp_first = n; F.tp_slots = 0; F.n = n;
    F.G = s->p.G; F.header = ff.header; F.mass = nullptr; F.dt_half = dt_half; F.vel = s->vel; F.acc_out = acc_out;
    if (sym && !mixed) {
        F.header = nullptr;
        kick_pack_kernel<<<(n + 255) / 256, 256, 0, s->stream>>>(s->rcl[0].rc, S.pc2, n, s->ksym_irc, s->ksym_thrpc);
        ++s->launches;
        GENGA_CUDA_TRY(cudaMemsetAsync(s->ksym_ctr, 0, sizeof(unsigned), s->stream));
        if (precheck) GENGA_CUDA_TRY(cudaMemsetAsync(&s->ctr->cand_count, 0, sizeof(unsigned long long), s->stream));
        const unsigned nb = (unsigned)s->ksym_blocks;
        const size_t smem = sym_smem(s->ksym_P);
#define GENGA_SYM_LAUNCH(PCK, TPK) kick_sym_kernel<PCK, TPK><<<nb, kSymT, smem, s->stream>>>(S)
        if (tp) { if (precheck) GENGA_SYM_LAUNCH(true, true); else GENGA_SYM_LAUNCH(false, true); }
        else { if (precheck) GENGA_SYM_LAUNCH(true, false); else GENGA_SYM_LAUNCH(false, false); }
#undef GENGA_SYM_LAUNCH
        GENGA_CUDA_TRY(cudaGetLastError());
    } else {
        if (sym) ff.ctr = s->ksym_ctr;
        if (precheck) ff.cand_count = &s->ctr->cand_count;
        GENGA_CUDA_TRY(launch_ff_pack(ff, s->stream, &s->launches));
        if (sym) {
            F.mass = s->mass;
            GENGA_CUDA_TRY(launch_sym_ff(S, precheck, s->ksym_blocks, s->stream));
            ++s->launches;
        } else {
            GENGA_CUDA_TRY(launch_tile_kick(S, s->ktile_chunk, s->ktile_nchunk, mixed, precheck, s->stream));
        }
    }
    if (tp) {                                      // test particles: partials of the large bodies' ranges only
        const int first = sym ? s->ksym_R * s->ksym_P * kSymT : (S.nm + kSymT - 1) / kSymT * kSymT;
        F.tp_first = std::min(first, n);
        F.tp_slots = sym ? s->ksym_R : ((S.nm + 63) / 64 * 32 + s->ktile_chunk - 1) / s->ktile_chunk;
    }
    GENGA_CUDA_TRY(launch_fold(F, sym && !mixed, s->stream));
    s->launches += 2;
    return cudaSuccess;
}

cudaError_t launch_precheck_only(genga_system *s) {
    const int n = (int)s->n;
    if (!s->kick_part) return cudaErrorInvalidValue;
    if (s->kick_chunk == 0) kick_geometry(n, s->num_sms, &s->kick_chunk, &s->kick_nchunk);
    KickArgs A = make_args(s);
    // (i-tile x j-chunk) grid like the kick; blocks wholly below the diagonal return at once
    dim3 grid((n + kPcThreads * kPcI - 1) / (kPcThreads * kPcI), s->kick_nchunk);
    GENGA_CUDA_TRY(cudaMemsetAsync(&s->ctr->cand_count, 0, sizeof(unsigned long long), s->stream));
    precheck_kernel<<<grid, kPcThreads, 0, s->stream>>>(A, s->p.f_pc); ++s->launches;
    return cudaGetLastError();
}

// Launches the kick (no pre-check) on caller-provided arrays; used by the
// allocation-free entry point.  k.scratch holds the packed bodies and the partial
// sums of the tiled kick (kick_tile.cu) where they fit, else thresholds and the
// partial sums of kick_kernel.
cudaError_t launch_kick_raw(const KickRaw &k, int num_sms, cudaStream_t stream) {
    const size_t N = (size_t)k.n;
    FoldArgs F;
    F.nslot = 0; F.tp_first = k.n; F.tp_slots = 0; F.n = k.n; F.G = k.G; F.header = nullptr; F.mass = nullptr;
    F.dt_half = k.dt_half; F.vel = k.vel; F.acc_out = k.acc_out;
    const size_t packed = (ff_bytes(k.n) / sizeof(double) + 31) / 32 * 32;      // doubles
    TilePlan tile;
    if (packed < k.room) tile = tile_plan(k.n, k.n, num_sms, k.mixed, k.room - packed);
    if (tile.chunk) {
        FfPack ff;
        ff.pos = k.pos; ff.m = k.mass; ff.rc = k.rc; ff.pc2 = nullptr; ff.n = k.n; ff.nT = (k.n + kSymT - 1) / kSymT;
        ff_place(ff, k.scratch, ff.nT);
        ff.ctr = nullptr; ff.cand_count = nullptr; ff.window = k.mixed ? kFfWindowMixed : kFfWindow64;
        ff.margin = k.mixed ? kFfMarginMixed : kFfMargin64;
        SymArgs S = {};
        S.x = k.pos; S.y = k.pos + N; S.z = k.pos + 2 * N; S.m = k.mass; S.rc = k.rc;
        S.n = S.nm = k.n; S.nT = ff.nT; S.part = k.scratch + packed;
        S.body = ff.body; S.ircf = ff.ircf; S.ff_header = ff.header; S.tmass = ff.tmass;
        int64_t launches = 0;
        GENGA_CUDA_TRY(launch_ff_pack(ff, stream, &launches));
        GENGA_CUDA_TRY(launch_tile_kick(S, tile.chunk, tile.nchunk, k.mixed, false, stream));
        F.part = S.part; F.nslot = tile.nchunk; F.header = ff.header;
        return launch_fold(F, false, stream);
    }
    const size_t part_off = (N + (N + 1) / 2 + 31) / 32 * 32;                   // 256-byte aligned
    const int max_nchunk = part_off < k.room ? (int)((k.room - part_off) / (6 * N)) : 0;
    if (max_nchunk < 1) return cudaErrorMemoryAllocation;
    int chunk, nchunk;
    kick_geometry(k.n, num_sms, &chunk, &nchunk);
    if (nchunk > max_nchunk) {
        const int tiles = (k.n + kTile - 1) / kTile;
        const int tiles_per_chunk = (tiles + max_nchunk - 1) / max_nchunk;
        chunk = tiles_per_chunk * kTile;
        nchunk = (k.n + chunk - 1) / chunk;
    }
    float *thr = (float *)k.scratch;
    raw_thresholds_kernel<<<(unsigned)((N + 255) / 256), 256, 0, stream>>>(k.n, k.rc, thr);
    GENGA_CUDA_TRY(cudaGetLastError());
    KickArgs A = {};
    A.x = k.pos; A.y = k.pos + k.n; A.z = k.pos + 2 * N; A.m = k.mass;
    A.rc = k.rc; A.thr_rc = thr;
    A.n = A.nm = k.n; A.chunk = chunk; A.part = k.scratch + part_off;
    dim3 grid((k.n + kKickThreads - 1) / kKickThreads, nchunk);
    if (k.mixed) kick_kernel<true><<<grid, kKickThreads, 0, stream>>>(A);
    else kick_kernel<false><<<grid, kKickThreads, 0, stream>>>(A);
    GENGA_CUDA_TRY(cudaGetLastError());
    F.part = A.part; F.nslot = nchunk;
    return launch_fold(F, true, stream);
}

int kick_nchunk_for(int n, int num_sms) {
    int c, nc;
    kick_geometry(n, num_sms, &c, &nc);
    return nc;
}

}  // namespace genga

using namespace genga;

extern "C" int genga_set_kick_layout(genga_system_t *s, int32_t layout, int32_t P) {
    if (!s || layout < GENGA_KICK_AUTO || layout > GENGA_KICK_SYMMETRIC || P < 0 || P > kSymMaxP)
        return GENGA_EINVAL;
    s->ksym_layout = layout;
    s->ksym_req_P = P;
    s->ksym_n = -1;                       // geometry redone by the next kick
    return GENGA_OK;
}

extern "C" int genga_get_kick_layout(genga_system_t *s, int32_t *layout, int32_t *P, int32_t *slots,
                                     int32_t *blocks) {
    if (!s) return GENGA_EINVAL;
    if (kick_reserve(s) != cudaSuccess) return GENGA_ECUDA;
    const bool sym = s->ksym_P > 0;
    if (layout) *layout = sym ? GENGA_KICK_SYMMETRIC : GENGA_KICK_TILED;
    if (P) *P = sym ? s->ksym_P : 0;
    if (slots) *slots = sym ? s->ksym_nS : s->ktile_nchunk;
    if (blocks) *blocks = sym ? s->ksym_blocks : (int32_t)((s->n + kSymT - 1) / kSymT * s->ktile_nchunk);
    return GENGA_OK;
}

