// kick_tile.cu -- the tiled all-pairs kick on packed bodies (kick_ff.cu): every
// ordered pair, one row i per thread against 64-body groups of j in shared
// memory, read by all lanes at once; a (tile of rows) x (chunk of steps) grid of
// equal blocks.  No sums travel between lanes, so a block can be as small as 8 of a
// group's 32 steps: the form for small N, and in FP64 for every N.
//
//   mixed   the pair arithmetic of kick_ff.cu (displacement, r^-3, K and the term
//           m_j r^-3 d as two floats each, sums in two floats handed to FP64 after
//           16 steps): ~105 FP32 operations per ordered pair.  Pairs of bodies whose
//           coordinates three floats do not hold go to a buffer, as below.
//   FP64    results of full double precision with 3 FP64 FMAs per ordered pair.
//           FP64 issues once in 64 cycles per sub-partition, so everything else is
//           on the FP32 pipe: displacement H + L + T, exactly (kick_ff.cu), the residual
//           e = 1 - |d y|^2 to 2^-56 from digits, m_j r^-3 = m_j y^3 (1 + 1.5 e +
//           1.875 e^2) as a double -- m_j y^3 as a float plus a whole number of
//           units of the last place of that double.  The FMAs take it times the
//           leading float H of each component (exact as a double); m_j r^-3 (L + T),
//           2^-24 of the term, is summed in two floats.  ~190 FP32 operations per
//           ordered pair, about as long (270 cycles per warp) as the three FMAs (192),
//           against 17 FP64 instructions (1,088) of CUDA's double rsqrt form and
//           10.5 (672) of the symmetric one.
//           Pairs that need more (changeover band, close pairs, r^-3 next to a power
//           of two, bodies whose coordinates three floats do not hold) go to a buffer and
//           are taken 32 at a time in FP64.  Where many coordinates are not held (kFfExact)
//           the displacement is an FP64 subtraction, which the FMAs then take whole: 6
//           FP64 instructions.
// Measured (whole kick, us; before: kick_kernel, or FP64 symmetric from 16,384 on):
//   FP64   N = 1,000: 39 (189), 2,048: 67 (193), 20,011: 2,867 (7,915); error against
//          64 bits 1.6e-16 of the norm at 20,011 (2.1e-16)
//   mixed  N = 1,000: 27 (101), 3,001: 59 (136), 4,096: 88 (246)
// Bound: FP64 pipe 75 % and FP32 pipe 72 % busy at N = 8,192 (both, in turns, by the
// few warps that 96 registers leave); below N ~ 2,000 the latency of one block.
#include <algorithm>
#include <cmath>

#include "ff_pair.cuh"

namespace genga {
namespace {

constexpr int kTlRows = kSymT;                 // rows per block, one per thread
constexpr int kTlFlush = 16;                   // steps (of two bodies j) between the sums' hand-over to FP64
// FP64, by measurement at N = 20,011 (ms): 2 steps unrolled and 5 blocks per SM by
// registers 3.02; 1 and 5: 3.14, 4 and 5: 3.05, 2 and 4: 3.31, 1 and 6: 3.34.
constexpr int kTlUnroll64 = 2, kTlBlocks64 = 5;
constexpr int kTlNear = 128;                   // FP64: buffered near pairs per warp

struct TlRow {                                 // a thread's row, in both halves: negated coordinates
    f2 h[3], m[3], l[3];
    float thr, tn;                             // bounds of r^2: changeover, near pairs
    int i;
};

template <bool PC>
__device__ __forceinline__ void tl_load_row(const SymArgs &A, int a, int r, float close2, TlRow &I) {
    const float4 *B = A.body + (size_t)a * kFfTile + (r >> 6) * 32 + (r & 31);
    const bool up = r & 32;
    const float4 q0 = B[0], q1 = B[kFfRow], q2 = B[2 * kFfRow], q3 = B[3 * kFfRow], q4 = B[4 * kFfRow],
                 q5 = B[5 * kFfRow], q6 = B[6 * kFfRow];
    I.i = a * kSymT + r;
    I.h[0] = f2_dup(-(up ? q0.y : q0.x)); I.h[1] = f2_dup(-(up ? q0.w : q0.z)); I.h[2] = f2_dup(-(up ? q1.y : q1.x));
    I.m[0] = f2_dup(-(up ? q2.y : q2.x)); I.m[1] = f2_dup(-(up ? q2.w : q2.z)); I.m[2] = f2_dup(-(up ? q3.y : q3.x));
    I.l[0] = f2_dup(-(up ? q4.y : q4.x)); I.l[1] = f2_dup(-(up ? q4.w : q4.z)); I.l[2] = f2_dup(-(up ? q5.y : q5.x));
    I.thr = fmaxf(up ? q5.w : q5.z, close2);
    I.tn = fmaxf(PC ? (up ? q6.w : q6.z) : I.thr, close2);
}

// The steps a block takes (A.P of the 32 per group: whole groups, or 16 or 8 steps of
// one), and the staging of a group: 7 rows of 32 float4.
struct TlRange { int g0, g1, k0, k1; };
__device__ __forceinline__ TlRange tl_range(const SymArgs &A) {
    TlRange r;
    const int c = blockIdx.y * A.P;
    r.g0 = c >> 5;
    r.k0 = c & 31;
    r.k1 = min(32, r.k0 + A.P);
    r.g1 = min(2 * A.nT, (c + A.P + 31) >> 5);
    if ((int)blockIdx.x * kSymT >= A.nm) r.g1 = min(r.g1, (A.nm + 63) / 64);   // test-particle rows
    return r;
}
__device__ __forceinline__ void tl_stage(const SymArgs &A, int g, float4 *grp) {
    const float4 *src = A.body + (size_t)(g >> 1) * kFfTile + (g & 1) * 32;
    for (int k = threadIdx.x; k < 7 * 32; k += kTlRows) grp[k] = src[(k >> 5) * kFfRow + (k & 31)];
}

// The warp's buffered pairs (row lane, body j) -- FP64: near ones; mixed: those that the
// packed coordinates do not give --, 32 at a time: every lane
// forms one pair's term m_j K r^-3 d in FP64 from the positions, then adds the
// terms of its own row in buffer order.
struct TlNear {
    uint2 q[kTlNear];
    double t[3][32];
};
__device__ __forceinline__ void tl_near_flush(const SymArgs &A, TlNear &B, int &cnt, int i0, double *sum, int lane) {
    for (int t0 = 0; t0 < cnt; t0 += 32) {
        __syncwarp();
        const int t = t0 + lane, m = min(32, cnt - t0);
        double tx = 0.0, ty = 0.0, tz = 0.0;
        if (lane < m) {
            const int i = i0 + (int)B.q[t].x, j = (int)B.q[t].y;
            const double dx = A.x[j] - A.x[i], dy = A.y[j] - A.y[i], dz = A.z[j] - A.z[i];
            const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
            const double y = rsqrt(r2);
            const double K = r2 < 1e300 ? changeover_fast(r2 * y, inv_rc(fmax(A.rc[i], A.rc[j]))) : 1.0;
            const double c = A.m[j] * (K * (y * y * y));
            tx = c * dx; ty = c * dy; tz = c * dz;
        }
        const unsigned row = B.q[t0].x;
        if (__all_sync(0xffffffffu, lane >= m || B.q[t0 + lane].x == row)) {
            // one row's (a body that is not held): a butterfly, 15 FP64 instructions instead of 96
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                tx += __shfl_xor_sync(0xffffffffu, tx, o);
                ty += __shfl_xor_sync(0xffffffffu, ty, o);
                tz += __shfl_xor_sync(0xffffffffu, tz, o);
            }
            if (lane == (int)row) { sum[0] += tx; sum[kTlRows] += ty; sum[2 * kTlRows] += tz; }
            continue;
        }
        B.t[0][lane] = tx; B.t[1][lane] = ty; B.t[2][lane] = tz;
        __syncwarp();
        unsigned mine = 0u;
        for (int e = 0; e < m; e++) mine |= (B.q[t0 + e].x == (unsigned)lane ? 1u : 0u) << e;
        while (mine) {
            const int e = __ffs(mine) - 1;
            mine &= mine - 1;
            sum[0] += B.t[0][e]; sum[kTlRows] += B.t[1][e]; sum[2 * kTlRows] += B.t[2][e];
        }
    }
    __syncwarp();
    cnt = 0;
}

// Mixed: the steps [k0, k1) of row I against the 64 bodies of group g; near: sums of the
// buffered pairs in the caller's units.
template <bool PC, int MODE>
__device__ __forceinline__ void tl_group(const SymArgs &A, const float4 *grp, int g, int k0, int k1, const TlRow &I, float close2,
                                         double mm, double (&acc)[3], double *near, TlNear &nb, int &npend, uint2 *pcbuf,
                                         int &pend, int lane) {
    constexpr bool EXACT = MODE == kFfExact, GEN = MODE == kFfGeneral || EXACT;
    const f2 away = f2_dup(kFfMasked2);
    const int es = EXACT ? A.ff_header[2] : 0;
#pragma unroll 1
    for (int tb = k0; tb < k1; tb += kTlFlush) {
        f2 sh[3], sl[3];
#pragma unroll
        for (int c = 0; c < 3; c++) sh[c] = sl[c] = 0ull;
#pragma unroll (EXACT ? 1 : 2)
        for (int k = tb; k < min(tb + kTlFlush, k1); k++) {
            const float4 q0 = grp[k], q1 = grp[32 + k], q2 = grp[64 + k], q3 = grp[96 + k], q4 = grp[128 + k],
                         q5 = grp[160 + k];
            const float2 tj = PC ? *reinterpret_cast<const float2 *>(&grp[192 + k].z) : make_float2(q5.z, q5.w);
            const int j = g * 64 + k;
            f2 H[3], L[3], s2, tail, w, wl;
            bool wx = true, wy = true;
            if (GEN) {
                const bool ti = I.i >= A.nm;
                wx = j != I.i && !(ti && j >= A.nm);
                wy = j + 32 != I.i && !(ti && j + 32 >= A.nm);
            }
            if (EXACT) {
                ff_disp_f64(A, min(I.i, A.n - 1), min(j, A.n - 1), min(j + 32, A.n - 1), es, H, L);
                wx = wx && I.i < A.n && j < A.n;
                wy = wy && I.i < A.n && j + 32 < A.n;
            } else {
                ff_disp(f2_lo(q0), f2_lo(q2), f2_lo(q4), I.h[0], I.m[0], I.l[0], H[0], L[0]);
                ff_disp(f2_hi(q0), f2_hi(q2), f2_hi(q4), I.h[1], I.m[1], I.l[1], H[1], L[1]);
                ff_disp(f2_lo(q1), f2_lo(q3), f2_lo(q5), I.h[2], I.m[2], I.l[2], H[2], L[2]);
            }
            ff_r2(H, L, s2, tail);
            if (GEN) {                             // (NaN times zero would be NaN)
                s2 = f2_select(wx, wy, s2, away);
                tail = f2_select(wx, wy, tail, 0ull);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    H[c] = f2_select(wx, wy, H[c], 0ull);
                    L[c] = f2_select(wx, wy, L[c], 0ull);
                }
            }
            ff_inv_r3(s2, tail, w, wl);
            const float2 S = f2_get(s2);
            const bool fx = EXACT && S.x > kFfExactFar2, fy = EXACT && S.y > kFfExactFar2;
            const bool nx = fx || !(S.x >= fmaxf(I.tn, tj.x)), ny = fy || !(S.y >= fmaxf(I.tn, tj.y));
            if (__any_sync(0xffffffffu, nx || ny)) {
                if (PC) {
                    sym_pc_push(pcbuf, pend, lane, nx && wx && j > I.i, I.i, j);
                    sym_pc_push(pcbuf, pend, lane, ny && wy && j + 32 > I.i, I.i, j + 32);
                    if (pend > kSymPcFlush) sym_pc_flush(A, pcbuf, pend, lane);
                }
                // pairs that the packed coordinates do not give (a body that is not held, or
                // closer than they tell): to the FP64 buffer, no term here
                const bool ox = fx || !(S.x >= close2), oy = fy || !(S.y >= close2);
                if (__any_sync(0xffffffffu, ox || oy)) {
                    const bool vi = I.i < A.n;                   // not a padding body
                    sym_pc_push(nb.q, npend, lane, ox && wx && vi && j < A.n, lane, j);
                    sym_pc_push(nb.q, npend, lane, oy && wy && vi && j + 32 < A.n, lane, j + 32);
                    if (npend > kTlNear - 64) tl_near_flush(A, nb, npend, I.i - lane, near, lane);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        H[c] = f2_select(ox, oy, 0ull, H[c]);
                        L[c] = f2_select(ox, oy, 0ull, L[c]);
                    }
                    w = f2_select(ox, oy, 0ull, w);
                    wl = f2_select(ox, oy, 0ull, wl);
                }
                // changeover band: K in float-float, 1/rc_ij = min(1/rc_i, 1/rc_j) (as float
                // pairs: rounding is monotone), r^-3 scaled by K
                const bool bx = !ox && S.x < fmaxf(I.thr, q5.z), by = !oy && S.y < fmaxf(I.thr, q5.w);
                if (bx || by) {
                    const float2 ci = A.ircf[I.i], Tl = f2_get(tail);
                    float2 W = f2_get(w), WL = f2_get(wl);
#pragma unroll 1
                    for (int h = 0; h < 2; h++) {
                        if (!(h ? by : bx)) continue;
                        const float2 cj = A.ircf[j + 32 * h];
                        const bool ti = ci.x < cj.x || (ci.x == cj.x && ci.y <= cj.y);
                        float wh = h ? W.y : W.x, wlo = h ? WL.y : WL.x, Kh, Kl;
                        ff_changeover(h ? S.y : S.x, h ? Tl.y : Tl.x, ti ? ci.x : cj.x, ti ? ci.y : cj.y, Kh, Kl);
                        ff_mul(wh, wlo, Kh, Kl);
                        if (Kh == 0.0f) wh = wlo = 0.0f;         // also where r^-3 overflows
                        if (h) { W.y = wh; WL.y = wlo; }
                        else { W.x = wh; WL.x = wlo; }
                    }
                    w = f2_make(W.x, W.y);
                    wl = f2_make(WL.x, WL.y);
                }
            }
            if (GEN) {
                w = f2_select(wx, wy, w, 0ull);
                wl = f2_select(wx, wy, wl, 0ull);
            }
            f2 ch = w, cl = wl, th[3], te[3];
            if (MODE != kFfUniform) ff_coeff(f2_hi(q1), f2_hi(q3), w, wl, ch, cl);
            ff_term(ch, cl, H, L, th, te);
#pragma unroll
            for (int c = 0; c < 3; c++) f2_acc(sh[c], sl[c], th[c], te[c]);
            if (k & 1) {                       // the low parts back below the last place of the high ones
#pragma unroll
                for (int c = 0; c < 3; c++) f2_fast_two_sum(sh[c], sl[c], sh[c], sl[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 a = f2_get(sh[c]), b = f2_get(sl[c]);
            float s, x;
            ff_two_sum(a.x, a.y, s, x);
            const double v = ff_sum_f64(s) + f64_of_f32_any(x + (b.x + b.y));
            acc[c] = MODE == kFfUniform ? fma(mm, v, acc[c]) : acc[c] + v;
        }
    }
}

template <bool PC>
__global__ void __launch_bounds__(kTlRows, 4)
kick_tile_ff_kernel(SymArgs A) {
    __shared__ float4 grp[7 * 32];
    __shared__ TlNear nb[4];
    __shared__ double nsum[3][kTlRows];
    __shared__ uint2 pcb[PC ? 4 : 1][PC ? kSymPcBuf : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, a = blockIdx.x;
    const TlRange R = tl_range(A);
    const bool exact = ff_exact_pairs(A.ff_header, A.n);
    const float close2 = exact ? kFfExactClose2 : kFfClose2;
    int pend = 0, npend = 0;
    TlRow I;
    tl_load_row<PC>(A, a, threadIdx.x, close2, I);
    double acc[3] = {0.0, 0.0, 0.0}, *near = &nsum[0][threadIdx.x];
#pragma unroll
    for (int c = 0; c < 3; c++) near[c * kTlRows] = 0.0;
    for (int g = R.g0; g < R.g1; g++) {
        __syncthreads();
        tl_stage(A, g, grp);
        __syncthreads();
        const double mm = A.tmass[g >> 1];
        const bool gen = (g >> 1) == a || ((a + 1) * kSymT > A.nm && (g + 1) * 64 > A.nm);
        if (exact) tl_group<PC, kFfExact>(A, grp, g, R.k0, R.k1, I, close2, 0.0, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        else if (gen) tl_group<PC, kFfGeneral>(A, grp, g, R.k0, R.k1, I, close2, 0.0, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        else if (mm > 0.0) tl_group<PC, kFfUniform>(A, grp, g, R.k0, R.k1, I, close2, mm, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        else tl_group<PC, kFfPlain>(A, grp, g, R.k0, R.k1, I, close2, 0.0, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
    }
    tl_near_flush(A, nb[w], npend, I.i - lane, near, lane);
    if (PC) sym_pc_flush(A, pcb[w], pend, lane);
    if (I.i < A.n) {
        const double back = scalbn(1.0, 2 * A.ff_header[2] - A.ff_header[1]);     // to the packed units
        double *p = A.part + (size_t)blockIdx.y * 3 * A.n + I.i;
#pragma unroll
        for (int c = 0; c < 3; c++) p[(size_t)c * A.n] = near[c * kTlRows] != 0.0 ? fma(back, near[c * kTlRows], acc[c]) : acc[c];
    }
}

// ---------------------------------------------------------------- FP64

// FP64: the steps [k0, k1) of row I against the 64 bodies of group g.  acc: sums of (m_j) r^-3 d
// in the packed units, near: those of the buffered pairs in the caller's units.
// kFfExact: the displacement from the positions, xyz those of the group in the packed units.
template <bool PC, int MODE>
__device__ __forceinline__ void tl_group64(const SymArgs &A, const float4 *grp, const double (*xyz)[64], int g, int k0, int k1, const TlRow &I,
                                           double (&acc)[3], double *near, TlNear &nb, int &npend,
                                           uint2 *pcbuf, int &pend, int lane) {
    constexpr bool EXACT = MODE == kFfExact, GEN = MODE == kFfGeneral || EXACT;
    double xi[3];
    if (EXACT) {
        const double xs = scalbn(1.0, -A.ff_header[2]);
        const int i = min(I.i, A.n - 1);
        xi[0] = A.x[i] * xs; xi[1] = A.y[i] * xs; xi[2] = A.z[i] * xs;
    }
    const f2 c15 = f2_dup(1.5f), c1875 = f2_dup(1.875f);
    // r^-3 (L + T): 2^-24 of the terms, so that two floats per sum do for a group
    f2 sh[3], sl[3];
#pragma unroll
    for (int c = 0; c < 3; c++) sh[c] = sl[c] = 0ull;
#pragma unroll (EXACT ? 1 : kTlUnroll64)
    for (int k = k0; k < k1; k++) {
        const float4 q0 = grp[k], q1 = grp[32 + k], q2 = grp[64 + k], q3 = grp[96 + k], q4 = grp[128 + k],
                     q5 = grp[160 + k];
        const float2 tj = PC ? *reinterpret_cast<const float2 *>(&grp[192 + k].z) : make_float2(q5.z, q5.w);
        const int j = g * 64 + k;
        bool wx = true, wy = true;
        if (GEN) {
            const bool ti = I.i >= A.nm;
            wx = j != I.i && I.i < A.n && j < A.n && !(ti && j >= A.nm);
            wy = j + 32 != I.i && I.i < A.n && j + 32 < A.n && !(ti && j + 32 >= A.nm);
        }
        f2 H[3], L[3], T[3];
        double ex[3], ey[3];                   // kFfExact: the two displacements
        if (EXACT) {
#pragma unroll
            for (int c = 0; c < 3; c++) {
                float hx, lx, tx, hy, ly, ty;
                ex[c] = xyz[c][k] - xi[c];
                ey[c] = xyz[c][k + 32] - xi[c];
                f64_split3(ex[c], 0, hx, lx, tx);
                f64_split3(ey[c], 0, hy, ly, ty);
                H[c] = f2_make(hx, hy); L[c] = f2_make(lx, ly); T[c] = f2_make(tx, ty);
            }
        } else {
            ff_disp3(f2_lo(q0), f2_lo(q2), f2_lo(q4), I.h[0], I.m[0], I.l[0], H[0], L[0], T[0]);
            ff_disp3(f2_hi(q0), f2_hi(q2), f2_hi(q4), I.h[1], I.m[1], I.l[1], H[1], L[1], T[1]);
            ff_disp3(f2_lo(q1), f2_lo(q3), f2_lo(q5), I.h[2], I.m[2], I.l[2], H[2], L[2], T[2]);
        }
        const f2 s = f2_fma(H[2], H[2], f2_fma(H[1], H[1], f2_mul(H[0], H[0])));
        const f2 y = f2_rsqrt(s);
        f2 eh, el;
        ff_residual(H, L, T, y, eh, el);
        // y^3 = wh + we + f + fe exactly; r^-3 = y^3 (1 + 1.5 e + 1.875 e^2) = wh + 1.5 x0 + (we + f) + small
        const f2 p = f2_mul(y, y), pe = f2_fma(y, y, f2_neg(p));
        const f2 wh = f2_mul(p, y), we = f2_fma(p, y, f2_neg(wh));
        const f2 f = f2_mul(pe, y), fe = f2_fma(pe, y, f2_neg(f));
        const f2 x0 = f2_mul(wh, eh), x0e = f2_fma(wh, eh, f2_neg(x0)), wf = f2_add(we, f);
        const f2 small = f2_fma(wh, f2_fma(f2_mul(c1875, eh), eh, f2_mul(c15, el)),
                                f2_fma(c15, x0e, f2_fma(f2_mul(c15, wf), eh, fe)));
        const f2 v = f2_fma(c15, x0, wf);  // r^-3 - wh as a float
        // base + a whole number of units: r^-3, or m_j r^-3 with m_j = mh + ml + mt, as a double
        f2 base = wh, sc, tu, lo;
        if (MODE == kFfUniform) {
            const float2 B = f2_get(base);
            sc = f2_make(ff_ulp_scale(B.x), ff_ulp_scale(B.y));
            ff_units(x0, f2_mul(c15, sc), tu, lo);
            ff_units_add(we, sc, tu, lo);
            ff_units_add(f, sc, tu, lo);
            ff_units_add(small, sc, tu, lo);
        } else {
            const f2 mh = f2_hi(q1), ml = f2_hi(q3), mt = *reinterpret_cast<const f2 *>(&grp[192 + k]);
            base = f2_mul(wh, mh);
            const float2 B = f2_get(base);
            sc = f2_make(ff_ulp_scale(B.x), ff_ulp_scale(B.y));
            const f2 ms = f2_mul(mh, sc), ls = f2_mul(ml, sc), x15 = f2_mul(c15, x0);
            ff_units(x15, ms, tu, lo);
            ff_units_add(f2_fma(wh, mh, f2_neg(base)), sc, tu, lo);
            ff_units_add(we, ms, tu, lo);
            ff_units_add(f, ms, tu, lo);
            ff_units_add(wh, ls, tu, lo);
            ff_units_add(f2_add(small, f2_fma(c15, x0, f2_neg(x15))), ms, tu, lo);
            lo = f2_fma(v, ls, f2_fma(wh, f2_mul(mt, sc), lo));
        }
        const float2 B = f2_get(base), TU = f2_get(tu), LO = f2_get(ff_units_end(lo));
        // times 2^896, to go with the components' 2^-896
        constexpr int UP = EXACT ? 0 : 896;
        double dx = ff_add_units<UP>(B.x, TU.x, LO.x), dy = ff_add_units<UP>(B.y, TU.y, LO.y);
        // near pairs; PC: the bounds tn include the changeover's
        const float2 S = f2_get(s);
        const bool px = !(S.x >= fmaxf(I.tn, tj.x)), py = !(S.y >= fmaxf(I.tn, tj.y));
        // next to a power of two the bits change scale: 1.5 e, |e| < 5.6e-7, and the products'
        // low parts are at most 17 last places (2^-24 of the base, below the power)
        const bool ux = ff_near_binade<24>(B.x) || !(S.x < 1e36f && B.x > 6e-23f);
        const bool uy = ff_near_binade<24>(B.y) || !(S.y < 1e36f && B.y > 6e-23f);
        f2 ch = wh, cl = v;
        if (__any_sync(0xffffffffu, px || py || ux || uy || !wx || !wy)) {
            if (PC) {
                sym_pc_push(pcbuf, pend, lane, px && wx && j > I.i, I.i, j);
                sym_pc_push(pcbuf, pend, lane, py && wy && j + 32 > I.i, I.i, j + 32);
                if (pend > kSymPcFlush) sym_pc_flush(A, pcbuf, pend, lane);
            }
            const bool bx = ux || !(S.x >= fmaxf(I.thr, q5.z)), by = uy || !(S.y >= fmaxf(I.thr, q5.w));
            // (a massless j's ux, uy hold: nothing to add, unless NaN or infinite)
            sym_pc_push(nb.q, npend, lane, bx && wx && (B.x != 0.0f || !(S.x < 1e36f)), lane, j);
            sym_pc_push(nb.q, npend, lane, by && wy && (B.y != 0.0f || !(S.y < 1e36f)), lane, j + 32);
            if (npend > kTlNear - 64) tl_near_flush(A, nb, npend, I.i - lane, near, lane);
            const bool ox = bx || !wx, oy = by || !wy;            // no term here
            if (ox) dx = 0.0;
            if (oy) dy = 0.0;
            ch = f2_select(ox, oy, 0ull, ch);
            cl = f2_select(ox, oy, 0ull, cl);
#pragma unroll
            for (int c = 0; c < 3; c++) H[c] = f2_select(ox, oy, 0ull, H[c]);
#pragma unroll
            for (int c = 0; c < 3; c++) L[c] = f2_select(ox, oy, 0ull, L[c]);
#pragma unroll
            for (int c = 0; c < 3; c++) T[c] = f2_select(ox, oy, 0ull, T[c]);
            if (EXACT)
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    if (ox) ex[c] = 0.0;
                    if (oy) ey[c] = 0.0;
                }
        }
        if (EXACT) {
#pragma unroll
            for (int c = 0; c < 3; c++) acc[c] = fma(dy, ey[c], fma(dx, ex[c], acc[c]));
            continue;
        }
        if (MODE != kFfUniform) {
            const f2 h0 = ch, l0 = cl;
            ff_coeff(f2_hi(q1), f2_hi(q3), h0, l0, ch, cl);
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 h = f2_get(H[c]);
            acc[c] = fma(dx, ff_bits_down896(h.x), acc[c]);
            acc[c] = fma(dy, ff_bits_down896(h.y), acc[c]);
            const f2 th = f2_mul(ch, L[c]);
            const f2 te = f2_fma(ch, T[c], f2_fma(cl, L[c], f2_fma(ch, L[c], f2_neg(th))));
            f2_acc(sh[c], sl[c], th, te);
        }
    }
    if constexpr (!EXACT) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 a = f2_get(sh[c]), b = f2_get(sl[c]);
            float s, x;
            ff_two_sum(a.x, a.y, s, x);
            acc[c] += f64_of_f32_any(s) + f64_of_f32_any(x + (b.x + b.y));
        }
    }
}

template <bool PC>
__global__ void __launch_bounds__(kTlRows, kTlBlocks64)
kick_tile_f64_kernel(SymArgs A) {
    __shared__ float4 grp[7 * 32];
    __shared__ double xyz[3][64];              // kFfExact: the group's positions
    __shared__ TlNear nb[4];
    __shared__ uint2 pcb[PC ? 4 : 1][PC ? kSymPcBuf : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, a = blockIdx.x;
    const TlRange R = tl_range(A);
    const bool exact = ff_exact_pairs(A.ff_header, A.n);
    const double back = scalbn(1.0, 2 * A.ff_header[2] - A.ff_header[1]);     // the near pairs' sums in the packed units
    const bool pads = A.n % kSymT != 0;
    int pend = 0, npend = 0;
    TlRow I;
    tl_load_row<PC>(A, a, threadIdx.x, exact ? kFfExactClose2 : kFfClose2, I);
    // sums kept out of the registers: of the near pairs; of up to 4 groups; of all
    // before them (TwoSum) with its compensation
    __shared__ double sums[12][kTlRows];
    double *near = &sums[0][threadIdx.x], *T = near + 3 * kTlRows, *S = near + 6 * kTlRows, *C = near + 9 * kTlRows;
#pragma unroll
    for (int k = 0; k < 12; k++) near[k * kTlRows] = 0.0;
    for (int g = R.g0; g < R.g1; g++) {
        __syncthreads();
        tl_stage(A, g, grp);
        if (exact && threadIdx.x < 64) {
            const double xs = scalbn(1.0, -A.ff_header[2]);
            const int j = min(g * 64 + (int)threadIdx.x, A.n - 1);
            xyz[0][threadIdx.x] = A.x[j] * xs; xyz[1][threadIdx.x] = A.y[j] * xs; xyz[2][threadIdx.x] = A.z[j] * xs;
        }
        __syncthreads();
        const double mm = A.tmass[g >> 1];
        const bool gen = (g >> 1) == a || ((a + 1) * kSymT > A.nm && (g + 1) * 64 > A.nm) ||
                         (pads && (a == A.nT - 1 || (g >> 1) == A.nT - 1));
        double acc[3] = {0.0, 0.0, 0.0};
        if (exact) tl_group64<PC, kFfExact>(A, grp, xyz, g, R.k0, R.k1, I, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        else if (gen) tl_group64<PC, kFfGeneral>(A, grp, xyz, g, R.k0, R.k1, I, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        else if (mm > 0.0)
            tl_group64<PC, kFfUniform>(A, grp, xyz, g, R.k0, R.k1, I, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        else tl_group64<PC, kFfPlain>(A, grp, xyz, g, R.k0, R.k1, I, acc, near, nb[w], npend, pcb[PC ? w : 0], pend, lane);
        const double f = !exact && !gen && mm > 0.0 ? mm : 1.0;
        const bool fold = ((g - R.g0) & 3) == 3 && g + 1 < R.g1;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            double t = fma(f, acc[c], T[c * kTlRows]);
            if (fold) {
                double e;
                if (near[c * kTlRows] != 0.0) {                  // (a body whose pairs are all taken in FP64)
                    t = fma(back, near[c * kTlRows], t);
                    near[c * kTlRows] = 0.0;
                }
                two_sum_ordered(S[c * kTlRows], t, t, e);
                S[c * kTlRows] = t;
                C[c * kTlRows] += e;
                t = 0.0;
            }
            T[c * kTlRows] = t;
        }
    }
    tl_near_flush(A, nb[w], npend, I.i - lane, near, lane);
    if (PC) sym_pc_flush(A, pcb[w], pend, lane);
    if (I.i < A.n) {
        double *p = A.part + (size_t)blockIdx.y * 3 * A.n + I.i;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            double t = T[c * kTlRows];
            if (near[c * kTlRows] != 0.0) t = fma(back, near[c * kTlRows], t);
            if (R.g1 - R.g0 > 4) t = S[c * kTlRows] + (C[c * kTlRows] + t);
            p[(size_t)c * A.n] = t;
        }
    }
}

}  // namespace

// Steps per chunk: SM cycles by waves over the resident blocks times a block's steps
// plus its start, and the fold.
TilePlan tile_plan(int n, int nm, int num_sms, bool mixed, size_t max_part) {
    TilePlan best;
    const int nT = (n + kSymT - 1) / kSymT;
    const long long steps = 64ll * nT;
    const size_t rows = 3;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, mixed ? (const void *)kick_tile_ff_kernel<false> : (const void *)kick_tile_f64_kernel<false>, kTlRows,
            0) != cudaSuccess || per_sm < 1)
        return best;
    // SM cycles per ordered pair of a full SM; per partial and body in the fold; start in steps
    const double c_pair = mixed ? 1.0 : 2.2, c_fin = 0.5, start = mixed ? 2.0 : 6.0;
    const double slots = (double)per_sm * num_sms;
    // of all the rows' groups, those that hold sources
    const double share = ((double)nm * n + (double)(n - nm) * nm) / ((double)n * n);
    for (long long P = 8;; P *= 2) {
        const long long nc = (steps + P - 1) / P;
        if (rows * nc * (size_t)n <= max_part && nc <= 65535) {
            const double w = share * nT * nc / slots, waves = w <= 1.0 ? 1.0 : std::max(std::ceil(w) - 0.5, w);
            const double t = waves * (P + start) * per_sm * 2.0 * kTlRows * c_pair + c_fin * rows * nc * n / num_sms;
            if (best.chunk == 0 || t < best.cycles) {
                best.chunk = (int)P;
                best.nchunk = (int)nc;
                best.cycles = t;
            }
        }
        if (P >= steps) break;
    }
    return best;
}

cudaError_t launch_tile_kick(const SymArgs &S, int chunk, int nchunk, bool mixed, bool precheck, cudaStream_t stream) {
    const dim3 grid(S.nT, nchunk);
    SymArgs A = S;
    A.P = chunk;
    if (mixed) {
        if (precheck) kick_tile_ff_kernel<true><<<grid, kTlRows, 0, stream>>>(A);
        else kick_tile_ff_kernel<false><<<grid, kTlRows, 0, stream>>>(A);
    } else {
        if (precheck) kick_tile_f64_kernel<true><<<grid, kTlRows, 0, stream>>>(A);
        else kick_tile_f64_kernel<false><<<grid, kTlRows, 0, stream>>>(A);
    }
    return cudaGetLastError();
}

}  // namespace genga
