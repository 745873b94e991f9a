// kick_ff.cu -- the mixed symmetric all-pairs kick: every unordered pair once,
// in float expansions on the FP32 pipe.
//
// GB300 executes 128 FP32 operations per clock and SM against ~1.8 FP64 ones, so
// 9 FP64 instructions per pair (3 displacements, 6 accumulations) cost 576
// cycles of a sub-partition per warp of pairs, while the whole pair takes 127
// to 135 FP32 operations.  Nothing here is less exact for it:
//   * a coordinate is the sum of three floats on two fixed grids, h (multiples
//     of 2^-23 S, S a power of two > every |coordinate| on its axis), m (of 2^-47 S)
//     and the remainder l.  Differences of h and of m are exact, so
//     h_j - h_i, m_j - m_i, l_j - l_i sum to the displacement with an error of
//     2^-72 S; a Fast2Sum step gives it as two floats (relative error 2^-48);
//   * r^2 is the exact sum of the squares in two floats (2^-48), r^-3 =
//     y^3 (1 + 1.5 e + 1.875 e^2) from the FP32 seed y and its residual
//     e = 1 - r^2 y^2, in two floats (2^-46);
//   * the force m_i m_j r^-3 d is formed once, as two floats (exact products by
//     FMA), and summed for both bodies in two floats by TwoSum; after 16 terms
//     the sums go to FP64.  A body's sum is divided by its mass in the fold of
//     the partial sums.  Between two tiles of equal masses each (a disk's
//     planetesimals) r^-3 d is summed and the product of the masses applied there.
// What bounds it is the register file: a packed operation reads up to six
// 32-bit registers per lane and the sub-partition delivers two per cycle
// (measured: 3 cycles for an FFMA2 of three different registers, 2 for an FADD2),
// so the choices below save operand reads -- the force formed once for both
// bodies instead of m_j r^-3 d and m_i r^-3 d, TwoSum instead of an ordered
// Fast2Sum (whose selects read as much as the three operations they save).
//
// What the packing kernel finds takes the instance of the pair loop that unusual
// inputs need:
//   * coordinates that three floats do not hold, because they are far smaller than
//     the largest on their axis (2^-25: 3e-8), or larger (S leaves out a few bodies
//     far outside the others).  A few: NaN in their place, which
//     takes these bodies' pairs to FP64 one by one (ff_one); many: kFfExact, every
//     displacement by FP64 subtraction, 3 FP64 instructions per pair;
//   * kFfTwoMass: a massless body, or one 2^-40 of the heaviest: m_j r^-3 d and
//     m_i r^-3 d are formed apart and nothing is divided.
//
// Two pairs per instruction (f32x2): a lane holds one body i and two travelling
// bodies j (l and l + 32 of a 64-body group).
#include "ff_pair.cuh"

namespace genga {
namespace {

constexpr int kFfThreads = 64;                 // two warps: 64 rows each of the 128-body tile

// Chosen by measurement at N = 65,540 (ms per kick): rows per lane 2 (9.5; 1:
// 10.3 -- the j data and shuffles serve two rows), 2 steps unrolled (1: 9.45, 4:
// 9.9).  Blocks per SM that the registers must allow: 5, which gives the compiler the 166
// to 168 it then takes, so that 6 are resident (8.96; bound at 6, 148 registers: 9.17,
// at 7: 9.16, at 4: 9.69).
constexpr int kFfR = 2;
constexpr int kFfUnroll = 2;
constexpr int kFfMinBlocks = 5;
// Terms summed in floats before the sums go to FP64, and steps between two
// renormalisations of the float sums: the rounding of the sums' low parts then
// stays below that of the terms (error of the accelerations of the 16,384-body
// disk 4.0e-15 of their norm; 32 and none: 6.9e-15; 9 FP64 instructions per pair: 5.5e-15).
constexpr int kFfFlush = 16, kFfRenorm = 2;

struct IBody {                                 // a lane's row, in both halves: negated coordinates, mass
    f2 h[3], m[3], l[3];
    f2 mh, ml;
    float thr, tn;                             // bounds of r^2: changeover, near pairs
    int i;
};

// sum += h + l, in the uniform instance times m_i m_j.
template <int MODE>
__device__ __forceinline__ void ff_flush(double &sum, double mm, float h, float l) {
    const double v = ff_sum_f64(h) + f64_of_f32_any(l);
    sum = MODE == kFfUniform ? fma(mm, v, sum) : sum + v;
}

// 32 steps of 32 kFfR of the warp's rows (from row0 of the tile on) against the
// 64 bodies of group jb / 64.  kFfGeneral: pairs masked (diagonal subtiles dsub,
// test particles) and kFfTwoMass; the other instances take every pair.  kFfExact:
// this with displacements by FP64 subtraction.  kFfUniform: two tiles of equal
// masses each, the product mm of the two applied to the sums.
template <bool PC, int MODE>
__device__ __forceinline__ void ff_rows(const SymArgs &A, const float4 *tile, double *js, double *is, int PT, int e0,
                                        int jb, int jglob, const IBody (&I)[kFfR], int flags, float close2, bool dsub, int row0,
                                        double mm, uint2 *pcbuf, int &pend, int lane) {
    constexpr bool EXACT = MODE == kFfExact, GEN = MODE == kFfGeneral || EXACT;
    f2 ih[kFfR][3], il[kFfR][3], jh[3], jl[3];
    const f2 away = f2_dup(kFfMasked2);
    const int es = EXACT ? A.ff_header[2] : 0;
    const float4 *group = tile + (jb >> 1);
#pragma unroll 1
    for (int tb = 0; tb < 32; tb += kFfFlush) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            jh[c] = jl[c] = 0ull;
#pragma unroll
            for (int r = 0; r < kFfR; r++) ih[r][c] = il[r][c] = 0ull;
        }
#pragma unroll (EXACT ? 1 : kFfUnroll)
        for (int t = tb; t < tb + kFfFlush; t++) {
            const int k = (lane + t) & 31;
            const float4 q0 = group[k], q1 = group[kFfRow + k], q2 = group[2 * kFfRow + k], q3 = group[3 * kFfRow + k],
                         q4 = group[4 * kFfRow + k], q5 = group[5 * kFfRow + k];
            // bounds of the near pairs: pre-check or, without it, changeover
            const float2 tj = PC ? *reinterpret_cast<const float2 *>(&group[6 * kFfRow + k].z) : make_float2(q5.z, q5.w);
            f2 H[kFfR][3], L[kFfR][3], w[kFfR], wl[kFfR];
            float2 S[kFfR], Tl[kFfR];
            bool want[kFfR][2], near = false;
#pragma unroll
            for (int r = 0; r < kFfR; r++) {
                want[r][0] = want[r][1] = true;    // this lane's two pairs are wanted
                if (GEN) {
                    const int i = I[r].i;
                    const bool up = i & 32;
                    if (dsub) {                    // every pair of the 64 x 64 diagonal subtile once
                        const bool tri = t >= 1 && (t < 16 || (t == 16 && lane < 16));
                        want[r][0] = !up && tri;
                        want[r][1] = up ? tri : true;
                    }
                    const int j = jglob + k;
                    want[r][0] = want[r][0] && !(i >= A.nm && j >= A.nm);
                    want[r][1] = want[r][1] && !(i >= A.nm && j + 32 >= A.nm);
                }
                if (EXACT) {
                    ff_disp_f64(A, min(I[r].i, A.n - 1), min(jglob + k, A.n - 1), min(jglob + k + 32, A.n - 1), es, H[r], L[r]);
                    want[r][0] = want[r][0] && I[r].i < A.n && jglob + k < A.n;
                    want[r][1] = want[r][1] && I[r].i < A.n && jglob + k + 32 < A.n;
                } else {
                    ff_disp(f2_lo(q0), f2_lo(q2), f2_lo(q4), I[r].h[0], I[r].m[0], I[r].l[0], H[r][0], L[r][0]);
                    ff_disp(f2_hi(q0), f2_hi(q2), f2_hi(q4), I[r].h[1], I[r].m[1], I[r].l[1], H[r][1], L[r][1]);
                    ff_disp(f2_lo(q1), f2_lo(q3), f2_lo(q5), I[r].h[2], I[r].m[2], I[r].l[2], H[r][2], L[r][2]);
                }
                f2 s2, tail;
                ff_r2(H[r], L[r], s2, tail);
                if (GEN) {                         // (NaN times zero would be NaN)
                    s2 = f2_select(want[r][0], want[r][1], s2, away);
                    tail = f2_select(want[r][0], want[r][1], tail, 0ull);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        H[r][c] = f2_select(want[r][0], want[r][1], H[r][c], 0ull);
                        L[r][c] = f2_select(want[r][0], want[r][1], L[r][c], 0ull);
                    }
                }
                S[r] = f2_get(s2);
                Tl[r] = f2_get(tail);
                ff_inv_r3(s2, tail, w[r], wl[r]);
                near = near || !(S[r].x >= fmaxf(I[r].tn, tj.x)) || !(S[r].y >= fmaxf(I[r].tn, tj.y));
                if (EXACT) near = near || S[r].x > kFfExactFar2 || S[r].y > kFfExactFar2;
            }
            if (PC ? __any_sync(0xffffffffu, near) : near) {
#pragma unroll
                for (int r = 0; r < kFfR; r++) {
                    if (PC) {                      // pre-check: the bounds tn include the changeover's
                        sym_pc_push(pcbuf, pend, lane, want[r][0] && !(S[r].x >= fmaxf(I[r].tn, tj.x)), I[r].i, jglob + k);
                        sym_pc_push(pcbuf, pend, lane, want[r][1] && !(S[r].y >= fmaxf(I[r].tn, tj.y)), I[r].i,
                                    jglob + k + 32);
                        if (pend > kSymPcFlush) sym_pc_flush(A, pcbuf, pend, lane);
                    }
                    // changeover band: K in float-float, 1/rc_ij = min(1/rc_i, 1/rc_j) (as float
                    // pairs: rounding is monotone), r^-3 scaled by K; and the pairs for ff_one
                    const bool fx = EXACT && S[r].x > kFfExactFar2, fy = EXACT && S[r].y > kFfExactFar2;
                    const bool bx = fx || !(S[r].x >= fmaxf(I[r].thr, q5.z)), by = fy || !(S[r].y >= fmaxf(I[r].thr, q5.w));
                    if (bx || by) {
                        const float2 ci = A.ircf[I[r].i];
                        float2 W = f2_get(w[r]), WL = f2_get(wl[r]);
#pragma unroll 1
                        for (int h = 0; h < 2; h++) {
                            if (!(h ? by : bx)) continue;
                            const float2 cj = A.ircf[jglob + k + 32 * h];
                            const bool ti = ci.x < cj.x || (ci.x == cj.x && ci.y <= cj.y);
                            const float ih = ti ? ci.x : cj.x, il = ti ? ci.y : cj.y;
                            float wh = h ? W.y : W.x, wlo = h ? WL.y : WL.x;
                            if (!((h ? S[r].y : S[r].x) >= close2) || (h ? fy : fx)) {
                                FfOne o;
                                ff_one(A, I[r].i, jglob + k + 32 * h, ih, il, o);
#pragma unroll
                                for (int c = 0; c < 3; c++) {
                                    const float2 u = f2_get(H[r][c]), v = f2_get(L[r][c]);
                                    H[r][c] = f2_make(h ? u.x : o.H[c], h ? o.H[c] : u.y);
                                    L[r][c] = f2_make(h ? v.x : o.L[c], h ? o.L[c] : v.y);
                                }
                                wh = o.w;
                                wlo = o.wl;
                            } else {
                                float Kh, Kl;
                                ff_changeover(h ? S[r].y : S[r].x, h ? Tl[r].y : Tl[r].x, ih, il, Kh, Kl);
                                ff_mul(wh, wlo, Kh, Kl);
                                if (Kh == 0.0f) wh = wlo = 0.0f;         // also where r^-3 overflows
                            }
                            if (h) { W.y = wh; WL.y = wlo; }
                            else { W.x = wh; WL.x = wlo; }
                        }
                        w[r] = f2_make(W.x, W.y);
                        wl[r] = f2_make(WL.x, WL.y);
                    }
                }
            }
            const f2 mjh = f2_hi(q1), mjl = f2_hi(q3);
#pragma unroll
            for (int r = 0; r < kFfR; r++) {
                f2 ch, cl, th[3], te[3];
                if (GEN) {
                    w[r] = f2_select(want[r][0], want[r][1], w[r], 0ull);
                    wl[r] = f2_select(want[r][0], want[r][1], wl[r], 0ull);
                }
                if (GEN && (flags & kFfTwoMass)) {
                    ff_coeff(mjh, mjl, w[r], wl[r], ch, cl);
                    ff_term(ch, cl, H[r], L[r], th, te);
#pragma unroll
                    for (int c = 0; c < 3; c++) f2_acc(ih[r][c], il[r][c], th[c], te[c]);
                    ff_coeff(I[r].mh, I[r].ml, w[r], wl[r], ch, cl);
                    ff_term(ch, cl, H[r], L[r], th, te);
#pragma unroll
                    for (int c = 0; c < 3; c++) f2_acc_neg(jh[c], jl[c], th[c], te[c]);
                } else {
                    if (MODE == kFfUniform) {
                        ch = w[r];
                        cl = wl[r];
                    } else {
                        const f2 mh = I[r].mh, Mh = f2_mul(mh, mjh);             // m_i m_j
                        const f2 Ml = f2_fma(I[r].ml, mjh, f2_fma(mh, mjl, f2_fma(mh, mjh, f2_neg(Mh))));
                        ff_coeff(Mh, Ml, w[r], wl[r], ch, cl);
                    }
                    ff_term(ch, cl, H[r], L[r], th, te);
#pragma unroll
                    for (int c = 0; c < 3; c++) f2_acc(ih[r][c], il[r][c], th[c], te[c]);
#pragma unroll
                    for (int c = 0; c < 3; c++) f2_acc_neg(jh[c], jl[c], th[c], te[c]);
                }
            }
            // the low parts back below the last place of the high ones
            if (t % kFfRenorm == kFfRenorm - 1) {
#pragma unroll
                for (int c = 0; c < 3; c++) {
#pragma unroll
                    for (int r = 0; r < kFfR; r++) f2_fast_two_sum(ih[r][c], il[r][c], ih[r][c], il[r][c]);
                    f2_fast_two_sum(jh[c], jl[c], jh[c], jl[c]);
                }
            }
            // pass the j sums on: lane L takes over lane L + 1's bodies
#pragma unroll
            for (int c = 0; c < 3; c++) {
                jh[c] = f2_shfl(jh[c], (lane + 1) & 31);
                jl[c] = f2_shfl(jl[c], (lane + 1) & 31);
            }
        }
        // the sums go to FP64; after the hand-overs a lane holds the bodies lane + tb + kFfFlush
        const int e = e0 + ((lane + tb + kFfFlush) & 31);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 h = f2_get(jh[c]), l = f2_get(jl[c]);
            ff_flush<MODE>(js[c * PT + e], mm, h.x, l.x);
            ff_flush<MODE>(js[c * PT + e + 32], mm, h.y, l.y);
#pragma unroll
            for (int r = 0; r < kFfR; r++) {
                const float2 a = f2_get(ih[r][c]), b = f2_get(il[r][c]);
                float s, x;
                ff_two_sum(a.x, a.y, s, x);
                ff_flush<MODE>(is[c * kSymT + row0 + 32 * r + lane], mm, s, x + (b.x + b.y));
            }
        }
    }
}

template <bool PC>
__device__ __forceinline__ void ff_load_row(const SymArgs &A, int a, int r, float close2, IBody &I) {
    const float4 *B = A.body + (size_t)a * kFfTile + (r >> 6) * 32 + (r & 31);
    const bool up = r & 32;
    const float4 q0 = B[0], q1 = B[kFfRow], q2 = B[2 * kFfRow], q3 = B[3 * kFfRow], q4 = B[4 * kFfRow],
                 q5 = B[5 * kFfRow];
    I.i = a * kSymT + r;
    I.h[0] = f2_dup(-(up ? q0.y : q0.x)); I.h[1] = f2_dup(-(up ? q0.w : q0.z)); I.h[2] = f2_dup(-(up ? q1.y : q1.x));
    I.m[0] = f2_dup(-(up ? q2.y : q2.x)); I.m[1] = f2_dup(-(up ? q2.w : q2.z)); I.m[2] = f2_dup(-(up ? q3.y : q3.x));
    I.l[0] = f2_dup(-(up ? q4.y : q4.x)); I.l[1] = f2_dup(-(up ? q4.w : q4.z)); I.l[2] = f2_dup(-(up ? q5.y : q5.x));
    I.mh = f2_dup(up ? q1.w : q1.z);
    I.ml = f2_dup(up ? q3.w : q3.z);
    const float4 q6 = B[6 * kFfRow];
    I.thr = fmaxf(up ? q5.w : q5.z, close2);
    I.tn = fmaxf(PC ? (up ? q6.w : q6.z) : I.thr, close2);
}

// EX: the kernel for bodies whose coordinates are not held (kFfExact); the other returns
// at once.  In one kernel the third instance costs the others 3 % (N = 131,071: 35.7 ms
// against 34.7), the launch that finds nothing to do 2 us.
template <bool PC, bool EX>
__global__ void __launch_bounds__(kFfThreads, kFfMinBlocks)
kick_sym_ff_kernel(SymArgs A)
{
    if (ff_exact_pairs(A.ff_header, A.n) != EX) return;
    extern __shared__ __align__(16) unsigned char ff_sh[];
    float4 *tile = reinterpret_cast<float4 *>(ff_sh);            // the j tile
    double *is = reinterpret_cast<double *>(tile + kFfTile);     // [3][kSymT]: the row tile's sums
    double *js = is + 3 * kSymT;                                 // [3][P * kSymT]: the item's j sums
    __shared__ int s_item;
    __shared__ uint2 pcb[PC ? 2 : 1][PC ? kSymPcBuf : 1];
    int pend = 0;                                                // candidates in this warp's buffer

    const int n = A.n, PT = A.P * kSymT;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int flags = A.ff_header[0];
    // (read: with the bound as a constant in the code the compiler's schedule is 3 % slower)
    const float close2 = EX ? kFfExactClose2 : reinterpret_cast<const float *>(A.ff_header)[4];
    for (;;) {
        __syncthreads();                       // the previous item's shared sums are written out
        if (threadIdx.x == 0) s_item = (int)atomicAdd(A.ctr, 1u);
        __syncthreads();
        const int it = s_item;
        if (it >= A.nItems) break;
        const int2 XY = A.items[it];
        const int a0 = XY.x * A.P, a1 = min(A.nT, a0 + A.P);
        const int b0 = XY.y * A.P, b1 = min(A.nT, b0 + A.P);
        const bool diag = XY.x == XY.y;
        for (int e = threadIdx.x; e < 3 * PT; e += kFfThreads) js[e] = 0.0;
        for (int a = a0; a < a1; a++) {
#pragma unroll
            for (int c = 0; c < 3; c++)        // a lane's own two rows
                is[c * kSymT + w * 64 + lane] = is[c * kSymT + w * 64 + 32 + lane] = 0.0;
            for (int b = diag ? a : b0; b < b1; b++) {
                __syncthreads();               // the tile buffer is free
                for (int k = threadIdx.x; k < kFfTile; k += kFfThreads) tile[k] = A.body[(size_t)b * kFfTile + k];
                __syncthreads();
                const bool same = a == b;
                // pairs to mask: the diagonal tile's, and two test particles'
                const bool gen = flags != 0 || same || ((a + 1) * kSymT > A.nm && (b + 1) * kSymT > A.nm);
                const double mm = A.tmass[a] * A.tmass[b];
                for (int s = 0; s < 2; s++) {
                    const int q = (w + s) & 1;
                    if (!same || q >= w) {
                        const bool dsub = same && q == w;
                        const int jb = q * 64, e0 = (b - b0) * kSymT + jb, jg = b * kSymT + jb;
#pragma unroll 1
                        for (int h = 0; h < 64; h += 32 * kFfR) {
                            IBody I[kFfR];
#pragma unroll
                            for (int r = 0; r < kFfR; r++) ff_load_row<PC>(A, a, w * 64 + h + 32 * r + lane, close2, I[r]);
                            if constexpr (EX)
                                ff_rows<PC, kFfExact>(A, tile, js, is, PT, e0, jb, jg, I, flags, close2, dsub, w * 64 + h,
                                                      0.0, pcb[PC ? w : 0], pend, lane);
                            else if (gen)
                                ff_rows<PC, kFfGeneral>(A, tile, js, is, PT, e0, jb, jg, I, flags, close2, dsub, w * 64 + h,
                                                        0.0, pcb[PC ? w : 0], pend, lane);
                            else if (mm > 0.0)
                                ff_rows<PC, kFfUniform>(A, tile, js, is, PT, e0, jb, jg, I, 0, close2, false, w * 64 + h, mm,
                                                        pcb[PC ? w : 0], pend, lane);
                            else
                                ff_rows<PC, kFfPlain>(A, tile, js, is, PT, e0, jb, jg, I, 0, close2, false, w * 64 + h, 0.0,
                                                      pcb[PC ? w : 0], pend, lane);
                        }
                    }
                    __syncthreads();           // group sums handed to the other warp
                }
            }
            // row a done: its sums over the tiles of Y (slot Y), or, in a
            // diagonal item, with the j sums of tile a, now complete (slot X)
            double *pp = A.part + (size_t)(diag ? XY.x : XY.y) * 3 * n;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int r = w * 64 + 32 * h + lane, i = a * kSymT + r;
                if (i >= n) continue;
#pragma unroll
                for (int c = 0; c < 3; c++)
                    pp[(size_t)c * n + i] =
                        diag ? is[c * kSymT + r] + js[c * PT + (a - b0) * kSymT + r] : is[c * kSymT + r];
            }
        }
        if (!diag) {                           // j sums of the Y tiles: slot X
            double *pp = A.part + (size_t)XY.x * 3 * n;
            const int nj = (b1 - b0) * kSymT;
            for (int e = threadIdx.x; e < nj; e += kFfThreads) {
                const int j = b0 * kSymT + e;
                if (j >= n) continue;
#pragma unroll
                for (int c = 0; c < 3; c++) pp[(size_t)c * n + j] = js[c * PT + e];
            }
        }
    }
    if (PC) sym_pc_flush(A, pcb[w], pend, lane);
}

// The exponent field of a finite double (0: zero or denormal, -1: infinite or NaN).
__device__ __forceinline__ int f64_field(double v) {
    const int f = (__double2hiint(v) >> 20) & 0x7ff;
    return f == 0x7ff ? -1 : f;
}

// Per block: largest exponent field on each axis, of the masses, smallest of the masses.
__global__ void __launch_bounds__(256) ff_bounds_kernel(int n, const double *pos, const double *mass, int4 *bounds, int *header) {
    __shared__ int sh[5][8];
    int v[5] = {0, 0, 0, 0, 0};                    // the last: 0x7ff - field
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += 256 * gridDim.x) {
        const int m = f64_field(mass[i]);
#pragma unroll
        for (int c = 0; c < 3; c++) v[c] = max(v[c], f64_field(pos[(size_t)c * n + i]));
        v[3] = max(v[3], m);
        if (m >= 0) v[4] = max(v[4], 0x7ff - m);
    }
#pragma unroll
    for (int c = 0; c < 5; c++) {
        v[c] = __reduce_max_sync(0xffffffffu, v[c]);
        if ((threadIdx.x & 31) == 0) sh[c][threadIdx.x >> 5] = v[c];
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        int m = 0;
        for (int k = 0; k < 8; k++) m = max(m, sh[threadIdx.x][k]);
        reinterpret_cast<int *>(bounds + 2 * blockIdx.x)[threadIdx.x] = m;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) header[3] = header[5] = 0;
}

// (Scaled) x = h + m + l: h a multiple of 2^-23 S, m of 2^-47 S (S = 2^e), l the rest
// rounded to a float.  mag1, mag2: 1.5 2^52 times the two grids' spacing, whose
// addition rounds a double to a multiple of the spacing.
__device__ __forceinline__ void ff_split(double x, double mag1, double mag2, float &h, float &m, float &l) {
    const double dh = (x + mag1) - mag1, r = x - dh;
    const double dm = (r + mag2) - mag2;
    h = (float)dh;
    m = (float)dm;
    l = (float)(r - dm);
}

// Four blocks per tile, one for each coordinate and one for masses, radii and the
// header: the work is FP64 instructions, ~60 per body, and four SMs do a tile in
// two thirds of the time of one (N = 2,048: 5.1 us against 6.9).
__global__ void __launch_bounds__(kSymT) ff_pack_kernel(FfPack A, int nbounds) {
    __shared__ int sh[5];
    __shared__ double tm;
    {
        // warp c, axis c: the largest field of the blocks, without those of more than
        // A.margin above what an eighth of them reach -- bodies far outside the others
        // (ejected ones) would otherwise set a grid too coarse for all; warp 3: masses
        const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
        int f[(kFfBoundBlocks + 31) / 32], m = 0, small = 0;
#pragma unroll
        for (int k = 0; k < (kFfBoundBlocks + 31) / 32; k++) {
            const int b = 32 * k + lane;
            f[k] = b < nbounds ? reinterpret_cast<const int *>(A.bounds + 2 * b)[c] : 0;
            m = max(m, f[k]);
            if (c == 3 && b < nbounds) small = max(small, A.bounds[2 * b + 1].x);
        }
        m = __reduce_max_sync(0xffffffffu, m);
        small = __reduce_max_sync(0xffffffffu, small);
        if (c < 3 && nbounds >= 8) {
            int q = 0;                         // largest field that more than an eighth reach
            for (int s = 1024; s; s >>= 1) {
                int above = 0;
#pragma unroll
                for (int k = 0; k < (kFfBoundBlocks + 31) / 32; k++) above += f[k] >= q + s;
                if (8 * __reduce_add_sync(0xffffffffu, above) > nbounds) q += s;
            }
            m = 0;
#pragma unroll
            for (int k = 0; k < (kFfBoundBlocks + 31) / 32; k++) m = max(m, f[k] <= q + A.margin ? f[k] : 0);
            m = __reduce_max_sync(0xffffffffu, m);
        }
        if (lane == 0) {
            sh[c] = m;
            if (c == 3) sh[4] = small;
        }
    }
    __syncthreads();
    int v[5];
#pragma unroll
    for (int c = 0; c < 5; c++) v[c] = sh[c];
    // S = 2^ex > every |coordinate| that is held; lengths are scaled by 2^-es, which puts S at 2^kFfScale,
    // masses by 2^-em, so that the floats' range does not depend on the caller's units
    const int ex = min(max(max(v[0], max(v[1], v[2])) - 1022, -200), 400);
    const int es = ex - kFfScale, em = min(max(v[3] - 1023, -200), 400);
    const double xscale = scalbn(1.0, -es);
    const int i = blockIdx.x * kSymT + threadIdx.x;
    // component of row q, first (0) or second (2) half: + 1 for the bodies l + 32
    float *B = reinterpret_cast<float *>(A.body + (size_t)(i >> 7) * kFfTile + ((i >> 6) & 1) * 32 + (i & 31)) +
               ((i >> 5) & 1);
    constexpr int R = 4 * kFfRow;
    if (blockIdx.y < 3) {
        const int c = blockIdx.y, q = c == 2 ? R : 2 * c;       // z: first half of the next row
        // the axis' own S = 2^ec > every |x| on it (2^-60 of the largest, if smaller), in units
        const int ec = min(max(v[c] - 1022, ex - 60), ex);
        float h = (float)pad_pos(i & (kSymT - 1)), m = 0.0f, l = 0.0f;
        bool out = false;
        if (i < A.n) {
            const double x = A.pos[(size_t)c * A.n + i];
            ff_split(x * xscale, scalbn(1.5, 52 - 23 + ec - es), scalbn(1.5, 52 - 47 + ec - es), h, m, l);
            // not held: 2^ec or more, or below 2^(ec - window); a zero is
            const int f = f64_field(x) - 1022;                  // |x| < 2^f
            out = x != 0.0 && (f > ec || f < ec - A.window || !(fabs(x) < __longlong_as_double(0x7ff0000000000000ll)));
            if (out) h = __uint_as_float(0x7fc00000u);
        }
        B[q] = h; B[2 * R + q] = m; B[4 * R + q] = l;
        const int nout = __syncthreads_count(out);
        if (nout && threadIdx.x == 0) atomicAdd(&A.header[3], nout);
        return;
    }
    if (i == 0) {
        A.header[0] = 0x7ff - v[4] <= v[3] - 40 ? kFfTwoMass : 0;
        A.header[1] = em;
        A.header[2] = es;
        reinterpret_cast<float *>(A.header)[4] = kFfClose2;
        if (A.ctr) *A.ctr = 0u;
        if (A.cand_count) *A.cand_count = 0ull;
    }
    int field = 0x7ff;
    if (i < A.n)
        field = max(f64_field(A.pos[i]), max(f64_field(A.pos[(size_t)A.n + i]), f64_field(A.pos[2 * (size_t)A.n + i])));
    const int inner = __syncthreads_count(field - 1022 <= ex - kFfInner);
    if (inner && threadIdx.x == 0) atomicAdd(&A.header[5], inner);
    // the common (scaled) mass of a full tile of equal masses, else 0
    const double ms = i < A.n ? A.m[i] * scalbn(1.0, -em) : 0.0;
    if (threadIdx.x == 0) tm = ms;
    __syncthreads();
    const int differ = __syncthreads_or(ms != tm || !(ms > 0.0));
    if (threadIdx.x == 0) A.tmass[blockIdx.x] = differ ? 0.0 : ms;
    float mh = 0.0f, ml = 0.0f, mt = 0.0f, thr = 0.0f, thp = 0.0f;
    float2 ircf = make_float2(0.0f, 0.0f);
    if (i < A.n) {
        const double rc = A.rc[i], rcs = rc * xscale, pc2 = A.pc2 ? A.pc2[i] * xscale * xscale : 0.0;
        mh = __double2float_rn(ms);
        ml = __double2float_rn(ms - (double)mh);
        mt = __double2float_rn((ms - (double)mh) - (double)ml);
        // upper bounds of rc^2 and pc2: rounded up, then 2^-16 more, so that any float
        // r^2 within 2^-20 of an r^2 below them is below them
        thr = __double2float_ru(rcs * rcs) * 1.0000153f;
        thp = fmaxf(__double2float_ru(pc2) * 1.0000153f, thr);
        ircf = ff_of_irc(inv_rc(rc) * scalbn(1.0, es));
    }
    B[R + 2] = mh;
    B[3 * R + 2] = ml;
    B[5 * R + 2] = thr;
    B[6 * R] = mt;
    B[6 * R + 2] = thp;
    A.ircf[i] = ircf;
}

}  // namespace

size_t sym_ff_smem(int P) {
    return (size_t)kFfTile * sizeof(float4) + (size_t)(P + 1) * kSymT * 3 * sizeof(double);
}

int sym_ff_blocks_per_sm(int P) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kick_sym_ff_kernel<true, false>, kFfThreads, sym_ff_smem(P)) !=
        cudaSuccess)
        return 0;
    return nb;
}

// Layout of the packed-body allocation: the arrays in this order, each a whole
// number of float4 per tile (but the bounds and the header, at the end).
static size_t ff_tile_bytes(size_t nT) {
    return nT * (sizeof(float4) * kFfTile + sizeof(float2) * kSymT + sizeof(float4)) + sizeof(int4) * (2 * kFfBoundBlocks + 2);
}

void ff_place(FfPack &k, void *mem, size_t nT) {
    k.body = (float4 *)mem;
    k.ircf = (float2 *)(k.body + nT * kFfTile);
    k.tmass = (double *)(k.ircf + nT * kSymT);
    k.bounds = (int4 *)(k.tmass + 2 * nT);
    k.header = (int *)(k.bounds + 2 * kFfBoundBlocks);
}

size_t ff_bytes(int n) { return ff_tile_bytes((size_t)((n + kSymT - 1) / kSymT)); }

cudaError_t ff_reserve(genga_system *s) {
    const size_t nT = (size_t)((s->n + kSymT - 1) / kSymT);
    if (nT <= s->ff_tiles) return cudaSuccess;
    if (s->ff) cudaFree(s->ff);
    s->ff = nullptr;
    s->ff_tiles = 0;
    GENGA_CUDA_TRY(cudaMalloc(&s->ff, ff_tile_bytes(nT)));
    s->ff_tiles = nT;
    return cudaSuccess;
}

FfPack ff_pack_args(const genga_system *s) {
    FfPack k;
    k.pos = s->pos; k.m = s->mass; k.rc = s->rcl[0].rc; k.pc2 = s->rcl[0].pc2;
    k.n = (int)s->n;
    k.nT = (int)((s->n + kSymT - 1) / kSymT);
    ff_place(k, s->ff, s->ff_tiles);
    k.window = s->p.precision == GENGA_MIXED ? kFfWindowMixed : kFfWindow64;
    k.margin = s->p.precision == GENGA_MIXED ? kFfMarginMixed : kFfMargin64;
    k.ctr = nullptr;
    k.cand_count = nullptr;
    return k;
}

cudaError_t launch_ff_pack(const FfPack &k, cudaStream_t stream, int64_t *launches) {
    const int nb = std::min(kFfBoundBlocks, (k.n + 255) / 256);
    ff_bounds_kernel<<<nb, 256, 0, stream>>>(k.n, k.pos, k.m, k.bounds, k.header);
    GENGA_CUDA_TRY(cudaGetLastError());
    ff_pack_kernel<<<dim3(k.nT, 4), kSymT, 0, stream>>>(k, nb);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_sym_ff(const SymArgs &S, bool precheck, int blocks, cudaStream_t stream) {
    const size_t smem = sym_ff_smem(S.P);
    if (precheck) kick_sym_ff_kernel<true, false><<<blocks, kFfThreads, smem, stream>>>(S);
    else kick_sym_ff_kernel<false, false><<<blocks, kFfThreads, smem, stream>>>(S);
    if (precheck) kick_sym_ff_kernel<true, true><<<blocks, kFfThreads, smem, stream>>>(S);
    else kick_sym_ff_kernel<false, true><<<blocks, kFfThreads, smem, stream>>>(S);
    return cudaGetLastError();
}

}  // namespace genga
