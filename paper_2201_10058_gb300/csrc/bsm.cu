// bsm.cu -- Bulirsch-Stoer for close-encounter groups of more than
// kBlockGroupMax members, spread over the whole GPU (the role of the paper's
// BS-M, Sec. 6.1), with every such group of the current grouping advanced
// together by one persistent cooperative kernel.
//
// One round is one attempt of every still-running group, at its own step H,
// in phases separated by grid-wide barriers:
//   start      derivative at the attempt's start, error scale, first
//              midpoint sub-step of all 8 extrapolation columns;
//   sub-step   it = 1..16 moves every column whose n_k = 2(k+1) still has
//              sub-steps left, over all (column, member) pairs (ping-pong
//              state buffers, so partner reads never race with writes);
//              for large batches of the forward ODE a pair phase first
//              evaluates each partner pair once per column and writes its two
//              terms to the pair's partner-list entries, which the sub-step
//              then sums per member (the same values, in the same order);
//              A column's last sub-step also forms its row of the extrapolation
//              table and sets the group's bit of the column unless its error is under
//              tolerance; the sub-steps end when every running group has a column
//              that is not (16,384-body step: 22.5 ms with all 16 sub-steps and a
//              phase of their own for the tables, 20.1 so; N = 2,048: 2.11, 1.86);
//   decide     one thread per group: first column k >= 1 under tolerance
//              -> accept (grow H by 1.5 if k < 4), else halve H; attempt
//              and time bookkeeping; done / failed status;
//   accept     members of accepting groups take the accepted column.
// Step control and iteration stay on the device: the host launches once and
// reads the result.  A group fails after bs_max_steps attempts, so at most
// bs_max_steps rounds run; every barrier wait has a time limit (2 s unless
// genga_set_wait_limits sets another) after which the kernel records a
// timeout and returns.  Scheme and acceptance rule
// are those of the in-block kernels (modified midpoint n = 2..16, Neville in
// h^2, error scale |y| + |H dy/dt| + 1e-300, the same force arithmetic).
// Data written by one block and read by another inside the kernel is read
// through L2 (ld.global.cg), never from a possibly stale L1 line.
//
// The ODE is a template policy: the group's forward ODE (6 values per member)
// or the adjoint's augmented backward ODE (13 values per member).
#include <algorithm>
#include <cstring>
#include <vector>

#include "common.cuh"

namespace genga {
namespace {

constexpr int kPMaxThreads = 512;
// Lanes per (column, member) item: 16 while all items then make at most this many
// warps per SM sub-partition, else 8, else 4.  A phase lasts as long as its longest
// partner list (a dense disk's reaches 80), which more lanes shorten; they cost FP64
// work in the butterfly.  Measured (ms per call): 4,096-body gradient (1,415 members) 16
// lanes 71.2, 8: 84, 4: 90; 16,384-body step (12,346 members) 16: 36.5, 8: 28.2, 4: 29.3.
constexpr int kItemWarps = 64;
// Members from which the pair form pays although one pass holds all items (1,415
// members: 67.6 against 71.2 ms; 276 members: 4.45 against 4.13).
constexpr int kPairMembers = 400;

struct GridBarrier {
    unsigned long long count;   // arrivals since the launch; top bit: a wait ran out
    unsigned err;               // the same, for the host: 1, 2 for the first wait
    unsigned running;           // groups still integrating
};

// One unordered pair of batched members (pair-centric mode): members m < p, the
// partner-list entries m -> p and p -> m, their masses.
struct alignas(32) PairRec {
    int m, p, q, q2;
    double mm, mp;
};

// Batch of groups: compact member index m in [0, M) over the groups.
struct BsmArgs {
    int M;                         // members over all batched groups
    int ng;                        // batched groups
    int nlev;                      // levels whose (1 - K) factors apply
    // per member, written before the persistent launch
    const int *mgroup;             // [M] batched group of m
    const int *mq0, *mq1;          // [M] partner range in the level CSR
    const int *pidx;               // [CSR entries] compact index of each partner
    const double *mmass;           // [M] mass
    const double *irc;             // [nlev][M] 1/rc per level
    double G, mu, dt, tol;
    int max_steps;
    // state, component-major over members ([..][D][M])
    double *Y, *F0, *SC;           // attempt start, its derivative, error scale
    double *ZM, *ZA, *ZB;          // [8] per column: previous midpoint state, two current buffers
    double *T, *DIAG;              // [8] latest row of the Neville table, diagonal T_kk of each column
    // per-group step control
    double *gt, *gH;
    double *gh;                    // [ng][8] midpoint sub-step H / n_k of each column this round, 0: done
    int *gstat;                    // 0 running, 1 done, 2 failed
    int *gkconv;                   // accepted column of the last round, -1 none
    long long *gatt, *gacc, *grej;
    unsigned *gfail;               // [ng] bit k: some component's error of column k is not under tolerance
    GridBarrier *bar;
    unsigned long long barrier_ns; // limit of one grid-barrier wait
    unsigned long long first_ns;   // added for the first: blocks start when the in-block kernels leave room
    unsigned barrier_absent;       // test hook: arrivals every barrier waits for in vain (0)
    // collisions (Sec. 7.1-7.2), used by the collision ODE instance
    CollArgs coll;
    const int *mbody;              // [M] body of each member
    const int *gbase;              // [ng + 1] first member of each group
    int *morder;                   // [M] members of each group by ascending body index
    int *malive;                   // [M] alive flags of the members
    double *mmass_rw;              // = mmass, written by mergers
    int *gseq;                     // [ng] mergers of each group so far
    unsigned long long *gdeep;     // [ng] deepest overlap fraction found (bits), zero between uses
    DevCounters *ctr;
    // pair-centric derivative (forward ODE without collisions, large batches):
    // each unordered pair once per column, its two terms written to the two
    // partner-list entries, then summed per member
    int pairs;                     // 1: this mode
    const int *pcount;             // pairs listed
    const PairRec *prec;           // [pairs]
    const double *pirc;            // [nlev][nq] 1/rc of each pair per level
    double2 *rec;                  // [8][entries][2]: (c, dx), (dy, dz) of each entry per column
    size_t nq;                     // entries (the stride of rec per column)
    double *star;                  // [8][M] -mu / r^3 of each member per column
};

__device__ __forceinline__ double ldc(const double *p) { return __ldcg(p); }
__device__ __forceinline__ int ldc(const int *p) { return __ldcg(p); }

__device__ __forceinline__ double step_of(const BsmArgs &A, int g) {
    const double H = ldc(&A.gH[g]);
    const double left = A.dt - ldc(&A.gt[g]);
    return H > left ? left : H;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier (all blocks co-resident: cooperative launch).  One thread per
// block arrives (release) at a counter that only grows and polls it (acquire)
// until the arrivals of `target` barriers' worth are in: one round trip through
// L2 after the last arrival, ~2 us against 4.7 us for a counter that the last
// block resets behind a generation word.  A wait longer than limit_ns sets the
// counter's top bit, which ends every other wait too.  The barrier completes when
// gridDim.x + absent blocks have arrived (absent = 0 in normal use; a test makes
// every wait run out with absent > 0).  Returns false if a wait ran out.
constexpr unsigned long long kBarrierErr = 1ull << 63;
__device__ bool grid_barrier(GridBarrier *b, unsigned long long limit_ns, unsigned long long first_ns, unsigned absent,
                             unsigned long long &target) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool first = target == 0ull;
        if (first) limit_ns += first_ns;
        target += gridDim.x + absent;
        asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(&b->count) : "memory");
        unsigned long long t0 = 0ull, v;
        for (unsigned polls = 1;; polls++) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&b->count) : "memory");
            if (v >= target) break;             // all arrived, or the top bit is set
            if ((polls & 63u) == 0u) {
                const unsigned long long now = global_ns();
                if (t0 == 0ull) t0 = now;
                if (now - t0 >= limit_ns) {
                    atomicOr(&b->count, kBarrierErr);
                    atomicCAS(&b->err, 0u, first ? 2u : 1u);
                    v = kBarrierErr;
                    break;
                }
            }
        }
        ok = (v & kBarrierErr) == 0ull;
    }
    __syncthreads();
    return ok != 0;
}

// W *= 1 - K(r / rc) for 1/rc = irc, from r^2 = d2 and yv = 1/r.  Outside the
// band (decided from FP32 copies with margins of 1e-4) K is 0 or 1 exactly and
// costs no FP64 operation; false: K = 1, W is zero.
__device__ __forceinline__ bool apply_changeover(float rf, double d, double irc, double &W) {
    const int side = changeover_side_f32(rf, __double2float_rz(irc));
    if (side > 0) return false;
    if (side == 0) W *= changeover_rest(d, irc);
    return true;
}
// FP32 r from r^2 (relative error 2^-21).
__device__ __forceinline__ float r_f32(double d2) {
    const float f = f32_of_f64_trunc(d2);
    return f * rsqrtf(f);
}

// Lanes per item in the derivative phases: the partner loop of one (column,
// member) item is split over L adjacent lanes.  Sums of the NV values of an item's
// lanes, to all of them: each exchange hands half of the values over while there
// are several (3 values over 16 lanes: 5 FP64 instructions instead of 12, 7: 8
// instead of 28), then one shuffle per value.
template <int L, int NV>
__device__ __forceinline__ void lane_sums(double (&v)[NV]) {
    static_assert((NV & (NV - 1)) == 0, "");
    const unsigned mk = (L < 32 ? ((1u << L) - 1u) : 0xffffffffu) << ((threadIdx.x & 31u) & ~(unsigned)(L - 1));
    int n = NV;
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool hi = threadIdx.x & o;
#pragma unroll
            for (int i = 0; i < NV / 2; i++)
                if (i < n) {
                    const double send = hi ? v[i] : v[i + n], keep = hi ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(mk, send, o);
                }
        } else {
            v[0] += __shfl_xor_sync(mk, v[0], o);
        }
    }
    constexpr int held = NV > L ? NV / L : 1, apart = L / (NV / held);     // values per lane; lanes between them
    double r[NV];
#pragma unroll
    for (int j = 0; j < NV; j++) r[j] = __shfl_sync(mk, v[j % held], j / held * apart, L);
#pragma unroll
    for (int j = 0; j < NV; j++) v[j] = r[j];
}

// Forward group ODE: y = (x, v); a = -mu x/r^3 + G sum_p m_p W (x_p - x)/r^3,
// W = prod_{levels} (1 - K).  Every lane of the item returns f.  With
// collisions (COLL) the members' masses and alive flags change inside the
// kernel (read through L2); a member merged away feels only the star, and a
// partner merged away has mass 0.
template <bool COLL_>
struct FwdOdeT {
    static constexpr int D = 6;
    static constexpr int NERR = 6;
    static constexpr bool COLL = COLL_;
    template <int L>
    __device__ static void deriv(const BsmArgs &A, const double *Z, int m, int lane, double *f) {
        const size_t ld = (size_t)A.M;
        const double x = ldc(&Z[0 * ld + m]), y = ldc(&Z[1 * ld + m]), z = ldc(&Z[2 * ld + m]);
        double p[4] = {0.0, 0.0, 0.0, 0.0};
        const int q0 = A.mq0[m], q1 = (COLL && !ldc(&A.malive[m])) ? q0 : A.mq1[m];
        // entry q0 - 1 is the star, at the origin: one more entry of the first lane
        // instead of the same term in all of them; its coefficient is the fourth sum
        for (int q = q0 - 1 + lane; q < q1; q += L) {
            const bool star = q < q0;
            const int sp = star ? m : A.pidx[q];
            double sx = ldc(&Z[0 * ld + sp]), sy = ldc(&Z[1 * ld + sp]), sz = ldc(&Z[2 * ld + sp]);
            if (star) sx = sy = sz = 0.0;
            const double dx = sx - x, dy = sy - y, dz = sz - z;
            const double d2 = fma(dz, dz, fma(dy, dy, dx * dx));
            const double yv = rsqrt_newton(d2);
            double W = 1.0;
            if (!star) {
                const float rf = r_f32(d2);
                bool in = true;
                for (int l = 0; l < A.nlev && in; l++)
                    in = apply_changeover(rf, d2 * yv,
                                          min_positive(A.irc[(size_t)l * ld + m], A.irc[(size_t)l * ld + sp]), W);
                if (!in) continue;
            }
            const double c = (star ? -A.mu : COLL ? ldc(&A.mmass[sp]) : A.mmass[sp]) * (W * (yv * yv * yv));
            if (star) { p[3] = c; continue; }
            p[0] = fma(c, dx, p[0]); p[1] = fma(c, dy, p[1]); p[2] = fma(c, dz, p[2]);
        }
        lane_sums<L>(p);
        f[0] = ldc(&Z[3 * ld + m]); f[1] = ldc(&Z[4 * ld + m]); f[2] = ldc(&Z[5 * ld + m]);
        f[3] = fma(p[3], x, A.G * p[0]); f[4] = fma(p[3], y, A.G * p[1]); f[5] = fma(p[3], z, A.G * p[2]);
    }
};
// The forward derivative of member m in column k from the entries' records
// (pair-centric mode): the same terms, summed in the same lane split and order.
template <int L>
__device__ __forceinline__ void fwd_deriv_rec(const BsmArgs &A, const double *Z, int k, int m, int lane,
                                              double *f) {
    const size_t ld = (size_t)A.M;
    const double x = ldc(&Z[0 * ld + m]), y = ldc(&Z[1 * ld + m]), z = ldc(&Z[2 * ld + m]);
    const double2 *R = A.rec + (size_t)k * 2 * A.nq;
    const double sst = __ldcg(&A.star[(size_t)k * A.M + m]);
    double p[4] = {0.0, 0.0, 0.0, 0.0};
    const int q0 = A.mq0[m], q1 = A.mq1[m];
#pragma unroll 4
    for (int q = lane ? q0 - 1 + lane : q0 - 1 + L; q < q1; q += L) {      // the split of FwdOdeT::deriv
        const double2 u = __ldcg(&R[2 * (size_t)q]), w = __ldcg(&R[2 * (size_t)q + 1]);
        p[0] = fma(u.x, u.y, p[0]); p[1] = fma(u.x, w.x, p[1]); p[2] = fma(u.x, w.y, p[2]);
    }
    lane_sums<L>(p);
    f[0] = ldc(&Z[3 * ld + m]); f[1] = ldc(&Z[4 * ld + m]); f[2] = ldc(&Z[5 * ld + m]);
    f[3] = fma(sst, x, A.G * p[0]); f[4] = fma(sst, y, A.G * p[1]); f[5] = fma(sst, z, A.G * p[2]);
}

using FwdOde = FwdOdeT<false>;
using FwdCollOde = FwdOdeT<true>;

// Adjoint augmented ODE in reversed time (level 0): y (6), lambda (6), the
// mass-gradient integral (1); with A = da/dx:
//   dy/dtau = -f(y),  dlx/dtau = A^T lv,  dlv/dtau = lx,
//   dg_a/dtau = G sum_p W lv_p . (x_a - x_p)/r^3   (da_p/dm_a).
struct AdjOde {
    static constexpr int D = 13;
    static constexpr int NERR = 6;
    static constexpr bool COLL = false;
    template <int L>
    __device__ static void deriv(const BsmArgs &A, const double *Z, int m, int lane, double *f) {
        const size_t ld = (size_t)A.M;
        const double x = ldc(&Z[0 * ld + m]), y = ldc(&Z[1 * ld + m]), z = ldc(&Z[2 * ld + m]);
        const double lvx = ldc(&Z[9 * ld + m]), lvy = ldc(&Z[10 * ld + m]), lvz = ldc(&Z[11 * ld + m]);
        const double mb = A.mmass[m];
        double px = 0.0, py = 0.0, pz = 0.0, gx = 0.0, gy = 0.0, gz = 0.0, gm = 0.0;
        const int q1 = A.mq1[m];
        for (int q = A.mq0[m] + lane; q < q1; q += L) {
            const int sp = A.pidx[q];
            const double dx = ldc(&Z[0 * ld + sp]) - x, dy = ldc(&Z[1 * ld + sp]) - y,
                         dz = ldc(&Z[2 * ld + sp]) - z;
            const double d2 = fma(dz, dz, fma(dy, dy, dx * dx));
            const double yv = rsqrt_newton(d2);
            const double d = d2 * yv, id2 = yv * yv, id3 = id2 * yv;
            double K, dK;
            changeover_fast_dr(d, min_positive(A.irc[m], A.irc[sp]), K, dK);
            const double W = 1.0 - K;
            const double Wp = -dK;
            const double mp = A.mmass[sp];
            const double cw = mp * W * id3;
            px = fma(cw, dx, px); py = fma(cw, dy, py); pz = fma(cw, dz, pz);
            const double qx = ldc(&Z[9 * ld + sp]), qy = ldc(&Z[10 * ld + sp]), qz = ldc(&Z[11 * ld + sp]);
            const double e0 = mb * qx - mp * lvx, e1 = mb * qy - mp * lvy, e2 = mb * qz - mp * lvz;
            const double de = dx * e0 + dy * e1 + dz * e2;
            const double aa = W * id3;
            const double bb = de * id2 * (Wp * id2 - 3.0 * W * id3);
            gx += aa * e0 + bb * dx; gy += aa * e1 + bb * dy; gz += aa * e2 + bb * dz;
            gm -= W * (qx * dx + qy * dy + qz * dz) * id3;
        }
        double p[8] = {px, py, pz, gx, gy, gz, gm, 0.0};
        lane_sums<L>(p);
        px = p[0]; py = p[1]; pz = p[2]; gx = p[3]; gy = p[4]; gz = p[5]; gm = p[6];
        const double r2 = fma(z, z, fma(y, y, x * x));
        const double ys = rsqrt_newton(r2);
        const double ir2 = ys * ys, ir3 = ir2 * ys;
        const double xl = x * lvx + y * lvy + z * lvz;
        const double tx = -A.mu * ir3 * (lvx - 3.0 * x * xl * ir2);
        const double ty = -A.mu * ir3 * (lvy - 3.0 * y * xl * ir2);
        const double tz = -A.mu * ir3 * (lvz - 3.0 * z * xl * ir2);
        const double ax = -A.mu * x * ir3 + A.G * px, ay = -A.mu * y * ir3 + A.G * py,
                     az = -A.mu * z * ir3 + A.G * pz;
        f[0] = -ldc(&Z[3 * ld + m]); f[1] = -ldc(&Z[4 * ld + m]); f[2] = -ldc(&Z[5 * ld + m]);
        f[3] = -ax; f[4] = -ay; f[5] = -az;
        f[6] = tx + A.G * gx; f[7] = ty + A.G * gy; f[8] = tz + A.G * gz;
        f[9] = ldc(&Z[6 * ld + m]); f[10] = ldc(&Z[7 * ld + m]); f[11] = ldc(&Z[8 * ld + m]);
        f[12] = A.G * gm;
    }
};

// ---------------------------------------------------------------- phases
// start and sub-step: item = L adjacent lanes; lane l writes the components l, l + L,
// ... (FP64 charges a warp instruction whatever its lanes).
template <int D, int L>
__device__ __forceinline__ double pick(const double *f, int base, int lane) {
    double v = f[base];
#pragma unroll
    for (int l = 1; l < L; l++)
        if (base + l < D && lane == l) v = f[base + l];
    return v;
}

template <class Ode, int L>
__device__ void phase_start(const BsmArgs &A, int m, int lane) {
    const int g = A.mgroup[m];
    if (ldc(&A.gstat[g]) != 0) return;
    constexpr int D = Ode::D;
    const size_t ld = (size_t)A.M, blk = (size_t)D * ld;
    const double H = step_of(A, g);
    double f[D];
    Ode::template deriv<L>(A, A.Y, m, lane, f);
#pragma unroll
    for (int b = 0; b < D; b += L) {
        const int c = b + lane;
        const double fc = pick<D, L>(f, b, lane);
        if (c >= D) break;
        const double y = ldc(&A.Y[c * ld + m]);
        A.F0[c * ld + m] = fc;
        A.SC[c * ld + m] = fabs(y) + fabs(H * fc) + 1e-300;
        for (int k = 0; k < 8; k++) {
            A.ZM[k * blk + c * ld + m] = y;
            A.ZA[k * blk + c * ld + m] = y + ldc(&A.gh[(size_t)g * 8 + k]) * fc;
        }
    }
}

// Column k of component c of member m is complete with the value cur: its row of the
// Neville table (the columns' latest values T[j], read from column k - 1's row), the
// diagonal, and the group's bit k of gfail unless |T_kk - T_k,k-1| <= tol scale (a NaN
// is not convergence).  K at compile time: no divisions and the row in registers.
template <class Ode, int K>
__device__ __forceinline__ void neville_row(const BsmArgs &A, size_t e, size_t blk, int c, int g, double cur) {
    double old[8];
#pragma unroll
    for (int j = 0; j < K; j++) old[j] = ldc(&A.T[j * blk + e]);
    const double lim = K >= 1 && c < Ode::NERR ? A.tol * ldc(&A.SC[e]) : 0.0;
    const unsigned seen = K >= 1 ? __ldcg(&A.gfail[g]) : 0u;
    double last = 0.0;
    A.T[e] = cur;
#pragma unroll
    for (int j = 1; j <= K; j++) {
        const double coef = (double)((K - j + 1) * (K - j + 1)) / (double)(j * (2 * K + 2 - j));
        last = cur;
        cur = fma(cur - old[j - 1], coef, cur);
        A.T[j * blk + e] = cur;
    }
    A.DIAG[K * blk + e] = cur;
    // (most bits are there already: an atomic only for one that is not)
    if (K >= 1 && c < Ode::NERR && !(fabs(cur - last) <= lim) && !(seen >> K & 1u)) atomicOr(&A.gfail[g], 1u << K);
}
template <class Ode>
__device__ __forceinline__ void neville(const BsmArgs &A, int k, size_t e, size_t blk, int c, int g, double cur) {
    switch (k) {
    case 0: neville_row<Ode, 0>(A, e, blk, c, g, cur); break;
    case 1: neville_row<Ode, 1>(A, e, blk, c, g, cur); break;
    case 2: neville_row<Ode, 2>(A, e, blk, c, g, cur); break;
    case 3: neville_row<Ode, 3>(A, e, blk, c, g, cur); break;
    case 4: neville_row<Ode, 4>(A, e, blk, c, g, cur); break;
    case 5: neville_row<Ode, 5>(A, e, blk, c, g, cur); break;
    case 6: neville_row<Ode, 6>(A, e, blk, c, g, cur); break;
    default: neville_row<Ode, 7>(A, e, blk, c, g, cur); break;
    }
}
// Whether a column k >= 1 of the first `complete` ones met the tolerance.  Final
// once the barrier behind the sub-step that completed the last of them has passed.
__device__ __forceinline__ bool converged(unsigned fail, int complete) {
    return (~fail & 0xfeu & ((1u << complete) - 1u)) != 0u;
}

// Group g takes no part in sub-step it: done, or with a column under tolerance.
__device__ __forceinline__ bool idle(const BsmArgs &A, int g, int it) {
    return ldc(&A.gstat[g]) != 0 || converged(__ldcg(&A.gfail[g]), (it - 1) / 2);
}

template <class Ode, int L>
__device__ void phase_substep(const BsmArgs &A, int k, int m, int it, int lane) {
    const int nk = 2 * (k + 1), g = A.mgroup[m];
    const double h = ldc(&A.gh[(size_t)g * 8 + k]);
    if (h == 0.0) return;                        // the group is done
    if (A.ng > 1 && converged(__ldcg(&A.gfail[g]), (it - 1) / 2)) return;      // or has its column
    constexpr int D = Ode::D;
    const size_t ld = (size_t)A.M, blk = (size_t)D * ld;
    const double *Zcur = ((it & 1) ? A.ZA : A.ZB) + k * blk;
    double *Znext = ((it & 1) ? A.ZB : A.ZA) + k * blk;
    double *ZM = A.ZM + k * blk;
    double f[D];
    if constexpr (D == 6 && !Ode::COLL) {
        if (A.pairs) fwd_deriv_rec<L>(A, Zcur, k, m, lane, f);
        else Ode::template deriv<L>(A, Zcur, m, lane, f);
    } else {
        Ode::template deriv<L>(A, Zcur, m, lane, f);
    }
    const double h2 = 2.0 * h;
#pragma unroll
    for (int b = 0; b < D; b += L) {
        const int c = b + lane;
        const double fc = pick<D, L>(f, b, lane);
        if (c >= D) break;
        const double zc = ldc(&Zcur[c * ld + m]), zm = ldc(&ZM[c * ld + m]);
        if (it < nk) {
            ZM[c * ld + m] = zc;
            Znext[c * ld + m] = zm + h2 * fc;
        } else {
            neville<Ode>(A, k, c * ld + m, blk, c, g, 0.5 * (zc + zm + h * fc));
        }
    }
}

// Pair-centric mode, before each sub-step: pair t of column k computes the
// terms member m's partner loop would (displacement from m to its partner p,
// W, m_p W / r^3) and those p's would (the displacement negated, exactly, and
// m_m W / r^3), into the records of entries m -> p and p -> m.
__device__ void phase_pairs(const BsmArgs &A, int k, long long pi, int it) {
    const PairRec r = A.prec[pi];
    if (A.ng > 1 && idle(A, A.mgroup[r.m], it)) return;
    const size_t ld = (size_t)A.M, blk = 6 * ld;
    const double *Z = ((it & 1) ? A.ZA : A.ZB) + k * blk;
    const double x = ldc(&Z[0 * ld + r.m]), y = ldc(&Z[1 * ld + r.m]), z = ldc(&Z[2 * ld + r.m]);
    const double dx = ldc(&Z[0 * ld + r.p]) - x, dy = ldc(&Z[1 * ld + r.p]) - y, dz = ldc(&Z[2 * ld + r.p]) - z;
    const double d2 = fma(dz, dz, fma(dy, dy, dx * dx));
    const float rf = r_f32(d2);
    double cm = 0.0, cp = 0.0;
    bool in = true;
    for (int l = 0; l < A.nlev && in; l++)          // beyond some rc: no term, no FP64 reciprocal root
        in = changeover_side_f32(rf, __double2float_rz(A.pirc[(size_t)l * A.nq + pi])) <= 0;
    if (in) {
        const double yv = rsqrt_newton(d2);
        const double d = d2 * yv;
        double W = 1.0;
        for (int l = 0; l < A.nlev; l++) apply_changeover(rf, d, A.pirc[(size_t)l * A.nq + pi], W);
        const double y3 = yv * yv * yv;
        const double g = W * y3;
        cm = r.mp * g;
        cp = r.mm * g;
    }
    double2 *R = A.rec + (size_t)k * 2 * A.nq;
    R[2 * (size_t)r.q] = make_double2(cm, dx);
    R[2 * (size_t)r.q + 1] = make_double2(dy, dz);
    R[2 * (size_t)r.q2] = make_double2(cp, -dx);
    R[2 * (size_t)r.q2 + 1] = make_double2(-dy, -dz);
}

// The same for the star's coefficient -mu / r^3 of member m: a full warp of members
// here, where the member phase would repeat it in every lane of an item.
__device__ void phase_star(const BsmArgs &A, int k, int m, int it) {
    if (A.ng > 1 && idle(A, A.mgroup[m], it)) return;
    const size_t ld = (size_t)A.M, blk = 6 * ld;
    const double *Z = ((it & 1) ? A.ZA : A.ZB) + k * blk;
    const double x = ldc(&Z[0 * ld + m]), y = ldc(&Z[1 * ld + m]), z = ldc(&Z[2 * ld + m]);
    const double ys = rsqrt_newton(fma(z, z, fma(y, y, x * x)));
    A.star[(size_t)k * ld + m] = -A.mu * (ys * ys * ys);
}

// Collisions (reading R25) of group g, by one thread: the separation of two
// members in the state Z (component-major over members, stride M).
__device__ __forceinline__ double member_dist(const BsmArgs &A, const double *Z, int a, int b) {
    const size_t ld = (size_t)A.M;
    return __dsqrt_rn(dist2_rn(__dsub_rn(ldc(&Z[0 * ld + b]), ldc(&Z[0 * ld + a])),
                               __dsub_rn(ldc(&Z[1 * ld + b]), ldc(&Z[1 * ld + a])),
                               __dsub_rn(ldc(&Z[2 * ld + b]), ldc(&Z[2 * ld + a]))));
}

// Member m's part of the search for overlapping pairs of alive members in its group's
// state Z: the deepest overlap fraction (R_m + R_p - r) / (R_m + R_p) over its pairs with
// a higher body goes to the group's maximum (as bits: positive doubles order so).
// By one thread per group it took most of a giant group's step: 16,000 bodies with
// collisions on one level 4,935 ms, 69 ms so (8,000: 716, 12; 4,096: 157, 5.2).
__device__ void phase_overlap(const BsmArgs &A, const double *Z, int m) {
    if (!ldc(&A.malive[m])) return;
    double deepest = 0.0;
    for (int q = A.mq0[m]; q < A.mq1[m]; q++) {
        const int p = A.pidx[q];
        if (A.mbody[p] <= A.mbody[m] || !ldc(&A.malive[p])) continue;
        const double r = member_dist(A, Z, m, p);
        const double Rs = __dadd_rn(ldc(&A.coll.radius[A.mbody[m]]), ldc(&A.coll.radius[A.mbody[p]]));
        if (r < Rs) deepest = fmax(deepest, __ddiv_rn(__dsub_rn(Rs, r), Rs));
    }
    if (deepest > 0.0) atomicMax(&A.gdeep[A.mgroup[m]], (unsigned long long)__double_as_longlong(deepest));
}
// The group's maximum, left at zero.
__device__ __forceinline__ double take_deepest(const BsmArgs &A, int g) {
    return __longlong_as_double((long long)atomicExch(&A.gdeep[g], 0ull));
}
// First column k >= 1 under tolerance of a finished attempt, -1: none.
__device__ __forceinline__ int first_converged(unsigned fail) {
    const unsigned conv = ~fail & 0xfeu;
    return conv ? __ffs(conv) - 1 : -1;
}

// Mergers of the overlapping pairs of alive members of group g in the state
// Y at time t of the call, in ascending (i, j) order (members by rank, partner
// lists ascending), each seeing the mergers before it.
__device__ void group_merge(const BsmArgs &A, int g, double t) {
    const size_t ld = (size_t)A.M;
    const int label = A.mbody[A.morder[A.gbase[g]]];
    int seq = A.gseq[g];
    for (int rk = A.gbase[g]; rk < A.gbase[g + 1]; rk++) {
        const int m = A.morder[rk];
        for (int q = A.mq0[m]; q < A.mq1[m]; q++) {
            const int p = A.pidx[q];
            const int im = A.mbody[m], ip = A.mbody[p];
            if (ip <= im || !ldc(&A.malive[m]) || !ldc(&A.malive[p])) continue;
            const double r = member_dist(A, A.Y, m, p);
            const double Rs = __dadd_rn(ldc(&A.coll.radius[im]), ldc(&A.coll.radius[ip]));
            if (!(r < Rs)) continue;
            double xa[3], va[3], xb[3], vb[3], xo[3], vo[3], dU, rr;
            for (int k = 0; k < 3; k++) {
                xa[k] = ldc(&A.Y[k * ld + m]); va[k] = ldc(&A.Y[(3 + k) * ld + m]);
                xb[k] = ldc(&A.Y[k * ld + p]); vb[k] = ldc(&A.Y[(3 + k) * ld + p]);
            }
            const int sv = merge_bodies(A.coll, (size_t)A.coll.n, im, ip, xa, va, xb, vb, xo, vo, &dU, &rr);
            const int ms = sv == im ? m : p, mo = sv == im ? p : m;
            for (int k = 0; k < 3; k++) { A.Y[k * ld + ms] = xo[k]; A.Y[(3 + k) * ld + ms] = vo[k]; }
            A.mmass_rw[ms] = A.coll.mass[sv];
            A.mmass_rw[mo] = 0.0;
            A.malive[mo] = 0;
            log_merger(A.coll, A.ctr, label, seq++, t, im, ip, r, Rs, dU);
        }
    }
    A.gseq[g] = seq;
}

// The columns' midpoint sub-steps of group g's next attempt.
__device__ __forceinline__ void column_steps(const BsmArgs &A, int g, double t, double H) {
    const double left = A.dt - t;
    if (H > left) H = left;
    for (int k = 0; k < 8; k++) A.gh[(size_t)g * 8 + k] = H / (2 * (k + 1));
}

// Item t of the columns k0, k0 + 1, ... of `per` items each: the column; t becomes
// the item within it.
__device__ __forceinline__ int column_of(long long &t, long long per, int k0) {
    int k = k0;
    while (t >= per) {
        t -= per;
        k++;
    }
    return k;
}

// Step control of group g (the in-block kernels' rule).  The group's
// counters are touched only by this thread, so plain accesses suffice for
// them; the words other blocks read go through L2.
template <class Ode>
__device__ void phase_decide(const BsmArgs &A, int g) {
    A.gkconv[g] = -1;
    if (ldc(&A.gstat[g]) != 0) return;
    double H = step_of(A, g);
    int kconv = first_converged(atomicExch(&A.gfail[g], 0u));
    // collision precision (Sec. 7.2): a step that ends with an overlap of
    // tol or more of the radius sum ends too late
    if (Ode::COLL && A.coll.tol > 0.0 && take_deepest(A, g) >= A.coll.tol) kconv = -1;
    const long long att = A.gatt[g] + 1;
    A.gatt[g] = att;
    double t = ldc(&A.gt[g]);
    if (kconv >= 0) {
        t += H;
        A.gacc[g] += 1;
        if (kconv < 4) H *= 1.5;
    } else {
        A.grej[g] += 1;
        H *= 0.5;
    }
    A.gt[g] = t;
    A.gH[g] = H;
    A.gkconv[g] = kconv;
    column_steps(A, g, t, H);
    int st = 0;
    if (!(t < A.dt)) st = 1;
    else if (att >= A.max_steps) st = 2;
    if (st) {
        for (int k = 0; k < 8; k++) A.gh[(size_t)g * 8 + k] = 0.0;
        A.gstat[g] = st;
        atomicSub(&A.bar->running, 1u);
    }
}

template <class Ode>
__device__ void phase_accept(const BsmArgs &A, long long t) {
    constexpr int D = Ode::D;
    const size_t blk = (size_t)D * A.M;
    const int m = (int)(t % A.M);
    const int k = ldc(&A.gkconv[A.mgroup[m]]);
    if (k >= 0) A.Y[t] = ldc(&A.DIAG[k * blk + t]);
}

template <class Ode, int L>
// Two blocks per SM (64 registers) for the forward ODE: the gathers through L2 want
// the warps (16,384-body step 22.5 ms; one block: 23.2).
__global__ void __launch_bounds__(kPMaxThreads, Ode::D == 6 && !Ode::COLL ? 2 : 1)
bsm_persistent_kernel(BsmArgs A) {
    constexpr int D = Ode::D;
    const long long nth = (long long)gridDim.x * blockDim.x;
    // consecutive warps' worth of work go to consecutive blocks, so that a phase
    // with few items (the last sub-steps: one column) still reaches every SM
    const long long tid = ((long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
    const long long M = A.M;
    // derivative phases: L adjacent lanes per item
    const long long item0 = tid / L, nitem = nth / L;
    const int lane = (int)(threadIdx.x % L);
    // pairs of the pair-centric mode (listed by bsm_pairs_kernel before the launch)
    const long long P = (D == 6 && !Ode::COLL && A.pairs) ? (long long)*A.pcount : 0;
    __shared__ unsigned running;
    unsigned long long arrived = 0ull;            // thread 0: arrivals the next barrier waits for
    if (Ode::COLL) {
        // pairs already overlapping when the integration starts merge at once
        for (long long m = tid; m < M; m += nth) phase_overlap(A, A.Y, (int)m);
        if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
        for (long long g = tid; g < A.ng; g += nth)
            if (take_deepest(A, (int)g) > 0.0) group_merge(A, (int)g, 0.0);
        if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
    }
    for (int round = 0; round < A.max_steps; round++) {
        // one read per block; the previous round ended with a barrier
        if (threadIdx.x == 0) running = atomicAdd(&A.bar->running, 0u);
        __syncthreads();
        if (running == 0u) break;
        for (long long t = item0; t < M; t += nitem) phase_start<Ode, L>(A, (int)t, lane);
        if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
        for (int it = 1; it <= 16; it++) {
            const int k0 = (it - 1) / 2;          // columns below have no sub-step left
            if (P > 0) {
                for (long long t = tid; t < (8 - k0) * (P + M); t += nth) {
                    long long pi = t;
                    const int k = column_of(pi, P + M, k0);
                    if (pi < P) phase_pairs(A, k, pi, it);
                    else phase_star(A, k, (int)(pi - P), it);
                }
                if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
            }
            for (long long t = item0; t < (8 - k0) * M; t += nitem) {
                long long m = t;
                const int k = column_of(m, M, k0);
                phase_substep<Ode, L>(A, k, (int)m, it, lane);
            }
            if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
            // a column was completed: done when every running group has one under
            // tolerance.  All blocks see the same bits: those of later columns, which
            // blocks ahead may be setting, do not count.
            if (it >= 4 && !(it & 1)) {
                bool open = false;
                for (int g = threadIdx.x; g < A.ng; g += blockDim.x)
                    open = open || (ldc(&A.gstat[g]) == 0 && !converged(__ldcg(&A.gfail[g]), it / 2));
                if (!__syncthreads_or(open)) break;
            }
        }
        if (Ode::COLL && A.coll.tol > 0.0) {
            for (long long m = tid; m < M; m += nth) {
                const int g = A.mgroup[m], k = ldc(&A.gstat[g]) == 0 ? first_converged(__ldcg(&A.gfail[g])) : -1;
                if (k >= 0) phase_overlap(A, A.DIAG + (size_t)k * D * M, (int)m);
            }
            if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
        }
        for (long long g = tid; g < A.ng; g += nth) phase_decide<Ode>(A, (int)g);
        if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
        for (long long t = tid; t < D * M; t += nth) phase_accept<Ode>(A, t);
        if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
        if (Ode::COLL) {
            // mergers at the end of every accepted step (same thread per group
            // as the decision, which wrote gkconv and gt)
            for (long long m = tid; m < M; m += nth)
                if (ldc(&A.gkconv[A.mgroup[m]]) >= 0) phase_overlap(A, A.Y, (int)m);
            if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
            for (long long g = tid; g < A.ng; g += nth)
                if (A.gkconv[g] >= 0 && take_deepest(A, (int)g) > 0.0) group_merge(A, (int)g, ldc(&A.gt[g]));
            if (!grid_barrier(A.bar, A.barrier_ns, A.first_ns, A.barrier_absent, arrived)) return;
        }
    }
}

// ---------------------------------------------------------------- set-up
struct RcPtrs {
    const double *p[kMaxLevels];
};

// Per member: group, body, partner range, compact partner indices, mass, 1/rc.
__global__ void bsm_members_kernel(int ng, const int *gbase, const int *gslot0, const int *member,
                                   const int *slotof, const int *off, const int *list, const double *mass,
                                   RcPtrs rc, int nlev, int M, int *mbody, int *mgroup, int *mq0, int *mq1,
                                   int *pidx, double *mmass, double *irc) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    int lo = 0, hi = ng - 1;                     // last group with gbase <= m
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (gbase[mid] <= m) lo = mid; else hi = mid - 1;
    }
    mgroup[m] = lo;
    const int b = member[gslot0[lo] + (m - gbase[lo])];
    mbody[m] = b;
    mmass[m] = mass[b];
    const int q0 = off[b], q1 = off[b + 1];
    mq0[m] = q0;
    mq1[m] = q1;
    // partners belong to the same group (connected components of the pair graph)
    for (int q = q0; q < q1; q++) pidx[q] = gbase[lo] + (slotof[list[q]] - gslot0[lo]);
    for (int l = 0; l < nlev; l++) irc[(size_t)l * M + m] = 1.0 / rc.p[l][b];
}

// Pair-centric mode: the unordered pairs of the batched members (each listed
// from its lower member, in any order) with the reverse entry (the rows are
// ascending in body index, so a binary search finds it), masses and 1/rc.
__global__ void bsm_pairs_kernel(int M, const int *mq0, const int *mq1, const int *pidx, const int *mbody,
                                 const int *list, const double *mmass, const double *irc, int nlev, size_t nq,
                                 int *pcount, PairRec *prec, double *pirc) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int bm = mbody[m];
    for (int q = mq0[m]; q < mq1[m]; q++) {
        const int p = pidx[q];
        if (p <= m) continue;
        int lo = mq0[p], hi = mq1[p] - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (list[mid] < bm) lo = mid + 1; else hi = mid;
        }
        const int k = atomicAdd(pcount, 1);
        PairRec r;
        r.m = m; r.p = p; r.q = q; r.q2 = lo;
        r.mm = mmass[m]; r.mp = mmass[p];
        prec[k] = r;
        for (int l = 0; l < nlev; l++) pirc[(size_t)l * nq + k] = fmin(irc[(size_t)l * M + m], irc[(size_t)l * M + p]);
    }
}

// Collisions: each member's alive flag, and the members of each group by
// ascending body index (rank = members of the group with a smaller body).
__global__ void bsm_coll_init_kernel(BsmArgs A) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= A.M) return;
    const int b = A.mbody[m];
    A.malive[m] = A.coll.alive[b];
    const int g = A.mgroup[m];
    int rank = 0;
    for (int q = A.gbase[g]; q < A.gbase[g + 1]; q++) rank += A.mbody[q] < b;
    A.morder[A.gbase[g] + rank] = m;
}

__global__ void bsm_init_groups_kernel(BsmArgs A) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g == 0) {
        A.bar->count = 0ull;
        A.bar->err = 0u;
        A.bar->running = (unsigned)A.ng;
    }
    if (g >= A.ng) return;
    A.gt[g] = 0.0;
    A.gH[g] = A.dt;
    A.gstat[g] = 0;
    A.gkconv[g] = -1;
    A.gatt[g] = 0;
    A.gacc[g] = 0;
    A.grej[g] = 0;
    if (A.gseq) A.gseq[g] = 0;
    if (A.gdeep) A.gdeep[g] = 0ull;
    A.gfail[g] = 0u;
    column_steps(A, g, 0.0, A.dt);
}

__global__ void bsm_gather_fwd(int n, int M, const int *mbody, const double *pos, const double *vel, double *Y) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int b = mbody[m];
    for (int c = 0; c < 3; c++) {
        Y[c * (size_t)M + m] = pos[c * (size_t)n + b];
        Y[(3 + c) * (size_t)M + m] = vel[c * (size_t)n + b];
    }
}
__global__ void bsm_scatter_fwd(int n, int M, const int *mbody, const double *Y, double *pos, double *vel) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int b = mbody[m];
    for (int c = 0; c < 3; c++) {
        pos[c * (size_t)n + b] = Y[c * (size_t)M + m];
        vel[c * (size_t)n + b] = Y[(3 + c) * (size_t)M + m];
    }
}
__global__ void bsm_gather_adj(int n, int M, const int *mbody, const double *x2, const double *v2,
                               const double *lx, const double *lv, double *Y) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int b = mbody[m];
    const size_t ld = (size_t)M;
    for (int c = 0; c < 3; c++) {
        Y[c * ld + m] = x2[c * (size_t)n + b];
        Y[(3 + c) * ld + m] = v2[c * (size_t)n + b];
        Y[(6 + c) * ld + m] = lx[c * (size_t)n + b];
        Y[(9 + c) * ld + m] = lv[c * (size_t)n + b];
    }
    Y[12 * ld + m] = 0.0;
}
__global__ void bsm_scatter_adj(int n, int M, const int *mbody, const double *Y, double *lx, double *lv,
                                double *lm) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int b = mbody[m];
    const size_t ld = (size_t)M;
    for (int c = 0; c < 3; c++) {
        lx[c * (size_t)n + b] = Y[(6 + c) * ld + m];
        lv[c * (size_t)n + b] = Y[(9 + c) * ld + m];
    }
    lm[b] += Y[12 * ld + m];
}

// Folds the groups' counters into the system's (one thread, group order).
__global__ void bsm_stats_kernel(BsmArgs A, DevCounters *ctr, int count_steps) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    unsigned long long acc = 0, rej = 0, att = 0, fail = 0;
    for (int g = 0; g < A.ng; g++) {
        acc += (unsigned long long)A.gacc[g];
        rej += (unsigned long long)A.grej[g];
        if ((unsigned long long)A.gatt[g] > att) att = (unsigned long long)A.gatt[g];
        fail += A.gstat[g] == 2 ? 1ull : 0ull;
    }
    if (count_steps) {
        atomicAdd(&ctr->bs_steps, acc);
        atomicAdd(&ctr->bs_rejects, rej);
        atomicMax(&ctr->bs_max_attempts, att);
    }
    if (fail) {
        atomicAdd(&ctr->bs_fail, fail);
        latch_error(ctr, kErrBS);
    }
}

// Device buffers of the batch, grown on demand, kept by the system.
struct BsmBuffers {
    void *raw = nullptr;
    size_t bytes = 0;
};

void *bsm_reserve(genga_system *s, size_t bytes) {
    BsmBuffers *b = static_cast<BsmBuffers *>(s->bsm);
    if (!b) {
        b = new BsmBuffers;
        s->bsm = b;
    }
    if (b->bytes < bytes) {
        if (b->raw) cudaFree(b->raw);
        b->raw = nullptr;
        b->bytes = 0;
        if (cudaMalloc(&b->raw, bytes) != cudaSuccess) return nullptr;
        b->bytes = bytes;
    }
    return b->raw;
}

// Host list of the groups with more than kBlockGroupMax members: (slot0, nm),
// ascending slot.
int batched_groups(genga_system *s, std::vector<int2> &out) {
    out.clear();
    DevCounters c;
    if (cudaMemcpyAsync(&c, s->ctr, sizeof(c), cudaMemcpyDeviceToHost, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return -1;
    ++s->host_syncs;
    if ((int)c.max_group <= kBlockGroupMax || c.ngroups == 0) return 0;
    std::vector<int> glist(c.ngroups), goff((size_t)s->n + 1);
    if (cudaMemcpyAsync(glist.data(), s->glist, sizeof(int) * c.ngroups, cudaMemcpyDeviceToHost, s->stream) !=
            cudaSuccess ||
        cudaMemcpyAsync(goff.data(), s->goff, sizeof(int) * goff.size(), cudaMemcpyDeviceToHost, s->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return -1;
    ++s->host_syncs;
    for (int g : glist) {
        const int nm = goff[(size_t)g + 1] - goff[(size_t)g];
        if (nm > kBlockGroupMax) out.push_back(make_int2(goff[(size_t)g], nm));
    }
    std::sort(out.begin(), out.end(), [](const int2 &a, const int2 &b) { return a.x < b.x; });
    return 0;
}

size_t aligned(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

template <typename T>
T *carve(char *&p, size_t count) {
    T *r = reinterpret_cast<T *>(p);
    p += aligned(sizeof(T) * count);
    return r;
}

// Runs every batched group over dt from the state `gather` writes into Y;
// `scatter` takes Y back.  Returns a genga error code.
template <class Ode, class Gather, class Scatter>
int bsm_run(genga_system *s, int level, double dt, const std::vector<int2> &groups, bool count_steps,
            Gather gather, Scatter scatter) {
    constexpr int D = Ode::D;
    const int ng = (int)groups.size();
    const int nlev = level + 1;
    std::vector<int> gbase(ng + 1), gslot0(ng);
    int M = 0;
    for (int g = 0; g < ng; g++) {
        gbase[g] = M;
        gslot0[g] = groups[g].x;
        M += groups[g].y;
    }
    gbase[ng] = M;
    const size_t blk = (size_t)D * M;
    const size_t nq = 2 * (size_t)s->csr[level].cap;
    // One persistent cooperative launch: one block per SM as large as the items
    // need (fewer arrivals at a grid barrier than with small blocks), more blocks
    // where they fill it.
    int L = 16;
    while (L > 4 && 8LL * M * L > (long long)kItemWarps * 4 * 32 * s->num_sms) L /= 2;
    const void *kernel = L == 16  ? (const void *)bsm_persistent_kernel<Ode, 16>
                         : L == 8 ? (const void *)bsm_persistent_kernel<Ode, 8>
                                  : (const void *)bsm_persistent_kernel<Ode, 4>;
    const long long want_threads = 8LL * M * L;
    const int threads = (int)std::min<long long>(kPMaxThreads,
                                                 ((want_threads + s->num_sms - 1) / s->num_sms + 31) / 32 * 32);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
        return GENGA_ECUDA;
    const long long want = (want_threads + threads - 1) / threads;
    const long long cap = (long long)per_sm * s->num_sms;
    const unsigned grid = (unsigned)std::max(1LL, std::min(want, cap));
    // pair-centric derivative from kPairMembers members on, and where a sub-step
    // phase takes more than two passes over its items: the FP64 work of the
    // partner terms, halved and evenly spread over the lanes, outweighs a second
    // barrier per sub-step
    const bool pairs = D == 6 && !Ode::COLL &&
                       (s->bs_pairs == GENGA_BS_PAIRS_ON ||
                        (s->bs_pairs == GENGA_BS_PAIRS_AUTO && (M >= kPairMembers || 8LL * M > 2LL * grid * (threads / L))));
    const size_t np = nq / 2;
    const size_t pbytes = pairs ? aligned(sizeof(double2) * 2 * 8 * nq) + aligned(sizeof(PairRec) * np) +
                                      aligned(sizeof(double) * nlev * nq) + aligned(sizeof(int)) + aligned(sizeof(double) * 8 * M)
                                : 0;
    const size_t bytes = pbytes + aligned(sizeof(double) * blk) * 3 + aligned(sizeof(double) * 8 * blk) * 5 +
                         aligned(sizeof(double) * (size_t)nlev * M) + aligned(sizeof(double) * M) +
                         aligned(sizeof(int) * M) * 4 + aligned(sizeof(int) * nq) +
                         aligned(sizeof(int) * (ng + 1)) + aligned(sizeof(int) * ng) * 4 +
                         aligned(sizeof(double) * ng) * 2 +
                         aligned(sizeof(long long) * ng) * 3 + aligned(sizeof(unsigned) * ng) + aligned(sizeof(double) * 8 * ng) +
                         aligned(sizeof(GridBarrier)) +
                         (Ode::COLL ? aligned(sizeof(int) * M) * 2 + aligned(sizeof(unsigned long long) * ng) : 0);
    char *p = static_cast<char *>(bsm_reserve(s, bytes));
    if (!p) return GENGA_ENOMEM;
    BsmArgs A;
    A.M = M; A.ng = ng; A.nlev = nlev;
    A.pairs = pairs ? 1 : 0;
    A.nq = nq;
    int *pcount = nullptr;
    PairRec *prec = nullptr;
    double *pirc = nullptr;
    A.rec = nullptr;
    A.star = nullptr;
    if (pairs) {
        A.rec = carve<double2>(p, 2 * 8 * nq);
        prec = carve<PairRec>(p, np);
        pirc = carve<double>(p, (size_t)nlev * nq);
        pcount = carve<int>(p, 1);
        A.star = carve<double>(p, 8 * (size_t)M);
    }
    A.pcount = pcount; A.prec = prec; A.pirc = pirc;
    A.Y = carve<double>(p, blk); A.F0 = carve<double>(p, blk); A.SC = carve<double>(p, blk);
    A.ZM = carve<double>(p, 8 * blk); A.ZA = carve<double>(p, 8 * blk); A.ZB = carve<double>(p, 8 * blk);
    A.T = carve<double>(p, 8 * blk); A.DIAG = carve<double>(p, 8 * blk);
    double *irc = carve<double>(p, (size_t)nlev * M), *mmass = carve<double>(p, M);
    int *mbody = carve<int>(p, M), *mgroup = carve<int>(p, M), *mq0 = carve<int>(p, M), *mq1 = carve<int>(p, M);
    int *pidx = carve<int>(p, nq);
    int *d_gbase = carve<int>(p, ng + 1), *d_gslot0 = carve<int>(p, ng);
    int *gseq = carve<int>(p, ng);
    A.gstat = carve<int>(p, ng);
    A.gkconv = carve<int>(p, ng);
    A.gt = carve<double>(p, ng);
    A.gH = carve<double>(p, ng);
    A.gatt = carve<long long>(p, ng);
    A.gacc = carve<long long>(p, ng);
    A.grej = carve<long long>(p, ng);
    A.gfail = carve<unsigned>(p, ng);
    A.gh = carve<double>(p, 8 * (size_t)ng);
    A.bar = carve<GridBarrier>(p, 1);
    A.mgroup = mgroup; A.mq0 = mq0; A.mq1 = mq1; A.pidx = pidx; A.mmass = mmass; A.irc = irc;
    A.mbody = mbody; A.gbase = d_gbase; A.mmass_rw = mmass; A.ctr = s->ctr;
    A.coll = coll_args(s);
    A.gseq = Ode::COLL ? gseq : nullptr;
    A.morder = Ode::COLL ? carve<int>(p, M) : nullptr;
    A.malive = Ode::COLL ? carve<int>(p, M) : nullptr;
    A.gdeep = Ode::COLL ? carve<unsigned long long>(p, ng) : nullptr;
    A.G = s->p.G; A.mu = s->p.G * s->p.m_star; A.dt = dt; A.tol = s->p.bs_tol;
    A.max_steps = s->p.bs_max_steps;
    A.barrier_ns = s->barrier_limit_ns;
    A.first_ns = s->bs_beside ? s->bs_group_limit_ns : 0ull;
    A.barrier_absent = s->barrier_absent;

    cudaStream_t st = s->stream;
    if (cudaMemcpyAsync(d_gbase, gbase.data(), sizeof(int) * (ng + 1), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(d_gslot0, gslot0.data(), sizeof(int) * ng, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return GENGA_ECUDA;
    RcPtrs rcp;
    for (int l = 0; l < kMaxLevels; l++) rcp.p[l] = s->rcl[l].rc;
    const unsigned gm = (unsigned)((M + 127) / 128);
    bsm_members_kernel<<<gm, 128, 0, st>>>(ng, d_gbase, d_gslot0, s->member, s->slotof, s->csr[level].off,
                                          s->csr[level].list, s->mass, rcp, nlev, M, mbody, mgroup, mq0, mq1,
                                          pidx, mmass, irc);
    bsm_init_groups_kernel<<<(unsigned)((ng + 127) / 128), 128, 0, st>>>(A);
    if (pairs) {
        if (cudaMemsetAsync(pcount, 0, sizeof(int), st) != cudaSuccess) return GENGA_ECUDA;
        bsm_pairs_kernel<<<gm, 128, 0, st>>>(M, mq0, mq1, pidx, mbody, s->csr[level].list, mmass, irc, nlev, nq, pcount,
                                             prec, pirc);
        ++s->launches;
    }
    if (Ode::COLL) {
        bsm_coll_init_kernel<<<gm, 128, 0, st>>>(A);
        ++s->launches;
    }
    gather(st, mbody, A.Y);
    s->launches += 3;
    if (cudaGetLastError() != cudaSuccess) return GENGA_ECUDA;

    void *args[] = {&A};
    if (cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(threads), args,
                                    0, st) != cudaSuccess)
        return GENGA_ECUDA;
    ++s->launches;
    GridBarrier hb;
    if (cudaMemcpyAsync(&hb, A.bar, sizeof(hb), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return GENGA_ECUDA;
    ++s->host_syncs;
    if (hb.err) {
        snprintf(s->err, sizeof(s->err),
                 "persistent Bulirsch-Stoer: a grid-barrier wait exceeded its limit of %.3g s",
                 1e-9 * (double)(A.barrier_ns + (hb.err == 2u ? A.first_ns : 0ull)));
        return GENGA_ETIMEOUT;
    }
    scatter(st, mbody, A.Y);
    bsm_stats_kernel<<<1, 1, 0, st>>>(A, s->ctr, count_steps ? 1 : 0);
    s->launches += 2;
    return cudaGetLastError() == cudaSuccess ? GENGA_OK : GENGA_ECUDA;
}

int members_of(const std::vector<int2> &groups) {
    int t = 0;
    for (const int2 &g : groups) t += g.y;
    return t;
}

}  // namespace

void bsm_release(genga_system *s) {
    BsmBuffers *b = static_cast<BsmBuffers *>(s->bsm);
    if (!b) return;
    if (b->raw) cudaFree(b->raw);
    delete b;
    s->bsm = nullptr;
}

// Forward BS of every group larger than kBlockGroupMax, from the level's
// pre-drift state into pos/vel.
int bsm_forward_groups(genga_system *s, int level, double dt_l) {
    std::vector<int2> groups;
    if (batched_groups(s, groups) != 0) return GENGA_ECUDA;
    if (groups.empty()) return GENGA_OK;
    const double *pre_pos = s->pre_pos[level], *pre_vel = s->pre_vel[level];
    double *pos = s->pos, *vel = s->vel;
    const int n = (int)s->n;
    const int M = members_of(groups);
    const unsigned gr = (unsigned)((M + 127) / 128);
    auto gather = [&](cudaStream_t st, const int *mbody, double *Y) {
        bsm_gather_fwd<<<gr, 128, 0, st>>>(n, M, mbody, pre_pos, pre_vel, Y);
    };
    auto scatter = [&](cudaStream_t st, const int *mbody, const double *Y) {
        bsm_scatter_fwd<<<gr, 128, 0, st>>>(n, M, mbody, Y, pos, vel);
    };
    if (s->coll_on) return bsm_run<FwdCollOde>(s, level, dt_l, groups, true, gather, scatter);
    return bsm_run<FwdOde>(s, level, dt_l, groups, true, gather, scatter);
}

// Bulirsch-Stoer of every group of the current grouping at `level`: the
// in-block kernels for groups of up to kBlockGroupMax members on the side
// streams, the persistent driver for the larger ones on the system's stream
// beside them.  The groups share no body, and both add to the counters by atomics.
// (The cooperative launch starts once all its blocks fit; the in-block kernels
// wait for nothing, so that is when they leave room at the latest.)  Both are
// bound by latency with little of the GPU in use unless a group is a giant:
// N = 2,048, FP64: 1.84 ms for both, 3.75 ms one after the other.
// Joins the side streams, whatever the result of the persistent driver.
static int bs_large_and_join(genga_system *s, int level, double dt_l, const unsigned *counts) {
    int rc = GENGA_OK;
    if (counts[kBuckets - 1]) {
        rc = phase_mark(s, GENGA_PH_BS_LARGE);
        for (int q = 0; q + 1 < kBuckets; q++) s->bs_beside = s->bs_beside || counts[q];
        if (rc == GENGA_OK) rc = bsm_forward_groups(s, level, dt_l);
        s->bs_beside = false;
        if (rc == GENGA_OK) rc = phase_mark(s, GENGA_PH_BS_SMALL);     // what is left of them
    }
    if (join_bs(s) != cudaSuccess) return rc != GENGA_OK ? rc : GENGA_ECUDA;
    return rc;
}

int run_bs(genga_system *s, int level, double dt_l, int64_t np) {
    if (np <= 0) return GENGA_OK;
    ++s->bs_call;                         // orders the merger records of the calls
    unsigned counts[kBuckets];
    int rc = phase_mark(s, GENGA_PH_BUCKETS);
    if (rc != GENGA_OK) return rc;
    if (bucket_groups(s, counts) != cudaSuccess) return GENGA_ECUDA;
    if ((rc = phase_mark(s, GENGA_PH_BS_SMALL)) != GENGA_OK) return rc;
    if (launch_bs(s, level, dt_l, counts) != cudaSuccess) {
        join_bs(s);
        return GENGA_ECUDA;
    }
    return bs_large_and_join(s, level, dt_l, counts);
}

extern "C" int genga_set_bs_pair_mode(genga_system_t *s, int32_t mode) {
    if (!s || mode < GENGA_BS_PAIRS_AUTO || mode > GENGA_BS_PAIRS_ON) return GENGA_EINVAL;
    s->bs_pairs = mode;
    return GENGA_OK;
}

int run_bs_dev(genga_system *s, int level, double dt_l) {
    ++s->bs_call;
    int rc = phase_mark(s, GENGA_PH_BUCKETS);
    if (rc != GENGA_OK) return rc;
    if (bucket_groups_async(s) != cudaSuccess) return GENGA_ECUDA;
    if ((rc = phase_mark(s, GENGA_PH_BS_SMALL)) != GENGA_OK) return rc;
    // the counts were copied before the kernels above run: the GPU keeps
    // working while the host reads them
    if (launch_bs(s, level, dt_l, nullptr) != cudaSuccess || cudaEventSynchronize(s->ev_counts) != cudaSuccess) {
        join_bs(s);
        return GENGA_ECUDA;
    }
    ++s->host_syncs;
    return bs_large_and_join(s, level, dt_l, s->bucket_host);
}

// Adjoint BS (backward, augmented) of every group larger than kBlockGroupMax.
int bsm_adjoint_groups(genga_system *s, const double *x2, const double *v2, double *lx, double *lv,
                       double *lm, double dt) {
    std::vector<int2> groups;
    if (batched_groups(s, groups) != 0) return GENGA_ECUDA;
    if (groups.empty()) return GENGA_OK;
    const int n = (int)s->n;
    const int M = members_of(groups);
    const unsigned gr = (unsigned)((M + 127) / 128);
    return bsm_run<AdjOde>(
        s, 0, dt, groups, false,
        [&](cudaStream_t st, const int *mbody, double *Y) {
            bsm_gather_adj<<<gr, 128, 0, st>>>(n, M, mbody, x2, v2, lx, lv, Y);
        },
        [&](cudaStream_t st, const int *mbody, const double *Y) {
            bsm_scatter_adj<<<gr, 128, 0, st>>>(n, M, mbody, Y, lx, lv, lm);
        });
}

}  // namespace genga
