// energy.cu -- the energy and angular-momentum report (Eq. H): kinetic and star
// terms, angular momentum and momentum per body, the pair potential over all
// unordered pairs, compensated sums in a fixed order.
//
// The pair potential is the whole cost.  An FP64 square root and division per
// ordered pair take ~30 FP64 instructions; here 1/r of an unordered pair is formed
// on the FP32 pipe (64 times faster) to the last place of an FP64 value, and one
// FP64 FMA per pair sums m_j / r_ij:
//   * displacement from the packed bodies (kick_ff.cu) as three floats, exact to
//     2^-72 of the largest coordinate;
//   * y = rsqrt(r^2) in FP32, q = d y per component; the residual e = 1 - |q|^2
//     (|e| < 2^-20.5) to 2^-56: q is cut into digits on the fixed grids 2^-11,
//     2^-22 and 2^-34 (|q| <= 1), whose products are whole multiples of 2^-44 and
//     whose sums fit a float, so only the last digits' products round;
//   * 1/r = y (1 + e/2 + 3 e^2/8): the correction as a whole number of units of
//     the last place of y as a double, added to its bits.
// ~130 FP32 operations, one FP64 and ~40 integer instructions per unordered pair,
// bound by the FP32 pipe and the register reads of its three-operand FMAs.
// N = 65,540: 10.9 ms, against 207 ms for the FP64 square root and division of
// every ordered pair (the same E and L to the last bit there).
#include <algorithm>

#include "ff_pair.cuh"

namespace genga {
namespace {

constexpr int kEnThreads = 128;                // a tile's rows
constexpr int kEnRows = 9;                     // per-body sums
constexpr int kEnBlocks = 1024;                // partial sums per row, at most

struct EnergyArgs {
    const double *x, *y, *z, *m;
    const float4 *body;
    const int *header;                         // of the packed bodies
    int n, nm, nT;
    double *part;                              // [2][gridDim.x]: sum, compensation
};

// Sum of all threads' (S, C) pairs in a fixed order (TwoSum tree), to thread 0.
template <int T>
__device__ __forceinline__ void block_sum2(double &S, double &C, double *sh) {
    __syncthreads();
    sh[threadIdx.x] = S;
    sh[T + threadIdx.x] = C;
    __syncthreads();
#pragma unroll
    for (int w = T / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            double t, e;
            two_sum(sh[threadIdx.x], sh[threadIdx.x + w], t, e);
            sh[threadIdx.x] = t;
            sh[T + threadIdx.x] += sh[T + threadIdx.x + w] + e;
        }
        __syncthreads();
    }
    S = sh[0];
    C = sh[T];
}

// 1/r in FP64: close pairs (r < 2^-17 S: 2^-72 S is more than 2^-55 of the distance, 0
// among them) and NaN, 1/r next to a power of two.
__device__ __noinline__ double rinv_fp64(const EnergyArgs &A, int i, int j) {
    const double dx = A.x[j] - A.x[i], dy = A.y[j] - A.y[i], dz = A.z[j] - A.z[i];
    return 1.0 / sqrt(dx * dx + dy * dy + dz * dz);
}

// (TS, TC) += m (S + C)
__device__ __forceinline__ void add_row(double &TS, double &TC, double m, double S, double C) {
    const double P = m * S;
    double s, e;
    two_sum(TS, P, s, e);
    TS = s;
    TC += e + (fma(m, S, -P) + m * C);
}

// The pairs i < j, by tiles (a, b), a <= b, in an order in which every block takes
// one contiguous range: row a of tiles is followed by row nT - 1 - a, so that two
// rows together always have nT + 1 tile pairs.
__global__ void __launch_bounds__(kEnThreads, 4)
energy_pairs_kernel(EnergyArgs A) {
    __shared__ float4 tile[6 * kFfRow];
    __shared__ double sm[kSymT];
    __shared__ double sh[2 * kEnThreads];
    const int nT = A.nT, tid = threadIdx.x;
    const long long total = (long long)nT * (nT + 1) / 2;
    const long long u0 = total * blockIdx.x / gridDim.x, u1 = total * (blockIdx.x + 1) / gridDim.x;
    constexpr float close2 = 0x1p-22f;                     // (2^-17 S)^2
    const double unit = scalbn(1.0, A.header[2]);          // of the packed bodies' lengths
    const f2 half = f2_dup(0.5f), c375 = f2_dup(0.375f);
    double TS = 0.0, TC = 0.0;                 // this thread's sum of m_i m_j / r_ij
    double S = 0.0, C = 0.0;                   // its row's sum of m_j / r_ij
    f2 nh[3], nm[3], nl[3];
    int row = -1, i = 0;
    for (long long u = u0; u < u1; u++) {
        const long long p = u / (nT + 1);
        const int t = (int)(u - p * (nT + 1));
        const bool second = t >= nT - (int)p;
        const int a = second ? nT - 1 - (int)p : (int)p;
        const int b = second ? a + (t - (nT - (int)p)) : (int)p + t;
        if (a != row) {
            if (row >= 0 && i < A.n) add_row(TS, TC, A.m[i], S, C);
            S = C = 0.0;
            row = a;
            i = a * kSymT + tid;
            const float4 *B = A.body + (size_t)a * kFfTile + (tid >> 6) * 32 + (tid & 31);
            const bool up = tid & 32;
            const float4 q0 = B[0], q1 = B[kFfRow], q2 = B[2 * kFfRow], q3 = B[3 * kFfRow], q4 = B[4 * kFfRow],
                         q5 = B[5 * kFfRow];
            nh[0] = f2_dup(-(up ? q0.y : q0.x)); nh[1] = f2_dup(-(up ? q0.w : q0.z)); nh[2] = f2_dup(-(up ? q1.y : q1.x));
            nm[0] = f2_dup(-(up ? q2.y : q2.x)); nm[1] = f2_dup(-(up ? q2.w : q2.z)); nm[2] = f2_dup(-(up ? q3.y : q3.x));
            nl[0] = f2_dup(-(up ? q4.y : q4.x)); nl[1] = f2_dup(-(up ? q4.w : q4.z)); nl[2] = f2_dup(-(up ? q5.y : q5.x));
        }
        if (a * kSymT >= A.nm) continue;       // test particles only (b >= a): block-uniform
        __syncthreads();                       // the tile buffer is free
        for (int k = tid; k < 6 * kFfRow; k += kEnThreads) tile[k] = A.body[(size_t)b * kFfTile + k];
        {
            const int j = b * kSymT + tid;
            sm[tid] = j < A.n ? A.m[j] : 0.0;
        }
        __syncthreads();
        const bool mask = a == b || ((a + 1) * kSymT > A.nm && (b + 1) * kSymT > A.nm);
        double s0 = 0.0, s1 = 0.0;
#pragma unroll 2
        for (int k = 0; k < kFfRow; k++) {
            const float4 q0 = tile[k], q1 = tile[kFfRow + k], q2 = tile[2 * kFfRow + k], q3 = tile[3 * kFfRow + k],
                         q4 = tile[4 * kFfRow + k], q5 = tile[5 * kFfRow + k];
            const int jx = (k >> 5) * 64 + (k & 31), jy = jx + 32;              // in the tile
            double mx = sm[jx], my = sm[jy];
            bool wx = true, wy = true;
            if (mask) {
                const int gx = b * kSymT + jx, gy = b * kSymT + jy;
                wx = gx > i && !(i >= A.nm && gx >= A.nm);
                wy = gy > i && !(i >= A.nm && gy >= A.nm);
                if (!wx) mx = 0.0;
                if (!wy) my = 0.0;
            }
            const f2 hj[3] = {f2_lo(q0), f2_hi(q0), f2_lo(q1)}, mj[3] = {f2_lo(q2), f2_hi(q2), f2_lo(q3)},
                     lj[3] = {f2_lo(q4), f2_hi(q4), f2_lo(q5)};
            f2 H[3], L[3], T[3];
#pragma unroll
            for (int c = 0; c < 3; c++) ff_disp3(hj[c], mj[c], lj[c], nh[c], nm[c], nl[c], H[c], L[c], T[c]);
            const f2 s = f2_fma(H[2], H[2], f2_fma(H[1], H[1], f2_mul(H[0], H[0])));
            const f2 y = f2_rsqrt(s);
            f2 eh, el;
            ff_residual(H, L, T, y, eh, el);
            // y (1 + e/2 + 3 e^2/8) - y = vh + vl
            const f2 x = f2_mul(y, eh), xe = f2_fma(y, eh, f2_neg(x));
            const f2 tt = f2_fma(f2_mul(c375, eh), eh, f2_mul(half, el));
            const float2 Y = f2_get(y), R2 = f2_get(s);
            const f2 sc = f2_make(ff_ulp_scale(Y.x), ff_ulp_scale(Y.y));
            f2 tu, lo;
            ff_units(f2_mul(half, x), sc, tu, lo);
            lo = f2_fma(f2_fma(y, tt, f2_mul(half, xe)), sc, lo);
            const float2 TU = f2_get(tu), LO = f2_get(ff_units_end(lo));
            double rx = ff_add_units(Y.x, TU.x, LO.x), ry = ff_add_units(Y.y, TU.y, LO.y);
            // next to a power of two the bits of y + v change scale; |e| < 5.6e-7, so that v is at
            // most 5 last places (2^-24 of y below the power)
            const bool ex = !(R2.x > close2 && R2.x < 1e36f) || ff_near_binade<8>(Y.x);
            const bool ey = !(R2.y > close2 && R2.y < 1e36f) || ff_near_binade<8>(Y.y);
            if (ex || ey) {
                if (ex && wx && i < A.n && b * kSymT + jx < A.n) rx = unit * rinv_fp64(A, i, b * kSymT + jx);
                if (ey && wy && i < A.n && b * kSymT + jy < A.n) ry = unit * rinv_fp64(A, i, b * kSymT + jy);
            }
            s0 = fma(mx, rx, s0);
            s1 = fma(my, ry, s1);
        }
        double v, e;
        two_sum(s0, s1, v, e);
        C += e;
        two_sum(S, v, v, e);
        S = v;
        C += e;
    }
    if (row >= 0 && i < A.n) add_row(TS, TC, A.m[i], S, C);
    block_sum2<kEnThreads>(TS, TC, sh);
    if (tid == 0) {
        A.part[blockIdx.x] = TS / unit;
        A.part[kEnBlocks + blockIdx.x] = TC / unit;
    }
}

// Per body: kinetic and star terms, angular momentum and momentum; block sums.
__global__ void __launch_bounds__(kEnThreads)
energy_bodies_kernel(int n, const double *pos, const double *vel, const double *mass, double G, double m_star,
                     double *part /* [9][2][kEnBlocks] */) {
    __shared__ double sh[2 * kEnThreads];
    const size_t N = (size_t)n;
    double S[kEnRows], C[kEnRows];
#pragma unroll
    for (int k = 0; k < kEnRows; k++) S[k] = C[k] = 0.0;
    for (int i = blockIdx.x * kEnThreads + threadIdx.x; i < n; i += kEnThreads * gridDim.x) {
        const double x = pos[i], y = pos[N + i], z = pos[2 * N + i];
        const double vx = vel[i], vy = vel[N + i], vz = vel[2 * N + i], m = mass[i];
        const double r = sqrt(x * x + y * y + z * z);
        const double v[kEnRows - 1] = {0.5 * m * (vx * vx + vy * vy + vz * vz), -G * m_star * m / r,
                                       m * (y * vz - z * vy), m * (z * vx - x * vz), m * (x * vy - y * vx),
                                       m * vx, m * vy, m * vz};
#pragma unroll
        for (int k = 0; k < kEnRows - 1; k++) {
            double s, e;
            two_sum(S[k], v[k], s, e);
            S[k] = s;
            C[k] += e;
        }
    }
#pragma unroll
    for (int k = 0; k < kEnRows - 1; k++) {
        block_sum2<kEnThreads>(S[k], C[k], sh);
        if (threadIdx.x == 0) {
            part[(size_t)k * 2 * kEnBlocks + blockIdx.x] = S[k];
            part[((size_t)k * 2 + 1) * kEnBlocks + blockIdx.x] = C[k];
        }
    }
}

// One block per row of partial sums (8 body rows, then the pairs).
__global__ void __launch_bounds__(kEnThreads)
energy_fold_kernel(const double *part, int nbody, int npair, double *out) {
    __shared__ double sh[2 * kEnThreads];
    const double *p = part + (size_t)blockIdx.x * 2 * kEnBlocks;
    const int n = (int)blockIdx.x == kEnRows - 1 ? npair : nbody;
    double S = 0.0, C = 0.0;
    for (int k = threadIdx.x; k < n; k += kEnThreads) {
        double s, e;
        two_sum(S, p[k], s, e);
        S = s;
        C += e + p[kEnBlocks + k];
    }
    block_sum2<kEnThreads>(S, C, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = isinf(S) ? S : S + C;       // bodies at one place
}

}  // namespace

// E = (kinetic + star + pairs) + |P|^2 / (2 m_star); L as summed.
cudaError_t launch_energy(genga_system *s, double *E_host, double *L_host) {
    const int n = (int)s->n;
    GENGA_CUDA_TRY(ff_reserve(s));
    if (!s->en_part)
        GENGA_CUDA_TRY(cudaMalloc((void **)&s->en_part, sizeof(double) * (kEnRows * 2 * kEnBlocks + kEnRows)));
    FfPack ff = ff_pack_args(s);
    ff.window = kFfWindowNone;
    ff.margin = kFfMargin64;
    GENGA_CUDA_TRY(launch_ff_pack(ff, s->stream, &s->launches));
    EnergyArgs A;
    A.x = s->pos; A.y = s->pos + n; A.z = s->pos + 2 * (size_t)n; A.m = s->mass;
    A.body = ff.body; A.header = ff.header; A.n = n; A.nm = tp_bound(s); A.nT = ff.nT;
    A.part = s->en_part + (size_t)(kEnRows - 1) * 2 * kEnBlocks;
    int per_sm = 0;
    GENGA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, energy_pairs_kernel, kEnThreads, 0));
    const long long tiles = (long long)ff.nT * (ff.nT + 1) / 2;
    const int npair = (int)std::min<long long>(tiles, std::min(kEnBlocks, std::max(1, per_sm) * s->num_sms));
    energy_pairs_kernel<<<npair, kEnThreads, 0, s->stream>>>(A);
    GENGA_CUDA_TRY(cudaGetLastError());
    const int nbody = std::min((n + kEnThreads - 1) / kEnThreads, s->num_sms);
    energy_bodies_kernel<<<nbody, kEnThreads, 0, s->stream>>>(n, s->pos, s->vel, s->mass, s->p.G, s->p.m_star,
                                                              s->en_part);
    GENGA_CUDA_TRY(cudaGetLastError());
    double *out = s->en_part + kEnRows * 2 * kEnBlocks;
    energy_fold_kernel<<<kEnRows, kEnThreads, 0, s->stream>>>(s->en_part, nbody, npair, out);
    GENGA_CUDA_TRY(cudaGetLastError());
    s->launches += 3;
    double h[kEnRows];
    GENGA_CUDA_TRY(cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, s->stream));
    GENGA_CUDA_TRY(cudaStreamSynchronize(s->stream));
    const double P2 = h[5] * h[5] + h[6] * h[6] + h[7] * h[7];
    *E_host = ((h[0] + h[1]) - s->p.G * h[8]) + P2 / (2.0 * s->p.m_star);
    L_host[0] = h[2]; L_host[1] = h[3]; L_host[2] = h[4];
    return cudaSuccess;
}

}  // namespace genga
