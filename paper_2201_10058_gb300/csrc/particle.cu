// particle.cu -- per-body kernels of the hybrid step (Appendix A): Rcrit
// (Eq. rcrit), HC (Eq. Hc), FG (Kepler part of Eq. Ha) with the pre-drift copy,
// and the level restore of the higher-level scheme (Sec. 6.3).
//
// These kernels are memory/latency bound (a few hundred bytes per body); they
// use one thread per body, coalesced SoA loads and no shared memory.  FG runs
// its Newton iteration per thread; its Stumpff functions need no
// transcendental calls (series + argument quartering).
#include <algorithm>

#include "common.cuh"

namespace genga {
namespace {

// ---------------------------------------------------------------- Rcrit
// rc_i = max(n1 R_H,i, n2 dt |v_i|), R_H,i = |x_i| (m_i/(3 m_star))^(1/3).
// |x| and |v| use the detection operation order (no contraction) so that the
// thresholds compare bit-for-bit with a plain CPU evaluation.
__device__ __forceinline__ void derive_thresholds(double rc, double f_pc, double *rc2, double *pc2,
                                                  float *thr_rc, double *irc) {
    *irc = __ddiv_rn(1.0, rc);
    const double r2 = __dmul_rn(rc, rc);
    const double t = __dmul_rn(f_pc, rc);
    const double p2 = __dmul_rn(t, t);
    *rc2 = r2;
    if (pc2) *pc2 = p2;
    // conservative FP32 upper bound (rounded up, + 2^-16)
    if (thr_rc) *thr_rc = fmaxf(__double2float_ru(r2) * 1.0000153f, 1.17549435e-38f);
}

__global__ void rcrit_kernel(int n, const double *pos, const double *vel, const double *mass,
                             double m_star, double dt, double n1, double n2, double f_pc,
                             RcritArrays out, const int *bodies, int nb, DevCounters *ctr) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    const int i = bodies ? bodies[k] : k;
    const double x = pos[i], y = pos[(size_t)n + i], z = pos[2 * (size_t)n + i];
    const double vx = vel[i], vy = vel[(size_t)n + i], vz = vel[2 * (size_t)n + i];
    const double r = sqrt(dist2_rn(x, y, z));
    const double vabs = sqrt(dist2_rn(vx, vy, vz));
    if (!(r > 0.0) || !isfinite(r) || !isfinite(vabs)) latch_error(ctr, kErrBadState);
    const double hill = __dmul_rn(r, cbrt(__ddiv_rn(mass[i], __dmul_rn(3.0, m_star))));
    const double a = __dmul_rn(n1, hill);
    const double b = __dmul_rn(__dmul_rn(n2, dt), vabs);
    const double rc = a > b ? a : b;
    out.rc[i] = rc;
    derive_thresholds(rc, f_pc, &out.rc2[i], out.pc2 ? &out.pc2[i] : nullptr,
                      out.thr_rc ? &out.thr_rc[i] : nullptr, &out.irc[i]);
}

__global__ void rcrit_derive_kernel(int n, double f_pc, RcritArrays a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    derive_thresholds(a.rc[i], f_pc, &a.rc2[i], &a.pc2[i], &a.thr_rc[i], &a.irc[i]);
}

// ---------------------------------------------------------------- HC
// P = sum_j m_j v_j in a fixed order (strided per-thread sums, then a fixed
// tree), shift = dt_half P / m_star; then x_i += shift.
constexpr int kHcThreads = 256;

// P = sum_j m_j v_j in a fixed order: each block sums a contiguous range of
// bodies (strided per-thread sums, then a fixed tree), and the last block to
// finish adds the block sums in block order; shift = dt_half P / m_star.  One
// launch over every SM (a single block was bound by one SM's FP64 rate).
__global__ void __launch_bounds__(kHcThreads)
hc_reduce_kernel(int n, const double *vel, const double *mass, double m_star, double dt_half,
                 double *part, DevCounters *ctr) {
    __shared__ double sp[3][kHcThreads];
    __shared__ bool last;
    const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
    const int j0 = (int)blockIdx.x * per, j1 = min(n, j0 + per);
    double p0 = 0.0, p1 = 0.0, p2 = 0.0;
    for (int j = j0 + (int)threadIdx.x; j < j1; j += kHcThreads) {
        const double mj = mass[j];
        p0 += mj * vel[j];
        p1 += mj * vel[(size_t)n + j];
        p2 += mj * vel[2 * (size_t)n + j];
    }
    sp[0][threadIdx.x] = p0; sp[1][threadIdx.x] = p1; sp[2][threadIdx.x] = p2;
    __syncthreads();
    for (int w = kHcThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            sp[0][threadIdx.x] += sp[0][threadIdx.x + w];
            sp[1][threadIdx.x] += sp[1][threadIdx.x + w];
            sp[2][threadIdx.x] += sp[2][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x < 3) part[3 * blockIdx.x + threadIdx.x] = sp[threadIdx.x][0];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctr->hc_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x < 3) {
        const volatile double *vp = part;
        double sum = 0.0;
        for (unsigned q = 0; q < gridDim.x; q++) sum += vp[3 * q + threadIdx.x];
        ctr->hc_shift[threadIdx.x] = dt_half * sum / m_star;
    }
    if (threadIdx.x == 0) ctr->hc_done = 0;
}

__global__ void hc_apply_kernel(int n, double *pos, const DevCounters *ctr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    pos[i] += ctr->hc_shift[0];
    pos[(size_t)n + i] += ctr->hc_shift[1];
    pos[2 * (size_t)n + i] += ctr->hc_shift[2];
}

// ---------------------------------------------------------------- FG
// kepler_drift() and stumpff() live in common.cuh (shared with the ensemble).

__global__ void drift_kernel(int n, double *pos, double *vel, double *pre_pos, double *pre_vel,
                             double mu, double dt, int max_iter, const int *bodies, int nb,
                             DevCounters *ctr) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    const int i = bodies ? bodies[k] : k;
    const size_t N = (size_t)n;
    double x = pos[i], y = pos[N + i], z = pos[2 * N + i];
    double vx = vel[i], vy = vel[N + i], vz = vel[2 * N + i];
    if (pre_pos) {
        pre_pos[i] = x; pre_pos[N + i] = y; pre_pos[2 * N + i] = z;
        pre_vel[i] = vx; pre_vel[N + i] = vy; pre_vel[2 * N + i] = vz;
    }
    if (!kepler_drift(x, y, z, vx, vy, vz, mu, dt, max_iter)) {
        latch_error(ctr, kErrKepler);
        atomicAdd(&ctr->kepler_fail, 1ull);
    }
    if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(vx) && isfinite(vy) && isfinite(vz)))
        latch_error(ctr, kErrBadState);
    pos[i] = x; pos[N + i] = y; pos[2 * N + i] = z;
    vel[i] = vx; vel[N + i] = vy; vel[2 * N + i] = vz;
}

__global__ void restore_kernel(int n, double *pos, double *vel, const double *pre_pos,
                               const double *pre_vel, const int *bodies, int nb) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    const int i = bodies[k];
    const size_t N = (size_t)n;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        pos[c * N + i] = pre_pos[c * N + i];
        vel[c * N + i] = pre_vel[c * N + i];
    }
}

}  // namespace

cudaError_t launch_rcrit(genga_system *s, int level, double dt, const int *bodies, int nb) {
    if (nb <= 0) return cudaSuccess;
    RcritArrays out = s->rcl[level];
    if (level > 0) { out.pc2 = nullptr; out.thr_rc = nullptr; }
    rcrit_kernel<<<(nb + 255) / 256, 256, 0, s->stream>>>((int)s->n, s->pos, s->vel, s->mass,
        s->p.m_star, dt, s->p.n1, s->p.n2, s->p.f_pc, out, bodies, nb, s->ctr); ++s->launches;
    return cudaGetLastError();
}

cudaError_t launch_rcrit_derive(genga_system *s) {
    const int n = (int)s->n;
    rcrit_derive_kernel<<<(n + 255) / 256, 256, 0, s->stream>>>(n, s->p.f_pc, s->rcl[0]); ++s->launches;
    return cudaGetLastError();
}

cudaError_t launch_hc(genga_system *s, double dt_half) {
    const int n = (int)s->n;
    const int nblk = std::max(1, std::min(s->num_sms, (n + kHcThreads - 1) / kHcThreads));
    hc_reduce_kernel<<<nblk, kHcThreads, 0, s->stream>>>(n, s->vel, s->mass, s->p.m_star, dt_half, s->red,
                                                        s->ctr); ++s->launches;
    GENGA_CUDA_TRY(cudaGetLastError());
    hc_apply_kernel<<<(n + 255) / 256, 256, 0, s->stream>>>(n, s->pos, s->ctr); ++s->launches;
    return cudaGetLastError();
}

cudaError_t launch_drift(genga_system *s, int level, double dt, const int *bodies, int nb) {
    if (nb <= 0) return cudaSuccess;
    drift_kernel<<<(nb + 127) / 128, 128, 0, s->stream>>>((int)s->n, s->pos, s->vel,
        s->pre_pos[level], s->pre_vel[level], s->p.G * s->p.m_star, dt, s->p.kepler_max_iter,
        bodies, nb, s->ctr); ++s->launches;
    return cudaGetLastError();
}

cudaError_t launch_restore(genga_system *s, int from_level, const int *bodies, int nb) {
    if (nb <= 0) return cudaSuccess;
    restore_kernel<<<(nb + 255) / 256, 256, 0, s->stream>>>((int)s->n, s->pos, s->vel,
        s->pre_pos[from_level], s->pre_vel[from_level], bodies, nb); ++s->launches;
    return cudaGetLastError();
}

}  // namespace genga
