// Individual time steps on rungs with the hierarchical kick-drift-kick leapfrog (Sec. 3.2).
//
// Particle i sits on rung r_i with step dt0 / 2^r_i (Sec. 3.2: time steps restricted to
// 2^-l of the base step).  The base step is cut into 2^R substeps of h = dt0 / 2^R; a
// particle is active at substep s when s is a multiple of 2^(R - r_i), i.e. where its
// kicks line up with those of the coarser rungs (Fig. KDK).  At substep s, for active
// particles: closing half kick with the force just computed, rung reassignment from
// Delta T_i = 0.2 sqrt(eps / |a_i|) (Sec. 3.2), opening half kick of the new step; then
// every particle drifts by h.  All of it in FP64.
//
// Rung choice is an integer decided by floating point, made reproducible by avoiding
// log2: r = the smallest r in [0, R] with dt0 <= Delta T * 2^r (scaling by 2^r is exact),
// with |a| = sqrt((ax^2 + ay^2) + az^2) and Delta T computed step by step without fused
// operations.  A particle may move to a coarser rung only at a substep where that rung
// is synchronised.
#include <math.h>

#include "f64bits.cuh"
#include "fmm_internal.cuh"

// The target rung in FP64: the definition.
__device__ __noinline__ int target_rung_f64(float ax, float ay, float az, double eps, double dt0, int R)
{
    double x = ax, y = ay, z = az;
    double a2 = __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
    double am = __dsqrt_rn(a2);
    if (!(am > 0.0)) return 0;
    double dt = __dmul_rn(0.2, __dsqrt_rn(__ddiv_rn(eps, am)));
    int r = 0;
    while (r < R && dt0 > ldexp(dt, r)) r++;
    return r;
}

// The same rung, decided in FP32 where FP32 can decide it.  dt0 <= Delta T 2^r is
// |a|^2 <= t0 16^r with t0 = (0.04 eps / dt0^2)^2 (t0 = 0: outside FP32's range, never decided here).
// The FP32 square is within 3e-7 of the exact one (three squares and two sums, each rounded once;
// the range below keeps lost subnormals far under that), t0's rounding within 6e-8 and the FP64
// definition's own roundings within 1e-14, so a square further than 1e-6 from the thresholds on both
// sides of it has the definition's rung; the others (one particle in about a million) take it.  The
// FP64 square roots and division (FP64 issues at 1/64 of the FP32 rate, and a warp pays in full for one
// active lane) made the kick-drift of a 256^3 box with a tenth active 1.62 ms, 0.8 TB/s; it took
// 0.46 ms, 2.8 TB/s, this way.
__device__ __forceinline__ int target_rung(float ax, float ay, float az, double eps, double dt0, int R, float t0)
{
    if (R == 0) return 0;  // a single rung: nothing to decide
    const float a2 = __fmaf_rn(ax, ax, __fmaf_rn(ay, ay, __fmul_rn(az, az)));
    if (a2 == 0.0f && ax == 0.0f && ay == 0.0f && az == 0.0f) return 0;
    if (t0 > 0.0f && a2 > 1e-30f && a2 < 1e37f) {
        int r = 0;
        float t = t0;
        while (r < R && a2 > t) {
            r++;
            t *= 16.0f;
        }
        const bool above = r == 0 || a2 > 0.0625f * t * 1.000001f, below = r == R || a2 < t * 0.999999f;
        if (above && below) return r;
    }
    return target_rung_f64(ax, ay, az, eps, dt0, R);
}

// t0 of target_rung; 0 where it or its first multiples leave FP32's normal range
static float rung_threshold(double eps, double dt0)
{
    const double q = 0.04 * eps / (dt0 * dt0), t = q * q;
    return t > 1e-36 && t < 1e36 ? (float)t : 0.0f;
}

__global__ void k_assign_rungs(const float* __restrict__ acc, unsigned char* __restrict__ rung, long long n,
                               double eps, double dt0, int R, float t0)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rung[i] = (unsigned char)target_rung(acc[i], acc[n + i], acc[2 * n + i], eps, dt0, R, t0);
}

// dt0 2^-k as ldexp gives it, by one exact multiplication with the power of two built from its bits
__device__ __forceinline__ double pow2_scale(double dt0, int k)
{
    return __dmul_rn(dt0, fmm_dfrom((unsigned long long)(1023 - k) << 52));
}

// FP64 issues at 1/64 of the FP32 rate on this GPU: the kicks and the drift are FP64 arithmetic, while
// the widening of the FP32 accelerations and the box check of the new position use the encodings
// (f64bits.cuh) and give the same values.
//
// A warp pays for an FP64 instruction in full however few of its lanes are active, and on a substep
// nearly every warp holds some of the active tenth.  So a block gathers its active particles in shared
// memory and kicks them with as few warps as hold them; the drift, of every particle, follows.  256^3 box,
// a tenth active: 0.353 ms, 4.2 TB/s, against 0.465 with every particle kicked in its own lane (6 blocks per
// SM; 0.39 with 5, 0.41 with 4).  Neither pipe alone bounds it: FP64 is busy for 62% of the time and DRAM for
// 57%, and the warps wait at the barriers, most of all for the accelerations, which are loaded behind one.
#define KD_THREADS 256
__global__ void __launch_bounds__(KD_THREADS, 6) k_kick_drift(
    double* __restrict__ pos, double* __restrict__ vel, const float* __restrict__ acc, unsigned char* __restrict__ rung,
    unsigned char* __restrict__ active_next, long long n, double eps, double dt0, int R, float t0, long long s, int closing,
    unsigned int* __restrict__ status)
{
    __shared__ double v[3][KD_THREADS];
    __shared__ unsigned char rs[KD_THREADS], list[KD_THREADS];
    __shared__ int count;
    const int tid = threadIdx.x;
    const long long first = (long long)blockIdx.x * KD_THREADS, i = first + tid;
    const bool valid = i < n;
    if (tid == 0) count = 0;
    int r = 0;
    double vx = 0.0, vy = 0.0, vz = 0.0, x = 0.0, y = 0.0, z = 0.0;
    if (valid) {
        r = rung[i];
        vx = vel[i];
        vy = vel[n + i];
        vz = vel[2 * n + i];
        x = pos[i];
        y = pos[n + i];
        z = pos[2 * n + i];
    }
    const bool active = valid && (s & ((1LL << (R - r)) - 1)) == 0;
    __syncthreads();
    const unsigned int m = __ballot_sync(FMM_FULL_MASK, active);
    int at = 0;
    if ((tid & 31) == 0 && m) at = atomicAdd(&count, __popc(m));
    at = __shfl_sync(FMM_FULL_MASK, at, 0) + __popc(m & fmm_lanemask_lt());
    if (active) {
        list[at] = (unsigned char)tid;
        rs[tid] = (unsigned char)r;
        v[0][tid] = vx;
        v[1][tid] = vy;
        v[2][tid] = vz;
    }
    __syncthreads();
    if (tid < count) {
        const int q = list[tid], ro = rs[q];
        const long long j = first + q;
        double wx = v[0][q], wy = v[1][q], wz = v[2][q];
        const float fx = acc[j], fy = acc[n + j], fz = acc[2 * n + j];
        const double ax = fmm_f2d(fx), ay = fmm_f2d(fy), az = fmm_f2d(fz);
        if (closing) {
            const double hk = pow2_scale(dt0, ro + 1);
            wx += ax * hk;
            wy += ay * hk;
            wz += az * hk;
        }
        int rn = target_rung(fx, fy, fz, eps, dt0, R, t0);
        while (rn < ro && (s & ((1LL << (R - rn)) - 1)) != 0) rn++;
        const double hk = pow2_scale(dt0, rn + 1);
        wx += ax * hk;
        wy += ay * hk;
        wz += az * hk;
        v[0][q] = wx;
        v[1][q] = wy;
        v[2][q] = wz;
        rs[q] = (unsigned char)rn;
    }
    __syncthreads();
    if (!valid) return;
    if (active) {
        r = rs[tid];
        rung[i] = (unsigned char)r;
        vel[i] = vx = v[0][tid];
        vel[n + i] = vy = v[1][tid];
        vel[2 * n + i] = vz = v[2][tid];
    }
    const double h = pow2_scale(dt0, R);
    x += vx * h;
    y += vy * h;
    z += vz * h;
    if (!(fmm_in_unit(x) && fmm_in_unit(y) && fmm_in_unit(z))) atomicOr(status, FMM_DEV_ERR_ARG);
    pos[i] = x;
    pos[n + i] = y;
    pos[2 * n + i] = z;
    long long s1 = s + 1;
    active_next[i] = ((s1 & ((1LL << (R - r)) - 1)) == 0) ? 1 : 0;
}

// The same with a single rung (the ordinary time step): substep 0 alone, every particle active and on rung 0 from here
// on, so there is nothing to gather or to decide.  The gathering kernel's barriers and shared memory cost it
// 8.5 us against 7.1 on 100,000 particles, 64.4 against 62.2 on 2 million and 570 against 561 on 20 million.
template <bool CLOSING>
__global__ void __launch_bounds__(KD_THREADS) k_kick_drift_single(double* __restrict__ pos, double* __restrict__ vel,
                                                                  const float* __restrict__ acc,
                                                                  unsigned char* __restrict__ rung,
                                                                  unsigned char* __restrict__ active_next, long long n,
                                                                  double dt0, double hk, unsigned int* __restrict__ status)
{
    const long long i = (long long)blockIdx.x * KD_THREADS + threadIdx.x;
    if (i >= n) return;
    double x[3], hc = hk;  // the closing half step is that of the rung so far
    if (CLOSING) {
        const int r = rung[i];
        if (r != 0) hc = pow2_scale(dt0, r + 1);
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const double f = fmm_f2d(acc[a * n + i]);
        double v = vel[a * n + i];
        if (CLOSING) v += f * hc;
        v += f * hk;
        vel[a * n + i] = v;
        x[a] = pos[a * n + i] + v * dt0;
        pos[a * n + i] = x[a];
    }
    if (!(fmm_in_unit(x[0]) && fmm_in_unit(x[1]) && fmm_in_unit(x[2]))) atomicOr(status, FMM_DEV_ERR_ARG);
    rung[i] = 0;
    active_next[i] = 1;
}

cudaError_t fmm_launch_kick_drift(double* pos, double* vel, const float* acc, unsigned char* rung,
                                  unsigned char* active_next, long long n, double eps, double dt0, int max_rung,
                                  int substep, int closing, DevCounters* ctr, cudaStream_t s)
{
    const unsigned blocks = (unsigned)fmm_ceil_div(n, KD_THREADS);
    const auto single = closing ? k_kick_drift_single<true> : k_kick_drift_single<false>;
    if (max_rung == 0)
        single<<<blocks, KD_THREADS, 0, s>>>(pos, vel, acc, rung, active_next, n, dt0, 0.5 * dt0, &ctr->status);
    else
        k_kick_drift<<<blocks, KD_THREADS, 0, s>>>(pos, vel, acc, rung, active_next, n, eps, dt0, max_rung,
                                                   rung_threshold(eps, dt0), substep, closing, &ctr->status);
    return cudaGetLastError();
}

// The same schedule on compressed storage (Sec. 3.4, memory): positions as 32-bit fixed-point
// coordinates x = u 2^-32 of the unit box, velocities as FP32.  Within a substep the kicks are FP64
// (v = fl64(v32), v += a hk for each half kick, each product and sum rounded once: no fused
// operations), and the velocity is stored rounded to FP32.  The drift moves u by the nearest integer
// of v32 h 2^32, computed in FP64 (x 2^32 is exact), ties to even.  In the periodic box (periodic != 0)
// u wraps modulo 2^32, which is the box's periodicity; in the isolated box a particle leaving
// [0, 1) sets the argument error bit and keeps its old position.
__global__ void k_kick_drift_i32(unsigned int* __restrict__ ipos, float* __restrict__ vel,
                                 const float* __restrict__ acc, unsigned char* __restrict__ rung,
                                 unsigned char* __restrict__ active_next, long long n, double eps, double dt0, int R,
                                 float t0, long long s, int closing, int periodic, unsigned int* __restrict__ status)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int r = rung[i];
    float v32[3] = {vel[i], vel[n + i], vel[2 * n + i]};
    if ((s & ((1LL << (R - r)) - 1)) == 0) {
        const float f[3] = {acc[i], acc[n + i], acc[2 * n + i]};
        double v[3] = {fmm_f2d(v32[0]), fmm_f2d(v32[1]), fmm_f2d(v32[2])};
        if (closing) {
            const double hk = pow2_scale(dt0, r + 1);
            for (int a = 0; a < 3; a++) v[a] = __dadd_rn(v[a], __dmul_rn(fmm_f2d(f[a]), hk));
        }
        int rt = target_rung(f[0], f[1], f[2], eps, dt0, R, t0);
        int rn = rt;
        if (rt < r) {
            rn = rt;
            while (rn < r && (s & ((1LL << (R - rn)) - 1)) != 0) rn++;
        }
        r = rn;
        rung[i] = (unsigned char)r;
        const double hk = pow2_scale(dt0, r + 1);
        for (int a = 0; a < 3; a++) {
            v[a] = __dadd_rn(v[a], __dmul_rn(fmm_f2d(f[a]), hk));
            v32[a] = fmm_d2f_rn(v[a]);
            vel[a * n + i] = v32[a];
        }
    }
    const double h = pow2_scale(dt0, R);
    long long u[3];
    bool out = false;
    for (int a = 0; a < 3; a++) {
        const long long d = __double2ll_rn(__dmul_rn(__dmul_rn(fmm_f2d(v32[a]), h), 4294967296.0));
        u[a] = (long long)ipos[a * n + i] + d;
        if (periodic) u[a] &= 0xffffffffLL;
        else if (u[a] < 0 || u[a] > 0xffffffffLL) out = true;
    }
    if (out) {
        atomicOr(status, FMM_DEV_ERR_ARG);
    } else {
        for (int a = 0; a < 3; a++) ipos[a * n + i] = (unsigned int)u[a];
    }
    long long s1 = s + 1;
    active_next[i] = ((s1 & ((1LL << (R - r)) - 1)) == 0) ? 1 : 0;
}

cudaError_t fmm_launch_kick_drift_i32(unsigned int* ipos, float* vel, const float* acc, unsigned char* rung,
                                      unsigned char* active_next, long long n, double eps, double dt0, int max_rung,
                                      int substep, int closing, int periodic, DevCounters* ctr, cudaStream_t s)
{
    k_kick_drift_i32<<<(unsigned)fmm_ceil_div(n, 256), 256, 0, s>>>(ipos, vel, acc, rung, active_next, n, eps, dt0,
                                                                    max_rung, rung_threshold(eps, dt0), substep, closing,
                                                                    periodic, &ctr->kdk_status);
    return cudaGetLastError();
}

cudaError_t fmm_launch_assign_rungs(const float* acc, unsigned char* rung, long long n, double eps, double dt0,
                                    int max_rung, cudaStream_t s)
{
    k_assign_rungs<<<(unsigned)fmm_ceil_div(n, 256), 256, 0, s>>>(acc, rung, n, eps, dt0, max_rung,
                                                                  rung_threshold(eps, dt0));
    return cudaGetLastError();
}
