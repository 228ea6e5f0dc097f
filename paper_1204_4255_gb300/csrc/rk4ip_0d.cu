// rk4ip_0d.cu -- RK4IP for zero-dimensional problems (ordinary SDEs), one thread per path.
//
// XMDS2 (arXiv:1204.4255) Sec. 2.5: fixed-step RK4 for Wiener-driven SDEs in
// Stratonovich form, many independent paths; Sec. 2.6: with no transverse
// dimension the interaction-picture factor exp(L dt/2) is the scalar exp(c0 dt/2).
// The state lives in registers for the whole run; a Philox draw per step.
//
// What bounds it: the chain of a step (a path's steps follow one another) with few
// warps to hide it -- 65536 paths are 13.5 warps an SM -- and the draw's ~150
// instructions.  The draws do not depend on the state, so kAhead steps' draws are
// made together, independent chains between two runs of dependent steps; the noise
// kind is a template argument (real noise takes the cosine alone); samples are found
// by a countdown (a 64-bit remainder a step cost as much as the step); and a block
// is two warps, so that the paths spread evenly over the SMs.  65536 paths x 1000
// steps, complex64, sampled every 100: 750 -> 471 us.
#include "kernels.h"

namespace xsde {
namespace {

constexpr int kThreads0D = 64;
constexpr int kAhead = 4;

// FINE: the problem has noise substeps
template <typename R, int NOISE, bool FINE> __global__ void __launch_bounds__(kThreads0D) rk4ip_0d_kernel(const Params0D<R> p) {
    using V = cx<R>;
    __shared__ double red[2][kThreads0D / 32];
    const int64_t lp = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = lp < p.npaths;
    const uint32_t gp = (uint32_t)(p.lt.path_offset + lp);
    V z = (active && XSDE_IN(lp, p.npaths, p.status)) ? p.psi[lp] : mk<V>(R(0), R(0));
    const V E = p.Ehalf;
    const R gdt = p.lt.gdt;
    const R sixth = R(1) / R(6), third = R(1) / R(3), half = R(0.5);
    const int idx0[3] = {0, 0, 0};
    const bool vtime = p.lt.pot == PM_TABLE && p.lt.V_nt > 1;
    const R Vstatic = vtime ? R(0) : potential(p.lt, 0, idx0, 0, 0);

    auto sample = [&](int64_t s, int64_t n) {
        const double m2 = active ? (double)cabs2(z) : 0.0;
        if (active) {
            const double v = (double)potential(p.lt, 0, idx0, 0, p.step0 + n);
            if ((p.sm.which & (MOM_NORM | MOM_ENERGY)) && p.sm.per_path &&
                XSDE_IN(s * p.npaths + lp, p.sm.nsamp * p.npaths, p.status)) {
                double *pq = p.sm.per_path + 2 * (s * p.npaths + lp);
                pq[0] = m2;
                pq[1] = (p.sm.h0 + v) * m2 + 0.5 * p.sm.g * m2 * m2;
            }
            if (!isfinite(m2)) atomicOr(p.status, ST_NONFINITE);
        }
        if ((p.sm.which & (MOM_MOD2 | MOM_MOD4)) && p.sm.per_point && XSDE_IN(s, p.sm.nsamp, p.status)) {
            double a = warp_sum(m2), b = warp_sum(m2 * m2);
            if ((threadIdx.x & 31) == 0) {
                red[0][threadIdx.x >> 5] = a;
                red[1][threadIdx.x >> 5] = b;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                double sa = 0.0, sb = 0.0;
                for (int w = 0; w < kThreads0D / 32; ++w) {
                    sa += red[0][w];
                    sb += red[1][w];
                }
                atomicAdd(p.sm.per_point + 2 * s, sa * p.sm.inv_paths);
                atomicAdd(p.sm.per_point + 2 * s + 1, sb * p.sm.inv_paths);
            }
            __syncthreads();
        }
    };
    auto step = [&](uint64_t sg, V xi) {
        const R v = vtime ? (XSDE_IN(sg, p.lt.V_nt, p.status) ? p.lt.V[sg] : R(0)) : Vstatic;
        const PointTerm<R> pt = point_term<NOISE>(p.lt, v, xi);
        const V aI = cmul(E, z);
        if (p.scheme == 1) {
            // semi-implicit midpoint: a_I = D a; m <- a_I + N(m)/2 (three times); a <- D(2m - a_I)
            V m = aI;
            for (int it = 0; it < 3; ++it) m = caxpy(aI, half, apply_N(m, pt, gdt));
            z = cmul(E, mk<V>(R(2) * m.x - aI.x, R(2) * m.y - aI.y));
            return;
        }
        // a_I = D a, k1 = D N(a), k2, k3, k4 = N(D(a_I + k3)), a <- D(acc) + k4/6
        const V k1 = cmul(E, apply_N(z, pt, gdt));
        const V k2 = apply_N(caxpy(aI, half, k1), pt, gdt);
        const V k3 = apply_N(caxpy(aI, half, k2), pt, gdt);
        const V k4 = apply_N(cmul(E, cadd(aI, k3)), pt, gdt);
        const V acc = caxpy(caxpy(caxpy(aI, sixth, k1), third, k2), third, k3);
        z = caxpy(cmul(E, acc), sixth, k4);
    };

    auto noise = [&](int64_t n) -> V {
        const uint32_t sg = (uint32_t)(p.step0 + n);
        if constexpr (NOISE == NM_NONE) return mk<V>(R(0), R(0));
        else if constexpr (FINE) return scaled_normals<R, NOISE == NM_ADD_COMPLEX>(p.lt, 0u, gp, sg);
        else return cscale(wiener_pair<R, NOISE == NM_ADD_COMPLEX>(p.lt.key, 0u, gp, sg), p.lt.nscale);
    };
    int64_t s = 0;
    for (int64_t n = 0;;) {
        // sample at n, then run to the next sample (or the end)
        if (p.sm.every > 0 && n == s * p.sm.every) sample(s++, n);
        if (n == p.nsteps) break;
        int64_t stop = p.nsteps;
        if (p.sm.every > 0 && s * p.sm.every < stop) stop = s * p.sm.every;
        for (; n + kAhead <= stop; n += kAhead) {
            V xi[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) xi[i] = noise(n + i);
#pragma unroll
            for (int i = 0; i < kAhead; ++i) step(p.step0 + n + i, xi[i]);
        }
        for (; n < stop; ++n) step(p.step0 + n, noise(n));
    }
    if (active && XSDE_IN(lp, p.npaths, p.status)) p.psi[lp] = z;
}

}  // namespace

template <typename R, int NOISE> static cudaError_t launch_0d_noise(const Params0D<R> &p, cudaStream_t s) {
    const unsigned blocks = (unsigned)((p.npaths + kThreads0D - 1) / kThreads0D);
    if (NOISE != NM_NONE && p.lt.substeps > 1) rk4ip_0d_kernel<R, NOISE, true><<<blocks, kThreads0D, 0, s>>>(p);
    else rk4ip_0d_kernel<R, NOISE, false><<<blocks, kThreads0D, 0, s>>>(p);
    return cudaGetLastError();
}

template <typename R> cudaError_t launch_rk4ip_0d(const Params0D<R> &p, cudaStream_t s) {
    switch (p.lt.noise) {
        case NM_ADD_REAL: return launch_0d_noise<R, NM_ADD_REAL>(p, s);
        case NM_ADD_COMPLEX: return launch_0d_noise<R, NM_ADD_COMPLEX>(p, s);
        case NM_MUL_REAL: return launch_0d_noise<R, NM_MUL_REAL>(p, s);
        default: return launch_0d_noise<R, NM_NONE>(p, s);
    }
}

template cudaError_t launch_rk4ip_0d<float>(const Params0D<float> &, cudaStream_t);
template cudaError_t launch_rk4ip_0d<double>(const Params0D<double> &, cudaStream_t);

}  // namespace xsde
