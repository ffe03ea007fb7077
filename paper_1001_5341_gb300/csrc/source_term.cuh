// source_term.cuh -- the moving shower's current on one Ez edge.
//
// The increment on edge (i, j, k+1/2) is amp_k(n) w_ij with amp_k(n) = qbar
// coef dC_k, the same for every edge of a plane.  All of it is FP64, as the
// integer node index floor(z/dx) must be decided in the same precision as the
// reference arithmetic, and GB300 issues FP64 at 1/64 of the FP32 rate: with
// the two or more divisions of amp_k done per edge, the one block of a launch
// that holds the shower ran 25 us longer than the others, which was 40 % of a
// whole step on a 96^3 grid.  So the few amplitudes of a step are computed
// once (by the host per launch, by one warp per work item in the batch
// kernel) and an edge costs one FP64 product.
#pragma once

#include "fdtd_internal.h"

namespace fdtd {

// E increment per unit lateral weight on the Ez edges of plane k during step
// n, from the charge carried across them (0 on planes without current); q: the
// charge table where the caller can read it.
__host__ __device__ inline double source_amp(const Source &s, const double *q, int k, long long n) {
    if (k < s.kmin || k > s.kmax) return 0.0;
    double za = s.z0 + s.v * (double)n * s.dt;
    double zb = s.z0 + s.v * (double)(n + 1) * s.dt;
    // C_k(z): fraction of the charge on nodes <= k of the untruncated CIC line
    double ua = za / s.dx, ub = zb / s.dx;
    double ka = floor(ua), kb = floor(ub);
    double ca = (double)k < ka ? 0.0 : ((double)k == ka ? 1.0 - (ua - ka) : 1.0);
    double cb = (double)k < kb ? 0.0 : ((double)k == kb ? 1.0 - (ub - kb) : 1.0);
    double dC = cb - ca;
    if (dC == 0.0) return 0.0;
    double zm = s.z0 + s.v * ((double)n + 0.5) * s.dt;
    double u = (zm - s.z0) / s.bin_dz;
    if (!(u >= 0.0) || u > (double)(s.nbins - 1)) return 0.0;
    int b = (int)floor(u);
    double qbar = b >= s.nbins - 1 ? q[s.nbins - 1] : q[b] * (1.0 - (u - b)) + q[b + 1] * (u - b);
    // -(dt/eps) J with J = -(dx/dt) qbar w dC / dx^3
    return qbar * s.coef * dC;
}

// A conservative window [klo, khi] of planes around the charge's path in step
// n, without amplitudes (tab = 0).
__host__ __device__ inline SourceStep source_window(const Source &s, long long n) {
    SourceStep w;
    w.n = n;
    w.klo = 1;
    w.khi = 0;  // empty
    w.kb = w.tab = 0;
    if (!s.active) return w;
    double za = s.z0 + s.v * (double)n * s.dt, zb = s.z0 + s.v * (double)(n + 1) * s.dt;
    double lo = za < zb ? za : zb, hi = za < zb ? zb : za;
    double klo = floor(lo / s.dx) - 2.0, khi = floor(hi / s.dx) + 2.0;
    if (khi < (double)s.kmin || klo > (double)s.kmax) return w;
    w.klo = klo < (double)s.kmin ? s.kmin : (int)klo;
    w.khi = khi > (double)s.kmax ? s.kmax : (int)khi;
    return w;
}

// The source of step n with its amplitudes, on the host (q: host table).  A
// window of more than SRC_PLANES planes (a charge that crosses several cells
// per step) keeps tab = 0, and every edge evaluates source_amp itself.
inline SourceStep source_step(const Source &s, const double *q, long long n) {
    SourceStep w = source_window(s, n);
    if (w.klo > w.khi || w.khi - w.klo >= SRC_PLANES) return w;
    w.kb = w.klo;
    w.tab = 1;
    int first = w.khi + 1, last = w.klo - 1;
    for (int k = w.klo; k <= w.khi; ++k) {
        const double a = source_amp(s, q, k, n);
        w.amp[k - w.kb] = a;
        if (a != 0.0) {
            if (first > k) first = k;
            last = k;
        }
    }
    w.klo = first;   // empty where every amplitude is zero
    w.khi = last;
    return w;
}

// The same by one warp into shared memory (32 lanes, one plane each).
__device__ __forceinline__ void source_step_warp(const Source &s, long long n, SourceStep *out) {
    const int lane = threadIdx.x & 31;
    const SourceStep w = source_window(s, n);
    const bool tab = w.klo <= w.khi && w.khi - w.klo < SRC_PLANES;
    const double a = tab && w.klo + lane <= w.khi ? source_amp(s, s.q, w.klo + lane, n) : 0.0;
    const unsigned nz = __ballot_sync(0xffffffffu, a != 0.0);
    if (lane < SRC_PLANES) out->amp[lane] = a;
    if (lane == 0) {
        out->n = n;
        out->kb = w.klo;
        out->tab = tab;
        out->klo = !tab ? w.klo : nz ? w.klo + __ffs(nz) - 1 : 1;
        out->khi = !tab ? w.khi : nz ? w.klo + 31 - __clz(nz) : 0;
    }
}

__device__ __forceinline__ float source_at(const Source &s, const SourceStep &w, int i, int j, int k) {
    if (k < w.klo || k > w.khi) return 0.0f;
    const int di = i - s.ic, dj = j - s.jc;
    if (di < -s.L || di > s.L || dj < -s.L || dj > s.L) return 0.0f;
    const double a = w.tab ? w.amp[k - w.kb] : source_amp(s, s.q, k, w.n);
    return (float)(a * s.w[(dj + s.L) * (2 * s.L + 1) + (di + s.L)]);
}

}  // namespace fdtd
