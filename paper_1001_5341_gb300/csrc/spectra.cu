// Spectra of detector traces (Sec. V): E_omega(f) = dt sum_m g_m x_{first+m}
// exp(i 2 pi f t_{first+m}), t_n = t0 + n dt, the time factor of eq. GreenMethod.
//
// The phase of (frequency, sample) is the same for every trace, so a block
// takes TB traces (4 or 8) and up to 128 frequencies, one per thread: a
// phase factor costs about ten instructions and is then used TB times, one
// packed multiply-add (two traces) for the real and one for the imaginary
// part.  Bound: instruction issue and its latencies, about four instructions
// a term; with one trace per block and sincospif for every term (40
// instructions a term) the 64 x 8204 samples x 1024 frequencies of the largest
// 2D run took 572 us, now 146 us.
//
// Phase factors.  A phase is the fraction of a cycle in 64-bit fixed point,
// so no rounding builds up along the trace.  Every eighth sample's factor is
// computed from its phase (sincospif of the top 24 bits, the next bits as a
// first-order correction); the others are that factor times the thread's fixed
// rotations e^{i 2 pi f 16 j dt}, one complex product.  A rotation's rounding
// error would enter every eighth sample alike, so its modulus is put right by
// one more multiply-add (without it the sums are 25 % further off).
//
// Sums.  Each block weights and tapers a tile of samples of its traces into
// shared memory (zero outside a trace's gate), the next tile's samples loaded
// meanwhile.  A thread sums eight samples (16 apart) in float32 and adds that
// to a two-float (hi, lo) total: as near the exact sum as the float64 totals of
// 32 strided samples before (32 to a sum here: twice as far off).  The totals
// are added in float64.  Where the frequencies are fewer than 128 the threads
// also split the samples, and where the blocks would not fill the GPU a cluster of up to eight blocks splits them further: the blocks
// of a cluster add their totals through distributed shared memory, so nothing
// is allocated and the order of every sum is fixed.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "f32x2.cuh"
#include "spectra.h"

namespace {

using namespace fdtd::px2;   // a pair holds two traces

constexpr int SPEC_THREADS = 128;
constexpr int SPEC_TILE = 128;        // samples staged at a time
constexpr int SPEC_RUN = 8;           // samples per exact phase factor
constexpr int SPEC_SUM = 8;           // of them per float32 sum
constexpr int SPEC_STRIDE = SPEC_TILE / SPEC_RUN;   // samples between them
constexpr int SPEC_MAX_COMP = 4;
constexpr int SPEC_MAX_SPLIT = 8;     // blocks of a cluster (the portable size)
constexpr int SPEC_MIN_TF = 8;        // fewest frequency lanes
static_assert(SPEC_RUN % SPEC_SUM == 0, "whole float32 sums");
static_assert(SPEC_THREADS == SPEC_TILE, "a thread stages one sample of every trace");
static_assert(SPEC_THREADS / SPEC_MIN_TF <= SPEC_STRIDE, "a sample lane takes every ts-th of a tile's runs");

struct TraceParam {
    float a[SPEC_MAX_COMP];           // component weights
    int first, count;                 // gate
};

struct FreqParam {
    unsigned long long a, b;          // cycles of f t0 and of f dt, fraction x 2^64
};

// Parameters that travel with the launch (the trace table, then the frequency
// table), so that a call of ordinary size needs no device allocation or copy.
template <int N>
struct Blob {
    alignas(16) unsigned char b[N];
};
constexpr int SPEC_SMALL = 3072, SPEC_LARGE = 30720;   // a launch carries up to 32764 bytes

// Fraction of x in [0, 1) as a 64-bit fixed-point number.
unsigned long long fixed_fraction(double x) {
    double fr = x - std::floor(x);
    if (!(fr >= 0.0 && fr < 1.0)) fr = 0.0;
    return (unsigned long long)std::ldexp(fr, 64);
}

// e^{i 2 pi p} of a phase in 64-bit fixed point: the top word in half-turns,
// its rounding to float32 put back as a rotation by the small remainder.
__device__ __forceinline__ void phase_factor(unsigned long long p, float &c, float &s) {
    const int top = (int)(p >> 32);
    const float t = (float)top;
    const float rest = (float)(top - (int)t) * 1.4629180792671596e-9f;   // pi 2^-31
    float s0, c0;
    sincospif(t * 4.656612873077393e-10f, &s0, &c0);
    c = fmaf(-s0, rest, c0);
    s = fmaf(c0, rest, s0);
}

// (hi, lo) += x, the rounding error of hi kept in lo
__device__ __forceinline__ void add_total(f32x2 &hi, f32x2 &lo, f32x2 x) {
    const f32x2 t = add2(hi, x), b = sub2(t, hi);
    lo = add2(lo, add2(sub2(hi, sub2(t, b)), sub2(x, b)));
    hi = t;
}

// Grid: x = blocks of a cluster (splits of the samples) x groups of TB traces,
// y = groups of tf frequencies.  Thread t: frequency lane t % tf, sample lane
// t / tf.  Parameters from dpar, or from the launch itself when it is null.
template <int TB, int N>
__global__ void __launch_bounds__(SPEC_THREADS)
k_trace_spectrum(const float *__restrict__ X, int n_traces, int n_t, int n_comp, int tf, int split,
                 const __grid_constant__ Blob<N> blob, const unsigned char *dpar, int foff, int n_freq, float taper,
                 double dt, float *__restrict__ out) {
    namespace cg = cooperative_groups;
    constexpr int ROW = TB + 4;       // floats per staged sample (16-byte rows, fewer bank conflicts)
    __shared__ __align__(16) float sv[SPEC_TILE * ROW];
    __shared__ double red[SPEC_THREADS * TB * 2];
    __shared__ TraceParam sp[TB];

    const unsigned char *par = dpar ? dpar : blob.b;
    const int tid = threadIdx.x;
    const int rank = blockIdx.x % split, tr0 = blockIdx.x / split * TB;
    const int fl = tid % tf, sl = tid / tf, ts = SPEC_THREADS / tf;
    const int kf = blockIdx.y * tf + fl;
    const int ntr = min(TB, n_traces - tr0);

    if (tid < TB) {
        TraceParam P{};
        if (tid < ntr) P = reinterpret_cast<const TraceParam *>(par)[tr0 + tid];
        sp[tid] = P;
    }
    __syncthreads();
    // the samples any of the block's traces needs, and this block's share of them
    int lo = n_t, hi = 0;
    for (int t = 0; t < ntr; ++t)
        if (sp[t].count > 0) {
            lo = min(lo, sp[t].first);
            hi = max(hi, sp[t].first + sp[t].count);
        }
    const int span = max(0, hi - lo);
    const int share = ((span + split - 1) / split + SPEC_TILE - 1) / SPEC_TILE * SPEC_TILE;
    const int beg = lo + min(span, rank * share), end = lo + min(span, rank * share + share);

    unsigned long long ph0 = 0ull, step = 0ull;
    if (kf < n_freq) {
        const FreqParam F = reinterpret_cast<const FreqParam *>(par + foff)[kf];
        ph0 = F.a;
        step = F.b;
    }
    float rc[SPEC_RUN], rs[SPEC_RUN], rm[SPEC_RUN];
#pragma unroll
    for (int j = 1; j < SPEC_RUN; ++j) {
        phase_factor(step * (unsigned long long)(j * SPEC_STRIDE), rc[j], rs[j]);
        // half of what |r|^2 lacks to one (r2: the rounding error of rs^2)
        const float s2 = rs[j] * rs[j], r2 = fmaf(rs[j], rs[j], -s2);
        rm[j] = 0.5f * (fmaf(-rc[j], rc[j], 1.f - s2) - r2);
    }

    f32x2 reh[TB / 2], rel[TB / 2], imh[TB / 2], iml[TB / 2];
#pragma unroll
    for (int t = 0; t < TB / 2; ++t) reh[t] = rel[t] = imh[t] = iml[t] = 0ull;

    // sample tid of the tile at n0 of every trace, weighted (untapered): loaded
    // before the previous tile is worked on
    const float half = 0.5f * taper;
    float nv[TB];
    auto load = [&](int n0) {
        const int n = n0 + tid;
#pragma unroll
        for (int t = 0; t < TB; ++t) {
            nv[t] = 0.f;
            if ((unsigned)(n - sp[t].first) < (unsigned)sp[t].count && n < end) {
                const float *x = X + ((size_t)(tr0 + t) * n_t + n) * n_comp;
                for (int c = 0; c < n_comp; ++c) nv[t] = fmaf(sp[t].a[c], x[c], nv[t]);
            }
        }
    };
    load(beg);
    for (int n0 = beg; n0 < end; n0 += SPEC_TILE) {
        __syncthreads();   // the previous tile is done with
#pragma unroll
        for (int t = 0; t < TB; ++t) {
            const int count = sp[t].count;
            if (taper > 0.f && count > 1) {
                const float u = (float)(n0 + tid - sp[t].first) * (1.f / (float)(count - 1));
                if (u < half)
                    nv[t] *= 0.5f * (1.f - cospif(2.f * u / taper));
                else if (u > 1.f - half)
                    nv[t] *= 0.5f * (1.f - cospif(2.f * (1.f - u) / taper));
            }
            sv[tid * ROW + t] = nv[t];
        }
        __syncthreads();
        if (n0 + SPEC_TILE < end) load(n0 + SPEC_TILE);
        for (int r = sl; r < SPEC_STRIDE; r += ts) {
            float c0, s0;
            phase_factor(ph0 + (unsigned long long)(n0 + r) * step, c0, s0);
            f32x2 re[TB / 2], im[TB / 2];
#pragma unroll
            for (int j = 0; j < SPEC_RUN; ++j) {   // samples past the end are staged as zeros
                float c = c0, s = s0;
                if (j) {
                    c = fmaf(-s0, rs[j], c0 * rc[j]);
                    s = fmaf(c0, rs[j], s0 * rc[j]);
                    c = fmaf(c, rm[j], c);
                    s = fmaf(s, rm[j], s);
                }
                const f32x2 cc = pack(c, c), ss = pack(s, s);
                const ulonglong2 *v = reinterpret_cast<const ulonglong2 *>(sv + (r + j * SPEC_STRIDE) * ROW);
#pragma unroll
                for (int t = 0; t < TB / 4; ++t) {
                    const ulonglong2 q = v[t];
                    const bool first = j % SPEC_SUM == 0;
                    re[2 * t] = first ? mul2(q.x, cc) : fma2(q.x, cc, re[2 * t]);
                    im[2 * t] = first ? mul2(q.x, ss) : fma2(q.x, ss, im[2 * t]);
                    re[2 * t + 1] = first ? mul2(q.y, cc) : fma2(q.y, cc, re[2 * t + 1]);
                    im[2 * t + 1] = first ? mul2(q.y, ss) : fma2(q.y, ss, im[2 * t + 1]);
                }
                if (j % SPEC_SUM == SPEC_SUM - 1)
#pragma unroll
                    for (int t = 0; t < TB / 2; ++t) {
                        add_total(reh[t], rel[t], re[t]);
                        add_total(imh[t], iml[t], im[t]);
                    }
            }
        }
    }

    // red[sample lane][trace][frequency lane][re, im]; an infinite total has no
    // meaningful rounding error
    auto total = [](float h, float l) { return isfinite(h) ? (double)h + (double)l : (double)h; };
#pragma unroll
    for (int t = 0; t < TB / 2; ++t) {
        double *r0 = red + ((size_t)(sl * TB + 2 * t) * tf + fl) * 2, *r1 = r0 + 2 * tf;
        const float2 a = unpack(reh[t]), b = unpack(rel[t]), c = unpack(imh[t]), d = unpack(iml[t]);
        r0[0] = total(a.x, b.x);
        r0[1] = total(c.x, d.x);
        r1[0] = total(a.y, b.y);
        r1[1] = total(c.y, d.y);
    }
    auto cluster = cg::this_cluster();
    cluster.sync();
    const int nout = TB * tf * 2;
    for (int o = rank * SPEC_THREADS + tid; o < nout; o += split * SPEC_THREADS) {
        const int t = o / (2 * tf), k = blockIdx.y * tf + o / 2 % tf;
        if (t >= ntr || k >= n_freq) continue;
        double sum = 0.0;
        for (int r = 0; r < split; ++r) {
            const double *q = cluster.map_shared_rank(red, r);
            for (int l = 0; l < ts; ++l) sum += q[(size_t)l * nout + o];
        }
        out[((size_t)(tr0 + t) * n_freq + k) * 2 + (o & 1)] = (float)(sum * dt);
    }
    cluster.sync();   // a block's totals stay until every block has read them
}

// Launch for TB traces per block; parameters by value where they fit.
template <int TB, int N>
cudaError_t launch_spectrum(dim3 grid, int split, cudaStream_t s, const float *X, int n_traces, int n_t, int n_comp,
                            int tf, const Blob<N> &blob, const unsigned char *dpar, int foff, int n_freq, float taper,
                            double dt, float *out) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(SPEC_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = split;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_trace_spectrum<TB, N>, X, n_traces, n_t, n_comp, tf, split, blob, dpar, foff,
                              n_freq, taper, dt, out);
}

template <int N>
cudaError_t launch_spectrum(int tb, dim3 grid, int split, cudaStream_t s, const float *X, int n_traces, int n_t,
                            int n_comp, int tf, const Blob<N> &blob, const unsigned char *dpar, int foff, int n_freq,
                            float taper, double dt, float *out) {
    auto f = tb == 4 ? launch_spectrum<4, N> : launch_spectrum<8, N>;
    return f(grid, split, s, X, n_traces, n_t, n_comp, tf, blob, dpar, foff, n_freq, taper, dt, out);
}

// Device (or managed) memory that kernels may read; a host pointer is refused
// before anything is launched.
bool device_pointer(const void *p) {
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" int fdtd_trace_spectrum(const float *traces, int n_traces, int n_t, int n_comp, const double *coef,
                                   const int *gate, double taper, double dt, double t0, const double *freq,
                                   int n_freq, float *out, int on_device, void *stream) {
    if (!traces || !freq || !out || n_traces < 1 || n_t < 1 || n_freq < 1 || n_comp < 1 ||
        n_comp > SPEC_MAX_COMP || !(taper >= 0.0 && taper <= 1.0) || !(dt > 0.0) || !std::isfinite(dt) ||
        !std::isfinite(t0))
        return FDTD_ERR_ARG;
    if (n_freq > 8 * 65535 || n_traces > 0x7fffffff / 2) return FDTD_ERR_ARG;
    if (!device_pointer(traces) || (on_device && !device_pointer(out))) return FDTD_ERR_ARG;

    std::vector<TraceParam> tp(n_traces);
    for (int p = 0; p < n_traces; ++p) {
        TraceParam &T = tp[p];
        for (int c = 0; c < SPEC_MAX_COMP; ++c) {
            double a = c < n_comp ? (coef ? coef[(size_t)p * n_comp + c] : (c == 0 ? 1.0 : 0.0)) : 0.0;
            if (!std::isfinite(a)) return FDTD_ERR_ARG;
            T.a[c] = (float)a;
        }
        T.first = gate ? gate[2 * p] : 0;
        T.count = gate ? gate[2 * p + 1] : n_t;
        if (T.first < 0 || T.count < 0 || (long long)T.first + T.count > n_t) return FDTD_ERR_ARG;
    }
    std::vector<FreqParam> fp(n_freq);
    for (int k = 0; k < n_freq; ++k) {
        const double f = freq[k];
        if (!std::isfinite(f) || !std::isfinite(f * t0) || !std::isfinite(f * dt)) return FDTD_ERR_ARG;
        fp[k].a = fixed_fraction(f * t0);
        fp[k].b = fixed_fraction(f * dt);
    }

    cudaStream_t s = (cudaStream_t)stream;
    const size_t tp_bytes = sizeof(TraceParam) * (size_t)n_traces;
    const size_t tp_pad = (tp_bytes + 15) & ~(size_t)15;
    const size_t par_bytes = tp_pad + sizeof(FreqParam) * (size_t)n_freq;
    const size_t out_bytes = sizeof(float) * 2 * (size_t)n_traces * n_freq;
    const bool carried = par_bytes <= (size_t)SPEC_LARGE;
    const size_t need = (carried ? 0 : par_bytes) + (on_device ? 0 : out_bytes);
    unsigned char *dev = nullptr;
    if (need > 0 && cudaMallocAsync((void **)&dev, need, s) != cudaSuccess) {
        cudaGetLastError();
        return FDTD_ERR_OOM;
    }
    const unsigned char *dpar = carried ? nullptr : dev;
    float *dout = on_device ? out : (float *)(dev + (carried ? 0 : par_bytes));
    int rc = FDTD_OK;
    if (!carried && (cudaMemcpyAsync(dev, tp.data(), tp_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess ||
                     cudaMemcpyAsync(dev + tp_pad, fp.data(), sizeof(FreqParam) * (size_t)n_freq,
                                     cudaMemcpyHostToDevice, s) != cudaSuccess))
        rc = FDTD_ERR_CUDA;
    if (rc == FDTD_OK) {
        // Lanes for up to 128 frequencies; the blocks of a cluster split the
        // samples while the grid stays within three blocks on each of 152 SMs
        // and every block has a tile or more.  Eight traces per block where
        // that fills the GPU with long shares (64 x 8204 samples x 1024
        // frequencies: 146 us, four traces 161), else four (143 x 1493 x 492:
        // 37 us, eight traces 45; 12 x 23635 x 10: 67 against 125); fewer
        // frequency lanes, so more blocks, where those are still too few
        // (3 x 4298 x 353: 21 us at 32 lanes, 33 at 128).
        constexpr long long SMS = 152;
        int tf = SPEC_MIN_TF, tb = 8, split = 1;
        while (tf < SPEC_THREADS && tf < n_freq) tf *= 2;
        long long groups = (n_traces + tb - 1) / tb, fgroups = (n_freq + tf - 1) / tf;
        auto splits = [&]() {
            int c = 1;
            while (c < SPEC_MAX_SPLIT && groups * fgroups * c < 3 * SMS && n_t / (2 * c) >= SPEC_TILE) c *= 2;
            return c;
        };
        split = splits();
        if (groups * fgroups * split < SMS || n_t / split < 4 * SPEC_TILE) {
            tb = 4;
            groups = (n_traces + tb - 1) / tb;
            split = splits();
            for (; groups * fgroups * split < SMS && tf > 32; split = splits()) {
                tf /= 2;
                fgroups = (n_freq + tf - 1) / tf;
            }
        }
        const dim3 grid((unsigned)(groups * split), (unsigned)fgroups);
        cudaError_t e;
        auto fill = [&](unsigned char *b) {
            if (!carried) return;
            std::memcpy(b, tp.data(), tp_bytes);
            std::memcpy(b + tp_pad, fp.data(), sizeof(FreqParam) * (size_t)n_freq);
        };
        if (!carried || par_bytes <= (size_t)SPEC_SMALL) {
            Blob<SPEC_SMALL> blob;
            fill(blob.b);
            e = launch_spectrum(tb, grid, split, s, traces, n_traces, n_t, n_comp, tf, blob, dpar, (int)tp_pad, n_freq,
                                (float)taper, dt, dout);
        } else {
            Blob<SPEC_LARGE> blob;
            fill(blob.b);
            e = launch_spectrum(tb, grid, split, s, traces, n_traces, n_t, n_comp, tf, blob, dpar, (int)tp_pad, n_freq,
                                (float)taper, dt, dout);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            rc = FDTD_ERR_CUDA;
        }
    }
    if (rc == FDTD_OK && !on_device) {
        if (cudaMemcpyAsync(out, dout, out_bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) rc = FDTD_ERR_CUDA;
    }
    if (dev) cudaFreeAsync(dev, s);
    if (!on_device && cudaStreamSynchronize(s) != cudaSuccess) rc = FDTD_ERR_CUDA;
    return rc;
}

extern "C" int fdtd_theta_coef(const double *theta, int n, double *coef) {
    if (!theta || !coef || n < 1) return FDTD_ERR_ARG;
    for (int t = 0; t < n; ++t)
        if (!std::isfinite(theta[t])) return FDTD_ERR_ARG;
    for (int t = 0; t < n; ++t) {
        coef[2 * t] = -std::sin(theta[t]);
        coef[2 * t + 1] = std::cos(theta[t]);
    }
    return FDTD_OK;
}
