// surrogate.cu -- forward/backward kernels and the optimiser step of the
// learned near-field surrogate (declarations and contracts: surrogate.h).
//
// The GEMM with 16-byte operand rows runs on the fifth-generation tensor cores
// (tcgen05, TMEM, TMA: gemm_tc.cu).  Other row strides and base addresses run on
// the warp-level mma.sync m16n8k16 bf16 instruction:
// 64x64 block tiles, 32-deep k slices staged in shared memory (either operand
// layout, transposed while staging), four warps of 32x32, f32 accumulators,
// fused bias / ReLU / bf16-copy epilogue.  The
// convolutions, the elementwise steps and the reductions are plain SIMT
// kernels: they are a few percent of the network's arithmetic.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/fdtd.h"
#include "../../include/surrogate.h"

namespace {

typedef unsigned short bf16raw;   // storage of one bfloat16

__device__ __forceinline__ float bf(const bf16raw v) { return __bfloat162float(__ushort_as_bfloat16(v)); }
__device__ __forceinline__ bf16raw tobf(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }

int launched() {
    if (cudaGetLastError() != cudaSuccess) return FDTD_ERR_CUDA;
    return FDTD_OK;
}

// ---- GEMM ------------------------------------------------------------------

constexpr int GBM = 64, GBN = 64, GBK = 32, GPAD = 8, GT = 128;

template <bool AK, bool BK>
__global__ void __launch_bounds__(GT) k_gemm(const bf16raw *__restrict__ A, int lda, const bf16raw *__restrict__ B,
                                             int ldb, float *Y, int ldy, bf16raw *Yb, int M, int N, int K,
                                             const float *__restrict__ bias, int relu, int accumulate) {
    __shared__ __align__(16) bf16raw As[GBM][GBK + GPAD];
    __shared__ __align__(16) bf16raw Bs[GBN][GBK + GPAD];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int wm = warp >> 1, wn = warp & 1;       // warp tile (32x32) inside the block tile
    const int g = lane >> 2, t4 = lane & 3;        // mma fragment coordinates
    const int m0 = blockIdx.y * GBM, n0 = blockIdx.x * GBN;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;

    for (int k0 = 0; k0 < K; k0 += GBK) {
        // stage A (64 x 32) and B (64 x 32), reading along the contiguous axis
#pragma unroll 4
        for (int e = t; e < GBM * GBK; e += GT) {
            int m, k;
            if (AK) { m = e / GBK; k = e % GBK; } else { m = e % GBM; k = e / GBM; }
            const int gm = m0 + m, gk = k0 + k;
            bf16raw v = 0;
            if (gm < M && gk < K) v = AK ? A[(long long)gm * lda + gk] : A[(long long)gk * lda + gm];
            As[m][k] = v;
        }
#pragma unroll 4
        for (int e = t; e < GBN * GBK; e += GT) {
            int n, k;
            if (BK) { n = e / GBK; k = e % GBK; } else { n = e % GBN; k = e / GBN; }
            const int gn = n0 + n, gk = k0 + k;
            bf16raw v = 0;
            if (gn < N && gk < K) v = BK ? B[(long long)gn * ldb + gk] : B[(long long)gk * ldb + gn];
            Bs[n][k] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GBK; kk += 16) {
            uint32_t a[2][4], b[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = wm * 32 + i * 16 + g;
                a[i][0] = *reinterpret_cast<const uint32_t *>(&As[r][kk + 2 * t4]);
                a[i][1] = *reinterpret_cast<const uint32_t *>(&As[r + 8][kk + 2 * t4]);
                a[i][2] = *reinterpret_cast<const uint32_t *>(&As[r][kk + 2 * t4 + 8]);
                a[i][3] = *reinterpret_cast<const uint32_t *>(&As[r + 8][kk + 2 * t4 + 8]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = wn * 32 + j * 8 + g;
                b[j][0] = *reinterpret_cast<const uint32_t *>(&Bs[c][kk + 2 * t4]);
                b[j][1] = *reinterpret_cast<const uint32_t *>(&Bs[c][kk + 2 * t4 + 8]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                        : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
                        : "r"(a[i][0]), "r"(a[i][1]), "r"(a[i][2]), "r"(a[i][3]), "r"(b[j][0]), "r"(b[j][1]));
        }
        __syncthreads();
    }
    // epilogue: c0,c1 at (row g, cols 2t4, 2t4+1), c2,c3 at row g+8
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int m = m0 + wm * 32 + i * 16 + g + (r >= 2 ? 8 : 0);
                const int n = n0 + wn * 32 + j * 8 + 2 * t4 + (r & 1);
                if (m >= M || n >= N) continue;
                const long long o = (long long)m * ldy + n;
                float v = acc[i][j][r];
                if (accumulate) v += Y[o];
                if (bias) v += bias[n];
                if (relu) v = fmaxf(v, 0.f);
                Y[o] = v;
                if (Yb) Yb[o] = tobf(v);
            }
}

// ---- convolution -------------------------------------------------------------

__global__ void k_conv_fwd(const float *__restrict__ x, int xs, const bf16raw *__restrict__ w,
                           const float *__restrict__ bias, float *y, int B, int cin, int lin, int cout, int k,
                           int stride, int pad, int lout, int relu) {
    const long long total = (long long)B * cout * lout;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < total;
         id += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(id % lout), o = (int)((id / lout) % cout), b = (int)(id / ((long long)lout * cout));
        float s = bias ? bias[o] : 0.f;
        const float *xb = x + (long long)b * xs;
        for (int c = 0; c < cin; ++c)
            for (int tt = 0; tt < k; ++tt) {
                const int i = l * stride + tt - pad;
                if (i >= 0 && i < lin) s += bf(w[(o * cin + c) * k + tt]) * xb[c * lin + i];
            }
        y[id] = relu ? fmaxf(s, 0.f) : s;
    }
}

__device__ __forceinline__ float block_sum(float v, float *red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    float s = 0.f;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;   // valid on thread 0
}

// dw[o][c][t], one block per (o, c); db[o] from the blocks with c == 0
__global__ void k_conv_bwd_w(const float *__restrict__ x, int xs, const float *__restrict__ y,
                             const float *__restrict__ dy, int dys, float *dw, float *db, int B, int cin, int lin,
                             int cout, int k, int stride, int pad, int lout) {
    __shared__ float red[32];
    const int o = blockIdx.x / cin, c = blockIdx.x % cin;
    float acc[8];
    for (int tt = 0; tt < 8; ++tt) acc[tt] = 0.f;
    float accb = 0.f;
    const long long total = (long long)B * lout;
    for (long long id = threadIdx.x; id < total; id += blockDim.x) {
        const int l = (int)(id % lout), b = (int)(id / lout);
        const long long yo = (long long)b * cout * lout + (long long)o * lout + l;
        const float dz = y[yo] > 0.f ? dy[(long long)b * dys + (long long)o * lout + l] : 0.f;
        if (dz == 0.f) continue;
        accb += dz;
        const float *xb = x + (long long)b * xs + (long long)c * lin;
        for (int tt = 0; tt < k; ++tt) {
            const int i = l * stride + tt - pad;
            if (i >= 0 && i < lin) acc[tt] += dz * xb[i];
        }
    }
    for (int tt = 0; tt < k; ++tt) {
        const float s = block_sum(acc[tt], red);
        if (threadIdx.x == 0) dw[(o * cin + c) * k + tt] = s;
    }
    const float sb = block_sum(accb, red);
    if (threadIdx.x == 0 && c == 0) db[o] = sb;
}

__global__ void k_conv_bwd_x(const bf16raw *__restrict__ w, const float *__restrict__ y,
                             const float *__restrict__ dy, int dys, float *dx, int B, int cin, int lin, int cout,
                             int k, int stride, int pad, int lout) {
    const long long total = (long long)B * cin * lin;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < total;
         id += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(id % lin), c = (int)((id / lin) % cin), b = (int)(id / ((long long)lin * cin));
        float s = 0.f;
        for (int tt = 0; tt < k; ++tt) {
            const int num = i + pad - tt;
            if (num < 0 || num % stride) continue;
            const int l = num / stride;
            if (l >= lout) continue;
            for (int o = 0; o < cout; ++o) {
                const long long yo = (long long)b * cout * lout + (long long)o * lout + l;
                if (y[yo] > 0.f) s += bf(w[(o * cin + c) * k + tt]) * dy[(long long)b * dys + (long long)o * lout + l];
            }
        }
        dx[id] = s;
    }
}

// ---- elementwise and reductions ------------------------------------------------

// V: elements a thread moves at once (4: float4 and 8-byte bf16 accesses)
template <int V>
__global__ void k_relu_bwd(const float *__restrict__ y, const float *__restrict__ dy, float *dz, bf16raw *dzb,
                           long long n) {
    const long long step = (long long)gridDim.x * blockDim.x * V;
    for (long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) * V; i < n; i += step) {
        if constexpr (V == 4) {
            const float4 a = *reinterpret_cast<const float4 *>(y + i), d = *reinterpret_cast<const float4 *>(dy + i);
            const float4 v = make_float4(a.x > 0.f ? d.x : 0.f, a.y > 0.f ? d.y : 0.f, a.z > 0.f ? d.z : 0.f,
                                         a.w > 0.f ? d.w : 0.f);
            *reinterpret_cast<float4 *>(dz + i) = v;
            if (dzb) *reinterpret_cast<ushort4 *>(dzb + i) = make_ushort4(tobf(v.x), tobf(v.y), tobf(v.z), tobf(v.w));
        } else {
            const float v = y[i] > 0.f ? dy[i] : 0.f;
            dz[i] = v;
            if (dzb) dzb[i] = tobf(v);
        }
    }
}

// Column sums.  A cluster of up to eight blocks takes 32 columns, each block a
// share of the rows, 32 warps over its rows with eight loads in flight; the
// blocks' sums meet in distributed shared memory in rank order.  (One block of
// eight warps per 32 columns: 41 us on 4096 x 1024, latency bound; now 7.8 us.)
constexpr int BG_W = 32;
__global__ void __launch_bounds__(32 * BG_W) k_bias_grad(const float *__restrict__ dz, int ldz, int M, int N, float *db,
                                                         int S) {
    namespace cg = cooperative_groups;
    __shared__ float red[BG_W][33], sum[32];
    const int rank = blockIdx.x % S, lane = threadIdx.x & 31, ry = threadIdx.x >> 5;
    const int col = blockIdx.x / S * 32 + lane;
    const int share = (M + S - 1) / S, m0 = min(M, rank * share), m1 = min(M, m0 + share);
    float s = 0.f;
    if (col < N) {
        const float *p = dz + col;
        int m = m0 + ry;
        for (; m + 7 * BG_W < m1; m += 8 * BG_W) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = p[(long long)(m + u * BG_W) * ldz];
            s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
        for (; m < m1; m += BG_W) s += p[(long long)m * ldz];
    }
    red[ry][lane] = s;
    __syncthreads();
    if (ry == 0) {
        float t = 0.f;
        for (int r = 0; r < BG_W; ++r) t += red[r][lane];
        sum[lane] = t;
    }
    auto cluster = cg::this_cluster();
    cluster.sync();
    if (rank == 0 && ry == 0 && col < N) {
        float t = 0.f;
        for (int r = 0; r < S; ++r) t += cluster.map_shared_rank(sum, r)[lane];
        db[col] = t;
    }
    cluster.sync();
}

__global__ void k_cast(const float *x, bf16raw *y, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = tobf(x[i]);
}

__global__ void k_concat(const float *a, int na, const float *c, int nc, bf16raw *out, int B) {
    const int w = na + nc;
    const long long n = (long long)B * w;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int f = (int)(i % w);
        const long long b = i / w;
        out[i] = tobf(f < na ? a[b * na + f] : c[b * nc + (f - na)]);
    }
}

__global__ void k_mse(const float *y, const float *t, long long n, float *dy, float *loss) {
    __shared__ float red[32];
    float s = 0.f;
    const float inv = 1.0f / (float)n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        dy[i] = 2.f * d * inv;
        s += d * d;
    }
    const float b = block_sum(s, red);
    if (loss && threadIdx.x == 0) atomicAdd(loss, b * inv);
}

__global__ void k_adam(float *w, bf16raw *wb, const float *g, float *m, float *v, long long n, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        if (wb) wb[i] = tobf(wi);
    }
}

// one warp per row: the row's peak |q|, then the division
__global__ void k_normalize(const float *q, int B, int n, float *qn, float *s) {
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= B) return;
    const float *qr = q + (long long)row * n;
    float m = 0.f;
    for (int i = lane; i < n; i += 32) m = fmaxf(m, fabsf(qr[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float inv = m > 0.f ? 1.f / m : 0.f;
    for (int i = lane; i < n; i += 32) qn[(long long)row * n + i] = qr[i] * inv;
    if (lane == 0) s[row] = m;
}

__global__ void k_features(const float *rz, int B, float r0, float rs, float z0, float zs, float *out) {
    const long long n = (long long)B * 64;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int f = (int)(i % 64);
        const long long b = i / 64;
        const float u = (rz[2 * b] - r0) / rs, v = (rz[2 * b + 1] - z0) / zs;
        float val = 0.f;
        if (f == 0) {
            val = u;
        } else if (f == 1) {
            val = v;
        } else if (f < 62) {
            const int q = (f - 2) / 4, r = (f - 2) % 4;
            const float a = 3.14159265358979f * (float)(q + 1) * (r < 2 ? u : v);
            val = (r & 1) ? cosf(a) : sinf(a);
        }
        out[i] = val;
    }
}

__global__ void k_scale_rows(float *y, int B, int n, const float *s, float c, int invert) {
    const long long total = (long long)B * n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const float sb = s[i / n];
        y[i] *= invert ? (sb != 0.f ? c / sb : 0.f) : c * sb;
    }
}

__global__ void k_pairs(const float *rz, int B, int K, float z0, float dz, float *out) {
    const long long n = (long long)B * K;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long b = i / K;
        const int k = (int)(i % K);
        out[2 * i] = rz[2 * b];
        out[2 * i + 1] = rz[2 * b + 1] - z0 - (float)k * dz;
    }
}

// retarded-time placement of bin k's response at antenna b: integer sample
// offset ci, interpolation weight f, amplitude 1/R
struct Place {
    int ci;
    float f, a;
};
__device__ __forceinline__ Place place(const float *rz, long long b, int k, int shift, float z0, float dz,
                                       float cps) {
    const float r = rz[2 * b], d = rz[2 * b + 1] - z0 - (float)k * dz;
    const float R = fmaxf(sqrtf(r * r + d * d), 0.5f * dz);
    const float c = (float)(shift * k) + R / cps;
    Place p;
    p.ci = (int)floorf(c);
    p.f = c - (float)p.ci;
    p.a = 1.f / R;
    return p;
}

// one thread per output sample, a loop over the bins
__global__ void k_assemble(const float *__restrict__ G, const float *__restrict__ qn, const float *__restrict__ rz,
                           int B, int K, int Tg, int shift, int T, float z0, float dz, float cps, int J0,
                           float *out) {
    const long long n = (long long)B * T;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n;
         id += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(id % T);
        const long long b = id / T;
        float s = 0.f;
        for (int k = 0; k < K; ++k) {
            const Place p = place(rz, b, k, shift, z0, dz, cps);
            const int j = i - p.ci + J0;
            if (j < 0) continue;
            const float *g = G + (b * K + k) * (long long)Tg;
            const float g0 = j < Tg ? g[j] : 0.f, g1 = (j >= 1 && j - 1 < Tg) ? g[j - 1] : 0.f;
            s += qn[b * K + k] * p.a * ((1.f - p.f) * g0 + p.f * g1);
        }
        out[id] = s;
    }
}

__global__ void k_assemble_bwd(const float *__restrict__ dout, const float *__restrict__ qn,
                               const float *__restrict__ rz, int B, int K, int Tg, int shift, int T, float z0,
                               float dz, float cps, int J0, float *dG, bf16raw *dGb) {
    const long long n = (long long)B * K * Tg;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n;
         id += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(id % Tg);
        const long long bk = id / Tg;
        const long long b = bk / K;
        const int k = (int)(bk % K);
        const Place p = place(rz, b, k, shift, z0, dz, cps);
        const int i0 = j + p.ci - J0, i1 = i0 + 1;
        const float d0 = (i0 >= 0 && i0 < T) ? dout[b * T + i0] : 0.f;
        const float d1 = (i1 >= 0 && i1 < T) ? dout[b * T + i1] : 0.f;
        const float v = qn[bk] * p.a * ((1.f - p.f) * d0 + p.f * d1);
        dG[id] = v;
        if (dGb) dGb[id] = tobf(v);
    }
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

int grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 4096) b = 4096;
    return (int)(b < 1 ? 1 : b);
}

// ---- lattice surrogate: bin responses on the grid's own lattice ----------------
// G[(ir * D + d) * T + tau] (bf16): response of antenna radial class ir to a
// unit profile bin at axial lattice offset d - moff (bins), tau samples after
// the bin's own time origin.  Antenna b has class ant[2b] and axial lattice
// index ant[2b+1]; bin k's offset is m - k, its time origin S k - J samples
// (J lead samples: the bin's charge starts to move one bin early).

__device__ __forceinline__ float val(const bf16raw v) { return bf(v); }
__device__ __forceinline__ float val(const float v) { return v; }

// Tab: bf16raw (with an optional second bf16 table Glo of the remainders) or float
template <typename Tab>
__global__ void __launch_bounds__(256) k_lat_fwd(const Tab *__restrict__ G, const bf16raw *__restrict__ Glo,
                                                 const float *__restrict__ q, const int *__restrict__ ant, int K,
                                                 int NR, int D, int T, int S, int J, int moff,
                                                 float *__restrict__ y) {
    __shared__ float qs[1024];
    const int b = blockIdx.y;
    for (int k = threadIdx.x; k < K; k += blockDim.x) qs[k] = q[(long long)b * K + k];
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int ir = ant[2 * b], m = ant[2 * b + 1];
    float acc = 0.f;
    if (ir >= 0 && ir < NR) {
        const long long base = (long long)ir * D * T;
        for (int k = 0; k < K && S * k - J <= t; ++k) {
            const int d = m - k + moff, tau = t - S * k + J;
            if (d >= 0 && d < D && tau < T && qs[k] != 0.f) {
                const long long i = base + (long long)d * T + tau;
                float gv = val(G[i]);
                if (Glo) gv += bf(Glo[i]);
                acc += qs[k] * gv;
            }
        }
    }
    y[(long long)b * T + t] = acc;
}

__global__ void __launch_bounds__(256) k_lat_bwd(const float *__restrict__ dy, const float *__restrict__ q,
                                                 const int *__restrict__ ant, int K, int NR, int D, int T, int S,
                                                 int J, int moff, float *__restrict__ dG) {
    __shared__ float qs[1024];
    const int b = blockIdx.y;
    for (int k = threadIdx.x; k < K; k += blockDim.x) qs[k] = q[(long long)b * K + k];
    __syncthreads();
    const int tau = blockIdx.x * blockDim.x + threadIdx.x;
    if (tau >= T) return;
    const int ir = ant[2 * b], m = ant[2 * b + 1];
    if (ir < 0 || ir >= NR) return;
    float *g = dG + (long long)ir * D * T;
    const float *r = dy + (long long)b * T;
    for (int k = 0; k < K && tau + S * k - J < T; ++k) {
        const int d = m - k + moff, t = tau + S * k - J;
        if (d >= 0 && d < D && t >= 0 && qs[k] != 0.f) atomicAdd(&g[(long long)d * T + tau], qs[k] * r[t]);
    }
}

// hi = bf16(x), lo = bf16(x - hi): x = hi + lo to about 2^-17 relative
__global__ void k_split_bf16(const float *__restrict__ x, bf16raw *__restrict__ hi, bf16raw *__restrict__ lo,
                             long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const bf16raw h = tobf(x[i]);
        hi[i] = h;
        lo[i] = tobf(x[i] - bf(h));
    }
}

// W[a][k][t] = G[ir_a][m_a - k + moff][t - S k + J] (0 where that time or the
// offset is off the table): antenna a's weights, a K x T matrix, for the GEMM
__global__ void k_lat_weights(const bf16raw *__restrict__ G, const int *__restrict__ ant, int K, int NR, int D,
                              int T, int S, int J, int moff, bf16raw *__restrict__ W) {
    const int a = blockIdx.z, k = blockIdx.y;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int ir = ant[2 * a], d = ant[2 * a + 1] - k + moff, tau = t - S * k + J;
    bf16raw v = 0;
    if (ir >= 0 && ir < NR && d >= 0 && d < D && tau >= 0 && tau < T) v = G[((long long)ir * D + d) * T + tau];
    W[((long long)a * K + k) * T + t] = v;
}

// The same weights K-major: W[a][t][koff + k] (row stride ldw), for the
// tcgen05 GEMM; one thread per (a, t, k), k fastest
__global__ void k_lat_weights_kmajor(const bf16raw *__restrict__ G, const int *__restrict__ ant, int A, int K, int NR,
                                     int D, int T, int S, int J, int moff, bf16raw *__restrict__ W, int ldw,
                                     int koff) {
    const long long n = (long long)A * T * K;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i % K);
        const long long at = i / K;
        const int t = (int)(at % T), a = (int)(at / T);
        const int ir = ant[2 * a], d = ant[2 * a + 1] - k + moff, tau = t - S * k + J;
        bf16raw v = 0;
        if (ir >= 0 && ir < NR && d >= 0 && d < D && tau >= 0 && tau < T) v = G[((long long)ir * D + d) * T + tau];
        W[at * ldw + koff + k] = v;
    }
}

// out[r] = [hi(x[r]), hi(x[r]), lo(x[r]), 0 ...] (row stride ld >= 3K): the A
// operand of the split-precision product [hi, hi, lo] [W_hi; W_lo; W_hi]
__global__ void k_split3_bf16(const float *__restrict__ x, int rows, int K, bf16raw *__restrict__ out, int ld) {
    const long long n = (long long)rows * ld;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % ld);
        const long long r = i / ld;
        bf16raw v = 0;
        if (c < 3 * K) {
            const float xv = x[r * K + c % K];
            const bf16raw h = tobf(xv);
            v = c < 2 * K ? h : tobf(xv - bf(h));
        }
        out[i] = v;
    }
}

// ---- one training step of the lattice table (sur_lattice_step) ----
//
// For the pairs of one radial class, with u = t - S m_b, the forward map is a
// matrix product, y_b(t) = sum_d Q_b[d] H[d][u], H[d][u] = G[ir][d][u + S d + c],
// c = J - S moff, Q_b[d] = q_b[m_b + moff - d] (zero outside 0..K-1), and the
// gradient its transpose, dH[d][u] = sum_b Q_b[d] dy_b(u + S m_b).  So a pass
// over the pairs class by class reads each table entry once per 32 pairs
// (pair by pair: 400 MB from L2 for 1024 pairs), and sums the gradient of an
// entry in registers (67 M atomic adds before), where the Adam update follows
// at once.  1024 pairs, 7.6 M entries: forward and loss 54 us (129 + 19
// before), gradient and update 58 us (119 + 40 + the clearing 6).  Bound by
// latency and issue (39 and 48 % active) ahead of DRAM (213 MB of table, moments
// and gradient, 31 us).
// Terms with q = 0 are left out, as an entry that is not finite would spread
// through them.

struct StepGeo {
    int B, K, NR, D, T, S, J, moff;
};
constexpr int ST_W = 8;            // warps of the forward kernel's blocks
constexpr int ST_P = 4;            // pairs per warp (forward)
constexpr int ST_U = 128;          // samples per block, four consecutive ones per lane
constexpr int ST_D = 128;          // table rows whose profile values are staged at a time (forward)
constexpr int ST_Q = ST_W * ST_P + 4;   // floats per staged row of profiles
constexpr int ST_RS = 32, ST_NS = 3;    // table rows per copy stage, stages in the ring
constexpr int ST_BW = 4, ST_R = 4;      // backward: warps per block, table rows per warp
constexpr size_t ST_SMEM = sizeof(float) * (ST_D * ST_Q + ST_NS * ST_RS * ST_U);

__device__ __forceinline__ void cp_async(float *dst, const float *src, int bytes, bool on) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (bytes == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(on ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(on ? 4 : 0) : "memory");
}
// four consecutive floats p[t .. t+3], zero outside [0, n); VEC: all inside or
// all outside, 16-byte aligned
template <bool VEC>
__device__ __forceinline__ void load4(float (&v)[4], const float *p, int t, int n) {
    if (VEC) {
        const float4 x = (unsigned)t < (unsigned)n ? *reinterpret_cast<const float4 *>(p + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (unsigned)(t + j) < (unsigned)n ? p[t + j] : 0.f;
    }
}
template <bool VEC>
__device__ __forceinline__ void store4(float *p, int t, int n, const float (&v)[4]) {
    if (VEC) {
        if ((unsigned)t < (unsigned)n) *reinterpret_cast<float4 *>(p + t) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((unsigned)(t + j) < (unsigned)n) p[t + j] = v[j];
    }
}

// Pairs by class, in their order: block c writes (b, m) to list[start[c] ..] and
// the range of m of its class.  Class NR holds the pairs that meet no table entry.
__global__ void __launch_bounds__(256) k_step_bucket(const int *__restrict__ ant, StepGeo g, int *start, int *mlo,
                                                     int *mhi, int2 *list) {
    __shared__ int wsum[8], s_lo, s_hi, s_base, s_before;
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    auto cls = [&](int b, int &m) {
        const int ir = ant[2 * b];
        m = ant[2 * b + 1];
        return ir < 0 || ir >= g.NR || m < -g.moff || m > g.D + g.K - 2 - g.moff ? g.NR : ir;
    };
    if (tid == 0) {
        s_before = 0;
        s_lo = 0x7fffffff;
        s_hi = -0x7fffffff;
    }
    __syncthreads();
    int before = 0, lo = 0x7fffffff, hi = -0x7fffffff;
    for (int b = tid; b < g.B; b += 256) {
        int m;
        const int k = cls(b, m);
        before += k < c;
        if (k == c) {
            lo = min(lo, m);
            hi = max(hi, m);
        }
    }
    atomicAdd(&s_before, before);
    atomicMin(&s_lo, lo);
    atomicMax(&s_hi, hi);
    __syncthreads();
    if (tid == 0) {
        start[c] = s_base = s_before;
        if (c == g.NR) start[c + 1] = g.B;
        mlo[c] = c == g.NR ? 0 : s_lo;
        mhi[c] = c == g.NR ? 0 : s_hi;
    }
    __syncthreads();
    for (int b0 = 0; b0 < g.B; b0 += 256) {
        int m;
        const bool in = b0 + tid < g.B && cls(b0 + tid, m) == c;
        const unsigned v = __ballot_sync(0xffffffffu, in);
        if (lane == 0) wsum[w] = __popc(v);
        __syncthreads();
        int at = s_base + __popc(v & ((1u << lane) - 1u)), all = 0;
        for (int k = 0; k < 8; ++k) {
            if (k < w) at += wsum[k];
            all += wsum[k];
        }
        if (in) list[at] = make_int2(b0 + tid, c == g.NR ? 0 : m);
        __syncthreads();
        if (tid == 0) s_base += all;
        __syncthreads();
    }
}

// The next up to 32 pairs of list[at, end) that pass `want(m)`, compacted into
// sb, sm (b = -1 past the last) by the first warp; returns where to go on.
template <typename F>
__device__ __forceinline__ int gather_pairs(const int2 *__restrict__ list, int at, int end, int *sb, int *sm, F want) {
    const int lane = threadIdx.x & 31;
    sb[lane] = -1;
    sm[lane] = 0;
    __syncwarp();
    int n = 0;
    while (n < 32 && at < end) {
        const int2 bm = at + lane < end ? list[at + lane] : make_int2(-1, 0);
        const bool in = bm.x >= 0 && want(bm.y);
        const unsigned v = __ballot_sync(0xffffffffu, in);
        const int slot = n + __popc(v & ((1u << lane) - 1u));
        if (in && slot < 32) {
            sb[slot] = bm.x;
            sm[slot] = bm.y;
        }
        const int all = __popc(v);
        if (n + all <= 32) {
            n += all;
            at += 32;
        } else {   // go on at the first pair that found no place
            at += __fns(v, 0, 32 - n + 1);
            n = 32;
        }
    }
    return at;
}

// Forward map, loss and its derivative: grid (tiles of u, classes + 1).  The
// table rows of the tile stream through a ring of asynchronous copies (they come
// from DRAM: with loads into registers a few rows ahead the kernel waited for
// them, 113 us), one stage of ST_RS rows for all warps of the block.
template <bool VEC>
__global__ void __launch_bounds__(32 * ST_W, 3) k_step_fwd(const float *__restrict__ G, const float *__restrict__ q,
                                                        const float *__restrict__ s,
                                                        const float *__restrict__ target,
                                                        const float *__restrict__ st, StepGeo g, float c_out,
                                                        const int *__restrict__ start, const int *__restrict__ mlo,
                                                        const int *__restrict__ mhi, const int2 *__restrict__ list,
                                                        float *__restrict__ dy, float *loss) {
    extern __shared__ __align__(16) float dyn[];
    float *Q = dyn, *ring = dyn + ST_D * ST_Q;
    __shared__ int sb[ST_W * ST_P], sm[ST_W * ST_P], s_at;
    __shared__ float red[32];
    const int cl = blockIdx.y, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int p0 = start[cl], p1 = start[cl + 1];
    if (p0 >= p1) return;
    const int lo = mlo[cl], hi = mhi[cl];
    const int u0 = -g.S * hi + blockIdx.x * ST_U;
    if (u0 > g.T - 1 - g.S * lo) return;
    const int c = g.J - g.S * g.moff;
    const float inv = 1.0f / (float)((long long)g.B * g.T);
    float sum = 0.f;
    for (int at = p0; at < p1;) {
        __syncthreads();
        if (w == 0) {   // pairs with a sample in this tile of u
            at = gather_pairs(list, at, p1, sb, sm, [&](int m) {
                return u0 + ST_U - 1 + g.S * m >= 0 && u0 + g.S * m < g.T;
            });
            if (lane == 0) s_at = at;
        }
        __syncthreads();
        at = s_at;
        // table rows that some of these pairs meet, and that hold a response
        // sample of this tile, 0 <= u + S d + c < T
        int d0 = g.D, d1 = -1;
        if (cl < g.NR)
            for (int i = 0; i < ST_W * ST_P; ++i)
                if (sb[i] >= 0) {
                    d0 = min(d0, sm[i] + g.moff - g.K + 1);
                    d1 = max(d1, sm[i] + g.moff);
                }
        if (g.S > 0) {
            const int a = -(u0 + ST_U - 1 + c), z = g.T - 1 - u0 - c;   // a <= S d <= z
            d0 = max(d0, a <= 0 ? 0 : (a + g.S - 1) / g.S);
            d1 = min(d1, z < 0 ? -1 : z / g.S);
        }
        d0 = max(d0, 0);
        d1 = min(d1, g.D - 1);
        const int nd = max(0, d1 + 1 - d0), stages = (nd + ST_RS - 1) / ST_RS;
        auto fetch = [&](int k) {   // rows d0 + k ST_RS .. of the tile, one commit group per stage
            if (k < stages) {
                float *r = ring + k % ST_NS * ST_RS * ST_U;
                constexpr int E = VEC ? 4 : 1;
#pragma unroll
                for (int e = tid * E; e < ST_RS * ST_U; e += 32 * ST_W * E) {
                    const int d = d0 + k * ST_RS + e / ST_U, tau = u0 + e % ST_U + g.S * d + c;
                    const bool on = d <= d1 && (unsigned)tau < (unsigned)g.T;
                    cp_async(r + e, on ? G + ((long long)cl * g.D + d) * g.T + tau : G, 4 * E, on);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        float acc[ST_P][4];
#pragma unroll
        for (int i = 0; i < ST_P; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 1
        for (int k = 0; k < ST_NS - 1; ++k) fetch(k);
        for (int k = 0; k < stages; ++k) {
            if (k * ST_RS % ST_D == 0) {   // the profile values of the next ST_D rows
                __syncthreads();
#pragma unroll
                for (int e = tid; e < ST_D * ST_W * ST_P; e += 32 * ST_W) {
                    const int dd = e % ST_D, i = e / ST_D, kk = sm[i] + g.moff - (d0 + k * ST_RS + dd);
                    Q[dd * ST_Q + i] = sb[i] >= 0 && kk >= 0 && kk < g.K ? q[(long long)sb[i] * g.K + kk] : 0.f;
                }
            }
            asm volatile("cp.async.wait_group %0;" ::"n"(ST_NS - 2) : "memory");
            __syncthreads();   // stage k is there, and stage k - 1 is done with
            fetch(k + ST_NS - 1);
            if (sb[w * ST_P] < 0) continue;   // no pair for this warp
            const float *r = ring + k % ST_NS * ST_RS * ST_U + 4 * lane;
            const float *qr = Q + (k * ST_RS % ST_D) * ST_Q + w * ST_P;
            const int n = min(ST_RS, nd - k * ST_RS);
#pragma unroll 4
            for (int e = 0; e < n; ++e) {
                const float4 h = *reinterpret_cast<const float4 *>(r + e * ST_U);
                const float4 v = *reinterpret_cast<const float4 *>(qr + e * ST_Q);
                const float qv[ST_P] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < ST_P; ++i)
                    if (qv[i] != 0.f) {
                        acc[i][0] = fmaf(qv[i], h.x, acc[i][0]);
                        acc[i][1] = fmaf(qv[i], h.y, acc[i][1]);
                        acc[i][2] = fmaf(qv[i], h.z, acc[i][2]);
                        acc[i][3] = fmaf(qv[i], h.w, acc[i][3]);
                    }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
        for (int i = 0; i < ST_P; ++i) {
            const int b = sb[w * ST_P + i];
            if (b < 0) continue;
            // the scaled output and target, and back (relative: by the target's own peak)
            const float sq = s[b], peak = st ? st[b] : 0.f;
            const float fy = st ? c_out * sq : 1.f, fr = st ? (peak != 0.f ? 1.f / peak : 0.f) : 1.f;
            const float ft = st ? 1.f : (sq != 0.f ? (1.f / c_out) / sq : 0.f);
            const int t = u0 + 4 * lane + g.S * sm[w * ST_P + i];
            float y[4], o[4];
            load4<VEC>(y, target + (long long)b * g.T, t, g.T);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float e = acc[i][j] * fy * fr - y[j] * ft;
                o[j] = 2.f * e * inv * fy * fr;
                if ((unsigned)(t + j) < (unsigned)g.T) sum += e * e;
            }
            store4<VEC>(dy + (long long)b * g.T, t, g.T, o);
        }
    }
    const float bs = block_sum(sum, red);
    if (tid == 0) atomicAdd(loss, bs * inv);
}

// Gradient and Adam update: grid (tiles of u, tiles of ST_BW ST_R table rows, classes).
template <bool VEC>
__global__ void __launch_bounds__(32 * ST_BW) k_step_bwd(const float *__restrict__ dy, const float *__restrict__ q,
                                                         StepGeo g, const int *__restrict__ start,
                                                         const int2 *__restrict__ list,
                                                         float *__restrict__ W, float *__restrict__ dG,
                                                         float *__restrict__ m1, float *__restrict__ m2, float lr,
                                                         float b1, float b2, float eps, float i1, float i2) {
    constexpr int NP = 32, ROWS = ST_BW * ST_R;   // pairs staged at a time, table rows of the block
    __shared__ __align__(16) float Q[NP][ROWS];
    __shared__ int sb[NP], sm[NP], s_at;
    const int cl = blockIdx.z, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int dt = blockIdx.y * ROWS, dw = dt + w * ST_R;
    const int c = g.J - g.S * g.moff;
    const int tau0 = blockIdx.x * ST_U + 4 * lane - g.S * (ST_R - 1);   // of row dw; row dw + i: + S i
    const int p0 = start[cl], p1 = start[cl + 1];
    // the table entries and moments, from DRAM to L2 while the gradient is summed
#pragma unroll
    for (int i = 0; i < ST_R; ++i) {
        const int tau = tau0 + g.S * i;
        if (dw + i >= g.D || (unsigned)tau >= (unsigned)g.T) continue;
        const long long o = ((long long)cl * g.D + dw + i) * g.T + tau;
        if (lane % 8 == 0) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(W + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(m1 + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(m2 + o));
        }
    }
    float acc[ST_R][4];
#pragma unroll
    for (int i = 0; i < ST_R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int at = p0; at < p1;) {
        __syncthreads();
        if (w == 0) {   // pairs that meet these table rows
            at = gather_pairs(list, at, p1, sb, sm, [&](int m) {
                return m + g.moff - dt >= 0 && m + g.moff - (dt + ROWS - 1) < g.K;
            });
            if (lane == 0) s_at = at;
        }
        __syncthreads();
        at = s_at;
#pragma unroll
        for (int e = tid; e < NP * ROWS; e += 32 * ST_BW) {
            const int i = e % ROWS, p = e / ROWS, k = sm[p] + g.moff - (dt + i);
            Q[p][i] = sb[p] >= 0 && k >= 0 && k < g.K ? q[(long long)sb[p] * g.K + k] : 0.f;
        }
        __syncthreads();
        // four pairs' samples in flight
        for (int pb = 0; pb < NP && sb[pb] >= 0; pb += 4) {
            float h[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e)   // a pair past the last has b = -1: an empty row
                load4<VEC>(h[e], dy + (long long)max(sb[pb + e], 0) * g.T, tau0 - g.S * dw - c + g.S * sm[pb + e],
                           sb[pb + e] >= 0 ? g.T : 0);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 v = *reinterpret_cast<const float4 *>(&Q[pb + e][w * ST_R]);
                const float qv[ST_R] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < ST_R; ++i)
                    if (qv[i] != 0.f)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(qv[i], h[e][j], acc[i][j]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < ST_R; ++i) {
        if (dw + i >= g.D) continue;
        const long long base = ((long long)cl * g.D + dw + i) * g.T;
        const int tau = tau0 + g.S * i;
        float a[4], v[4], x[4];
        load4<VEC>(a, m1 + base, tau, g.T);
        load4<VEC>(v, m2 + base, tau, g.T);
        load4<VEC>(x, W + base, tau, g.T);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float gi = acc[i][j];
            a[j] = b1 * a[j] + (1.f - b1) * gi;
            v[j] = b2 * v[j] + (1.f - b2) * gi * gi;
            x[j] = x[j] - lr * (a[j] * i1) / (sqrtf(v[j] * i2) + eps);
        }
        store4<VEC>(dG + base, tau, g.T, acc[i]);
        store4<VEC>(m1 + base, tau, g.T, a);
        store4<VEC>(m2 + base, tau, g.T, v);
        store4<VEC>(W + base, tau, g.T, x);
    }
}

// ---- serving every profile at every antenna (sur_lattice_serve) ----

// One warp per profile: its peak s, and the split of the normalised profile as
// the A operand [hi, hi, lo], each part KS columns (zeros past K).
__global__ void k_serve_profiles(const float *__restrict__ q, int P, int K, int KS, bf16raw *__restrict__ out,
                                 float *__restrict__ s) {
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= P) return;
    const float *qr = q + (long long)row * K;
    float m = 0.f;
    for (int i = lane; i < K; i += 32) m = fmaxf(m, fabsf(qr[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float inv = m > 0.f ? 1.f / m : 0.f;
    bf16raw *o = out + (long long)row * 3 * KS;
    for (int i = lane; i < KS; i += 32) {
        const float x = i < K ? qr[i] * inv : 0.f;
        const bf16raw h = tobf(x);
        o[i] = o[KS + i] = h;
        o[2 * KS + i] = tobf(x - bf(h));
    }
    if (lane == 0) s[row] = m;
}

// The B operands: W[a][k][t] = Ghi[ir][d][t - S k + J] for k < K, the same of Glo
// from row KS, zeros where the table has no such entry.  A block copies rows k
// (a warp each) of one antenna and part, eight t per lane: the table row is read
// and W written along t, so both are coalesced (gathered K-major, two bytes a
// lane along k, the same weights took 3 x 34.6 us for 64 antennas, now one launch of 10 us).
// VEC: S, J and T are multiples of four and the tables 8-byte aligned, so that a
// lane's eight entries are two 8-byte loads.
template <bool VEC>
__global__ void __launch_bounds__(256) k_serve_weights(const bf16raw *__restrict__ Ghi, const bf16raw *__restrict__ Glo,
                                                       const int *__restrict__ ant, int K, int KS, int NR, int D, int T,
                                                       int TW, int S, int J, int moff, bf16raw *__restrict__ W) {
    const int a = blockIdx.y, row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;   // row of 2 KS
    const int k = row < KS ? row : row - KS;
    const int ir = ant[2 * a], d = ant[2 * a + 1] - k + moff;
    const bool on = k < K && ir >= 0 && ir < NR && d >= 0 && d < D;
    const bf16raw *g = (row < KS ? Ghi : Glo) + ((long long)(on ? ir : 0) * D + (on ? d : 0)) * T;
    bf16raw *w = W + ((long long)a * 2 * KS + row) * TW;
    const int off = J - S * k;
    for (int t = 8 * lane; t < TW; t += 256) {
        ushort4 v[2] = {make_ushort4(0, 0, 0, 0), make_ushort4(0, 0, 0, 0)};
        if (on) {
            if (VEC) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int tau = t + 4 * h + off;   // a multiple of four: a quad lies inside the row or outside
                    if (tau >= 0 && tau < T && t + 4 * h < T) v[h] = *reinterpret_cast<const ushort4 *>(g + tau);
                }
            } else {
                bf16raw *e = reinterpret_cast<bf16raw *>(v);
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    const int tau = t + h + off;
                    if (tau >= 0 && tau < T && t + h < T) e[h] = g[tau];
                }
            }
        }
        *reinterpret_cast<uint4 *>(w + t) = *reinterpret_cast<const uint4 *>(v);
    }
}

struct ServeLayout {
    int KS, TW;                       // K rounded up to 64, T to 8
    long long q, s, w, bytes;         // offsets of Q3, the peaks and W
};
ServeLayout serve_layout(int P, int A, int K, int T) {
    ServeLayout L;
    L.KS = (K + 63) / 64 * 64;
    L.TW = (T + 7) / 8 * 8;
    const auto up = [](long long n) { return (n + 255) / 256 * 256; };
    L.q = 0;
    L.s = up(2LL * P * 3 * L.KS);
    L.w = L.s + up(4LL * P);
    L.bytes = L.w + up(2LL * A * 2 * L.KS * L.TW);
    return L;
}

}  // namespace

namespace fdtd {
namespace gtc {
// gemm_tc.cu: the tcgen05 kernel's layout for this product (-1: none), the
// path selected by sur_gemm_set_path, and its launch
int tc_layout(const void *A, int lda, int a_kmajor, const void *B, int ldb, int b_kmajor, int K);
int tc_path();
int gemm_tc(int layout, const void *A, int lda, int a_kmajor, const void *B, int ldb, int b_kmajor, float *Y, int ldy,
            void *Yb, int M, int N, int K, const float *bias, int relu, int accumulate, cudaStream_t s);
int serve_gemm(const void *Q, const void *W, int ldw, float *Y, int M, int N, int KS, int batch, const float *row_scale,
               float alpha, cudaStream_t s);
}  // namespace gtc
}  // namespace fdtd

extern "C" {

int sur_gemm_bf16(const void *A, int lda, int a_kmajor, const void *B, int ldb, int b_kmajor, float *Y, int ldy,
                  void *Yb, int M, int N, int K, const float *bias, int relu, int accumulate, void *stream) {
    if (!A || !B || !Y || M < 1 || N < 1 || K < 1 || lda < 1 || ldb < 1 || ldy < N) return FDTD_ERR_ARG;
    if ((a_kmajor ? lda < K : lda < M) || (b_kmajor ? ldb < K : ldb < N)) return FDTD_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // operands with 16-byte rows: the tcgen05 kernels; else mma.sync
    const int layout = fdtd::gtc::tc_layout(A, lda, a_kmajor, B, ldb, b_kmajor, K);
    if (layout >= 0) 
        return fdtd::gtc::gemm_tc(layout, A, lda, a_kmajor, B, ldb, b_kmajor, Y, ldy, Yb, M, N, K, bias, relu, accumulate,
                                  s);
    if (fdtd::gtc::tc_path() >= 2) return FDTD_ERR_ARG;   // the tcgen05 kernel alone was asked for
    const dim3 grid((N + GBN - 1) / GBN, (M + GBM - 1) / GBM);
    const bf16raw *a = static_cast<const bf16raw *>(A), *b = static_cast<const bf16raw *>(B);
    bf16raw *yb = static_cast<bf16raw *>(Yb);
    if (a_kmajor && b_kmajor)
        k_gemm<true, true><<<grid, GT, 0, s>>>(a, lda, b, ldb, Y, ldy, yb, M, N, K, bias, relu, accumulate);
    else if (a_kmajor)
        k_gemm<true, false><<<grid, GT, 0, s>>>(a, lda, b, ldb, Y, ldy, yb, M, N, K, bias, relu, accumulate);
    else if (b_kmajor)
        k_gemm<false, true><<<grid, GT, 0, s>>>(a, lda, b, ldb, Y, ldy, yb, M, N, K, bias, relu, accumulate);
    else
        k_gemm<false, false><<<grid, GT, 0, s>>>(a, lda, b, ldb, Y, ldy, yb, M, N, K, bias, relu, accumulate);
    return launched();
}

int sur_conv1d_fwd(const float *x, int xs, const void *w, const float *bias, float *y, int B, int cin, int lin,
                   int cout, int k, int stride, int pad, int relu, void *stream) {
    if (!x || !w || !y || B < 1 || cin < 1 || lin < 1 || cout < 1 || k < 1 || k > 8 || stride < 1 || pad < 0 ||
        xs < cin * lin)
        return FDTD_ERR_ARG;
    const int lout = (lin + 2 * pad - k) / stride + 1;
    if (lout < 1) return FDTD_ERR_ARG;
    const long long n = (long long)B * cout * lout;
    k_conv_fwd<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        x, xs, static_cast<const bf16raw *>(w), bias, y, B, cin, lin, cout, k, stride, pad, lout, relu);
    return launched();
}

int sur_conv1d_bwd(const float *x, int xs, const void *w, const float *y, const float *dy, int dys, float *dx,
                   float *dw, float *db, int B, int cin, int lin, int cout, int k, int stride, int pad,
                   void *stream) {
    if (!x || !w || !y || !dy || !dw || !db || B < 1 || cin < 1 || lin < 1 || cout < 1 || k < 1 || k > 8 ||
        stride < 1 || pad < 0 || xs < cin * lin)
        return FDTD_ERR_ARG;
    const int lout = (lin + 2 * pad - k) / stride + 1;
    if (lout < 1 || dys < cout * lout) return FDTD_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    k_conv_bwd_w<<<cout * cin, 256, 0, s>>>(x, xs, y, dy, dys, dw, db, B, cin, lin, cout, k, stride, pad, lout);
    if (dx) {
        const long long n = (long long)B * cin * lin;
        k_conv_bwd_x<<<grid_for(n, 256), 256, 0, s>>>(static_cast<const bf16raw *>(w), y, dy, dys, dx, B, cin,
                                                        lin, cout, k, stride, pad, lout);
    }
    return launched();
}

int sur_relu_bwd(const float *y, const float *dy, float *dz, void *dzb, long long n, void *stream) {
    if (!y || !dy || !dz || n < 1) return FDTD_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    bf16raw *zb = static_cast<bf16raw *>(dzb);
    // 16-byte accesses where every array allows them (4096 x 1024: 18.5 us scalar, 8.9 us)
    if (n % 4 == 0 && aligned16(y) && aligned16(dy) && aligned16(dz) && (reinterpret_cast<uintptr_t>(dzb) & 7) == 0)
        k_relu_bwd<4><<<grid_for(n / 4, 256), 256, 0, s>>>(y, dy, dz, zb, n);
    else
        k_relu_bwd<1><<<grid_for(n, 256), 256, 0, s>>>(y, dy, dz, zb, n);
    return launched();
}

int sur_bias_grad(const float *dz, int ldz, int M, int N, float *db, void *stream) {
    if (!dz || !db || M < 1 || N < 1 || ldz < N) return FDTD_ERR_ARG;
    int S = 1;   // blocks per 32 columns: while they fit two per SM and have 256 rows or more each
    while (S < 8 && (long long)((N + 31) / 32) * S * 2 <= 2 * 152 && M / (2 * S) >= 256) S *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((N + 31) / 32 * S));
    cfg.blockDim = dim3(32 * BG_W);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = S;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k_bias_grad, dz, ldz, M, N, db, S) != cudaSuccess) {
        cudaGetLastError();
        return FDTD_ERR_CUDA;
    }
    return FDTD_OK;
}

int sur_cast_bf16(const float *x, void *y, long long n, void *stream) {
    if (!x || !y || n < 1) return FDTD_ERR_ARG;
    k_cast<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(x, static_cast<bf16raw *>(y), n);
    return launched();
}

int sur_concat_bf16(const float *a, int na, const float *c, int nc, void *out, int B, void *stream) {
    if (!a || !c || !out || na < 1 || nc < 1 || B < 1) return FDTD_ERR_ARG;
    const long long n = (long long)B * (na + nc);
    k_concat<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(a, na, c, nc,
                                                                               static_cast<bf16raw *>(out), B);
    return launched();
}

int sur_mse(const float *y, const float *t, long long n, float *dy, float *loss, void *stream) {
    if (!y || !t || !dy || n < 1) return FDTD_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (loss && cudaMemsetAsync(loss, 0, sizeof(float), s) != cudaSuccess) return FDTD_ERR_CUDA;
    k_mse<<<grid_for(n, 256), 256, 0, s>>>(y, t, n, dy, loss);
    return launched();
}

int sur_adam(float *w, void *wb, const float *g, float *m, float *v, long long n, float lr, float b1, float b2,
             float eps, int t, void *stream) {
    if (!w || !g || !m || !v || n < 1 || t < 1) return FDTD_ERR_ARG;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    k_adam<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(w, static_cast<bf16raw *>(wb), g, m, v,
                                                                              n, lr, b1, b2, eps, c1, c2);
    return launched();
}

int sur_normalize_rows(const float *q, int B, int n, float *qn, float *s, void *stream) {
    if (!q || !qn || !s || B < 1 || n < 1) return FDTD_ERR_ARG;
    k_normalize<<<(B + 7) / 8, 256, 0, static_cast<cudaStream_t>(stream)>>>(q, B, n, qn, s);
    return launched();
}

int sur_antenna_features(const float *rz, int B, float r0, float rs, float z0, float zs, float *out, void *stream) {
    if (!rz || !out || B < 1 || !(rs != 0.f) || !(zs != 0.f)) return FDTD_ERR_ARG;
    k_features<<<grid_for((long long)B * 64, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(rz, B, r0, rs, z0, zs,
                                                                                               out);
    return launched();
}

int sur_scale_rows(float *y, int B, int n, const float *s, float c, int invert, void *stream) {
    if (!y || !s || B < 1 || n < 1) return FDTD_ERR_ARG;
    k_scale_rows<<<grid_for((long long)B * n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(y, B, n, s, c,
                                                                                               invert);
    return launched();
}

int sur_pairs(const float *rz, int B, int K, float z0, float dz, float *out, void *stream) {
    if (!rz || !out || B < 1 || K < 1) return FDTD_ERR_ARG;
    k_pairs<<<grid_for((long long)B * K, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(rz, B, K, z0, dz, out);
    return launched();
}

int sur_assemble(const float *G, const float *qn, const float *rz, int B, int K, int Tg, int shift, int T, float z0,
                 float dz, float cps, int J0, float *out, void *stream) {
    if (!G || !qn || !rz || !out || B < 1 || K < 1 || Tg < 1 || shift < 0 || T < 1 || !(dz > 0.f) || !(cps > 0.f) ||
        J0 < 0)
        return FDTD_ERR_ARG;
    k_assemble<<<grid_for((long long)B * T, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        G, qn, rz, B, K, Tg, shift, T, z0, dz, cps, J0, out);
    return launched();
}

int sur_assemble_bwd(const float *dout, const float *qn, const float *rz, int B, int K, int Tg, int shift, int T,
                     float z0, float dz, float cps, int J0, float *dG, void *dGb, void *stream) {
    if (!dout || !qn || !rz || !dG || B < 1 || K < 1 || Tg < 1 || shift < 0 || T < 1 || !(dz > 0.f) ||
        !(cps > 0.f) || J0 < 0)
        return FDTD_ERR_ARG;
    k_assemble_bwd<<<grid_for((long long)B * K * Tg, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        dout, qn, rz, B, K, Tg, shift, T, z0, dz, cps, J0, dG, static_cast<bf16raw *>(dGb));
    return launched();
}

int sur_lattice_fwd(const void *G, const void *Glo, const float *q, const int *ant, int B, int K, int NR, int D,
                    int T, int S, int J, int moff, float *y, void *stream) {
    if (!G || !q || !ant || !y || B < 1 || B > 65535 || K < 1 || K > 1024 || NR < 1 || D < 1 || T < 1 || S < 0 ||
        J < 0)
        return FDTD_ERR_ARG;
    k_lat_fwd<bf16raw><<<dim3((T + 255) / 256, B), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const bf16raw *>(G), static_cast<const bf16raw *>(Glo), q, ant, K, NR, D, T, S, J, moff, y);
    return launched();
}

int sur_lattice_fwd_f32(const float *G, const float *q, const int *ant, int B, int K, int NR, int D, int T, int S,
                        int J, int moff, float *y, void *stream) {
    if (!G || !q || !ant || !y || B < 1 || B > 65535 || K < 1 || K > 1024 || NR < 1 || D < 1 || T < 1 || S < 0 ||
        J < 0)
        return FDTD_ERR_ARG;
    k_lat_fwd<float><<<dim3((T + 255) / 256, B), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        G, nullptr, q, ant, K, NR, D, T, S, J, moff, y);
    return launched();
}

int sur_split_bf16(const float *x, void *hi, void *lo, long long n, void *stream) {
    if (!x || !hi || !lo || n < 1) return FDTD_ERR_ARG;
    k_split_bf16<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        x, static_cast<bf16raw *>(hi), static_cast<bf16raw *>(lo), n);
    return launched();
}

int sur_lattice_bwd(const float *dy, const float *q, const int *ant, int B, int K, int NR, int D, int T, int S,
                    int J, int moff, float *dG, void *stream) {
    if (!dy || !q || !ant || !dG || B < 1 || B > 65535 || K < 1 || K > 1024 || NR < 1 || D < 1 || T < 1 || S < 0 ||
        J < 0)
        return FDTD_ERR_ARG;
    k_lat_bwd<<<dim3((T + 255) / 256, B), 256, 0, static_cast<cudaStream_t>(stream)>>>(dy, q, ant, K, NR, D, T, S,
                                                                                         J, moff, dG);
    return launched();
}

int sur_lattice_weights_kmajor(const void *G, const int *ant, int A, int K, int NR, int D, int T, int S, int J,
                               int moff, void *W, int ldw, int koff, void *stream) {
    if (!G || !ant || !W || A < 1 || K < 1 || NR < 1 || D < 1 || T < 1 || S < 0 || J < 0 || koff < 0 ||
        ldw < koff + K)
        return FDTD_ERR_ARG;
    const long long n = (long long)A * T * K;
    k_lat_weights_kmajor<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const bf16raw *>(G), ant, A, K, NR, D, T, S, J, moff, static_cast<bf16raw *>(W), ldw, koff);
    return launched();
}

int sur_split3_bf16(const float *x, int rows, int K, void *out, int ld, void *stream) {
    if (!x || !out || rows < 1 || K < 1 || ld < 3 * K) return FDTD_ERR_ARG;
    k_split3_bf16<<<grid_for((long long)rows * ld, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        x, rows, K, static_cast<bf16raw *>(out), ld);
    return launched();
}

int sur_lattice_weights(const void *G, const int *ant, int A, int K, int NR, int D, int T, int S, int J, int moff,
                        void *W, void *stream) {
    if (!G || !ant || !W || A < 1 || A > 65535 || K < 1 || K > 65535 || NR < 1 || D < 1 || T < 1 || S < 0 || J < 0)
        return FDTD_ERR_ARG;
    k_lat_weights<<<dim3((T + 255) / 256, K, A), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const bf16raw *>(G), ant, K, NR, D, T, S, J, moff, static_cast<bf16raw *>(W));
    return launched();
}

long long sur_lattice_serve_bytes(int P, int A, int K, int T) {
    if (P < 1 || A < 1 || K < 1 || T < 1) return FDTD_ERR_ARG;
    return serve_layout(P, A, K, T).bytes;
}

int sur_lattice_serve(const void *Ghi, const void *Glo, const float *q, const int *ant, int P, int A, int K, int NR,
                      int D, int T, int S, int J, int moff, float c_out, void *work, long long work_bytes, float *out,
                      void *stream) {
    if (!Ghi || !Glo || !q || !ant || !work || !out || P < 1 || A < 1 || A > 65535 || K < 1 || NR < 1 || D < 1 || T < 1 ||
        S < 0 || J < 0 || !aligned16(work))
        return FDTD_ERR_ARG;
    const ServeLayout L = serve_layout(P, A, K, T);
    if (work_bytes < L.bytes) return FDTD_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *w = static_cast<char *>(work);
    bf16raw *Q = reinterpret_cast<bf16raw *>(w + L.q), *W = reinterpret_cast<bf16raw *>(w + L.w);
    float *s = reinterpret_cast<float *>(w + L.s);
    k_serve_profiles<<<(P + 7) / 8, 256, 0, st>>>(q, P, K, L.KS, Q, s);
    const dim3 grid(2 * L.KS / 8, A);
    const bf16raw *hi = static_cast<const bf16raw *>(Ghi), *lo = static_cast<const bf16raw *>(Glo);
    const bool vec = S % 4 == 0 && J % 4 == 0 && T % 4 == 0 &&
                     ((reinterpret_cast<uintptr_t>(Ghi) | reinterpret_cast<uintptr_t>(Glo)) & 7) == 0;
    if (vec)
        k_serve_weights<true><<<grid, 256, 0, st>>>(hi, lo, ant, K, L.KS, NR, D, T, L.TW, S, J, moff, W);
    else
        k_serve_weights<false><<<grid, 256, 0, st>>>(hi, lo, ant, K, L.KS, NR, D, T, L.TW, S, J, moff, W);
    const int rc = launched();
    if (rc != FDTD_OK) return rc;
    return fdtd::gtc::serve_gemm(Q, W, L.TW, out, P, T, L.KS, A, s, c_out, st);
}

long long sur_lattice_step_bytes(int B, int NR) {
    if (B < 1 || NR < 1) return FDTD_ERR_ARG;
    return 4LL * (3LL * NR + 4 + 2LL * B);
}

int sur_lattice_step(float *G, float *dG, float *m, float *v, const float *qn, const float *s, const int *ant,
                     const float *target, const float *st, int B, int K, int NR, int D, int T, int S, int J, int moff,
                     float c_out, float lr, float b1, float b2, float eps, int t, float *dy, float *loss, void *work,
                     long long work_bytes, void *stream) {
    if (!G || !dG || !m || !v || !qn || !s || !ant || !target || !dy || !loss || !work || B < 1 || B > 65535 || K < 1 ||
        K > 1024 || NR < 1 || NR > 65534 || D < 1 || T < 1 || S < 0 || J < 0 || t < 1 ||
        (reinterpret_cast<uintptr_t>(work) & 7) || work_bytes < sur_lattice_step_bytes(B, NR))
        return FDTD_ERR_ARG;
    // positions along u and tau stay well inside 32 bits
    if ((long long)S * (D + 2LL * K + (moff < 0 ? -(long long)moff : moff)) + T + J > (1LL << 30)) return FDTD_ERR_ARG;
    const StepGeo g{B, K, NR, D, T, S, J, moff};
    cudaStream_t q = static_cast<cudaStream_t>(stream);
    int2 *list = static_cast<int2 *>(work);
    int *start = reinterpret_cast<int *>(list + B), *mlo = start + NR + 2, *mhi = mlo + NR + 1;
    if (cudaMemsetAsync(loss, 0, sizeof(float), q) != cudaSuccess) return FDTD_ERR_CUDA;
    k_step_bucket<<<NR + 1, 256, 0, q>>>(ant, g, start, mlo, mhi, list);
    // u of a class spans T + S (range of m), m in [-moff, D + K - 2 - moff]
    const long long span = T + (long long)S * (D + K - 2);
    const dim3 gf((unsigned)((span + ST_U - 1) / ST_U), NR + 1);
    const dim3 gb((unsigned)((T + (long long)S * (ST_R - 1) + ST_U - 1) / ST_U), (D + ST_BW * ST_R - 1) / (ST_BW * ST_R), NR);
    const float i1 = 1.f / (1.f - powf(b1, (float)t)), i2 = 1.f / (1.f - powf(b2, (float)t));
    // 16-byte accesses where every row and lag allows them
    const bool vec = S % 4 == 0 && J % 4 == 0 && T % 4 == 0 && aligned16(G) && aligned16(dG) && aligned16(m) &&
                     aligned16(v) && aligned16(target) && aligned16(dy);
    const void *fwd = vec ? (const void *)k_step_fwd<true> : (const void *)k_step_fwd<false>;
    if (cudaFuncSetAttribute(fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ST_SMEM) != cudaSuccess) {
        cudaGetLastError();
        return FDTD_ERR_CUDA;
    }
    if (vec) {
        k_step_fwd<true><<<gf, 32 * ST_W, ST_SMEM, q>>>(G, qn, s, target, st, g, c_out, start, mlo, mhi, list, dy,
                                                        loss);
        k_step_bwd<true><<<gb, 32 * ST_BW, 0, q>>>(dy, qn, g, start, list, G, dG, m, v, lr, b1, b2, eps, i1, i2);
    } else {
        k_step_fwd<false><<<gf, 32 * ST_W, ST_SMEM, q>>>(G, qn, s, target, st, g, c_out, start, mlo, mhi, list, dy,
                                                         loss);
        k_step_bwd<false><<<gb, 32 * ST_BW, 0, q>>>(dy, qn, g, start, list, G, dG, m, v, lr, b1, b2, eps, i1, i2);
    }
    return launched();
}

}  // extern "C"
