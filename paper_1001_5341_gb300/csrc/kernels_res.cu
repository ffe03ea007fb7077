// kernels_res.cu -- many steps of a small grid in one launch, its fields
// resident in registers and shared memory (PEC and first-order Mur grids; the
// Yee leapfrog of Sec. III.A with the shower current of Sec. III.B).
//
// A 96^3 step is 0.9 M cell-updates, under a microsecond of arithmetic on 152
// SMs, but the one-step path spends 18.6 us on it (22.8 with Mur faces): three
// launches, each with its pipeline to fill.  Here one cooperative launch runs up
// to RES_STEPS steps of 5.7 us (6.8); 32^3: 14.5 -> 3.8 us, and already 11.9 in
// runs of two steps.  A block owns a brick of the node grid, all x columns (at
// most 128) by up to RW rows by up to KZ planes; warp w holds row j0 + w, lane L
// the columns 4L .. 4L+3 of its planes: Ey, Ez and Hy in registers, and what the
// neighbouring rows read -- Ex, Ez, Hx and Hz -- in shared memory (Ex only
// there: 20 warps leave 96 registers a thread, and a spilled register costs more
// here than a shared read, because 190 KB of shared memory leave little L1).
//
// Per step:
//   H phase  H^{n+1/2} of the brick from E^n: row j+1 from the shared rows of E,
//            plane k+1 from the next plane, column i+1 by shuffle; the row and the
//            plane of the bricks after this one from those bricks;
//   E phase  E^{n+1} likewise from row j-1, plane k-1 and column i-1, the current,
//            and the Mur faces (x and z faces from the own warp's values, y faces
//            after the block's barrier from the row next to them).
// Two halo warps fetch the rows of the bricks after and before; one warp tabulates
// the current of the next E phase and records the detectors, which takes both off
// the rows' path (1.1 and 0.7 us a step there).
// Bricks exchange what their neighbours read -- E (Ex, Ez) of their first row and
// (Ex, Ey) of their first plane to the brick before, H (Hx, Hz) of their last row
// and (Hx, Hy) of their last plane to the brick after -- as indivisible 16-byte
// words {three values, tag}, the tag counting the steps: a reader polls the words
// themselves, so an exchange costs one store and one load through L2 and no flag
// or fence.  The two exchanges of a step, about 1.7 us each, are what bounds a
// small brick; 96^3 adds the shared-memory traffic of 68 row-planes a block.
// A word is overwritten only after its reader has used it: the owner of a row or
// plane publishes E^{n+1} after it has received the neighbour's H^{n+1/2}, which
// the neighbour computes from E^n, and the other way round.  Every poll is bounded.
// Blocks meet through barriers A (H phase done) and B (E phase done); neighbour
// to neighbour barriers between the rows instead measured 9.7 us against 8.1.
//
// The expressions are those of the tile path (kernels_vtile.cu) and of k_mur, so
// the fields are bit for bit the same.
#include <cuda_runtime.h>

#include <algorithm>
#include <new>
#include <vector>

#include "fdtd_internal.h"
#include "source_term.cuh"
#include "tma_pipe.cuh"

namespace fdtd {
namespace {

using namespace tma;

constexpr int RW = 17;              // most rows of a brick
constexpr int KZ = 4;               // most planes of a brick
constexpr int NH = KZ / 2;          // halo warps, two planes each
constexpr int NWB = RW + NH + 1;    // warps: rows, halo, current
constexpr int NTB = 32 * NWB;
constexpr int COLS = 128;
constexpr int RES_STEPS = 64;       // most steps per launch
constexpr int ROWF = 2 * COLS;      // floats of a shared row (two components)
constexpr int SET = (RW + 1) * KZ * ROWF;   // rows of the brick and one halo row
constexpr int FACE = KZ * ROWF;             // old E of the row next to a y face, per side
constexpr int CUR = RW * KZ * COLS;         // increments of the current
constexpr int EYROWS = RW * KZ * COLS;      // a brick's Ey, in global memory
constexpr size_t RES_SMEM = (2 * SET + 2 * FACE + CUR) * sizeof(float);
constexpr int EY_REC = 1 << 20;
constexpr int MAX_REC = 1024;       // most detector records of a brick (beyond: the one-step path)
// 16-byte words received by a brick: E of row j1 and of plane k1, H of row j0-1 and of plane k0-1;
// three words per lane for four columns of two components
constexpr int XW = 3 * 32;
constexpr int X_EY = 0, X_EZ = X_EY + KZ * XW, X_HY = X_EZ + RW * XW, X_HZ = X_HY + KZ * XW, X_WORDS = X_HZ + RW * XW;

struct ResArgs {
    Grid g;
    const float *in;            // the current set
    float *out;                 // the set that takes the result
    float kE, kH, m;
    int by, bz;                 // bricks along y and z
    int n;                      // steps
    unsigned tag0;              // tag of E^n at the start; step s publishes tag0 + s + 1
    uint4 *xch;                 // [brick][X_WORDS]
    Source src;
    const SourceStep *ss;       // [n]
    const int2 *bricks;         // [bricks + 1] first detector record, rows whose Ey is recorded
    const int2 *rec;            // records: place in shared memory (Ey: past EY_REC, in the brick's `ey`), slot
    float *ey;                  // [brick][RW][KZ][COLS], rows that detectors read
    float *rbuf;                // [n][slots]
    int slots;
    int *flags;
};

// One 16-byte access, indivisible (the scalar b128 form): {three values, tag}.
__device__ __forceinline__ void put(uint4 *p, float a, float b, float c, unsigned tag) {
    asm volatile(
        "{.reg .b64 l, h; .reg .b128 w; mov.b64 l, {%1, %2}; mov.b64 h, {%3, %4}; mov.b128 w, {l, h};\n\t"
        "st.relaxed.gpu.global.b128 [%0], w;}" ::"l"(p),
        "f"(a), "f"(b), "f"(c), "r"(tag)
        : "memory");
}
struct Word {
    float a, b, c;
    unsigned tag;
};
__device__ __forceinline__ Word get(const uint4 *p) {
    Word w;
    asm volatile(
        "{.reg .b64 l, h; .reg .b128 w; ld.relaxed.gpu.global.b128 w, [%4]; mov.b128 {l, h}, w;\n\t"
        "mov.b64 {%0, %1}, l; mov.b64 {%2, %3}, h;}"
        : "=f"(w.a), "=f"(w.b), "=f"(w.c), "=r"(w.tag)
        : "l"(p)
        : "memory");
    return w;
}
// four columns of two components
__device__ __forceinline__ void publish(uint4 *p, int lane, float4 x, float4 y, unsigned tag) {
    put(p + lane, x.x, x.y, x.z, tag);
    put(p + 32 + lane, x.w, y.x, y.y, tag);
    put(p + 64 + lane, y.z, y.w, 0.f, tag);
}
struct Words {
    Word u, v, w;
};
__device__ __forceinline__ Words peek(const uint4 *p, int lane) {
    return Words{get(p + lane), get(p + 32 + lane), get(p + 64 + lane)};
}
__device__ __forceinline__ bool tagged(const Words &a, unsigned tag) {
    return a.u.tag == tag && a.v.tag == tag && a.w.tag == tag;
}
__device__ __forceinline__ float4 first(const Words &a) { return make_float4(a.u.a, a.u.b, a.u.c, a.v.a); }
__device__ __forceinline__ float4 second(const Words &a) { return make_float4(a.v.b, a.v.c, a.w.a, a.w.b); }
constexpr long long WAIT_CYCLES = 4LL << 30;   // bound of a poll: about two seconds
// poll until the words carry the tag, from a first look a; a poll that gives up
// is recorded, and the thread polls no more
__device__ __forceinline__ void receive(const uint4 *p, int lane, unsigned tag, float4 &x, float4 &y, bool &dead,
                                        Words a) {
    if (!tagged(a, tag)) {
        const long long t0 = clock64();
        while (!dead) {
            a = peek(p, lane);
            if (tagged(a, tag)) break;
            if (clock64() - t0 > WAIT_CYCLES) dead = true;
        }
    }
    x = first(a);
    y = second(a);
}

__device__ __forceinline__ float4 shift_r(float4 v) {   // column i+1
    return make_float4(v.y, v.z, v.w, __shfl_down_sync(0xffffffffu, v.x, 1));
}
__device__ __forceinline__ float4 shift_l(float4 v) {   // column i-1
    const float w = __shfl_up_sync(0xffffffffu, v.w, 1);
    return make_float4(w, v.x, v.y, v.z);
}
// first-order Mur: E0' = E1 + m (E1' - E0)
__device__ __forceinline__ float mur1(float e1, float m, float e1n, float e0) { return e1 + m * (e1n - e0); }
__device__ __forceinline__ float4 mur4(float4 e0, float4 e1, float m, float4 e1n) {
    return make_float4(mur1(e1.x, m, e1n.x, e0.x), mur1(e1.y, m, e1n.y, e0.y), mur1(e1.z, m, e1n.z, e0.z),
                       mur1(e1.w, m, e1n.w, e0.w));
}
// a value on an x face: Mur, or as it was
__device__ __forceinline__ float face(bool mur, float e1, float m, float e1n, float e0) {
    return mur ? mur1(e1, m, e1n, e0) : e0;
}

__global__ void __launch_bounds__(32) k_res_source(Source s, long long n0, SourceStep *out) {
    __shared__ SourceStep w;
    source_step_warp(s, n0 + blockIdx.x, &w);
    __syncwarp();
    const int words = sizeof(SourceStep) / 4;
    for (int t = threadIdx.x; t < words; t += 32)
        reinterpret_cast<int *>(out + blockIdx.x)[t] = reinterpret_cast<const int *>(&w)[t];
}

// all warps of the block, from the row warps' loop and from the others'
__device__ __forceinline__ void block_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(NTB) : "memory"); }

template <int N>
struct Planes {
    static constexpr int value = N;
};

template <bool MUR>
__global__ void __launch_bounds__(NTB, 1) k_res(const ResArgs A) {
    extern __shared__ __align__(128) float smem[];
    // rows [row][plane][2][COLS] of (Ex, Ez) and (Hx, Hz), old (Ex, Ez) next to the
    // y faces [side][plane][2][COLS], increments of Ez [row][plane][COLS]
    float *XE = smem, *XH = smem + SET, *FO = smem + 2 * SET, *CI = FO + 2 * FACE;
    __shared__ __align__(8) uint64_t halo[2], fdone;   // E row j1, H row j0-1 arrived; Mur row ny done
    __shared__ int cur_lo, cur_hi;              // planes of the brick with current in this step
    const Grid &g = A.g;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const int bj = blockIdx.x % A.by, bk = blockIdx.x / A.by;
    const int j0 = bj * (ny + 1) / A.by, j1 = (bj + 1) * (ny + 1) / A.by;
    const int k0 = bk * (nz + 1) / A.bz, k1 = (bk + 1) * (nz + 1) / A.bz;
    const int nj = j1 - j0, nk = k1 - k0;
    const bool up_y = j1 <= ny, dn_y = j0 > 0, up_z = k1 <= nz, dn_z = k0 > 0;   // bricks beyond
    // word offsets: this brick's inbox, and those of the bricks after and before it
    const int box = blockIdx.x * X_WORDS, box_y = X_WORDS, box_z = A.by * X_WORDS;
    bool dead = false;

    if (tid == 0) {
        mbar_init(&halo[0], NH);
        mbar_init(&halo[1], NH);
        mbar_init(&fdone, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const bool row = w < nj, halow = w >= RW && w < RW + NH, curw = w == RW + NH;
    const int j = j0 + w, col = 4 * lane;
    auto srow = [&](float *base, int r, int p, int c) { return base + ((r * KZ + p) * 2 + c) * COLS + col; };

    // edges of the x faces are left alone by the Mur update of the other faces
    auto keep = [&](float4 n, float4 o) {
        if (lane == 0) n.x = o.x;
        if (col == nx) n.x = o.x;
        if (col + 1 == nx) n.y = o.y;
        if (col + 2 == nx) n.z = o.z;
        if (col + 3 == nx) n.w = o.w;
        return n;
    };

    float4 Ey[KZ], Ez[KZ], Hy[KZ];
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool inrow = col < g.pitch;   // pitch is a multiple of 32
#pragma unroll
    for (int p = 0; p < KZ; ++p) {
        Ey[p] = Ez[p] = Hy[p] = z4;
        if (row && p < nk) {
            const float *f = A.in + gidx(g, 0, j, k0 + p) + col;
            float4 ex = z4, hx = z4, hz = z4;
            if (inrow) {
                ex = *reinterpret_cast<const float4 *>(f);
                Ey[p] = *reinterpret_cast<const float4 *>(f + g.comp);
                Ez[p] = *reinterpret_cast<const float4 *>(f + 2 * g.comp);
                hx = *reinterpret_cast<const float4 *>(f + 3 * g.comp);
                Hy[p] = *reinterpret_cast<const float4 *>(f + 4 * g.comp);
                hz = *reinterpret_cast<const float4 *>(f + 5 * g.comp);
            }
            sts4(srow(XH, w, p, 0), hx);
            sts4(srow(XH, w, p, 1), hz);
            sts4(srow(XE, w, p, 0), ex);
            sts4(srow(XE, w, p, 1), Ez[p]);
        }
    }
    for (int t = tid; t < CUR; t += NTB) CI[t] = 0.f;   // columns without current stay zero
    // E of the first plane to the brick below, of the first row to the brick before
    auto publish_e_plane = [&](float4 ex, float4 ey, unsigned tag) {
        publish(A.xch + box - box_z + X_EZ + w * XW, lane, ex, ey, tag);
    };
    auto publish_e_row = [&](int p, float4 ex, float4 ez, unsigned tag) {
        publish(A.xch + box - box_y + X_EY + p * XW, lane, ex, ez, tag);
    };
    if (row) {
        if (dn_z) publish_e_plane(lds4(srow(XE, w, 0, 0)), Ey[0], A.tag0);
        if (dn_y && w == 0) {
#pragma unroll
            for (int p = 0; p < KZ; ++p)
                if (p < nk) publish_e_row(p, lds4(srow(XE, 0, p, 0)), Ez[p], A.tag0);
        }
    }
    // two planes' rows of (E or H) from the brick after or before into row slot r
    auto receive_rows = [&](const uint4 *in, float *X, int r, unsigned tag) {
        const int p = 2 * (w - RW);
        if (p >= nk) return;
        const uint4 *q = in + p * XW;
        const bool two = p + 1 < nk;
        Words a, b;
        const long long t0 = clock64();
        do {
            a = peek(q, lane);
            if (two) b = peek(q + XW, lane);
            if (dead || (tagged(a, tag) && (!two || tagged(b, tag)))) break;
            if (clock64() - t0 > WAIT_CYCLES) dead = true;
        } while (true);
        sts4(srow(X, r, p, 0), first(a));
        sts4(srow(X, r, p, 1), second(a));
        if (two) {
            sts4(srow(X, r, p + 1, 0), first(b));
            sts4(srow(X, r, p + 1, 1), second(b));
        }
    };
    const bool yface = MUR && row && (j == 0 || j == ny);
    const int nxq = nx & 3, nxl = nx >> 2;   // place of column nx
    const bool srcrow = A.src.active && row && j >= A.src.jc - A.src.L && j <= A.src.jc + A.src.L;
    const bool cur_rows = A.src.active && j0 <= A.src.jc + A.src.L && j1 > A.src.jc - A.src.L;
    const int2 recs = A.bricks ? A.bricks[blockIdx.x] : make_int2(0, 0);
    const int nrec = A.bricks ? A.bricks[blockIdx.x + 1].x - recs.x : 0;
    auto eyp = [&]() { return A.ey + (size_t)blockIdx.x * EYROWS; };
    const bool eyrow = row && (recs.y >> w & 1);
    __syncthreads();

    if (!row) {   // halo warps, the current's warp and warps beyond the brick's rows
        const int2 rec = curw && lane < nrec ? A.rec[recs.x + lane] : make_int2(0, 0);
        // detector records of step s, between its E phase and the next one's
        auto record = [&](int s) {
            for (int t = lane; t < nrec; t += 32) {
                const int2 e = t == lane ? rec : A.rec[recs.x + t];
                A.rbuf[(size_t)s * A.slots + e.y] = e.x < EY_REC ? smem[e.x] : __ldcg(eyp() + e.x - EY_REC);
            }
        };
        for (int s = 0; s < A.n; ++s) {
            const unsigned te = A.tag0 + s;
            if (halow && up_y) {
                receive_rows(A.xch + box + X_EY, XE, nj, te);
                __syncwarp();
                if (lane == 0) mbar_arrive(&halo[0]);
            }
            if (curw && cur_rows) {
                const SourceStep &ss = A.ss[s];
                const int a = max(ss.klo, k0), b = min(ss.khi, k1 - 1), L = A.src.L, W = 2 * L + 1;
                const int r0 = max(A.src.jc - L - j0, 0), r1 = min(A.src.jc + L - j0, nj - 1);
                for (int k = a; k <= b; ++k) {
                    const double amp = ss.tab ? ss.amp[k - ss.kb] : source_amp(A.src, A.src.q, k, ss.n);
                    for (int i = lane; i < W; i += 32) {
                        float *c = CI + (k - k0) * COLS + A.src.ic - L + i;
                        const double *wt = A.src.w + (r0 + j0 - A.src.jc + L) * W + i;
#pragma unroll 4
                        for (int r = r0; r <= r1; ++r) c[r * KZ * COLS] = (float)(amp * wt[(r - r0) * W]);
                    }
                }
                if (lane == 0) {
                    cur_lo = a - k0;
                    cur_hi = b - k0;
                }
            }
            if (curw && s > 0) record(s - 1);
            block_barrier();
            if (halow && dn_y) {
                receive_rows(A.xch + box + X_HY, XH, RW, te + 1);
                __syncwarp();
                if (lane == 0) mbar_arrive(&halo[1]);
            }
            block_barrier();
        }
        if (curw) record(A.n - 1);
        if (dead) atomicOr(A.flags, 1);
        return;
    }
    // the steps of a row, for a brick of NK planes
    auto run = [&](auto planes) {
        constexpr int NK = decltype(planes)::value;
        const bool jfirst = w > 0 || dn_y, jlast = w < nj - 1 || up_y;   // beyond row 0, below row ny
        for (int s = 0; s < A.n; ++s) {
            const unsigned te = A.tag0 + s, th = te + 1;   // tags of E^n, of H^{n+1/2} and E^{n+1}
            // ---- H phase ----
            {
                const uint4 *q = A.xch + box + X_EZ + w * XW;
                if (w == nj - 1 && up_y && !dead && !mbar_wait(&halo[0], s & 1)) dead = true;
                if (MUR && j == ny - 1 && s > 0 && !dead && !mbar_wait(&fdone, (s - 1) & 1)) dead = true;
                float4 exK = lds4(srow(XE, w, 0, 0));
#pragma unroll
                for (int p = 0; p < NK; ++p) {
                    const bool kfirst = p > 0 || dn_z, klast = p < NK - 1 || up_z;   // beyond plane 0, below plane nz
                    const float4 ex = exK;
                    float4 eyK = z4;
                    if (p < NK - 1) {
                        exK = lds4(srow(XE, w, p < NK - 1 ? p + 1 : p, 0));
                        eyK = Ey[p < NK - 1 ? p + 1 : p];
                    } else if (up_z) {
                        receive(q, lane, te, exK, eyK, dead, peek(q, lane));
                    }
                    const float4 exU = lds4(srow(XE, w + 1, p, 0)), ezU = lds4(srow(XE, w + 1, p, 1));
                    float4 hx = lds4(srow(XH, w, p, 0)), hz = lds4(srow(XH, w, p, 1));
                    if (jlast && klast) {
                        hx = axpy(hx, -A.kH, (ezU - Ez[p]) - (eyK - Ey[p]));
                        if (jfirst) Hy[p] = axpy(Hy[p], -A.kH, (exK - ex) - (shift_r(Ez[p]) - Ez[p]));
                        if (kfirst) hz = axpy(hz, -A.kH, (shift_r(Ey[p]) - Ey[p]) - (exU - ex));
                        sts4(srow(XH, w, p, 0), hx);
                        sts4(srow(XH, w, p, 1), hz);
                    }
                    if (p == NK - 1 && up_z) publish(A.xch + box + box_z + X_HZ + w * XW, lane, hx, Hy[p], th);
                    if (w == nj - 1 && up_y) publish(A.xch + box + box_y + X_HY + p * XW, lane, hx, hz, th);
                }
            }
            block_barrier();
            // ---- E phase ----
            {
                const uint4 *q = A.xch + box + X_HZ + w * XW;
                int plo = 1, phi = 0;   // planes with current
                if (srcrow) {
                    plo = cur_lo;
                    phi = cur_hi;
                }
                if (w == 0 && dn_y && !dead && !mbar_wait(&halo[1], s & 1)) dead = true;
                const int wd = w > 0 ? w - 1 : RW;   // shared row of j-1
                [[maybe_unused]] float4 oxz = z4, oyz = z4;   // old Ex, Ey of plane 1
#pragma unroll
                for (int pp = 0; pp < NK; ++pp) {
                    const int p = NK - 1 - pp;   // the first plane last: it waits for the brick below
                    const bool kfirst = p > 0 || dn_z, klast = p < NK - 1 || up_z;   // beyond plane 0, below plane nz
                    const float4 hx = lds4(srow(XH, w, p, 0)), hz = lds4(srow(XH, w, p, 1));
                    const float4 hxD = lds4(srow(XH, wd, p, 0)), hzD = lds4(srow(XH, wd, p, 1));
                    float4 hxK = z4, hyK = z4;
                    if (p > 0) {
                        hxK = lds4(srow(XH, w, p > 0 ? p - 1 : 0, 0));
                        hyK = Hy[p > 0 ? p - 1 : 0];
                    } else if (dn_z) {
                        receive(q, lane, th, hxK, hyK, dead, peek(q, lane));
                    }
                    const float4 oy = Ey[p], oz = Ez[p];
                    float4 ex = lds4(srow(XE, w, p, 0));
                    if (MUR && (j == 1 || j == ny - 1)) {
                        float *o = FO + (j == 1 ? 0 : FACE) + p * ROWF + col;
                        sts4(o, ex);
                        sts4(o + COLS, oz);
                    }
                    [[maybe_unused]] const float4 ox = ex;
                    const float4 lhz = shift_l(hz), lhy = shift_l(Hy[p]);
                    if (jfirst && jlast && kfirst && klast)
                        ex = axpy(ex, A.kE, (hz - hzD) - (Hy[p] - hyK));
                    if (jlast && kfirst && klast) Ey[p] = axpy(Ey[p], A.kE, (hx - hxK) - (hz - lhz));
                    if (jfirst && jlast && klast) {
                        Ez[p] = axpy(Ez[p], A.kE, (Hy[p] - lhy) - (hx - hxD));
                        if (p >= plo && p <= phi) {
                            const float4 c = lds4(CI + (w * KZ + p) * COLS + col);
                            Ez[p] = make_float4(Ez[p].x + c.x, Ez[p].y + c.y, Ez[p].z + c.z, Ez[p].w + c.w);
                        }
                    }
                    // x faces: columns 0 and nx, from columns 1 and nx - 1 (Mur) or as they were; the
                    // columns beyond nx, Hx of column 0 and Ex, Hy, Hz of column nx hold what no
                    // other column reads
                    if (klast) {
                        const bool fy = jlast && kfirst, fz = jfirst && jlast;
                        float yo = 0.f, yn = 0.f, zo = 0.f, zn = 0.f;   // column nx - 1, old and new
                        if (nxq == 0 && MUR) {
                            yo = __shfl_up_sync(0xffffffffu, oy.w, 1);
                            yn = __shfl_up_sync(0xffffffffu, Ey[p].w, 1);
                            zo = __shfl_up_sync(0xffffffffu, oz.w, 1);
                            zn = __shfl_up_sync(0xffffffffu, Ez[p].w, 1);
                        }
                        if (lane == 0) {
                            if (fy) Ey[p].x = face(MUR, oy.y, A.m, Ey[p].y, oy.x);
                            if (fz) Ez[p].x = face(MUR, oz.y, A.m, Ez[p].y, oz.x);
                        }
                        if (lane == nxl) {
                            if (nxq == 0) {
                                if (fy) Ey[p].x = face(MUR, yo, A.m, yn, oy.x);
                                if (fz) Ez[p].x = face(MUR, zo, A.m, zn, oz.x);
                            } else if (nxq == 1) {
                                if (fy) Ey[p].y = face(MUR, oy.x, A.m, Ey[p].x, oy.y);
                                if (fz) Ez[p].y = face(MUR, oz.x, A.m, Ez[p].x, oz.y);
                            } else if (nxq == 2) {
                                if (fy) Ey[p].z = face(MUR, oy.y, A.m, Ey[p].y, oy.z);
                                if (fz) Ez[p].z = face(MUR, oz.y, A.m, Ez[p].y, oz.z);
                            } else {
                                if (fy) Ey[p].w = face(MUR, oy.z, A.m, Ey[p].z, oy.w);
                                if (fz) Ez[p].w = face(MUR, oz.z, A.m, Ez[p].z, oz.w);
                            }
                        }
                    }
                    if constexpr (MUR) {
                        // z faces
                        if (p == 0 && !dn_z) {
                            if (jfirst && jlast) ex = mur4(ex, oxz, A.m, lds4(srow(XE, w, 1, 0)));
                            if (jlast) Ey[0] = keep(mur4(Ey[0], oyz, A.m, Ey[1]), Ey[0]);
                        }
                        if (p == NK - 2 && !up_z) {   // plane nz is the next one
                            const int pn = p < NK - 1 ? p + 1 : p;
                            if (jfirst && jlast)
                                sts4(srow(XE, w, pn, 0), mur4(lds4(srow(XE, w, pn, 0)), ox, A.m, ex));
                            if (jlast) Ey[pn] = keep(mur4(Ey[pn], oy, A.m, Ey[p]), Ey[pn]);
                        }
                        if (p == 1 && !dn_z) {   // comes before plane 0
                            oxz = ox;
                            oyz = oy;
                        }
                    }
                    sts4(srow(XE, w, p, 0), ex);
                    sts4(srow(XE, w, p, 1), Ez[p]);
                    if (eyrow) __stcg(reinterpret_cast<float4 *>(eyp() + (w * KZ + p) * COLS + col), Ey[p]);
                    // never a y face (a brick has two rows or more); Ex of plane nz is not used there
                    if (w == 0 && dn_y) publish_e_row(p, ex, Ez[p], th);
                    if (p == 0 && dn_z && !yface) publish_e_plane(ex, Ey[p], th);
                }
            }
            block_barrier();
            if (yface) {
                // y faces from the row next to them, old (FO) and new
                const int wi = j == 0 ? w + 1 : w - 1;
                const float *o = FO + (j == 0 ? 0 : FACE) + col;
#pragma unroll
                for (int p = 0; p < NK; ++p) {
                    const bool kfirst = p > 0 || dn_z, klast = p < NK - 1 || up_z;   // beyond plane 0, below plane nz
                    float4 ex = lds4(srow(XE, w, p, 0));
                    if (kfirst && klast) ex = mur4(ex, lds4(o + p * ROWF), A.m, lds4(srow(XE, wi, p, 0)));
                    if (klast) Ez[p] = keep(mur4(Ez[p], lds4(o + p * ROWF + COLS), A.m, lds4(srow(XE, wi, p, 1))), Ez[p]);
                    sts4(srow(XE, w, p, 0), ex);
                    sts4(srow(XE, w, p, 1), Ez[p]);
                    if (p == 0 && dn_z) publish_e_plane(ex, Ey[p], th);
                }
                __syncwarp();
                if (j == ny && lane == 0) mbar_arrive(&fdone);   // the row before it reads this one
            }
        }
    };
    if (nk == 2) run(Planes<2>{});
    if (nk == 3) run(Planes<3>{});
    if (nk == 4) run(Planes<4>{});
    // columns that no update writes keep what they were: all from `hi` on, and Hx of column 0
    auto store = [&](const float *in, float *out, float4 v, int hi, bool lo) {
        const float4 o = *reinterpret_cast<const float4 *>(in);
        *reinterpret_cast<float4 *>(out) = make_float4(col < hi && !lo ? v.x : o.x, col + 1 < hi ? v.y : o.y,
                                                       col + 2 < hi ? v.z : o.z, col + 3 < hi ? v.w : o.w);
    };
    if (inrow)
#pragma unroll
        for (int p = 0; p < KZ; ++p)
            if (p < nk) {
                const long long c = gidx(g, 0, j, k0 + p) + col;
                store(A.in + c, A.out + c, lds4(srow(XE, w, p, 0)), nx, false);
                store(A.in + c + g.comp, A.out + c + g.comp, Ey[p], nx + 1, false);
                store(A.in + c + 2 * g.comp, A.out + c + 2 * g.comp, Ez[p], nx + 1, false);
                store(A.in + c + 3 * g.comp, A.out + c + 3 * g.comp, lds4(srow(XH, w, p, 0)), nx, lane == 0);
                store(A.in + c + 4 * g.comp, A.out + c + 4 * g.comp, Hy[p], nx, false);
                store(A.in + c + 5 * g.comp, A.out + c + 5 * g.comp, lds4(srow(XH, w, p, 1)), nx, false);
            }
    if (dead) atomicOr(A.flags, 1);
}

struct ResState {
    int by, bz;
    unsigned tag;             // tag of the next launch's E^n
    uint4 *xch;
    SourceStep *ss;           // [RES_STEPS]
    bool probes_ok;           // the detectors' records fit
    int2 *bricks, *rec;
    float *ey;
    float *rbuf;              // [RES_STEPS][6 np]
};

void (*kernel(const fdtd_ctx *h))(ResArgs) { return h->boundary == FDTD_MUR1 ? k_res<true> : k_res<false>; }

void free_records(ResState *st) {
    if (st->bricks) cudaFree(st->bricks);
    if (st->rec) cudaFree(st->rec);
    if (st->ey) cudaFree(st->ey);
    if (st->rbuf) cudaFree(st->rbuf);
    st->bricks = nullptr;
    st->rec = nullptr;
    st->ey = nullptr;
    st->rbuf = nullptr;
}

// Detector records per brick; slot 6 t + v of detector t in the order in which
// `readout` takes the six values.  False when a brick would hold too many or
// memory runs out.
bool build_records(fdtd_ctx *h, ResState *st) {
    st->probes_ok = false;
    free_records(st);
    if (h->np == 0) return st->probes_ok = true;
    const Grid &g = h->g;
    const int bricks = st->by * st->bz;
    try {
        auto brick_of = [](int i, int n, int b) {   // the b-th of n near-equal parts that holds node i
            int p = (int)((long long)i * b / (n + 1));
            while ((long long)(p + 1) * (n + 1) / b <= i) ++p;
            while ((long long)p * (n + 1) / b > i) --p;
            return p;
        };
        const size_t n = 6 * (size_t)h->np;
        std::vector<int> key(n);
        std::vector<int2> off((size_t)bricks + 1, make_int2(0, 0)), val(n), rec(n);
        for (int t = 0; t < h->np; ++t) {
            const int i = h->h_ijk[3 * t], j = h->h_ijk[3 * t + 1], k = h->h_ijk[3 * t + 2];
            const int at[6][4] = {{0, i - 1, j, k}, {0, i, j, k}, {1, i, j - 1, k}, {1, i, j, k}, {2, i, j, k - 1}, {2, i, j, k}};
            for (int v = 0; v < 6; ++v) {
                const int bj = brick_of(at[v][2], g.ny, st->by), bk = brick_of(at[v][3], g.nz, st->bz), b = bk * st->by + bj;
                const int r = at[v][2] - (int)((long long)bj * (g.ny + 1) / st->by);
                const int rp = r * KZ + at[v][3] - (int)((long long)bk * (g.nz + 1) / st->bz);
                key[6 * t + v] = b;
                val[6 * t + v] = make_int2(at[v][0] == 1 ? EY_REC + rp * COLS + at[v][1]
                                                         : (2 * rp + at[v][0] / 2) * COLS + at[v][1], 6 * t + v);
                off[b + 1].x++;
                if (at[v][0] == 1) off[b].y |= 1 << r;
            }
        }
        for (int b = 1; b <= bricks; ++b) {
            if (off[b].x > MAX_REC) return false;
            off[b].x += off[b - 1].x;
        }
        std::vector<int2> at(off);
        for (size_t q = 0; q < n; ++q) rec[at[key[q]].x++] = val[q];
        if (cudaMalloc(&st->bricks, off.size() * sizeof(int2)) != cudaSuccess ||
            cudaMalloc(&st->rec, n * sizeof(int2)) != cudaSuccess ||
            cudaMalloc(&st->ey, sizeof(float) * EYROWS * bricks) != cudaSuccess ||
            cudaMalloc(&st->rbuf, sizeof(float) * RES_STEPS * n) != cudaSuccess ||
            cudaMemcpy(st->bricks, off.data(), off.size() * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(st->rec, rec.data(), n * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess) {
            cudaGetLastError();
            free_records(st);
            return false;
        }
    } catch (const std::bad_alloc &) {
        return false;
    }
    return st->probes_ok = true;
}

}  // namespace

// Bricks for the grid, or no resident path (h->res stays null): up to 128
// columns of nodes, no CPML, bricks of two or more rows and planes, one per SM.
// Among the splits that fit, the smallest brick.
void res_prepare(fdtd_ctx *h) {
    const Grid &g = h->g;
    if (h->P > 0 || g.nx > COLS - 1 || h->num_sms < 1) return;
    int by = 0, bz = 0, best = RW * KZ + 1;
    for (int y = (g.ny + 1 + RW - 1) / RW; 2 * y <= g.ny + 1; ++y)
        for (int z = (g.nz + 1 + KZ - 1) / KZ; 2 * z <= g.nz + 1 && y * z <= h->num_sms; ++z) {
            const int cells = ((g.ny + y) / y) * ((g.nz + z) / z);
            if (cells < best) {
                best = cells;
                by = y;
                bz = z;
            }
        }
    if (by == 0) return;
    int coop = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->dev) != cudaSuccess || !coop ||
        cudaFuncSetAttribute(kernel(h), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RES_SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel(h), NTB, RES_SMEM) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return;
    }
    ResState *st = new (std::nothrow) ResState();
    if (!st) return;
    st->by = by;
    st->bz = bz;
    st->tag = 1;              // the exchange words start with tag 0
    st->probes_ok = true;     // no detectors yet
    const size_t bytes = sizeof(uint4) * X_WORDS * (size_t)by * bz;
    if (cudaMalloc(&st->xch, bytes) != cudaSuccess || cudaMalloc(&st->ss, sizeof(SourceStep) * RES_STEPS) != cudaSuccess ||
        cudaMemsetAsync(st->xch, 0, bytes, h->stream) != cudaSuccess) {
        cudaGetLastError();
        if (st->xch) cudaFree(st->xch);
        if (st->ss) cudaFree(st->ss);
        delete st;
        return;
    }
    h->res = st;
}

void res_release(fdtd_ctx *h) {
    ResState *st = static_cast<ResState *>(h->res);
    if (!st) return;
    free_records(st);
    cudaFree(st->xch);
    cudaFree(st->ss);
    delete st;
    h->res = nullptr;
}

// Whether the resident path takes the handle's next steps: not while launches
// are timed (those are single steps).  The caller leaves it out while the stream
// is captured: a replay would find its exchange tags already there.
bool res_ready(const fdtd_ctx *h) {
    const ResState *st = static_cast<const ResState *>(h->res);
    return st && !h->timing.on && st->probes_ok;
}

void res_set_probes(fdtd_ctx *h) {
    if (h->res) build_records(h, static_cast<ResState *>(h->res));
}

int res_steps() { return RES_STEPS; }

// n <= RES_STEPS steps on stream s, detectors included; false if the launch was refused.
bool launch_res(fdtd_ctx *h, int n, cudaStream_t s) {
    ResState *st = static_cast<ResState *>(h->res);
    ResArgs a;
    a.g = h->g;
    a.in = h->fields[h->cur];
    a.out = h->fields[h->cur ^ 1];
    a.kE = (float)h->kE;
    a.kH = (float)h->kH;
    a.m = (float)h->mur_m;
    a.by = st->by;
    a.bz = st->bz;
    a.n = n;
    a.tag0 = st->tag;
    a.xch = st->xch;
    a.src = h->src;
    a.ss = st->ss;
    a.bricks = h->np > 0 ? st->bricks : nullptr;
    a.rec = st->rec;
    a.ey = st->ey;
    a.rbuf = st->rbuf;
    a.slots = 6 * h->np;
    a.flags = h->d_flags;
    if (h->src.active) {
        k_res_source<<<n, 32, 0, s>>>(h->src, h->steps, st->ss);
        h->launches++;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(st->by * st->bz));
    cfg.blockDim = dim3(NTB);
    cfg.dynamicSmemBytes = RES_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel(h), a) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    h->launches++;
    st->tag += (unsigned)n + 1;
    if (h->np > 0) {
        launch_record_probes(h, s, st->rbuf, n);
        h->launches++;
    }
    h->cur ^= 1;
    h->steps += n;
    return true;
}

}  // namespace fdtd
