// swe_prep.cu -- grid pre-processing of libswe (Sections 3.8 and 3.9):
// corner bathymetry from cell averages, land erosion, refinement and
// coarsening by two. The corner bathymetry is a march, a warp per strip of
// columns, bound by instruction issue; the others are memory-bound stencils, two
// or four cells per thread with vector loads and stores where the caller's layout
// allows them, else one. Nothing here allocates.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <type_traits>

#include "../../include/swe.h"
#include "swe_kernels.h"

namespace {

using swe::kLand;

constexpr int kMaxIter = 4096;           // iterations whose statistics fit the work area
constexpr int kBX = 32, kBY = 8;

int prep_fail(cudaError_t e) { return swe::record_cuda_error(e); }

long long round_up(long long v, long long m) { return (v + m - 1) / m * m; }

dim3 grid_for(long long nx, long long ny) {
    return dim3((unsigned)((nx + kBX - 1) / kBX), (unsigned)((ny + kBY - 1) / kBY));
}

// Non-negative floats order like their bit patterns.
__device__ __forceinline__ void atomic_max_nonneg(unsigned int *acc, float v) {
    atomicMax(acc, __float_as_uint(v));
}

// Block maximum of v over the threads with `have`, one atomic per block
// (every thread of the block must call it).
__device__ __forceinline__ void block_max_to(unsigned int *acc, float v, bool have) {
    __shared__ float part[kBX * kBY / 32];
    v = have ? v : 0.f;
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0 && acc) {
        float m = 0.f;
        for (int w = 0; w < kBX * kBY / 32; w++) m = fmaxf(m, part[w]);
        atomic_max_nonneg(acc, m);
    }
}

// ---------------------------------------------------------------------------
// corner bathymetry (Section 3.8), FP32: GB300's FP64 rate is a small
// fraction of its FP32 rate, and the corners feed the FP32 stage kernels

// max |Hm - H*(i, j)| over the cells -> *acc, H* the mean of the cell's four
// corners (the misfit of the final corners).
__global__ void __launch_bounds__(kBX * kBY) residual_kernel(const float *Hm, long long pitch,
                                                             const float *Hc, long long cpitch,
                                                             int nx, int ny, unsigned int *acc) {
    const int i = blockIdx.x * kBX + threadIdx.x % kBX;
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    const bool in = i < nx && j < ny;
    float r = 0.f;
    if (in) {
        const float *c = Hc + (long long)j * cpitch + i;
        const float mid = 0.25f * (((c[0] + c[1]) + c[cpitch]) + c[cpitch + 1]);
        r = Hm[(long long)j * pitch + i] - mid;
    }
    block_max_to(acc, fabsf(r), in);
}

// The smaller magnitude of a and b with the product of their signs; first: NaN
// where either is.
__device__ __forceinline__ float min_xor_nan(float a, float b) {
    float r;
    asm("min.NaN.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float min_xor(float a, float b) {
    float r;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Generalised minmod of (theta b, (b + f)/2, theta f) over theta in five
// operations, with c = 1 / (2 theta) (zero where b or f is NaN).
__device__ __forceinline__ float limited(float b, float f, float c) {
    const float m = fmaxf(min_xor_nan(b, f), 0.f);
    return min_xor(m, c * (b + f));
}

// One iteration of the corner reconstruction (INIT: the initial guess, X
// unused). A warp marches up a strip of columns with everything in registers;
// lane l holds corner and cell column c = 26 strip - 3 + l, and as corner row
// k arrives
//   A  the field F whose slopes are taken on cell row k - 1: Hm itself for the
//      initial guess, else the residual dH = Hm - H*(i, j) of X;
//   B  eqn:recon_1: its limited slopes along x, and those along y of cell row
//      k - 2 (beyond an edge a value is linearly extrapolated, so a cell at an
//      edge has the same difference on both sides);
//   C  eqn:recon_2, eqn:recon_3: T = X + the mean of the planar estimates of
//      the cells meeting at a corner of row k - 2;
//   D  the smoothing pass Y = T + w (mean of T's 4 neighbours - T) of corner
//      row k - 3 (beyond an edge T is extrapolated: the two neighbours
//      across it sum to 2 T); the initial guess is T as it stands.
// The strip's stencil reaches three columns to each side, so 26 of 32 lanes
// produce output, and an item of `rows` corner rows marches rows + 6. The
// misfit max|dH| of X and the largest change max|Y - X| go to misfit and
// change unless they are NULL.
//
// Bound by instruction issue: 2048 x 1500 takes 10.2 M warp instructions an
// iteration (106 thread instructions per corner) and 18 us, where the same on
// shared-memory tiles took 37.4 M and 45 us (halo recomputation, index
// arithmetic and every intermediate through shared memory). Loading one row
// ahead left it waiting on loads (23 us); the edge logic in every row took
// 21.1 M instructions (33 us). Launches that may start while the iteration
// before drains took ten iterations with the erosion from 197 to 175 us.
constexpr int kBathyStrip = 26, kBathyWarps = 4;

template <bool INIT, bool STATS>
__global__ void __launch_bounds__(kBathyWarps * 32) bathy_march_kernel(
    const float *Hm, long long pitch, int nx, int ny, const float *X, long long xp, float *Y, long long yp,
    float half_theta, float inv_2theta, float wgt, int rows, unsigned int *misfit, unsigned int *change) {
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = (blockIdx.x * kBathyWarps + warp) * kBathyStrip - 3;
    const int c = base + lane;
    const int J0 = blockIdx.y * rows, J1 = min(J0 + rows, ny + 1);
    float mis = 0.f, chg = 0.f;
    // the next iteration's blocks may start; this one's first loads need the
    // iteration before it. That one, and the two before it, may still run while
    // this block is resident, so a line of either plane that an L1 holds can be
    // two iterations old and no plane is read-only for this kernel's lifetime:
    // the planes are read from L2 (__ldcg), never through the non-coherent path.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (base + 3 <= nx) {                        // (warp-uniform: the strip has a corner)
        const bool corner = c >= 0 && c <= nx, cell = c >= 0 && c < nx;
        const bool out = lane >= 3 && lane < 3 + kBathyStrip && c <= nx;
        const bool edge = base <= 0 || base + 32 >= nx;     // (warp-uniform) some lane is at or beyond an edge
        const bool rim = c == 0 || c == nx;
        const float cx = rim ? 1.f : 0.5f;       // one over the cell columns meeting at the corner
        float x1 = 0.f, x2 = 0.f, x3 = 0.f;      // X of corner rows k-1, k-2, k-3
        float s1 = 0.f, h1 = 0.f;                // X summed along x and Hm of row k-1
        float D2 = 0.f, A2 = 0.f, B2 = 0.f, dS = 0.f;   // cell row k-2: F, F -+ half slope, difference below
        float n3 = 0.f;                          // cell row k-3: estimates at its north corners
        float T3 = 0.f, T4 = 0.f;                // T of corner rows k-3 and k-4
        const float *px = X + (long long)(J0 - 3) * xp + c, *ph = Hm + (long long)(J0 - 3) * pitch + c;
        float *py = Y + (long long)(J0 - 6) * yp + c;       // the row written
        const auto row = [&](int k, float x, float h, auto general) {
            constexpr bool G = decltype(general)::value;   // some lane or row at an edge
            // A: cell row k - 1
            const float s = INIT ? 0.f : x + __shfl_down_sync(full, x, 1);
            float D = INIT ? h1 : fmaf(-0.25f, s1 + s, h1);
            if (G && (k - 1 < 0 || k - 1 >= ny || !cell)) D = 0.f;
            if (STATS && out && k - 1 >= J0 && k - 1 < J1) mis = fmaxf(mis, fabsf(D));
            // B: slopes
            float b = D - __shfl_up_sync(full, D, 1), f = __shfl_down_sync(full, b, 1);
            if (G) {
                if (c == 0) b = nx > 1 ? f : 0.f;
                if (c == nx - 1) f = nx > 1 ? b : 0.f;
                if (!cell) b = 0.f;
            }
            const float lx = limited(b, f, inv_2theta);
            float dN = D - D2, lo = dS;
            if (G && k - 1 >= ny) dN = ny > 1 ? dS : 0.f;
            if (G && k - 2 <= 0) lo = ny > 1 ? dN : 0.f;
            float hy = half_theta * limited(lo, dN, inv_2theta);
            if (G && (k - 2 < 0 || k - 2 >= ny || !cell)) hy = 0.f;
            // C: T of corner row k - 2
            const float sumD = A2 + __shfl_up_sync(full, B2, 1), sumh = hy + __shfl_up_sync(full, hy, 1);
            const float scale = G ? cx * (k - 2 <= 0 || k - 2 >= ny ? 1.f : 0.5f) : 0.25f;
            const float T2 = fmaf(scale, n3 + (sumD - sumh), x2);
            n3 = sumD + sumh;
            // D: output corner row k - 3
            float v = T3;
            if (!INIT) {
                float we = __shfl_up_sync(full, T3, 1) + __shfl_down_sync(full, T3, 1), sn = T4 + T2;
                if (G && rim) we = 2.f * T3;
                if (G && (k - 3 <= 0 || k - 3 >= ny)) sn = 2.f * T3;
                v = fmaf(wgt, fmaf(0.25f, we + sn, -T3), T3);
            }
            if (out && k - 3 >= J0 && k - 3 < J1) {
                *py = v;
                if (STATS) chg = fmaxf(chg, fabsf(v - x3));
            }
            py += yp;
            if (STATS) x3 = x2;
            x2 = x1; x1 = x;
            s1 = s; h1 = h;
            D2 = D; A2 = fmaf(-half_theta, lx, D); B2 = fmaf(half_theta, lx, D); dS = dN;
            T4 = T3; T3 = T2;
        };
        // rows in groups of four, the loads of a group in flight while the one
        // before is worked on; groups whose march meets no edge of the plane
        // run without the edge logic (k0: the group's first row)
        const auto inside = [&](int k0) { return !edge && k0 >= 4 && k0 + 4 <= ny; };
        const auto load = [&](int k0, float *x, float *h) {
            if (inside(k0)) {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    x[q] = INIT ? 0.f : __ldcg(px + q * xp);
                    h[q] = __ldcg(ph + q * pitch);
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const int k = k0 + q;
                    x[q] = !INIT && corner && k >= 0 && k <= ny ? __ldcg(px + q * xp) : 0.f;
                    h[q] = cell && k >= 0 && k < ny ? __ldcg(ph + q * pitch) : 0.f;
                }
            }
            px += 4 * xp;
            ph += 4 * pitch;
        };
        float x[4], h[4];
        load(J0 - 3, x, h);
        for (int k0 = J0 - 3; k0 < J1 + 3; k0 += 4) {
            float xn[4], hn[4];
            load(k0 + 4, xn, hn);
            if (inside(k0)) {
#pragma unroll
                for (int q = 0; q < 4; q++) row(k0 + q, x[q], h[q], std::false_type());
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++) row(k0 + q, x[q], h[q], std::true_type());
            }
#pragma unroll
            for (int q = 0; q < 4; q++) { x[q] = xn[q]; h[q] = hn[q]; }
        }
    }
    if (!STATS) return;
    __shared__ float part[2][kBathyWarps];
    for (int o = 16; o > 0; o >>= 1) {
        mis = fmaxf(mis, __shfl_xor_sync(full, mis, o));
        chg = fmaxf(chg, __shfl_xor_sync(full, chg, o));
    }
    if (lane == 0) { part[0][warp] = mis; part[1][warp] = chg; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kBathyWarps; w++) { mis = fmaxf(mis, part[0][w]); chg = fmaxf(chg, part[1][w]); }
        if (misfit) atomic_max_nonneg(misfit, mis);
        atomic_max_nonneg(change, chg);
    }
}

// Corner rows per item: the six halo rows weigh little on long items, but
// small planes are cut finer so that the chip has some 32 warps per SM
// (2048 x 1500, ten iterations with the erosion before them: 213, 206, 197 and
// 197 us for 20, 24, 32 and 48 warps).
int bathy_rows(int nx, int ny) {
    const long long strips = (nx + 1 + kBathyStrip - 1) / kBathyStrip;
    const long long want = 152LL * 32;
    long long rows = strips * (ny + 1) / want;
    return (int)(rows < 4 ? 4 : rows > 64 ? 64 : rows);
}

// Work area: one corner plane (the iterations alternate between it and the
// caller's corners, ending in the caller's) and the per-iteration statistics.
struct BathyWork {
    float *corners;
    unsigned int *stats;
    long long tp;
};

BathyWork bathy_layout(void *work, int nx, int ny) {
    BathyWork w;
    w.tp = round_up((long long)nx + 1, 32);
    char *p = static_cast<char *>(work);
    w.corners = reinterpret_cast<float *>(p);
    w.stats = reinterpret_cast<unsigned int *>(p + round_up(w.tp * (ny + 1) * 4, 256));
    return w;
}

size_t bathy_bytes(int nx, int ny) {
    const long long tp = round_up((long long)nx + 1, 32);
    return (size_t)round_up(tp * (ny + 1) * 4, 256) + 2 * kMaxIter * sizeof(unsigned int);
}

// ---------------------------------------------------------------------------
// land erosion (Section 3.8)

// One cell (i, j) of the erosion step (shared by the one-cell kernel and the
// ragged end of a row in the four-cell kernel).
__device__ __forceinline__ void erode_cell(const unsigned char *land, const float *eta, const float *Hm,
                                           long long pitch, int nx, int ny, float land_depth, int i, int j,
                                           unsigned char *land_out, float *eta_out, float *Hm_out) {
    const long long s = (long long)j * pitch + i;
    const bool l = land[s] != 0;
    // outside the domain counts as land
    const bool lw = i == 0 || land[s - 1] != 0, le = i == nx - 1 || land[s + 1] != 0;
    const bool ls = j == 0 || land[s - pitch] != 0, ln = j == ny - 1 || land[s + pitch] != 0;
    const bool stays = l && lw && le && ls && ln;
    const bool opened = l && !stays;
    float e = eta[s], h = Hm[s];
    if (opened) {
        // gray dilation: the largest eta among the water 4-neighbours
        float m = -INFINITY;
        if (!lw) m = fmaxf(m, eta[s - 1]);
        if (!le) m = fmaxf(m, eta[s + 1]);
        if (!ls) m = fmaxf(m, eta[s - pitch]);
        if (!ln) m = fmaxf(m, eta[s + pitch]);
        e = m;
        h = land_depth;
    }
    land_out[s] = stays ? 1 : 0;
    eta_out[s] = e;
    Hm_out[s] = h;
}

__global__ void __launch_bounds__(kBX * kBY) erode_kernel(const unsigned char *land, const float *eta,
                                                          const float *Hm, long long pitch, int nx,
                                                          int ny, float land_depth, unsigned char *land_out,
                                                          float *eta_out, float *Hm_out) {
    const int i = blockIdx.x * kBX + threadIdx.x % kBX;
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    if (i >= nx || j >= ny) return;
    erode_cell(land, eta, Hm, pitch, nx, ny, land_depth, i, j, land_out, eta_out, Hm_out);
}

// The same step, four consecutive cells per thread with vector loads and
// stores (pitch a multiple of 4, float planes 16-byte and byte planes
// 4-byte aligned): five byte-plane loads and two float4 loads for four
// cells instead of twenty-eight scalar loads. The same selections and the
// same order of maxima as erode_cell, so the same bits.
__global__ void __launch_bounds__(kBX * kBY) erode4_kernel(const unsigned char *land, const float *eta,
                                                           const float *Hm, long long pitch, int nx,
                                                           int ny, float land_depth, unsigned char *land_out,
                                                           float *eta_out, float *Hm_out) {
    const int i0 = 4 * (blockIdx.x * kBX + threadIdx.x % kBX);
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    if (i0 >= nx || j >= ny) return;
    if (i0 + 4 > nx) {                          // the ragged end of a row
        for (int i = i0; i < nx; i++)
            erode_cell(land, eta, Hm, pitch, nx, ny, land_depth, i, j, land_out, eta_out, Hm_out);
        return;
    }
    const long long s = (long long)j * pitch + i0;
    const uchar4 one = make_uchar4(1, 1, 1, 1);
    const uchar4 L = *reinterpret_cast<const uchar4 *>(land + s);
    const uchar4 LS = j > 0 ? *reinterpret_cast<const uchar4 *>(land + s - pitch) : one;
    const uchar4 LN = j < ny - 1 ? *reinterpret_cast<const uchar4 *>(land + s + pitch) : one;
    const bool lW = i0 == 0 || land[s - 1] != 0;
    const bool lE = i0 + 4 >= nx || land[s + 4] != 0;
    const float4 E = *reinterpret_cast<const float4 *>(eta + s);
    const float4 D = *reinterpret_cast<const float4 *>(Hm + s);
    const bool l[4] = {L.x != 0, L.y != 0, L.z != 0, L.w != 0};
    const bool ls[4] = {LS.x != 0, LS.y != 0, LS.z != 0, LS.w != 0};
    const bool ln[4] = {LN.x != 0, LN.y != 0, LN.z != 0, LN.w != 0};
    const float ein[4] = {E.x, E.y, E.z, E.w};
    float e[4] = {E.x, E.y, E.z, E.w}, h[4] = {D.x, D.y, D.z, D.w};
    unsigned char stay[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const bool lw = k == 0 ? lW : l[k - 1], le = k == 3 ? lE : l[k + 1];
        const bool stays = l[k] && lw && le && ls[k] && ln[k];
        if (l[k] && !stays) {
            float m = -INFINITY;
            if (!lw) m = fmaxf(m, k == 0 ? eta[s - 1] : ein[k - 1]);
            if (!le) m = fmaxf(m, k == 3 ? eta[s + 4] : ein[k + 1]);
            if (!ls[k]) m = fmaxf(m, eta[s + k - pitch]);
            if (!ln[k]) m = fmaxf(m, eta[s + k + pitch]);
            e[k] = m;
            h[k] = land_depth;
        }
        stay[k] = stays ? 1 : 0;
    }
    *reinterpret_cast<uchar4 *>(land_out + s) = make_uchar4(stay[0], stay[1], stay[2], stay[3]);
    *reinterpret_cast<float4 *>(eta_out + s) = make_float4(e[0], e[1], e[2], e[3]);
    *reinterpret_cast<float4 *>(Hm_out + s) = make_float4(h[0], h[1], h[2], h[3]);
}

// ---------------------------------------------------------------------------
// refinement and coarsening by two (Section 3.9), FP32

__device__ __forceinline__ bool corner_land(const float *H, long long cp, int j, int i) {
    const float *c = H + (long long)j * cp + i;
    return (c[0] == kLand) | (c[1] == kLand) | (c[cp] == kLand) | (c[cp + 1] == kLand);
}

struct Planes3 {
    const float *q[3];
};
struct OutPlanes3 {
    float *q[3];
};

// The four children of a water cell with value c and one-sided
// differences bx, fx (x) and by, fy (y): limited slopes, children at
// x +- 1/4, y +- 1/4 of the cell (lo: the lower row of children). theta: 1 /
// (2 theta) and theta / 4.
__device__ __forceinline__ void refine_children(float c, float bx, float fx, float by, float fy, float2 theta,
                                                float2 &lo, float2 &hi) {
    const float sx = theta.y * limited(bx, fx, theta.x), sy = theta.y * limited(by, fy, theta.x);
    lo.x = (c - sx) - sy;
    lo.y = (c + sx) - sy;
    hi.x = (c - sx) + sy;
    hi.y = (c + sx) + sy;
}

// One coarse cell (i, j) of the refinement (the one-cell kernel, and the odd
// last cell of a row in the two-cell kernel).
__device__ __forceinline__ void refine_cell(const Planes3 &in, long long pitch, const float *H, long long cp,
                                            int nx, int ny, float2 theta, const OutPlanes3 &out, long long fp,
                                            int i, int j) {
    const bool land = corner_land(H, cp, j, i);
    // a neighbour that is land or outside gives a zero one-sided difference
    const bool nw = i > 0 && !corner_land(H, cp, j, i - 1);
    const bool ne = i < nx - 1 && !corner_land(H, cp, j, i + 1);
    const bool ns = j > 0 && !corner_land(H, cp, j - 1, i);
    const bool nn = j < ny - 1 && !corner_land(H, cp, j + 1, i);
    const long long s = (long long)j * pitch + i;
    const long long f0 = (long long)(2 * j) * fp + 2 * i;
    for (int v = 0; v < 3; v++) {
        float2 lo = make_float2(0.f, 0.f), hi = make_float2(0.f, 0.f);
        if (!land) {
            const float *p = in.q[v] + s;
            const float c = p[0];
            refine_children(c, nw ? c - p[-1] : 0.f, ne ? p[1] - c : 0.f, ns ? c - p[-pitch] : 0.f,
                            nn ? p[pitch] - c : 0.f, theta, lo, hi);
        }
        *reinterpret_cast<float2 *>(out.q[v] + f0) = lo;
        *reinterpret_cast<float2 *>(out.q[v] + f0 + fp) = hi;
    }
}

__global__ void __launch_bounds__(kBX * kBY) refine_cells_kernel(Planes3 in, long long pitch, const float *H,
                                                                 long long cp, int nx, int ny, float2 theta,
                                                                 OutPlanes3 out, long long fp) {
    const int i = blockIdx.x * kBX + threadIdx.x % kBX;
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    if (i >= nx || j >= ny) return;
    refine_cell(in, pitch, H, cp, nx, ny, theta, out, fp, i, j);
}

// Fine intersections of the coarse corners a = (J, I), b = (J, I + 1), c =
// (J + 1, I), d = (J + 1, I + 1): the midpoints of a|b and a|c, the centre.
__device__ __forceinline__ float mid2(float a, float b) {
    return (a == kLand || b == kLand) ? kLand : 0.5f * (a + b);
}
__device__ __forceinline__ float mid4(float a, float b, float c, float d) {
    const bool l = (a == kLand) | (b == kLand) | (c == kLand) | (d == kLand);
    return l ? kLand : 0.25f * (((a + b) + c) + d);
}

__device__ __forceinline__ void store4(float *o, float4 v, bool vec) {
    if (vec) {
        *reinterpret_cast<float4 *>(o) = v;
    } else {
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
}

// The same refinement with the fine corners, two coarse cells (i0, i0 + 1) per
// thread (coarse pitch even, coarse planes 8-byte aligned; fine pitch a
// multiple of 4, fine planes 16-byte aligned; corner planes laid out so too are
// read and written as vectors, vec_H and vec_F): float2 loads, the land of the
// six cells around from one read of their corners, which also gives the fine
// corners of rows 2j and 2j + 1 (row j = ny only has those), and float4 stores.
// The same selections and arithmetic as refine_cell and refine_corners_kernel,
// so the same bits. HBM-bound.
__global__ void __launch_bounds__(kBX * kBY) refine2_kernel(Planes3 in, long long pitch, const float *H,
                                                            long long cp, int nx, int ny, float2 theta,
                                                            OutPlanes3 out, long long fp, float *F, long long fcp,
                                                            bool vec_H, bool vec_F) {
    const int i0 = 2 * (blockIdx.x * kBX + threadIdx.x % kBX);
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    if (i0 > nx || j > ny) return;
    const bool has_w = i0 > 0, two = i0 + 1 < nx, has_e = i0 + 2 < nx, has_s = j > 0, top = j == ny;
    // corners of rows j, j + 1 at columns i0 - 1 .. i0 + 3 (where they exist)
    const float *c = H + (long long)j * cp + i0, *cu = top ? c : c + cp;
    const bool any1 = i0 + 1 <= nx, any2 = i0 + 2 <= nx, any3 = i0 + 3 <= nx;
    float A[5], B[5];
    if (vec_H && any3) {
        const float2 a0 = *reinterpret_cast<const float2 *>(c), a1 = *reinterpret_cast<const float2 *>(c + 2);
        const float2 b0 = *reinterpret_cast<const float2 *>(cu), b1 = *reinterpret_cast<const float2 *>(cu + 2);
        A[1] = a0.x; A[2] = a0.y; A[3] = a1.x; A[4] = a1.y;
        B[1] = b0.x; B[2] = b0.y; B[3] = b1.x; B[4] = b1.y;
    } else {
        A[1] = c[0]; A[2] = any1 ? c[1] : 0.f; A[3] = any2 ? c[2] : 0.f; A[4] = any3 ? c[3] : 0.f;
        B[1] = cu[0]; B[2] = any1 ? cu[1] : 0.f; B[3] = any2 ? cu[2] : 0.f; B[4] = any3 ? cu[3] : 0.f;
    }
    A[0] = has_w ? c[-1] : 0.f;
    B[0] = has_w ? cu[-1] : 0.f;
    // fine corners of rows 2j and 2j + 1, columns 2 i0 .. 2 i0 + 3 (as far as 2 nx)
    float *o = F + (long long)(2 * j) * fcp + 2 * i0;
    if (two) {
        store4(o, make_float4(A[1], mid2(A[1], A[2]), A[2], mid2(A[2], A[3])), vec_F);
        if (!top)
            store4(o + fcp, make_float4(mid2(A[1], B[1]), mid4(A[1], A[2], B[1], B[2]), mid2(A[2], B[2]),
                                        mid4(A[2], A[3], B[2], B[3])), vec_F);
    } else {
        o[0] = A[1];
        if (!top) o[fcp] = mid2(A[1], B[1]);
        if (any1) {                              // the odd last cell of a row
            o[1] = mid2(A[1], A[2]);
            o[2] = A[2];
            if (!top) {
                o[fcp + 1] = mid4(A[1], A[2], B[1], B[2]);
                o[fcp + 2] = mid2(A[2], B[2]);
            }
        }
    }
    if (two && !has_e) {                         // the last corner column of an even row
        o[4] = A[3];
        if (!top) o[fcp + 4] = mid2(A[3], B[3]);
    }
    if (top || i0 >= nx) return;
    if (!two) {
        refine_cell(in, pitch, H, cp, nx, ny, theta, out, fp, i0, j);
        return;
    }
    const bool has_n = j < ny - 1;
    bool a[5], b[5];                             // corner is LAND, rows j and j + 1
#pragma unroll
    for (int x = 0; x < 5; x++) {
        const bool ok = (x > 0 || has_w) && (x < 4 || has_e);
        a[x] = ok && A[x] == kLand;
        b[x] = ok && B[x] == kLand;
    }
    const bool landW = a[0] | a[1] | b[0] | b[1], land0 = a[1] | a[2] | b[1] | b[2];
    const bool land1 = a[2] | a[3] | b[2] | b[3], landE = a[3] | a[4] | b[3] | b[4];
    bool landS0 = true, landS1 = true, landN0 = true, landN1 = true;
    if (has_s) {
        const float *d = c - cp;
        const bool s0 = d[0] == kLand, s1 = d[1] == kLand, s2 = d[2] == kLand;
        landS0 = s0 | s1 | a[1] | a[2];
        landS1 = s1 | s2 | a[2] | a[3];
    }
    if (has_n) {
        const float *d = c + 2 * cp;
        const bool n0 = d[0] == kLand, n1 = d[1] == kLand, n2 = d[2] == kLand;
        landN0 = b[1] | b[2] | n0 | n1;
        landN1 = b[2] | b[3] | n1 | n2;
    }
    const bool nw0 = has_w && !landW, ne0 = !land1, ns0 = has_s && !landS0, nn0 = has_n && !landN0;
    const bool nw1 = !land0, ne1 = has_e && !landE, ns1 = has_s && !landS1, nn1 = has_n && !landN1;
    const long long s = (long long)j * pitch + i0;
    const long long f0 = (long long)(2 * j) * fp + 2 * i0;
#pragma unroll
    for (int v = 0; v < 3; v++) {
        const float *p = in.q[v] + s;
        const float2 P = *reinterpret_cast<const float2 *>(p);
        const float pw = has_w ? p[-1] : 0.f, pe = has_e ? p[2] : 0.f;
        const float2 S = has_s ? *reinterpret_cast<const float2 *>(p - pitch) : make_float2(0.f, 0.f);
        const float2 N = has_n ? *reinterpret_cast<const float2 *>(p + pitch) : make_float2(0.f, 0.f);
        float2 lo0 = make_float2(0.f, 0.f), hi0 = lo0, lo1 = lo0, hi1 = lo0;
        if (!land0)
            refine_children(P.x, nw0 ? P.x - pw : 0.f, ne0 ? P.y - P.x : 0.f, ns0 ? P.x - S.x : 0.f,
                            nn0 ? N.x - P.x : 0.f, theta, lo0, hi0);
        if (!land1)
            refine_children(P.y, nw1 ? P.y - P.x : 0.f, ne1 ? pe - P.y : 0.f, ns1 ? P.y - S.y : 0.f,
                            nn1 ? N.y - P.y : 0.f, theta, lo1, hi1);
        *reinterpret_cast<float4 *>(out.q[v] + f0) = make_float4(lo0.x, lo0.y, lo1.x, lo1.y);
        *reinterpret_cast<float4 *>(out.q[v] + f0 + fp) = make_float4(hi0.x, hi0.y, hi1.x, hi1.y);
    }
}

// Fine intersections owned by coarse corner (J, I): (2J, 2I) and, where they
// exist, the edge midpoints (2J, 2I+1), (2J+1, 2I) and the centre (2J+1, 2I+1).
__global__ void __launch_bounds__(kBX * kBY) refine_corners_kernel(const float *H, long long cp, int nx, int ny,
                                                                   float *F, long long fcp) {
    const int I = blockIdx.x * kBX + threadIdx.x % kBX;
    const int J = blockIdx.y * kBY + threadIdx.x / kBX;
    if (I > nx || J > ny) return;
    const float *c = H + (long long)J * cp + I;
    float *o = F + (long long)(2 * J) * fcp + 2 * I;
    const float a = c[0];
    o[0] = a;
    if (I < nx) o[1] = mid2(a, c[1]);
    if (J < ny) o[fcp] = mid2(a, c[cp]);
    if (I < nx && J < ny) o[fcp + 1] = mid4(a, c[1], c[cp], c[cp + 1]);
}

// s / n for n = 1 .. 4: only a third needs a division.
__device__ __forceinline__ float mean_of(float s, float n) {
    return n == 3.f ? s / 3.f : s * (n == 4.f ? 0.25f : n == 2.f ? 0.5f : 1.f);
}

// One coarse cell (i, j) of the coarsening (the one-cell kernel, and the odd
// last cell of a row in the two-cell kernel).
__device__ __forceinline__ void coarsen_cell(const Planes3 &fin, long long fp, const float *Hf, long long fcp,
                                             const OutPlanes3 &out, long long pitch, int i, int j) {
    // the coarse cell is land if one of its sampled corners is
    const float *cc = Hf + (long long)(2 * j) * fcp + 2 * i;
    const bool cland = (cc[0] == kLand) | (cc[2] == kLand) | (cc[2 * fcp] == kLand) | (cc[2 * fcp + 2] == kLand);
    bool wet[4];
    float n_wet = 0.f;
    for (int b = 0; b < 2; b++)
        for (int a = 0; a < 2; a++) {
            wet[2 * b + a] = !corner_land(Hf, fcp, 2 * j + b, 2 * i + a);
            n_wet += wet[2 * b + a] ? 1.f : 0.f;
        }
    const long long f0 = (long long)(2 * j) * fp + 2 * i;
    for (int v = 0; v < 3; v++) {
        const float2 lo = *reinterpret_cast<const float2 *>(fin.q[v] + f0);
        const float2 hi = *reinterpret_cast<const float2 *>(fin.q[v] + f0 + fp);
        const float s = (((wet[0] ? lo.x : 0.f) + (wet[1] ? lo.y : 0.f)) + (wet[2] ? hi.x : 0.f)) +
                        (wet[3] ? hi.y : 0.f);
        out.q[v][(long long)j * pitch + i] = (cland || n_wet == 0.f) ? 0.f : mean_of(s, n_wet);
    }
}

__global__ void __launch_bounds__(kBX * kBY) coarsen_cells_kernel(Planes3 fin, long long fp, const float *Hf,
                                                                  long long fcp, int nx, int ny, OutPlanes3 out,
                                                                  long long pitch) {
    const int i = blockIdx.x * kBX + threadIdx.x % kBX;
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    if (i >= nx || j >= ny) return;
    coarsen_cell(fin, fp, Hf, fcp, out, pitch, i, j);
}

// The same coarsening with the coarse corners, two coarse cells (i0, i0 + 1)
// per thread (fine pitch a multiple of 4, fine planes 16-byte aligned; coarse
// pitch even, coarse planes 8-byte aligned; corner planes laid out so too are
// read and written as vectors, vec_F and vec_H): one read of the 3 x 5 fine
// corners they share, which holds the coarse corners of row j too (row j = ny
// only has those), float4 loads of the children, float2 stores. The same
// selections and arithmetic as coarsen_cell, so the same bits. HBM-bound.
__global__ void __launch_bounds__(kBX * kBY) coarsen2_kernel(Planes3 fin, long long fp, const float *Hf,
                                                             long long fcp, int nx, int ny, OutPlanes3 out,
                                                             long long pitch, float *H, long long cp, bool vec_F,
                                                             bool vec_H) {
    const int i0 = 2 * (blockIdx.x * kBX + threadIdx.x % kBX);
    const int j = blockIdx.y * kBY + threadIdx.x / kBX;
    if (i0 > nx || j > ny) return;
    const float *cc = Hf + (long long)(2 * j) * fcp + 2 * i0;
    float *o = H + (long long)j * cp + i0;
    if (i0 + 1 >= nx || j == ny) {               // the odd last cell of a row, the last corners
        for (int k = 0; k < 3 && i0 + k <= nx; k++)
            if (k < 2 || i0 + 2 == nx) o[k] = cc[2 * k];
        if (i0 < nx && i0 + 1 >= nx && j < ny) coarsen_cell(fin, fp, Hf, fcp, out, pitch, i0, j);
        return;
    }
    // fine corners of rows 2j .. 2j + 2, columns 2 i0 .. 2 i0 + 4: LAND?
    bool L[3][5];
#pragma unroll
    for (int b = 0; b < 3; b++) {
        const float *r = cc + b * fcp;
        const float4 h = vec_F ? *reinterpret_cast<const float4 *>(r) : make_float4(r[0], r[1], r[2], r[3]);
        const float h4 = r[4];
        L[b][0] = h.x == kLand; L[b][1] = h.y == kLand; L[b][2] = h.z == kLand; L[b][3] = h.w == kLand;
        L[b][4] = h4 == kLand;
        if (b == 0) {
            if (vec_H) *reinterpret_cast<float2 *>(o) = make_float2(h.x, h.z);
            else { o[0] = h.x; o[1] = h.z; }
            if (i0 + 2 == nx) o[2] = h4;
        }
    }
    bool cland[2], wet[2][4];
    float n_wet[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        cland[k] = L[0][2 * k] | L[0][2 * k + 2] | L[2][2 * k] | L[2][2 * k + 2];
        n_wet[k] = 0.f;
#pragma unroll
        for (int b = 0; b < 2; b++)
#pragma unroll
            for (int a = 0; a < 2; a++) {
                const int x = 2 * k + a;
                wet[k][2 * b + a] = !(L[b][x] | L[b][x + 1] | L[b + 1][x] | L[b + 1][x + 1]);
                n_wet[k] += wet[k][2 * b + a] ? 1.f : 0.f;
            }
    }
    const long long f0 = (long long)(2 * j) * fp + 2 * i0;
#pragma unroll
    for (int v = 0; v < 3; v++) {
        const float4 lo = *reinterpret_cast<const float4 *>(fin.q[v] + f0);
        const float4 hi = *reinterpret_cast<const float4 *>(fin.q[v] + f0 + fp);
        const float s0 = (((wet[0][0] ? lo.x : 0.f) + (wet[0][1] ? lo.y : 0.f)) + (wet[0][2] ? hi.x : 0.f)) +
                         (wet[0][3] ? hi.y : 0.f);
        const float s1 = (((wet[1][0] ? lo.z : 0.f) + (wet[1][1] ? lo.w : 0.f)) + (wet[1][2] ? hi.z : 0.f)) +
                         (wet[1][3] ? hi.w : 0.f);
        *reinterpret_cast<float2 *>(out.q[v] + (long long)j * pitch + i0) =
            make_float2((cland[0] || n_wet[0] == 0.f) ? 0.f : mean_of(s0, n_wet[0]),
                        (cland[1] || n_wet[1] == 0.f) ? 0.f : mean_of(s1, n_wet[1]));
    }
}

__global__ void __launch_bounds__(kBX * kBY) coarsen_corners_kernel(const float *Hf, long long fcp, int nx, int ny,
                                                                    float *H, long long cp) {
    const int I = blockIdx.x * kBX + threadIdx.x % kBX;
    const int J = blockIdx.y * kBY + threadIdx.x / kBX;
    if (I > nx || J > ny) return;
    H[(long long)J * cp + I] = Hf[(long long)(2 * J) * fcp + 2 * I];
}

bool aligned8(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; }

}  // namespace

extern "C" {

size_t swe_bathymetry_work_bytes(int nx, int ny) {
    if (nx < 1 || ny < 1) return 0;
    return bathy_bytes(nx, ny);
}

int swe_bathymetry_reconstruct(const float *Hm, long long pitch, int nx, int ny, float *Hc,
                               long long cpitch, void *work, int n_iter, double theta,
                               double smooth, double *stats, void *stream) {
    swe::TraceRange trace("swe_bathymetry_reconstruct");
    if (!Hm || !Hc || !work || nx < 1 || ny < 1 || pitch < nx || cpitch < (long long)nx + 1)
        return SWE_ERR_INVALID_ARG;
    if (n_iter < 0 || n_iter > kMaxIter || !(theta >= 1.0 && theta <= 2.0) ||
        !(smooth >= 0.0 && smooth <= 1.0))
        return SWE_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(work) & 255u) != 0) return SWE_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const BathyWork w = bathy_layout(work, nx, ny);
    const int rows = bathy_rows(nx, ny);
    const int strips = (nx + 1 + kBathyStrip - 1) / kBathyStrip;
    const dim3 grid((unsigned)((strips + kBathyWarps - 1) / kBathyWarps), (unsigned)((ny + 1 + rows - 1) / rows));
    const float ht = 0.5f * (float)theta, i2t = (float)(0.5 / theta), sm = (float)smooth;
    // (the statistics are gathered only for a caller that wants them)
    cudaError_t e = stats ? cudaMemsetAsync(w.stats, 0, 2 * (size_t)n_iter * sizeof(unsigned int), st) : cudaSuccess;
    if (e != cudaSuccess) return prep_fail(e);
    // corners after k iterations live in plane (n_iter - k) % 2: 0 the caller's, 1 the work area's
    float *plane[2] = {Hc, w.corners};
    const long long pp[2] = {cpitch, w.tp};
    int cur = n_iter % 2;
    const auto iteration = stats ? bathy_march_kernel<false, true> : bathy_march_kernel<false, false>;
    // launches that may start while the one before them drains
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof attr);
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kBathyWarps * 32);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const float *no_corners = nullptr;
    unsigned int *none = nullptr;
    e = cudaLaunchKernelEx(&cfg, bathy_march_kernel<true, false>, Hm, pitch, nx, ny, no_corners, 0LL, plane[cur], pp[cur],
                           ht, i2t, sm, rows, none, none);
    for (int k = 0; k < n_iter && e == cudaSuccess; k++) {
        // the misfit of the previous iteration's corners (none for the initial guess)
        e = cudaLaunchKernelEx(&cfg, iteration, Hm, pitch, nx, ny, (const float *)plane[cur], pp[cur], plane[cur ^ 1],
                               pp[cur ^ 1], ht, i2t, sm, rows, stats && k > 0 ? w.stats + 2 * (k - 1) : none,
                               stats ? w.stats + 2 * k + 1 : none);
        cur ^= 1;
    }
    if (e != cudaSuccess) return prep_fail(e);
    if (stats && n_iter > 0)
        residual_kernel<<<grid_for(nx, ny), kBX * kBY, 0, st>>>(Hm, pitch, Hc, cpitch, nx, ny,
                                                                w.stats + 2 * (n_iter - 1));
    if ((e = cudaGetLastError()) != cudaSuccess) return prep_fail(e);
    if (stats && n_iter > 0) {
        unsigned int bits[2 * kMaxIter];
        e = cudaMemcpyAsync(bits, w.stats, 2 * (size_t)n_iter * sizeof(unsigned int), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return prep_fail(e);
        for (int k = 0; k < 2 * n_iter; k++) {
            float f;
            memcpy(&f, &bits[k], sizeof f);
            stats[k] = f;
        }
    }
    return SWE_OK;
}

int swe_land_erode(const unsigned char *land, const float *eta, const float *Hm,
                   long long pitch, int nx, int ny, double land_depth,
                   unsigned char *land_out, float *eta_out, float *Hm_out, void *stream) {
    swe::TraceRange trace("swe_land_erode");
    if (!land || !eta || !Hm || !land_out || !eta_out || !Hm_out || nx < 1 || ny < 1 || pitch < nx)
        return SWE_ERR_INVALID_ARG;
    if ((const void *)land_out == (const void *)land || eta_out == eta || Hm_out == Hm)
        return SWE_ERR_INVALID_ARG;
    if (!(land_depth >= 0.0)) return SWE_ERR_INVALID_ARG;
    auto al = [](const void *p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; };
    if (pitch % 4 == 0 && al(land, 4) && al(land_out, 4) && al(eta, 16) && al(Hm, 16) && al(eta_out, 16) &&
        al(Hm_out, 16))
        erode4_kernel<<<grid_for(((long long)nx + 3) / 4, ny), kBX * kBY, 0, (cudaStream_t)stream>>>(
            land, eta, Hm, pitch, nx, ny, (float)land_depth, land_out, eta_out, Hm_out);
    else
        erode_kernel<<<grid_for(nx, ny), kBX * kBY, 0, (cudaStream_t)stream>>>(
            land, eta, Hm, pitch, nx, ny, (float)land_depth, land_out, eta_out, Hm_out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SWE_OK : prep_fail(e);
}

int swe_refine2(const float *eta, const float *hu, const float *hv, long long pitch,
                const float *H, long long cpitch, int nx, int ny, double theta,
                float *eta_f, float *hu_f, float *hv_f, long long fpitch, float *H_f,
                long long fcpitch, void *stream) {
    swe::TraceRange trace("swe_refine2");
    if (!eta || !hu || !hv || !H || !eta_f || !hu_f || !hv_f || !H_f) return SWE_ERR_INVALID_ARG;
    if (nx < 1 || ny < 1 || nx > 65536 || ny > 65536 || pitch < nx || cpitch < (long long)nx + 1)
        return SWE_ERR_INVALID_ARG;
    if (fpitch < 2LL * nx || (fpitch & 1) || fcpitch < 2LL * nx + 1) return SWE_ERR_INVALID_ARG;
    if (!aligned8(eta_f) || !aligned8(hu_f) || !aligned8(hv_f)) return SWE_ERR_INVALID_ARG;
    if (!(theta >= 1.0 && theta <= 2.0)) return SWE_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    Planes3 in{{eta, hu, hv}};
    const float2 th = make_float2((float)(0.5 / theta), (float)(0.25 * theta));
    OutPlanes3 out{{eta_f, hu_f, hv_f}};
    auto al = [](const void *p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; };
    if (pitch % 2 == 0 && fpitch % 4 == 0 && al(eta, 8) && al(hu, 8) && al(hv, 8) && al(eta_f, 16) &&
        al(hu_f, 16) && al(hv_f, 16)) {
        refine2_kernel<<<grid_for((long long)nx / 2 + 1, ny + 1), kBX * kBY, 0, st>>>(
            in, pitch, H, cpitch, nx, ny, th, out, fpitch, H_f, fcpitch, cpitch % 2 == 0 && al(H, 8),
            fcpitch % 4 == 0 && al(H_f, 16));
    } else {
        refine_cells_kernel<<<grid_for(nx, ny), kBX * kBY, 0, st>>>(in, pitch, H, cpitch, nx, ny, th,
                                                                    out, fpitch);
        refine_corners_kernel<<<grid_for(nx + 1, ny + 1), kBX * kBY, 0, st>>>(H, cpitch, nx, ny, H_f, fcpitch);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SWE_OK : prep_fail(e);
}

int swe_coarsen2(const float *eta_f, const float *hu_f, const float *hv_f, long long fpitch,
                 const float *H_f, long long fcpitch, int nx, int ny, float *eta, float *hu,
                 float *hv, long long pitch, float *H, long long cpitch, void *stream) {
    swe::TraceRange trace("swe_coarsen2");
    if (!eta_f || !hu_f || !hv_f || !H_f || !eta || !hu || !hv || !H) return SWE_ERR_INVALID_ARG;
    if (nx < 1 || ny < 1 || nx > 65536 || ny > 65536 || pitch < nx || cpitch < (long long)nx + 1)
        return SWE_ERR_INVALID_ARG;
    if (fpitch < 2LL * nx || (fpitch & 1) || fcpitch < 2LL * nx + 1) return SWE_ERR_INVALID_ARG;
    if (!aligned8(eta_f) || !aligned8(hu_f) || !aligned8(hv_f)) return SWE_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    Planes3 fin{{eta_f, hu_f, hv_f}};
    OutPlanes3 out{{eta, hu, hv}};
    auto al = [](const void *p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; };
    if (fpitch % 4 == 0 && pitch % 2 == 0 && al(eta_f, 16) && al(hu_f, 16) && al(hv_f, 16) && al(eta, 8) &&
        al(hu, 8) && al(hv, 8)) {
        coarsen2_kernel<<<grid_for((long long)nx / 2 + 1, ny + 1), kBX * kBY, 0, st>>>(
            fin, fpitch, H_f, fcpitch, nx, ny, out, pitch, H, cpitch, fcpitch % 4 == 0 && al(H_f, 16),
            cpitch % 2 == 0 && al(H, 8));
    } else {
        coarsen_cells_kernel<<<grid_for(nx, ny), kBX * kBY, 0, st>>>(fin, fpitch, H_f, fcpitch, nx, ny, out,
                                                                     pitch);
        coarsen_corners_kernel<<<grid_for(nx + 1, ny + 1), kBX * kBY, 0, st>>>(H_f, fcpitch, nx, ny, H, cpitch);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SWE_OK : prep_fail(e);
}

}  // extern "C"
