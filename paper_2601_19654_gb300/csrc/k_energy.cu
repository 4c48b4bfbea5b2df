// Energy, angular momentum and momentum of each system in democratic
// heliocentric variables (Sec. 2.1.1 item (7), mxx_en; the Hamiltonian split
// is footnote 1 of Sec. 2.1.1):
//   E = sum 1/2 m |V|^2 - sum G M0 m / |x| + |P|^2 / (2 M0) - sum_{i<j} G m_i m_j / r_ij,
//   P = sum m V,  L = sum m x x V.
// FP64 throughout; every partial is summed in a fixed order.
#include <cuda.h>   // driver types only: cuCtxGetCurrent / cuCtxGetId are reached through the runtime
#include <algorithm>
#include <cmath>
#include <mutex>

#include "opal_internal.cuh"

namespace opal {

constexpr int kEnThreads = 128;
constexpr int kEnTile = 128;       // bodies of an i-tile and of a j-tile of the pair sum
// Blocks of the pair sum an SM holds: 4 (127 registers) with two pairs under way a thread
// 0.527 ms at 16384 bodies; 3: 0.548, 5: 0.539, 6: 0.541;
// one pair at a time 0.544 to 0.561, four 0.538.
constexpr int kEnBlocks = 4;
constexpr int kEnShortRun = 32;    // sources of a unit when there are few tiles

// ---------------------------------------------------------------------------
// Pair potential, sum_{i<j} m_i m_j / r_ij, of n bodies.
//
// On this chip FP64 runs at 1/62 of the FP32 rate (measured: 1.25 against 78
// TFLOP/s), so the sum in plain FP64 (about 20 FP64 instructions a pair with
// the square root and the division) was bound by the FP64 pipe: 6.1 ms at
// 16384 bodies and 765 ms at 131072.  From kEnSplitMin bodies on a pair's
// term is formed in pairs of floats instead (hi + lo; every product's and
// sum's rounding error is taken along by an FMA or Knuth's TwoSum), about 100
// FP32 instructions, which the FP32 pipe bounds.  A term is then right to about
// 2^-47 of itself, independently from pair to pair:
//  - coordinates and masses are split into three floats, which hold a double
//    exactly (a body's own rounding would be in all its pairs);
//  - pairs closer than 1/128 of the i-body's distance take the FP64
//    expression, and so do pairs with more than 2^-12 of the sum (by its lower
//    bound (sum m_i m_j)^2 / sum m_i m_j (|x_i| + |x_j|), as r_ij <= |x_i| +
//    |x_j|), so the errors of the others average: 2^-47 * 2^-6 of the sum at
//    most, less with more pairs;
//  - terms about as small as a rounding join a sum before it is rounded (as
//    the addend of an FMA): added to a rounded float they would be lost
//    whatever their sign, and the sum over the pairs biased.
// Measured against the sum of FP64 terms added without rounding, 512 to 131072
// bodies: both forms within 4e-16 of it, and at 131072 bodies with two giants
// this one 4e-16, the FP64 one 1.3e-15.  16384 bodies: 6.1 to 0.53 ms; 131072:
// 765 to 29.7 ms (2.9e11 pairs/s; the 110 instructions of a pair at the FP32
// pipe's full rate would take 25 ms).  Below 512 bodies the errors have too
// few pairs to average over, and the sum stays in FP64.  Bodies whose coordinates or masses leave the range in which no part of a float
// pair under- or overflows take FP64 too, tile by tile, so any units work.
constexpr int64_t kEnSplitMin = 512;

// FP64 arrays of the bodies, component c of body i at c[i * stride]; alive may be null
struct EnSrc {
    const double *x, *y, *z, *m;
    const int32_t* alive;
    int stride;
};

// the float pairs of one body: a = hi of x, y, z, m; b = lo.  a.x is a NaN when
// the body is out of the range of the float form.
__device__ __forceinline__ void en_split(double x, double y, double z, double m, float4& a, float4& b) {
    split_hl(x, a.x, b.x);
    split_hl(y, a.y, b.y);
    split_hl(z, a.z, b.z);
    split_hl(m, a.w, b.w);
    const float big = fmaxf(fabsf(a.x), fmaxf(fabsf(a.y), fabsf(a.z)));
    const bool ok = big > 0x1p-30f && big < 0x1p30f && (a.w == 0.0f || (a.w > 0x1p-50f && a.w < 0x1p50f)) &&
                    isfinite(x) && isfinite(y) && isfinite(z) && isfinite(m) && (m == 0.0 || a.w != 0.0f);
    if (!ok) a.x = __int_as_float(0x7fffffff);
}

// a + b = s + e exactly
__device__ __forceinline__ void en_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
}

// One unit: body i (this thread's; a, b its float pairs, li its index in the
// tile) against nj staged sources, those with index above its own when the
// tiles are the same (diag).  The sum of m_j / r_ij comes back in FP64.
// `wide`: a body of the unit is out of the float range (or there are few
// bodies): FP64.
struct EnTile {
    float4 a[kEnTile], b[kEnTile], c[kEnTile];   // first, second and third floats of x, y, z, m
    double x[kEnTile], y[kEnTile], z[kEnTile], m[kEnTile];
};

// what two floats leave of a double (exact)
__device__ __forceinline__ float en_third(double v, float a, float b) { return (float)(v - (double)a - (double)b); }

template <bool DIAG>
__device__ __forceinline__ double en_unit_split(const EnTile& T, int nj, int first, float4 a, float4 b, double xi,
                                                double yi, double zi, float most) {
    const float big = fmaxf(fabsf(a.x), fmaxf(fabsf(a.y), fabsf(a.z)));
    const float thr = big * big * 0x1p-14f;   // nearer than 1/128 of the largest coordinate: FP64
    const float ax = en_third(xi, a.x, b.x), ay = en_third(yi, a.y, b.y), az = en_third(zi, a.z, b.z);
    float sh = 0.0f, sl = 0.0f;
    double e = 0.0;
#pragma unroll 2
    for (int jj = 0; jj < nj; jj++) {
        const float4 c = T.a[jj], g = T.b[jj], k = T.c[jj];
        float dx, dy, dz, ex, ey, ez, t;
        en_two_sum(c.x, -a.x, dx, ex);
        en_two_sum(c.y, -a.y, dy, ey);
        en_two_sum(c.z, -a.z, dz, ez);
        ex = __fadd_rn(__fadd_rn(ex, __fsub_rn(g.x, b.x)), __fsub_rn(k.x, ax));
        ey = __fadd_rn(__fadd_rn(ey, __fsub_rn(g.y, b.y)), __fsub_rn(k.y, ay));
        ez = __fadd_rn(__fadd_rn(ez, __fsub_rn(g.z, b.z)), __fsub_rn(k.z, az));
        t = __fadd_rn(dx, ex); ex = __fsub_rn(ex, __fsub_rn(t, dx)); dx = t;
        t = __fadd_rn(dy, ey); ey = __fsub_rn(ey, __fsub_rn(t, dy)); dy = t;
        t = __fadd_rn(dz, ez); ez = __fsub_rn(ez, __fsub_rn(t, dz)); dz = t;
        // r^2 = rh + rl, rl = 2 (dx ex + ...) + (ex^2 + ...) and the roundings
        const float px = __fmul_rn(dx, dx), py = __fmul_rn(dy, dy), pz = __fmul_rn(dz, dz);
        const float qx = __fmaf_rn(dx, dx, -px), qy = __fmaf_rn(dy, dy, -py), qz = __fmaf_rn(dz, dz, -pz);
        float et, rh, er;
        en_two_sum(px, py, t, et);
        en_two_sum(t, pz, rh, er);
        const float sq = __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
        const float cr = __fmaf_rn(dz, ez, __fmaf_rn(dy, ey, __fmaf_rn(dx, ex, __fmul_rn(0.5f, sq))));
        const float rl =
            __fmaf_rn(2.0f, cr, __fadd_rn(__fadd_rn(__fadd_rn(qx, qy), qz), __fadd_rn(et, er)));
        // m y (1 + d/2 + 3/8 d^2), d = 1 - r^2 y^2: the next term is below 2^-66
        float y;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(rh));
        const float yh = __fmul_rn(y, y), yl = __fmaf_rn(y, y, -yh);
        float d = __fmaf_rn(-rh, yh, 1.0f);
        d = __fmaf_rn(-rh, yl, d);
        d = __fmaf_rn(-rl, yh, d);
        float wh = __fmul_rn(c.w, y), wl = __fmaf_rn(c.w, y, -wh);
        wl = __fadd_rn(wl, __fmaf_rn(g.w, y, __fmul_rn(k.w, y)));
        wl = __fadd_rn(wl, __fmaf_rn(wh, __fmul_rn(0.5f, d), __fmul_rn(wh, __fmul_rn(__fmul_rn(0.375f, d), d))));
        // (r = 0 makes y infinite: the tests below take such a pair out before its NaN is added)
        const bool own = DIAG && first + jj <= (int)threadIdx.x;   // another thread's pair, or the body itself
        const bool fp64 = (rh < thr || wh > most) && !own;
        if (fp64 || own) wh = wl = 0.0f;
        float s, es;
        en_two_sum(sh, wh, s, es);
        sh = s;
        sl = __fadd_rn(sl, __fadd_rn(es, wl));
        if (fp64 && T.m[jj] != 0.0) {
            const double fx = T.x[jj] - xi, fy = T.y[jj] - yi, fz = T.z[jj] - zi;
            e += T.m[jj] / sqrt(fx * fx + fy * fy + fz * fz);
        }
    }
    return e + ((double)sh + (double)sl);
}

__device__ __forceinline__ double en_unit_wide(const EnTile& T, int nj, int from, double xi, double yi, double zi) {
    double e = 0.0;
    for (int jj = from; jj < nj; jj++) {
        if (T.m[jj] == 0.0) continue;
        const double fx = T.x[jj] - xi, fy = T.y[jj] - yi, fz = T.z[jj] - zi;
        e += T.m[jj] / sqrt(fx * fx + fy * fy + fz * fz);
    }
    return e;
}

// The pair sum of n bodies from off on (sa, sb their float pairs).  A unit is
// an i-tile against a run of `run` sources (a whole j-tile, or a quarter of
// one when there are few) of a j-tile at or above it; block b takes units b,
// b + gridDim.x, ..., so that the order of every sum is fixed, and its total
// goes to out[b].  rows: the body kernel's rows (row_n doubles each) of these
// bodies, from column c0 on the sums of m, m^2 and m |x|.
__global__ void __launch_bounds__(kEnThreads, kEnBlocks) k_energy_pairs(int64_t n, int64_t off, EnSrc src,
                                                             const float4* __restrict__ sa,
                                                             const float4* __restrict__ sb, int run,
                                                             const double* __restrict__ rows, int row_n, int c0,
                                                             double* __restrict__ out) {
    __shared__ EnTile T;
    __shared__ double red[3][kEnThreads];
    const int64_t nt = (n + kEnTile - 1) / kEnTile;
    const int parts = kEnTile / run;
    const int64_t units = nt * (nt + 1) / 2 * parts;
    const bool few = n < kEnSplitMin;
    double most = 0.0;   // m_i times a term's limit in float form
    if (!few) {
        double v[3] = {0.0, 0.0, 0.0};
        for (int64_t b = threadIdx.x; b < nt; b += kEnThreads)
            for (int c = 0; c < 3; c++) v[c] += rows[b * row_n + c0 + c];
        for (int c = 0; c < 3; c++) red[c][threadIdx.x] = v[c];
        __syncthreads();
        for (int w = kEnThreads / 2; w >= 1; w >>= 1) {
            if (threadIdx.x < w)
                for (int c = 0; c < 3; c++) red[c][threadIdx.x] += red[c][threadIdx.x + w];
            __syncthreads();
        }
        const double mm = red[0][0] * red[0][0] - red[1][0];
        most = 0x1p-12 * mm / (2.0 * red[0][0]) * (0.5 * mm / red[2][0]);
    }
    double total = 0.0;
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const int64_t w = u / parts;
        const int first = (int)(u % parts) * run;
        // tiles (A, B), A <= B, in the order B (B + 1) / 2 + A
        int64_t B = (int64_t)((sqrtf(8.0f * (float)w + 1.0f) - 1.0f) * 0.5f);
        while (B * (B + 1) / 2 > w) B--;
        while ((B + 1) * (B + 2) / 2 <= w) B++;
        const int64_t A = w - B * (B + 1) / 2;
        const int64_t j0 = B * kEnTile + first, i = A * kEnTile + threadIdx.x;
        const int nj = (int)(n - j0 < run ? n - j0 : run);
        if (nj <= 0) continue;   // (the same for the whole block)
        __syncthreads();
        bool wide = few;
        if ((int)threadIdx.x < nj) {
            const int64_t g = off + j0 + threadIdx.x, s = g * src.stride;
            const float4 a = sa[g], b = sb[g];
            const double x = src.x[s], y = src.y[s], z = src.z[s];
            const double m = src.alive && !src.alive[g] ? 0.0 : src.m[g];
            T.a[threadIdx.x] = a;
            T.b[threadIdx.x] = b;
            T.c[threadIdx.x] =
                make_float4(en_third(x, a.x, b.x), en_third(y, a.y, b.y), en_third(z, a.z, b.z), en_third(m, a.w, b.w));
            T.x[threadIdx.x] = x;
            T.y[threadIdx.x] = y;
            T.z[threadIdx.x] = z;
            T.m[threadIdx.x] = m;
            wide |= isnan(a.x);
        }
        float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
        double xi = 0.0, yi = 0.0, zi = 0.0, mi = 0.0;
        if (i < n) {
            const int64_t g = off + i, s = g * src.stride;
            a = sa[g];
            b = sb[g];
            xi = src.x[s];
            yi = src.y[s];
            zi = src.z[s];
            mi = src.alive && !src.alive[g] ? 0.0 : src.m[g];
            wide |= isnan(a.x);
        }
        wide = __syncthreads_or(wide);
        if (mi == 0.0) continue;   // (no barrier between here and the next unit's first)
        const float lim = (float)(most / mi);
        double e;
        if (wide) e = en_unit_wide(T, nj, A == B ? max(0, (int)threadIdx.x + 1 - first) : 0, xi, yi, zi);
        else if (A == B) e = en_unit_split<true>(T, nj, first, a, b, xi, yi, zi, lim);
        else e = en_unit_split<false>(T, nj, first, a, b, xi, yi, zi, lim);
        total += mi * e;
    }
    __syncthreads();
    red[0][threadIdx.x] = total;
    __syncthreads();
    for (int w = kEnThreads / 2; w >= 1; w >>= 1) {
        if (threadIdx.x < w) red[0][threadIdx.x] += red[0][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = red[0][0];
}

// grid and run length of the pair sum of n bodies: whole j-tiles once they
// give every block that fits a unit, else quarters
static void en_shape(int64_t n, int nsm, int& grid, int& run) {
    const int64_t nt = (n + kEnTile - 1) / kEnTile, tiles = nt * (nt + 1) / 2;
    const int most = std::min(kEnBlocks * nsm, kEnMaxGrid);
    run = tiles >= most ? kEnTile : kEnShortRun;
    grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles * (kEnTile / run), most));
}

// body terms of one system from off on: per 128-body block, kEnSums sums (kinetic +
// central, P, L, then m, m^2 and m |x|), and the float pairs of its bodies for the pair sum
__global__ void __launch_bounds__(kEnThreads) k_energy_body(Dev d, int64_t off, double* body_part, float4* sa,
                                                            float4* sb) {
    __shared__ double red[kEnSums][kEnThreads];
    const int64_t b = off + (int64_t)blockIdx.x * kEnThreads + threadIdx.x;
    double v[kEnSums] = {};
    const double x = d.x[b], y = d.y[b], z = d.z[b];
    const bool alive = d.alive[b] != 0;
    const double m = alive ? d.m[b] : 0.0;
    float4 fa, fb;
    en_split(x, y, z, m, fa, fb);
    sa[b] = fa;
    sb[b] = fb;
    if (alive) {
        const double vx = d.vx[b], vy = d.vy[b], vz = d.vz[b];
        const double r = sqrt(x * x + y * y + z * z);
        v[0] = 0.5 * m * (vx * vx + vy * vy + vz * vz) - d.p.G * d.M0s[d.body_sys[b]] * m / r;
        v[1] = m * vx;
        v[2] = m * vy;
        v[3] = m * vz;
        v[4] = m * (y * vz - z * vy);
        v[5] = m * (z * vx - x * vz);
        v[6] = m * (x * vy - y * vx);
        v[7] = m;
        v[8] = m * m;
        v[9] = m * r;
    }
    for (int c = 0; c < kEnSums; c++) red[c][threadIdx.x] = v[c];
    __syncthreads();
    for (int w = kEnThreads / 2; w >= 1; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < kEnSums; c++) red[c][threadIdx.x] += red[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < kEnSums) body_part[(int64_t)blockIdx.x * kEnSums + threadIdx.x] = red[threadIdx.x][0];
}

// one block: fixed-order sums of the system's partials (nb body blocks, np pair partials)
__global__ void k_energy_final(Dev d, int s, int64_t nb, int np, const double* body_part, const double* pair_part,
                               double* out) {
    __shared__ double red[8][256];
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t k = threadIdx.x; k < nb; k += blockDim.x)
        for (int c = 0; c < 7; c++) v[c] += body_part[k * kEnSums + c];
    for (int k = threadIdx.x; k < np; k += blockDim.x) v[7] += pair_part[k];
    for (int c = 0; c < 8; c++) red[c][threadIdx.x] = v[c];
    __syncthreads();
    for (int w = blockDim.x / 2; w >= 1; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < 8; c++) red[c][threadIdx.x] += red[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double Px = red[1][0], Py = red[2][0], Pz = red[3][0];
        double E = red[0][0] + (Px * Px + Py * Py + Pz * Pz) / (2.0 * d.M0s[s]) - d.p.G * red[7][0];
        out[0] = E;
        out[1] = red[4][0]; out[2] = red[5][0]; out[3] = red[6][0];
        out[4] = Px; out[5] = Py; out[6] = Pz;
        out[7] = d.E_lost[s];
    }
}

void launch_energy(const Dev& d, int sys, const SysInfo& si, int nsm, float4* sa, float4* sb, double* pair_part,
                   double* body_part, double* out, cudaStream_t s) {
    const int64_t nb = si.cap / kEnThreads;
    int grid, run;
    en_shape(si.nb, nsm, grid, run);   // small bodies carry no mass: no pair of theirs adds anything
    k_energy_body<<<(unsigned)nb, kEnThreads, 0, s>>>(d, si.off, body_part, sa, sb);
    k_energy_pairs<<<grid, kEnThreads, 0, s>>>(si.nb, si.off, EnSrc{d.x, d.y, d.z, d.m, d.alive, 1}, sa, sb, run,
                                               body_part, kEnSums, 7, pair_part);
    k_energy_final<<<1, 256, 0, s>>>(d, sys, nb, grid, body_part, pair_part, out);
}

// ---------------------------------------------------------------------------
// The same energy, L and P from caller-owned device arrays of one system,
// with no allocation: the per-block partial sums live in a file-scope device
// array of fixed size, found once per device with cudaGetSymbolAddress.
// Inputs are heliocentric x and v; with u = sum m v / (M0 + sum m) the
// barycentric velocities are V = v - u, so
//   sum 1/2 m |V|^2 = sum 1/2 m |v|^2 - u . sum m v + 1/2 |u|^2 sum m,
//   P = sum m v - u sum m,  L = sum m x x v - (sum m x) x u,
// which lets one pass over the bodies gather every term.

constexpr int kNaThreads = 128;
constexpr int kNaMaxBlocks = 1024;
constexpr int64_t kNaMaxBodies = (int64_t)kNaThreads * kNaMaxBlocks;   // 131072
constexpr int kNaSums = 14;   // 1/2 m v^2, m v (3), m/|x|, m x (3), m x x v (3), m, m^2, m |x|
constexpr int kNaMaxDevices = 64;

// Every slot a call reads is written earlier in the same call (body block b
// writes row b and its bodies' float pairs, pair block b writes pair[b]), so
// nothing here has to start at zero.  4.3 MB of device memory.
struct NaMem {
    float4 a[kNaMaxBodies], b[kNaMaxBodies];
    double part[kNaMaxBlocks * kNaSums];
    double pair[kEnMaxGrid];
};
static __device__ __align__(256) NaMem g_na_mem;

__global__ void __launch_bounds__(kNaThreads) k_energy_na_body(int64_t n, const double* __restrict__ m,
                                                               const double* __restrict__ x,
                                                               const double* __restrict__ v, NaMem* mem) {
    __shared__ double red[kNaSums][kNaThreads];
    const int64_t i = (int64_t)blockIdx.x * kNaThreads + threadIdx.x;
    double s[kNaSums];
    for (int c = 0; c < kNaSums; c++) s[c] = 0.0;
    if (i < n) {
        const double mi = m[i], xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2];
        const double vx = v[3 * i], vy = v[3 * i + 1], vz = v[3 * i + 2];
        float4 fa, fb;
        en_split(xi, yi, zi, mi, fa, fb);
        mem->a[i] = fa;
        mem->b[i] = fb;
        if (mi != 0.0) {
            s[0] = 0.5 * mi * (vx * vx + vy * vy + vz * vz);
            s[1] = mi * vx;
            s[2] = mi * vy;
            s[3] = mi * vz;
            const double r = sqrt(xi * xi + yi * yi + zi * zi);
            s[4] = mi / r;
            s[5] = mi * xi;
            s[6] = mi * yi;
            s[7] = mi * zi;
            s[8] = mi * (yi * vz - zi * vy);
            s[9] = mi * (zi * vx - xi * vz);
            s[10] = mi * (xi * vy - yi * vx);
            s[11] = mi;
            s[12] = mi * mi;
            s[13] = mi * r;
        }
    }
    for (int c = 0; c < kNaSums; c++) red[c][threadIdx.x] = s[c];
    __syncthreads();
    for (int w = kNaThreads / 2; w >= 1; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < kNaSums; c++) red[c][threadIdx.x] += red[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < kNaSums) mem->part[(int64_t)blockIdx.x * kNaSums + threadIdx.x] = red[threadIdx.x][0];
}

// one block: fixed-order sums of the nb body rows and np pair partials, then E, L, P
__global__ void __launch_bounds__(256) k_energy_na_final(int nb, int np, double G, double M0, const NaMem* mem,
                                                         double* __restrict__ out) {
    __shared__ double red[kNaSums + 1][256];   // 30 KB
    double s[kNaSums + 1];
    for (int c = 0; c <= kNaSums; c++) s[c] = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        for (int c = 0; c < kNaSums; c++) s[c] += mem->part[(int64_t)b * kNaSums + c];
    for (int b = threadIdx.x; b < np; b += blockDim.x) s[kNaSums] += mem->pair[b];
    for (int c = 0; c <= kNaSums; c++) red[c][threadIdx.x] = s[c];
    __syncthreads();
    for (int w = blockDim.x / 2; w >= 1; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c <= kNaSums; c++) red[c][threadIdx.x] += red[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double kin = red[0][0], mv[3] = {red[1][0], red[2][0], red[3][0]}, msum = red[11][0];
        const double pot_sun = red[4][0], mx[3] = {red[5][0], red[6][0], red[7][0]};
        const double lh[3] = {red[8][0], red[9][0], red[10][0]}, pair = red[kNaSums][0];
        double u[3], P[3];
        for (int k = 0; k < 3; k++) {
            u[k] = mv[k] / (M0 + msum);
            P[k] = mv[k] - u[k] * msum;
        }
        const double kinV = kin - (u[0] * mv[0] + u[1] * mv[1] + u[2] * mv[2]) +
                            0.5 * msum * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
        out[0] = kinV - G * M0 * pot_sun + (P[0] * P[0] + P[1] * P[1] + P[2] * P[2]) / (2.0 * M0) - G * pair;
        out[1] = lh[0] - (mx[1] * u[2] - mx[2] * u[1]);
        out[2] = lh[1] - (mx[2] * u[0] - mx[0] * u[2]);
        out[3] = lh[2] - (mx[0] * u[1] - mx[1] * u[0]);
        out[4] = P[0];
        out[5] = P[1];
        out[6] = P[2];
    }
}

namespace {

std::mutex g_na_mu;
// per device: the scratch's device address and the context it belongs to
struct NaScratch {
    unsigned long long ctx_id;
    NaMem* ptr;
    int nsm;   // SMs of the device (the pair sum's grid)
};
NaScratch g_na[kNaMaxDevices] = {};
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);
CtxGetCurrentFn g_ctx_current = nullptr;
CtxGetIdFn g_ctx_id = nullptr;

// unique id of the current context (0 if none is current yet); caller holds g_na_mu
opal_status na_context_id(unsigned long long* id) {
    if (!g_ctx_current || !g_ctx_id) {
        void* f1 = nullptr;
        void* f2 = nullptr;
        cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) != cudaSuccess ||
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) != cudaSuccess ||
            q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2) {
            cudaGetLastError();
            set_thread_error("the driver's context queries (cuCtxGetCurrent, cuCtxGetId) are unavailable");
            return OPAL_ECUDA;
        }
        g_ctx_current = (CtxGetCurrentFn)f1;
        g_ctx_id = (CtxGetIdFn)f2;
    }
    CUcontext ctx = nullptr;
    if (g_ctx_current(&ctx) != CUDA_SUCCESS) {
        set_thread_error("cuCtxGetCurrent failed");
        return OPAL_ECUDA;
    }
    *id = 0;
    if (ctx && g_ctx_id(ctx, id) != CUDA_SUCCESS) {
        set_thread_error("cuCtxGetId failed");
        return OPAL_ECUDA;
    }
    return OPAL_OK;
}

// the device address of g_na_mem in the current device's context, looked up
// once per device and context (a device reset or a new primary context makes
// the module load again at another address, so the lookup is redone)
opal_status na_scratch(NaMem** out, int* nsm) {
    int dev = -1;
    cudaError_t rc = cudaGetDevice(&dev);
    if (rc != cudaSuccess) {
        set_thread_error("cudaGetDevice failed: %s", cudaGetErrorString(rc));
        return OPAL_ECUDA;
    }
    if (dev < 0 || dev >= kNaMaxDevices) {
        set_thread_error("device ordinal %d is beyond the %d devices this path supports", dev, kNaMaxDevices);
        return OPAL_EINVAL;
    }
    std::lock_guard<std::mutex> lock(g_na_mu);
    unsigned long long id = 0;
    opal_status st = na_context_id(&id);
    if (st != OPAL_OK) return st;
    if (!g_na[dev].ptr || id == 0 || g_na[dev].ctx_id != id) {
        void* p = nullptr;
        rc = cudaGetSymbolAddress(&p, g_na_mem);
        if (rc != cudaSuccess || !p) {
            set_thread_error("cudaGetSymbolAddress of the energy scratch failed on device %d: %s", dev,
                             cudaGetErrorString(rc));
            return OPAL_ECUDA;
        }
        st = na_context_id(&id);   // the lookup made the primary context current if none was
        if (st != OPAL_OK) return st;
        g_na[dev].ctx_id = id;
        rc = cudaDeviceGetAttribute(&g_na[dev].nsm, cudaDevAttrMultiProcessorCount, dev);
        if (rc != cudaSuccess) {
            set_thread_error("cudaDeviceGetAttribute failed: %s", cudaGetErrorString(rc));
            return OPAL_ECUDA;
        }
        g_na[dev].ptr = (NaMem*)p;
    }
    *out = g_na[dev].ptr;
    *nsm = g_na[dev].nsm;
    return OPAL_OK;
}

// a pointer the kernels may read or write: device (or managed) memory of the
// current device, aligned for doubles
opal_status na_check_ptr(const void* p, const char* name) {
    if (!p) {
        set_thread_error("%s is NULL", name);
        return OPAL_EINVAL;
    }
    if (((uintptr_t)p & 7u) != 0) {
        set_thread_error("%s is not 8-byte aligned", name);
        return OPAL_EINVAL;
    }
    cudaPointerAttributes a{};
    cudaError_t rc = cudaPointerGetAttributes(&a, p);
    if (rc != cudaSuccess) {
        cudaGetLastError();
        set_thread_error("%s: cudaPointerGetAttributes failed: %s", name, cudaGetErrorString(rc));
        return OPAL_EINVAL;
    }
    int dev = -1;
    cudaGetDevice(&dev);
    if (!((a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged)) {
        set_thread_error("%s is not device memory of the current device %d", name, dev);
        return OPAL_EINVAL;
    }
    return OPAL_OK;
}

}  // namespace

}  // namespace opal

using namespace opal;

extern "C" opal_status opal_energy_momentum_noalloc(int64_t n, double G, double M0, const double* m,
                                                    const double* x, const double* v, double* out,
                                                    void* stream) {
    if (n < 0) {
        set_thread_error("n = %lld < 0", (long long)n);
        return OPAL_EINVAL;
    }
    if (n > kNaMaxBodies) {
        set_thread_error("n = %lld exceeds the %lld-body limit of opal_energy_momentum_noalloc (its fixed scratch "
                         "holds %d blocks of %d bodies); use opal_energy_momentum",
                         (long long)n, (long long)kNaMaxBodies, kNaMaxBlocks, kNaThreads);
        return OPAL_EINVAL;
    }
    if (!(std::isfinite(G) && G > 0.0) || !(std::isfinite(M0) && M0 > 0.0)) {
        set_thread_error("G and M0 must be finite and > 0");
        return OPAL_EINVAL;
    }
    opal_status st = na_check_ptr(out, "out");
    if (st == OPAL_OK && n > 0) st = na_check_ptr(m, "m");
    if (st == OPAL_OK && n > 0) st = na_check_ptr(x, "x");
    if (st == OPAL_OK && n > 0) st = na_check_ptr(v, "v");
    if (st != OPAL_OK) return st;
    NaMem* mem = nullptr;
    int nsm = 1;
    st = na_scratch(&mem, &nsm);
    if (st != OPAL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (int)((n + kNaThreads - 1) / kNaThreads);
    int grid = 0, run = 0;
    if (nb > 0) {
        en_shape(n, nsm, grid, run);
        k_energy_na_body<<<nb, kNaThreads, 0, s>>>(n, m, x, v, mem);
        k_energy_pairs<<<grid, kNaThreads, 0, s>>>(n, 0, EnSrc{x, x + 1, x + 2, m, nullptr, 3}, mem->a, mem->b, run,
                                                   mem->part, kNaSums, 11, mem->pair);
    }
    k_energy_na_final<<<1, 256, 0, s>>>(nb, grid, G, M0, mem, out);
    cudaError_t rc = cudaGetLastError();
    if (rc != cudaSuccess) {
        set_thread_error("launch of the energy kernels failed: %s", cudaGetErrorString(rc));
        return OPAL_ECUDA;
    }
    return OPAL_OK;
}
