// Energy, angular momentum and momentum of each system in democratic
// heliocentric variables (Sec. 2.1.1 item (7), mxx_en; the Hamiltonian split
// is footnote 1 of Sec. 2.1.1):
//   E = sum 1/2 m |V|^2 - sum G M0 m / |x| + |P|^2 / (2 M0) - sum_{i<j} G m_i m_j / r_ij,
//   P = sum m V,  L = sum m x x V.
// Every sum is FP64, in a fixed order.  The pair sum takes 1 / r_ij to FP64's precision from the
// FP32 and integer pipes (en_recip); everything else is FP64 arithmetic.
#include <cuda.h>   // driver types only: cuCtxGetCurrent / cuCtxGetId are reached through the runtime
#include <algorithm>
#include <cmath>
#include <mutex>

#include "opal_internal.cuh"

namespace opal {

constexpr int kEnThreads = 128;
constexpr int kEnTile = 128;       // bodies of an i-tile and of a j-tile of the pair sum
// Blocks of the pair sum an SM holds: 6 (78 registers) 0.729 ms at 16384 bodies and 43.3 at 131072;
// 3: 0.782 and 46.8, 4: 0.759 and 45.7, 5: 0.740 and 44.2.
constexpr int kEnBlocks = 6;
constexpr int kEnShortRun = 32;    // sources of a unit when there are few tiles

// ---------------------------------------------------------------------------
// Pair potential, sum_{i<j} m_i m_j / r_ij, of n bodies.
//
// On this chip FP64 runs at 1/62 of the FP32 rate (measured: 1.25 against 78 TFLOP/s): a warp's FP64
// instruction takes its scheduler 64 cycles.  A pair in plain FP64 with the square root and the
// division is about 20 of them, with the hardware's approximate reciprocal square root 13.  Here 1 / r
// is formed as a double by about 133 FP32 operations (two pairs a packed instruction) and 20 integer ones, and
// one FP64 FMA adds m_j / r to the thread's sum beside them.  Plain FP64: 16384 bodies 6.1 ms, 131072 bodies 765
// (each pair from both sides); the 13 instructions at the pipe's rate 2.8 and 178; so 0.73 and 43.3 (the packed
// pipe busy 0.7 of the time; unpacked 0.77 and 46.0).  Pairs of floats (0.53 and 29.7) kept 47 bits of a term.
//
// The FP32 part, for bodies of two tiles whose coordinates lie below X, a power of two (everything
// in units of X, so any units of length work):
//  - a coordinate is three floats a + b + c, a a multiple of 2^-22, b of 2^-45, c the rest, so that the
//    differences of the a's and of the b's are exact (those of the c's to 2^-70); their sum by one
//    FastTwoSum is D1 + D2, |D2| <= half an ulp of D1;
//  - y = the approximate 1 / r of D1 alone, off by 2^-21.6 at most; with v = y (D1 + D2 + D3), a unit
//    vector but for y's error, 1 / r = y (1 - d)^(-1/2), d = 1 - v.v, |d| < 2^-20;
//  - v's components are cut into V (a multiple of 2^-11), A (of 2^-21), B1 (of 2^-31) and C, so that 1 -
//    V.V - 2 V.A - A.A - 2 V.B1, nearly all of which cancels, is exact in FP32 (multiples of 2^-42, the
//    partial results below 2^-18 from A.A on); the rest of d, 2 V.C + 2 A.B + B.B, is below 2^-29, in floats;
//  - 1 / r = y (1 + d/2 + 3/8 d^2) (the next term is below 2^-61) as the 53-bit mantissa of
//    a double: y's 24 bits and, 29 places lower, y (d/2 + 3/8 d^2), a product of integers rounded once.
// Error of 1 / r against 113-bit arithmetic, 200000 pairs for each power of two of r from X down to
// 2^-13 X: 0.52 to 0.53 x 2^-53 rms and 2.7 x 2^-53 at most, mean below 0.002 x 2^-53 (1 / sqrt of the
// FP64 square: 0.69 to 0.72, 2.8 and 0.004; at 2^-14 X the two rms meet, c's rounding grows as X / r).
// A pair closer than 2^-13 X takes the FP64 expression, and so do tiles whose coordinates leave
// the range of the scaling (or are not finite).

// FP64 arrays of the bodies, component c of body i at c[i * stride]; alive may be null
struct EnSrc {
    const double *x, *y, *z, *m;
    const int32_t* alive;
    int stride;
};

// the sources of a unit: a, b and c of x, y, z (component 3 q + k), and the FP64 values
struct EnTile {
    float part[9][kEnTile];
    double m[kEnTile], x[kEnTile], y[kEnTile], z[kEnTile];
};

// scale: 1 / X
__device__ __forceinline__ void en_split(double v, double scale, float& a, float& b, float& c) {
    const double s = v * scale, kA = 0x1.8p30, kB = 0x1.8p7;   // (ulps 2^-22 and 2^-45)
    const double da = (s + kA) - kA, rest = s - da, db = (rest + kB) - kB;
    a = trunc_f(da);   // (exact, and so is b)
    b = trunc_f(db);
    c = trunc_f(rest - db);
}

// 1 / |j - i| of two sources j (j2: their nine floats; n: i's, negated), a packed instruction for both where there
// is one.  Not good (the result means nothing): a separation below 2^-13, zero included, or 1 / r on
// the other side of a power of two than y, where a mantissa's unit is another (one pair in some 10^6).
__device__ __forceinline__ void en_recip(const float (&n)[9], const float2 (&j2)[9], double (&out)[2], bool (&good)[2]) {
    auto all = [](float v) { return make_float2(v, v); };
    auto sub = [&](float2 a, float2 b) { return __ffma2_rn(b, all(-1.0f), a); };
    auto cut = [&](float2 a, float k) { return __fadd2_rn(__fadd2_rn(a, all(k)), all(-k)); };   // to a multiple of k's ulp
    auto dot = [](const float2 (&a)[3], const float2 (&b)[3], float2 c) {
        return __ffma2_rn(a[2], b[2], __ffma2_rn(a[1], b[1], __ffma2_rn(a[0], b[0], c)));
    };
    float2 D1[3], D2[3], V[3], A[3], B[3], C[3], b1[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float2 p = __fadd2_rn(j2[k], all(n[k])), q = __fadd2_rn(j2[3 + k], all(n[3 + k]));
        D1[k] = __fadd2_rn(p, q);
        D2[k] = sub(q, sub(D1[k], p));
    }
    const float2 r2 = __ffma2_rn(D1[2], D1[2], __ffma2_rn(D1[1], D1[1], __fmul2_rn(D1[0], D1[0])));
    float2 y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(r2.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(r2.y));
#pragma unroll
    for (int k = 0; k < 3; k++) {
        // v = P + pe + Q + s, the first three exact
        const float2 P = __fmul2_rn(y, D1[k]), pe = __ffma2_rn(y, D1[k], make_float2(-P.x, -P.y)), Q = __fmul2_rn(y, D2[k]);
        const float2 s = __ffma2_rn(y, __fadd2_rn(j2[6 + k], all(n[6 + k])), __ffma2_rn(y, D2[k], make_float2(-Q.x, -Q.y)));
        V[k] = cut(P, 0x1.8p12f);
        const float2 f = sub(P, V[k]);
        A[k] = cut(f, 0x1.8p2f);
        const float2 f2 = sub(f, A[k]);
        const float2 g = __fadd2_rn(pe, Q), gv = sub(g, pe);
        const float2 ge = __fadd2_rn(sub(pe, sub(g, gv)), sub(Q, gv));   // g + ge = pe + Q
        b1[k] = cut(__fadd2_rn(f2, g), 0x1.8p-8f);
        C[k] = __fadd2_rn(__fadd2_rn(sub(f2, b1[k]), g), __fadd2_rn(ge, s));
        B[k] = __fadd2_rn(b1[k], C[k]);
    }
    const float2 zero = all(0.0f), two = all(2.0f);
    float2 h = dot(V, V, all(-1.0f));                        // -d = h + l
    h = __ffma2_rn(two, dot(V, A, zero), h);
    h = dot(A, A, h);
    h = __ffma2_rn(two, dot(V, b1, zero), h);
    const float2 l = dot(B, B, __fmul2_rn(two, dot(A, B, dot(V, C, zero))));
    // d/2 as h/2 in units of 2^-52 (h is an integer of 22 bits in units of 2^-42, taken from the
    // low bits of its sum with 1.5 x 2^23) and l/2 - 3/8 d^2 in units of 2^-54, both negative
    const float2 d = __fadd2_rn(h, l);
    const float2 hm = __ffma2_rn(h, all(0x1p42f), all(0x1.8p23f));
    const float2 lm = __ffma2_rn(__fmul2_rn(d, d), all(-0x1.8p52f), __fmul2_rn(l, all(0x1p53f)));
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const int ch = (int)((__float_as_uint(e ? hm.y : hm.x) << 9) ^ 0x80000000u), cl = __float2int_rn(e ? lm.y : lm.x);
        const unsigned yb = __float_as_uint(e ? y.y : y.x);
        const int Y = (int)((yb & 0x7fffffu) | 0x800000u);
        const long long z = ((long long)Y * ch + (long long)(Y >> 2) * cl + (1 << 22)) >> 23;
        const long long y64 = ((long long)yb << 29) + (896LL << 52), u = y64 - z;
        good[e] = (e ? r2.y : r2.x) >= 0x1p-26f && (u ^ y64) >> 52 == 0;
        out[e] = __longlong_as_double(u);
    }
}

// the pair's term in FP64 (out of line: few pairs take it)
__device__ __noinline__ double en_term(const EnTile& T, int jj, double xi, double yi, double zi) {
    if (T.m[jj] == 0.0) return 0.0;
    const double fx = T.x[jj] - xi, fy = T.y[jj] - yi, fz = T.z[jj] - zi;
    return T.m[jj] / sqrt(fx * fx + fy * fy + fz * fz);
}

// One unit: body i (this thread's) against nj staged sources, those with index above its own
// when the tiles are the same (DIAG); the sum of m_j / r_ij.
template <bool DIAG>
__device__ __forceinline__ double en_unit(const EnTile& T, int nj, int first, double scale, double xi, double yi, double zi) {
    float n[9];
    en_split(-xi, scale, n[0], n[3], n[6]);
    en_split(-yi, scale, n[1], n[4], n[7]);
    en_split(-zi, scale, n[2], n[5], n[8]);
    double e = 0.0, near = 0.0;
#pragma unroll 1
    for (int jj = 0; jj < nj; jj += 2) {
        float2 j2[9];
#pragma unroll
        for (int q = 0; q < 9; q++) j2[q] = *reinterpret_cast<const float2*>(&T.part[q][jj]);
        const double2 m = *reinterpret_cast<const double2*>(&T.m[jj]);
        double s[2];
        bool good[2];
        en_recip(n, j2, s, good);
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const bool own = DIAG && first + jj + k <= (int)threadIdx.x;   // another thread's pair, or the body itself
            if (good[k]) e = fma(own ? 0.0 : k ? m.y : m.x, s[k], e);
            else if (!own) near += en_term(T, jj + k, xi, yi, zi);
        }
    }
    return fma(e, scale, near);
}

__device__ __forceinline__ double en_unit_wide(const EnTile& T, int nj, int from, double xi, double yi, double zi) {
    double e = 0.0;
    for (int jj = from; jj < nj; jj++) e += en_term(T, jj, xi, yi, zi);
    return e;
}

// The pair sum of n bodies from off on.  A unit is an i-tile against a run of `run` sources (a whole
// j-tile, or a quarter of one when there are few) of a j-tile at or above it; block b takes units b,
// b + gridDim.x, ..., so that the order of every sum is fixed, and its total goes to out[b].
__global__ void __launch_bounds__(kEnThreads, kEnBlocks) k_energy_pairs(int64_t n, int64_t off, EnSrc src, int run,
                                                                     double* __restrict__ out) {
    __shared__ __align__(16) EnTile T;
    __shared__ double red[kEnThreads];
    __shared__ int top[kEnThreads / 32];
    const int64_t nt = (n + kEnTile - 1) / kEnTile;
    const int parts = kEnTile / run;
    const int64_t units = nt * (nt + 1) / 2 * parts;
    // a body (a massless one adds nothing wherever it is, and is put at the origin), and the
    // high word of its largest coordinate
    auto load = [&](int64_t k, double& x, double& y, double& z, double& m) {
        const int64_t g = off + k, s = g * src.stride;
        m = src.alive && !src.alive[g] ? 0.0 : src.m[g];
        const bool any = m != 0.0;
        x = any ? src.x[s] : 0.0;
        y = any ? src.y[s] : 0.0;
        z = any ? src.z[s] : 0.0;
        return max(__double2hiint(fabs(x)), max(__double2hiint(fabs(y)), __double2hiint(fabs(z))));
    };
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
        double xj = 0.0, yj = 0.0, zj = 0.0, mj = 0.0, xi = 0.0, yi = 0.0, zi = 0.0, mi = 0.0;
        int hi = 0;
        if ((int)threadIdx.x < nj) hi = load(j0 + threadIdx.x, xj, yj, zj, mj);
        if (i < n) hi = max(hi, load(i, xi, yi, zi, mi));
        hi = __reduce_max_sync(0xffffffffu, hi);
        __syncthreads();   // (the unit before this one is done with the tile)
        if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = hi;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kEnThreads / 32; q++) hi = max(hi, top[q]);
        const int k = hi >> 20;                          // coordinates below X = 2^(k - 1022)
        const bool wide = k < 64 || k > 1983;            // (no scaling: FP64)
        const double scale = __hiloint2double((2045 - k) << 20, 0);
        if ((int)threadIdx.x < (nj + 1) / 2 * 2) {   // (a last one without mass where nj is odd)
            const int t = threadIdx.x;
            T.x[t] = xj;
            T.y[t] = yj;
            T.z[t] = zj;
            T.m[t] = mj;
            en_split(xj, scale, T.part[0][t], T.part[3][t], T.part[6][t]);
            en_split(yj, scale, T.part[1][t], T.part[4][t], T.part[7][t]);
            en_split(zj, scale, T.part[2][t], T.part[5][t], T.part[8][t]);
        }
        __syncthreads();
        if (mi == 0.0) continue;   // (no barrier between here and the next unit's first)
        double e;
        if (wide) e = en_unit_wide(T, nj, A == B ? max(0, (int)threadIdx.x + 1 - first) : 0, xi, yi, zi);
        else if (A == B) e = en_unit<true>(T, nj, first, scale, xi, yi, zi);
        else e = en_unit<false>(T, nj, first, scale, xi, yi, zi);
        total += mi * e;
    }
    red[threadIdx.x] = total;
    __syncthreads();
    for (int w = kEnThreads / 2; w >= 1; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

// grid and run length of the pair sum of n bodies: whole j-tiles once they
// give every block that fits a unit, else quarters
static void en_shape(int64_t n, int nsm, int& grid, int& run) {
    const int64_t nt = (n + kEnTile - 1) / kEnTile, tiles = nt * (nt + 1) / 2;
    const int most = std::min(kEnBlocks * nsm, kEnMaxGrid);
    run = tiles >= most ? kEnTile : kEnShortRun;
    grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles * (kEnTile / run), most));
}

// body terms of one system from off on: per 128-body block, kEnSums sums (kinetic + central, P, L)
__global__ void __launch_bounds__(kEnThreads) k_energy_body(Dev d, int64_t off, double* body_part) {
    __shared__ double red[kEnSums][kEnThreads];
    const int64_t b = off + (int64_t)blockIdx.x * kEnThreads + threadIdx.x;
    double v[kEnSums] = {};
    if (d.alive[b]) {
        const double m = d.m[b], x = d.x[b], y = d.y[b], z = d.z[b], vx = d.vx[b], vy = d.vy[b], vz = d.vz[b];
        v[0] = 0.5 * m * (vx * vx + vy * vy + vz * vz) - d.p.G * d.M0s[d.body_sys[b]] * m / sqrt(x * x + y * y + z * z);
        v[1] = m * vx;
        v[2] = m * vy;
        v[3] = m * vz;
        v[4] = m * (y * vz - z * vy);
        v[5] = m * (z * vx - x * vz);
        v[6] = m * (x * vy - y * vx);
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
        for (int c = 0; c < kEnSums; c++) v[c] += body_part[k * kEnSums + c];
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

void launch_energy(const Dev& d, int sys, const SysInfo& si, int nsm, double* pair_part, double* body_part,
                   double* out, cudaStream_t s) {
    const int64_t nb = si.cap / kEnThreads;
    int grid, run;
    en_shape(si.nb, nsm, grid, run);   // small bodies carry no mass: no pair of theirs adds anything
    k_energy_body<<<(unsigned)nb, kEnThreads, 0, s>>>(d, si.off, body_part);
    k_energy_pairs<<<grid, kEnThreads, 0, s>>>(si.nb, si.off, EnSrc{d.x, d.y, d.z, d.m, d.alive, 1}, run,
                                               pair_part);
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
constexpr int kNaSums = 12;   // 1/2 m v^2, m v (3), m/|x|, m x (3), m x x v (3), m
constexpr int kNaMaxDevices = 64;

// Every slot a call reads is written earlier in the same call (body block b
// writes row b, pair block b writes pair[b]), so nothing here has to start at zero.
struct NaMem {
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
        if (mi != 0.0) {
            s[0] = 0.5 * mi * (vx * vx + vy * vy + vz * vz);
            s[1] = mi * vx;
            s[2] = mi * vy;
            s[3] = mi * vz;
            s[4] = mi / sqrt(xi * xi + yi * yi + zi * zi);
            s[5] = mi * xi;
            s[6] = mi * yi;
            s[7] = mi * zi;
            s[8] = mi * (yi * vz - zi * vy);
            s[9] = mi * (zi * vx - xi * vz);
            s[10] = mi * (xi * vy - yi * vx);
            s[11] = mi;
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
    __shared__ double red[kNaSums + 1][256];   // 27 KB
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
        k_energy_pairs<<<grid, kNaThreads, 0, s>>>(n, 0, EnSrc{x, x + 1, x + 2, m, nullptr, 3}, run, mem->pair);
    }
    k_energy_na_final<<<1, 256, 0, s>>>(nb, grid, G, M0, mem, out);
    cudaError_t rc = cudaGetLastError();
    if (rc != cudaSuccess) {
        set_thread_error("launch of the energy kernels failed: %s", cudaGetErrorString(rc));
        return OPAL_ECUDA;
    }
    return OPAL_OK;
}
