// Bulirsch-Stoer integration of each encounter group over the step, with
// perfect-merger collisions (Sec. 2.1.1 footnote 2: the bodies in a close
// encounter have their interaction and Keplerian Hamiltonians advanced by BS;
// Sec. 3.2 listing: they restart from the saved x0, v0; mce_coll, Sec. 2.1.2).
//
// Equations of a group, democratic heliocentric variables:
//   dx_b/dt = V_b,
//   dV_b/dt = -G M0 x_b/|x_b|^3 + sum_{c in group} G m_c (1 - K(r_bc; rc_bc)) (x_c - x_b)/r_bc^3.
// A substep of length H: modified midpoint with n_k = 2, 4, ..., 16 steps and
// Neville extrapolation in h^2; row k (k >= 1) is accepted when
//   max_b max(|dX_b|/|X_b|, |dV_b|/|V_b|) <= bs_tol,  d = T[k][k] - T[k][k-1].
// Step control as the oracle's: first substep = the whole step; accepted at
// k <= 2 -> double, at k >= 6 -> halve; not accepted by k = 7 -> retry at
// half length; the substep count is capped.
//
// Layout: one thread per (sequence k, member b); all eight midpoint
// sequences advance in lockstep, one derivative evaluation per round.
// Sequence k finishes at round n_k = 2k + 2, row k is extrapolated at once
// (row k - 1 is two rounds old), and the group stops at the first row that
// passes the test, as the sequential method does.  On this chip a warp's FP64
// instruction holds its scheduler's FP64 unit for 64 cycles whatever the number
// of active lanes, so a round lasts as long as its longest warp has FP64
// instructions, and warps beyond one a scheduler wait for each other.  The
// small-group kernel also tries the step sizes H, H/2, H/4, H/8 at once, on as
// many SMs: the first one accepted in that order is the one the sequential
// method would reach after its rejections, so only the cost of rejections
// changes.
#include <cooperative_groups.h>

#include <type_traits>

#include <algorithm>

#include "opal_internal.cuh"

namespace opal {

namespace cg = cooperative_groups;

// Few groups (kBsManyGroups or fewer in a step): the lockstep kernels (all
// sequences at once) give each group the shortest chain of dependent
// operations.  Many groups: those of up to four members make their first
// attempt, the whole step, in the packed kernel (one lane per member, many
// groups per warp), which settles most of them; the ones it rejects go on to
// the lockstep kernel, which starts them again from the beginning.  Groups of
// more than four members always go to their lockstep kernels, beside all this.

// Groups of 17 to 64 members: one block, one thread per (sequence, member).
constexpr int kBsThreads = 512;
struct BsSh {
    static constexpr int M = kBsThreads / kBsRows;
    double y[6][M];                  // current state, component-major: X, Y, Z, VX, VY, VZ
    double pos[kBsRows][3][M];       // positions of each sequence's evaluation in progress
    float4 posf[kBsRows][M];         // the same in float, with rc (rounded up), for near_pair
    double row[kBsRows][6][M];       // the last extrapolated row of each member
    double diag[kBsRows][6][M];      // T[k][k] of every finished row (the accepted one is kept)
    double raw[6][M];                // midpoint result of the sequence finishing this round
    double df2[6][M], cur2[6][M];    // per component: squared change and squared value
    int ok[kBsRows][M];              // each member passes the acceptance test, per finished row
    double m[M], R[M], rc[M];
    float rcf[M];                    // rc rounded up
    // per member: rc^2, 1 / (0.9 rc) and 0.1 rc (a pair uses the member with the larger rc)
    double prc2[M], pinv[M], pc01[M];
    int alive[M], gid[M];
    int big[M];                      // a big body (a source of force), not a small one
    int kacc;                        // accepted row of the substep, -1 while none
    int collide, nmerge;
    double El;
};

// Perfect merger of members b and q of a group held in S (y[6][.], m, R, gid,
// alive), M0 the star's mass: mass, momentum and centre of mass kept, R = cbrt(R_b^3 + R_q^3),
// the heavier body (lower id on a tie) survives; El gets the energy removed.
template <class SH>
__device__ void bs_merge(SH& S, const Params& p, double M0, int b, int q, double& El, int& nmerge) {
    const double G = p.G;
    double mb = S.m[b], mq = S.m[q], M = mb + mq;
    double d[3] = {S.y[0][q] - S.y[0][b], S.y[1][q] - S.y[1][b], S.y[2][q] - S.y[2][b]};
    double xn[3], vn[3];
    for (int k = 0; k < 3; k++) {
        xn[k] = (mb * S.y[k][b] + mq * S.y[k][q]) / M;
        vn[k] = (mb * S.y[3 + k][b] + mq * S.y[3 + k][q]) / M;
    }
    double vb2 = S.y[3][b] * S.y[3][b] + S.y[4][b] * S.y[4][b] + S.y[5][b] * S.y[5][b];
    double vq2 = S.y[3][q] * S.y[3][q] + S.y[4][q] * S.y[4][q] + S.y[5][q] * S.y[5][q];
    double rb = sqrt(S.y[0][b] * S.y[0][b] + S.y[1][b] * S.y[1][b] + S.y[2][b] * S.y[2][b]);
    double rq = sqrt(S.y[0][q] * S.y[0][q] + S.y[1][q] * S.y[1][q] + S.y[2][q] * S.y[2][q]);
    double rbq = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    double e_before = 0.5 * mb * vb2 + 0.5 * mq * vq2 - G * M0 * mb / rb - G * M0 * mq / rq - G * mb * mq / rbq;
    double vn2 = vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2];
    double rn = sqrt(xn[0] * xn[0] + xn[1] * xn[1] + xn[2] * xn[2]);
    double e_after = 0.5 * M * vn2 - G * M0 * M / rn;
    El += e_before - e_after;
    int keep, gone;
    if (mb > mq) keep = b, gone = q;
    else if (mq > mb) keep = q, gone = b;
    else keep = (S.gid[b] < S.gid[q]) ? b : q, gone = (keep == b) ? q : b;
    double Rn = cbrt(S.R[b] * S.R[b] * S.R[b] + S.R[q] * S.R[q] * S.R[q]);
    for (int k = 0; k < 3; k++) {
        S.y[k][keep] = xn[k];
        S.y[3 + k][keep] = vn[k];
    }
    S.m[keep] = M;
    S.R[keep] = Rn;
    S.m[gone] = 0.0;
    S.alive[gone] = 0;
    nmerge++;
}

// x^2 + y^2 + z^2, contracted one way wherever it is inlined (an encounter's
// result then does not depend on which kernel integrates its group)
__device__ __forceinline__ double bs_sq3(double x, double y, double z) {
    return fma(z, z, fma(x, x, __dmul_rn(y, y)));
}

// (1 - K) weighted attraction of a member at (xb, yb, zb) towards one at
// (xo, yo, zo) of mass mo, added to (ax, ay, az).  rc, rc2, c01, inv belong to
// the member with the larger rc (rc_bo = max(rc_b, rc_o)): rc, rc^2, 0.1 rc and
// 1 / (0.9 rc), so K needs no division by rc.  Callers pass big members only:
// a small body pulls nothing (Sec. 2.1: only big bodies are gravity sources).
// bs_factor gives the separation and its factor (0 out of range).
__device__ __forceinline__ double bs_factor(const Params& p, double xb, double yb, double zb, double xo, double yo,
                                            double zo, double mo, double rc, double rc2, double c01, double inv,
                                            double& dx, double& dy, double& dz) {
    dx = xo - xb, dy = yo - yb, dz = zo - zb;
    const double dr2 = bs_sq3(dx, dy, dz);
    if (ge_nonneg(dr2, rc2)) return 0.0;   // 1 - K = 0 at or beyond rc
    const double dri = rsqrt(dr2), dr = __dmul_rn(dr2, dri);
    if (ge_nonneg(dr, rc)) return 0.0;
    return mutual_factor(p.G * mo * (dri * dri * dri), __dmul_rn(dr - c01, inv), p.changeover);
}
__device__ __forceinline__ void bs_pair(const Params& p, double xb, double yb, double zb, double xo, double yo,
                                        double zo, double mo, double rc, double rc2, double c01, double inv,
                                        double& ax, double& ay, double& az) {
    double dx, dy, dz;
    const double t = bs_factor(p, xb, yb, zb, xo, yo, zo, mo, rc, rc2, c01, inv, dx, dy, dz);
    if (!(__double_as_longlong(t) << 1)) return;
    ax = fma(t, dx, ax);
    ay = fma(t, dy, ay);
    az = fma(t, dz, az);
}

// FP32 test that never turns away a pair closer than max(rc_b, rc_o): most pairs
// of a group are farther apart than that, and the FP64 test of one (the
// separation and its square, six instructions of the FP64 unit, the resource
// that bounds these kernels) cost more than the few near pairs' terms.  a, b:
// positions cut to floats, with rc rounded up.  A float separation is off by
// at most 2^-23 (|x_a| + |x_b|) and its own rounding, and |x_b| <= |x_a| + |dx|,
// so 2^-21 of the coordinates of a alone and a factor 1 + 1e-5 cover it.
__device__ __forceinline__ bool near_pair(const float4& a, const float4& b) {
    const float dx = b.x - a.x, dy = b.y - a.y, dz = b.z - a.z;
    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    const float t = (fmaxf(a.w, b.w) + 0x1p-21f * (fabsf(a.x) + fabsf(a.y) + fabsf(a.z))) * 1.00001f;
    return !(r2 > t * t);
}
__device__ __forceinline__ float4 near_record(double x, double y, double z, float rc) {
    return make_float4(trunc_f(x), trunc_f(y), trunc_f(z), rc);
}

// acceleration of member b of sequence k at its position (x, y, z): the
// stellar term, then the mutual terms in ascending order of the other member
// (the oracle's order)
__device__ __forceinline__ void bs_accel(const BsSh& S, const Params& p, double GM0, int nm, int k, int b, double xb,
                                         double yb, double zb, double& ax, double& ay, double& az) {
    double r2 = bs_sq3(xb, yb, zb), ri = rsqrt(r2);
    double s = -GM0 * (ri * ri * ri);
    ax = s * xb;
    ay = s * yb;
    az = s * zb;
    const float4 me = S.posf[k][b];
    unsigned long long near = 0;   // bit j: the j-th other member may be in range
    for (int j = 0; j < nm - 1; j++) {
        const int o = j + (j >= b ? 1 : 0);
        if (near_pair(me, S.posf[k][o]) && S.alive[o] && S.big[o]) near |= 1ull << j;
    }
    for (; near; near &= near - 1) {
        const int j = __ffsll((long long)near) - 1;
        const int o = j + (j >= b ? 1 : 0);
        const int w = gt_nonneg(S.rc[b], S.rc[o]) ? b : o;   // rc_bo = max(rc_b, rc_o)
        bs_pair(p, xb, yb, zb, S.pos[k][0][o], S.pos[k][1][o], S.pos[k][2][o], S.m[o], S.rc[w], S.prc2[w], S.pc01[w],
                S.pinv[w], ax, ay, az);
    }
}

__global__ void __launch_bounds__(kBsThreads, 1) k_bs(Dev d) {
    OPAL_TIMELINE_SCOPE(kTlBs64);
    constexpr int M = BsSh::M, NT = kBsThreads;
    extern __shared__ __align__(16) unsigned char bs_smem[];   // one BsSh (dynamic: above the static limit)
    BsSh& S = *reinterpret_cast<BsSh*>(bs_smem);
    if (d.ctl->status) return;
    const Params p = d.p;
    const int ng = d.ctl->nlarge;
    const int tid = threadIdx.x;
    const int cap = p.bs_max_substeps;
    const double tol2 = p.bs_tol * p.bs_tol;
    __shared__ int s_gi;
    for (;;) {
        // blocks take groups from a queue, so a long group holds up only its own block
        __syncthreads();
        if (tid == 0) s_gi = atomicAdd(&d.ctl->qlock[2], 1);
        __syncthreads();
        const int gi = s_gi;
        if (gi >= ng) break;
        const int g = d.glarge[gi];
        const int mb = d.goff[g], nm = d.goff[g + 1] - mb;
        if (nm > M) {
            if (tid == 0) set_status(d.ctl, kEoverflow, 1000000 + g);
            return;
        }
        const int k = tid / nm, b = tid % nm;   // sequence, member
        const bool act = k < kBsRows;
        const double M0g = d.M0s[d.body_sys[d.members[mb]]];   // the star of the group's system
        if (tid < nm) {
            int gb = d.members[mb + tid];
            S.gid[tid] = gb;
            S.y[0][tid] = d.x0[gb];
            S.y[1][tid] = d.y0[gb];
            S.y[2][tid] = d.z0[gb];
            S.y[3][tid] = d.vx0[gb];
            S.y[4][tid] = d.vy0[gb];
            S.y[5][tid] = d.vz0[gb];
            S.m[tid] = d.m[gb];
            S.R[tid] = d.R[gb];
            S.rc[tid] = d.rc[gb];
            S.alive[tid] = d.alive[gb];
            const SysInfo& gs = d.sys[d.body_sys[gb]];
            S.big[tid] = gb - gs.off < gs.nb;
        }
        if (tid == 0) {
            S.El = 0.0;
            S.nmerge = 0;
        }
        __syncthreads();
        if (tid < nm) {
            const double rcp = S.rc[tid];
            S.prc2[tid] = rcp * rcp;
            S.pc01[tid] = 0.1 * rcp;
            S.pinv[tid] = 1.0 / (0.9 * rcp);
            S.rcf[tid] = __double2float_ru(rcp);
        }
        __syncthreads();
        const double dt = p.dt;
        const int n = 2 * (k + 1);
        double t = 0.0, H = dt;
        int nsub = 0, failed = 0;
        for (;;) {
            const double rem = dt - t;
            int last = 0;
            if (fabs(H) >= fabs(rem)) {
                H = rem;
                last = 1;
            }
            const double h = H / n;
            double za[6], zb[6];
            if (act)
                for (int c = 0; c < 6; c++) za[c] = zb[c] = S.y[c][b];
            if (tid == 0) S.kacc = -1;
            __syncthreads();
            for (int r = 0; r <= 2 * kBsRows; r++) {
                const bool live = act && r <= n;
                if (live) {
                    const double* zp = (r == 0) ? za : zb;
                    S.pos[k][0][b] = zp[0];
                    S.pos[k][1][b] = zp[1];
                    S.pos[k][2][b] = zp[2];
                    S.posf[k][b] = near_record(zp[0], zp[1], zp[2], S.rcf[b]);
                }
                __syncthreads();
                double f[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
                if (live && S.alive[b]) {
                    const double* zp = (r == 0) ? za : zb;
                    f[0] = zp[3];
                    f[1] = zp[4];
                    f[2] = zp[5];
                    bs_accel(S, p, p.G * M0g, nm, k, b, zp[0], zp[1], zp[2], f[3], f[4], f[5]);
                }
                if (live) {
                    if (r == 0) {
                        for (int c = 0; c < 6; c++) zb[c] = za[c] + h * f[c];
                    } else if (r < n) {
                        for (int c = 0; c < 6; c++) {
                            double znew = za[c] + 2.0 * h * f[c];
                            za[c] = zb[c];
                            zb[c] = znew;
                        }
                    } else {
                        // sequence k done: its midpoint result, extrapolated below
                        for (int c = 0; c < 6; c++) S.raw[c][b] = 0.5 * (zb[c] + za[c] + h * f[c]);
                    }
                }
                if (r >= 2 && (r & 1) == 0) {
                    // row kr of the tableau, one lane per (component, member) of each
                    // attempt: the six Neville chains of a member run side by side
                    const int kr = r / 2 - 1;
                    __syncthreads();
                    if (tid < 6 * nm) {
                        const int c = tid / nm, bb = tid % nm;
                        double cur = S.raw[c][bb];
                        double prev_col = 0.0;
                        for (int j = 1; j <= kr; j++) {
                            const double up = S.row[j - 1][c][bb];
                            S.row[j - 1][c][bb] = cur;
                            prev_col = cur;
                            cur = cur + (cur - up) * kNeville[kr][j];
                        }
                        S.row[kr][c][bb] = cur;
                        S.diag[kr][c][bb] = cur;
                        const double df = cur - prev_col;
                        S.df2[c][bb] = df * df;
                        S.cur2[c][bb] = cur * cur;
                    }
                    __syncthreads();
                    if (tid < nm) {
                        // this member passes the acceptance test: |dX|^2 <= tol^2 |X|^2
                        // and the same for V (the test without its divisions); a NaN fails
                        int pass = 1;
                        if (kr >= 1 && S.alive[tid]) {
                            const double dsq_x = S.df2[0][tid] + S.df2[1][tid] + S.df2[2][tid];
                            const double nx = S.cur2[0][tid] + S.cur2[1][tid] + S.cur2[2][tid];
                            const double dsq_v = S.df2[3][tid] + S.df2[4][tid] + S.df2[5][tid];
                            const double nv = S.cur2[3][tid] + S.cur2[4][tid] + S.cur2[5][tid];
                            pass = dsq_x <= tol2 * fmax(nx, 2.3e-308) && dsq_v <= tol2 * fmax(nv, 2.3e-308);
                        }
                        S.ok[kr][tid] = pass;
                    }
                }
                __syncthreads();
                if (r >= 4 && (r & 1) == 0) {
                    const int kr = r / 2 - 1;           // row finished this round
                    if (tid == 0) {
                        int all = 1;
                        for (int q = 0; q < nm; q++) all &= S.ok[kr][q];
                        if (all) S.kacc = kr;
                    }
                    __syncthreads();
                    if (S.kacc >= 0) break;
                }
            }
            const int kacc = S.kacc;
            nsub++;
            if (kacc >= 0) {
                if (tid < 6 * nm) S.y[tid / nm][tid % nm] = S.diag[kacc][tid / nm][tid % nm];
                t = last ? dt : t + H;
                if (tid == 0) S.collide = 0;
                __syncthreads();
                // any pair in contact?  (exact sequential resolution only if so)
                for (int e = tid; e < nm * nm; e += NT) {
                    int u = e / nm, w = e % nm;
                    if (w > u && S.alive[u] && S.alive[w] && bs_can_touch(S.m[u], S.m[w])) {
                        double dx = S.y[0][w] - S.y[0][u], dy = S.y[1][w] - S.y[1][u],
                               dz = S.y[2][w] - S.y[2][u];
                        if (sqrt(dx * dx + dy * dy + dz * dz) <= S.R[u] + S.R[w]) S.collide = 1;
                    }
                }
                __syncthreads();
                if (S.collide && tid == 0) {
                    for (int u = 0; u < nm; u++)
                        for (int w = u + 1; w < nm && S.alive[u]; w++) {
                            if (!S.alive[w] || !bs_can_touch(S.m[u], S.m[w])) continue;
                            double dx = S.y[0][w] - S.y[0][u], dy = S.y[1][w] - S.y[1][u],
                                   dz = S.y[2][w] - S.y[2][u];
                            if (sqrt(dx * dx + dy * dy + dz * dz) <= S.R[u] + S.R[w])
                                bs_merge(S, p, M0g, u, w, S.El, S.nmerge);
                        }
                }
                __syncthreads();
                if (last) break;
                if (kacc <= 2) H *= 2.0;
                else if (kacc >= 6) H *= 0.5;
            } else {
                H *= 0.5;
            }
            if (nsub >= cap) {
                failed = 1;
                break;
            }
        }
        __syncthreads();
        if (failed) {
            if (tid == 0) set_status(d.ctl, kEbs, g);
            return;
        }
        // results go to the member's slot of the side buffer; the state itself
        // is updated after the step's kick, which runs beside this kernel
        if (tid < nm) {
            double* o = d.bsout + (int64_t)kBsOut * (mb + tid);
            for (int c = 0; c < 6; c++) o[c] = S.y[c][tid];
            o[6] = S.m[tid];
            o[7] = S.R[tid];
            o[8] = (double)S.alive[tid];
        }
        if (tid == 0) {
            d.glost[g] = S.El;
            if (S.nmerge) atomicAdd(&d.ctl->nmerge, S.nmerge);
            atomicAdd(&d.ctl->nsub, (unsigned long long)nsub);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Many groups: the first attempt of each group of up to four members (the
// whole step as one substep), with one lane per member and many groups to a
// warp; a group whose attempt is rejected goes on the list the lockstep kernel
// takes next.  A warp works through the size classes (groups of 3-4, then of 2
// members) in turn; its lanes form 32 / Wc segments of Wc lanes, and each
// segment takes groups of the class from a queue, the next one as soon as its
// group is done.  Every lane runs the same instructions on each pass of the
// loop: one derivative at the member's evaluation point, then the midpoint
// step or, at the end of a sequence, its row of the extrapolation tableau and
// the group's decision.  The sequences n_k run one after another as in the
// sequential method, so a pass does the work of up to 32 members.  What a
// group shares (positions for the forces, the error maximum, contacts) goes
// through shared memory within its segment.  (Larger groups left this kernel:
// their chains of up to 15 pairs a pass held the whole warp, and the step,
// for 2.6 ms on the ensemble before their lockstep kernel could start.)
constexpr int kPkWarps = 4;    // warps per block

struct PkWarp {
    double row[kBsRows][6][32];          // each lane's extrapolation tableau (in place)
    double y[6][32];                     // states at a substep's end (contacts, mergers)
    double px[32], py[32], pz[32];       // positions of the current evaluation
    float4 pf[32];                       // the same in float, with rc (rounded up), for near_pair
    double m[32], R[32], rc[32], prc2[32], pinv[32], pc01[32];
    float rcf[32];                       // rc rounded up
    int alive[32], gid[32];
    int big[32];                         // a big body (a source of force), not a small one
    int seg_g[16];                       // group each segment took from the queue
};

__global__ void __launch_bounds__(32 * kPkWarps) k_bs_packed(Dev d) {
    OPAL_TIMELINE_SCOPE(kTlBsPacked);
    extern __shared__ __align__(16) unsigned char pk_smem[];
    const int lane = threadIdx.x & 31;
    PkWarp& W = reinterpret_cast<PkWarp*>(pk_smem)[threadIdx.x >> 5];
    if (d.ctl->status) return;
    if (d.ctl->ngroups <= kBsManyGroups) return;   // few groups: the lockstep kernels take them
    const Params p = d.p;
    const double tol2 = p.bs_tol * p.bs_tol, dt = p.dt;
    const int cap = p.bs_max_substeps;
    for (int c = 1; c >= 0; c--) {
        const int Wc = 2 << c;                      // 4, then 2 lanes a segment
        const int nq = d.ctl->ncls[c];
        const int seg = lane / Wc, sl = lane % Wc, base = seg * Wc;
        const unsigned segmask = ((1u << Wc) - 1u) << base;
        int g = -1, sz = 0, mslot = 0;
        double M0g = p.M0, GM0 = p.G * p.M0;   // the star of the segment's group
        double yv[6] = {0, 0, 0, 0, 0, 0}, z0[6] = {0, 0, 0, 0, 0, 0}, z1[6] = {0, 0, 0, 0, 0, 0};
        double t = 0.0, H = 0.0, El = 0.0;
        int k = 0, ms = 0, nsub = 0, last = 0, nmerge = 0;
        bool need = true;
        for (;;) {
            // segments that need a group take the next one of the class
            if (need && sl == 0) {
                const int q = atomicAdd(&d.ctl->qcls[c], 1);
                W.seg_g[seg] = q < nq ? d.gcls[c * d.gcap + q] : -1;
            }
            __syncwarp();
            if (need) {
                need = false;
                g = W.seg_g[seg];
                sz = g >= 0 ? d.goff[g + 1] - d.goff[g] : 0;
                if (g >= 0) {
                    M0g = d.M0s[d.body_sys[d.members[d.goff[g]]]];
                    GM0 = p.G * M0g;
                }
                W.alive[lane] = 0;
                W.big[lane] = 0;
                if (sl < sz) {
                    mslot = d.goff[g] + sl;
                    const int gb = d.members[mslot];
                    W.gid[lane] = gb;
                    yv[0] = d.x0[gb]; yv[1] = d.y0[gb]; yv[2] = d.z0[gb];
                    yv[3] = d.vx0[gb]; yv[4] = d.vy0[gb]; yv[5] = d.vz0[gb];
                    W.m[lane] = d.m[gb];
                    W.R[lane] = d.R[gb];
                    const double rc = d.rc[gb];
                    W.rc[lane] = rc;
                    W.rcf[lane] = __double2float_ru(rc);
                    W.prc2[lane] = rc * rc;
                    W.pc01[lane] = 0.1 * rc;
                    W.pinv[lane] = 1.0 / (0.9 * rc);
                    W.alive[lane] = d.alive[gb];
                    const SysInfo& gs = d.sys[d.body_sys[gb]];
                    W.big[lane] = gb - gs.off < gs.nb;
                }
                t = 0.0;
                H = dt;
                last = 0;
                if (fabs(H) >= fabs(dt - t)) {
                    H = dt - t;
                    last = 1;
                }
                k = 0;
                ms = 0;
                nsub = 0;
                El = 0.0;
                nmerge = 0;
            }
            __syncwarp();
            const bool active = g >= 0;
            if (!__any_sync(0xffffffffu, active)) break;   // the class is done for the whole warp
            const bool live = active && sl < sz;
            // evaluation point: the substep's start (ms == 0) or the midpoint chain
            {
                const bool st = ms == 0;
                W.px[lane] = st ? yv[0] : z1[0];
                W.py[lane] = st ? yv[1] : z1[1];
                W.pz[lane] = st ? yv[2] : z1[2];
                W.pf[lane] = near_record(W.px[lane], W.py[lane], W.pz[lane], W.rcf[lane]);
            }
            __syncwarp();
            double f[6] = {0, 0, 0, 0, 0, 0};
            if (live && W.alive[lane]) {
                const double P0 = W.px[lane], P1 = W.py[lane], P2 = W.pz[lane];
                const bool st = ms == 0;
                f[0] = st ? yv[3] : z1[3];
                f[1] = st ? yv[4] : z1[4];
                f[2] = st ? yv[5] : z1[5];
                const double r2 = bs_sq3(P0, P1, P2), ri = rsqrt(r2);
                const double sk = -GM0 * (ri * ri * ri);
                double ax = sk * P0, ay = sk * P1, az = sk * P2;
                const float4 me = W.pf[lane];
                unsigned near = 0;   // bit j: the j-th other lane of the segment may be in range
                for (int j = 0; j < Wc - 1; j++) {
                    const int o = base + j + (j >= sl ? 1 : 0);
                    if (near_pair(me, W.pf[o]) && W.alive[o] && W.big[o]) near |= 1u << j;
                }
                for (; near; near &= near - 1) {   // ascending
                    const int j = __ffs(near) - 1;
                    const int o = base + j + (j >= sl ? 1 : 0);
                    const int w = gt_nonneg(W.rc[lane], W.rc[o]) ? lane : o;
                    bs_pair(p, P0, P1, P2, W.px[o], W.py[o], W.pz[o], W.m[o], W.rc[w], W.prc2[w], W.pc01[w],
                            W.pinv[w], ax, ay, az);
                }
                f[3] = ax;
                f[4] = ay;
                f[5] = az;
            }
            const int n = 2 * (k + 1);
            const double h = H / n;
            const int stage = ms == 0 ? 0 : (ms < n ? 1 : 2);
            double cur[6] = {0, 0, 0, 0, 0, 0};
            bool pass = true;   // lanes without a live member never hold a segment back
            if (stage < 2) {
                // first step z1 = y + h f; then z0 <- z1, z1 <- z0 + 2 h f
                for (int q = 0; q < 6; q++) {
                    const double b0 = stage == 0 ? yv[q] : z0[q];
                    const double zn = b0 + (stage == 0 ? h : 2.0 * h) * f[q];
                    z0[q] = stage == 0 ? yv[q] : z1[q];
                    z1[q] = zn;
                }
            } else if (live) {
                double dsq_x = 0.0, dsq_v = 0.0, nx = 0.0, nv = 0.0;
                for (int q = 0; q < 6; q++) {
                    double cv = 0.5 * (z1[q] + z0[q] + h * f[q]), pv = 0.0;
                    for (int j = 1; j <= k; j++) {
                        const double up = W.row[j - 1][q][lane];
                        W.row[j - 1][q][lane] = cv;
                        pv = cv;
                        cv = cv + (cv - up) * kNeville[k][j];
                    }
                    W.row[k][q][lane] = cv;
                    cur[q] = cv;
                    const double df = cv - pv;
                    if (q < 3) {
                        dsq_x += df * df;
                        nx += cv * cv;
                    } else {
                        dsq_v += df * df;
                        nv += cv * cv;
                    }
                }
                if (k >= 1 && W.alive[lane]) {
                    // |dX|^2 <= tol^2 |X|^2 and the same for V; a NaN fails it
                    pass = dsq_x <= tol2 * fmax(nx, 2.3e-308) && dsq_v <= tol2 * fmax(nv, 2.3e-308);
                }
            }
            // the segment's members all pass (a ballot: no FP64 work)
            const bool seg_pass = (__ballot_sync(0xffffffffu, pass) & segmask) == segmask;
            // 0: on with the sequence, 1: next sequence, 2: accept row k, 3: reject the substep
            int decision = 0;
            if (active && stage == 2) {
                const bool acc = k >= 1 && seg_pass;
                decision = acc ? 2 : (k == kBsRows - 1 ? 3 : 1);
            }
            if (decision == 2 && live)
                for (int q = 0; q < 6; q++) W.y[q][lane] = cur[q];
            __syncwarp();
            // contacts after an accepted substep: each lane tests its pairs with
            // later members; the segment's first lane merges in the sequential order
            bool touch = false;
            if (decision == 2 && live && W.alive[lane])
                for (int o = lane + 1; o < base + sz; o++) {
                    if (!W.alive[o] || !bs_can_touch(W.m[lane], W.m[o])) continue;
                    const double ddx = cur[0] - W.y[0][o], ddy = cur[1] - W.y[1][o], ddz = cur[2] - W.y[2][o];
                    const double rs = W.R[lane] + W.R[o];
                    if (ddx * ddx + ddy * ddy + ddz * ddz <= rs * rs * (1.0 + 1e-9)) touch = true;
                }
            const unsigned tb = __ballot_sync(0xffffffffu, touch);
            if (decision == 2 && sl == 0 && (tb & segmask)) {
                for (int u = base; u < base + sz; u++)
                    for (int w = u + 1; w < base + sz && W.alive[u]; w++) {
                        if (!W.alive[w] || !bs_can_touch(W.m[u], W.m[w])) continue;
                        const double ddx = W.y[0][w] - W.y[0][u], ddy = W.y[1][w] - W.y[1][u],
                                     ddz = W.y[2][w] - W.y[2][u];
                        if (sqrt(ddx * ddx + ddy * ddy + ddz * ddz) <= W.R[u] + W.R[w])
                            bs_merge(W, p, M0g, u, w, El, nmerge);
                    }
            }
            __syncwarp();
            if (decision == 2 && live)
                for (int q = 0; q < 6; q++) yv[q] = W.y[q][lane];
            // step control (the same on every lane of a segment)
            if (active) {
                if (stage < 2) {
                    ms++;
                } else {
                    ms = 0;
                    if (decision == 1) {
                        k++;
                    } else {
                        nsub++;
                        bool fin = false, failed = false, hard = false;
                        if (decision == 2) {
                            t = last ? dt : t + H;
                            if (last) fin = true;
                            else if (k <= 2) H *= 2.0;
                            else if (k >= 6) H *= 0.5;
                        } else {
                            hard = fin = true;   // first attempt rejected: the lockstep kernels redo the group
                        }
                        if (!fin && nsub >= cap) fin = failed = true;
                        k = 0;
                        if (fin && hard) {
                            if (sl == 0) {
                                const int q = atomicAdd(&d.ctl->nhard, 1);
                                if (q < d.gcap) d.ghard[q] = g;
                                else set_status(d.ctl, kEoverflow, -7);
                            }
                            need = true;
                        } else if (fin) {
                            if (live) {
                                double* o = d.bsout + (int64_t)kBsOut * mslot;
                                for (int q = 0; q < 6; q++) o[q] = yv[q];
                                o[6] = W.m[lane];
                                o[7] = W.R[lane];
                                o[8] = (double)W.alive[lane];
                            }
                            if (sl == 0) {
                                d.glost[g] = El;
                                if (nmerge) atomicAdd(&d.ctl->nmerge, nmerge);
                                atomicAdd(&d.ctl->nsub, (unsigned long long)nsub);
                                if (failed) set_status(d.ctl, kEbs, g);
                            }
                            need = true;
                        } else {
                            last = 0;
                            if (fabs(H) >= fabs(dt - t)) {
                                H = dt - t;
                                last = 1;
                            }
                        }
                    }
                }
            }
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// Groups of up to 16 members (nearly every encounter): k_bs_ws<1> up to four
// members, k_bs_ws<4> five to sixteen.  The attempts (step sizes H, H/2, H/4,
// H/8, or H and H/2) are the blocks of a cluster; when every one is rejected
// the next round tries the following halvings, so the sizes tried and
// accepted are those of the sequential scheme.  Inside a block four roles share
// the work of a round (a warp each up to four members; else R warps, a quarter of the
// members, for roles 0 and 3 and half of the other warps each for roles 1 and 2), since a warp's FP64 instruction holds its scheduler's
// FP64 unit for 64 cycles whatever its dependences, so that what shortens a
// round is fewer instructions on the warp that waits:
//   role 0 keeps each (sequence, member) state and takes the midpoint steps;
//   roles 1 and 2 evaluate the (1 - K) mutual terms at the even and at the
//          odd evaluation points;
//   role 3 evaluates the stellar term at every point, in order, and then, two
//          points after a sequence has ended, its row of the extrapolation
//          tableau and the acceptance test, beside the other roles.
// In the midpoint sequence x_{m+1} = x_{m-1} + 2h v_m, v_{m+1} = v_{m-1} +
// 2h a(x_m), the position x_{m+2} needs a(x_m) but not a(x_{m+1}), so the
// accelerations at two successive points are computed at once: as soon as
// a(x_m) arrives, role 0 forms v_{m+1} and x_{m+2} and hands x_{m+2} to the
// role of its parity while the other role is still on a(x_{m+1}).  The
// arithmetic is that of the sequential scheme; up to four members a point's
// acceleration is the stellar term plus the sum of the mutual terms, above
// that the mutual terms are added to the stellar one in `sp` interleaved parts
// (as when sp lanes shared a member's terms), combined by a tree.  Four named
// barriers hand over positions and accelerations, one pair per parity, each
// met by role 0, the mutual role of its parity and the stellar role (above
// four members two more hand the stellar terms to the mutual roles); buffers
// are doubled by parity.  Lanes: k * nm + b (sequence k, member b).  Attempt 0
// announces its acceptance to the other blocks through distributed shared
// memory.
// Cycles of a substep accepted at the fourth row, one pair alone on its SM
// (1001 bodies): 63000 with the rows in role 0 and the addresses formed in the
// loops, 54000 so; the 16384-body disk's slowest group 163000 to 125000-139000,
// a dense ensemble's of six members 15900 to 9200 a round.
// what a member's pair with its j-th other member takes besides the positions
struct WsPair {
    double gm;                           // G m of the other member
    double rc, rc2, c01, inv;            // of the one with the larger rc: rc, rc^2, 0.1 rc, 1 / (0.9 rc)
    float rcf;                           // rc rounded up
    int src;                             // the other member is alive and big (a source of force)
};

// the unordered pairs with a source of a group of 5-16 members, and their terms
// at the points of both parities: separation (of the second from the first) and
// the factors of the term on the first and on the second
template <int RMAX>
struct WsTasks {
    static constexpr int kPairs = 4 * RMAX * (4 * RMAX - 1) / 2;
    int np;
    short first[kPairs], second[kPairs];
    short task[4 * RMAX][4 * RMAX - 1];      // of a member and its j-th other: pair index, -1 none
    double sep[2][kBsRows][3][kPairs], fac[2][kBsRows][2][kPairs];
};
template <>
struct WsTasks<1> {};

template <int RMAX>
struct WsSh {
    static constexpr int M = 4 * RMAX;
    WsTasks<RMAX> T;
    double y[6][M];                      // current state, component-major
    double pos[2][kBsRows][3][M];        // evaluation points, by parity of the round
    float4 posf[2][kBsRows][M];          // the same in float, with rc (rounded up), for near_pair
    double acc[2][kBsRows][3][M];        // mutual terms there (above four members: the whole acceleration)
    double sacc[2][kBsRows][3][M];       // stellar terms there
    double row[kBsRows][6][M];           // the last extrapolated row of each member
    double diag[kBsRows][6][M];          // T[k][k] of every finished row
    double raw[2][6][M];                 // midpoint result of a finished sequence, by parity of its row
    double df2[6][M], cur2[6][M];
    double m[M], R[M], rc[M];
    WsPair pc[M][M - 1];                 // set for a group and again after a merger
    int alive[M], gid[M], big[M];
    int kacc;                            // this block's attempt: accepted row, -1 while none
    int halt;                            // role 0's warps leave the rounds together (RMAX > 1)
    int stop;                            // role 0 tells the evaluating roles that the rounds are over
    int decision;                        // the substep number attempt 0 announced
    int dec, gi, collide, nmerge;
    int kq[4];
    double El;
};

constexpr int kBarPos0 = 1, kBarPos1 = 2;   // named barriers: evaluation points written (role 0 -> 1 or 2, and 3)
constexpr int kBarAcc0 = 3, kBarAcc1 = 4;   // accelerations written (role 1 or 2, and 3 -> 0)
constexpr int kBarStar0 = 5, kBarStar1 = 6; // stellar terms written (role 3 -> 1 or 2; RMAX > 1)
constexpr int kBarRow = 7, kBarHalt = 8;    // within role 3 (a row's squares written), within role 0 (halt written)
constexpr int kBarPair0 = 9, kBarPair1 = 10;   // within role 1 or 2 (the pairs' terms written; RMAX > 1)

// a named barrier met by the given number of threads (a multiple of 32)
__device__ __forceinline__ void ws_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void ws_bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Attempts a cluster: four when the encounter integrator has the GPU to
// itself (a rejected substep costs no extra round unless all four fail);
// two beside the kick, whose blocks then get the registers the other two
// would hold (measured on the 16384-body disk: the kick and the encounter
// branch end together, and the step is 2-3% shorter than with four).
constexpr int kWsAttemptsAlone = 4, kWsAttemptsBeside = 2, kWsAttemptsMid = 2;

// dsq <= tol2 * max(nsq, 2.3e-308) for squares (>= +0) on the integer units; a NaN fails
__device__ __forceinline__ bool ws_passes(double dsq, double nsq, double tol2) {
    const double n = __longlong_as_double(max(__double_as_longlong(nsq), __double_as_longlong(2.3e-308)));
    return __double_as_longlong(dsq) <= 0x7ff0000000000000ll && !gt_nonneg(dsq, tol2 * n);
}

// the pair's contact test: |d| <= rs, with the square root only near it
__device__ __forceinline__ bool ws_touch(double dx, double dy, double dz, double rs) {
    const double d2 = dx * dx + dy * dy + dz * dz;
    if (gt_nonneg(d2, rs * rs * (1.0 + 1e-9))) return false;
    return sqrt(d2) <= rs;
}

// (1 - K) factor of a pair at separation (dx, dy, dz): 0 out of range
__device__ __forceinline__ double ws_factor(const WsPair& c, int form, double dx, double dy, double dz) {
    const double dr2 = bs_sq3(dx, dy, dz);
    if (ge_nonneg(dr2, c.rc2)) return 0.0;   // 1 - K = 0 at or beyond rc
    const double dri = rsqrt(dr2), dr = __dmul_rn(dr2, dri);
    if (ge_nonneg(dr, c.rc)) return 0.0;
    return mutual_factor(c.gm * (dri * dri * dri), __dmul_rn(dr - c.c01, c.inv), form);
}

// FP32 test of near_pair with the pair's radius
__device__ __forceinline__ bool ws_near(const float4& a, const float4& b, float rcf) {
    const float dx = b.x - a.x, dy = b.y - a.y, dz = b.z - a.z;
    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    const float t = (rcf + a.w) * 1.00001f;
    return !(r2 > t * t);
}
__device__ __forceinline__ float4 ws_record(double x, double y, double z) {
    const float fx = trunc_f(x), fy = trunc_f(y), fz = trunc_f(z);
    return make_float4(fx, fy, fz, 0x1p-21f * (fabsf(fx) + fabsf(fy) + fabsf(fz)));
}

// A member's acceleration above four members: the stellar term and the mutual
// terms added in up to four interleaved parts, the parts by the tree
// (0 + 2) + (1 + 3) (parts without a term left out: they would add zeros).
struct WsParts {
    double s[4][3];
    unsigned used = 0;
    __device__ __forceinline__ WsParts(double x, double y, double z) {
        for (int q = 1; q < 4; q++)
            for (int c = 0; c < 3; c++) s[q][c] = 0.0;
        s[0][0] = x, s[0][1] = y, s[0][2] = z;
    }
    __device__ __forceinline__ void add(int part, double tf, double dx, double dy, double dz) {
        used |= 1u << part;
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (part == q) {
                s[q][0] = fma(tf, dx, s[q][0]);
                s[q][1] = fma(tf, dy, s[q][1]);
                s[q][2] = fma(tf, dz, s[q][2]);
            }
    }
    __device__ __forceinline__ void total() {
        if (used & 4u)
            for (int c = 0; c < 3; c++) s[0][c] += s[2][c];
        if (used & 8u)
            for (int c = 0; c < 3; c++) s[1][c] += s[3][c];
        if (used & 10u)
            for (int c = 0; c < 3; c++) s[0][c] += s[1][c];
    }
};

template <class SH>
__device__ __forceinline__ void ws_pairs(SH& S, const Params& p, int nm, int tid, int nt) {
    for (int e = tid; e < nm * (nm - 1); e += nt) {
        const int b = e / (nm - 1), j = e % (nm - 1), o = j + (j >= b ? 1 : 0);
        const double rc = gt_nonneg(S.rc[b], S.rc[o]) ? S.rc[b] : S.rc[o];   // rc_bo = max(rc_b, rc_o)
        WsPair& c = S.pc[b][j];
        c.gm = p.G * S.m[o];
        c.rc = rc;
        c.rc2 = rc * rc;
        c.c01 = 0.1 * rc;
        c.inv = 1.0 / (0.9 * rc);
        c.rcf = __double2float_ru(rc);
        c.src = S.alive[o] && S.big[o];
    }
}

// the group's list of pairs with a source (one thread: a group's setup, or after a merger)
template <class SH>
__device__ __forceinline__ void ws_list(SH& S, int nm) {
    int np = 0;
    for (int u = 0; u < nm; u++)
        for (int w = u + 1; w < nm; w++) {
            const bool any = S.alive[u] && S.alive[w] && (S.big[u] || S.big[w]);
            S.T.task[u][w - 1] = S.T.task[w][u] = (short)(any ? np : -1);
            if (any) {
                S.T.first[np] = (short)u;
                S.T.second[np] = (short)w;
                np++;
            }
        }
    S.T.np = np;
}

// The rounds of one substep, for the warps of the four roles (see above).  NM:
// the members, 0 when known only at run time (nm).  A lane's addresses and
// constants are set before its loop: alone on its scheduler, a warp pays four
// to six cycles for every dependent instruction beside the FP64 ones.
template <int RMAX, int NM, class PEER>
__device__ __forceinline__ void ws_rounds(WsSh<RMAX>& S, const Params& p, double GM0, double tol2, int nm_rt, int R,
                                          int RM, int role, int li, int sp, double Ha, int arank, int ca, int epoch,
                                          bool dense, PEER peer) {
    constexpr int M = WsSh<RMAX>::M;
    const int nm = NM ? NM : nm_rt;
    // threads at a barrier: positions (roles 0, 1 or 2, 3), accelerations, stellar terms
    const int nbp = 32 * (2 * R + RM), nb3 = 96 * R, nb2 = 64 * R;
    const int k = li / nm, b = li - k * nm;
    const bool act = k < kBsRows;
    const int n = act ? 2 * (k + 1) : -1;              // (an idle lane takes no point)
    const int kk = act ? k : 0;
    const bool alive = act && S.alive[b];
    if (role == 0) {
        // ---- role 0: states and midpoint steps.  At iteration m a lane
        // holds x_{m-1}, x_m, x_{m+1} and v_{m-1}, v_m.
        const double h = Ha / (2 * (k + 1)), h2 = 2.0 * h;
        double Xm[3], X0[3], X1[3], Vm[3], V0[3];
        for (int c = 0; c < 3; c++) Xm[c] = X0[c] = X1[c] = Vm[c] = V0[c] = 0.0;
        if (act) {
            for (int c = 0; c < 3; c++) {
                X0[c] = Xm[c] = S.y[c][b];
                V0[c] = Vm[c] = S.y[3 + c][b];
                S.pos[0][k][c][b] = X0[c];
                X1[c] = X0[c] + h * V0[c];   // x_1 = x_0 + h v_0
                S.pos[1][k][c][b] = X1[c];
            }
            if (NM != 2) {
                S.posf[0][k][b] = ws_record(X0[0], X0[1], X0[2]);
                S.posf[1][k][b] = ws_record(X1[0], X1[1], X1[2]);
            }
        }
        if (li == 0) {
            S.kacc = -1;
            S.stop = 0;
        }
        ws_bar_arrive(kBarPos0, nbp);        // points 0 and 1
        ws_bar_arrive(kBarPos1, nbp);
        for (int m = 0;; m++) {
            const int par = m & 1;
            double(*const pos)[M] = S.pos[par][kk];
            ws_bar_sync(par ? kBarAcc1 : kBarAcc0, nb3);   // a(x_m)
            if (m <= n) {
                double a[3] = {0.0, 0.0, 0.0};
                if (alive)
                    for (int c = 0; c < 3; c++)
                        a[c] = RMAX == 1 ? S.sacc[par][kk][c][b] + S.acc[par][kk][c][b] : S.acc[par][kk][c][b];
                if (m < n) {
                    const double hm = m == 0 ? h : h2;     // (v_{-1} is v_0)
                    for (int c = 0; c < 3; c++) {
                        const double vn = Vm[c] + hm * a[c];
                        // the point two ahead: x_{m+2} = x_m + 2h v_{m+1}
                        const double x2 = X0[c] + h2 * vn;
                        pos[c][b] = x2;                    // (past the sequence's end nobody reads it)
                        Xm[c] = X0[c];
                        X0[c] = X1[c];
                        X1[c] = x2;
                        Vm[c] = V0[c];
                        V0[c] = vn;
                    }
                    if (NM != 2) S.posf[par][kk][b] = ws_record(X1[0], X1[1], X1[2]);
                } else {
                    // sequence k done: its midpoint result 1/2 (z_n + z_{n-1} + h f(z_n))
                    for (int c = 0; c < 3; c++) {
                        S.raw[k & 1][c][b] = 0.5 * (X0[c] + Xm[c] + h * V0[c]);
                        S.raw[k & 1][3 + c][b] = 0.5 * (V0[c] + Vm[c] + h * a[c]);
                    }
                }
            }
            __syncwarp();
            ws_bar_arrive(par ? kBarPos1 : kBarPos0, nbp);   // point m + 2, and row m / 2 - 1
            // stop: this attempt accepted, attempt 0 announced, or every sequence done
            // (one look for all warps of the role, so that they leave together)
            int st = 0;
            if (RMAX == 1 || li == 0)
                st = *reinterpret_cast<volatile int*>(&S.kacc) >= 0 ||
                     *reinterpret_cast<volatile int*>(&S.decision) == epoch || m == 2 * kBsRows;
            if (RMAX == 1) {
                st = __shfl_sync(0xffffffffu, st, 0);
            } else {
                if (li == 0) S.halt = st;
                ws_bar_sync(kBarHalt, 32 * R);
                st = S.halt;   // (written again only after every warp has met the next Acc barrier)
            }
            if (st) {
                // the evaluations of points m + 1 and m + 2 are under way: take
                // (and drop) them, then release the roles with the stop flag
                ws_bar_sync(par ? kBarAcc0 : kBarAcc1, nb3);
                ws_bar_sync(par ? kBarAcc1 : kBarAcc0, nb3);
                if (li == 0) S.stop = 1;
                ws_bar_arrive(kBarPos0, nbp);
                ws_bar_arrive(kBarPos1, nbp);
                break;
            }
        }
    } else if (role == 3) {
        // ---- role 3: the stellar term at every point, in order, and the rows.
        // At the stop, role 0 releases both position barriers: this role
        // meets the second one too, which the other parity's role waits at.
        const int rc = li / nm, rb = li - rc * nm;     // component and member of a row's lane
        for (int m = 0;; m++) {
            const int par = m & 1;
            ws_bar_sync(par ? kBarPos1 : kBarPos0, nbp);
            if (*reinterpret_cast<volatile int*>(&S.stop)) {
                ws_bar_sync(par ? kBarPos0 : kBarPos1, nbp);
                break;
            }
            if (m <= n && alive) {
                const double px = S.pos[par][kk][0][b], py = S.pos[par][kk][1][b], pz = S.pos[par][kk][2][b];
                const double r2 = bs_sq3(px, py, pz), ri = rsqrt(r2);
                const double sk = -GM0 * (ri * ri * ri);
                S.sacc[par][kk][0][b] = sk * px;
                S.sacc[par][kk][1][b] = sk * py;
                S.sacc[par][kk][2][b] = sk * pz;
            }
            __syncwarp();
            if (RMAX > 1) ws_bar_arrive(par ? kBarStar1 : kBarStar0, nb2);
            ws_bar_arrive(par ? kBarAcc1 : kBarAcc0, nb3);
            if (m >= 4 && par == 0) {
                // row kr of the tableau: sequence kr ended at point m - 2.  Its raw
                // result is there since this point's position barrier, and its buffer
                // is next written after this role has arrived at point m + 2.
                const int kr = m / 2 - 2;
                if (rc < 6) {
                    double cur = S.raw[kr & 1][rc][rb], prev_col = 0.0;
                    for (int j = 1; j <= kr; j++) {
                        const double up = S.row[j - 1][rc][rb];
                        S.row[j - 1][rc][rb] = cur;
                        prev_col = cur;
                        cur = cur + (cur - up) * kNeville[kr][j];
                    }
                    S.row[kr][rc][rb] = cur;
                    S.diag[kr][rc][rb] = cur;
                    const double df = cur - prev_col;
                    S.df2[rc][rb] = df * df;
                    S.cur2[rc][rb] = cur * cur;
                }
                if (kr >= 1) {
                    if (RMAX == 1) __syncwarp();
                    else ws_bar_sync(kBarRow, 32 * R);
                    if (li < 32) {
                        bool pass = true;
                        if (li < nm && S.alive[li]) {
                            const double dsq_x = S.df2[0][li] + S.df2[1][li] + S.df2[2][li];
                            const double nx = S.cur2[0][li] + S.cur2[1][li] + S.cur2[2][li];
                            const double dsq_v = S.df2[3][li] + S.df2[4][li] + S.df2[5][li];
                            const double nv = S.cur2[3][li] + S.cur2[4][li] + S.cur2[5][li];
                            pass = ws_passes(dsq_x, nx, tol2) && ws_passes(dsq_v, nv, tol2);
                        }
                        // rows are tested in order: the first that passes is kept
                        if (__all_sync(0xffffffffu, pass) && li == 0 && S.kacc < 0) {
                            S.kacc = kr;
                            if (arank == 0)
                                for (int q = 0; q < ca; q++) peer(q)->decision = epoch;
                        }
                    }
                }
            }
        }
    } else if (role < 3) {
        // ---- roles 1 and 2: mutual terms at the points of their parity
        const int par = role - 1, form = p.changeover;
        const double(*const pk)[M] = S.pos[par][kk];
        const float4* const pf = S.posf[par][kk];
        const WsPair* const pc = S.pc[b];
        double(*const acc)[M] = S.acc[par][kk];
        // pairs as tasks where a lane would have several near ones to take one after another
        // (three big members) and the tasks are at most two a lane
        bool tasks = false;
        if constexpr (RMAX > 1) tasks = dense && kBsRows * S.T.np <= 64 * RM;
        for (int m = par;; m += 2) {
            ws_bar_sync(par ? kBarPos1 : kBarPos0, nbp);
            if (*reinterpret_cast<volatile int*>(&S.stop)) break;
            const bool live = m <= n && alive;
            if (RMAX == 1) {
                if (live) {
                    const double px = pk[0][b], py = pk[1][b], pz = pk[2][b];
                    double ax = 0.0, ay = 0.0, az = 0.0;
                    auto pair = [&](int j) {
                        const int o = j + (j >= b ? 1 : 0);
                        const double dx = pk[0][o] - px, dy = pk[1][o] - py, dz = pk[2][o] - pz;
                        const double tf = ws_factor(pc[j], form, dx, dy, dz);
                        if (__double_as_longlong(tf) << 1) {
                            ax = fma(tf, dx, ax);
                            ay = fma(tf, dy, ay);
                            az = fma(tf, dz, az);
                        }
                    };
                    if (NM == 2) {
                        if (pc[0].src) pair(0);
                    } else {
                        const float4 me = pf[b];
                        unsigned near = 0;   // bit j: the j-th other member (ascending) may be in range
#pragma unroll
                        for (int j = 0; j < (NM ? NM : M) - 1; j++)
                            if (j < nm - 1 && pc[j].src && ws_near(me, pf[j + (j >= b ? 1 : 0)], pc[j].rcf))
                                near |= 1u << j;
                        for (; near; near &= near - 1) pair(__ffs(near) - 1);
                    }
                    acc[0][b] = ax;
                    acc[1][b] = ay;
                    acc[2][b] = az;
                }
            } else if (!tasks) {
                // a lane's own terms, its first while the stellar terms are on their way
                if (li < 32 * R) {   // (whole warps)
                    unsigned near = 0;
                    double px = 0.0, py = 0.0, pz = 0.0;
                    if (live) {
                        px = pk[0][b], py = pk[1][b], pz = pk[2][b];
                        const float4 me = pf[b];
                        for (int j = 0; j < nm - 1; j++)
                            if (pc[j].src && ws_near(me, pf[j + (j >= b ? 1 : 0)], pc[j].rcf)) near |= 1u << j;
                    }
                    double tf = 0.0, dx = 0.0, dy = 0.0, dz = 0.0;
                    int part = 0;
                    auto next = [&] {
                        const int j = __ffs(near) - 1, o = j + (j >= b ? 1 : 0);
                        near &= near - 1;
                        part = j & (sp - 1);
                        dx = pk[0][o] - px, dy = pk[1][o] - py, dz = pk[2][o] - pz;
                        tf = ws_factor(pc[j], form, dx, dy, dz);
                    };
                    bool have = near != 0;
                    if (have) next();
                    __syncwarp();
                    ws_bar_sync(par ? kBarStar1 : kBarStar0, nb2);
                    if (live) {
                        WsParts a(S.sacc[par][kk][0][b], S.sacc[par][kk][1][b], S.sacc[par][kk][2][b]);
                        while (have) {
                            if (__double_as_longlong(tf) << 1) a.add(part, tf, dx, dy, dz);   // (in range after all)
                            have = near != 0;
                            if (have) next();
                        }
                        a.total();
                        for (int c = 0; c < 3; c++) acc[c][b] = a.s[0][c];
                    }
                }
            } else if constexpr (RMAX > 1) {
                // the pairs of the sequences still running, one a lane, both ways at once: the
                // factors share the separation, 1 / r^3 and the changeover
                const int np = S.T.np, k0 = m <= 2 ? 0 : (m + 1) / 2 - 1;   // sequences with n >= m
                for (int e = li; e < (kBsRows - k0) * np; e += 32 * RM) {
                    const int q = e / np, pr = e - q * np, ks = k0 + q;
                    const int u = S.T.first[pr], w = S.T.second[pr];
                    const WsPair& c = S.pc[u][w - 1];
                    double fu = 0.0, fw = 0.0;
                    if (ws_near(S.posf[par][ks][u], S.posf[par][ks][w], c.rcf)) {
                        const double(*const x)[M] = S.pos[par][ks];
                        const double dx = x[0][w] - x[0][u], dy = x[1][w] - x[1][u], dz = x[2][w] - x[2][u];
                        const double dr2 = bs_sq3(dx, dy, dz);
                        if (!ge_nonneg(dr2, c.rc2)) {
                            const double dri = rsqrt(dr2), dr = __dmul_rn(dr2, dri);
                            if (!ge_nonneg(dr, c.rc)) {
                                const double ri3 = dri * dri * dri, y = __dmul_rn(dr - c.c01, c.inv);
                                if (c.src) fu = mutual_factor(c.gm * ri3, y, form);
                                const WsPair& cw = S.pc[w][u];
                                if (cw.src) fw = mutual_factor(cw.gm * ri3, y, form);
                            }
                        }
                        S.T.sep[par][ks][0][pr] = dx;
                        S.T.sep[par][ks][1][pr] = dy;
                        S.T.sep[par][ks][2][pr] = dz;
                    }
                    S.T.fac[par][ks][0][pr] = fu;
                    S.T.fac[par][ks][1][pr] = fw;
                }
                __syncwarp();
                ws_bar_sync(par ? kBarPair1 : kBarPair0, 32 * RM);
                if (li < 32 * R) {   // (whole warps) each member's terms, in the order of its others
                    ws_bar_sync(par ? kBarStar1 : kBarStar0, nb2);
                    if (live) {
                        WsParts a(S.sacc[par][kk][0][b], S.sacc[par][kk][1][b], S.sacc[par][kk][2][b]);
                        for (int j = 0; j < nm - 1; j++) {
                            const int pr = S.T.task[b][j];
                            if (pr < 0) continue;
                            const int way = j >= b ? 0 : 1;
                            double tf = S.T.fac[par][kk][way][pr];
                            if (!(__double_as_longlong(tf) << 1)) continue;
                            // (the separation of the first from the second has the other sign)
                            if (way) tf = -tf;
                            a.add(j & (sp - 1), tf, S.T.sep[par][kk][0][pr], S.T.sep[par][kk][1][pr],
                                  S.T.sep[par][kk][2][pr]);
                        }
                        a.total();
                        for (int c = 0; c < 3; c++) acc[c][b] = a.s[0][c];
                    }
                }
            }
            __syncwarp();
            if (RMAX == 1 || li < 32 * R) ws_bar_arrive(par ? kBarAcc1 : kBarAcc0, nb3);
        }
    }
}

// Registers: six blocks an SM of the small form beside the kick's; the other holds its 512 threads
// alone at 128, without spills (held to 96, 80 or 64 it spills 16 to 52 bytes, and steps of 16 and 256
// systems, 33000 and 263000 bodies and the disk are the same within 1%).
template <int RMAX, int CA>
__global__ void __launch_bounds__(128 * RMAX, RMAX == 1 ? 6 : 1) k_bs_ws(Dev d) {
    OPAL_TIMELINE_SCOPE((RMAX == 1 ? kTlBsWs : kTlBs16));
    constexpr int NT = 128 * RMAX;
    extern __shared__ __align__(16) unsigned char ws_smem[];   // one WsSh
    WsSh<RMAX>& S = *reinterpret_cast<WsSh<RMAX>*>(ws_smem);
    __shared__ int s_gi;
    constexpr int M = WsSh<RMAX>::M;
    static_assert(CA >= 1 && CA <= 4, "one to four attempts a cluster");
    cg::cluster_group cl = cg::this_cluster();
    // (no status check: every block of a cluster must take the same path, and
    // another kernel may set the status while the cluster's blocks start)
    const Params p = d.p;
    const bool many = d.ctl->ngroups > kBsManyGroups;
    // the groups it looks at: up to four members, all of them or what the packed
    // kernel left; above, the list of those of 5-16 members
    const int* list = RMAX > 1 ? d.gmid : (many ? d.ghard : nullptr);
    const int ng = RMAX > 1 ? d.ctl->nmid : (many ? d.ctl->nhard : d.ctl->ngroups);
    // Many groups: every block its own group, one attempt (no block waits for
    // another of its cluster).  The groups then fill the SMs' FP64 units, and
    // the further attempts, few of which are ever taken (62 substeps in 59
    // rounds of the ensemble's longest group), would slow all of them down.
    const bool solo = RMAX > 1 ? many || ng > kBsSoloMid : d.ctl->ngroups > kBsSoloGroups;
    const int ca = solo ? 1 : CA;
    const int arank = solo ? 0 : (int)cl.block_rank();
    auto csync = [&] {
        if (ca > 1) cl.sync();
        else __syncthreads();
    };
    auto peer = [&](int q) { return ca > 1 ? cl.map_shared_rank(&S, q) : &S; };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cap = p.bs_max_substeps;
    const double tol2 = p.bs_tol * p.bs_tol;
    int epoch = 0;
    if (tid == 0) S.decision = -1;
    for (;;) {
        __syncthreads();
        if (arank == 0 && tid == 0) S.gi = atomicAdd(&d.ctl->qlock[RMAX == 1 ? 0 : 1], 1);
        csync();
        if (tid == 0) s_gi = peer(0)->gi;
        csync();
        const int gi = s_gi;
        if (gi >= ng) break;
        const int g = list ? list[gi] : gi;
        const int mb = d.goff[g], nm = d.goff[g + 1] - mb;
        if (nm > M) continue;                // a larger group: another lockstep kernel's
        const double M0g = d.M0s[d.body_sys[d.members[mb]]], GM0 = p.G * M0g;   // the group's star
        const int R = RMAX == 1 ? 1 : (nm + 3) / 4;        // warps of roles 0 and 3
        // and of roles 1 and 2: the rest of the block's in halves (above four members)
        const int RM = RMAX == 1 ? 1 : 2 * RMAX - R;
        const int role = warp < R ? 0 : (warp < R + RM ? 1 : (warp < R + 2 * RM ? 2 : 3));
        const int li = (warp - (role == 0 ? 0 : (role == 1 ? R : (role == 2 ? R + RM : R + 2 * RM)))) * 32 + lane;
        int nbg = 0;
        if (RMAX > 1)
            for (int q = 0; q < nm; q++) {
                const int gb = d.members[mb + q];
                const SysInfo& gs = d.sys[d.body_sys[gb]];
                nbg += gb - gs.off < gs.nb ? 1 : 0;
            }
        int sp_full = 1;                                   // parts a member's mutual terms are added in
        while (RMAX > 1 && 2 * sp_full * kBsRows * nm <= 256 && 2 * sp_full <= nbg) sp_full *= 2;
        if (tid < nm) {
            const int gb = d.members[mb + tid];
            S.gid[tid] = gb;
            S.y[0][tid] = d.x0[gb];
            S.y[1][tid] = d.y0[gb];
            S.y[2][tid] = d.z0[gb];
            S.y[3][tid] = d.vx0[gb];
            S.y[4][tid] = d.vy0[gb];
            S.y[5][tid] = d.vz0[gb];
            S.m[tid] = d.m[gb];
            S.R[tid] = d.R[gb];
            S.rc[tid] = d.rc[gb];
            S.alive[tid] = d.alive[gb];
            const SysInfo& gs = d.sys[d.body_sys[gb]];
            S.big[tid] = gb - gs.off < gs.nb;
        }
        if (tid == 0) {
            S.El = 0.0;
            S.nmerge = 0;
        }
        __syncthreads();
        ws_pairs(S, p, nm, tid, NT);
        if constexpr (RMAX > 1)
            if (tid == NT - 1) ws_list(S, nm);
        __syncthreads();
        const double dt = p.dt;
        double t = 0.0, H = dt;
        int nsub = 0, failed = 0, finished = 0;
        while (!finished && !failed) {
            double rem = dt - t;
            int last0 = 0;
            if (fabs(H) >= fabs(rem)) {
                H = rem;
                last0 = 1;
            }
            epoch++;
            // with many groups the whole step is tried first with the terms in
            // one part (the order the packed kernel's attempts have)
            const int sp = RMAX > 1 && many && nsub == 0 ? 1 : sp_full;
            const double Ha = ldexp(H, -arank);
            auto rounds = [&](auto members) {
                ws_rounds<RMAX, decltype(members)::value>(S, p, GM0, tol2, nm, R, RM, role, li, sp, Ha, arank, ca,
                                                          epoch, nbg >= 3, peer);
            };
            if (RMAX > 1) rounds(std::integral_constant<int, 0>());
            else if (nm == 2) rounds(std::integral_constant<int, 2>());
            else if (nm == 3) rounds(std::integral_constant<int, 3>());
            else if (nm == 4) rounds(std::integral_constant<int, 4>());
            else rounds(std::integral_constant<int, 0>());   // (one member: the test hook)
            __syncthreads();
            // every block is out of its rounds: the first accepted attempt in
            // halving order is taken, the same in every block
            csync();
            if (tid == 0) {
                int dcs = ca;
                for (int q = ca - 1; q >= 0; q--) {
                    S.kq[q] = peer(q)->kacc;
                    if (S.kq[q] >= 0) dcs = q;
                }
                S.dec = dcs;
            }
            __syncthreads();
            const int dec = S.dec;
            // replay the sequential control flow over the attempts just made
            for (int q = 0; q < ca; q++) {
                nsub++;
                const double Hq = ldexp(H, -q);
                if (q == dec) {
                    const int kacc = S.kq[q];
                    if (tid < 6 * nm) S.y[tid / nm][tid % nm] = peer(q)->diag[kacc][tid / nm][tid % nm];
                    const int lastq = (q == 0) ? last0 : 0;
                    t = lastq ? dt : t + Hq;
                    if (tid == 0) S.collide = 0;
                    __syncthreads();
                    // any pair in contact?  (exact sequential resolution only if so)
                    for (int e = tid; e < nm * nm; e += NT) {
                        const int u = e / nm, w = e % nm;
                        if (w > u && S.alive[u] && S.alive[w] && bs_can_touch(S.m[u], S.m[w])) {
                            const double dx = S.y[0][w] - S.y[0][u], dy = S.y[1][w] - S.y[1][u],
                                         dz = S.y[2][w] - S.y[2][u];
                            if (ws_touch(dx, dy, dz, S.R[u] + S.R[w])) S.collide = 1;
                        }
                    }
                    __syncthreads();
                    if (S.collide && tid == 0) {
                        for (int u = 0; u < nm; u++)
                            for (int w = u + 1; w < nm && S.alive[u]; w++) {
                                if (!S.alive[w] || !bs_can_touch(S.m[u], S.m[w])) continue;
                                const double dx = S.y[0][w] - S.y[0][u], dy = S.y[1][w] - S.y[1][u],
                                             dz = S.y[2][w] - S.y[2][u];
                                if (ws_touch(dx, dy, dz, S.R[u] + S.R[w]))
                                    bs_merge(S, p, M0g, u, w, S.El, S.nmerge);
                            }
                    }
                    __syncthreads();
                    if (lastq) {
                        finished = 1;
                        break;
                    }
                    if (S.collide) {   // masses and live flags may have changed
                        ws_pairs(S, p, nm, tid, NT);
                        if constexpr (RMAX > 1)
                            if (tid == NT - 1) ws_list(S, nm);
                        __syncthreads();
                    }
                    H = Hq;
                    if (kacc <= 2) H *= 2.0;
                    else if (kacc >= 6) H *= 0.5;
                    if (nsub >= cap) failed = 1;
                    break;
                }
                if (nsub >= cap) {   // attempt q rejected
                    failed = 1;
                    break;
                }
            }
            if (dec == ca && !failed) H = ldexp(H, -ca);   // every attempt rejected
            // no block resets its accepted row or overwrites its tableau before
            // every block has read them
            csync();
        }
        if (failed) {
            if (tid == 0 && arank == 0) set_status(d.ctl, kEbs, g);
            return;
        }
        if (tid < nm && arank == 0) {
            double* o = d.bsout + (int64_t)kBsOut * (mb + tid);
            for (int c = 0; c < 6; c++) o[c] = S.y[c][tid];
            o[6] = S.m[tid];
            o[7] = S.R[tid];
            o[8] = (double)S.alive[tid];
        }
        if (tid == 0 && arank == 0) {
            d.glost[g] = S.El;
            if (S.nmerge) atomicAdd(&d.ctl->nmerge, S.nmerge);
            atomicAdd(&d.ctl->nsub, (unsigned long long)nsub);
        }
    }
}

cudaError_t bs_setup() {
    cudaError_t e = cudaFuncSetAttribute(k_bs_packed, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kPkWarps * sizeof(PkWarp)));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_bs_ws<4, kWsAttemptsMid>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(WsSh<4>));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_bs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BsSh));
}

void launch_bs_packed(const Dev& d, int nsm, cudaStream_t s) {
    // one block of four warps an SM, one a scheduler (a scheduler's FP64 unit takes 64 cycles a warp
    // instruction, so a second warp there would wait for the first): the ensemble's first attempts
    // 2.6 ms with two warps, 1.52 with four, 1.45 with eight, a few hundred groups 0.41, 0.42 and 0.46
    if (d.ntot / 2 <= kBsManyGroups) return;   // (a group has two members at least)
    k_bs_packed<<<nsm, 32 * kPkWarps, kPkWarps * sizeof(PkWarp), s>>>(d);
    prof_mark("bs: many groups, packed");
}

// The encounter kernels after grouping: the packed kernel (unless the caller
// has launched it) and the groups of up to 4 members on s, those of 5-16 on the
// branch s2 and the larger ones on s3 (s2 == s: one after the other).  Within a stream priority,
// blocks are placed in launch order, and a kernel whose blocks do not fit yet
// holds back the kernels launched after it.  beside (the kick runs beside, on a
// stream of lower priority than s2, which is lower than s; the packed kernel
// has run before the kick's fork): the small-group kernel goes first, since
// beside the kick's blocks only its blocks fit (a larger-group block takes half
// an SM's registers or more).  Otherwise the larger-group kernels go first, on a
// branch of the same priority (their longest group is an ensemble's longest
// chain), and the packed and small-group blocks fill the room they leave.  The
// small-group clusters hold two attempts beside the kick, four otherwise.
cudaError_t launch_bs(const Dev& d, int nsm, cudaStream_t s, cudaStream_t s2, cudaStream_t s3, cudaEvent_t fork,
                      cudaEvent_t join, cudaEvent_t join3, bool beside) {
    cudaError_t err = cudaSuccess;   // the first failed launch, if any (the cluster and cooperative ones)
    if (d.nmax <= 4) s2 = s3 = s;    // (no larger groups)
    if (s2 != s) {
        cudaEventRecord(fork, s);
        cudaStreamWaitEvent(s2, fork, 0);
        if (s3 != s2) cudaStreamWaitEvent(s3, fork, 0);
    }
    auto clusters = [&](auto kernel, size_t smem, int ca, int blocks, int threads, cudaStream_t st) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((blocks + ca - 1) / ca * ca));
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = ca;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, d);
        if (err == cudaSuccess) err = e;
    };
    // no more blocks than groups of at least so many members can form
    const int64_t bodies = (int64_t)d.nmax * d.nsys;
    auto room = [&](int least, int64_t blocks) { return (int)std::min<int64_t>(blocks, std::max<int64_t>(1, bodies / least)); };
    auto larger = [&] {
        if (d.nmax <= 4) return;   // (kernels whose groups cannot form are left out)
        clusters(k_bs_ws<4, kWsAttemptsMid>, sizeof(WsSh<4>), kWsAttemptsMid,
                 kWsAttemptsMid * room(5, nsm / kWsAttemptsMid), 512, s2);
        if (s2 == s) prof_mark("bs: groups of 5-16");
        if (d.nmax <= 16) return;
        k_bs<<<room(17, nsm), kBsThreads, sizeof(BsSh), s3>>>(d);
        if (s2 == s) prof_mark("bs: groups of 17-64");
        if (d.nmax <= 64) return;
        const cudaError_t e = launch_bs_huge(d, nsm, s3);
        if (err == cudaSuccess) err = e;
    };
    if (!beside) {
        larger();
        launch_bs_packed(d, nsm, s);
    }
    // groups of up to 4 members: clusters of two or four blocks, one attempt each
    if (beside) clusters(k_bs_ws<1, kWsAttemptsBeside>, sizeof(WsSh<1>), kWsAttemptsBeside,
                         kWsAttemptsBeside * room(2, 2 * nsm), 128, s);
    else clusters(k_bs_ws<1, kWsAttemptsAlone>, sizeof(WsSh<1>), kWsAttemptsAlone,
                  kWsAttemptsAlone * room(2, 2 * nsm), 128, s);
    prof_mark("bs: groups <= 4");
    if (beside) larger();
    if (s2 != s) {
        cudaEventRecord(join, s2);
        cudaStreamWaitEvent(s, join, 0);
        if (s3 != s2) {
            cudaEventRecord(join3, s3);
            cudaStreamWaitEvent(s, join3, 0);
        }
    }
    return err;
}

}  // namespace opal
