// Bulirsch-Stoer of an encounter group of more than 64 members (a giant
// planet's critical sphere holding hundreds of small bodies), on the whole
// GPU: the blocks of a team in step through barriers of the team.
//
// The method is the sequential one of the small-group kernels (Sec. 2.1.1
// footnote 2; modified midpoint n_k = 2, 4, ..., 16, Neville extrapolation in
// h^2, the same acceptance test and step control, perfect mergers in the
// sequential order after each accepted substep).  The midpoint sequences advance in
// lockstep, one barrier a round: round r evaluates the derivative at the r-th
// point of every sequence with n_k >= r (round 0 at the substep's start) and
// takes the step; rows k >= 1 of the tableau are tested in the sequential order.
//
// What bounds it: a round is latency, the barrier (3 us with its fences), loads of what other
// SMs wrote (1 us a trip) and the FP64 instructions of one warp on its scheduler, about
// 64 cycles each.
//  - Members lie in spatial order, a lane a member, 32 to a warp.  Which members can come
//    near one another is searched once a substep, with the contacts at its start, and
//    listed for each warp (huge_search): the points of all sequences and rounds lie within
//    a bound of the start carried along with the group, which each member checks as it
//    moves (a round in which one has not kept it takes every pair).  A round tests the
//    listed pairs in FP32 and takes the few inside their critical radius in FP64, a lane a pair.
//    A search each round, by boxes, took half of it.
//  - Members of wide critical radius (a giant planet: the whole group is near it) are kept
//    out of that search.  Every lane takes its member's pair with each of them, and the
//    same (1 - K) / r^3 serves both: the wide member's side is summed over the warp, the
//    block, and then, in the next round, by every block for itself from the blocks' sums.
//    So every block holds the wide members' state (in shared memory, the same bits in each),
//    which saves the second barrier a round in which one block would step them.
//  - The tableau row of a sequence that has ended is formed a round later, by warps of its
//    own beside the other sequences' steps (up to 120 FP64 operations of a lane, which made
//    the ending sequence's units the longest by half); it is tested a round later too.
//  - Two teams of blocks, each on every SM, take the groups in turn: the latencies of two
//    groups overlap.
//  - Where most pairs are near (no boxes or lists help) the FP64 pipes bound it: fewer members
//    to a warp, as many as spread the sequences that are left over all warps.  A group with a few near ones
//    to each member takes fewer members to a warp too, and lists.
//  - The loops of a round are kept small and the long parts out of line: a warp runs them once
//    through, and with everything inlined the instruction caches bound it.
// Two steps of 131072 bodies with Jupiter's and Saturn's groups of 1665 and 800 members: 1063
// to 116 ms in one system (a round of the larger 37 to 19 us, and half of the rounds hidden behind it), in
// others 4.8 to 9.2 times less than before, by the substeps that their steps take;
// 150 members all near one another 6.9 to 5.7 ms, 600 of them 1.075 s before and after.
// Every thread takes the same decisions from the same values, so the control flow is
// identical in all blocks of a team.  A barrier that waits longer than its limit
// (four seconds; a test hook sets it shorter) sets an abort flag: every block
// leaves and the step reports OPAL_EBS.
#include <algorithm>

#include "opal_internal.cuh"

namespace opal {

constexpr int kHugeThreads = 32 * (kHugeUnitWarps + 1);   // the last warp serves the wide members
constexpr float kHugeFar = 3.0e18f;   // float coordinate of slots that are no candidates (finite squares)

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Barrier of a team's blocks (all blocks of the launch are resident); false once aborted.
// The count only grows: a block waits until it reaches target, the arrivals up to this
// barrier (one trip to the other SMs where resetting a count and then raising a flag
// take two).  Each wait is bounded by wait_ns of the global timer.  hold (a test hook):
// wait for one arrival more, so that every wait runs out, as if a block never arrived.
__device__ bool huge_sync(HugeCtl* hc, unsigned int target, unsigned long long wait_ns, int hold) {
    __shared__ int ok;   // (one reading of the flag for the whole block)
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned int* count = &hc->bar_count;
        const unsigned int want = target + (unsigned)hold;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        atomicAdd(&hc->bar_count, 1u);
        const unsigned long long t0 = global_ns();
        for (unsigned int poll = 1; (int)(*count - want) < 0; poll++) {
            if (poll % 16) continue;
            if (*(volatile int*)&hc->abort) break;
            if (global_ns() - t0 > wait_ns) {
                atomicExch(&hc->abort, 1);
                break;
            }
        }
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        ok = *(volatile int*)&hc->abort == 0;
    }
    __syncthreads();
    return ok != 0;
}

// Arrays of evaluation points: parity of the round x 8 + sequence, and two for the
// substep's start (the current one, and the one that a tableau row proposes).
constexpr int kHugeY = 2 * kBsRows;
__device__ __forceinline__ double* huge_pos(const HugeBuf& H, int a) { return H.pos + (int64_t)a * 3 * H.cap; }
__device__ __forceinline__ float4* huge_posf(const HugeBuf& H, int a) { return H.posf + (int64_t)a * H.cap; }
__device__ __forceinline__ float4* huge_box(const HugeBuf& H, int a) {   // (of the start arrays)
    return H.box + (int64_t)(a - kHugeY) * 3 * huge_boxes(H.cap);
}
// what a member can reach in h, apart from the group's drift; m: its motion (w: radius),
// speed against the drift (x, half as much again) and acceleration (y, taken four times)
__device__ __forceinline__ float4* huge_mot(const HugeBuf& H, int a) { return H.mot + (int64_t)(a - kHugeY) * H.cap; }
__device__ __forceinline__ float huge_reach(float4 m, float h) { return h * fmaf(2.0f * h, m.y, m.x); }

// G m (1 - K) / r^3 (gm: G m) of a pair inside the larger critical radius of the two, else 0.
// The arithmetic, its order and its contraction are written out: with one term near it, a
// member's acceleration then has the same bits in whatever order this kernel sums the others,
// and a step decision within rounding of the tolerance falls the same way.
// (Hardware approximations in place of the library's rsqrt and division save 10 of 34 FP64
// operations and nothing of a round's time; step decisions then fell differently in one run
// of eight, after which bodies deep inside the giant's sphere differed by up to 3e-7.)  Not
// inlined: a round's code runs once through, and what does not stay in the instruction caches
// costs more than the call.
__device__ __noinline__ double huge_factor(double dx, double dy, double dz, double rcb, double pinvb, double rco,
                                           double pinvo, double gm, int form) {
    const bool first = gt_nonneg(rcb, rco);
    const double rc = first ? rcb : rco;
    const double dr2 = fma(dz, dz, fma(dx, dx, __dmul_rn(dy, dy)));
    if (ge_nonneg(dr2, __dmul_rn(rc, rc))) return 0.0;   // 1 - K = 0 at or beyond rc
    const double dri = rsqrt(dr2), dr = __dmul_rn(dr2, dri);
    if (ge_nonneg(dr, rc)) return 0.0;
    const double y = __dmul_rn(fma(-0.1, rc, dr), first ? pinvb : pinvo);
    return mutual_factor(__dmul_rn(gm, __dmul_rn(__dmul_rn(dri, dri), dri)), y, form);
}

// Sums over the warp of three doubles, in six additions: lanes 0, 8 and 16 hold
// them (every lane of the warp calls it).
__device__ __forceinline__ double warp_sum3(double a, double b, double c) {
    const unsigned full = 0xffffffffu;
    const bool h = threadIdx.x & 16, g = threadIdx.x & 8;
    double p = h ? c : a, q = h ? 0.0 : b;
    p += __shfl_xor_sync(full, h ? a : c, 16);
    const double qo = __shfl_xor_sync(full, h ? b : 0.0, 16);
    q += qo;
    double v = g ? q : p;
    v += __shfl_xor_sync(full, g ? p : q, 8);
    v += __shfl_xor_sync(full, v, 4);
    v += __shfl_xor_sync(full, v, 2);
    v += __shfl_xor_sync(full, v, 1);
    return v;
}

// Gap between a point (or box) and a box, squared: FP32 subtraction, squares and sums
// round monotonically, so a box's gap is at most a pair's (the factor 1.001 of the tests
// covers a contraction into an FMA).
__device__ __forceinline__ float gap2(float4 alo, float4 ahi, float4 blo, float4 bhi) {
    const float gx = fmaxf(0.0f, fmaxf(blo.x - ahi.x, alo.x - bhi.x));
    const float gy = fmaxf(0.0f, fmaxf(blo.y - ahi.y, alo.y - bhi.y));
    const float gz = fmaxf(0.0f, fmaxf(blo.z - ahi.z, alo.z - bhi.z));
    return gx * gx + gy * gy + gz * gz;
}
__device__ __forceinline__ float huge_slack(float4 p) { return 1e-5f * (1.0f + fabsf(p.x) + fabsf(p.y) + fabsf(p.z)); }

// The box of a warp's members (have) to the box array: lo, hi, and the largest of rc and
// twice the radius, of the speeds and of the accelerations.
__device__ __noinline__ void box_store(bool have, float4 p, float4 m, float4* dst) {
    int lo[3], hi[3];
    const float c[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        lo[k] = __reduce_min_sync(0xffffffffu, have ? ford(c[k]) : 0x7fffffff);
        hi[k] = __reduce_max_sync(0xffffffffu, have ? ford(c[k]) : (int)0x80000000);
    }
    auto most = [&](float v) { return __int_as_float(__reduce_max_sync(0xffffffffu, have ? __float_as_int(v) : 0)); };   // (v >= 0)
    const float e = most(fmaxf(fabsf(p.w), 2.0f * m.w)), s = most(m.x), ac = most(m.y);
    if ((threadIdx.x & 31) == 0) {
        const bool none = lo[0] == 0x7fffffff;
        dst[0] = none ? make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.0f) : make_float4(fordinv(lo[0]), fordinv(lo[1]), fordinv(lo[2]), 0.0f);
        dst[1] = none ? make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.0f) : make_float4(fordinv(hi[0]), fordinv(hi[1]), fordinv(hi[2]), 0.0f);
        dst[2] = make_float4(s, ac, 0.0f, e);
    }
}

// Pairs of a warp's L members (slots L u + lane; have: a live member that is not wide)
// with the massive others that are not wide, near enough at the substep's start (array a)
// that they may come within the critical radius or touch in a substep of h.
// kHugeList: to the warp's list (its count -1 if it has no room), which then serves every
// round of every sequence of the substep.  kHugeCount: their number, to hc->nnear.
// pb: the member's place in float with rc (negative: a massless body), mo its motion.
// A warp tests the boxes of the other warps' members against its own, then its members
// against a box that is near, then the few members near it against the 32 slots there,
// four at a time, with the loads of the next three runs of 32 in flight, all in FP32 with a margin
// far above its rounding.  Every lane of the warp calls it.
enum { kHugeList, kHugeCount };
constexpr int kHugeTry = 4;
struct HugeQueue {
    float4 mem[32];              // the warp's members in float
    float reach[32];
    unsigned mine[32];           // lanes whose pair is each member's
    int j[32];                   // near runs of 32 slots, and which of the warp's members are near each
    unsigned near[32];
};
template <int MODE>
__device__ __noinline__ void huge_search(const HugeBuf& H, HugeCtl* hc, int a, int L, int u, int M, bool have, float4 pb,
                                         float4 mo, float h, HugeQueue& Q) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, nb = (M + L - 1) / L;
    const int run = 32 / L;                  // the boxes of one run of 32 slots
    const unsigned sub = 0xffffffffu >> (32 - run);
    const float4* bx = huge_box(H, a);
    const float4* pf = huge_posf(H, a);
    const float4* mt = huge_mot(H, a);
    // a pair is near within the larger of the two's sizes (rc, or twice the radius, so that a contact
    // is one) and what both can reach
    auto size = [](float w, float4 m) { return fmaxf(w, 2.0f * m.w); };
    const float sz = size(fabsf(pb.w), mo), rch = huge_reach(mo, h);
    const float4 ulo = bx[3 * u], uhi = bx[3 * u + 1], um = bx[3 * u + 2];
    const float usz = um.w, urch = huge_reach(um, h);
    const float slack = huge_slack(make_float4(fmaxf(fabsf(ulo.x), fabsf(uhi.x)), fmaxf(fabsf(ulo.y), fabsf(uhi.y)),
                                               fmaxf(fabsf(ulo.z), fabsf(uhi.z)), 0.0f));
    int* list = H.list + (int64_t)u * kHugeListed;
    __syncwarp();
    Q.mem[lane] = make_float4(pb.x, pb.y, pb.z, sz);
    Q.reach[lane] = rch;
    int cnt = 0;   // pairs, the same for every lane
    const int any_have = __any_sync(full, have);
    for (int j0 = 0; any_have && j0 < nb; j0 += 32) {
        float4 lo = make_float4(0.0f, 0.0f, 0.0f, 0.0f), hi = lo;
        float bsz = 0.0f, brch = 0.0f;
        bool live = false;
        if (j0 + lane < nb) {
            lo = bx[3 * (j0 + lane)];
            hi = bx[3 * (j0 + lane) + 1];
            const float4 m = bx[3 * (j0 + lane) + 2];
            bsz = m.w;
            brch = huge_reach(m, h);
            const float lim = fmaxf(usz, bsz) + urch + brch + slack;
            live = !(gap2(ulo, uhi, lo, hi) > lim * lim * 1.001f);
        }
        unsigned lm = __ballot_sync(full, live);
        int nq = 0;
#pragma unroll 1
        while (lm) {
            const int f = __ffs(lm) - 1;
            lm &= ~(sub << (f / run * run));
            bool near = have;
            if (L == 32) {   // (with fewer members a warp they are all tried)
                const float4 l = make_float4(__shfl_sync(full, lo.x, f), __shfl_sync(full, lo.y, f), __shfl_sync(full, lo.z, f), 0.0f);
                const float4 h = make_float4(__shfl_sync(full, hi.x, f), __shfl_sync(full, hi.y, f), __shfl_sync(full, hi.z, f), 0.0f);
                const float bl = fmaxf(sz, __shfl_sync(full, bsz, f)) + rch + __shfl_sync(full, brch, f) + slack;
                near = have && !(gap2(pb, pb, l, h) > bl * bl * 1.001f);
            }
            const unsigned nm = __ballot_sync(full, near);
            if (nm && lane == 0) {
                Q.j[nq] = (j0 + f) / run;
                Q.near[nq] = nm;
            }
            nq += nm ? 1 : 0;
        }
        __syncwarp();
        // the others of run q, and the next two
        float4 po[3], qo[3];
        auto fetch = [&](int q, float4& p, float4& m) {
            const int o = q < nq ? 32 * Q.j[q] + lane : M;
            p = o < M ? pf[o] : make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f);
            m = o < M ? mt[o] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        };
#pragma unroll
        for (int q = 0; q < 3; q++) fetch(q, po[q], qo[q]);
#pragma unroll 1
        for (int q = 0; q < nq; q++) {
            const float4 p = po[0];
            const float osz = size(fabsf(p.w), qo[0]), orch = huge_reach(qo[0], h) + slack;
            const int o = 32 * Q.j[q] + lane;
            const bool src = __float_as_int(p.w) >= 0;   // (a massless body is no source)
            po[0] = po[1];
            qo[0] = qo[1];
            po[1] = po[2];
            qo[1] = qo[2];
            fetch(q + 3, po[2], qo[2]);
            unsigned nm = Q.near[q];
#pragma unroll 1
            while (nm) {
                int s[kHugeTry];
                unsigned hm[kHugeTry], any = 0;
#pragma unroll
                for (int e = 0; e < kHugeTry; e++) {
                    const bool one = nm != 0;
                    s[e] = one ? __ffs(nm) - 1 : 0;
                    nm &= nm - 1;   // (0 stays 0)
                    const float4 b = Q.mem[s[e]];
                    const float dx = p.x - b.x, dy = p.y - b.y, dz = p.z - b.z;
                    const float lim = fmaxf(b.w, osz) + Q.reach[s[e]] + orch;
                    const bool hit = one && src && o != L * u + s[e] && dx * dx + dy * dy + dz * dz < lim * lim;
                    hm[e] = __ballot_sync(full, hit);
                    any |= hm[e];
                }
                if (!any) continue;
#pragma unroll
                for (int e = 0; e < kHugeTry; e++) {
                    const int at = cnt + __popc(hm[e] & ((1u << lane) - 1u));
                    if (MODE == kHugeList && ((hm[e] >> lane) & 1u) && at < kHugeListed) list[at] = s[e] | (o << 5);
                    cnt += __popc(hm[e]);
                }
            }
        }
        __syncwarp();
    }
    if (MODE == kHugeCount) {
        if (lane == 0 && cnt) atomicAdd(&hc->nnear, cnt);
        return;
    }
    if (lane == 0) H.listed[u] = cnt <= kHugeListed ? cnt : -1;
}

// The contacts of one pair of slots at the start array a (the lower member first): a both
// massive pair is met from either side, and taken from the lower slot's
__device__ __forceinline__ void huge_contact(const HugeBuf& H, HugeCtl* hc, int a, int i, int o) {
    const double* pos = huge_pos(H, a);
    const int64_t c = H.cap;
    if (o < i && !le_zero(H.m[i])) return;
    const double dx = pos[o] - pos[i], dy = pos[c + o] - pos[c + i], dz = pos[2 * c + o] - pos[2 * c + i];
    const double rt = H.R[i] + H.R[o];
    if (dx * dx + dy * dy + dz * dz <= rt * rt * (1.0 + 1e-9)) {
        const int q = atomicAdd(&hc->ncand, 1);
        if (q < kHugeCand) hc->cand[q] = H.gid[i] < H.gid[o] ? make_int2(i, o) : make_int2(o, i);
    }
}

// The FP64 terms of a warp's listed pairs (n of them) at the points of array a, added to acc:
// an FP32 test, then a pair a lane; each member adds its pairs in the list's order.
__device__ __noinline__ void huge_listed(const Dev& d, const HugeBuf& H, int a, int u, int n, double x, double y, double z,
                                         float4 pb, double rc, double pinv, HugeQueue& Q, double (&acc)[3]) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, form = d.p.changeover;
    const float4* pf = huge_posf(H, a);
    const double* pos = huge_pos(H, a);
    const int* list = H.list + (int64_t)u * kHugeListed;
    const int64_t c = H.cap;
    __syncwarp();
    Q.mem[lane] = make_float4(pb.x, pb.y, pb.z, fabsf(pb.w));
    __syncwarp();
    for (int e0 = 0; e0 < n; e0 += 32) {
        const int ent = e0 + lane < n ? list[e0 + lane] : 0, s = ent & 31, o = ent >> 5;
        const float4 b = Q.mem[s], p = pf[o];
        const float dx = p.x - b.x, dy = p.y - b.y, dz = p.z - b.z;
        const float lim = fmaxf(b.w, fabsf(p.w)) + huge_slack(b);
        const bool hit = e0 + lane < n && dx * dx + dy * dy + dz * dz < lim * lim;
        if (!__any_sync(full, hit)) continue;
        Q.mine[lane] = 0u;
        __syncwarp();
        const double xs = __shfl_sync(full, x, s), ys = __shfl_sync(full, y, s), zs = __shfl_sync(full, z, s);
        const double rs = __shfl_sync(full, rc, s), ps = __shfl_sync(full, pinv, s);
        double tx = 0.0, ty = 0.0, tz = 0.0;
        if (hit) {
            const double ex = pos[o] - xs, ey = pos[c + o] - ys, ez = pos[2 * c + o] - zs;
            const double w = huge_factor(ex, ey, ez, rs, ps, H.rc[o], H.pinv[o], d.p.G * H.m[o], form);
            tx = w * ex;
            ty = w * ey;
            tz = w * ez;
            atomicOr(&Q.mine[s], 1u << lane);
        }
        __syncwarp();
        unsigned mine = Q.mine[lane];
        while (__any_sync(full, mine != 0)) {
            const int src = mine ? __ffs(mine) - 1 : lane;
            const double vx = __shfl_sync(full, tx, src), vy = __shfl_sync(full, ty, src), vz = __shfl_sync(full, tz, src);
            if (mine) {
                acc[0] += vx;
                acc[1] += vy;
                acc[2] += vz;
            }
            mine &= mine - 1;
        }
        __syncwarp();
    }
}

// The same for all others, where most pairs are near or the lists do not serve: a member at a time, the
// others across the lanes, summed over the warp once a member.
__device__ __noinline__ void huge_dense(const Dev& d, const HugeBuf& H, int a, int L, int u, int M, bool have, double x, double y,
                           double z, float4 pb, double rc, double pinv, double (&acc)[3]) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, form = d.p.changeover;
    const float4* pf = huge_posf(H, a);
    const double* pos = huge_pos(H, a);
    const int64_t c = H.cap;
    const float slack = huge_slack(pb);
    for (unsigned nm = __ballot_sync(full, have); nm; nm &= nm - 1) {
        const int s = __ffs(nm) - 1;
        const float fx = __shfl_sync(full, pb.x, s), fy = __shfl_sync(full, pb.y, s), fz = __shfl_sync(full, pb.z, s);
        const float fw = __shfl_sync(full, fabsf(pb.w), s), sl = __shfl_sync(full, slack, s);
        const double xs = __shfl_sync(full, x, s), ys = __shfl_sync(full, y, s), zs = __shfl_sync(full, z, s);
        const double rs = __shfl_sync(full, rc, s), ps = __shfl_sync(full, pinv, s);
        double tx = 0.0, ty = 0.0, tz = 0.0;
        float4 po[4];
        for (int o0 = lane; o0 - lane < M; o0 += 128) {   // (four loads in flight)
#pragma unroll
            for (int q = 0; q < 4; q++) po[q] = o0 + 32 * q < M ? pf[o0 + 32 * q] : make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f);
            unsigned hit = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float dx = po[q].x - fx, dy = po[q].y - fy, dz = po[q].z - fz;
                const float lim = fmaxf(fw, fabsf(po[q].w)) + sl;
                if (dx * dx + dy * dy + dz * dz < lim * lim && __float_as_int(po[q].w) >= 0 && o0 + 32 * q != L * u + s)
                    hit |= 1u << q;
            }
#pragma unroll 1
            for (int q = 0; q < 4; q++) {
                if (!((hit >> q) & 1u)) continue;
                const int o = o0 + 32 * q;
                const double ex = pos[o] - xs, ey = pos[c + o] - ys, ez = pos[2 * c + o] - zs;
                const double w = huge_factor(ex, ey, ez, rs, ps, H.rc[o], H.pinv[o], d.p.G * H.m[o], form);
                tx = fma(w, ex, tx);
                ty = fma(w, ey, ty);
                tz = fma(w, ez, tz);
            }
        }
        __syncwarp();
        const double v = warp_sum3(tx, ty, tz);
        const double vx = __shfl_sync(full, v, 0), vy = __shfl_sync(full, v, 8), vz = __shfl_sync(full, v, 16);
        if (lane == s) {
            acc[0] += vx;
            acc[1] += vy;
            acc[2] += vz;
        }
    }
}

// 2D Morton key of a point quantised to 16 bits an axis
__device__ __forceinline__ unsigned int spread16(unsigned int v) {
    v &= 0xffffu;
    v = (v | (v << 8)) & 0x00ff00ffu;
    v = (v | (v << 4)) & 0x0f0f0f0fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

// exact contact test of two members, by slot (the small-group kernels' comparison);
// two small bodies never touch.  pos, vel: the substep's start
__device__ __forceinline__ bool huge_touch(const HugeBuf& H, const double* pos, int u, int w) {
    if (!bs_can_touch(H.m[u], H.m[w])) return false;
    const int64_t c = H.cap;
    const double dx = pos[w] - pos[u], dy = pos[c + w] - pos[c + u], dz = pos[2 * c + w] - pos[2 * c + u];
    return sqrt(dx * dx + dy * dy + dz * dz) <= H.R[u] + H.R[w];
}

// perfect merger of the members in slots b and q (as the small-group kernels merge)
__device__ void huge_merge(const Dev& d, const HugeBuf& H, double* pos, double* vel, double M0, int b, int q, double& El,
                           int& survivor) {
    const int64_t c = H.cap;
    const double G = d.p.G;
    const double mb = H.m[b], mq = H.m[q], M = mb + mq;
    double X[2][6];
    for (int k = 0; k < 3; k++) {
        X[0][k] = pos[k * c + b];
        X[1][k] = pos[k * c + q];
        X[0][3 + k] = vel[k * c + b];
        X[1][3 + k] = vel[k * c + q];
    }
    double dd[3] = {X[1][0] - X[0][0], X[1][1] - X[0][1], X[1][2] - X[0][2]};
    double xn[3], vn[3];
    for (int k = 0; k < 3; k++) {
        xn[k] = (mb * X[0][k] + mq * X[1][k]) / M;
        vn[k] = (mb * X[0][3 + k] + mq * X[1][3 + k]) / M;
    }
    const double vb2 = X[0][3] * X[0][3] + X[0][4] * X[0][4] + X[0][5] * X[0][5];
    const double vq2 = X[1][3] * X[1][3] + X[1][4] * X[1][4] + X[1][5] * X[1][5];
    const double rb = sqrt(X[0][0] * X[0][0] + X[0][1] * X[0][1] + X[0][2] * X[0][2]);
    const double rq = sqrt(X[1][0] * X[1][0] + X[1][1] * X[1][1] + X[1][2] * X[1][2]);
    const double rbq = sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]);
    const double e_before = 0.5 * mb * vb2 + 0.5 * mq * vq2 - G * M0 * mb / rb - G * M0 * mq / rq - G * mb * mq / rbq;
    const double vn2 = vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2];
    const double rn = sqrt(xn[0] * xn[0] + xn[1] * xn[1] + xn[2] * xn[2]);
    const double e_after = 0.5 * M * vn2 - G * M0 * M / rn;
    El += e_before - e_after;
    int keep, gone;
    if (mb > mq) keep = b, gone = q;
    else if (mq > mb) keep = q, gone = b;
    else keep = (H.gid[b] < H.gid[q]) ? b : q, gone = (keep == b) ? q : b;
    const double Rn = cbrt(H.R[b] * H.R[b] * H.R[b] + H.R[q] * H.R[q] * H.R[q]);
    for (int k = 0; k < 3; k++) {
        pos[k * c + keep] = xn[k];
        vel[k * c + keep] = vn[k];
    }
    H.m[keep] = M;
    H.R[keep] = Rn;
    H.m[gone] = 0.0;
    H.alive[gone] = 0;
    survivor = keep;
}

// lexicographic order of pairs of slots by their bodies (the sequential sweep's order)
__device__ __forceinline__ bool pair_before(const HugeBuf& H, int2 a, int2 b) {
    const int ax = H.gid[a.x], bx = H.gid[b.x];
    return ax < bx || (ax == bx && H.gid[a.y] < H.gid[b.y]);
}

// the sequential sweep over the contacts found, by one thread: sorted, then in
// order; a merger moves its survivor, whose new contacts later in the order join the list
__device__ void huge_sweep(const Dev& d, const HugeBuf& H, HugeCtl* hc, int M, double* pos, double* vel, double M0) {
    int nc = min(hc->ncand, kHugeCand);
    if (hc->ncand > kHugeCand) set_status(d.ctl, kEoverflow, -8);
    for (int i = 1; i < nc; i++) {
        const int2 x = hc->cand[i];
        int j = i - 1;
        while (j >= 0 && pair_before(H, x, hc->cand[j])) {
            hc->cand[j + 1] = hc->cand[j];
            j--;
        }
        hc->cand[j + 1] = x;
    }
    for (int i = 0; i < nc; i++) {
        const int2 pr = hc->cand[i];
        if (!H.alive[pr.x] || !H.alive[pr.y] || !huge_touch(H, pos, pr.x, pr.y)) continue;
        double El = hc->El;
        int sv = -1;
        huge_merge(d, H, pos, vel, M0, pr.x, pr.y, El, sv);
        hc->El = El;
        hc->nmerge++;
        for (int x = 0; x < M; x++) {
            if (x == sv || !H.alive[x] || !huge_touch(H, pos, sv, x)) continue;
            const int2 np = H.gid[sv] < H.gid[x] ? make_int2(sv, x) : make_int2(x, sv);
            if (!pair_before(H, pr, np)) continue;   // the sweep is past that pair
            bool have = false;
            for (int j = i + 1; j < nc; j++)
                if (hc->cand[j].x == np.x && hc->cand[j].y == np.y) have = true;
            if (have) continue;
            if (nc >= kHugeCand) {
                set_status(d.ctl, kEoverflow, -8);
                break;
            }
            int j = nc++;
            while (j > i + 1 && pair_before(H, np, hc->cand[j - 1])) {
                hc->cand[j] = hc->cand[j - 1];
                j--;
            }
            hc->cand[j] = np;
        }
    }
}

// Row k of the tableau for the member in slot i (in place; sequences end in order), from the
// sequence's last value; a failed test marks hc->err.  With k >= 1 the row also proposes
// the next substep's start: its place, velocity, motion and box.  own: a slot that is not wide,
// have: its member is alive.  Every lane of the warp calls it.
__device__ __noinline__ void huge_row(const HugeBuf& H, HugeCtl* hc, int k, int ysel, int u, int i, bool slot, bool own,
                                      bool have, int attempt, double tol2, const double (&vg)[3], bool dense) {
    const int64_t c = H.cap;
    const int B = kHugeY + (ysel ^ 1);
    bool good = true;   // |dX|^2 <= tol^2 |X|^2 and the same for V; a NaN fails it
    float4 pf = make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f), mn = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float v2 = 0.0f;
    if (have) {
        pf.w = huge_posf(H, kHugeY + ysel)[i].w;
        mn.y = H.ska[i];
        mn.w = huge_mot(H, kHugeY + ysel)[i].w;
    }
#pragma unroll 1
    for (int e3 = 0; e3 < 6; e3 += 3) {   // (three components' loads together)
        double up[3][kBsRows], sq = 0.0, nr = 0.0;
#pragma unroll
        for (int e = 0; e < 3; e++) up[e][0] = own ? H.sk[(e3 + e) * c + i] : 0.0;
#pragma unroll
        for (int j = 1; j < kBsRows; j++)
#pragma unroll
            for (int e = 0; e < 3; e++) up[e][j] = own && j <= k ? H.row[((int64_t)(j - 1) * 6 + e3 + e) * c + i] : 0.0;
#pragma unroll
        for (int e = 0; e < 3; e++) {
            double cv = up[e][0], pv = 0.0;
#pragma unroll
            for (int j = 1; j < kBsRows; j++)
                if (j <= k) {
                    if (own) H.row[((int64_t)(j - 1) * 6 + e3 + e) * c + i] = cv;
                    pv = cv;
                    cv = cv + (cv - up[e][j]) * kNeville[k][j];
                }
            if (own) H.row[((int64_t)k * 6 + e3 + e) * c + i] = cv;
            const double df = cv - pv;
            sq += df * df;
            nr += cv * cv;
            if (own && k >= 1) {
                if (e3 == 0) huge_pos(H, B)[e * c + i] = cv;
                else H.yv[((int64_t)(ysel ^ 1) * 3 + e) * c + i] = cv;
            }
            const float fv = trunc_f(e3 == 0 ? cv : cv - vg[e]);
            if (e3 == 0 && have) (e == 0 ? pf.x : e == 1 ? pf.y : pf.z) = fv;
            if (e3 == 3) v2 = fmaf(fv, fv, v2);
        }
        good = good && sq <= tol2 * fmax(nr, 2.3e-308);
    }
    if (k == 0) return;
    if (have && !good) *(volatile int*)&hc->err[k] = attempt;
    if (have) mn.x = 1.5f * sqrtf(v2);
    if (slot) {
        huge_posf(H, B)[i] = pf;
        huge_mot(H, B)[i] = mn;
    }
    if (!dense) box_store(have, pf, mn, huge_box(H, B) + 3 * u);
}

// A block's copy of the wide members, the same in every block of the team.
struct HugeSh {
    double y[kHugeWide][6], ty[kHugeWide][6];   // substep's start, and the state a row proposes
    double z0[kBsRows][kHugeWide][6], z1[kBsRows][kHugeWide][6], row[kBsRows][kHugeWide][6];
    double base[kBsRows][kHugeWide][3];         // star and other wide members at this round's points
    double F[kBsRows][kHugeWide][3];            // the whole acceleration at the last round's
    double red[kHugeUnitWarps][kHugeWide][3];   // the warps' sums of the members' side
    double m[kHugeWide], gm[kHugeWide], igm[kHugeWide];   // (G m and its reciprocal)
    double rc[kHugeWide], pinv[kHugeWide], R[kHugeWide];
    double sq[kHugeWide][6][2];                 // squares of a row's error and value
    int alive[kHugeWide], slot[kHugeWide];
    HugeQueue q[kHugeUnitWarps];
    int nwide;
    int fail[kBsRows];                          // the last attempt in which one of them failed each row's test
};

__global__ void __launch_bounds__(kHugeThreads, 3) k_bs_huge(Dev d, int nsm) {
    OPAL_TIMELINE_SCOPE(kTlBsHuge);
    __shared__ HugeSh S;
    const int nh = d.ctl->nhuge;
    if (nh == 0) return;   // fixed before the launch: the same in every block
    // one group alone: all blocks are its team (until it turns out not to need them)
    int nblk = nh == 1 ? kHugeTeams * nsm : nsm;
    const int team = (int)blockIdx.x / nblk, blk = (int)blockIdx.x % nblk;
    HugeCtl* hc = d.hctl + team;
    const unsigned long long wait_ns = (unsigned long long)d.huge_wait_ns;
    const int hold = d.huge_hold;
    unsigned int arrivals = 0;   // of the team up to the next barrier
    auto sync = [&] {
        arrivals += (unsigned)nblk;
        return huge_sync(hc, arrivals, wait_ns, hold);
    };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool lead = blk == 0 && tid == 0;
    // status set before this kernel: block 0 looks, everyone follows
    if (lead) hc->skip = *(volatile int*)&d.ctl->status;
    if (!sync()) {
        if (lead) set_status(d.ctl, kEbs, kHugeAbortDetail);   // no group started: a barrier wait ran out
        return;
    }
    if (*(volatile int*)&hc->skip) return;
    const Params& p = d.p;
    const HugeBuf& H = d.hb[team];
    const int64_t c = H.cap;
    const double dt = p.dt, tol2 = p.bs_tol * p.bs_tol, G = p.G;
    const int form = p.changeover;
    int64_t gt = (int64_t)blk * kHugeThreads + tid, nt = (int64_t)nblk * kHugeThreads;
    int gw = blk * kHugeUnitWarps + warp, nw = nblk * kHugeUnitWarps;   // (unit warps)
    int attempt = 0;   // substeps tried by this team: marks a row's failure in hc->err
    for (int hi = team; hi < nh; hi += kHugeTeams) {
        const int g = d.ghuge[hi];
        const int m0 = d.goff[g], M = d.goff[g + 1] - m0;
        const double M0g = d.M0s[d.body_sys[d.members[m0]]], GM0 = G * M0g;   // the group's star
        if (lead) {
            hc->El = 0.0;
            hc->nmerge = 0;
            hc->ncand = 0;
            hc->nnear = 0;
            hc->bb[0] = hc->bb[2] = 0x7fffffff;
            hc->bb[1] = hc->bb[3] = (int)0x80000000;
            hc->rcmm[0] = 0;
            hc->rcmm[1] = 0x7fffffff;
        }
        // The members in spatial order, once a step: a 2D Morton key of each
        // start position over the group's box, ranked (ties by member), so that
        // 32 consecutive slots are compact.
        bool ok = sync();
        if (ok) {
            int lx = 0x7fffffff, hx = (int)0x80000000, ly = 0x7fffffff, hy = (int)0x80000000;
            int rmax = 0, rmin = 0x7fffffff;
            for (int64_t b = gt; b < M; b += nt) {
                const int gb = d.members[m0 + b];
                const int fx = ford((float)d.x0[gb]), fy = ford((float)d.y0[gb]);
                lx = min(lx, fx);
                hx = max(hx, fx);
                ly = min(ly, fy);
                hy = max(hy, fy);
                if (d.alive[gb]) {
                    const int rb = __float_as_int(__double2float_ru(d.rc[gb]));   // rc >= 0: bits order as values
                    rmax = max(rmax, rb);
                    rmin = min(rmin, rb);
                }
            }
            lx = __reduce_min_sync(0xffffffffu, lx);
            hx = __reduce_max_sync(0xffffffffu, hx);
            ly = __reduce_min_sync(0xffffffffu, ly);
            hy = __reduce_max_sync(0xffffffffu, hy);
            rmax = __reduce_max_sync(0xffffffffu, rmax);
            rmin = __reduce_min_sync(0xffffffffu, rmin);
            if (lane == 0) {

                atomicMin(&hc->bb[0], lx);
                atomicMax(&hc->bb[1], hx);
                atomicMin(&hc->bb[2], ly);
                atomicMax(&hc->bb[3], hy);
                atomicMax(&hc->rcmm[0], rmax);
                atomicMin(&hc->rcmm[1], rmin);
            }
            ok = sync();
        }
        if (ok) {
            const float x0 = fordinv(*(volatile int*)&hc->bb[0]), x1 = fordinv(*(volatile int*)&hc->bb[1]);
            const float y0 = fordinv(*(volatile int*)&hc->bb[2]), y1 = fordinv(*(volatile int*)&hc->bb[3]);
            const float sx = 65535.0f / fmaxf(x1 - x0, 1e-30f), sy = 65535.0f / fmaxf(y1 - y0, 1e-30f);
            for (int64_t b = gt; b < M; b += nt) {
                const int gb = d.members[m0 + b];
                const unsigned qx = (unsigned)fminf(65535.0f, fmaxf(0.0f, ((float)d.x0[gb] - x0) * sx));
                const unsigned qy = (unsigned)fminf(65535.0f, fmaxf(0.0f, ((float)d.y0[gb] - y0) * sy));
                H.key[b] = spread16(qx) | (spread16(qy) << 1);
            }
            ok = sync();
        }
        int ysel = 0;   // which of the two start arrays is current
        if (ok) {
            for (int64_t b = gt; b < M; b += nt) {
                const unsigned kb = H.key[b];
                int rank = 0;
                for (int o = 0; o < M; o++) {
                    const unsigned ko = H.key[o];
                    rank += (ko < kb || (ko == kb && o < (int)b)) ? 1 : 0;
                }
                const int gb = d.members[m0 + b];
                H.perm[rank] = (int)b;
                if (b == 0) hc->ref = rank;
                H.gid[rank] = gb;
                double* pos = huge_pos(H, kHugeY);
                pos[rank] = d.x0[gb];
                pos[c + rank] = d.y0[gb];
                pos[2 * c + rank] = d.z0[gb];
                H.yv[rank] = d.vx0[gb];
                H.yv[c + rank] = d.vy0[gb];
                H.yv[2 * c + rank] = d.vz0[gb];
                H.m[rank] = d.m[gb];
                H.R[rank] = d.R[gb];
                H.rc[rank] = d.rc[gb];
                H.pinv[rank] = 1.0 / (0.9 * d.rc[gb]);
                H.alive[rank] = d.alive[gb];
            }
            ok = sync();   // the slots are complete before anyone reads them
        }
        if (!ok) {
            if (lead) set_status(d.ctl, kEbs, kHugeAbortDetail + 1 + g);
            return;
        }
        // wide members: rc above a quarter of the largest, when that is over 8 times the
        // smallest; the first kHugeWide of them in slot order (any others are searched as the rest)
        if (warp == 0) {
            const float rmx = __int_as_float(*(volatile int*)&hc->rcmm[0]);
            const float rmn = __int_as_float(*(volatile int*)&hc->rcmm[1]);
            int n = 0;
            if (rmx > 8.0f * rmn)
                for (int i0 = 0; i0 < M && n < kHugeWide; i0 += 32) {
                    const int i = i0 + lane;
                    const bool w = i < M && H.alive[i] && __double2float_ru(H.rc[i]) > 0.25f * rmx;
                    const unsigned bm = __ballot_sync(0xffffffffu, w);
                    const int at = n + __popc(bm & ((1u << lane) - 1u));
                    if (w && at < kHugeWide) S.slot[at] = i;
                    n = min(kHugeWide, n + __popc(bm));
                }
            if (lane == 0) S.nwide = n;
            if (lane < kBsRows) S.fail[lane] = 0;
        }
        __syncthreads();
        const int nwide = S.nwide;
        auto is_wide = [&](int i) {
            bool w = false;
            for (int q = 0; q < nwide; q++) w |= S.slot[q] == i;
            return w;
        };
        // members a warp takes, and the warps' and the blocks' units of a sequence
        int L, nu, nv;
        auto units = [&](int l) {
            L = l;
            nu = (M + L - 1) / L;
            nv = (nu + kHugeUnitWarps - 1) / kHugeUnitWarps;
        };
        units(32);
        bool dense = false;   // most pairs near: no boxes, a warp's share by the sequences that are left
        // from the slots' state: the block's copy of the wide members, and the float
        // places and boxes of the current start array
        auto refresh = [&] {
            const double* pos = huge_pos(H, kHugeY + ysel);
            const double* vel = H.yv + (int64_t)ysel * 3 * c;
            if (dense) units(32);
            const int ref = *(volatile int*)&hc->ref;
            double vr[3];
            for (int e = 0; e < 3; e++) vr[e] = vel[e * c + (nwide > 0 ? S.slot[0] : ref)];
            for (int q = tid; q < nwide; q += kHugeThreads) {
                const int i = S.slot[q];
                for (int e = 0; e < 3; e++) {
                    S.y[q][e] = pos[e * c + i];
                    S.y[q][3 + e] = vel[e * c + i];
                }
                S.m[q] = H.m[i];
                S.gm[q] = G * H.m[i];
                S.igm[q] = S.gm[q] > 0.0 ? 1.0 / S.gm[q] : 0.0;
                S.R[q] = H.R[i];
                S.rc[q] = H.rc[i];
                S.pinv[q] = H.pinv[i];
                S.alive[q] = H.alive[i];
            }
            __syncthreads();
            if (warp < kHugeUnitWarps)
                for (int u = gw; u < nu; u += nw) {
                    const int i = L * u + lane;
                    const bool slot = lane < L && i < M, have = slot && H.alive[i] && !is_wide(i);
                    float4 pf = make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f);
                    if (have) {
                        const float rc = __double2float_ru(H.rc[i]);
                        pf = make_float4((float)pos[i], (float)pos[c + i], (float)pos[2 * c + i], le_zero(H.m[i]) ? -rc : rc);
                    }
                    if (slot) huge_posf(H, kHugeY + ysel)[i] = pf;
                    float4 mo = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (have) {
                        float v2 = 0.0f;
                        for (int e = 0; e < 3; e++) {
                            const float q = (float)(vel[e * c + i] - vr[e]);
                            v2 = fmaf(q, q, v2);
                        }
                        float ac = (float)GM0 / (pf.x * pf.x + pf.y * pf.y + pf.z * pf.z);
                        for (int w = 0; w < nwide; w++) {
                            const float dx = (float)S.y[w][0] - pf.x, dy = (float)S.y[w][1] - pf.y, dz = (float)S.y[w][2] - pf.z;
                            ac += (float)(G * S.m[w]) / fmaxf(dx * dx + dy * dy + dz * dz, 1e-20f);
                        }
                        mo = make_float4(1.5f * sqrtf(v2), ac, 0.0f, __double2float_ru(H.R[i]));
                    }
                    if (slot) huge_mot(H, kHugeY + ysel)[i] = mo;
                    if (!dense) box_store(have, pf, mo, huge_box(H, kHugeY + ysel) + 3 * u);
                }
            return sync();
        };
        ok = refresh();
        if (ok) {
            // A group in which a member is near more than one other (without the wide ones) is
            // bound by those pairs: fewer members to a warp then spread them over the SMs
            if (warp < kHugeUnitWarps)
                for (int u = gw; u < nu; u += nw) {
                    const int i = 32 * u + lane;
                    const bool have = i < M && H.alive[i] && !is_wide(i);
                    const float4 pf = i < M ? huge_posf(H, kHugeY)[i] : make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f);
                    huge_search<kHugeCount>(H, hc, kHugeY, 32, u, M, have, pf,
                                            i < M ? huge_mot(H, kHugeY)[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f), 0.0f, S.q[warp]);
                }
            ok = sync();
        }
        if (ok) {
            const int near = *(volatile int*)&hc->nnear;
            dense = near > (int64_t)M * M / 8;
            if (!dense && nblk > nsm) {   // blocks beyond one an SM would only make the barriers longer
                if (blk >= nsm) return;
                nblk = nsm;
                nt = (int64_t)nblk * kHugeThreads;
                nw = nblk * kHugeUnitWarps;
            }
            if (!dense && near > M) {
                int l = 2;
                while (l < 32 && ((M + l - 1) / l > kHugeSmallBoxes || (M + l - 1) / l * kBsRows > nw)) l *= 2;
                units(l);
                ok = refresh();
            }
        }
        if (!ok) {
            if (lead) set_status(d.ctl, kEbs, kHugeAbortDetail + 1 + g);
            return;
        }
        // the substep's pair lists and the contacts at its start, hs its length: while a member
        // stays within its reach of the group's drift (checked as it moves) the lists serve
        double vg[3] = {0.0, 0.0, 0.0};   // the drift: the first wide member's velocity, or the lowest member's
        float hlist = 0.0f;
        auto lists = [&](double hs, bool contacts) {
            const int A = kHugeY + ysel;
            const double* pos = huge_pos(H, A);
            const int ref = *(volatile int*)&hc->ref;
            for (int e = 0; e < 3; e++) vg[e] = nwide > 0 ? S.y[0][3 + e] : H.yv[((int64_t)ysel * 3 + e) * c + ref];
            hlist = fabsf((float)hs) * 1.0001f;
            if (warp < kHugeUnitWarps)
                for (int u = gw; u < nu; u += nw) {
                    const int i = L * u + lane;
                    const bool slot = lane < L && i < M, have = slot && H.alive[i] && !is_wide(i);
                    const float4 pb = slot ? huge_posf(H, A)[i] : make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f);
                    const float4 mo = slot ? huge_mot(H, A)[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    const float R = mo.w;
                    int n = -1;
                    if (!dense) {
                        huge_search<kHugeList>(H, hc, A, L, u, M, have, pb, mo, hlist, S.q[warp]);
                        __syncwarp();
                        n = H.listed[u];
                        for (int e = lane; contacts && e < n; e += 32) {
                            const int ent = H.list[(int64_t)u * kHugeListed + e], s = ent & 31, o = ent >> 5;
                            const float4 b = S.q[warp].mem[s], q = huge_posf(H, A)[o];
                            const float dx = q.x - b.x, dy = q.y - b.y, dz = q.z - b.z, lim = huge_mot(H, A)[L * u + s].w + huge_mot(H, A)[o].w + huge_slack(b);
                            if (dx * dx + dy * dy + dz * dz < lim * lim) huge_contact(H, hc, A, L * u + s, o);
                        }
                    }
                    if (contacts && n < 0)
                        for (unsigned nm = __ballot_sync(0xffffffffu, have); nm; nm &= nm - 1) {
                            const int s = __ffs(nm) - 1;
                            const float bx = __shfl_sync(0xffffffffu, pb.x, s), by = __shfl_sync(0xffffffffu, pb.y, s),
                                        bz = __shfl_sync(0xffffffffu, pb.z, s), bR = __shfl_sync(0xffffffffu, R, s);
                            const float sl = huge_slack(make_float4(bx, by, bz, 0.0f));
                            for (int o = lane; o < M; o += 32) {
                                const float4 q = huge_posf(H, A)[o];
                                const float dx = q.x - bx, dy = q.y - by, dz = q.z - bz, lim = bR + huge_mot(H, A)[o].w + sl;
                                if (o != L * u + s && __float_as_int(q.w) >= 0 && dx * dx + dy * dy + dz * dz < lim * lim)
                                    huge_contact(H, hc, A, L * u + s, o);
                            }
                        }
                    for (int w = 0; contacts && w < nwide; w++) {
                        if (!have || !S.alive[w]) continue;
                        const float fx = (float)S.y[w][0] - pb.x, fy = (float)S.y[w][1] - pb.y, fz = (float)S.y[w][2] - pb.z;
                        const float lim = R + __double2float_ru(S.R[w]) + huge_slack(pb);
                        if (!(fx * fx + fy * fy + fz * fz < lim * lim)) continue;
                        const double dx = S.y[w][0] - pos[i], dy = S.y[w][1] - pos[c + i], dz = S.y[w][2] - pos[2 * c + i];
                        const double rt = H.R[i] + S.R[w];
                        if (bs_can_touch(H.m[i], S.m[w]) && dx * dx + dy * dy + dz * dz <= rt * rt * (1.0 + 1e-9)) {
                            const int q = atomicAdd(&hc->ncand, 1), o = S.slot[w];
                            if (q < kHugeCand) hc->cand[q] = H.gid[i] < H.gid[o] ? make_int2(i, o) : make_int2(o, i);
                        }
                    }
                }
            if (contacts && blk == 0)   // the wide members with one another
                for (int q = tid; q < nwide * nwide; q += kHugeThreads) {
                    const int w = q / nwide, o = q % nwide;
                    if (o <= w || !S.alive[w] || !S.alive[o] || !bs_can_touch(S.m[w], S.m[o])) continue;
                    const double dx = S.y[o][0] - S.y[w][0], dy = S.y[o][1] - S.y[w][1], dz = S.y[o][2] - S.y[w][2];
                    const double rt = S.R[w] + S.R[o];
                    if (dx * dx + dy * dy + dz * dz <= rt * rt * (1.0 + 1e-9)) {
                        const int e = atomicAdd(&hc->ncand, 1), a = S.slot[w], b = S.slot[o];
                        if (e < kHugeCand) hc->cand[e] = H.gid[a] < H.gid[b] ? make_int2(a, b) : make_int2(b, a);
                    }
                }
            return sync();
        };
        double t = 0.0, Hs = dt;
        int nsub = 0;
        bool failed = false;
        if (!dense && !lists(dt, false)) {
            if (lead) set_status(d.ctl, kEbs, kHugeAbortDetail + 1 + g);
            return;
        }
        for (;;) {
            const double rem = dt - t;
            int last = 0;
            if (fabs(Hs) >= fabs(rem)) {
                Hs = rem;
                last = 1;
            }
            int kacc = -1;
            bool far = false;
            attempt++;
            for (int r = 0;; r++) {
                // (L, nu and nv are those of round r - 1 up to here)
                bool joined = nwide == 0 || r == 0 || r > 2 * kBsRows;   // the wide members' places of this round are there
                // the wide members' step of round r - 1, whose members' sums are in by now: the sums
                // by the block, the step by the last warp beside the others' first loads
                if (r > 0 && r <= 2 * kBsRows + 1 && nwide > 0) {
                    // a few threads a sum, its block sums in turn, then the threads in a tree
                    const int np = r == 1 ? kBsRows : kBsRows - max(0, r / 2 - 1), outs = np * nwide * 3;
                    int tpo = 1;
                    while (tpo < 8 && outs * tpo * 2 <= kHugeThreads) tpo *= 2;
                    for (int o0 = 0; o0 < outs * tpo; o0 += kHugeThreads) {   // (every lane runs every pass)
                        const int q = (o0 + tid) / tpo, part = (o0 + tid) % tpo;
                        const bool in = q < outs;
                        const int k = kBsRows - np + q / (nwide * 3), w = q / 3 % nwide, e = q % 3;
                        double s = 0.0;
                        if (in) {
                            const double* src = H.react + (((int64_t)((r - 1) & 1) * kBsRows + k) * nv * kHugeWide + w) * 3 + e;
#pragma unroll 4
                            for (int v = part; v < nv; v += tpo) s += __ldcg(src + (int64_t)v * kHugeWide * 3);
                        }
                        for (int o = 1; o < tpo; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                        if (in && part == 0) S.F[k][w][e] = S.base[k][w][e] + s;
                    }
                    __syncthreads();
                }
                if (r > 0 && r <= 2 * kBsRows + 1 && nwide > 0 && warp == kHugeUnitWarps) {
                    const int rp = r - 1, kp0 = rp == 0 ? 0 : max(0, (rp + 1) / 2 - 1), np = kBsRows - kp0;
                    __syncwarp();
                    for (int q = lane; q < np * nwide * 6; q += 32) {
                        const int k = kp0 + q / (nwide * 6), w = q / 6 % nwide, e = q % 6, n = 2 * (k + 1);
                        const double h = Hs / n;
                        const bool al = S.alive[w] != 0;
                        if (rp == 0) {
                            const double yq = S.y[w][e];
                            const double f = !al ? 0.0 : (e < 3 ? S.y[w][3 + e] : S.F[k][w][e - 3]);
                            S.z0[k][w][e] = yq;
                            S.row[k][w][e] = yq + h * f;   // (to z1 below: others still read the velocities)
                        } else {
                            const double f = !al ? 0.0 : (e < 3 ? S.z1[k][w][3 + e] : S.F[k][w][e - 3]);
                            const double z1 = S.z1[k][w][e], z0 = S.z0[k][w][e];
                            if (rp < n) {
                                S.z0[k][w][e] = z0 + 2.0 * h * f;   // the new z1 (swapped below)
                            } else {
                                double cv = 0.5 * (z1 + z0 + h * f), pv = 0.0;
                                for (int j = 1; j <= k; j++) {
                                    const double up = S.row[j - 1][w][e];
                                    S.row[j - 1][w][e] = cv;
                                    pv = cv;
                                    cv = cv + (cv - up) * kNeville[k][j];
                                }
                                S.row[k][w][e] = cv;
                                S.ty[w][e] = cv;
                                S.sq[w][e][0] = (cv - pv) * (cv - pv);
                                S.sq[w][e][1] = cv * cv;
                            }
                        }
                    }
                    __syncwarp();
                    for (int q = lane; q < np * nwide * 6; q += 32) {
                        const int k = kp0 + q / (nwide * 6), w = q / 6 % nwide, e = q % 6, n = 2 * (k + 1);
                        if (rp == 0) {
                            S.z1[k][w][e] = S.row[k][w][e];
                        } else if (rp < n) {
                            const double zn = S.z0[k][w][e];
                            S.z0[k][w][e] = S.z1[k][w][e];
                            S.z1[k][w][e] = zn;
                        }
                    }
                    if (rp >= 4 && rp % 2 == 0) {
                        // this row of a wide member: its error, and block 0 keeps the proposed state in its slot
                        for (int w = lane; w < nwide; w += 32) {
                            const double(*s)[2] = S.sq[w];
                            const double dx = s[0][0] + s[1][0] + s[2][0], nx = s[0][1] + s[1][1] + s[2][1];
                            const double dv = s[3][0] + s[4][0] + s[5][0], nvv = s[3][1] + s[4][1] + s[5][1];
                            if (S.alive[w] && !(dx <= tol2 * fmax(nx, 2.3e-308) && dv <= tol2 * fmax(nvv, 2.3e-308)))
                                S.fail[rp / 2 - 1] = attempt;
                            if (blk == 0) {
                                const int i = S.slot[w];
                                for (int e = 0; e < 3; e++) {
                                    huge_pos(H, kHugeY + (ysel ^ 1))[e * c + i] = S.ty[w][e];
                                    H.yv[((int64_t)(ysel ^ 1) * 3 + e) * c + i] = S.ty[w][3 + e];
                                }
                            }
                        }
                    }
                    __syncwarp();
                }
                if (r >= 6 && r % 2 == 0) {
                    // row kf >= 1, whose sequence ended in round r - 2: accepted unless a member's test failed
                    const int kf = r / 2 - 2;
                    if (*(volatile int*)&hc->err[kf] != attempt && (nwide == 0 || S.fail[kf] != attempt)) {   // (the same for every thread)
                        kacc = kf;
                        break;
                    }
                }
                if (r > 2 * kBsRows + 1) break;   // rejected
                const int k0 = r == 0 ? 0 : max(0, (r + 1) / 2 - 1);
                // (round 0's derivative is every sequence's; each takes it itself unless the pairs bound it)
                const int nact = dense && r == 0 ? 1 : kBsRows - k0;
                // the row of the sequence that ended last round, by units of their own: beside the
                // other sequences' steps, where it would else be the longest of them
                const int krow = r >= 3 && r % 2 == 1 ? (r - 3) / 2 : -1;
                // a member has moved past reach: the lists do not serve the rest of this attempt
                // (the mark of round r is in place before it: the same for every thread)
                if (!dense && *(volatile int*)&hc->moved[r & 1] == 32 * attempt + r) far = true;
                if (dense) units(min(32, (M * max(1, nact) + nw - 1) / nw));
                // a block's units: four warps' members of one sequence
                for (int unit = blk; unit == blk || unit < (nact + (krow >= 0)) * nv; unit += nblk) {
                    const bool act = unit < nact * nv;   // (a block without units only joins)
                    const int v = unit % nv, u = v * kHugeUnitWarps + warp;
                    if (!act && unit < (nact + (krow >= 0)) * nv && warp < kHugeUnitWarps && u < nu) {
                        const int i = L * u + lane;
                        const bool slot = lane < L && i < M, own = slot && !is_wide(i);
                        huge_row(H, hc, krow, ysel, u, i, slot, own, own && H.alive[i], attempt, tol2, vg, dense);
                    }
                    const int k = k0 + unit / nv;
                    const int kz = dense && r == 0 ? kBsRows - 1 : k;   // the derivative serves k .. kz
                    const bool mine = act && warp < kHugeUnitWarps && u < nu;
                    const int i = L * u + lane;
                    const bool slot = mine && lane < L && i < M;
                    const bool own = slot && !is_wide(i);        // a state this lane steps
                    const bool have = own && H.alive[i];
                    double P[3] = {1.0, 1.0, 1.0}, V[3] = {0.0, 0.0, 0.0}, Z[6], rc = 0.0, pinv = 0.0, mb = 0.0;
                    double acc[3] = {0.0, 0.0, 0.0};
                    float4 pb = make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f), mo = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (mine) {
                        const int A = r == 0 ? kHugeY + ysel : (r & 1) * kBsRows + k;
                        const double* pos = huge_pos(H, A);
                        const double* vel = r == 0 ? H.yv + (int64_t)ysel * 3 * c : H.zv + (int64_t)k * 3 * c;
                        const int listed = dense ? -1 : H.listed[u];   // (dense: more units than the lists have room for)
                        if (own) mo = huge_mot(H, kHugeY + ysel)[i];
                        if (own) {
                            pb = huge_posf(H, A)[i];
#pragma unroll
                            for (int e = 0; e < 3; e++) {
                                P[e] = pos[e * c + i];
                                V[e] = vel[e * c + i];
                            }
                            rc = H.rc[i];
                            pinv = H.pinv[i];
                            mb = H.m[i];
                        }
#pragma unroll
                        for (int e = 0; e < 6; e++) Z[e] = own && r > 0 ? H.z0[((int64_t)k * 6 + e) * c + i] : 0.0;
                        if (have) {
                            const double ri = rsqrt(fma(P[2], P[2], fma(P[1], P[1], __dmul_rn(P[0], P[0]))));
                            const double sk = -GM0 * (ri * ri * ri);
#pragma unroll
                            for (int e = 0; e < 3; e++) acc[e] = sk * P[e];
                        }
                        if (dense || far || listed < 0) huge_dense(d, H, A, L, u, M, have, P[0], P[1], P[2], pb, rc, pinv, acc);
                        else if (listed > 0) huge_listed(d, H, A, u, listed, P[0], P[1], P[2], pb, rc, pinv, S.q[warp], acc);
                    }
                    if (!joined) {
                        __syncthreads();
                        joined = true;
                    }
                    if (mine) {
                        // the wide members, both sides
                        for (int w = 0; w < nwide; w++) {
                            const double* Q = r == 0 ? S.y[w] : S.z1[k][w];
                            double s = 0.0, dx = 0.0, dy = 0.0, dz = 0.0;
                            if (have && S.alive[w]) {
                                dx = Q[0] - P[0];
                                dy = Q[1] - P[1];
                                dz = Q[2] - P[2];
                                s = huge_factor(dx, dy, dz, rc, pinv, S.rc[w], S.pinv[w], S.gm[w], form);
                            }
                            double sum = 0.0;
                            if (__any_sync(0xffffffffu, s != 0.0)) {
                                const double sb = -(s * S.igm[w]) * (G * mb);
                                acc[0] = __dadd_rn(acc[0], __dmul_rn(s, dx));
                                acc[1] = __dadd_rn(acc[1], __dmul_rn(s, dy));
                                acc[2] = __dadd_rn(acc[2], __dmul_rn(s, dz));
                                sum = warp_sum3(sb * dx, sb * dy, sb * dz);
                            }
                            if ((lane & 7) == 0 && lane < 24) S.red[warp][w][lane >> 3] = sum;
                        }
                        const double f[6] = {have ? V[0] : 0.0, have ? V[1] : 0.0, have ? V[2] : 0.0, acc[0], acc[1], acc[2]};
                        // the step, or at the sequence's end its row
                        for (int ks = k; ks <= kz; ks++) {
                            const int n = 2 * (ks + 1);
                            const double h = Hs / n;
                            double* z0p = H.z0 + (int64_t)ks * 6 * c;
                            if (r == n) {
                                // the sequence's end: its last value, for its row
#pragma unroll
                                for (int e = 0; e < 6; e++) {
                                    const double z1 = e < 3 ? P[e] : V[e - 3];
                                    if (own) H.sk[e * c + i] = 0.5 * (z1 + Z[e] + h * f[e]);
                                }
                                float a2 = 0.0f;
#pragma unroll
                                for (int e = 0; e < 3; e++) {
                                    const float qa = trunc_f(acc[e]);
                                    a2 = fmaf(qa, qa, a2);
                                }
                                if (own) H.ska[i] = sqrtf(a2);
                                continue;
                            }
                            const int B = ((r + 1) & 1) * kBsRows + ks;
                            double Y[6];
#pragma unroll
                            for (int e = 0; e < 6; e++) {
                                const double z1 = e < 3 ? P[e] : V[e - 3];
                                Y[e] = r == 0 ? z1 + h * f[e] : Z[e] + 2.0 * h * f[e];
                                if (own) z0p[e * c + i] = z1;
                            }
                            if (have && !dense) {
                                // the new point lies within reach of the start carried along with the group
                                const double* y0 = huge_pos(H, kHugeY + ysel);
                                const double tau = h * (r + 1);
                                float m2 = 0.0f;
#pragma unroll
                                for (int e = 0; e < 3; e++) {
                                    const float q = trunc_f(Y[e] - fma(vg[e], tau, y0[e * c + i]));
                                    m2 = fmaf(q, q, m2);
                                }
                                const float reach = huge_reach(mo, hlist);
                                if (!(m2 <= reach * reach)) *(volatile int*)&hc->moved[(r + 1) & 1] = 32 * attempt + r + 1;
                            }
                            float4 pf = make_float4(kHugeFar, kHugeFar, kHugeFar, 0.0f);
                            if (have) pf = make_float4(trunc_f(Y[0]), trunc_f(Y[1]), trunc_f(Y[2]), pb.w);
                            if (own) {
                                double* zv = H.zv + (int64_t)ks * 3 * c;
                                double* o = huge_pos(H, B);
#pragma unroll
                                for (int e = 0; e < 3; e++) {
                                    zv[e * c + i] = Y[3 + e];
                                    o[e * c + i] = Y[e];
                                }
                            }
                            if (slot) huge_posf(H, B)[i] = pf;
                        }
                    } else if (act && warp < kHugeUnitWarps) {
                        for (int q = lane; q < nwide * 3; q += 32) S.red[warp][q / 3][q % 3] = 0.0;
                    }
                    if (unit == blk && warp == kHugeUnitWarps) {
                        // the wide members' accelerations by the star and one another at this round's points
                        for (int q = lane; q < (kBsRows - k0) * nwide; q += 32) {
                            const int k = k0 + q / nwide, w = q % nwide;
                            if (!S.alive[w]) continue;
                            const double* P = r == 0 ? S.y[w] : S.z1[k][w];
                            const double ri = rsqrt(fma(P[2], P[2], fma(P[1], P[1], __dmul_rn(P[0], P[0]))));
                            const double sk = -GM0 * (ri * ri * ri);
                            double ax = sk * P[0], ay = sk * P[1], az = sk * P[2];
                            for (int o = 0; o < nwide; o++) {
                                if (o == w || !S.alive[o] || le_zero(S.m[o])) continue;
                                const double* Q = r == 0 ? S.y[o] : S.z1[k][o];
                                const double dx = Q[0] - P[0], dy = Q[1] - P[1], dz = Q[2] - P[2];
                                const double s = huge_factor(dx, dy, dz, S.rc[w], S.pinv[w], S.rc[o], S.pinv[o], G * S.m[o], form);
                                ax = __dadd_rn(ax, __dmul_rn(s, dx));
                                ay = __dadd_rn(ay, __dmul_rn(s, dy));
                                az = __dadd_rn(az, __dmul_rn(s, dz));
                            }
                            S.base[k][w][0] = ax;
                            S.base[k][w][1] = ay;
                            S.base[k][w][2] = az;
                        }
                    }
                    if (act && nwide > 0) {
                        __syncthreads();
                        for (int q = tid; q < nwide * 3; q += kHugeThreads) {
                            double s = 0.0;
                            for (int o = 0; o < kHugeUnitWarps; o++) s += S.red[o][q / 3][q % 3];
                            for (int ks = k; ks <= kz; ks++)
                                H.react[((((int64_t)(r & 1) * kBsRows + ks) * nv + v) * kHugeWide + q / 3) * 3 + q % 3] = s;
                        }
                        __syncthreads();
                    }
                }
                if (!(ok = sync())) break;
            }
            if (!ok) break;
            nsub++;
            if (kacc >= 0) {
                ysel ^= 1;
                for (int q = tid; q < nwide * 6; q += kHugeThreads) S.y[q / 6][q % 6] = S.ty[q / 6][q % 6];
                __syncthreads();
                t = last ? dt : t + Hs;
                if (kacc <= 2) Hs *= 2.0;
                else if (kacc >= 6) Hs *= 0.5;
                // contacts: candidates in parallel, with the next substep's lists, then the sequential sweep by one thread
                double* pos = huge_pos(H, kHugeY + ysel);
                if (!(ok = lists(last ? 0.0 : fmin(fabs(Hs), fabs(dt - t)), true))) break;
                const int nc = *(volatile int*)&hc->ncand;
                if (nc > 0) {
                    if (!(ok = sync())) break;   // everyone has read the count
                    if (lead) {
                        huge_sweep(d, H, hc, M, pos, H.yv + (int64_t)ysel * 3 * c, M0g);
                        hc->ncand = 0;
                    }
                    if (!(ok = sync())) break;
                    if (!(ok = refresh())) break;   // places, masses and flags as the mergers left them
                    if (!last && !dense && !(ok = lists(fmin(fabs(Hs), fabs(dt - t)), false))) break;
                }
                if (last) break;
            } else {
                // (with a barrier: round 0 writes sums that the last round's end has read)
                Hs *= 0.5;
                if (!(ok = dense ? sync() : lists(Hs, false))) break;
            }
            if (nsub >= p.bs_max_substeps) {
                failed = true;
                break;
            }
        }
        if (!ok) {
            if (lead) set_status(d.ctl, kEbs, kHugeAbortDetail + 1 + g);
            return;
        }
        // (the last sync is behind every write of the current start array but block 0's of
        // the wide members, which came before it too: rows end before their round's check)
        for (int64_t i = gt; i < M; i += nt) {
            double* o = d.bsout + (int64_t)kBsOut * (m0 + H.perm[i]);
            for (int e = 0; e < 3; e++) {
                o[e] = huge_pos(H, kHugeY + ysel)[e * c + i];
                o[3 + e] = H.yv[((int64_t)ysel * 3 + e) * c + i];
            }
            o[6] = H.m[i];
            o[7] = H.R[i];
            o[8] = (double)H.alive[i];
        }
        if (lead) {
            d.glost[g] = hc->El;
            if (hc->nmerge) atomicAdd(&d.ctl->nmerge, hc->nmerge);
            atomicAdd(&d.ctl->nsub, (unsigned long long)nsub);
            if (failed) set_status(d.ctl, kEbs, g);
        }
        if (!sync()) return;   // the buffers are free for the next group
    }
}

cudaError_t launch_bs_huge(const Dev& d, int nsm, cudaStream_t s) {
    // all blocks must be resident at once for the barriers: a cooperative launch
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(kHugeTeams * nsm));
    cfg.blockDim = dim3(kHugeThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_bs_huge, d, nsm);
    prof_mark("bs: groups of more than 64");
    return e;
}

}  // namespace opal
