// lbgb_moment.cu -- the time step at tau = 1 on the moments of the sites (FP32
// arithmetic).
//
// At omega = 1 the collided populations of a site are the equilibrium of its
// densities and its shifted velocity (Eq. 16: f*_i = f^eq_i(rho^k, u + F^k/rho^k)),
// and with tau_A = tau_B the mixture velocity needs the total momentum only
// (Eq. 14).  A step that is followed by another one in the same lb_step call
// therefore needs no populations: rho^k(t+1) and j(t+1) = sum_k j^k(t+1) are
// sums over the equilibria of the 18 neighbours and of the site itself
// (Eqs. 3, 6, 7),
//   rho^k(x, t+1) = sum_i f*^k_i(x - c_i, t),  j(x, t+1) = sum_k sum_i c_i f*^k_i(x - c_i, t),
// with the bounce-back values of the links that come from particle nodes
// (Eqs. 17-19) or from beyond a z face (Eqs. 9, 10).  One kernel per step
// reads rho^k, j and the link classes and writes rho^k and j: 44 bytes a site
// instead of the 349 of a density pass and a population push.  The first step
// of a call starts from the populations (density pass) and the last one pushes
// them, so that the state a call leaves is the populations.
//
// A lane holds two sites of a column of the block, side by side in packed
// values (f32x2 instructions advance both); a warp holds two rows of 32 sites
// and marches along z; a block holds MROWS rows, and one more warp holds the
// row on each side of them.  Every lane forms the 19 links of its sites in
// registers (opposite links share their even part); the links that cross x
// travel by warp shuffles, those that cross y between warps through shared
// memory, and a plane's sums reach the planes below, at and above it in
// registers.  With the shifted velocity as h = 3/2 (u + F/rho) a link is
//   f*_i = w_i (P + q (c.h) + q),  q = 2 rho c.h,  P = rho (1 - 2/3 h.h),
// in units of 1/36 (weights 12, 2, 1); the sums are scaled at the end.
//
// What bounds it: instruction issue (60 % active) and the shared-memory and
// shuffle pipe (64 %), some 490 warp instructions per two rows and plane; its 44
// bytes a site (DRAM sees 46) run at 0.33 of the copy bandwidth.  The two sites of a lane
// share loop, address and exchange work, and pack without regrouping (the
// components of one site would need their sum A + B unpacked for j): one
// site a lane took 790 instructions per 32 sites and plane.  Everything a
// plane needs is copied to shared memory (cp.async) one to two planes ahead:
// read to registers before the barrier instead, a third of the issue slots
// waited for it (392 -> 327 us).  256^3 periodic, two components, one step:
// density pass and push 882 us, here 330; one component 410 -> 157; with
// particles 512 x 512 x 256 at a volume fraction of 0.15 (k_moments and
// k_bounce_links) 4.12 -> 1.77 ms.
//
// The links are summed as deviations from those of a fluid of a reference
// density at rest (P less that density).  Where the densities are nearly uniform
// the reference is their mean initial value: the sums of rho and j then stay
// small and keep the precision that sums of the links themselves lose (48 x 40 x
// 36, deviations of 1 %, 100 steps: the rms error of rho 1.0e-7 against 1.3e-7
// by sums of the links and 1.6e-6 by sums of populations, of u 5e-9, 8e-9, 1.3e-8).
// A density far below the reference would be left with the rounding of the
// reference (0: with a residue of either sign).  So the references of a step are
// 0 once the step before, or the density pass, has met a density below half of
// them (L.spread; a site keeps its rest population, so that a density falls by
// a factor of about 3 at most meanwhile): the sums of the links are each rounded
// by their own size, and a component that is absent adds up to 0.  In slabs and
// droplets of 0, 1e-4, 1e-2 and 0.05 against 0.7 to 1.3 the rms errors are then
// those of sums of populations divided by 1.25 after 2 steps, 2.5 after 20, 7 after
// 100, 30 after 1000 (rho, each relative to itself) and 1.25, 2.2, 2.0, 1.4 (u;
// geometric means over 9 such states).
#include "lbgb_internal.cuh"

namespace lbgb {

// ----------------------------------------- two FP32 values side by side
struct alignas(8) F2 {
    union {
        unsigned long long v;
        struct {
            float x, y;
        };
    };
};
__device__ __forceinline__ F2 f2(float x, float y) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ F2 f2(float x) { return f2(x, x); }
__device__ __forceinline__ float lo(F2 a) {
    [[maybe_unused]] float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return x;
}
__device__ __forceinline__ float hi(F2 a) {
    [[maybe_unused]] float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return y;
}
__device__ __forceinline__ F2 operator+(F2 x, F2 y) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 x, F2 y) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 x, F2 y) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 x, F2 y, F2 z) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(x.v), "l"(y.v), "l"(z.v));
    return r;
}
__device__ __forceinline__ F2 shfl2(F2 a, int lane) {
    return f2(__shfl_sync(0xffffffffu, lo(a), lane), __shfl_sync(0xffffffffu, hi(a), lane));
}
// 1/x of normal values: the approximate reciprocal and one Newton-Raphson step,
// which rounds correctly (the bits of __frcp_rn at all 2^23 mantissas of 1/2^30,
// 1/2^10, 1/2 to 2, 2^10 and 2^100)
__device__ __forceinline__ F2 rcp_newton(F2 x) {
    float a, b;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(lo(x)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(hi(x)));
    const F2 r = f2(a, b);
    return fma2(fma2(f2(-1.f) * x, r, f2(1.f)), r, r);
}

// ------------------------------------------------------------ the kernel
// The two outer lanes on each side of a warp serve its neighbours only (the
// sums S = sum_i w_i psi(x + c_i) c_i of a lane need the psi of the next one,
// its sums the links of the next one), so a row advances 28 sites, or 32 on
// a lattice of nx = 32, whose rows close on themselves.
constexpr int MROWS = 8, MW = MROWS / 2;  // rows of a block, and their warps
constexpr int MNT = 32 * (MW + 1);  // the warps of the rows and one for the rows beside them

// The boundary sites of a step (fluid sites next to particle nodes), listed by
// k_moments for k_bounce_links: each block lists its own in a segment of its
// sites' number, by word: the site, its link classes, h (x A, x B, y A, ..) and rho.
constexpr int MREC = 10;
struct LinkList {
    unsigned* rec;  // [MREC][N]
    int* count;     // per block; with LIST_PLAIN if the step sums without a reference
};
constexpr int LIST_PLAIN = 1 << 30;
// first entry of the segment of the block at (x0, y0, z0) with H rows and nz planes
__device__ __forceinline__ long long segment_of(const Lattice& L, int x0, int y0, int H, int z0, int nz) {
    return (long long)L.nx * L.ny * z0 + (long long)nz * ((long long)y0 * L.nx + (long long)H * x0);
}

template <int NK, bool PART>
struct alignas(16) MomentShared {
    // the links that cross y, by parity of the plane, towards y + 1 / y - 1,
    // for the two rows of the warp that takes them: those within the plane,
    // those to the plane above and below, the momentum of the first along x
    static constexpr int NV = 3 * NK + 1;
    F2 cross[2][2][NV][MW][32];
    // psi of the columns of the block, the rows and two on each side of them,
    // of the plane in use, the next one and the one being copied
    F2 psi[NK == 2 ? 3 : 1][NK == 2 ? MROWS + 4 : 1][NK == 2 ? 32 : 1];
    // likewise j (x, y, z) and, for one component, rho, of the rows and one on
    // each side, of the plane in use and the next two, and the link classes
    float own[3][NK == 2 ? 3 : 4][MROWS + 2][32];
    uint32_t nb[PART ? 3 : 1][PART ? MROWS + 2 : 1][PART ? 32 : 1];
    float ref[NK];  // reference densities of the step
    int count;      // boundary sites listed so far
};

// the links along +c and -c of weight 1/36 (r2 = 2 rho) or 1/18 (r2 = 4 rho,
// P doubled), ch = c.h
__device__ __forceinline__ void link_pair(F2 ch, F2 r2, F2 P, F2& fp, F2& fm) {
    const F2 q = r2 * ch, e = fma2(q, ch, P);
    fp = e + q;
    fm = e - q;
}

// the links m of the lane and those that join them along x (from the lane on
// the left: a, on the right: b), and the momentum along x these bring
template <int NK>
__device__ __forceinline__ void join_x(const F2 (&m)[NK], const F2 (&a)[NK], const F2 (&b)[NK], int lane, F2 (&g)[NK],
                                       F2& jx) {
    F2 l[NK], r[NK];
#pragma unroll
    for (int k = 0; k < NK; k++) {
        l[k] = shfl2(a[k], (lane - 1) & 31);
        r[k] = shfl2(b[k], (lane + 1) & 31);
        g[k] = m[k] + (l[k] + r[k]);
    }
    jx = NK == 2 ? (l[0] + l[NK - 1]) - (r[0] + r[NK - 1]) : l[0] - r[0];
}

template <int NK>
__device__ __forceinline__ F2 total(const F2 (&a)[NK]) {
    return NK == 2 ? a[0] + a[NK - 1] : a[0];
}

// sums of S in progress along the march of one row (the two components side
// by side): g the links within a plane and from the plane below, b and c those
// that leave a plane, p the psi of the plane
struct PsiMarch {
    F2 gx, gy, bx, by, c0, c1, p;
};

// psi of the next plane around the site, p[y][x]: S of the plane before it,
// component by component
__device__ __forceinline__ void psi_march(PsiMarch& m, const F2 (&p)[3][3], float (&SA)[3], float (&SB)[3]) {
    const F2 wd = f2(1.f / 36.f), wa = f2(1.f / 18.f);
    const F2 dx = p[1][2] - p[1][0], dy = p[2][1] - p[0][1];
    const F2 d1 = p[2][2] - p[0][0], d2 = p[0][2] - p[2][0];  // along (1, 1) and (1, -1)
    const F2 bx = wd * dx, by = wd * dy;
    const F2 c = fma2(wa, p[1][1], wd * ((p[1][2] + p[1][0]) + (p[2][1] + p[0][1])));
    SA[0] = lo(m.gx) + lo(bx);
    SB[0] = hi(m.gx) + hi(bx);
    SA[1] = lo(m.gy) + lo(by);
    SB[1] = hi(m.gy) + hi(by);
    SA[2] = lo(c) - lo(m.c0);
    SB[2] = hi(c) - hi(m.c0);
    m.gx = fma2(wa, dx, wd * (d1 + d2)) + m.bx;
    m.gy = fma2(wa, dy, wd * (d1 - d2)) + m.by;
    m.bx = bx;
    m.by = by;
    m.c0 = m.c1;
    m.c1 = c;
    m.p = p[1][1];
}

__device__ __forceinline__ bool beyond(const Lattice& L, int q) { return (q < 0 || q >= L.nz) && !L.per[2]; }
__device__ __forceinline__ long long plane_at(const Lattice& L, int q) {
    return (long long)L.nx * L.ny * (q < 0 ? q + L.nz : (q >= L.nz ? q - L.nz : q));
}

__device__ __forceinline__ void block_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// The copies of the rows of a plane into shared memory, 16 bytes of psi (two
// sites) and 8 bytes of the other arrays (two sites) each, by the warps of
// the rows and the ring warp (a row starts at an even x, and nx is even: no
// copy crosses an edge).  The psi of plane q + 3 and the others of plane q + 2
// are issued while psi of plane q + 1 and the others of plane q are in use, so
// that a lane holds none of them while they travel.
template <int NK, bool PART>
struct PlaneCopy {
    static constexpr int NT = 32 * (MW + 1), NC = ((MROWS + 4) * 16 + NT - 1) / NT;
    static_assert((MROWS + 2) * 16 == NT, "one copy per thread and array");
    int pxy[NC], xy;  // the sites in a plane (pxy -1: none)

    __device__ __forceinline__ void place(const Lattice& L, int x, int y, int H) {
        auto site = [&](int t, int dy) { return (x + 2 * (t % 16) + L.nx) % L.nx + L.nx * ((y + t / 16 - dy + 2 * L.ny) % L.ny); };
#pragma unroll
        for (int c = 0; c < NC; c++) {
            const int t = threadIdx.x + c * NT;
            pxy[c] = t / 16 < H + 4 ? site(t, 2) : -1;
        }
        xy = site(threadIdx.x, 1);
    }
    __device__ __forceinline__ void psi(const Lattice& L, MomentShared<NK, PART>& sh, int q, int slot) {
        if constexpr (NK == 2) {
            const F2* base = (const F2*)L.psi + plane_at(L, q);
            if (beyond(L, q)) base = (const F2*)L.psi_wall + (q < 0 ? 0 : (long long)L.nx * L.ny);
#pragma unroll
            for (int c = 0; c < NC; c++)
                if (pxy[c] >= 0) cp_async_16(&sh.psi[slot][0][0] + 2 * (threadIdx.x + c * NT), base + pxy[c]);
        }
    }
    __device__ __forceinline__ void others(const Lattice& L, MomentShared<NK, PART>& sh, int q, int slot) {
        const long long s = plane_at(L, q) + xy;
        const float* mom = (const float*)L.mom + s;
#pragma unroll
        for (int d = 0; d < 3; d++) cp_async_8(&sh.own[slot][d][0][0] + 2 * threadIdx.x, mom), mom += L.pstride;
        if (NK == 1) cp_async_8(&sh.own[slot][NK == 1 ? 3 : 0][0][0] + 2 * threadIdx.x, (const float*)L.psi + s);
        if (PART) cp_async_8(&sh.nb[slot][0][0] + 2 * threadIdx.x, L.nb + s);
    }
};
// all copies but those of the last group are there
__device__ __forceinline__ void wait_but_last() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// the three slots of the staged planes: in use, next, being copied (psi runs
// one plane ahead of the others)
struct Slots {
    int a, b, c;
    __device__ __forceinline__ void next() {
        const int t = a;
        a = b;
        b = c;
        c = t;
    }
};

// What a lane keeps of its two sites while it marches.
template <int NK, bool PART>
struct MomentLane {
    int lane, row[2];  // rows of the block (1: the first)
    uint32_t nbn[2];   // link classes of the plane
    // of the densities met: the signs of their distances above L.rlow (any site),
    // and the largest as bits, which a negative one or no number exceeds (fluid)
    unsigned below, top;
    PsiMarch march[2];

    __device__ __forceinline__ void place(int l, int ra, int rb) {
        lane = l;
        row[0] = ra + 1;
        row[1] = rb + 1;
        const F2 zero = f2(0.f);
#pragma unroll
        for (int r = 0; r < 2; r++) march[r] = {zero, zero, zero, zero, zero, zero, zero};
        nbn[0] = nbn[1] = 0;
        below = top = 0;
    }
    // with the psi plane of a slot: S of the plane before it, by row and component
    __device__ __forceinline__ void advance(const MomentShared<NK, PART>& sh, int slot, float (&S)[2][2][3]) {
#pragma unroll
        for (int r = 0; r < 2; r++) {
            F2 p[3][3];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const F2* q = sh.psi[slot][row[r] + d];
                p[d][0] = q[(lane - 1) & 31];
                p[d][1] = q[lane];
                p[d][2] = q[(lane + 1) & 31];
            }
            psi_march(march[r], p, S[r][0], S[r][1]);
        }
    }
    // The densities of a step are judged here, where k_moments reads them (those
    // of the last step of a call by the kernel that pushes the populations): all
    // links that came back from particles and faces are in them by now.
    // What is below L.rlow is looked for by each warp among its sites, or, with
    // particles, by the ring warp in the staged psi of plane z + 1, where the march
    // of the others has no register to spare.  (256^3 without and with 2407
    // particles: k_moments 327 -> 326 and 372 -> 377 us a step; with a branch
    // for the unusual densities, or their smallest ones kept, 331 to 345 and 392 to 402.)
    __device__ __forceinline__ void meet(F2 d) { below |= __float_as_uint(lo(d)) | __float_as_uint(hi(d)); }
    __device__ __forceinline__ void meet_rows(const Lattice& L, const MomentShared<NK, PART>& sh, int slot, int H) {
        if constexpr (NK == 2)
            for (int y = 0; y < H; y++) meet(sh.psi[slot][y + 2][lane] - f2(L.rlow[0], L.rlow[1]));
    }
    __device__ __forceinline__ void judge(const F2 (&r)[NK]) {
        const unsigned none = NK == 1 ? 1u : 0u;  // one component: 0 is no density
#pragma unroll
        for (int k = 0; k < NK; k++)
            top = max(top, max(__float_as_uint(lo(r[k])) - none, __float_as_uint(hi(r[k])) - none));
    }
    // what the lanes `own` have met
    __device__ __forceinline__ void report(const Lattice& L, bool own) const {
        if (__any_sync(0xffffffffu, own && (below >> 31)) && lane == 0) note_spread(L, L.turn == 2 ? 0 : L.turn + 1);
        if (__any_sync(0xffffffffu, own && top >= __float_as_uint(1e30f)) && lane == 0) atomicOr(L.flags, FLAG_NONFINITE);
    }
    // h, rho and P of the sites of plane z, from the psi of plane z + 1 and the
    // other arrays of plane z in a slot; off: bits of the sites without fluid
    __device__ __forceinline__ unsigned collide(const Lattice& L, const MomentShared<NK, PART>& sh, int slot, int z,
                                                F2 (&h)[NK][3], F2 (&r)[NK], F2 (&P)[NK]) {
        const bool out = beyond(L, z);
        unsigned off = out ? 3u : 0u;
        if (PART) {
            nbn[0] = sh.nb[slot][row[0]][lane];
            nbn[1] = sh.nb[slot][row[1]][lane];
        }
        auto both = [&](int a) { return f2(sh.own[slot][a][row[0]][lane], sh.own[slot][a][row[1]][lane]); };
        if (PART) off |= (nbn[0] & NB_SOLID ? 1u : 0u) | (nbn[1] & NB_SOLID ? 2u : 0u);
        F2 rt;
        if constexpr (NK == 2) {
            r[0] = f2(lo(march[0].p), lo(march[1].p));
            r[1] = f2(hi(march[0].p), hi(march[1].p));
            if (!PART) meet(r[0] - f2(L.rlow[0])), meet(r[1] - f2(L.rlow[1]));
            if (PART) {
                r[0] = f2(off & 1u ? 0.f : lo(r[0]), off & 2u ? 0.f : hi(r[0]));
                r[1] = f2(off & 1u ? 0.f : lo(r[1]), off & 2u ? 0.f : hi(r[1]));
            }
            rt = r[0] + r[1];
        } else {
            r[0] = rt = both(NK == 1 ? 3 : 0);
            meet(r[0] - f2(L.rlow[0]));
        }
        if (!out) judge(r);
        if (PART) rt = f2(off & 1u ? 1.f : lo(rt), off & 2u ? 1.f : hi(rt));
        if (out) {
#pragma unroll
            for (int k = 0; k < NK; k++) r[k] = f2(0.f);
            rt = f2(1.f);
        }
        const F2 ir = f2(1.5f) * rcp_newton(rt);
        if constexpr (NK == 2) {
            float S[2][2][3];
            advance(sh, slot, S);
            const F2 mG = f2(-1.5f * L.PF.G);
#pragma unroll
            for (int d = 0; d < 3; d++) {
                // F^k / rho^k = g - G S of the other component (at a density
                // of 0 the velocity of a component does not matter)
                const F2 u = fma2(both(d), ir, f2(1.5f * L.PF.body_force[d]));
                h[0][d] = fma2(mG, f2(S[0][1][d], S[1][1][d]), u);
                h[1][d] = fma2(mG, f2(S[0][0][d], S[1][0][d]), u);
            }
        } else {
#pragma unroll
            for (int d = 0; d < 3; d++) h[0][d] = fma2(both(d), ir, f2(1.5f * L.PF.body_force[d]));
        }
#pragma unroll
        for (int k = 0; k < NK; k++) {
            const F2 hh = fma2(h[k][2], h[k][2], fma2(h[k][1], h[k][1], h[k][0] * h[k][0]));
            P[k] = fma2(r[k] * hh, f2(-2.f / 3.f), r[k] - f2(sh.ref[k]));
        }
        return off;
    }
};

// sums of a plane in progress: rho and j; j along z in two parts, of the links
// within the column of x and of those that cross y: each part meets the links
// from above that cancel it in a fluid at rest (their sum, rounded first,
// would leave a momentum along z of the same sign in all of a uniform phase)
template <int NK>
struct MomentSum {
    F2 r[NK], j[4];
};

// the links that cross y of the two sites: towards y + 1 within the plane
// (with the links that join them along x, jyp their momentum along x) and to
// the planes above and below; towards y - 1 likewise
template <int NK>
struct CrossLinks {
    F2 yp[NK], ym[NK], jyp, jym, pa[NK], pb[NK], ma[NK], mb[NK];
};

template <int NK>
__device__ __forceinline__ void cross_links(const F2 (&h)[NK][3], const F2 (&r2)[NK], const F2 (&r4)[NK],
                                            const F2 (&P)[NK], const F2 (&P2)[NK], int lane, CrossLinks<NK>& c) {
    F2 a[NK], ai[NK], d[NK], di[NK], m[NK], mi[NK];
#pragma unroll
    for (int k = 0; k < NK; k++) {
        link_pair(h[k][1], r4[k], P2[k], m[k], mi[k]);                 // (0, +-1, 0)
        link_pair(h[k][0] + h[k][1], r2[k], P[k], a[k], ai[k]);       // +-(1, 1, 0)
        link_pair(h[k][0] - h[k][1], r2[k], P[k], d[k], di[k]);       // +-(1, -1, 0)
    }
    join_x<NK>(m, a, di, lane, c.yp, c.jyp);
    join_x<NK>(mi, d, ai, lane, c.ym, c.jym);
#pragma unroll
    for (int k = 0; k < NK; k++) {
        link_pair(h[k][1] + h[k][2], r2[k], P[k], c.pa[k], c.mb[k]);  // +-(0, 1, 1)
        link_pair(h[k][1] - h[k][2], r2[k], P[k], c.pb[k], c.ma[k]);  // +-(0, 1, -1)
    }
}

// rho^k(t+1), j(t+1) into psi_o [N][NK], mom_o [3][pstride] from L.psi, L.mom
// (one component: rho [N] and j) of time t.  PART: the lattice has particles.
// TW sites a row and warp, from lane (32 - TW) / 2 on.  Every warp of the
// block passes one barrier per plane z0 - 1 .. z1, in the loop of its role.
template <int NK, bool PART>
__global__ void __launch_bounds__(MNT, NK == 1 ? 4 : 3)
    k_moments(const __grid_constant__ Lattice L, float* __restrict__ psi_o, float* __restrict__ mom_o, LinkList list,
              int zc, int TW) {
    chain_begin();
    typedef MomentShared<NK, PART> SH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SH& sh = *reinterpret_cast<SH*>(smem_raw);
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int edge = (32 - TW) / 2, x0 = blockIdx.x * TW, y0 = blockIdx.y * MROWS, H = min(MROWS, L.ny - y0);
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, L.nz);
    // warp w of nw holds rows w and w + nw of the block (of an odd H the last
    // one the row beside the block as its second), the ring warp the rows H
    // and -1
    const int nw = (H + 1) / 2;
    if (PART && threadIdx.x == 0) sh.count = 0;
    // psi of the planes z0 - 2 .. z0 and the other arrays of plane z0 - 1; the
    // slots go round with the planes
    PlaneCopy<NK, PART> copy;
    copy.place(L, x0 - edge, y0, H);
    for (int q = 0; q < 3; q++) copy.psi(L, sh, z0 - 2 + q, q);
    copy.others(L, sh, z0 - 1, 2);
    cp_async_commit();
    // (while the copies are under way)
    if (threadIdx.x < NK) sh.ref[threadIdx.x] = L.spread[L.turn] ? 0.f : L.rref[threadIdx.x];
    if (threadIdx.x == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) L.spread[L.turn == 0 ? 2 : L.turn - 1] = 0;
    cp_async_wait_all();
    block_barrier();
    if (warp == MW) {
        MomentLane<NK, PART> me;
        me.place(lane, H, -1);
        if constexpr (NK == 2) {
            float S[2][2][3];
            me.advance(sh, 0, S);
            me.advance(sh, 1, S);
        }
        block_barrier();
        copy.psi(L, sh, z0 + 1, 0);
        copy.others(L, sh, z0, 0);
        cp_async_commit();
        Slots slot = {2, 0, 1};
        for (int z = z0 - 1; z <= z1; z++, slot.next()) {
            F2 h[NK][3], r[NK], P[NK], r2[NK], r4[NK], P2[NK];
            copy.psi(L, sh, min(z + 3, z1 + 1), slot.c);
            copy.others(L, sh, min(z + 2, z1), slot.c);
            cp_async_commit();
            if (PART && !beyond(L, z + 1)) me.meet_rows(L, sh, slot.a, H);
            me.collide(L, sh, slot.a, z, h, r, P);
#pragma unroll
            for (int k = 0; k < NK; k++) {
                r2[k] = r[k] + r[k];
                r4[k] = r2[k] + r2[k];
                P2[k] = P[k] + P[k];
            }
            CrossLinks<NK> c;
            cross_links<NK>(h, r2, r4, P, P2, lane, c);
            // row -1 stands before row 0 (the first row of warp 0), row H
            // after row H - 1 (a second row; of an odd H it is held twice)
            float* up = &sh.cross[z & 1][0][0][0][lane].x;
            float* dn = &sh.cross[z & 1][1][0][nw - 1][lane].x + 1;
            constexpr int V = 2 * 32 * MW;
#pragma unroll
            for (int k = 0; k < NK; k++) {
                up[k * V] = hi(c.yp[k]);
                up[(NK + k) * V] = hi(c.pa[k]);
                up[(2 * NK + k) * V] = hi(c.pb[k]);
                if (H % 2 == 0) {
                    dn[k * V] = lo(c.ym[k]);
                    dn[(NK + k) * V] = lo(c.ma[k]);
                    dn[(2 * NK + k) * V] = lo(c.mb[k]);
                }
            }
            up[3 * NK * V] = hi(c.jyp);
            if (H % 2 == 0) dn[3 * NK * V] = lo(c.jym);
            wait_but_last();
            block_barrier();
        }
        cp_async_wait_all();
        if (PART) me.report(L, true);
    } else if (warp >= nw) {
        block_barrier();
        copy.psi(L, sh, z0 + 1, 0);
        copy.others(L, sh, z0, 0);
        cp_async_commit();
        Slots slot = {2, 0, 1};
        for (int z = z0 - 1; z <= z1; z++, slot.next()) {
            copy.psi(L, sh, min(z + 3, z1 + 1), slot.c);
            copy.others(L, sh, min(z + 2, z1), slot.c);
            cp_async_commit();
            wait_but_last();
            block_barrier();
        }
        cp_async_wait_all();
    } else {
        const bool cols = lane >= edge && lane < edge + TW && x0 + lane - edge < L.nx;
        const bool own0 = cols, own1 = cols && warp + nw < H;
        const long long nxy = (long long)L.nx * L.ny, ps = L.pstride;
        // the sites in a plane (columns of their own are within the lattice)
        const unsigned at[2] = {(unsigned)(x0 + lane - edge + L.nx * (y0 + warp)), (unsigned)(x0 + lane - edge + L.nx * (y0 + warp + nw))};
        MomentLane<NK, PART> me;
        me.place(lane, warp, warp + nw);
        if constexpr (NK == 2) {
            float S[2][2][3];
            me.advance(sh, 0, S);
            me.advance(sh, 1, S);
        }
        block_barrier();
        copy.psi(L, sh, z0 + 1, 0);
        copy.others(L, sh, z0, 0);
        cp_async_commit();
        Slots slot = {2, 0, 1};
        unsigned solid = 0;  // particle nodes of the two sites: bits 0, 1 this plane, bits 2, 3 the one before
        const long long seg = PART ? segment_of(L, x0, y0, H, z0, z1 - z0) : 0;
        const F2 zero = f2(0.f);
        MomentSum<NK> below, level;  // sums in progress of the plane before and of this one
#pragma unroll
        for (int k = 0; k < NK; k++) below.r[k] = level.r[k] = zero;
#pragma unroll
        for (int d = 0; d < 4; d++) below.j[d] = level.j[d] = zero;
#pragma unroll 1
        for (int z = z0 - 1; z <= z1; z++, slot.next()) {  // the plane whose links are formed
            const int b = z & 1;
            copy.psi(L, sh, min(z + 3, z1 + 1), slot.c);
            copy.others(L, sh, min(z + 2, z1), slot.c);
            cp_async_commit();
            MomentSum<NK> above;
            {
                F2 h[NK][3], r[NK], P[NK], r2[NK], r4[NK], P2[NK];
                const unsigned off = me.collide(L, sh, slot.a, z, h, r, P);
                if constexpr (PART) {
                    solid = solid << 2 | off;
                    if (z >= z0 && z < z1) {
                        const bool fr[2] = {own0 && !(off & 1u) && (me.nbn[0] & NB_LINKS),
                                            own1 && !(off & 2u) && (me.nbn[1] & NB_LINKS)};
                        const unsigned m0 = __ballot_sync(0xffffffffu, fr[0]), m1 = __ballot_sync(0xffffffffu, fr[1]);
                        if (m0 | m1) {
                            int n = 0;
                            if (lane == 0) n = atomicAdd(&sh.count, __popc(m0) + __popc(m1));
                            n = __shfl_sync(0xffffffffu, n, 0);
                            const unsigned under = (1u << lane) - 1u;
                            const int e[2] = {n + __popc(m0 & under), n + __popc(m0) + __popc(m1 & under)};
#pragma unroll
                            for (int a = 0; a < 2; a++) {
                                if (!fr[a]) continue;
                                unsigned* rec = list.rec + seg + e[a];
                                auto put = [&](unsigned v) { *rec = v, rec += L.N; };
                                put(at[a] + (unsigned)nxy * (unsigned)z);
                                put(me.nbn[a]);
#pragma unroll
                                for (int d = 0; d < 3; d++) {
                                    put(__float_as_uint(a == 0 ? lo(h[0][d]) : hi(h[0][d])));
                                    put(__float_as_uint(a == 0 ? lo(h[NK - 1][d]) : hi(h[NK - 1][d])));
                                }
                                put(__float_as_uint(a == 0 ? lo(r[0]) : hi(r[0])));
                                put(__float_as_uint(a == 0 ? lo(r[NK - 1]) : hi(r[NK - 1])));
                            }
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < NK; k++) {
                    r2[k] = r[k] + r[k];
                    r4[k] = r2[k] + r2[k];
                    P2[k] = P[k] + P[k];
                }
                {
                    CrossLinks<NK> c;
                    cross_links<NK>(h, r2, r4, P, P2, lane, c);
                    auto& up = sh.cross[b][0];
                    auto& dn = sh.cross[b][1];
                    // to the warp of the rows after this warp's; of the last
                    // warp the first row stands before row nw, the second row
                    // of warp 0
                    if (warp < nw - 1) {
#pragma unroll
                        for (int k = 0; k < NK; k++) {
                            up[k][warp + 1][lane] = c.yp[k];
                            up[NK + k][warp + 1][lane] = c.pa[k];
                            up[2 * NK + k][warp + 1][lane] = c.pb[k];
                        }
                        up[3 * NK][warp + 1][lane] = c.jyp;
                    } else {
#pragma unroll
                        for (int k = 0; k < NK; k++) {
                            up[k][0][lane].y = lo(c.yp[k]);
                            up[NK + k][0][lane].y = lo(c.pa[k]);
                            up[2 * NK + k][0][lane].y = lo(c.pb[k]);
                        }
                        up[3 * NK][0][lane].y = lo(c.jyp);
                    }
                    // and to the warp of the rows before them; of warp 0 the
                    // second row stands after row nw - 1, the first row of the last warp
                    if (warp > 0) {
#pragma unroll
                        for (int k = 0; k < NK; k++) {
                            dn[k][warp - 1][lane] = c.ym[k];
                            dn[NK + k][warp - 1][lane] = c.ma[k];
                            dn[2 * NK + k][warp - 1][lane] = c.mb[k];
                        }
                        dn[3 * NK][warp - 1][lane] = c.jym;
                    } else {
#pragma unroll
                        for (int k = 0; k < NK; k++) {
                            dn[k][nw - 1][lane].x = hi(c.ym[k]);
                            dn[NK + k][nw - 1][lane].x = hi(c.ma[k]);
                            dn[2 * NK + k][nw - 1][lane].x = hi(c.mb[k]);
                        }
                        dn[3 * NK][nw - 1][lane].x = hi(c.jym);
                    }
                }
                F2 m[NK], a[NK], ai[NK], c[NK], ci[NK], g[NK], jx, zm[NK];
#pragma unroll
                for (int k = 0; k < NK; k++) {
                    link_pair(h[k][2], r4[k], P2[k], m[k], zm[k]);                 // (0, 0, +-1)
                    link_pair(h[k][0] + h[k][2], r2[k], P[k], a[k], ai[k]);       // +-(1, 0, 1)
                    link_pair(h[k][0] - h[k][2], r2[k], P[k], c[k], ci[k]);       // +-(1, 0, -1)
                }
                // to the plane above, the plane below, and the plane itself
                join_x<NK>(m, a, ci, lane, above.r, above.j[0]);
                join_x<NK>(zm, c, ai, lane, g, jx);
#pragma unroll
                for (int k = 0; k < NK; k++) below.r[k] = below.r[k] + g[k];
                below.j[0] = below.j[0] + jx;
                below.j[2] = below.j[2] - total<NK>(g);
#pragma unroll
                for (int k = 0; k < NK; k++) {
                    link_pair(h[k][0], r4[k], P2[k], a[k], ai[k]);                // (+-1, 0, 0)
                    m[k] = fma2(f2(12.f), P[k], level.r[k]);                      // the rest population
                }
                join_x<NK>(m, a, ai, lane, level.r, jx);
                level.j[0] = level.j[0] + jx;
            }
            wait_but_last();
            block_barrier();
            // what comes from the rows before along y (p), and after (m)
            const auto& up = sh.cross[b][0];
            const auto& dn = sh.cross[b][1];
            F2 p[NK], m[NK], t[NK], o[NK], j[3];
#pragma unroll
            for (int k = 0; k < NK; k++) {
                p[k] = up[2 * NK + k][warp][lane];
                m[k] = dn[2 * NK + k][warp][lane];
                t[k] = p[k] + m[k];
                o[k] = below.r[k] + t[k];  // the plane below is complete
            }
            j[0] = below.j[0];
            j[1] = below.j[1] + (total<NK>(p) - total<NK>(m));
            j[2] = below.j[2] + (below.j[3] - total<NK>(t));
#pragma unroll
            for (int k = 0; k < NK; k++) {
                p[k] = up[k][warp][lane];
                m[k] = dn[k][warp][lane];
                below.r[k] = level.r[k] + (p[k] + m[k]);
            }
            below.j[0] = level.j[0] + (up[3 * NK][warp][lane] + dn[3 * NK][warp][lane]);
            below.j[1] = level.j[1] + (total<NK>(p) - total<NK>(m));
            below.j[2] = level.j[2];
            below.j[3] = level.j[3];
#pragma unroll
            for (int k = 0; k < NK; k++) {
                p[k] = up[NK + k][warp][lane];
                m[k] = dn[NK + k][warp][lane];
                t[k] = p[k] + m[k];
                level.r[k] = above.r[k] + t[k];
            }
            level.j[0] = above.j[0];
            level.j[1] = total<NK>(p) - total<NK>(m);
            level.j[2] = total<NK>(above.r);
            level.j[3] = total<NK>(t);
            if (z <= z0) continue;
            // 1/36 as a rounded value and the rest of it: the rounded value
            // alone would let the sums grow by 2e-8 a step
            constexpr float h36 = 1.0f / 36.0f, l36 = (float)(1.0 / 36.0 - (double)h36);
#pragma unroll
            for (int k = 0; k < NK; k++) o[k] = fma2(o[k], f2(h36), o[k] * f2(l36)) + f2(sh.ref[k]);
#pragma unroll
            for (int d = 0; d < 3; d++) j[d] = fma2(j[d], f2(h36), j[d] * f2(l36));
            float* psi_z = psi_o + NK * nxy * (z - 1);
            float* mom_z = mom_o + nxy * (z - 1);
#pragma unroll
            for (int e = 0; e < 2; e++) {
                if (!(e == 0 ? own0 : own1)) continue;
                float ra = e == 0 ? lo(o[0]) : hi(o[0]), rb = e == 0 ? lo(o[NK - 1]) : hi(o[NK - 1]);
                const bool off = PART && (solid & (e == 0 ? 4u : 8u));
                if (off) ra = L.rref[0], rb = L.rref[NK - 1];  // (any density that is not below L.rlow)
                if (NK == 2)
                    reinterpret_cast<float2*>(psi_z)[at[e]] = make_float2(ra, rb);
                else
                    psi_z[at[e]] = ra;
                float* mz = mom_z;
#pragma unroll
                for (int d = 0; d < 3; d++) mz[at[e]] = off ? 0.f : (e == 0 ? lo(j[d]) : hi(j[d])), mz += ps;
            }
        }
        cp_async_wait_all();
        me.report(L, cols);
    }
    if constexpr (PART) {
        block_barrier();
        if (threadIdx.x == 0) list.count[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = sh.count | (L.spread[L.turn] ? LIST_PLAIN : 0);
    }
}

// The bounce-back links of the listed boundary sites (`parts` blocks per
// segment of the grid of k_moments): the values that come back (Eqs. 17, 18)
// added to the sums k_moments left in psi_o, mom_o, and the forces and torques
// they hand to the particles (Eqs. 19, 22, 23).  A kernel of its own: a site's
// particle is two dependent loads away, which inside the march of k_moments
// every plane of a block waited for (256^3, 2407 particles: 654 us together, 366
// + 128 us apart; at the end of each block, 15 warps on an SM, 512 x 512 x 256
// took 1994 us instead of 1286 + 474).  It is bound by the latency of those
// loads: the sums are fetched beside them, and the links of a site are
// evaluated by opposite pairs without branches (103 -> 88 us at 256^3).  The
// sites of a warp mostly belong to a few particles in runs: the fixed-point
// words of a run are summed across the lanes and added once (integer sums: the
// bits do not depend on the grouping).
__global__ void __launch_bounds__(128) k_bounce_links(const __grid_constant__ Lattice L, float* __restrict__ psi_o,
                                                       float* __restrict__ mom_o, LinkList list, int zc, int TW,
                                                       int parts, long long unit) {
    chain_begin();
    const int bx = blockIdx.x / parts, z0 = blockIdx.z * zc, x0 = bx * TW, y0 = blockIdx.y * MROWS;
    const int count = list.count[bx + gridDim.x / parts * (blockIdx.y + gridDim.y * blockIdx.z)];
    const int n = count & ~LIST_PLAIN;
    const bool plain = count & LIST_PLAIN;
    const F2 ref = plain ? f2(0.f) : f2(L.rref[0], L.rref[1]);
    if (plain) unit = 0;
    const unsigned* seg = list.rec + segment_of(L, x0, y0, min(MROWS, L.ny - y0), z0, min(zc, L.nz - z0));
    const int lane = threadIdx.x & 31, nx = L.nx, nxy = L.nx * L.ny;
    for (int k0 = (int)(blockIdx.x % parts * 128 + threadIdx.x) - lane; k0 < n; k0 += 128 * parts) {
        const int k = k0 + lane;
        int p = -1, exact[3] = {0, 0, 0};
        float F[3] = {0, 0, 0}, T[3] = {0, 0, 0};
        if (k < n) {
            const unsigned* rec = seg + k;
            auto get = [&]() { const unsigned v = *rec; rec += L.N; return v; };
            const unsigned s = get(), nbc = get(), bits = nbc & NB_LINKS;
            F2 h[3], r;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const float a = __uint_as_float(get());
                h[d] = f2(a, __uint_as_float(get()));
            }
            const float ra = __uint_as_float(get());
            r = f2(ra, __uint_as_float(get()));
            // the sums that the links are added to, on their way while the
            // particle is looked up
            F2* ps = reinterpret_cast<F2*>(psi_o) + s;
            float* mo = mom_o + s;
            const F2 sum = *ps;
            const float js[3] = {mo[0], mo[L.pstride], mo[2 * L.pstride]};
            const int z = (int)(s / (unsigned)nxy), yx = (int)(s - (unsigned)z * (unsigned)nxy), y = yx / nx, x = yx - y * nx;
            const int dxp = x == nx - 1 ? 1 - nx : 1, dxm = x == 0 ? nx - 1 : -1;
            const int dyp = y == L.ny - 1 ? nx - nxy : nx, dym = y == 0 ? nxy - nx : -nx;
            const int dzp = z == L.nz - 1 ? nxy - (int)L.N : nxy, dzm = z == 0 ? (int)L.N - nxy : -nxy;
            auto owner_of = [&](int i) {
                const int ax = rc(0, i), ay = rc(1, i), az = rc(2, i);
                return L.owner[s + (unsigned)((ax > 0 ? dxp : (ax < 0 ? dxm : 0)) + (ay > 0 ? dyp : (ay < 0 ? dym : 0)) +
                                              (az > 0 ? dzp : (az < 0 ? dzm : 0)))];
            };
            // (as in k_moments, deviations from a fluid of the reference density at rest)
            const F2 hh = fma2(h[2], h[2], fma2(h[1], h[1], h[0] * h[0]));
            const F2 P = fma2(r * hh, f2(-2.f / 3.f), r - ref), P2 = P + P, r2 = r + r, r4 = r2 + r2;
            F2 back = f2(0.f);
            float j[3] = {0, 0, 0};
            // a link f*_i and what comes back, f*_i - 6 w_i rho c_i.u_w (Eq. 17):
            // added to back and j; returns the momentum handed over (Eq. 19)
            auto link = [&](int i, F2 ch, float cu, float ax, float ay, float az) {
                const F2 q = (i <= 6 ? r4 : r2) * ch, f0 = fma2(q, ch, i <= 6 ? P2 : P) + q;
                const F2 fb = fma2(i <= 6 ? r2 : r, f2(-6.f * cu), f0);
                back = back + fb;
                const float sb = lo(fb) + hi(fb);
                j[0] -= ax * sb;
                j[1] -= ay * sb;
                j[2] -= az * sb;
                return lo(f0) + hi(f0) + sb;
            };
            // the links of that fluid: their number (by weight) and its sums along
            // each axis, for the exact part of the sums
            const float nw = (float)(2 * __popc(bits & 0x7eu) + __popc(bits & 0x7ff80u));
            int nd[3];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                unsigned up = 0, dn = 0;
#pragma unroll
                for (int i = 7; i < Q; i++) {
                    const int c = d == 0 ? cx(i) : (d == 1 ? cy(i) : cz(i));
                    up |= c > 0 ? 1u << i : 0u;
                    dn |= c < 0 ? 1u << i : 0u;
                }
                nd[d] = __popc(bits & up) - __popc(bits & dn) + 2 * (int)((bits >> (2 * d + 1)) & 1u) -
                        2 * (int)((bits >> (2 * d + 2)) & 1u);
            }
            const float rr = lo(ref) + hi(ref);
            float U[3], rel[3];
            if (nbc & NB_MULTI) {
                // next to two particles: each link with its own, forces added directly
                for (unsigned m = bits; m; m &= m - 1) {
                    const int i = __ffs(m) - 1, o = owner_of(i);
                    const float ax = (float)rc(0, i), ay = (float)rc(1, i), az = (float)rc(2, i);
                    particle_u0<float>(L, o, x, y, z, U, rel);
                    const float fl = link(i, f2(ax) * h[0] + f2(ay) * h[1] + f2(az) * h[2],
                                          ax * U[0] + ay * U[1] + az * U[2], ax, ay, az) * (1.f / 36.f) +
                                     (i <= 6 ? 4.f : 2.f) * rr * (1.f / 36.f);
                    const float f[3] = {ax * fl, ay * fl, az * fl};
                    const float t[3] = {rel[1] * f[2] - rel[2] * f[1], rel[2] * f[0] - rel[0] * f[2], rel[0] * f[1] - rel[1] * f[0]};
                    commit_link_forces<float>(L, o, f, t);
                }
            } else {
                p = owner_of(__ffs(bits) - 1);
                particle_u0<float>(L, p, x, y, z, U, rel);
                const float V[3] = {-6.f * U[0], -6.f * U[1], -6.f * U[2]};
                // the opposite links of a pair hand over e + q, e - q and get back
                // e + o, e - o; those the site has count by the sum and the
                // difference of their bits: no branch (half of the lanes of a warp
                // have a given link, so branches ran for all of them)
#pragma unroll
                for (int i = 1; i < Q; i += 2) {
                    const float up = (bits >> i) & 1u ? 1.f : 0.f, dn = (bits >> (i + 1)) & 1u ? 1.f : 0.f;
                    const float m = up + dn, df = up - dn;
                    F2 ch = f2(0.f);
                    bool any = false;
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        const int c = d == 0 ? cx(i) : (d == 1 ? cy(i) : cz(i));
                        if (c == 0) continue;
                        ch = !any ? (c > 0 ? h[d] : f2(0.f) - h[d]) : (c > 0 ? ch + h[d] : ch - h[d]);
                        any = true;
                    }
                    const F2 q = (i <= 6 ? r4 : r2) * ch, e = fma2(q, ch, i <= 6 ? P2 : P);
                    const F2 o = fma2(i <= 6 ? r2 : r, f2(along<float>(i, V)), q);
                    back = fma2(f2(m), e, fma2(f2(df), o, back));
                    const float es = df * (lo(e) + hi(e)), os = lo(o) + hi(o), qs = lo(q) + hi(q);
                    const float jb = fmaf(m, os, es), fl = jb + fmaf(m, qs, es);
                    if (cx(i)) j[0] -= cx(i) * jb, F[0] += cx(i) * fl;
                    if (cy(i)) j[1] -= cy(i) * jb, F[1] += cy(i) * fl;
                    if (cz(i)) j[2] -= cz(i) * jb, F[2] += cz(i) * fl;
                }
                // Eq. 23 with r_w - r_p = (x - r_p) + c_i/2: the c_i/2 part is
                // parallel to the link force and drops out of the torque
                float G[3];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    F[d] *= 1.f / 36.f;
                    exact[d] = nd[d];
                    G[d] = fmaf((float)nd[d], 2.f * rr * (1.f / 36.f), F[d]);
                }
                T[0] = rel[1] * G[2] - rel[2] * G[1];
                T[1] = rel[2] * G[0] - rel[0] * G[2];
                T[2] = rel[0] * G[1] - rel[1] * G[0];
            }
            back = fma2(f2(nw), ref, back);
#pragma unroll
            for (int d = 0; d < 3; d++) j[d] = fmaf((float)-nd[d], rr, j[d]);
            constexpr float h36 = 1.0f / 36.0f, l36 = (float)(1.0 / 36.0 - (double)h36);
            *ps = fma2(back, f2(h36), fma2(back, f2(l36), sum));
#pragma unroll
            for (int d = 0; d < 3; d++) *mo = fmaf(j[d], h36, fmaf(j[d], l36, js[d])), mo += L.pstride;
        }
        add_runs(L, ACC_FLIQ, p, F, T, exact, unit);
    }
}

// The links that come back from the z faces, added to the sums of the planes
// next to them: walls and velocity faces (Eq. 9), pressure faces (Eq. 10),
// equilibrium faces.  k_moments leaves them out (their sources lie beyond the
// lattice); one thread per site of a plane forms the site's five collided
// links into the face from psi and mom of time t.
template <int NK>
__global__ void k_moment_faces(const __grid_constant__ Lattice L, float* __restrict__ psi_o, float* __restrict__ mom_o) {
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, face = blockIdx.z;
    if (x >= L.nx) return;
    const int z = face == 0 ? 0 : L.nz - 1;
    const long long xy = x + (long long)L.nx * y, s = xy + (long long)L.nx * L.ny * z;
    if (NK == 2 && L.mask[s]) return;
    const float* psi = (const float*)L.psi;
    const float* mom = (const float*)L.mom;
    float rho[NK], u[3], us[NK][3];
#pragma unroll
    for (int k = 0; k < NK; k++) rho[k] = psi[NK * s + k];
    const float ir = 1.0f / (NK == 2 ? rho[0] + rho[NK - 1] : rho[0]);
#pragma unroll
    for (int d = 0; d < 3; d++) u[d] = mom[d * L.pstride + s] * ir;
    if constexpr (NK == 2) {
        float one[2] = {1.f, 1.f}, F[2][3];  // F^k / rho^k
        sc_force<float>(L, site_nbr(L, x, y, z), one, F);
#pragma unroll
        for (int k = 0; k < 2; k++)
#pragma unroll
            for (int d = 0; d < 3; d++) us[k][d] = u[d] + F[k][d];
    } else {
#pragma unroll
        for (int d = 0; d < 3; d++) us[0][d] = u[d] + L.PF.body_force[d];
    }
    const float* uw = face == 0 ? L.PF.wall_u_lo : L.PF.wall_u_hi;
    const int type = L.P.open[face];
    const bool plain = L.spread[L.turn];
    const bool ext = L.P.open_extrap && (type == 1 || type == 2);
    // the face values of the column (k_face_values): rho_w^k, u_w
    const float* fv = (const float*)L.face + 5 * ((long long)face * L.nx * L.ny + xy);
    if (type == 1 && ext)
        for (int d = 0; d < 3; d++) u[d] = fv[2 + d];
    const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2], uwu = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
    float add[NK] = {}, j[3] = {0, 0, 0};
#pragma unroll
    for (int i = 1; i < Q; i++) {
        if (cz(i) != -1) continue;
        // the link (cx, cy, -1) into the lower face, (cx, cy, 1) into the upper one
        const float az = face == 0 ? -1.f : 1.f;
        const float cw = cx(i) * uw[0] + cy(i) * uw[1] + az * uw[2], cu = cx(i) * u[0] + cy(i) * u[1] + az * u[2];
        float sum = 0;
#pragma unroll
        for (int k = 0; k < NK; k++) {
            const float cs = cx(i) * us[k][0] + cy(i) * us[k][1] + az * us[k][2];
            const float ss = us[k][0] * us[k][0] + us[k][1] * us[k][1] + us[k][2] * us[k][2];
            // less the link of the reference fluid (see k_moments), in units of 1/36
            const float W = i <= 6 ? 2.f : 1.f, ref = plain ? 0.f : L.rref[k], ro = (float)L.P.open_rho[face][k];
            const float fs = W * ((rho[k] - ref) + rho[k] * (3.f * cs + 4.5f * cs * cs - 1.5f * ss));
            float fb;
            if (type == 1) fb = W * (2.f * (ro - ref) + ro * (9.f * cu * cu - 3.f * uu)) - fs;
            else if (type == 3) fb = W * ((ro - ref) + ro * (4.5f * cw * cw - 3.f * cw - 1.5f * uwu));
            else fb = fs - 6.f * W * (ext ? fv[k] : rho[k]) * cw;
            add[k] += fb;
            sum += fb;
        }
        j[0] -= cx(i) * sum;
        j[1] -= cy(i) * sum;
        j[2] -= az * sum;
    }
    // the reference fluid's links: weight 6 in all, along z only
    constexpr float h36 = 1.0f / 36.0f, l36 = (float)(1.0 / 36.0 - (double)h36);
    float ref = 0;
#pragma unroll
    for (int k = 0; k < NK; k++) {
        add[k] += plain ? 0.f : 6.f * L.rref[k];
        ref += plain ? 0.f : 6.f * L.rref[k];
        psi_o[NK * s + k] = fmaf(add[k], h36, fmaf(add[k], l36, psi_o[NK * s + k]));
    }
    j[2] += face == 0 ? ref : -ref;
#pragma unroll
    for (int d = 0; d < 3; d++) mom_o[d * L.pstride + s] = fmaf(j[d], h36, fmaf(j[d], l36, mom_o[d * L.pstride + s]));
}

// z chunk: the whole-wave count times the planes a block passes (its chunk and
// the four planes that fill the march) is smallest
static int moment_chunk(const Lattice& L, long long tiles, int per_sm) {
    const long long R = (long long)device_sms() * per_sm;
    int best = L.nz;
    long long cost = -1;
    // (each chunk once: a long lattice has as many numbers of chunks as planes, and
    // the host would look through all of them in every step)
    for (int zc = L.nz;;) {
        const long long n = (L.nz + zc - 1) / zc, c = ((tiles * n + R - 1) / R) * (zc + 4);
        if (cost < 0 || c < cost) {
            cost = c;
            best = zc;
        }
        if (zc <= 2) break;
        const int m = (L.nz + zc - 2) / (zc - 1);  // chunks of fewer planes than zc
        zc = (L.nz + m - 1) / m;
    }
    return best;
}

template <int NK, bool PART>
static int launch_moments_t(const Lattice& L, void* psi_o, void* mom_o, cudaStream_t st) {
    const size_t smem = sizeof(MomentShared<NK, PART>);
    const int per_sm = kernel_setup<k_moments<NK, PART>>(MNT, smem);
    const int TW = L.nx == 32 ? 32 : 28;
    const unsigned gx = (unsigned)((L.nx + TW - 1) / TW), gy = (unsigned)((L.ny + MROWS - 1) / MROWS);
    const int zc = moment_chunk(L, (long long)gx * gy, per_sm);
    const dim3 grid(gx, gy, (unsigned)((L.nz + zc - 1) / zc));
    // the list of boundary sites lies in the second population buffer, which a
    // step of this kind does not touch (MREC words and a part of a count a
    // site, of at least 76 bytes a site)
    LinkList list = {(unsigned*)L.f_nxt, (int*)L.f_nxt + (size_t)MREC * L.N};
    float *po = (float*)psi_o, *mo = (float*)mom_o;
    int n = 1;
    launch_after(k_moments<NK, PART>, grid, MNT, smem, st, L, po, mo, list, zc, TW);
    if (PART) {
        // about a fifth of the sites are boundary sites in a dense suspension:
        // blocks for two or three rounds over a segment
        const int parts = (zc * TW * MROWS + 128 * 16 - 1) / (128 * 16);
        // what a link of weight 1/36 of the reference fluid hands over (2 f*_i of
        // both components), in fixed point
        const long long unit = llrint(((double)L.rref[0] + (double)L.rref[1]) * (2.0 / 36.0 * 1099511627776.0));
        launch_after(k_bounce_links, dim3(gx * parts, gy, grid.z), 128, 0, st, L, po, mo, list, zc, TW, parts, unit);
        n++;
    }
    if (!L.per[2]) {
        k_moment_faces<NK><<<dim3((unsigned)((L.nx + 127) / 128), (unsigned)L.ny, 2), 128, 0, st>>>(L, po, mo);
        n++;
    }
    return n;
}

int launch_moments(const Lattice& L, void* psi_o, void* mom_o, cudaStream_t st) {
    if (L.ncomp == 1) return launch_moments_t<1, false>(L, psi_o, mom_o, st);
    if (L.nc > 0) return launch_moments_t<2, true>(L, psi_o, mom_o, st);
    return launch_moments_t<2, false>(L, psi_o, mom_o, st);
}

}  // namespace lbgb
