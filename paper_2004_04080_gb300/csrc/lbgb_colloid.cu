// lbgb_colloid.cu -- particle kernels: node map and remap (destroy / create),
// wetting virtual densities with the solid-node Shan-Chen force, Ladd link
// forces, pair forces (cell list) and the rotational leap-frog integrator.
//
// Per-particle lattice work runs one 16x8 thread block per particle over the
// box of lattice points around its sphere.  Geometry is evaluated in the
// compute type of the populations (FP32 for the FP32 / FP16 forms): FP64
// arithmetic on GB300 runs at a small fraction of the FP32 rate and costs a
// whole warp even in a divergent branch, so it is kept out of per-link code.
// Node membership |x - r_p|^2 < R^2 is nevertheless decided exactly: points
// whose FP32 distance is within a safe margin of the sphere are re-tested in
// FP64.  Every term of a per-particle sum is added in fixed point (acc_add),
// so the totals do not depend on the order of the threads.
#include "lbgb_internal.cuh"

namespace lbgb {

constexpr int BXP = 16, BYP = 8, PB = BXP * BYP;  // particle block
// a particle moves less than 1/2 along each axis in a step (checked by the
// integrator), so less than sqrt(3)/2; the box of the remap reaches beyond that
constexpr float REMAP_REACH = 0.88f;
constexpr double REMAP_PAD = 0.95;

// geometry of particle p in compute type C
template <typename C>
struct PGeo {
    int lo[3], ext[3];  // box of lattice points
    int ip[3];          // floor(r_p)
    C fr[3];            // r_p - floor(r_p)
    C v[3], w[3];       // v(t-1/2), omega(t-1/2)
    double R;
    C R2;
};

template <typename C>
__device__ __forceinline__ PGeo<C> pgeo(const Lattice& L, int p, double pad) {
    PGeo<C> g;
    g.R = L.rad[p];
    g.R2 = C(g.R) * C(g.R);
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (sizeof(C) == 8) {
            double r = L.pos[3 * p + d];
            g.lo[d] = (int)floor(r - g.R - pad);
            g.ext[d] = (int)ceil(r + g.R + pad) - g.lo[d] + 1;
            g.ip[d] = (int)floor(r);
            g.fr[d] = C(r - (double)g.ip[d]);
            g.v[d] = C(L.vel[3 * p + d]);
            g.w[d] = C(L.omg[3 * p + d]);
        } else {
            // box from the snapshot: r = ip + fr with fr in [0, 1) (the box only
            // has to cover the working shell, which it does with a wide margin)
            g.ip[d] = L.ipos[3 * p + d];
            g.fr[d] = C(L.fsnap[9 * p + d]);
            g.v[d] = C(L.fsnap[9 * p + 3 + d]);
            g.w[d] = C(L.fsnap[9 * p + 6 + d]);
            float Rp = float(g.R) + float(pad);
            g.lo[d] = g.ip[d] + (int)floorf(float(g.fr[d]) - Rp);
            g.ext[d] = g.ip[d] + (int)ceilf(float(g.fr[d]) + Rp) - g.lo[d] + 1;
        }
    }
    return g;
}

// exact membership |a - r_p|^2 < R^2 (FP64 without contraction, as a plain
// double evaluation would decide it)
__device__ __noinline__ bool inside_exact(const Lattice& L, int p, int a, int b, int c) {
    double dx = (double)a - L.pos[3 * p], dy = (double)b - L.pos[3 * p + 1], dz = (double)c - L.pos[3 * p + 2];
    double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    double R = L.rad[p];
    return d2 < __dmul_rn(R, R);
}

template <typename C>
__device__ __forceinline__ bool inside(const Lattice& L, int p, const PGeo<C>& g, const C (&d)[3], int a, int b,
                                       int c) {
    if (sizeof(C) == 8) return inside_exact(L, p, a, b, c);
    C d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    C gap = d2 - g.R2;
    if (gap > C(1e-2) || gap < C(-1e-2)) return gap < C(0);
    return inside_exact(L, p, a, b, c);
}

// Visit the box points of particle p; f(X, Y, Z, s, a, b, c, d) gets the
// wrapped site, its index, the unwrapped point and its offset from r_p.
template <typename C, typename Fn>
__device__ __forceinline__ void for_box(const Lattice& L, const PGeo<C>& g, Fn&& fn) {
    for (int zz = 0; zz < g.ext[2]; zz++) {
        int c = g.lo[2] + zz;
        if (!L.per[2] && (c < 0 || c >= L.nz)) continue;
        int Z = c < 0 ? c + L.nz : (c >= L.nz ? c - L.nz : c);
        for (int yy = threadIdx.y; yy < g.ext[1]; yy += BYP) {
            int b = g.lo[1] + yy;
            int Y = b < 0 ? b + L.ny : (b >= L.ny ? b - L.ny : b);
            for (int xx = threadIdx.x; xx < g.ext[0]; xx += BXP) {
                int a = g.lo[0] + xx;
                int X = a < 0 ? a + L.nx : (a >= L.nx ? a - L.nx : a);
                long long s = (long long)X + (long long)L.nx * ((long long)Y + (long long)L.ny * Z);
                C d[3] = {C(a - g.ip[0]) - g.fr[0], C(b - g.ip[1]) - g.fr[1], C(c - g.ip[2]) - g.fr[2]};
                fn(X, Y, Z, s, a, b, c, d);
            }
        }
    }
}

// Visit the box points of particle p whose distance from the centre lies in
// [R + lo, R + hi), one (y, z) row of the box per thread: the x range of a row
// that reaches the shell is found from the row's distance to the centre (one
// or two intervals), so a thin shell costs its own points instead of the
// whole box.  The shell is found in FP32 with a margin of 0.02 in x (far above
// its rounding); what a point is, fn decides.  Sites are indexed in 32 bits.
template <typename C, typename Fn>
__device__ __forceinline__ void for_band(const Lattice& L, const PGeo<C>& g, float lo, float hi, Fn&& fn) {
    constexpr float margin = 0.02f;
    const int tid = threadIdx.y * BXP + threadIdx.x;
    const int nrow = g.ext[1] * g.ext[2];
    const float Rin = fmaxf(float(g.R) + lo, 0.f), Rout = float(g.R) + hi;
    const float fx = float(g.fr[0]), fy = float(g.fr[1]), fz = float(g.fr[2]);
    for (int r = tid; r < nrow; r += PB) {
        const int zz = r / g.ext[1], b = g.lo[1] + r - zz * g.ext[1], c = g.lo[2] + zz;
        const float y = float(b - g.ip[1]) - fy, z = float(c - g.ip[2]) - fz;
        const float q = y * y + z * z, ho = Rout * Rout - q, hin = Rin * Rin - q;
        if (!(ho > 0.f) || (!L.per[2] && (c < 0 || c >= L.nz))) continue;
        const float xo = sqrtf(ho) + margin, xi = hin > 0.f ? sqrtf(hin) - margin : 0.f;
        const int Y = b < 0 ? b + L.ny : (b >= L.ny ? b - L.ny : b);
        const int Z = c < 0 ? c + L.nz : (c >= L.nz ? c - L.nz : c);
        const int row = L.nx * (Y + L.ny * Z);
        // |x - r_p| in [xi, xo]: the left and right intervals (one if xi <= 0)
        const int aL0 = (int)ceilf(fx - xo), aR1 = (int)floorf(fx + xo);
        const int aL1 = xi > 0.f ? (int)floorf(fx - xi) : aR1, aR0 = xi > 0.f ? (int)ceilf(fx + xi) : aR1 + 1;
        const int nl = aL1 - aL0 + 1, total = max(nl, 0) + max(aR1 - aR0 + 1, 0);
        for (int t = 0; t < total; t++) {
            const int a = t < nl ? aL0 + t : aR0 + t - max(nl, 0);
            const int ax = a + g.ip[0];
            const C d[3] = {C(a) - g.fr[0], C(b - g.ip[1]) - g.fr[1], C(c - g.ip[2]) - g.fr[2]};
            const int X = ax < 0 ? ax + L.nx : (ax >= L.nx ? ax - L.nx : ax);
            fn(X, Y, Z, (long long)(row + X), ax, b, c, d);
        }
    }
}

template <typename C>
__device__ __forceinline__ void crs(const C (&a)[3], const C (&b)[3], C (&o)[3]) {
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

template <int PREC>
__device__ __forceinline__ typename Prec<PREC>::C site_rho(const Lattice& L, long long s, int k) {
    typedef typename Prec<PREC>::S S;
    typedef typename Prec<PREC>::C C;
    const S* f = (const S*)L.f_cur;
    C r = 0;
#pragma unroll
    for (int i = 0; i < Q; i++)
        r += ld_pop(f + pop_index(k * Q + i, s, L.pstride), pop_shift<S, C>(L, k, i));
    return r;
}

// rho^k of a fluid node, from the populations or (MOM) from the moments
template <int PREC, bool MOM>
__device__ __forceinline__ typename Prec<PREC>::C node_rho(const Lattice& L, long long s, int k) {
    typedef typename Prec<PREC>::C C;
    if (MOM) return ((const C*)L.psi)[2 * s + k];
    return site_rho<PREC>(L, s, k);
}

// a node a particle covers holds no fluid (MOM: the density pass is not run
// again), but a density of use to k_moments
template <int PREC, bool MOM>
__device__ __forceinline__ void clear_moments(const Lattice& L, long long s) {
    typedef typename Prec<PREC>::C C;
    if (MOM) {
        for (int k = 0; k < 2; k++) ((C*)L.psi)[2 * s + k] = C(L.rref[k]);
        for (int d = 0; d < 3; d++) ((C*)L.mom)[d * L.pstride + s] = C(0);
    }
}

// -------------------------------------------------- FP32 snapshot
__global__ void k_snapshot(Lattice L) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= L.nc) return;
    for (int d = 0; d < 3; d++) {
        double r = L.pos[3 * p + d];
        int ip = (int)floor(r);
        L.ipos[3 * p + d] = ip;
        L.fsnap[9 * p + d] = float(r - (double)ip);
        L.fsnap[9 * p + 3 + d] = float(L.vel[3 * p + d]);
        L.fsnap[9 * p + 6 + d] = float(L.omg[3 * p + d]);
    }
}

// ------------------------------------------------------ initial node map
// First map after particles are added: nodes are claimed without momentum
// bookkeeping (Sec. 2.4).
template <int PREC>
__global__ void __launch_bounds__(PB) k_map_initial(Lattice L, int first) {
    typedef typename Prec<PREC>::C C;
    int p = first + blockIdx.x;
    PGeo<C> g = pgeo<C>(L, p, 0.0);
    for_box<C>(L, g, [&](int, int, int, long long s, int a, int b, int c, const C (&d)[3]) {
        if (!inside<C>(L, p, g, d, a, b, c)) return;
        int old = atomicCAS(L.owner + s, -1, p);
        if (old != -1 && old != p) atomicOr(L.flags, FLAG_OVERLAP);
        L.mask[s] = 1;
    });
}

// ------------------------------------------------------------- remap
// The nodes the remap of a step changes are marked in evt and listed (nb_chg,
// up to NB_CHG_CAP): the refill, the commit and the link classes then visit
// only them.  When more change, the list is left incomplete and every kernel
// that uses it scans evt (the link classes: every site) instead.  The list is
// empty at the start of a step (k_integrate leaves it so).
__device__ __forceinline__ void list_changed(const Lattice& L, long long s) {
    const int q = atomicAdd(L.nb_chg, 1);
    if (q < NB_CHG_CAP) L.nb_chg[8 + q] = (int)s;
}

// x_s - r_p (minimum image) and the particle's v, omega, in the compute type:
// FP32 / FP16 from the snapshot (integer cell + offset), FP64 from the state
template <typename C>
__device__ __forceinline__ void particle_frame(const Lattice& L, int p, int x, int y, int z, C (&d)[3], C (&v)[3],
                                               C (&w)[3]) {
    const int xs[3] = {x, y, z}, Ls[3] = {L.nx, L.ny, L.nz};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        int ip;
        C fr;
        if (sizeof(C) == 8) {
            const double r = L.pos[3 * p + c];
            ip = (int)floor(r);
            fr = C(r - (double)ip);
            v[c] = C(L.vel[3 * p + c]);
            w[c] = C(L.omg[3 * p + c]);
        } else {
            ip = L.ipos[3 * p + c];
            fr = C(L.fsnap[9 * p + c]);
            v[c] = C(L.fsnap[9 * p + 3 + c]);
            w[c] = C(L.fsnap[9 * p + 6 + c]);
        }
        int dd = xs[c] - ip;
        if (L.per[c]) {
            if (2 * dd > Ls[c]) dd -= Ls[c];
            else if (2 * dd < -Ls[c]) dd += Ls[c];
        }
        d[c] = C(dd) - fr;
    }
}

// Classify the points around particle p at its new position r_p(t):
//   fluid node now inside -> destroy (Eq. 24): its momentum rho u goes to p
//   node of p now outside -> create (handled by k_remap_create)
// The node map is that of the position before the last move v, so a node
// changes side only if it is within |v| of the surface: only that shell (with
// a margin far above the rounding of the FP32 distances) is visited, row by
// row of the box.  The first step of a call (wide) visits a shell of 0.65 at
// least, so that particles which overlapped before it are reported by every
// call that steps them.  A shell of 0.65 for every particle read the
// owner map of ten times the points: 512 x 512 x 256, 14,444 particles, 302
// us against 101 (96^3 FP64: 90 against 27).  Points outside the shell are found
// in FP32 before any FP64 distance is formed (39 us before at 96^3).
template <int PREC, bool MOM>
__global__ void __launch_bounds__(PB) k_remap_classify(const __grid_constant__ Lattice L, bool wide) {
    chain_begin();
    typedef typename Prec<PREC>::C C;
    int p = blockIdx.x;
    PGeo<C> g = pgeo<C>(L, p, REMAP_PAD);
    const float v2 = float(g.v[0]) * float(g.v[0]) + float(g.v[1]) * float(g.v[1]) + float(g.v[2]) * float(g.v[2]);
    const float reach = fminf(fmaxf(sqrtf(v2) + 0.01f, wide ? 0.65f : 0.f), REMAP_REACH);
    for_band<C>(L, g, -reach, reach, [&](int, int, int, long long s, int a, int b, int c, const C (&d)[3]) {
        int o = L.owner[s];
        if (inside<C>(L, p, g, d, a, b, c)) {
            if (o == -1) {
                if (atomicCAS(L.evt + s, 0, 4 * (p + 1) + 1) != 0) {
                    atomicOr(L.flags, FLAG_OVERLAP);
                    return;
                }
                list_changed(L, s);
                C mom[3], tq[3];
                if (MOM) {  // rho u = j at equal tau
                    for (int m = 0; m < 3; m++) mom[m] = ((const C*)L.mom)[m * L.pstride + s];
                } else {
                    C fv[2][Q], rho[2], j[2][3], u[3], om;
                    load_site<PREC>(L, (const typename Prec<PREC>::S*)L.f_cur, s, fv, rho, j);
                    mixture<C>(L, rho, j, u, om);
                    C rt = rho[0] + rho[1];
                    for (int m = 0; m < 3; m++) mom[m] = rt * u[m];
                }
                crs<C>(d, mom, tq);
                for (int m = 0; m < 3; m++) {
                    acc_add(L, acc_slot(L, ACC_FD, p, m), mom[m]);
                    acc_add(L, acc_slot(L, ACC_TD, p, m), tq[m]);
                }
            } else if (o != p) {
                atomicOr(L.flags, FLAG_OVERLAP);
            }
        } else if (o == p) {
            L.evt[s] = 4 * (p + 1) + 2;
            list_changed(L, s);
        }
    });
}

// Refill of node s, which particle p released (Eq. 25), by one warp:
// f = f^eq(rhobar^k, u_w) (MOM: its moments) with rhobar^k the w_i-weighted
// mean over neighbours that are fluid before and after the remap (a lane per
// neighbour, summed in link order), u_w = v_p + omega_p x (r - r_p); the
// momentum (rhobar) u_w it carries off is a term of F_c, T_c.
template <int PREC, bool MOM>
__device__ __forceinline__ void refill_node(const Lattice& L, long long s, int p, int lane) {
    typedef typename Prec<PREC>::S S;
    typedef typename Prec<PREC>::C C;
    const long long xy = (long long)L.nx * L.ny;
    const int Z = (int)(s / xy), r = (int)(s - (long long)Z * xy), Y = r / L.nx, X = r - Y * L.nx;
    const int link = lane < Q ? lane : 0, ax = rc(0, link), ay = rc(1, link), az = rc(2, link);
    C d[3], v[3], w[3], wxd[3], uw[3], rho[2] = {0, 0}, wl = 0;
    const SiteNbr n = site_nbr(L, X, Y, Z);
    if (link > 0 && !(az < 0 && n.wall_lo) && !(az > 0 && n.wall_hi)) {
        const int x = ax > 0 ? n.xp : (ax < 0 ? n.xm : X), y = ay > 0 ? n.yp : (ay < 0 ? n.ym : Y);
        const int z = az > 0 ? n.zp : (az < 0 ? n.zm : Z);
        const long long m = (long long)x + (long long)L.nx * ((long long)y + (long long)L.ny * z);
        const int o = L.owner[m], e = L.evt[m];
        if (o == -1 && e == 0) {
            wl = link <= 6 ? wgt<C>(1) : wgt<C>(7);
            for (int k = 0; k < 2; k++) rho[k] = node_rho<PREC, MOM>(L, m, k);
        }
    }
    particle_frame<C>(L, p, X, Y, Z, d, v, w);
    crs<C>(w, d, wxd);
    for (int m = 0; m < 3; m++) uw[m] = v[m] + wxd[m];
    C num[2] = {0, 0}, den = 0, rb[2];
#pragma unroll
    for (int i = 1; i < Q; i++) {
        const C wi = __shfl_sync(0xffffffffu, wl, i);
        for (int k = 0; k < 2; k++) num[k] += wi * __shfl_sync(0xffffffffu, rho[k], i);
        den += wi;
    }
    for (int k = 0; k < 2; k++) rb[k] = den > C(0) ? num[k] / den : C(L.P.rho0[k]);
    if (MOM) {
        if (lane == 0) {
            if (rb[0] < C(L.rlow[0]) || rb[1] < C(L.rlow[1])) note_spread(L, L.turn);
            for (int k = 0; k < 2; k++) ((C*)L.psi)[2 * s + k] = rb[k];
            for (int m = 0; m < 3; m++) ((C*)L.mom)[m * L.pstride + s] = (rb[0] + rb[1]) * uw[m];
        }
    } else if (lane < Q) {
        const C uu = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
        const C cu = C(ax) * uw[0] + C(ay) * uw[1] + C(az) * uw[2];
        const C wi = link == 0 ? wgt<C>(0) : (link <= 6 ? wgt<C>(1) : wgt<C>(7));
        S* f = (S*)L.f_cur + 2 * ((long long)link * L.pstride + SKEW + s - ax);  // pair_index
        for (int k = 0; k < 2; k++) {
            const C fe = wi * rb[k] * (C(1) + C(3) * cu + C(4.5) * cu * cu - C(1.5) * uu);
            st_pop(f + k, fe, sizeof(S) == 2 ? wi * prm<C>(L.P.rho0[k], L.PF.rho0[k]) : C(0));
        }
    }
    const C rt = rb[0] + rb[1];
    const C mom[3] = {-rt * uw[0], -rt * uw[1], -rt * uw[2]};
    C tq[3];
    crs<C>(d, mom, tq);
    if (lane < 6)
        acc_add(L, acc_slot(L, lane < 3 ? ACC_FC : ACC_TC, p, lane % 3),
                lane == 0 ? mom[0] : (lane == 1 ? mom[1] : (lane == 2 ? mom[2] : (lane == 3 ? tq[0] : (lane == 4 ? tq[1] : tq[2])))));
}

// The refill of the nodes the particles released, a warp per node: one thread
// per node took the 18 neighbours (and 19 populations of each) one after the
// other, 39 us a step at 128^3 with 801 particles against 6.
template <int PREC, bool MOM>
__global__ void __launch_bounds__(128) k_remap_create(const __grid_constant__ Lattice L) {
    chain_begin();
    const int cnt = *L.nb_chg, lane = threadIdx.x & 31;
    const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)(gridDim.x * blockDim.x >> 5);
    if (cnt <= NB_CHG_CAP) {
        for (int t = warp; t < cnt; t += nw) {
            const long long s = L.nb_chg[8 + t];
            const int code = L.evt[s];
            if ((code & 3) == 2) refill_node<PREC, MOM>(L, s, code / 4 - 1, lane);
        }
        return;
    }
    for (long long b = 32ll * warp; b < L.N; b += 32ll * nw) {
        const int code = b + lane < L.N ? L.evt[b + lane] : 0;
        for (unsigned m = __ballot_sync(0xffffffffu, (code & 3) == 2); m; m &= m - 1) {
            const int i = __ffs(m) - 1;
            refill_node<PREC, MOM>(L, b + i, __shfl_sync(0xffffffffu, code, i) / 4 - 1, lane);
        }
    }
}

// Commit the new node map.
template <int PREC, bool MOM>
__global__ void k_remap_commit(const __grid_constant__ Lattice L) {
    chain_begin();
    const int cnt = *L.nb_chg;
    const bool listed = cnt <= NB_CHG_CAP;
    const long long n = listed ? cnt : L.N;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const long long s = listed ? L.nb_chg[8 + t] : t;
        const int e = L.evt[s], p = e / 4 - 1;
        if (e == 0) continue;
        if ((e & 3) == 1) {
            int old = atomicCAS(L.owner + s, -1, p);
            if (old != -1) atomicOr(L.flags, FLAG_OVERLAP);
            L.mask[s] = 1;
            clear_moments<PREC, MOM>(L, s);
        } else if ((e & 3) == 2) {
            L.owner[s] = -1;
            L.mask[s] = 0;
        }
        L.evt[s] = 0;
    }
}

// The link-class word of site s = (x, y, z) from the owner map (NB_*); the 18
// loads are independent.
__device__ uint32_t link_classes(const Lattice& L, int x, int y, int z, long long s) {
    const SiteNbr n = site_nbr(L, x, y, z);
    int o[Q];
    o[0] = L.owner[s];
#pragma unroll
    for (int i = 1; i < Q; i++) o[i] = nbr_is_wall(n, i) ? -2 : L.owner[nbr_index(L, n, i)];
    const bool solid = o[0] >= 0;
    uint32_t bits = 0, multi = 0;
    int p0 = -1;
#pragma unroll
    for (int i = 1; i < Q; i++) {
        if (o[i] == -2) continue;
        const bool ms = o[i] >= 0;
        bits |= (uint32_t)(ms != solid) << i;
        if (!solid && ms) {
            multi |= p0 >= 0 && o[i] != p0 ? NB_MULTI : 0u;
            p0 = p0 < 0 ? o[i] : p0;
        }
    }
    return bits | multi | (solid ? NB_SOLID : 0u);
}

// every site (grid: x chunks, y, z)
__global__ void k_link_classes_all(Lattice L) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= L.nx) return;
    const long long s = (long long)x + (long long)L.nx * ((long long)y + (long long)L.ny * z);
    L.nb[s] = link_classes(L, x, y, z, s);
}

// The sites within one link of the nodes the remap changed (the map is
// final): a site next to two changed nodes is rewritten with the same word
// by both.  When more nodes changed than the list holds, every site.
__global__ void k_link_classes_changed(Lattice L) {
    chain_begin();
    const int cnt = *L.nb_chg;
    const long long nt = (long long)gridDim.x * blockDim.x;
    long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (cnt > NB_CHG_CAP) {
        for (long long s = t0; s < L.N; s += nt) {
            const long long xy = (long long)L.nx * L.ny;
            const int z = (int)(s / xy), r = (int)(s - (long long)z * xy), y = r / L.nx, x = r - y * L.nx;
            L.nb[s] = link_classes(L, x, y, z, s);
        }
        return;
    }
    for (long long t = t0; t < (long long)cnt * Q; t += nt) {
        const long long c = L.nb_chg[8 + t / Q];
        const int i = (int)(t % Q);
        const long long xy = (long long)L.nx * L.ny;
        const int z = (int)(c / xy), r = (int)(c - (long long)z * xy), y = r / L.nx, x = r - y * L.nx;
        const SiteNbr n = site_nbr(L, x, y, z);
        if (i > 0 && nbr_is_wall(n, i)) continue;
        int X = x, Y = y, Z = z;
        if (i > 0) {
            X = rc(0, i) > 0 ? n.xp : (rc(0, i) < 0 ? n.xm : x);
            Y = rc(1, i) > 0 ? n.yp : (rc(1, i) < 0 ? n.ym : y);
            Z = rc(2, i) > 0 ? n.zp : (rc(2, i) < 0 ? n.zm : z);
        }
        const long long s = (long long)X + (long long)L.nx * ((long long)Y + (long long)L.ny * Z);
        L.nb[s] = link_classes(L, X, Y, Z, s);
    }
}

// ------------------------------------------------------------ wetting
// Eq. 20 on every frontier node s (a particle node with at least one fluid
// neighbour): psi^k(s) = (1 + zeta^k) sum w_i rho^k / sum w_i over the fluid
// neighbours (with the Janus switch s of the node: 1 + s zeta^A, 1 - s zeta^B)
// neighbours, and Eq. 21 (repulsive sign):
// F_s = -G sum_k psi^k(s) sum w_i rho^kbar(s + c_i) c_i, added with its torque
// (x_s - r_p) x F_s to the fixed-point sums F_s, T_s of the owning particle
// (zero at the start of the step).  The link classes of a particle node are
// the links to its fluid neighbours, so a block reads the link classes of a
// 32 x 8 tile for a chunk of planes (4 bytes a site), packs the frontier nodes
// onto consecutive threads, and each thread gathers the densities of its
// node's fluid neighbours (a third of the 18), which are those of the fluid
// nodes at this time.  It is bound by the latency of these gathers and by
// issue (55 %).  (Copying psi and the owner map of the tile and its ring to
// shared memory instead moved 20 bytes a site for the 6 % of the sites that
// are frontier nodes: 512 x 512 x 256, 14,444 particles, 530 us against 298
// now; 96^3 FP64 115 against 88, with sums in integer weights.)
constexpr int VTX = 32, VTY = 8, VZC = 16;  // tile and planes per block (4096 sites: 12 bits of an entry)

template <int PREC>
__global__ void __launch_bounds__(VTX* VTY) k_virtual(const __grid_constant__ Lattice L, int store_terms, int zc) {
    chain_begin();
    typedef typename Prec<PREC>::C C;
    struct alignas(2 * sizeof(C)) Pair {
        C a, b;
    };
    constexpr int NT = VTX * VTY;
    __shared__ unsigned cand[NT * VZC];  // link bits 1..18 above the site's place in the tile
    __shared__ int wcnt[NT / 32];

    const int x0 = blockIdx.x * VTX, y0 = blockIdx.y * VTY;
    const int W = min(VTX, L.nx - x0), H = min(VTY, L.ny - y0);
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, L.nz), nz_b = z1 - z0;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * VTX + tx, lane = tid & 31, warp = tid >> 5;
    const bool act = tx < W && ty < H;
    const long long nxy = (long long)L.nx * L.ny;
    C* psi = (C*)L.psi;
    const int own_xy = act ? x0 + tx + L.nx * (y0 + ty) : 0;
    // the frontier nodes of the tile's own column (a particle node with a
    // fluid neighbour: its link classes), one bit per plane of the chunk
    unsigned front = 0;
    uint32_t c[VZC];
#pragma unroll
    for (int q = 0; q < VZC; q++) c[q] = act && q < nz_b ? L.nb[nxy * (z0 + q) + own_xy] : 0u;
    {
#pragma unroll
        for (int q = 0; q < VZC; q++) front |= (unsigned)((c[q] & NB_SOLID) && (c[q] & NB_LINKS)) << q;
    }
    // the frontier nodes of the chunk, packed onto consecutive threads (in
    // plane, warp and lane order: fixed by the geometry)
    const int mine = __popc(front);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wcnt[warp] = incl;
    __syncthreads();
    int off = incl - mine, tot = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; w++) {
        off += w < warp ? wcnt[w] : 0;
        tot += wcnt[w];
    }
#pragma unroll
    for (int q = 0; q < VZC; q++)
        if ((front >> q) & 1u) cand[off++] = (c[q] & NB_LINKS) << 12 | (unsigned)(q * NT + tid);
    __syncthreads();
    const C G36 = -prm<C>(L.P.G, L.PF.G) / C(36), zA = C(1) + C(L.P.zeta[0]), zB = C(1) + C(L.P.zeta[1]);
    // whole warps step through the list together (lanes past its end carry
    // no term) for the sums over runs of lanes
    for (int base = warp * 32; base < tot; base += NT) {
        const int k = base + lane;
        bool has = false;
        int p = -1;
        C fs[3] = {0, 0, 0}, tq[3] = {0, 0, 0};
        if (k < tot) {
            const unsigned e = cand[k], fluid = e >> 12;
            const int q = (int)(e & 4095u) / NT, t = (int)(e & 4095u) % NT, x = x0 + t % VTX, y = y0 + t / VTX, z = z0 + q;
            const unsigned s = (unsigned)(x + L.nx * y) + (unsigned)nxy * (unsigned)z;
            p = L.owner[s];
            const int nxi = L.nx, pl = (int)nxy;
            const int dxp = x == nxi - 1 ? 1 - nxi : 1, dxm = x == 0 ? nxi - 1 : -1;
            const int dyp = y == L.ny - 1 ? nxi - pl : nxi, dym = y == 0 ? pl - nxi : -nxi;
            const int dzp = z == L.nz - 1 ? pl - (int)L.N : pl, dzm = z == 0 ? (int)L.N - pl : -pl;
            Pair r[Q];
#pragma unroll
            for (int i = 1; i < Q; i++) {
                const int o = (cx(i) > 0 ? dxp : (cx(i) < 0 ? dxm : 0)) + (cy(i) > 0 ? dyp : (cy(i) < 0 ? dym : 0)) +
                              (cz(i) > 0 ? dzp : (cz(i) < 0 ? dzm : 0));
                r[i] = Pair{C(0), C(0)};
                if ((fluid >> i) & 1u) r[i] = reinterpret_cast<const Pair*>(psi)[s + (unsigned)o];
            }
            // sums in units of 1/36 (weights 2 and 1)
            C num[2] = {0, 0};
            C sA[3] = {0, 0, 0}, sB[3] = {0, 0, 0};
#pragma unroll
            for (int i = 1; i < Q; i++) {
                const C ra = i <= 6 ? C(2) * r[i].a : r[i].a, rb = i <= 6 ? C(2) * r[i].b : r[i].b;
                num[0] += ra;
                num[1] += rb;
                if (cx(i)) sA[0] += C(cx(i)) * ra, sB[0] += C(cx(i)) * rb;
                if (cy(i)) sA[1] += C(cy(i)) * ra, sB[1] += C(cy(i)) * rb;
                if (cz(i)) sA[2] += C(cz(i)) * ra, sB[2] += C(cz(i)) * rb;
            }
            const C den = C(2 * __popc(fluid & 0x7eu) + __popc(fluid & 0x7ff80u));
            if (den > C(0)) {
                C d[3];
                // x_s - r_p (minimum image) from the integer cell and offset of r_p
                const int xs[3] = {x, y, z}, Ls[3] = {L.nx, L.ny, L.nz};
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    int ip;
                    C fr;
                    if (sizeof(C) == 8) {
                        double r = L.pos[3 * p + c];
                        ip = (int)floor(r);
                        fr = C(r - (double)ip);
                    } else {
                        ip = L.ipos[3 * p + c];
                        fr = C(L.fsnap[9 * p + c]);
                    }
                    int dd = xs[c] - ip;
                    if (L.per[c]) {
                        if (2 * dd > Ls[c]) dd -= Ls[c];
                        else if (2 * dd < -Ls[c]) dd += Ls[c];
                    }
                    d[c] = C(dd) - fr;
                }
                C fa = zA, fb = zB;
                if (L.P.janus) {
                    const C sw = janus_switch<C>(L, p, d);
                    fa = C(1) + sw * C(L.P.zeta[0]);
                    fb = C(1) - sw * C(L.P.zeta[1]);
                }
                const C iden = C(1) / den, pa = fa * (num[0] * iden);
                const C pb = fb * (num[1] * iden);
                reinterpret_cast<Pair*>(psi)[s] = Pair{pa, pb};
                if (store_terms) {
#pragma unroll
                    for (int c = 0; c < 3; c++) fs[c] = G36 * (pa * sB[c] + pb * sA[c]);
                    crs<C>(d, fs, tq);
                    has = true;
                }
            }
        }
        if (!store_terms) continue;  // uniform across the block
        add_runs(L, ACC_FS, has ? p : -1, fs, tq);
    }
}

// -------------------------------------------------------- pair forces
// Eq. 26 (Hertz, repulsive, r floored at r_cap) and Eq. 27 (lubrication) on
// particle i due to j, in FP64.
__device__ void pair_force(const Lattice& L, int i, int j, const double (&ri)[3], double Ri,
                           const double (&vi)[3], double nu, double (&fo)[3]) {
    double rij[3];
    for (int d = 0; d < 3; d++) {
        double dd = L.pos[3 * j + d] - ri[d];
        if (L.per[d]) {
            double Ld = (d == 0 ? L.nx : (d == 1 ? L.ny : L.nz));
            dd -= Ld * floor(dd / Ld + 0.5);
        }
        rij[d] = dd;
    }
    fo[0] = fo[1] = fo[2] = 0.0;
    double r = sqrt(rij[0] * rij[0] + rij[1] * rij[1] + rij[2] * rij[2]);
    if (!(r > 0.0)) return;
    if (L.P.hertz_K != 0.0 && r < L.P.hertz_sigma) {
        double rr = r < L.P.hertz_rcap ? L.P.hertz_rcap : r;
        double mag = 2.5 * L.P.hertz_K * pow(L.P.hertz_sigma - rr, 1.5);
        for (int d = 0; d < 3; d++) fo[d] += -mag * rij[d] / r;
    }
    if (L.P.lub_on) {
        double Rj = L.rad[j];
        double h = r - (Ri + Rj);
        if (h < L.P.lub_hn) {
            double red = Ri * Rj / (Ri + Rj), vr = 0.0;
            if (h < L.P.lub_hmin) h = L.P.lub_hmin;
            for (int d = 0; d < 3; d++) vr += (vi[d] - L.vel[3 * j + d]) * rij[d] / r;
            double mag = -6.0 * 3.14159265358979323846 * nu * L.P.lub_scale * red * red *
                         (1.0 / h - 1.0 / L.P.lub_hn) * vr;
            for (int d = 0; d < 3; d++) fo[d] += mag * rij[d] / r;
        }
    }
}

struct CellGrid {
    int n[3];         // cells per axis (>= 3 each when used)
    float inv[3];     // cells per lattice unit
    int* count;       // [ncell] counts, reused as fill cursors
    int* start;       // [ncell + 1]
    int* items;       // [nc]
};

__device__ __forceinline__ int cell_coord(float x, float inv, int n) {
    int c = (int)(x * inv);
    return c < 0 ? 0 : (c >= n ? n - 1 : c);
}

// The cell list serves the pair-list build: the cell kernels do nothing in a
// step that keeps the list (flag clear).
__global__ void k_cells_count(Lattice L, CellGrid cg) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= L.nc || !*L.vl_flag) return;
    int c0 = cell_coord(float(L.pos[3 * p]), cg.inv[0], cg.n[0]);
    int c1 = cell_coord(float(L.pos[3 * p + 1]), cg.inv[1], cg.n[1]);
    int c2 = cell_coord(float(L.pos[3 * p + 2]), cg.inv[2], cg.n[2]);
    atomicAdd(cg.count + (c0 + cg.n[0] * (c1 + cg.n[1] * c2)), 1);
}

// exclusive scan of the counts (one block); counts are reset to serve as cursors
__global__ void __launch_bounds__(1024) k_cells_scan(CellGrid cg, const int* flag) {
    if (!*flag) return;
    __shared__ int part[1024];
    int nc = cg.n[0] * cg.n[1] * cg.n[2];
    int per = (nc + 1023) / 1024;
    int b = threadIdx.x * per, e = min(nc, b + per);
    int sum = 0;
    for (int c = b; c < e; c++) sum += cg.count[c];
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        int v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = part[threadIdx.x] - sum;
    for (int c = b; c < e; c++) {
        cg.start[c] = run;
        run += cg.count[c];
        cg.count[c] = 0;
    }
    if (threadIdx.x == 1023) cg.start[nc] = part[1023];
}

__global__ void k_cells_fill(Lattice L, CellGrid cg) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= L.nc || !*L.vl_flag) return;
    int c0 = cell_coord(float(L.pos[3 * p]), cg.inv[0], cg.n[0]);
    int c1 = cell_coord(float(L.pos[3 * p + 1]), cg.inv[1], cg.n[1]);
    int c2 = cell_coord(float(L.pos[3 * p + 2]), cg.inv[2], cg.n[2]);
    int c = c0 + cg.n[0] * (c1 + cg.n[1] * c2);
    cg.items[cg.start[c] + atomicAdd(cg.count + c, 1)] = p;
}

// Pair list (App. A rcut / delr): a particle's neighbours within the list
// radius rl = max(rcut, interaction range) + delr, sorted by index, are kept
// until some particle has moved more than delr / 2 since the build; the pair
// forces then reach only listed pairs.  Every pair within the interaction
// range at any step before the next build was within rl at the build.
__global__ void k_pair_check(Lattice L, double half_skin) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= L.nc) return;
    double d2 = 0.0;
    for (int d = 0; d < 3; d++) {
        double dd = L.pos[3 * p + d] - L.vl_ref[3 * p + d];
        if (L.per[d]) {
            double Ld = (d == 0 ? L.nx : (d == 1 ? L.ny : L.nz));
            dd -= Ld * floor(dd / Ld + 0.5);
        }
        d2 += dd * dd;
    }
    if (!(d2 <= half_skin * half_skin)) atomicOr(L.vl_flag, 1);
}

// Build the list of particle i (when the flag is set): candidates from the 27
// neighbouring cells, or among all particles when the grid has fewer than 3
// cells along an axis; more than PAIR_LIST_MAX neighbours is reported as an
// overlap.
__global__ void __launch_bounds__(128) k_pair_list(Lattice L, CellGrid cg, int use_cells, float rl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.nc || !*L.vl_flag) return;
    if (i == 0) atomicAdd(L.vl_builds, 1ull);
    float rif[3];
    for (int d = 0; d < 3; d++) {
        L.vl_ref[3 * i + d] = L.pos[3 * i + d];
        rif[d] = float(L.pos[3 * i + d]);
    }
    float Lf[3] = {float(L.nx), float(L.ny), float(L.nz)};
    float iLf[3] = {1.f / Lf[0], 1.f / Lf[1], 1.f / Lf[2]};
    int* cand = L.vl_nb + (size_t)i * PAIR_LIST_MAX;
    int nc = 0;
    auto test = [&](int j) {
        if (j == i) return;
        float r2 = 0.f;
        for (int d = 0; d < 3; d++) {
            float df = float(L.pos[3 * j + d]) - rif[d];
            if (L.per[d]) df -= Lf[d] * rintf(df * iLf[d]);
            r2 += df * df;
        }
        if (r2 >= rl * rl) return;
        if (nc < PAIR_LIST_MAX) {
            // insertion keeps the list sorted by j
            int q = nc++;
            while (q > 0 && cand[q - 1] > j) {
                cand[q] = cand[q - 1];
                q--;
            }
            cand[q] = j;
        } else {
            atomicOr(L.flags, FLAG_OVERLAP);
        }
    };
    if (rl > 0.f) {
        if (use_cells) {
            int c0 = cell_coord(rif[0], cg.inv[0], cg.n[0]);
            int c1 = cell_coord(rif[1], cg.inv[1], cg.n[1]);
            int c2 = cell_coord(rif[2], cg.inv[2], cg.n[2]);
            for (int dz = -1; dz <= 1; dz++) {
                int z = c2 + dz;
                if (z < 0 || z >= cg.n[2]) {
                    if (!L.per[2]) continue;
                    z = (z + cg.n[2]) % cg.n[2];
                }
                for (int dy = -1; dy <= 1; dy++) {
                    int y = (c1 + dy + cg.n[1]) % cg.n[1];
                    for (int dx = -1; dx <= 1; dx++) {
                        int x = (c0 + dx + cg.n[0]) % cg.n[0];
                        int c = x + cg.n[0] * (y + cg.n[1] * z);
                        for (int q = cg.start[c]; q < cg.start[c + 1]; q++) test(cg.items[q]);
                    }
                }
            }
        } else {
            for (int j = 0; j < L.nc; j++) test(j);
        }
    }
    L.vl_cnt[i] = nc;
}

// Pair forces on particle i summed over its listed neighbours in index
// order, plus the soft side walls.
__global__ void __launch_bounds__(128) k_pairs(Lattice L) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.nc) return;
    double ri[3], vi[3];
    for (int d = 0; d < 3; d++) {
        ri[d] = L.pos[3 * i + d];
        vi[d] = L.vel[3 * i + d];
    }
    double Ri = L.rad[i];
    double nu = 0.5 * ((L.P.tau[0] - 0.5) / 3.0 + (L.P.tau[1] - 0.5) / 3.0);
    NSum acc[3] = {{0, 0}, {0, 0}, {0, 0}};
    const int n = L.vl_cnt[i];
    const int* nb = L.vl_nb + (size_t)i * PAIR_LIST_MAX;
    for (int q = 0; q < n; q++) {
        double fo[3];
        pair_force(L, i, nb[q], ri, Ri, vi, nu, fo);
        for (int d = 0; d < 3; d++) acc[d].add(fo[d]);
    }
    if (!L.per[2] && L.P.side_wall_k != 0.0) {
        double hlo = ri[2] + 0.5, hhi = (double(L.nz) - 0.5) - ri[2];
        if (hlo < L.P.side_wall_d) acc[2].add(L.P.side_wall_k * (L.P.side_wall_d - hlo));
        if (hhi < L.P.side_wall_d) acc[2].add(-L.P.side_wall_k * (L.P.side_wall_d - hhi));
    }
    for (int d = 0; d < 3; d++) L.Fpair[3 * i + d] = acc[d].value();
}

// --------------------------------------------------------- integrator
// Eq. 35 totals, Eq. 32 leap-frog, Eqs. 33-34 quaternions; then the FP32
// snapshot of the new state.  A particle faster than 1/2 lattice unit along an axis
// is reported (the remap assumes smaller moves).  The step's fixed-point sums
// are read and cleared for the next step, and the list of changed nodes
// emptied.
//
// Eq. 33 is qdot = q (0, w*) / 2 with the body-frame w* = R(q/|q|)^T w, which
// is (0, w) q / 2 with w in the space frame, linear in q, so the implicit
// mid-step equation of Eq. 34, qdot = (0, w) (q + qdot / 2) / 2, has the closed
// form qdot = ((0, w) q / 2 - w.w q / 8) / (1 + w.w / 16), the fixed point of
// the iteration that Eq. 34 prescribes.  (Iterated, with two roots and eight
// divisions in FP64 each time: 40 us a step whatever the number of particles,
// FP64 running two lanes a cycle on an SM; one thread per particle took 11 us,
// four lanes, one per axis and component of the quaternion, take 8.6 us with 801
// particles, and 14.7 instead of 23 with 14,444.)
__global__ void __launch_bounds__(32) k_integrate(const __grid_constant__ Lattice L) {
    chain_begin();
    const int t = blockIdx.x * blockDim.x + threadIdx.x, d = t & 3, a = d < 3 ? d : 0, p = min(t >> 2, L.nc - 1);
    const bool live = (t >> 2) < L.nc, axis = live && d < 3;
    const unsigned all = 0xffffffffu;
    if (t == 0) *L.nb_chg = 0;
    const int i = 3 * p + a;
    double term[ACC_TERMS];
#pragma unroll
    for (int k = 0; k < ACC_TERMS; k++) term[k] = acc_value(L, acc_slot(L, k, p, a));
    const bool first = !L.prev_valid[p];
    const double Fp = first ? term[ACC_FLIQ] : L.Fliq_prev[i], Tp = first ? term[ACC_TLIQ] : L.Tliq_prev[i];
    const double im = 1.0 / L.mass[p], R = L.rad[p];
    double v = L.vel[i], r = L.pos[i], w = L.omg[i], q = L.quat[4 * p + d];
    const double F = 0.5 * (Fp + term[ACC_FLIQ]) + term[ACC_FD] + term[ACC_FC] + term[ACC_FS] + L.Fpair[i];
    const double T = 0.5 * (Tp + term[ACC_TLIQ]) + term[ACC_TD] + term[ACC_TC] + term[ACC_TS];
    const int n = a == 0 ? L.nx : (a == 1 ? L.ny : L.nz);
    v += F * im;
    r += v;
    if (L.per[a] && !(r >= 0.0 && r < (double)n)) r = r - (double)n * floor(r / (double)n);
    __syncwarp(all);  // every lane has read the sums and prev_valid
    if (axis) {
        double* terms[ACC_TERMS] = {L.Fliq, L.Tliq, L.Fd, L.Td, L.Fc, L.Tc, L.Fs, L.Ts};
#pragma unroll
        for (int k = 0; k < ACC_TERMS; k++) {
            unsigned long long* slot = acc_slot(L, k, p, a);
            slot[0] = slot[1] = 0ull;
            terms[k][i] = term[k];
        }
        L.Ftot[i] = F;
        L.Ttot[i] = T;
        L.Fliq_prev[i] = term[ACC_FLIQ];
        L.Tliq_prev[i] = term[ACC_TLIQ];
        L.vel[i] = v;
        L.pos[i] = r;
        if (!(fabs(v) < 0.5)) atomicOr(L.flags, FLAG_NONFINITE);
        if (a == 0) L.prev_valid[p] = 1;
    }
    if (L.P.rotate) {
        w += T * (im / (0.4 * R * R));
        const double w0 = __shfl_sync(all, w, 0, 4), w1 = __shfl_sync(all, w, 1, 4), w2 = __shfl_sync(all, w, 2, 4);
        const double q0 = __shfl_sync(all, q, 0, 4), q1 = __shfl_sync(all, q, 1, 4), q2 = __shfl_sync(all, q, 2, 4),
                     q3 = __shfl_sync(all, q, 3, 4);
        const double ww = w0 * w0 + w1 * w1 + w2 * w2;
        // component d of (0, w) q
        const double x = d == 0 ? -w0 : (d == 1 ? w0 : (d == 2 ? w1 : w2));
        const double y = d == 0 ? -w1 : (d == 1 ? w1 : (d == 2 ? w2 : w0));
        const double z = d == 0 ? -w2 : (d == 1 ? -w2 : (d == 2 ? -w0 : -w1));
        const double wq = x * (d == 0 ? q1 : q0) + y * (d == 1 ? q3 : (d == 2 ? q1 : q2)) +
                          z * (d == 0 || d == 2 ? q3 : (d == 1 ? q2 : q1));
        q += (0.5 * wq - 0.125 * ww * q) / (1.0 + 0.0625 * ww);
        double nq = q * q;
        nq += __shfl_xor_sync(all, nq, 1, 4);
        nq += __shfl_xor_sync(all, nq, 2, 4);
        q = q / sqrt(nq);
        if (axis) L.omg[i] = w;
        if (live) L.quat[4 * p + d] = q;
    }
    if (axis) {
        const int ip = (int)floor(r);
        L.ipos[i] = ip;
        L.fsnap[9 * p + a] = float(r - (double)ip);
        L.fsnap[9 * p + 3 + a] = float(v);
        L.fsnap[9 * p + 6 + a] = float(w);
    }
}

// ---------------------------------------------------------- launchers
#define DISPATCHC(prec, call)                                 \
    switch (prec) {                                           \
        case LB_FP64: { const int P = LB_FP64; call; break; } \
        case LB_FP32: { const int P = LB_FP32; call; break; } \
        default:      { const int P = LB_FP16; call; break; } \
    }

static const dim3 PBLK(BXP, BYP);

int launch_snapshot(const Lattice& L, cudaStream_t st) {
    if (L.nc <= 0) return 0;
    k_snapshot<<<(L.nc + 127) / 128, 128, 0, st>>>(L);
    return 1;
}

int launch_map_initial(const Lattice& L, int prec, int first, int count, cudaStream_t st) {
    if (count <= 0) return 0;
    DISPATCHC(prec, (k_map_initial<P><<<count, PBLK, 0, st>>>(L, first)));
    return 1;
}

template <int P, bool MOM>
static void launch_remap_t(const Lattice& L, bool wide, cudaStream_t st) {
    k_remap_classify<P, MOM><<<L.nc, PBLK, 0, st>>>(L, wide);
    launch_after(k_remap_create<P, MOM>, (unsigned)(16 * device_sms()), 128, 0, st, L);
    launch_after(k_remap_commit<P, MOM>, (unsigned)(2 * device_sms()), 128, 0, st, L);
}

int launch_clear_terms(const Lattice& L, cudaStream_t st) {
    if (L.nc <= 0) return 0;
    cudaMemsetAsync(L.acc, 0, (size_t)ACC_TERMS * L.maxc * 6 * sizeof(unsigned long long), st);
    cudaMemsetAsync(L.nb_chg, 0, sizeof(int), st);
    return 0;
}

int launch_remap(const Lattice& L, int prec, bool moments, bool wide, cudaStream_t st) {
    if (L.nc <= 0) return 0;
    if (moments) {
        DISPATCHC(prec, (launch_remap_t<P, true>(L, wide, st)));
    } else {
        DISPATCHC(prec, (launch_remap_t<P, false>(L, wide, st)));
    }
    return 3;
}

int launch_link_classes(const Lattice& L, bool full, cudaStream_t st) {
    if (full) {
        const int bx = L.nx >= 128 ? 128 : ((L.nx + 31) / 32) * 32;
        k_link_classes_all<<<dim3((unsigned)((L.nx + bx - 1) / bx), (unsigned)L.ny, (unsigned)L.nz), bx, 0, st>>>(L);
    } else {
        launch_after(k_link_classes_changed, (unsigned)(4 * device_sms()), 256, 0, st, L);
    }
    return 1;
}

int launch_virtual(const Lattice& L, int prec, int store_terms, cudaStream_t st) {
    if (L.nc <= 0) return 0;
    // full chunks where the lattice has blocks for all SMs several times over,
    // thinner ones where it has not (32^3: 10.4 us with two chunks, 7.4 with 16)
    const long long tiles = (long long)((L.nx + VTX - 1) / VTX) * ((L.ny + VTY - 1) / VTY);
    const long long zw = tiles * L.nz / (4 * device_sms());
    const int zc = (int)(zw < 2 ? 2 : (zw > VZC ? VZC : zw));
    dim3 grid((L.nx + VTX - 1) / VTX, (L.ny + VTY - 1) / VTY, (L.nz + zc - 1) / zc);
    DISPATCHC(prec, (launch_after(k_virtual<P>, grid, dim3(VTX, VTY), 0, st, L, store_terms, zc)));
    return 1;
}

int launch_pairs(const Lattice& L, void* cells, size_t cell_cap, bool force_build, cudaStream_t st) {
    if (L.nc <= 0) return 0;
    // interaction range: Hertz contact, and lubrication up to 2 R_max + h_n
    double rc = L.P.hertz_K != 0.0 ? L.P.hertz_sigma : 0.0;
    if (L.P.lub_on) rc = fmax(rc, 2.0 * L.rmax + L.P.lub_hn);
    if (rc > 0.0) rc = fmax(rc, L.P.rcut);
    float rl = rc > 0.0 ? float(rc + L.P.delr) + 0.05f : 0.f;
    CellGrid cg;
    int Ls[3] = {L.nx, L.ny, L.nz};
    long long ncell = 1;
    int use_cells = rl > 0.f && L.nc > 64;
    for (int d = 0; d < 3; d++) {
        int n = rl > 0.f ? (int)(Ls[d] / rl) : 1;
        if (n > 64) n = 64;
        if (n < 3) use_cells = 0;
        cg.n[d] = n < 1 ? 1 : n;
        cg.inv[d] = float(cg.n[d]) / float(Ls[d]);
        ncell *= cg.n[d];
    }
    if ((size_t)(2 * ncell + 1 + L.nc) * sizeof(int) > cell_cap) use_cells = 0;
    int n = 0;
    cg.count = (int*)cells;
    cg.start = cg.count + ncell;
    cg.items = cg.start + ncell + 1;
    // rebuild flag: forced (new particles or parameters, or no skin), else
    // set by the particles that moved more than delr / 2
    const bool every_step = force_build || !(L.P.delr > 0.0);
    cudaMemsetAsync(L.vl_flag, every_step ? 0xff : 0, sizeof(int), st);
    if (!every_step) {
        k_pair_check<<<(L.nc + 127) / 128, 128, 0, st>>>(L, 0.5 * L.P.delr);
        n++;
    }
    if (use_cells) {
        cudaMemsetAsync(cg.count, 0, ncell * sizeof(int), st);
        k_cells_count<<<(L.nc + 127) / 128, 128, 0, st>>>(L, cg);
        k_cells_scan<<<1, 1024, 0, st>>>(cg, L.vl_flag);
        k_cells_fill<<<(L.nc + 127) / 128, 128, 0, st>>>(L, cg);
        n += 3;
    }
    k_pair_list<<<(L.nc + 127) / 128, 128, 0, st>>>(L, cg, use_cells, rl);
    k_pairs<<<(L.nc + 127) / 128, 128, 0, st>>>(L);
    return n + 2;
}

int launch_integrate(const Lattice& L, cudaStream_t st) {
    if (L.nc <= 0) return 0;
    k_integrate<<<(L.nc + 7) / 8, 32, 0, st>>>(L);
    return 1;
}

}  // namespace lbgb
