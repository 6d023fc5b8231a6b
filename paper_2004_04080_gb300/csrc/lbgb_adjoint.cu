// lbgb_adjoint.cu -- reverse mode of the lattice step for fixed particles.
//
// With the particles held fixed (infinite mass, zero velocity) the node map
// is static and the time step is a smooth map f(t) -> f(t+1) of the
// populations with parameters tau_A, tau_B, G, zeta_A, zeta_B.  Its adjoint
// takes lambda(t+1) = dJ/df(t+1) to lambda(t) = dJ/df(t) and accumulates the
// parameter gradients.  The forward quantities of step t are recomputed from
// the stored populations f(t) (the caller keeps sqrt(N) checkpoints and
// re-runs each segment).
//
// An adjoint field is stored as lambda_i(x) = L_i(x) + R(x): 2 x 19 local
// values L and a per-site, per-component scalar R added to every link (the
// density adjoint arriving through the Shan-Chen halo), so the non-local part
// costs 2 values per site instead of 38.  Layout in the compute type:
// [L: 2][19][pstride] then [R: 2][pstride].
//
// Forward map at a fluid site x (Sec. 2.3, Eqs. 5-7, 11, 13-16, with the
// readings of the forward kernels):
//   rho^k = sum f^k_i, j^k = sum f^k_i c_i
//   S^k = sum_i w_i psi^k(x + c_i) c_i,  F^A = -G rho^A S^B + rho^A g (A<->B)
//   u = (om_A j^A + om_B j^B) / (om_A rho^A + om_B rho^B), om_k = 1/tau_k
//   om = 1/(3 nubar + 1/2), 1/nubar = sum_k (rho^k/rho)/nu_k, nu_k = (tau_k - 1/2)/3
//   v^k = u + F^k/rho^k
//   f*^k_i = (1 - om)(f^k_i - E_i(rho^k, u)) + E_i(rho^k, v^k)
//   push to x + c_i, or bounce back (Eqs. 8, 9, 17 with u_w = 0 on particles)
// psi is rho on fluid nodes, the virtual density (Eq. 20) on particle frontier
// nodes and the wall density beyond walls; the link forces of Eq. 19 are
// F_p = sum_links sum_k 2 f*^k_i c_i.
#include "lbgb_internal.cuh"

namespace lbgb {

constexpr int ADJ_VALUES = 5;  // dJ/d tau_A, tau_B, G, zeta_A, zeta_B

struct AdjArgs {
    const void* adj_in;   // lambda(t+1)
    void* adj_out;        // lambda(t)
    void* sbar;           // [2][3][N]: adjoint of S^k at fluid sites
    void* coef;           // [2][N]: per particle node, dJ/dpsi (1+zeta)/W
    void* coef_wall;      // [2 walls][2][nx ny]
    const double* dJdF;   // [nc][3] dJ/dF_liq of this step (device) or null
    double* red;          // block partials [blocks][ADJ_VALUES][2]
};

// weighted moments of an adjoint vector mu over the lattice:
// m0 = sum w mu, m1 = sum w mu c, m2 = sum w mu c c^T (xx, yy, zz, xy, xz, yz)
template <typename C>
struct Mom {
    C m0, m1[3], m2[6];
};

template <typename C>
__device__ __forceinline__ void moments_of(const C (&mu)[Q], Mom<C>& M) {
    // by opposite pairs, no products by the zeros of c_i: 60 operations (200
    // link by link)
    C ax = 0, dg = 0, sd[6] = {0, 0, 0, 0, 0, 0}, sa[3], da[3], dd[3] = {0, 0, 0};
#pragma unroll
    for (int i = 1; i < Q; i += 2) {  // opp(i) = i + 1
        const C sum = mu[i] + mu[i + 1], dif = mu[i] - mu[i + 1];
        const int c[3] = {cx(i), cy(i), cz(i)};
        if (i <= 6) {
            ax += sum;
            const int d = c[0] ? 0 : (c[1] ? 1 : 2);
            sa[d] = sum;
            da[d] = c[d] > 0 ? dif : -dif;
            continue;
        }
        dg += sum;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (c[d] > 0) dd[d] += dif;
            if (c[d] < 0) dd[d] -= dif;
            if (c[d] != 0) sd[d] += sum;
        }
        const int q = c[2] == 0 ? 3 : (c[1] == 0 ? 4 : 5);  // xy, xz, yz
        const int sign = (c[0] ? c[0] : c[1]) * (c[2] ? c[2] : c[1]);
        if (sign > 0) sd[q] += sum; else sd[q] -= sum;
    }
    const C w0 = wgt<C>(0), w1 = wgt<C>(1), w2 = wgt<C>(7);
    M.m0 = w0 * mu[0] + (w1 * ax + w2 * dg);
#pragma unroll
    for (int d = 0; d < 3; d++) {
        M.m1[d] = w1 * da[d] + w2 * dd[d];
        M.m2[d] = w1 * sa[d] + w2 * sd[d];
        M.m2[3 + d] = w2 * sd[3 + d];
    }
}

// sum_i mu_i E_i(rho,u)/rho = m0 + 3 m1.u + 9/2 u^T m2 u - 3/2 u.u m0
template <typename C>
__device__ __forceinline__ C mom_shape(const Mom<C>& M, const C (&u)[3]) {
    C uMu = M.m2[0] * u[0] * u[0] + M.m2[1] * u[1] * u[1] + M.m2[2] * u[2] * u[2] +
            C(2) * (M.m2[3] * u[0] * u[1] + M.m2[4] * u[0] * u[2] + M.m2[5] * u[1] * u[2]);
    C uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    return M.m0 + C(3) * (M.m1[0] * u[0] + M.m1[1] * u[1] + M.m1[2] * u[2]) + C(4.5) * uMu - C(1.5) * uu * M.m0;
}

// sum_i mu_i dE_i(rho,u)/du / rho = 3 m1 + 9 m2 u - 3 u m0
template <typename C>
__device__ __forceinline__ void mom_grad(const Mom<C>& M, const C (&u)[3], C (&g)[3]) {
    C m2u0 = M.m2[0] * u[0] + M.m2[3] * u[1] + M.m2[4] * u[2];
    C m2u1 = M.m2[3] * u[0] + M.m2[1] * u[1] + M.m2[5] * u[2];
    C m2u2 = M.m2[4] * u[0] + M.m2[5] * u[1] + M.m2[2] * u[2];
    g[0] = C(3) * M.m1[0] + C(9) * m2u0 - C(3) * u[0] * M.m0;
    g[1] = C(3) * M.m1[1] + C(9) * m2u1 - C(3) * u[1] * M.m0;
    g[2] = C(3) * M.m1[2] + C(9) * m2u2 - C(3) * u[2] * M.m0;
}

// sums over the block of NV doubles per thread, thread 0 writing value v to
// out[v * stride] (warp shuffles, then warps in order; blockDim.x a multiple of 32)
template <int NV>
__device__ __forceinline__ void block_sum_store(double (&v)[NV], double* out, long long stride) {
    __shared__ double sh[NV][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int m = 0; m < NV; m++)
        for (int off = 16; off > 0; off >>= 1) v[m] += __shfl_down_sync(0xffffffffu, v[m], off);
    if (lane == 0)
#pragma unroll
        for (int m = 0; m < NV; m++) sh[m][warp] = v[m];
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += sh[threadIdx.x][w];
        out[threadIdx.x * stride] = t;
    }
}

// Local adjoint of the collision and streaming at each fluid site.
template <int PREC>
__global__ void __launch_bounds__(128, (PREC == LB_FP64 ? 2 : 4)) k_adj_local(Lattice L, AdjArgs A) {
    typedef typename Prec<PREC>::S S;
    typedef typename Prec<PREC>::C C;
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y, z = blockIdx.z;
    C part[3] = {0, 0, 0};
    long long s = (long long)x + (long long)L.nx * ((long long)y + (long long)L.ny * z);
    const C* Lin = (const C*)A.adj_in;
    const C* Rin = Lin + 2 * Q * L.pstride;
    C* Lout = (C*)A.adj_out;
    C* sb = (C*)A.sbar;
    const uint32_t nbc = x < L.nx ? L.nb[s] : NB_SOLID;
    if (!(nbc & NB_SOLID)) {
        SiteNbr n = site_nbr(L, x, y, z);
        C fv[2][Q], rho[2], j[2][3], u[3], om;
        load_site<PREC>(L, (const S*)L.f_cur, s, fv, rho, j);
        // F^A / rho^A = g - G S^B and F^B / rho^B = g - G S^A (acc), 36 S in grad
        C grad[2][3], acc[2][3];
        {
            const C* psi = (const C*)L.psi;
            const C* pw = (const C*)L.psi_wall;
            const long long nxy = (long long)L.nx * L.ny;
            C ps[Q][2];
#pragma unroll
            for (int i = 1; i < Q; i++) {
                const C* q = psi;
                long long m;
                if (nbr_is_wall(n, i)) {
                    const int X = cx(i) == 0 ? n.x : (cx(i) > 0 ? n.xp : n.xm);
                    const int Y = cy(i) == 0 ? n.y : (cy(i) > 0 ? n.yp : n.ym);
                    q = pw;
                    m = (cz(i) < 0 ? 0 : nxy) + (long long)X + (long long)L.nx * Y;
                } else {
                    m = nbr_index(L, n, i);
                }
                ps[i][0] = q[2 * m];
                ps[i][1] = q[2 * m + 1];
            }
            link_gradient<C>(grad, [&](int i, int k) { return ps[i][k]; });
        }
        const C G = prm<C>(L.P.G, L.PF.G), G36 = G * wgt<C>(7);
        mixture<C>(L, rho, j, u, om);
        const C tiny = sizeof(C) == 8 ? C(1e-300) : C(1e-30);
        C v[2][3];
#pragma unroll
        for (int k = 0; k < 2; k++)
#pragma unroll
            for (int d = 0; d < 3; d++) {
                acc[k][d] = prm<C>(L.P.body_force[d], L.PF.body_force[d]) - G36 * grad[1 - k][d];
                v[k][d] = rho[k] > tiny ? u[d] + acc[k][d] : u[d];
            }
        C a = C(1) - om;
        // incoming adjoint mu = dJ/df*, and the wall bounce-back density term
        C mu[2][Q];
        C rbar[2] = {0, 0};
        const double* uwlo = L.P.wall_u_lo;
        const double* uwhi = L.P.wall_u_hi;
        // the population of the neighbour, or, of a link into a wall or a fixed
        // particle, the site's own one of the opposite link: the class bits
        // pick the address, so that all loads are under way together (a branch
        // per link on the neighbour's mask took the loads one after the other:
        // 96 -> 47 us at 64^3)
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const bool wall = i != 0 && nbr_is_wall(n, i), own = i == 0 || wall || ((nbc >> i) & 1u);
            const long long m = own ? s : nbr_index(L, n, i);
            const long long e = (own ? opp(i) : i) * L.pstride + m;
#pragma unroll
            for (int k = 0; k < 2; k++) mu[k][i] = Lin[k * Q * L.pstride + e] + Rin[k * L.pstride + m];
        }
        if (n.wall_lo || n.wall_hi) {
#pragma unroll
            for (int i = 1; i < Q; i++) {
                if (cz(i) == 0 || !nbr_is_wall(n, i)) continue;
                const double* uw = cz(i) < 0 ? uwlo : uwhi;
                const C cu = C(cx(i) * uw[0] + cy(i) * uw[1] + cz(i) * uw[2]);
                for (int k = 0; k < 2; k++) rbar[k] += mu[k][i] * (-C(6) * wgt<C>(i) * cu);
            }
        }
        if (A.dJdF && (nbc & NB_LINKS)) {
            // plus the link force of Eq. 19 on a fixed particle
#pragma unroll
            for (int i = 1; i < Q; i++) {
                if (!((nbc >> i) & 1u)) continue;
                const double* gp = A.dJdF + 3 * L.owner[nbr_index(L, n, i)];
                const C gc = C(2) * C(cx(i) * gp[0] + cy(i) * gp[1] + cz(i) * gp[2]);
                for (int k = 0; k < 2; k++) mu[k][i] += gc;
            }
        }
        // backward through the collision
        C ubar[3] = {0, 0, 0}, abar = 0, Fbar[2][3];
        for (int k = 0; k < 2; k++) {
            Mom<C> M;
            moments_of<C>(mu[k], M);
            C P = 0;
#pragma unroll
            for (int i = 0; i < Q; i++) P += mu[k][i] * fv[k][i];
            C shu = mom_shape<C>(M, u), shv = mom_shape<C>(M, v[k]);
            abar += P - rho[k] * shu;
            rbar[k] += -a * shu + shv;
            C gu[3], gv[3];
            mom_grad<C>(M, u, gu);
            mom_grad<C>(M, v[k], gv);
            for (int d = 0; d < 3; d++) {
                ubar[d] += -a * rho[k] * gu[d];
                ubar[d] += rho[k] * gv[d];
                // dJ/dF^k = gv; F^k / rho^k does not depend on rho^k
                Fbar[k][d] = rho[k] > tiny ? gv[d] : C(0);
            }
        }
        // forces: F^A = -G rho^A S^B + rho^A g, F^B = -G rho^B S^A + rho^B g
        C SAbar[3], SBbar[3], Gbar = 0;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            SBbar[d] = -G * rho[0] * Fbar[0][d];
            SAbar[d] = -G * rho[1] * Fbar[1][d];
            Gbar -= wgt<C>(7) * (rho[0] * Fbar[0][d] * grad[1][d] + rho[1] * Fbar[1][d] * grad[0][d]);
        }
        // mixture velocity
        const C w0 = prm<C>(L.inv_tau[0], L.PF.inv_tau[0]), w1 = prm<C>(L.inv_tau[1], L.PF.inv_tau[1]);
        const C iD = C(1) / (w0 * rho[0] + w1 * rho[1]);
        C jbar[2][3];
        const C Dbar = -(ubar[0] * u[0] + ubar[1] * u[1] + ubar[2] * u[2]) * iD;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            jbar[0][d] = w0 * ubar[d] * iD;
            jbar[1][d] = w1 * ubar[d] * iD;
        }
        rbar[0] += w0 * Dbar;
        rbar[1] += w1 * Dbar;
        const C wbar0 = (ubar[0] * j[0][0] + ubar[1] * j[0][1] + ubar[2] * j[0][2]) * iD + Dbar * rho[0];
        const C wbar1 = (ubar[0] * j[1][0] + ubar[1] * j[1][1] + ubar[2] * j[1][2]) * iD + Dbar * rho[1];
        C taub0 = -wbar0 * w0 * w0, taub1 = -wbar1 * w1 * w1;
        // relaxation frequency of the mixture
        const C in0 = prm<C>(L.inv_nu[0], L.PF.inv_nu[0]), in1 = prm<C>(L.inv_nu[1], L.PF.inv_nu[1]);
        const C irt = C(1) / (rho[0] + rho[1]), x0 = rho[0] * irt, x1 = rho[1] * irt;
        const C q = x0 * in0 + x1 * in1;
        const C nub = C(1) / q;
        const C nubbar = C(3) * abar * om * om;  // om = 1 / (3 nub + 1/2), a = 1 - om
        const C qbar = -nubbar * (nub * nub);
        rbar[0] += qbar * (in0 - q) * irt;
        rbar[1] += qbar * (in1 - q) * irt;
        taub0 -= qbar * (x0 * in0 * in0) * C(1.0 / 3.0);
        taub1 -= qbar * (x1 * in1 * in1) * C(1.0 / 3.0);
        // local adjoint of the populations
#pragma unroll
        for (int k = 0; k < 2; k++)
#pragma unroll
            for (int i = 0; i < Q; i++)
                Lout[((long long)(k * Q + i)) * L.pstride + s] =
                    a * mu[k][i] + rbar[k] + along<C>(i, jbar[k]);
        for (int d = 0; d < 3; d++) {
            sb[(0 * 3 + d) * L.N + s] = SAbar[d];
            sb[(1 * 3 + d) * L.N + s] = SBbar[d];
        }
        part[0] = taub0;
        part[1] = taub1;
        part[2] = Gbar;
    }
    // block partials of the parameter gradients (FP64 across threads)
    int nb = gridDim.x * gridDim.y * gridDim.z;
    int b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    double sums[3] = {double(part[0]), double(part[1]), double(part[2])};
    block_sum_store<3>(sums, A.red + b, nb);
}

// dJ/dpsi^k(y) = sum_i w_i c_i . Sbar^k(y - c_i) over fluid x = y - c_i.  On
// fluid nodes it is the density adjoint R; on particle frontier nodes it
// becomes coef = dJ/dpsi (1 + zeta^k) / W (W = sum of the fluid-neighbour
// weights, Eq. 20) and contributes dJ/dzeta^k = dJ/dpsi psi/(1 + zeta^k);
// with the Janus switch s of the node the factor is 1 + s_k zeta^k
// (s_A = s, s_B = -s) and the contribution dJ/dpsi s_k psi/(1 + s_k zeta^k).
template <int PREC>
__global__ void __launch_bounds__(128) k_adj_gather(Lattice L, AdjArgs A) {
    typedef typename Prec<PREC>::C C;
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y, z = blockIdx.z;
    C zp[2] = {0, 0};
    if (x < L.nx) {
        long long s = (long long)x + (long long)L.nx * ((long long)y + (long long)L.ny * z);
        SiteNbr n = site_nbr(L, x, y, z);
        const C* sb = (const C*)A.sbar;
        const uint32_t nbc = L.nb[s];
        const bool solid = nbc & NB_SOLID;
        C pb[2] = {0, 0}, W = 0;
#pragma unroll
        for (int i = 1; i < Q; i++) {
            // the site x = y - c_i is the neighbour along opp(i)
            int io = opp(i);
            const bool fluid = !nbr_is_wall(n, io) && (solid == (bool)((nbc >> io) & 1u));
            const long long m = fluid ? nbr_index(L, n, io) : s;
            const C w = fluid ? wgt<C>(i) : C(0);
            W += w;
#pragma unroll
            for (int k = 0; k < 2; k++) {
                C q[3];
#pragma unroll
                for (int d = 0; d < 3; d++)
                    if (d == 0 ? cx(i) : (d == 1 ? cy(i) : cz(i))) q[d] = sb[(k * 3 + d) * L.N + m];
                pb[k] += fluid ? w * along<C>(i, q) : C(0);
            }
        }
        C* Rout = (C*)A.adj_out + 2 * Q * L.pstride;
        C* cf = (C*)A.coef;
        if (!solid) {
            Rout[s] = pb[0];
            Rout[L.pstride + s] = pb[1];
        } else {
            const C* psi = (const C*)L.psi;
            // the node's wetting factors 1 + s_k zeta^k: s_k = 1 without the
            // Janus switch, s_A = s and s_B = -s with it
            C sk[2] = {C(1), C(1)};
            if (L.P.janus) {
                const int p = L.owner[s];
                const int xs[3] = {x, y, z}, Ls[3] = {L.nx, L.ny, L.nz};
                C d[3];
                for (int c = 0; c < 3; c++) {
                    double dd = (double)xs[c] - L.pos[3 * p + c];
                    if (L.per[c]) dd -= (double)Ls[c] * rint(dd / (double)Ls[c]);
                    d[c] = C(dd);
                }
                const C sw = janus_switch<C>(L, p, d);
                sk[0] = sw;
                sk[1] = -sw;
            }
            for (int k = 0; k < 2; k++) {
                C zk = C(1) + sk[k] * C(L.P.zeta[k]);
                cf[k * L.N + s] = W > C(0) ? pb[k] * zk / W : C(0);
                zp[k] = W > C(0) ? pb[k] * sk[k] * psi[2 * s + k] / zk : C(0);
            }
        }
    }
    int nb = gridDim.x * gridDim.y * gridDim.z;
    int b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    double sums[2] = {double(zp[0]), double(zp[1])};
    block_sum_store<2>(sums, A.red + 3ll * nb + b, nb);
}

// wall nodes: dJ/dpsi_wall from the fluid plane next to the wall, turned into
// coef_wall = dJ/dpsi_wall / W (the wall density is a plain mean)
template <typename C>
__global__ void k_adj_wall(Lattice L, AdjArgs A) {
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y, side = blockIdx.z;
    if (x >= L.nx) return;
    int zf = side == 0 ? 0 : L.nz - 1;
    int dz = side == 0 ? -1 : 1;  // links from the fluid plane into the wall
    const C* sb = (const C*)A.sbar;
    C pb[2] = {0, 0}, W = 0;
    long long nxy = (long long)L.nx * L.ny;
    for (int i = 1; i < Q; i++) {
        if (cz(i) != dz) continue;
        // fluid site x_f = wall site - c_i
        int X = x - cx(i), Y = y - cy(i);
        X = X < 0 ? X + L.nx : (X >= L.nx ? X - L.nx : X);
        Y = Y < 0 ? Y + L.ny : (Y >= L.ny ? Y - L.ny : Y);
        long long m = (long long)X + (long long)L.nx * ((long long)Y + (long long)L.ny * zf);
        if (L.mask[m]) continue;
        C w = wgt<C>(i);
        W += w;
        for (int k = 0; k < 2; k++)
            pb[k] += w * (C(cx(i)) * sb[(k * 3 + 0) * L.N + m] + C(cy(i)) * sb[(k * 3 + 1) * L.N + m] +
                          C(cz(i)) * sb[(k * 3 + 2) * L.N + m]);
    }
    C* cw = (C*)A.coef_wall;
    long long w = (long long)x + (long long)L.nx * y;
    for (int k = 0; k < 2; k++) cw[(side * 2 + k) * nxy + w] = W > C(0) ? pb[k] / W : C(0);
}

// fluid sites next to particle or wall nodes receive the virtual / wall
// density adjoint: R^k(x) += sum_j w_j coef^k(x + c_j)
template <int PREC>
__global__ void __launch_bounds__(128) k_adj_scatter(Lattice L, AdjArgs A) {
    typedef typename Prec<PREC>::C C;
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y, z = blockIdx.z;
    if (x >= L.nx) return;
    long long s = (long long)x + (long long)L.nx * ((long long)y + (long long)L.ny * z);
    const uint32_t nbc = L.nb[s];
    if (nbc & NB_SOLID) return;
    SiteNbr n = site_nbr(L, x, y, z);
    if (!(nbc & NB_LINKS) && !n.wall_lo && !n.wall_hi) return;
    const C* cf = (const C*)A.coef;
    const C* cw = (const C*)A.coef_wall;
    long long nxy = (long long)L.nx * L.ny;
    C add[2] = {0, 0};
#pragma unroll
    for (int j = 1; j < Q; j++) {
        C w = wgt<C>(j);
        if (nbr_is_wall(n, j)) {
            int X = cx(j) == 0 ? n.x : (cx(j) > 0 ? n.xp : n.xm);
            int Y = cy(j) == 0 ? n.y : (cy(j) > 0 ? n.yp : n.ym);
            int side = cz(j) < 0 ? 0 : 1;
            long long wi = (long long)X + (long long)L.nx * Y;
            add[0] += w * cw[(side * 2 + 0) * nxy + wi];
            add[1] += w * cw[(side * 2 + 1) * nxy + wi];
            continue;
        }
        if (!((nbc >> j) & 1u)) continue;
        long long m = nbr_index(L, n, j);
        add[0] += w * cf[m];
        add[1] += w * cf[L.N + m];
    }
    C* Rout = (C*)A.adj_out + 2 * Q * L.pstride;
    Rout[s] += add[0];
    Rout[L.pstride + s] += add[1];
}

// Sums of the nb partials of each of gridDim.x values, red[v][nb], stored to
// out[v], or added to it: a block of 256 threads per value, each thread the
// partials t, t + 256, ... (Neumaier), then lanes and warps merge in a fixed
// order.  (One warp per value and, for the objective, one thread took 51 us
// and 563 us of dependent additions at 64^3; 14 us each now.)
__global__ void __launch_bounds__(256) k_sum_partials(const double* __restrict__ red, int nb, double* out, bool add) {
    __shared__ NSum part[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* r = red + (long long)blockIdx.x * nb;
    NSum t = {0.0, 0.0};
    auto across = [&](int from) {
        for (int off = from; off > 0; off >>= 1) {
            NSum o = {__shfl_down_sync(0xffffffffu, t.s, off), __shfl_down_sync(0xffffffffu, t.c, off)};
            if (lane < off) t.merge(o);
        }
    };
    for (int b = threadIdx.x; b < nb; b += 256) t.add(r[b]);
    across(16);
    if (lane == 0) part[warp] = t;
    __syncthreads();
    if (warp > 0) return;
    if (lane < 8) t = part[lane];
    across(4);
    if (lane == 0) out[blockIdx.x] = (add ? out[blockIdx.x] : 0.0) + t.value();
}

// dJ/dF_p for J = weight sum_p sqrt(|F_p|^2 + eps^2)
__global__ void k_drag_gradient(int n, const double* F, double weight, double eps, double* out) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    double f0 = F[3 * p], f1 = F[3 * p + 1], f2 = F[3 * p + 2];
    double sc = weight / sqrt(f0 * f0 + f1 * f1 + f2 * f2 + eps * eps);
    out[3 * p] = sc * f0;
    out[3 * p + 1] = sc * f1;
    out[3 * p + 2] = sc * f2;
}

// Seed of the interface measure A = sum_x (1 - phi^2), phi = (rho_A - rho_B)/
// (rho_A + rho_B), over fluid nodes: L = 0, R^k = dA/drho^k, and block
// partials of A itself.
template <int PREC>
__global__ void __launch_bounds__(128) k_adj_seed_interface(Lattice L, void* adj, double* red, double weight) {
    typedef typename Prec<PREC>::C C;
    typedef typename Prec<PREC>::S S;
    long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double val = 0.0;
    if (s < L.N) {
        C* Lout = (C*)adj;
        C* Rout = Lout + 2 * Q * L.pstride;
        for (int q = 0; q < 2 * Q; q++) Lout[(long long)q * L.pstride + s] = 0;
        C r0 = 0, r1 = 0;
        if (!L.mask[s]) {
            C fv[2][Q], rho[2], j[2][3];
            load_site<PREC>(L, (const S*)L.f_cur, s, fv, rho, j);
            C rt = rho[0] + rho[1];
            C phi = (rho[0] - rho[1]) / rt;
            r0 = C(weight) * (-C(4) * phi * rho[1] / (rt * rt));
            r1 = C(weight) * (C(4) * phi * rho[0] / (rt * rt));
            val = double(C(1) - phi * phi);
        }
        Rout[s] = r0;
        Rout[L.pstride + s] = r1;
    }
    double sums[1] = {val};
    block_sum_store<1>(sums, red + blockIdx.x, 1);
}

// dJ/drho^k(0) = sum_i w_i lambda^k_i(0) for f(0) = f^eq(rho^k(0), 0) = w_i rho^k(0)
template <int PREC>
__global__ void k_adj_initial(Lattice L, const void* adj, double* grad) {
    typedef typename Prec<PREC>::C C;
    long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= L.N) return;
    const C* Lin = (const C*)adj;
    const C* Rin = Lin + 2 * Q * L.pstride;
    for (int k = 0; k < 2; k++) {
        double g = 0.0;
        if (!L.mask[s]) {
            C acc = 0;
            for (int i = 0; i < Q; i++) acc += wgt<C>(i) * Lin[((long long)(k * Q + i)) * L.pstride + s];
            g = double(acc + Rin[k * L.pstride + s]);
        }
        grad[k * L.N + s] = g;
    }
}

// ---------------------------------------------------------- launchers
#define DISPATCHA(prec, call)                                 \
    switch (prec) {                                           \
        case LB_FP64: { const int P = LB_FP64; call; break; } \
        case LB_FP32: { const int P = LB_FP32; call; break; } \
        default:      { const int P = LB_FP16; call; break; } \
    }

size_t adjoint_field_bytes(const Lattice& L, int prec) {
    size_t c = prec == LB_FP64 ? 8 : 4;
    return (size_t)(2 * Q + 2) * L.pstride * c;
}

size_t adjoint_scratch_bytes(const Lattice& L, int prec) {
    size_t c = prec == LB_FP64 ? 8 : 4;
    size_t nxy = (size_t)L.nx * L.ny;
    dim3 g((L.nx + 127) / 128, L.ny, L.nz);
    size_t nb = (size_t)g.x * g.y * g.z;
    size_t nb1 = (size_t)((L.N + 127) / 128);
    return 6 * L.N * c + 2 * L.N * c + 4 * nxy * c + (ADJ_VALUES * (nb > nb1 ? nb : nb1) + 16) * 8 + 4096;
}

static AdjArgs adj_args(const Lattice& L, int prec, const void* in, void* out, void* scratch,
                        const double* dJdF) {
    size_t c = prec == LB_FP64 ? 8 : 4;
    size_t nxy = (size_t)L.nx * L.ny;
    char* p = (char*)scratch;
    AdjArgs A;
    A.adj_in = in;
    A.adj_out = out;
    A.sbar = p; p += 6 * L.N * c;
    A.coef = p; p += 2 * L.N * c;
    A.coef_wall = p; p += 4 * nxy * c;
    p = (char*)(((uintptr_t)p + 255) & ~(uintptr_t)255);
    A.red = (double*)p;
    A.dJdF = dJdF;
    return A;
}

// one adjoint step; the 5 parameter gradients of this step are added to grads_dev
int launch_adjoint_step(const Lattice& L, int prec, const void* in, void* out, void* scratch,
                        const double* dJdF_dev, double* grads_dev, cudaStream_t st) {
    AdjArgs A = adj_args(L, prec, in, out, scratch, dJdF_dev);
    dim3 g((L.nx + 127) / 128, L.ny, L.nz);
    int bx = L.nx >= 128 ? 128 : ((L.nx + 31) / 32) * 32;
    dim3 gg((L.nx + bx - 1) / bx, L.ny, L.nz);
    int nb = gg.x * gg.y * gg.z;
    int n = 0;
    DISPATCHA(prec, (k_adj_local<P><<<gg, bx, 0, st>>>(L, A)));
    n++;
    if (!L.per[2]) {
        dim3 gw((L.nx + 127) / 128, L.ny, 2);
        if (prec == LB_FP64) k_adj_wall<double><<<gw, 128, 0, st>>>(L, A);
        else k_adj_wall<float><<<gw, 128, 0, st>>>(L, A);
        n++;
    } else {
        size_t c = prec == LB_FP64 ? 8 : 4;
        cudaMemsetAsync(A.coef_wall, 0, 4 * (size_t)L.nx * L.ny * c, st);
    }
    DISPATCHA(prec, (k_adj_gather<P><<<gg, bx, 0, st>>>(L, A)));
    DISPATCHA(prec, (k_adj_scatter<P><<<gg, bx, 0, st>>>(L, A)));
    k_sum_partials<<<ADJ_VALUES, 256, 0, st>>>(A.red, nb, grads_dev, true);
    (void)g;
    return n + 3;
}

int launch_adjoint_seed(const Lattice& L, int prec, void* adj, void* scratch, double weight, double* value_dev,
                        cudaStream_t st) {
    AdjArgs A = adj_args(L, prec, nullptr, adj, scratch, nullptr);
    int nb = (int)((L.N + 127) / 128);
    DISPATCHA(prec, (k_adj_seed_interface<P><<<nb, 128, 0, st>>>(L, adj, A.red, weight)));
    k_sum_partials<<<1, 256, 0, st>>>(A.red, nb, value_dev, false);
    return 2;
}

int launch_drag_gradient(int n, const double* F, double weight, double eps, double* out, cudaStream_t st) {
    if (n <= 0) return 0;
    k_drag_gradient<<<(n + 127) / 128, 128, 0, st>>>(n, F, weight, eps, out);
    return 1;
}

int launch_adjoint_initial(const Lattice& L, int prec, const void* adj, double* grad, cudaStream_t st) {
    DISPATCHA(prec, (k_adj_initial<P><<<(unsigned)((L.N + 255) / 256), 256, 0, st>>>(L, adj, grad)));
    return 1;
}

}  // namespace lbgb
