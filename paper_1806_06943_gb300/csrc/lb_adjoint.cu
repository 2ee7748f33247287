// lb_adjoint.cu -- discrete adjoint of one FP64 time step of the two-range
// pseudopotential lattice Boltzmann method (the step of lb_kernels.cuh:
// Eqs. 1-3, 5, 6, 8, 9 and half-way bounce-back), for gradients of an
// observable with respect to theta = (G_AB, G1, G2, tau_A, tau_B).
//
// Forward step at node x (species k, direction i):
//   rho_k = sum_i f_k,i,  psi_k = 1 - exp(-rho_k)
//   S1_k = sum_i w_i psi_k(x+e_i) e_i,  S2_k = sum_j p_j psi_k(x+e_j) e_j,
//   S3_k = sum_i w_i rho_kbar(x+e_i) e_i
//   F_k = -G1 psi_k S1_k - G2 psi_k S2_k - G_AB rho_k S3_k + rho_k g
//   m_k = sum_i f_k,i e_i + F_k / 2,  u = sum_k om_k m_k / sum_k om_k rho_k
//   f*_k,i = f_k,i - om_k (f_k,i - feq_i(rho_k, u)) + (1 - om_k/2) w_i [3(e_i - u) + 9 (e_i.u) e_i].F_k
//   f_k,i(x + e_i, t+1) = f*_k,i(x)   (or f_k,opp(i)(x, t+1) at a wall)
// Reverse of it, given lam = dJ/df(t+1):
//   lam*_k,i(x) = lam_k,i(x + e_i) (or lam_k,opp(i)(x) at a wall)      [pull]
//   phase A (local at x): the adjoints of u, F_k, m_k, the local parts of
//     the adjoints of rho_k and psi_k, the stencil sources
//     S1bar = -G1 psi F_bar, S2bar = -G2 psi F_bar, S3bar = -G_AB rho F_bar,
//     and the parameter-gradient contributions (per-node sums, FP64)
//   phase B (gather at y): psi_bar(y) += sum over the nodes x whose stencils
//     read y of w e . S1bar(x) + p e . S2bar(x); rho_bar(y) += exp(-rho) psi_bar
//     + w e . S3bar_kbar(x); lam_k,i(y, t) = (1 - om_k) lam*_k,i + m_bar_k . e_i + rho_bar_k.
// Ghost rows beyond a wall: a mirrored ghost passes its adjoint to the fluid
// node it copies; a fixed ghost is a constant and receives none.
#include <cuda_runtime.h>

#include "lb_kernels.cuh"
#include "lb_launch.h"

namespace lbk {

namespace {

// slots of the per-node buffer between the two phases
enum AdjSlot {
    aPsiA = 0, aPsiB, aRhoA, aRhoB,             // local psi_bar, rho_bar
    aMAx, aMAy, aMBx, aMBy,                      // m_bar
    aTAx, aTAy, aTBx, aTBy,                      // psi F_bar: S1bar = -G1 T, S2bar = -G2 T
    aQAx, aQAy, aQBx, aQBy,                      // rho F_bar: S3bar = -G_AB Q
    kAdjSlots
};
static_assert(kAdjSlots == kAdjSlotCount, "the host sizes the buffer");
// parameter-gradient accumulators, a plane each
enum AdjGrad { gGAB = 0, gG1, gG2, gOmA, gOmB, kAdjGrads };
static_assert(kAdjGrads == kAdjGradPlanes, "the host sizes the buffer");

__device__ __forceinline__ int wrapi(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// lam*(x, i): the adjoint of the population pushed from x in direction i
__device__ __forceinline__ double pull_lam(const Lat<double> &L, const double *__restrict__ lam, int k, int i, int x,
                                           int y)
{
    int xd = wrapi(x + ex9(i), L.nx), yd = y + ey9(i);
    int dir = i;
    if (yd < 0 || yd >= L.ny) {
        if (L.walls) {
            dir = opp9(i);
            xd = x;
            yd = y;
        } else {
            yd = wrapi(yd, L.ny);
        }
    }
    return lam[(size_t)(k * 9 + dir) * L.plane + (size_t)yd * L.pitch + xd];
}

}  // namespace

// D2Q9 and D2Q25 sums sum_j w_j s(x + e_j) e_j of a staged plane from
// differences of opposite neighbours (the inner ones serve both).
__device__ __forceinline__ void adj_sums(const Arith64<false> &A, const double (*s)[SW], int cx, int cy, double (&s9)[2],
                                         double (*s25)[2])
{
    constexpr double W1 = 1.0 / 9.0, W2 = 1.0 / 36.0;
    auto D = [&](int dx, int dy) { return A.sub(s[cy + dy][cx + dx], s[cy - dy][cx - dx]); };
    const double dE = D(1, 0), dN = D(0, 1), d1 = D(1, 1), d2 = D(1, -1);
    const double p = A.add(d1, d2), q = A.sub(d1, d2);
    s9[0] = __fma_rn(W1, dE, W2 * p);
    s9[1] = __fma_rn(W1, dN, W2 * q);
    if (!s25) return;
    double x = (2.0 * p25(4)) * D(2, 0), y = (2.0 * p25(4)) * D(0, 2);
#pragma unroll
    for (int a = 1; a <= 2; ++a)
#pragma unroll
        for (int b = 1; b <= 2; ++b) {
            if (a == 1 && b == 1) continue;
            const double e1 = D(a, b), e2 = D(a, -b);
            x = __fma_rn(p25(a * a + b * b) * a, A.add(e1, e2), x);
            y = __fma_rn(p25(a * a + b * b) * b, A.sub(e1, e2), y);
        }
    (*s25)[0] = __fma_rn(p25(1), dE, __fma_rn(p25(2), p, x));
    (*s25)[1] = __fma_rn(p25(1), dN, __fma_rn(p25(2), q, y));
}

// Phase A.  seed_kind: 0 = adjoint of a time step (lam_next given); 1 = seed
// of mu_r at this state (d J / d Q in seed_a, per-node m_bar from ubar); 2 =
// seed of the Laplace pressure jump (c_in = seed_a for r < R/2, c_out = seed_b
// for r > R + 6, probe in L).  rho: the densities and exp(-rho) of k_adj_density.
//
// Everything the collision's adjoint needs of lam* are its moments of second
// order with the weights w_i: with M0, M1, M2 the sums of w_i lam*_i (1, e,
// e e), V = 3 M1 - 3 u M0 + 9 M2 u and a = 1 - omega/2,
//   u_bar = omega rho V + a (9 M2 F - 3 F M0),   F_bar = a V,
//   rho_bar = omega P,  P = M0 + 3 M1.u + 4.5 u.M2 u - 1.5 u.u M0,
//   omega_bar = rho P - sum_i lam*_i f_i - V.F / 2,
// which takes a third of the FP64 instructions (they bound the kernel) of the
// sums written per direction: 415 a node instead of 1414, 214 -> 67 us on a
// 512 x 128 lattice; k_adj_gather, with one combined stencil, 158 instead of
// 559, 90 -> 30 us.
__global__ void __launch_bounds__(kThreads, 4) k_adj_local(const Lat<double> L, const double *__restrict__ f,
                                                           const double *__restrict__ rho, const double *__restrict__ lam_next,
                                                           double *__restrict__ abuf, double *__restrict__ gpart, int seed_kind,
                                                           double seed_a, double seed_b)
{
    __shared__ double srho[2][SH][SW];
    __shared__ double spsi[2][SH][SW];
    const int tiles_x = (L.nx + TX - 1) / TX;
    const int x0 = (blockIdx.x % tiles_x) * TX, y0 = (blockIdx.x / tiles_x) * TY;
    const int tid = threadIdx.y * TX + threadIdx.x;
    const Arith64<false> A(opaque_one());
    for (int idx = tid; idx < SW * SH; idx += kThreads) {
        const int sx = idx % SW, sy = idx / SW;
        const int gx = wrap_index(x0 + sx - HALO, L.nx);
        int gy = y0 + sy - HALO;
        bool fixed = false;
        if (gy < 0 || gy >= L.ny) {
            if (!L.walls) {
                gy = wrap_index(gy, L.ny);
            } else if (L.wall_mode == 1) {
                fixed = true;
            } else {
                gy = gy < 0 ? -1 - gy : 2 * L.ny - 1 - gy;
                gy = gy < 0 ? 0 : (gy >= L.ny ? L.ny - 1 : gy);  // rows no valid node reads
            }
        }
        const size_t c = (size_t)gy * L.pitch + gx;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            srho[k][sy][sx] = fixed ? L.wall_rho[k] : rho[(size_t)k * L.plane + c];
            spsi[k][sy][sx] = fixed ? psi64(L.wall_rho[k], A.one, L.exp_table) : A.sub(1.0, rho[(size_t)(2 + k) * L.plane + c]);
        }
    }
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    const size_t c = (size_t)y * L.pitch + x;
    double S1[2][2], S2[2][2], S3[2][2], F[2][2], m[2][2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        double fk[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) fk[i] = f[(size_t)(k * 9 + i) * L.plane + c];
        adj_sums(A, spsi[k], cx, cy, S1[k], &S2[k]);
        adj_sums(A, srho[1 - k], cx, cy, S3[k], nullptr);
        const double r = srho[k][cy][cx], ps = spsi[k][cy][cx];
#pragma unroll
        for (int a = 0; a < 2; ++a)
            F[k][a] = __fma_rn(-ps, __fma_rn(L.G1, S1[k][a], L.G2 * S2[k][a]), r * __fma_rn(-L.GAB, S3[k][a], L.g[a]));
        const double d57 = A.sub(fk[5], fk[7]), d86 = A.sub(fk[8], fk[6]);
        m[k][0] = __fma_rn(0.5, F[k][0], A.add(A.sub(fk[1], fk[3]), A.add(d57, d86)));
        m[k][1] = __fma_rn(0.5, F[k][1], A.add(A.sub(fk[2], fk[4]), A.sub(d57, d86)));
    }
    const double r[2] = {srho[0][cy][cx], srho[1][cy][cx]};
    const double om[2] = {L.omega[0], L.omega[1]};
    double aV[2][2] = {{0.0, 0.0}, {0.0, 0.0}}, rb[2] = {0.0, 0.0}, mb[2][2] = {{0.0, 0.0}, {0.0, 0.0}}, omb[2] = {0.0, 0.0};
    double gr[kAdjGrads] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (seed_kind == 0) {
        const double rD = 1.0 / __fma_rn(om[0], r[0], om[1] * r[1]);
        const double u[2] = {__fma_rn(om[0], m[0][0], om[1] * m[1][0]) * rD, __fma_rn(om[0], m[0][1], om[1] * m[1][1]) * rD};
        const double uu15 = 1.5 * __fma_rn(u[0], u[0], u[1] * u[1]);
        double ub[2] = {0.0, 0.0};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            constexpr double w0 = 4.0 / 9.0, w1 = 1.0 / 9.0, w2 = 1.0 / 36.0;
            double l[9], lf = 0.0;
#pragma unroll
            for (int i = 0; i < 9; ++i) l[i] = pull_lam(L, lam_next, k, i, x, y);
#pragma unroll
            for (int i = 0; i < 9; ++i) lf = __fma_rn(l[i], f[(size_t)(k * 9 + i) * L.plane + c], lf);
            const double ax = A.add(l[1], l[3]), ay = A.add(l[2], l[4]), p57 = A.add(l[5], l[7]), p68 = A.add(l[6], l[8]);
            const double m57 = A.sub(l[5], l[7]), m68 = A.sub(l[6], l[8]), dg = w2 * A.add(p57, p68);
            const double M0 = __fma_rn(w0, l[0], __fma_rn(w1, A.add(ax, ay), dg));
            const double M1x = __fma_rn(w1, A.sub(l[1], l[3]), w2 * A.sub(m57, m68));
            const double M1y = __fma_rn(w1, A.sub(l[2], l[4]), w2 * A.add(m57, m68));
            const double Mxx = __fma_rn(w1, ax, dg), Myy = __fma_rn(w1, ay, dg), Mxy = w2 * A.sub(p57, p68);
            const double Mux = __fma_rn(Mxx, u[0], Mxy * u[1]), Muy = __fma_rn(Mxy, u[0], Myy * u[1]);
            const double Vx = __fma_rn(9.0, Mux, 3.0 * __fma_rn(-u[0], M0, M1x));
            const double Vy = __fma_rn(9.0, Muy, 3.0 * __fma_rn(-u[1], M0, M1y));
            const double a = __fma_rn(-0.5, om[k], 1.0), omr = om[k] * r[k], a9 = 9.0 * a, a3M = -3.0 * a * M0;
            ub[0] = __fma_rn(omr, Vx, __fma_rn(a9, __fma_rn(Mxx, F[k][0], Mxy * F[k][1]), __fma_rn(a3M, F[k][0], ub[0])));
            ub[1] = __fma_rn(omr, Vy, __fma_rn(a9, __fma_rn(Mxy, F[k][0], Myy * F[k][1]), __fma_rn(a3M, F[k][1], ub[1])));
            aV[k][0] = a * Vx;
            aV[k][1] = a * Vy;
            double P = __fma_rn(-uu15, M0, M0);
            P = __fma_rn(3.0, __fma_rn(M1x, u[0], M1y * u[1]), P);
            P = __fma_rn(4.5, __fma_rn(u[0], Mux, u[1] * Muy), P);
            rb[k] = om[k] * P;
            omb[k] = __fma_rn(-0.5, __fma_rn(Vx, F[k][0], Vy * F[k][1]), __fma_rn(r[k], P, -lf));
        }
        // u = N / D
        const double Nb[2] = {ub[0] * rD, ub[1] * rD};
        const double Db = -__fma_rn(Nb[0], u[0], Nb[1] * u[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            mb[k][0] = om[k] * Nb[0];
            mb[k][1] = om[k] * Nb[1];
            omb[k] = __fma_rn(Nb[0], m[k][0], __fma_rn(Nb[1], m[k][1], __fma_rn(Db, r[k], omb[k])));
            rb[k] = __fma_rn(om[k], Db, rb[k]);
        }
    } else if (seed_kind == 1) {
        // J = Q0 / Q, Q = (1/nx) sum ubar_x, ubar = (m_A + m_B) / (rho_A + rho_B)
        const double rt = r[0] + r[1], ubx = (m[0][0] + m[1][0]) / rt;
        const double s = seed_a / L.nx;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            mb[k][0] = s / rt;
            rb[k] = -s * ubx / rt;
        }
    } else {
        // J = <p_b>_in - <p_b>_out, Eq. (11)
        double dx = fabs((double)x - L.probe[0]), dy = fabs((double)y - L.probe[1]);
        if (dx > 0.5 * L.nx) dx = L.nx - dx;
        if (!L.walls && dy > 0.5 * L.ny) dy = L.ny - dy;
        const double rr = sqrt(dx * dx + dy * dy), R = L.probe[2];
        const double cw = (rr < 0.5 * R ? seed_a : 0.0) + (rr > R + 6.0 ? seed_b : 0.0);
        if (cw != 0.0) {
            const double Gs = L.G1 + L.G2, ps[2] = {spsi[0][cy][cx], spsi[1][cy][cx]};
#pragma unroll
            for (int k = 0; k < 2; ++k)
                rb[k] = cw * ((1.0 + Gs * ps[k] * rho[(size_t)(2 + k) * L.plane + c]) / 3.0 + L.GAB * r[1 - k] / 3.0);
            gr[gG1] += cw * 0.5 * (ps[0] * ps[0] + ps[1] * ps[1]) / 3.0;
            gr[gG2] += cw * 0.5 * (ps[0] * ps[0] + ps[1] * ps[1]) / 3.0;
            gr[gGAB] += cw * r[0] * r[1] / 3.0;
        }
    }
    auto put = [&](int slot, double v) { abuf[(size_t)slot * L.plane + c] = v; };
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        // m = j + F/2, then F = -psi (G1 S1 + G2 S2) - G_AB rho S3 + rho g
        const double Fb[2] = {__fma_rn(0.5, mb[k][0], aV[k][0]), __fma_rn(0.5, mb[k][1], aV[k][1])};
        const double ps = spsi[k][cy][cx], T[2] = {ps * Fb[0], ps * Fb[1]}, Q[2] = {r[k] * Fb[0], r[k] * Fb[1]};
        const double f1 = __fma_rn(Fb[0], S1[k][0], Fb[1] * S1[k][1]), f2 = __fma_rn(Fb[0], S2[k][0], Fb[1] * S2[k][1]);
        const double f3 = __fma_rn(Fb[0], S3[k][0], Fb[1] * S3[k][1]);
        put(aPsiA + k, -__fma_rn(L.G1, f1, L.G2 * f2));
        put(aRhoA + k, __fma_rn(-L.GAB, f3, __fma_rn(Fb[0], L.g[0], __fma_rn(Fb[1], L.g[1], rb[k]))));
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            put(aMAx + 2 * k + a, mb[k][a]);
            put(aTAx + 2 * k + a, T[a]);
            put(aQAx + 2 * k + a, Q[a]);
        }
        gr[gG1] = __fma_rn(-ps, f1, gr[gG1]);
        gr[gG2] = __fma_rn(-ps, f2, gr[gG2]);
        gr[gGAB] = __fma_rn(-r[k], f3, gr[gGAB]);
    }
    gr[gOmA] = omb[0];
    gr[gOmB] = omb[1];
    // the node's running sums over the steps (reduced once, by k_adj_reduce:
    // a reduction per step would cost as many FP64 instructions as a stencil)
#pragma unroll
    for (int a = 0; a < kAdjGrads; ++a) {
        double *g = &gpart[(size_t)a * L.plane + c];
        *g = A.add(*g, gr[a]);
    }
}

// sum_e c(|e|^2) e_x v(x + e) over D2Q25 of a staged plane (AX = 0; e_y for
// AX = 1), c(1), c(2) given and c = G2 p beyond.
template <int AX>
__device__ __forceinline__ double gather25(const Arith64<false> &A, const double (*v)[SW], int cx, int cy, double c1,
                                           double c2, double G2)
{
    auto at = [&](int along, int across) { return AX == 0 ? v[cy + across][cx + along] : v[cy + along][cx + across]; };
    auto two = [&](int along, int across) {   // both sides across the axis
        return A.add(A.sub(at(along, across), at(-along, across)), A.sub(at(along, -across), at(-along, -across)));
    };
    double o = p25(8) * 2.0 * two(2, 2);
    o = __fma_rn(p25(5) * 2.0, two(2, 1), o);
    o = __fma_rn(p25(5), two(1, 2), o);
    o = __fma_rn(p25(4) * 2.0, A.sub(at(2, 0), at(-2, 0)), o);
    return __fma_rn(c1, A.sub(at(1, 0), at(-1, 0)), __fma_rn(c2, two(1, 1), G2 * o));
}

template <int AX>
__device__ __forceinline__ double gather9(const Arith64<false> &A, const double (*v)[SW], int cx, int cy)
{
    auto at = [&](int along, int across) { return AX == 0 ? v[cy + across][cx + along] : v[cy + along][cx + across]; };
    const double d = A.add(A.sub(at(1, 1), at(-1, 1)), A.sub(at(1, -1), at(-1, -1)));
    return __fma_rn(1.0 / 9.0, A.sub(at(1, 0), at(-1, 0)), (1.0 / 36.0) * d);
}

// Phase B: gather the stencil adjoints and form lam(t).  psi_bar takes
// sum_e (G1 w + G2 p) e.T(x + e) and rho_bar of a species G_AB sum_e w e.Q(x + e)
// of the other (the stencils are odd, so a transposed one is its negative), from
// T and Q of the tile and its halo staged in shared memory.  Ghost rows beyond
// a wall hold no node and give nothing; what the stencils of nodes near a
// mirroring wall read from a ghost row goes to the fluid node it copies.
__global__ void __launch_bounds__(kThreads) k_adj_gather(const Lat<double> L, const double *__restrict__ rho,
                                                         const double *__restrict__ lam_next,
                                                         const double *__restrict__ abuf, double *__restrict__ lam_out,
                                                         int seed)
{
    __shared__ double sv[8][SH][SW];   // T A x, y, B x, y, then Q
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int tid = threadIdx.y * TX + threadIdx.x;
    for (int idx = tid; idx < SW * SH; idx += kThreads) {
        const int sx = idx % SW, sy = idx / SW;
        const int gx = wrap_index(x0 + sx - HALO, L.nx);
        int gy = y0 + sy - HALO;
        const bool ghost = L.walls && (gy < 0 || gy >= L.ny);
        gy = ghost ? 0 : wrap_index(gy, L.ny);
#pragma unroll
        for (int v = 0; v < 8; ++v)
            sv[v][sy][sx] = ghost ? 0.0 : abuf[(size_t)(aTAx + v) * L.plane + (size_t)gy * L.pitch + gx];
    }
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    const size_t c = (size_t)y * L.pitch + x;
    const Arith64<false> A(opaque_one());
    const double c1 = -L.cw[0], c2 = -L.cw[1];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        double psb = A.add(gather25<0>(A, sv[2 * k], cx, cy, c1, c2, L.G2), gather25<1>(A, sv[2 * k + 1], cx, cy, c1, c2, L.G2));
        double q = A.add(gather9<0>(A, sv[6 - 2 * k], cx, cy), gather9<1>(A, sv[7 - 2 * k], cx, cy));
        if (L.walls && L.wall_mode == 0 && (y < HALO || y >= L.ny - HALO)) {
            // the mirrored ghost rows this node is copied to: row g of the
            // ghosts, read by nodes of row g - ey with stencil vectors (dx, ey)
            for (int side = 0; side < 2; ++side) {
                const int g = side == 0 ? -1 - y : 2 * L.ny - 1 - y;
                for (int j = 0; j < 25; ++j) {
                    const int dx = j % 5 - 2, ey = j / 5 - 2, e2 = dx * dx + ey * ey, row = g - ey;
                    if (e2 == 0 || row < 0 || row >= L.ny || (side == 0 ? g + HALO < 0 : g - HALO >= L.ny)) continue;
                    const int xs = wrapi(x - dx, L.nx);
                    auto V = [&](int slot) { return abuf[(size_t)slot * L.plane + (size_t)row * L.pitch + xs]; };
                    const double w = e2 == 1 ? 1.0 / 9.0 : e2 == 2 ? 1.0 / 36.0 : 0.0;
                    psb -= (L.G1 * w + L.G2 * p25(e2)) * (dx * V(aTAx + 2 * k) + ey * V(aTAy + 2 * k));
                    if (e2 <= 2) q -= w * (dx * V(aQBx - 2 * k) + ey * V(aQBy - 2 * k));
                }
            }
        }
        psb = A.add(psb, abuf[(size_t)(aPsiA + k) * L.plane + c]);
        const double rb = __fma_rn(rho[(size_t)(2 + k) * L.plane + c], psb,
                                   __fma_rn(L.GAB, q, abuf[(size_t)(aRhoA + k) * L.plane + c]));
        const double mx = abuf[(size_t)(aMAx + 2 * k) * L.plane + c], my = abuf[(size_t)(aMAy + 2 * k) * L.plane + c];
        const double s = A.add(mx, my), d = A.sub(mx, my), h = __fma_rn(-1.0, L.omega[k], 1.0);
        // m_bar . e_i + rho_bar
        const double base[9] = {rb, A.add(rb, mx), A.add(rb, my), A.sub(rb, mx), A.sub(rb, my), A.add(rb, s), A.sub(rb, d),
                                A.sub(rb, s), A.add(rb, d)};
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double ls = seed ? 0.0 : pull_lam(L, lam_next, k, i, x, y);
            lam_out[(size_t)(k * 9 + i) * L.plane + c] = __fma_rn(h, ls, base[i]);
        }
    }
}

// rho_k = sum_i f_k,i and exp(-rho_k) (planes 0, 1 and 2, 3 of rho) for the
// adjoint's recomputed states
__global__ void k_adj_density(const Lat<double> L, const double *__restrict__ f, double *__restrict__ rho)
{
    const int x = blockIdx.x * TX + threadIdx.x;
    const int y = blockIdx.y * TY + threadIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const size_t c = (size_t)y * L.pitch + x;
    const double one = opaque_one();
    for (int k = 0; k < 2; ++k) {
        double v[9];
        for (int i = 0; i < 9; ++i) v[i] = f[(size_t)(k * 9 + i) * L.plane + c];
        const double r = zeroth_moment<double>(v, one);
        rho[(size_t)k * L.plane + c] = r;
        rho[(size_t)(2 + k) * L.plane + c] = exp_minus(r, one, L.exp_table);
    }
}

// Fixed-order reduction of the per-node gradient sums: one block a parameter.
__global__ void __launch_bounds__(1024) k_adj_reduce(const double *__restrict__ gpart, size_t plane, double *__restrict__ out)
{
    __shared__ double s[1024];
    double v = 0.0;
    for (size_t i = threadIdx.x; i < plane; i += 1024) v += gpart[blockIdx.x * plane + i];
    s[threadIdx.x] = v;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = s[0];
}

cudaError_t adj_density(const Lat<double> &L, const double *f, double *rho, cudaStream_t s)
{
    k_adj_density<<<dim3((L.nx + TX - 1) / TX, (L.ny + TY - 1) / TY), dim3(TX, TY), 0, s>>>(L, f, rho);
    return cudaGetLastError();
}

cudaError_t adj_step(const Lat<double> &L, const double *f, const double *rho, const double *lam_next, double *abuf,
                     double *gpart, double *lam_out, int seed_kind, double seed_a, double seed_b, cudaStream_t s)
{
    const int tiles = ((L.nx + TX - 1) / TX) * ((L.ny + TY - 1) / TY);
    k_adj_local<<<tiles, dim3(TX, TY), 0, s>>>(L, f, rho, lam_next, abuf, gpart, seed_kind, seed_a, seed_b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_adj_gather<<<dim3((L.nx + TX - 1) / TX, (L.ny + TY - 1) / TY), dim3(TX, TY), 0, s>>>(L, rho, lam_next, abuf,
                                                                                          lam_out, seed_kind != 0);
    return cudaGetLastError();
}

cudaError_t adj_reduce(const Lat<double> &L, const double *gpart, double *out, cudaStream_t s)
{
    k_adj_reduce<<<kAdjGrads, 1024, 0, s>>>(gpart, L.plane, out);
    return cudaGetLastError();
}

}  // namespace lbk
