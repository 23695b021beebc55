// Generic kernels: any lattice size >= 4 in every dimension, one thread per
// site. The step runs as launches in site order -- phi (zeroth moment of g),
// mu or the chemical stress where the collision does not form them from phi,
// and collide+propagate -- and the same file holds the
// initialiser, the macroscopic output, the FP64 conservation sums, the
// codec I/O and propagation alone. Templates only: instantiated per storage
// precision by ld_prec_f64.cu and ld_prec_lp.cu.
#pragma once
#include "ld_common.cuh"
#include "ld_internal.h"

namespace ld {
namespace {

constexpr int kThreads = 256;

inline Geom to_dev(const GeomH& h) { return Geom{h.nx, h.ny, h.nz, h.n, h.npad}; }

inline unsigned blocks_for(long long n) { return (unsigned)((n + kThreads - 1) / kThreads); }

__device__ __forceinline__ void site_coords(const Geom& g, long long s, int& x, int& y, int& z) {
    const unsigned i = (unsigned)s, t = i / (unsigned)g.nx;  // n < 2^31 (ld_create)
    x = (int)(i - t * (unsigned)g.nx);
    z = (int)(t / (unsigned)g.ny);
    y = (int)(t - (unsigned)z * (unsigned)g.ny);
}

__device__ __forceinline__ long long site_of(const Geom& g, int x, int y, int z) {
    return (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * z);
}

// Coordinate after a displacement of -1, 0 or +1 (periodic).
__device__ __forceinline__ int step_coord(int a, int d, int n) {
    return d > 0 ? wrap_inc(a, n) : (d < 0 ? wrap_dec(a, n) : a);
}

// ---------------------------------------------------------------------------
// The step as launches in site order, kRowThreads consecutive sites per block,
// across the ends of rows: consecutive blocks cover consecutive addresses of
// every stream, the order that lets HBM run at its copy rate, and every block
// is full whatever nx is (blocks of one row's sites left 41 % of the threads
// idle at nx = 150). A site's coordinates come from its index by two
// multiplications (FastDiv). Element offsets i npad + s are of type I: 32-bit
// where 19 npad fits.

// Quotient of 0 <= a < 2^31 by a fixed 2 <= d < 2^31 (Granlund & Montgomery
// 1994): m = ceil(2^(31+l)/d) < 2^32 with l = ceil(log2 d), q = a m / 2^(31+l).
struct FastDiv {
    unsigned m;
    int shift;
    __device__ __forceinline__ int div(int a) const { return (int)(__umulhi((unsigned)a, m) >> shift); }
};
inline FastDiv fast_div(int d) {
    int l = 1;
    while ((1LL << l) < d) ++l;
    return FastDiv{(unsigned)(((1ULL << (31 + l)) + (unsigned)d - 1) / (unsigned)d), l - 1};
}

struct RowGeom {
    int nx, ny, nz, n;
    FastDiv dx, dy;
};

inline RowGeom row_geom(const GeomH& h) {
    return RowGeom{h.nx, h.ny, h.nz, (int)h.n, fast_div(h.nx), fast_div(h.ny)};
}

inline unsigned row_blocks(const GeomH& h) { return (unsigned)((h.n + kRowThreads - 1) / kRowThreads); }

// Site of this thread (false past the end of the lattice).
__device__ __forceinline__ bool row_site(const RowGeom& rg, int& x, int& y, int& z, int& s) {
    s = (int)(blockIdx.x * kRowThreads + threadIdx.x);
    if ((unsigned)s >= (unsigned)rg.n) return false;
    const int row = rg.dx.div(s);
    x = s - row * rg.nx;
    z = rg.dy.div(row);
    y = row - z * rg.ny;
    return true;
}

// N consecutive stored values, one load (s a multiple of N).
template <int N, class S>
struct alignas(N * sizeof(S)) SiteVec {
    S v[N];
};

// Stage 1: phi = sum_i g_i (the stored state is the post-propagation one), two
// sites per thread with 32- and 16-bit storage. npad is even: the second site
// may be the first of the padding, whose phi nothing reads.
template <int P>
__host__ __device__ constexpr int phi_sites() {
    return sizeof(typename Prec<P>::store_t) == 8 ? 1 : 2;
}
template <int P, class I, int N>
__global__ void __launch_bounds__(kRowThreads) k_phi(int n, I npad, const typename Prec<P>::store_t* __restrict__ gs,
                                                     const float* __restrict__ ref,
                                                     typename Prec<P>::real_t* __restrict__ phi, int* __restrict__ status) {
    using R = typename Prec<P>::real_t;
    using S = typename Prec<P>::store_t;
    const int s = (int)((blockIdx.x * kRowThreads + threadIdx.x) * N);
    if ((unsigned)s >= (unsigned)n || !site_ok(s, n, status)) return;
    SiteVec<N, S> v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = *reinterpret_cast<const SiteVec<N, S>*>(gs + i * npad + s);
    SiteVec<N, R> acc{};
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int e = 0; e < N; ++e) acc.v[e] += Prec<P>::decode(v[i].v[e], ref[Q + i]);
    *reinterpret_cast<SiteVec<N, R>*>(phi + s) = acc;
}

// Stage 2: mu = A phi + B phi^3 - kappa lap(phi), with the 7-point or the
// 19-point Laplacian.
template <class R>
__global__ void __launch_bounds__(kRowThreads) k_mu(RowGeom rg, Model<R> m, const R* __restrict__ phi,
                                                    R* __restrict__ mu) {
    int x, y, z, s;
    if (!row_site(rg, x, y, z, s)) return;
    const int nx = rg.nx, plane = rg.nx * rg.ny;
    const int xp = x + 1 == nx ? 1 - nx : 1, xm = x == 0 ? nx - 1 : -1;
    const int yp = y + 1 == rg.ny ? (1 - rg.ny) * nx : nx, ym = y == 0 ? (rg.ny - 1) * nx : -nx;
    const int zp = z + 1 == rg.nz ? (1 - rg.nz) * plane : plane, zm = z == 0 ? (rg.nz - 1) * plane : -plane;
    if (m.iso) {
        auto nb = [&](int i) {
            return phi[s + (cx(i) > 0 ? xp : (cx(i) < 0 ? xm : 0)) + (cy(i) > 0 ? yp : (cy(i) < 0 ? ym : 0)) +
                       (cz(i) > 0 ? zp : (cz(i) < 0 ? zm : 0))];
        };
        mu[s] = chem_potential_lap(phi[s], lap19(phi[s], nb), m);
        return;
    }
    const R nb = phi[s + xp] + phi[s + xm] + phi[s + yp] + phi[s + ym] + phi[s + zp] + phi[s + zm];
    mu[s] = chem_potential(phi[s], nb, m);
}

// Neighbour offsets of a row-ordered site (periodic).
struct RowNbr {
    int xp, xm, yp, ym, zp, zm;
    __device__ __forceinline__ int of(int i) const {
        return (cx(i) > 0 ? xp : (cx(i) < 0 ? xm : 0)) + (cy(i) > 0 ? yp : (cy(i) < 0 ? ym : 0)) +
               (cz(i) > 0 ? zp : (cz(i) < 0 ? zm : 0));
    }
};
__device__ __forceinline__ RowNbr row_nbr(const RowGeom& rg, int x, int y, int z) {
    const int nx = rg.nx, plane = rg.nx * rg.ny;
    return RowNbr{x + 1 == nx ? 1 - nx : 1,
                  x == 0 ? nx - 1 : -1,
                  y + 1 == rg.ny ? (1 - rg.ny) * nx : nx,
                  y == 0 ? (rg.ny - 1) * nx : -nx,
                  z + 1 == rg.nz ? (1 - rg.nz) * plane : plane,
                  z == 0 ? (rg.nz - 1) * plane : -plane};
}

// Gradient of a field at s with the selected stencils (7-point: central
// difference; 19-point: grad19), in the type of the field.
template <class T>
__device__ __forceinline__ void grad_at(int iso, const T* h, int s, const RowNbr& o, T& gx, T& gy, T& gz) {
    if (iso) {
        auto nb = [&](int i) { return h[s + o.of(i)]; };
        grad19(nb, gx, gy, gz);
    } else {
        gx = T(0.5) * (h[s + o.xp] - h[s + o.xm]);
        gy = T(0.5) * (h[s + o.yp] - h[s + o.ym]);
        gz = T(0.5) * (h[s + o.zp] - h[s + o.zm]);
    }
}

// Stage 2b (LD_FORCE_STRESS): chemical stress P[6][npad] (xx, yy, zz, xy,
// xz, yz) from grad phi and lap(phi) with the selected stencils:
//   iso = A/2 phi^2 + 3B/4 phi^4 - kappa phi lap - kappa/2 |grad phi|^2,
//   P_aa = iso + kappa (d_a phi)^2, P_ab = kappa d_a phi d_b phi,
// each expression in that operation order. Takes the place of k_mu: the step
// needs mu at the site alone with this force, and it has the Laplacian at hand.
template <class R, class I>
__global__ void __launch_bounds__(kRowThreads) k_stress(RowGeom rg, I npad, Model<R> m, const R* __restrict__ phi,
                                                        R* __restrict__ P, R* __restrict__ mu) {
    int x, y, z, s;
    if (!row_site(rg, x, y, z, s)) return;
    const RowNbr o = row_nbr(rg, x, y, z);
    const R ph = phi[s];
    R gx, gy, gz, lap;
    grad_at(m.iso, phi, s, o, gx, gy, gz);
    if (m.iso) {
        auto nb = [&](int i) { return phi[s + o.of(i)]; };
        lap = lap19(ph, nb);
        mu[s] = chem_potential_lap(ph, lap, m);
    } else {
        const R nb = phi[s + o.xp] + phi[s + o.xm] + phi[s + o.yp] + phi[s + o.ym] + phi[s + o.zp] + phi[s + o.zm];
        mu[s] = chem_potential(ph, nb, m);
        lap = nb - R(6) * ph;
    }
    const R pb = R(0.5) * m.A * ph * ph + R(0.75) * m.B * ph * ph * ph * ph;
    const R iso = pb - m.kappa * ph * lap - R(0.5) * m.kappa * (gx * gx + gy * gy + gz * gz);
    P[s] = iso + m.kappa * gx * gx;
    P[npad + s] = iso + m.kappa * gy * gy;
    P[2 * npad + s] = iso + m.kappa * gz * gz;
    P[3 * npad + s] = m.kappa * gx * gy;
    P[4 * npad + s] = m.kappa * gx * gz;
    P[5 * npad + s] = m.kappa * gy * gz;
}

// F = -div P at s: F_a = -((D_x P_ax + D_y P_ay) + D_z P_az), D the selected
// gradient, components of P indexed xx 0, yy 1, zz 2, xy 3, xz 4, yz 5.
template <class T, class I>
__device__ __forceinline__ void stress_force_at(int iso, const T* P, I npad, int s, const RowNbr& o, T& Fx, T& Fy,
                                                T& Fz) {
    T d[6][3];
#pragma unroll
    for (int c = 0; c < 6; ++c) grad_at(iso, P + c * npad, s, o, d[c][0], d[c][1], d[c][2]);
    Fx = -((d[0][0] + d[3][1]) + d[4][2]);
    Fy = -((d[3][0] + d[1][1]) + d[5][2]);
    Fz = -((d[4][0] + d[5][1]) + d[2][2]);
}

// A field by offsets from site s; the debug build reads only inside the lattice.
template <class R>
struct FieldAt {
    const R* h;  // the field at s
    int s, n;
    int* status;
    __device__ __forceinline__ R operator[](int d) const { return site_ok((long long)s + d, n, status) ? h[d] : R(0); }
};

// grad mu by central differences (as unscaled differences, twice the gradient)
// and mu at a site from phi alone: mu at the site and its six neighbours, each
// the operations of k_mu, from the 25 phi within two sites.
template <class R>
__device__ __forceinline__ void mu_diffs_of_phi(const RowGeom& rg, const Model<R>& m, const R* phi, int x, int y, int z,
                                                int s, const RowNbr& o, int* status, R& mu, R& dx, R& dy, R& dz) {
    const int nx = rg.nx, plane = rg.nx * rg.ny;
    const int x2 = x + 2 >= nx ? 2 - nx : 2, xm2 = x < 2 ? nx - 2 : -2;
    const int y2 = (y + 2 >= rg.ny ? 2 - rg.ny : 2) * nx, ym2 = (y < 2 ? rg.ny - 2 : -2) * nx;
    const int z2 = (z + 2 >= rg.nz ? 2 - rg.nz : 2) * plane, zm2 = (z < 2 ? rg.nz - 2 : -2) * plane;
    const FieldAt<R> p{phi + s, s, rg.n, status};
    const R c = p[0], xp = p[o.xp], xm = p[o.xm], yp = p[o.yp], ym = p[o.ym], zp = p[o.zp], zm = p[o.zm];
    const R xpyp = p[o.xp + o.yp], xpym = p[o.xp + o.ym], xmyp = p[o.xm + o.yp], xmym = p[o.xm + o.ym];
    const R xpzp = p[o.xp + o.zp], xpzm = p[o.xp + o.zm], xmzp = p[o.xm + o.zp], xmzm = p[o.xm + o.zm];
    const R ypzp = p[o.yp + o.zp], ypzm = p[o.yp + o.zm], ymzp = p[o.ym + o.zp], ymzm = p[o.ym + o.zm];
    mu = chem_potential(c, xp + xm + yp + ym + zp + zm, m);
    dx = chem_potential(xp, p[x2] + c + xpyp + xpym + xpzp + xpzm, m) -
         chem_potential(xm, c + p[xm2] + xmyp + xmym + xmzp + xmzm, m);
    dy = chem_potential(yp, xpyp + xmyp + p[y2] + c + ypzp + ypzm, m) -
         chem_potential(ym, xpym + xmym + c + p[ym2] + ymzp + ymzm, m);
    dz = chem_potential(zp, xpzp + xmzp + ypzp + ymzp + p[z2] + c, m) -
         chem_potential(zm, xpzm + xmzm + ypzm + ymzm + c + p[zm2], m);
}

// The force -div P (7-point stencils) and mu at a site from phi alone: the
// components P_ab that the divergence reads at the six neighbours, each the
// operations of k_stress, from the 25 phi within two sites.
template <class R>
__device__ __forceinline__ void stress_force_of_phi(const RowGeom& rg, const Model<R>& m, const R* phi, int x, int y,
                                                    int z, int s, const RowNbr& o, int* status, R& mu, R& Fx, R& Fy, R& Fz) {
    const int nx = rg.nx, plane = rg.nx * rg.ny;
    const int x2 = x + 2 >= nx ? 2 - nx : 2, xm2 = x < 2 ? nx - 2 : -2;
    const int y2 = (y + 2 >= rg.ny ? 2 - rg.ny : 2) * nx, ym2 = (y < 2 ? rg.ny - 2 : -2) * nx;
    const int z2 = (z + 2 >= rg.nz ? 2 - rg.nz : 2) * plane, zm2 = (z < 2 ? rg.nz - 2 : -2) * plane;
    const FieldAt<R> p{phi + s, s, rg.n, status};
    const R c = p[0], xp = p[o.xp], xm = p[o.xm], yp = p[o.yp], ym = p[o.ym], zp = p[o.zp], zm = p[o.zm];
    const R xpyp = p[o.xp + o.yp], xpym = p[o.xp + o.ym], xmyp = p[o.xm + o.yp], xmym = p[o.xm + o.ym];
    const R xpzp = p[o.xp + o.zp], xpzm = p[o.xp + o.zm], xmzp = p[o.xm + o.zp], xmzm = p[o.xm + o.zm];
    const R ypzp = p[o.yp + o.zp], ypzm = p[o.yp + o.zm], ymzp = p[o.ym + o.zp], ymzm = p[o.ym + o.zm];
    mu = chem_potential(c, xp + xm + yp + ym + zp + zm, m);
    // P_xb, P_yb, P_zb (b the axis of the neighbour) from its phi and six neighbours
    struct Col {
        R x, y, z;
    };
    auto column = [&](int b, R ph, R pxp, R pxm, R pyp, R pym, R pzp, R pzm) {
        const R gx = R(0.5) * (pxp - pxm), gy = R(0.5) * (pyp - pym), gz = R(0.5) * (pzp - pzm);
        const R lap = pxp + pxm + pyp + pym + pzp + pzm - R(6) * ph;
        const R pb = R(0.5) * m.A * ph * ph + R(0.75) * m.B * ph * ph * ph * ph;
        const R iso = pb - m.kappa * ph * lap - R(0.5) * m.kappa * (gx * gx + gy * gy + gz * gz);
        const R gb = b == 0 ? gx : (b == 1 ? gy : gz);
        Col r{m.kappa * gx * gb, m.kappa * gy * gb, m.kappa * gz * gb};
        (b == 0 ? r.x : (b == 1 ? r.y : r.z)) += iso;
        return r;
    };
    const Col a = column(0, xp, p[x2], c, xpyp, xpym, xpzp, xpzm), b = column(0, xm, c, p[xm2], xmyp, xmym, xmzp, xmzm);
    const Col d = column(1, yp, xpyp, xmyp, p[y2], c, ypzp, ypzm), e = column(1, ym, xpym, xmym, c, p[ym2], ymzp, ymzm);
    const Col f = column(2, zp, xpzp, xmzp, ypzp, ymzp, p[z2], c), g = column(2, zm, xpzm, xmzm, ypzm, ymzm, c, p[zm2]);
    Fx = -((R(0.5) * (a.x - b.x) + R(0.5) * (d.x - e.x)) + R(0.5) * (f.x - g.x));
    Fy = -((R(0.5) * (a.y - b.y) + R(0.5) * (d.y - e.y)) + R(0.5) * (f.y - g.y));
    Fz = -((R(0.5) * (a.z - b.z) + R(0.5) * (d.z - e.z)) + R(0.5) * (f.z - g.z));
}

// How the step's collision comes by mu and the force: from the fields that
// k_mu or k_stress wrote (kFar; kFarStress in FP32 storage with the stress
// force), or from phi itself, without those launches: kNearMu with the
// potential force, kNearStress with the stress force. The near forms take the
// 7-point stencils (the 19-point ones would need 19 phi at each of 18
// neighbours) and FP32 arithmetic (in FP64 they would add 60 and 200
// instructions to the pipe that bounds the step), so FP32 comes to the far
// ones with the 19-point stencils only. One FP32 kernel for both forces and
// either stencil held its 38 early loads through all of it and spilled: the
// stress force at 192^3 took 762 us a step (four launches a step before: 708),
// in a kernel of its own 640. The 16-bit forms load g after the f stores.
enum { kFar = 0, kNearMu = 1, kNearStress = 2, kFarStress = 3 };
__host__ __device__ constexpr bool is_near(int form) { return form == kNearMu || form == kNearStress; }
template <int P>
__host__ __device__ constexpr bool far_stress_apart() {
    return sizeof(typename Prec<P>::store_t) == 4;
}
template <int P>
int collide_form(const ld_ctx* c) {
    if (sizeof(typename Prec<P>::real_t) == 8) return kFar;
    if (c->prm.stencil == LD_STENCIL_7) return c->stress ? kNearStress : kNearMu;
    return far_stress_apart<P>() && c->stress ? kFarStress : kFar;
}

// Resident blocks per SM the collision kernel is compiled for: with FP32
// arithmetic 6 x 128 threads (80 registers), 5 (96) where it forms mu from phi;
// 3 with FP64.
template <int P, int FORM>
constexpr int rows_blocks_per_sm() {
    return sizeof(typename Prec<P>::real_t) == 4 ? (is_near(FORM) ? 5 : 6) : 3;
}

// Stage 3: force, velocity, collisions of f and g, and propagation (push: the
// post-collision value of direction i goes to x + c_i) with streaming stores;
// FORM: where mu and the force come from (near forms write mu to mu_out when
// it is not null); SR: the 16-bit stores rounded stochastically from `sr`.
template <int P, class I, int FORM, bool SR>
__global__ void __launch_bounds__(kRowThreads, (rows_blocks_per_sm<P, FORM>()))
    k_collide(RowGeom rg, I npad, Model<typename Prec<P>::real_t> m, SrStream sr, const typename Prec<P>::store_t* __restrict__ fs,
              const typename Prec<P>::store_t* __restrict__ gs, typename Prec<P>::store_t* __restrict__ fd,
              typename Prec<P>::store_t* __restrict__ gd, const typename Prec<P>::real_t* __restrict__ phi,
              const typename Prec<P>::real_t* __restrict__ mu, const float* __restrict__ ref,
              const typename Prec<P>::real_t* __restrict__ stress, typename Prec<P>::real_t* __restrict__ mu_out,
              int* __restrict__ status) {
    using R = typename Prec<P>::real_t;
    using S = typename Prec<P>::store_t;
    __shared__ float refs[2 * Q];  // codec references, read once per block
    if (threadIdx.x < 2 * Q) refs[threadIdx.x] = ref[threadIdx.x];
    __syncthreads();
    int x, y, z, s;
    if (!row_site(rg, x, y, z, s)) return;
    const long long n = rg.n;
    if (!site_ok(s, n, status)) return;
    // FP32 and FP64 issue all 38 loads first; the 16-bit forms issue g after
    // the f stores (each 16-bit value held early would take a register).
    constexpr bool kEarlyG = sizeof(S) >= 4;
    S fr[Q], gr[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        fr[i] = __ldcs(fs + i * npad + s);
        if (kEarlyG) gr[i] = __ldcs(gs + i * npad + s);
    }
    const RowNbr o = row_nbr(rg, x, y, z);
    const int oxp = o.xp, oxm = o.xm, oyp = o.yp, oym = o.ym, ozp = o.zp, ozm = o.zm;
    const R ph = phi[s];
    R muc, Fx, Fy, Fz;
    if constexpr (FORM == kNearStress) {
        stress_force_of_phi(rg, m, phi, x, y, z, s, o, status, muc, Fx, Fy, Fz);
        if (mu_out) mu_out[s] = muc;
    } else if constexpr (FORM == kNearMu) {
        R dx, dy, dz;
        mu_diffs_of_phi(rg, m, phi, x, y, z, s, o, status, muc, dx, dy, dz);
        force_of_diffs(ph, dx, dy, dz, Fx, Fy, Fz);
        if (mu_out) mu_out[s] = muc;
    } else {
        constexpr bool kApart = far_stress_apart<P>();
        const int iso = kApart ? 1 : m.iso;
        muc = mu[s];
        if (kApart ? FORM == kFarStress : stress != nullptr) {  // F = -div P
            stress_force_at(iso, stress, npad, s, o, Fx, Fy, Fz);
        } else if (iso) {  // F = -phi grad(mu)
            R gmx, gmy, gmz;
            grad_at(1, mu, s, o, gmx, gmy, gmz);
            Fx = -ph * gmx, Fy = -ph * gmy, Fz = -ph * gmz;
        } else {
            force_of_diffs(ph, mu[s + oxp] - mu[s + oxm], mu[s + oyp] - mu[s + oym], mu[s + ozp] - mu[s + ozm], Fx, Fy,
                           Fz);
        }
    }

    R f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = Prec<P>::decode(fr[i], refs[i]);
    R rho, jx, jy, jz;
    moments_f(f, rho, jx, jy, jz);
    R ux, uy, uz;
    guo_velocity(rho, jx, jy, jz, Fx, Fy, Fz, ux, uy, uz);
    if (m.trt)
        collide_f_trt(f, rho, ux, uy, uz, Fx, Fy, Fz, m);
    else
        collide_f(f, rho, ux, uy, uz, Fx, Fy, Fz, m);
    const unsigned long long sr_st = SR ? sr.base + (unsigned long long)s * kSrGamma : 0ull;
    unsigned long long sr_w = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int d = s + (cx(i) > 0 ? oxp : (cx(i) < 0 ? oxm : 0)) + (cy(i) > 0 ? oyp : (cy(i) < 0 ? oym : 0)) +
                      (cz(i) > 0 ? ozp : (cz(i) < 0 ? ozm : 0));
        S v;
        if constexpr (SR)
            v = Prec<P>::encode_sr(f[i], refs[i], sr_key(sr, sr_st, 0, i, sr_w));
        else
            v = Prec<P>::encode(f[i], refs[i]);
        if (site_ok(d, n, status)) __stcs(fd + i * npad + d, v);
    }
    R gg[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) gg[i] = Prec<P>::decode(kEarlyG ? gr[i] : __ldcs(gs + i * npad + s), refs[Q + i]);
    collide_g(gg, ph, muc, ux, uy, uz, m);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int d = s + (cx(i) > 0 ? oxp : (cx(i) < 0 ? oxm : 0)) + (cy(i) > 0 ? oyp : (cy(i) < 0 ? oym : 0)) +
                      (cz(i) > 0 ? ozp : (cz(i) < 0 ? ozm : 0));
        S v;
        if constexpr (SR)
            v = Prec<P>::encode_sr(gg[i], refs[Q + i], sr_key(sr, sr_st, 1, i, sr_w));
        else
            v = Prec<P>::encode(gg[i], refs[Q + i]);
        if (site_ok(d, n, status)) __stcs(gd + i * npad + d, v);
    }
}

// ---------------------------------------------------------------------------
// Initial state: f = feq(rho, u), g = geq(phi, u, mu(phi)), computed in the
// arithmetic type of the precision from the FP64 inputs, then encoded.
template <int P>
__global__ void __launch_bounds__(kThreads)
    k_init(Geom g, Model<typename Prec<P>::real_t> m, double rho0, const double* __restrict__ phi,
           const double* __restrict__ rho_in, const double* __restrict__ u_in, const float* __restrict__ ref,
           typename Prec<P>::store_t* __restrict__ fd, typename Prec<P>::store_t* __restrict__ gd) {
    using R = typename Prec<P>::real_t;
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.n) return;
    int x, y, z;
    site_coords(g, s, x, y, z);
    const R p = (R)phi[s];
    R lap;
    if (m.iso) {
        lap = R(0);
#pragma unroll
        for (int i = 1; i < Q; ++i)
            lap = init_mad(
                lap19_coef<R>(i),
                (R)phi[site_of(g, step_coord(x, cx(i), g.nx), step_coord(y, cy(i), g.ny), step_coord(z, cz(i), g.nz))] - p,
                lap);
    } else {
        lap = (R)phi[site_of(g, wrap_inc(x, g.nx), y, z)] + (R)phi[site_of(g, wrap_dec(x, g.nx), y, z)]
            + (R)phi[site_of(g, x, wrap_inc(y, g.ny), z)] + (R)phi[site_of(g, x, wrap_dec(y, g.ny), z)]
            + (R)phi[site_of(g, x, y, wrap_inc(z, g.nz))] + (R)phi[site_of(g, x, y, wrap_dec(z, g.nz))];
        lap = init_mad(R(-6), p, lap);
    }
    const R mu = init_mad(-m.kappa, lap, init_mad(m.A, p, m.B * p * p * p));
    const R rho = (R)(rho_in ? rho_in[s] : rho0);
    R ux = R(0), uy = R(0), uz = R(0);
    if (u_in) {
        ux = (R)u_in[s];
        uy = (R)u_in[g.n + s];
        uz = (R)u_in[2 * g.n + s];
    }
    equilibria(rho, p, mu, m.Gamma, ux, uy, uz, init_uu(ux, uy, uz), [&](int i, R feq, R geq) {
        fd[i * g.npad + s] = Prec<P>::encode_r(feq, ref[i]);
        gd[i * g.npad + s] = Prec<P>::encode_r(geq, ref[Q + i]);
    });
}

// Deviation references from the total of phi (in totals[0]): f_i: w_i rho0;
// g_i: geq_i(phibar, 0, A phibar + B phibar^3).
// Deviation references of the 16-bit forms: f_i w_i rho0; g_i geq_i(pb, 0, mu(pb))
// with pb the mean of the initial phi: totals[0] / n (mean_given = false) or
// `mean` itself (a part of a larger lattice that takes the whole one's mean).
__global__ void k_refs(const double* __restrict__ totals, long long n, double mean, int mean_given, Model<double> m,
                       double rho0, float* __restrict__ ref) {
    const int i = threadIdx.x;
    if (i >= Q) return;
    const double pb = mean_given ? mean : totals[0] / (double)n;
    const double mub = m.A * pb + m.B * pb * pb * pb;
    ref[i] = (float)(wgt<double>(i) * rho0);
    ref[Q + i] = (float)(wgt<double>(i) * (pb + 4.5 * (m.Gamma * mub - pb / 3.0) * (c2(i) - 1)));
}

__global__ void k_default_refs(double rho0, float* __restrict__ ref) {
    const int i = threadIdx.x;
    if (i >= Q) return;
    ref[i] = (float)(wgt<double>(i) * rho0);
    ref[Q + i] = 0.0f;
}

// ---------------------------------------------------------------------------
// Deterministic FP64 reductions: fixed grid, fixed per-thread order, fixed
// shuffle tree; then one ordered pass over the block partials.
template <int K>
__device__ __forceinline__ void block_sum_store(double (&v)[K], double* __restrict__ out_block) {
    __shared__ double red[kRedThreads / 32][K];
#pragma unroll
    for (int k = 0; k < K; ++k)
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) red[warp][k] = v[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double a = lane < kRedThreads / 32 ? red[lane][k] : 0.0;
            for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
            if (lane == 0) out_block[k] = a;
        }
    }
}

__global__ void __launch_bounds__(kRedThreads) k_sum_field(long long n, const double* __restrict__ x,
                                                           double* __restrict__ partials) {
    double v[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += stride) v[0] += x[s];
    block_sum_store<1>(v, partials + (long long)blockIdx.x * kRedFields);
}

// Sites per thread and iteration of k_totals: two where registers allow, to
// keep more bytes in flight (one site at a time took 0.50 ms at 256^3 in FP32
// and 1.58 ms in the 16-bit forms, whose 38 references were also read again at
// every site).
template <int P>
__host__ __device__ constexpr int totals_sites() {
    return sizeof(typename Prec<P>::store_t) == 8 ? 1 : 2;
}
// Blocks of k_totals: three per SM of the GPU's 152, one wave (a fixed number,
// so that the order of the sums does not depend on the device).
constexpr int kTotalsBlocks = 3 * 152;

// Each site's moments are summed in the arithmetic type of the precision (as
// the step itself forms them); sites accumulate in FP64.
template <int P>
__global__ void __launch_bounds__(kRedThreads, 3)
    k_totals(Geom g, const typename Prec<P>::store_t* __restrict__ fs,
             const typename Prec<P>::store_t* __restrict__ gs, const float* __restrict__ ref_g,
             double* __restrict__ partials) {
    using R = typename Prec<P>::real_t;
    using S = typename Prec<P>::store_t;
    constexpr int N = totals_sites<P>();
    using V = SiteVec<N, S>;
    __shared__ float ref[2 * Q];
    if (threadIdx.x < 2 * Q) ref[threadIdx.x] = ref_g[threadIdx.x];
    __syncthreads();
    const volatile float* vref = ref;  // read where used: 38 values held across the loop would spill
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const long long stride = (long long)gridDim.x * blockDim.x * N;
    for (long long s = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * N; s < g.n; s += stride) {
        // npad is a multiple of 64: the last vector may reach past n, into the
        // row's padding, whose sites are not added
        V fv[Q], gv[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            fv[i] = *reinterpret_cast<const V*>(fs + i * g.npad + s);
            gv[i] = *reinterpret_cast<const V*>(gs + i * g.npad + s);
        }
        R m[N][5] = {};
        if constexpr (sizeof(R) == 8) {
            R f[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                f[i] = fv[i].v[0];
                m[0][1] += gv[i].v[0];
            }
            moments_f(f, m[0][0], m[0][2], m[0][3], m[0][4]);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float rf = Prec<P>::kDev ? vref[i] : 0.0f, rg = Prec<P>::kDev ? vref[Q + i] : 0.0f;
#pragma unroll
                for (int e = 0; e < N; ++e) {
                    const R fi = Prec<P>::decode(fv[i].v[e], rf);
                    m[e][0] += fi;
                    add_c(i, fi, m[e][2], m[e][3], m[e][4]);
                    m[e][1] += Prec<P>::decode(gv[i].v[e], rg);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < N; ++e)
            if (s + e < g.n)
#pragma unroll
                for (int k = 0; k < 5; ++k) v[k] += (double)m[e][k];
    }
    block_sum_store<5>(v, partials + (long long)blockIdx.x * kRedFields);
}

// Final ordered pass: out[k] = sum over the nblocks blocks of partials[b][k].
__global__ void __launch_bounds__(kRedBlocks) k_finalize(const double* __restrict__ partials, int nblocks, int nfields,
                                                         double* __restrict__ out) {
    __shared__ double red[kRedBlocks / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < nfields; ++k) {
        double a = (int)threadIdx.x < nblocks ? partials[(long long)threadIdx.x * kRedFields + k] : 0.0;
        for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
        if (lane == 0) red[warp] = a;
        __syncthreads();
        if (warp == 0) {
            double b = red[lane];
            for (int off = 16; off > 0; off >>= 1) b += __shfl_down_sync(0xffffffffu, b, off);
            if (lane == 0) out[k] = b;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Macroscopic output (double): rho, u = (j + F/2)/rho, phi, grad phi.
//
// The outputs are FP64, and the FP64 pipe (two instructions per clock and SM)
// bounds this kernel: with 38 conversions, 95 additions and three divisions a
// site it took 5.70 ms at 256^3 in FP32 storage, where its bytes need 0.55
// ms. So FP32 and the 16-bit forms sum the stored values, which are floats, in
// FP32 arithmetic with every rounding error kept (Sum3), and widen floats to
// double with integer instructions: 27 FP64 instructions a site. Sites where
// that is not exact (a sum that leaves the range of floats, values that span
// more than 48 bits, subnormal values, NaN) take the FP64 form instead, a
// branch around a call: predicated instructions would occupy the FP64 pipe in
// every thread (measured: 72 instructions a site, 2.28 ms).

// x as a double times 2^-shift by integer instructions; clears ok unless x
// is zero or normal.
template <int shift>
__device__ __forceinline__ double widen(float x, bool& ok) {
    const unsigned u = (unsigned)__float_as_int(x), mag = u & 0x7fffffffu;
    ok = ok && (mag - 0x00800000u < 0x7f000000u || mag == 0u);
    const unsigned hi = mag == 0u ? 0u : (mag >> 3) + ((896u - shift) << 20);
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// A sum of floats s + e + t with the rounding errors of s kept in e and those
// of e in t (cascaded summation, Rump, Ogita & Oishi 2008).
struct Sum3 {
    float s, e, t;
    __device__ __forceinline__ static void two_sum(float& a, float b, float& err) {
        const float r = __fadd_rn(a, b), z = __fsub_rn(r, a);
        err = __fadd_rn(__fsub_rn(a, __fsub_rn(r, z)), __fsub_rn(b, z));
        a = r;
    }
    __device__ __forceinline__ void add(float x) {
        float r;
        two_sum(s, x, r);
        two_sum(e, r, r);
        t = __fadd_rn(t, r);
    }
    // s + e; clears ok unless that is the whole sum (t is NaN where s overflowed)
    __device__ __forceinline__ double value(bool& ok) const {
        ok = ok && t == 0.0f;
        return widen<0>(s, ok) + widen<0>(e, ok);
    }
};

// The arguments of k_macros (outputs may be null).
template <int P>
struct MacrosArgs {
    Geom g;
    const typename Prec<P>::store_t *fs, *gs;
    const typename Prec<P>::real_t *phi, *mu, *stress;  // stress: null unless F = -div P
    const float* ref;
    double *rho_out, *u_out, *phi_out, *gphi_out;
    int iso;
};

// One site. FAST: the float sums and integer conversions above; returns false,
// with nothing written, where they are not exact. ref_sum: the sums of the
// references of the deviation forms (sum r_i, sum q_i; r_i = r_-i, so they
// cancel in j).
template <int P, bool FAST>
__device__ __forceinline__ bool macros_site(const MacrosArgs<P>& a, unsigned s, const RowNbr& o, const float* ref,
                                            const double* ref_sum) {
    using R = typename Prec<P>::real_t;
    const long long n = a.g.n, npad = a.g.npad;
    const bool need_f = a.rho_out || a.u_out;
    bool ok = true;
    double rho = 0.0, ph, j[3];
    if constexpr (FAST) {
        Sum3 r{0.0f, 0.0f, 0.0f}, x = r, y = r, z = r, p = r;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            p.add(to_float(a.gs[i * npad + s]));
            if (!need_f) continue;
            const float v = to_float(a.fs[i * npad + s]);
            r.add(v);
            if (cx(i) != 0) x.add(cx(i) > 0 ? v : -v);
            if (cy(i) != 0) y.add(cy(i) > 0 ? v : -v);
            if (cz(i) != 0) z.add(cz(i) > 0 ? v : -v);
        }
        rho = r.value(ok);
        ph = p.value(ok);
        j[0] = x.value(ok);
        j[1] = y.value(ok);
        j[2] = z.value(ok);
        if (Prec<P>::kDev) {
            rho += ref_sum[0];
            ph += ref_sum[1];
        }
    } else {
        if (need_f) {
            double f[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) f[i] = Prec<P>::decode_d(a.fs[i * npad + s], ref[i]);
            moments_f(f, rho, j[0], j[1], j[2]);
        }
        ph = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) ph += Prec<P>::decode_d(a.gs[i * npad + s], ref[Q + i]);
    }
    // the difference of two field values, and half of it
    auto diff = [&](const R* h, int d0, int d1) -> double {
        if constexpr (FAST)
            return widen<0>(h[s + d0], ok) - widen<0>(h[s + d1], ok);
        else
            return (double)h[s + d0] - (double)h[s + d1];
    };
    auto half_diff = [&](const R* h, int d0, int d1) -> double {
        if constexpr (FAST)
            return widen<1>(h[s + d0], ok) - widen<1>(h[s + d1], ok);
        else
            return 0.5 * ((double)h[s + d0] - (double)h[s + d1]);
    };
    // gradient of a field with the selected stencil
    auto grad = [&](const R* h, double (&v)[3]) {
        if (a.iso) {  // from the differences of opposite neighbours: axis 1/6, diagonal 1/12
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = 2.0 * diff(h, o.of(2 * c + 1), o.of(2 * c + 2));
#pragma unroll
            for (int i = 7; i < Q; i += 2) add_c(i, diff(h, o.of(i), o.of(i + 1)), v[0], v[1], v[2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] *= 1.0 / 12.0;
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = half_diff(h, o.of(2 * c + 1), o.of(2 * c + 2));
        }
    };
    double u[3], gp[3];
    if (a.u_out) {
        double num[3];  // j + F/2
        if (a.stress) {  // F = -div P
            double d[6][3];
#pragma unroll
            for (int c = 0; c < 6; ++c) grad(a.stress + c * npad, d[c]);
            num[0] = __fma_rn(-0.5, (d[0][0] + d[3][1]) + d[4][2], j[0]);
            num[1] = __fma_rn(-0.5, (d[3][0] + d[1][1]) + d[5][2], j[1]);
            num[2] = __fma_rn(-0.5, (d[4][0] + d[5][1]) + d[2][2], j[2]);
        } else {  // F = -phi grad(mu)
            double gm[3];
            grad(a.mu, gm);
            const double h = -0.5 * ph;
#pragma unroll
            for (int c = 0; c < 3; ++c) num[c] = __fma_rn(h, gm[c], j[c]);
        }
        double inv;
        if constexpr (FAST) {  // 1/rho to about 46 bits, which the residuals of div_by take to the last
            const float f = (float)rho;
            const double r = widen<0>(__frcp_rn(f), ok);
            ok = ok && fabsf(f) > 1e-30f && fabsf(f) < 1e30f;
            inv = __fma_rn(__fma_rn(-rho, r, 1.0), r, r);
        } else {
            inv = __drcp_rn(rho);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = div_by(num[c], rho, inv);
        if constexpr (!FAST) {  // (FAST takes only densities within the range of floats)
            if (__builtin_expect(any_nonfinite(u[0], u[1], u[2]), 0)) {
                // j is the sum of c_i f_i over every i: an infinite f_i leaves no component of it a value
                double z = 0.0;
#pragma unroll 1
                for (int i = 0; i < Q; ++i) z = __fma_rn(0.0, Prec<P>::decode_d(a.fs[i * npad + s], ref[i]), z);
#pragma unroll
                for (int c = 0; c < 3; ++c) u[c] = z == 0.0 ? __ddiv_rn(num[c], rho) : z;
            }
        }
    }
    if (a.gphi_out) grad(a.phi, gp);
    if (FAST && !ok) return false;
    if (a.rho_out) a.rho_out[s] = rho;
    if (a.phi_out) a.phi_out[s] = ph;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (a.u_out) a.u_out[c * n + s] = u[c];
        if (a.gphi_out) a.gphi_out[c * n + s] = gp[c];
    }
    return true;
}
template <int P>
__device__ __noinline__ void macros_site_exact(const MacrosArgs<P>& a, unsigned s, const RowNbr& o) {
    macros_site<P, false>(a, s, o, a.ref, nullptr);
}

template <int P>
__global__ void __launch_bounds__(kThreads, 4) k_macros(const __grid_constant__ MacrosArgs<P> a) {
    constexpr bool kFast = sizeof(typename Prec<P>::store_t) < 8;
    __shared__ double ref_sum[2];
    if (Prec<P>::kDev) {
        if (threadIdx.x < 2) {
            double v = 0.0;
            for (int i = 0; i < Q; ++i) v += (double)a.ref[threadIdx.x * Q + i];
            ref_sum[threadIdx.x] = v;
        }
        __syncthreads();
    }
    const unsigned s = blockIdx.x * blockDim.x + threadIdx.x;  // n < 2^31
    if (s >= a.g.n) return;
    const unsigned row = s / (unsigned)a.g.nx;
    const int x = (int)(s - row * (unsigned)a.g.nx), z = (int)(row / (unsigned)a.g.ny);
    const RowNbr o = row_nbr(RowGeom{a.g.nx, a.g.ny, a.g.nz, 0, {}, {}}, x, (int)(row - (unsigned)z * a.g.ny), z);
    if constexpr (kFast) {
        if (!macros_site<P, true>(a, s, o, a.ref, ref_sum)) macros_site_exact<P>(a, s, o);
    } else {
        macros_site<P, false>(a, s, o, a.ref, nullptr);
    }
}

// Distributions out (decoded, stride n) and in (encoded).
template <int P>
__global__ void __launch_bounds__(kThreads) k_decode(Geom g, const typename Prec<P>::store_t* __restrict__ src,
                                                     const float* __restrict__ ref, double* __restrict__ out) {
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.n) return;
#pragma unroll
    for (int i = 0; i < Q; ++i) out[i * g.n + s] = Prec<P>::decode_d(src[i * g.npad + s], ref[i]);
}

template <int P>
__global__ void __launch_bounds__(kThreads) k_encode(Geom g, const double* __restrict__ in,
                                                     const float* __restrict__ ref,
                                                     typename Prec<P>::store_t* __restrict__ dst) {
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.n) return;
#pragma unroll
    for (int i = 0; i < Q; ++i) dst[i * g.npad + s] = Prec<P>::encode_d(in[i * g.n + s], ref[i]);
}

// Propagation alone on raw storage words (T has the storage width).
template <class T>
__global__ void __launch_bounds__(kThreads) k_propagate(Geom g, int reverse, const T* __restrict__ src,
                                                        T* __restrict__ dst) {
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.n) return;
    int x, y, z;
    site_coords(g, s, x, y, z);
#pragma unroll
    for (int i = 0; i < 2 * Q; ++i) {  // f components then g components
        const int q = i % Q;
        const long long o = site_of(g, step_coord(x, cx(q), g.nx), step_coord(y, cy(q), g.ny),
                                    step_coord(z, cz(q), g.nz));
        if (reverse)
            dst[i * g.npad + s] = src[i * g.npad + o];
        else
            dst[i * g.npad + o] = src[i * g.npad + s];
    }
}

// ---------------------------------------------------------------------------
template <int P>
cudaError_t init_p(ld_ctx* c, const double* phi, const double* rho, const double* u, const double* ref_mean) {
    using S = typename Prec<P>::store_t;
    const Geom g = to_dev(c->geom);
    const Model<double> m = model_of<double>(c->prm);
    if (Prec<P>::kDev) {
        if (!ref_mean) {
            k_sum_field<<<kRedBlocks, kRedThreads, 0, c->stream>>>(g.n, phi, c->partials);
            k_finalize<<<1, kRedBlocks, 0, c->stream>>>(c->partials, kRedBlocks, 1, c->totals);
        }
        k_refs<<<1, 32, 0, c->stream>>>(c->totals, g.n, ref_mean ? *ref_mean : 0.0, ref_mean ? 1 : 0, m, c->prm.rho0,
                                        c->ref);
    } else {
        k_default_refs<<<1, 32, 0, c->stream>>>(c->prm.rho0, c->ref);
    }
    k_init<P><<<blocks_for(g.n), kThreads, 0, c->stream>>>(g, model_of<typename Prec<P>::real_t>(c->prm),
                                                           c->prm.rho0, phi, rho, u, c->ref,
                                                           (S*)f_of(c, c->cur), (S*)g_of(c, c->cur));
    return cudaGetLastError();
}

inline bool offsets_fit_int(const ld_ctx* c) { return (long long)Q * c->geom.npad <= 0x7fffffffLL; }

template <int P, class I>
void launch_phi(ld_ctx* c, const void* state, typename Prec<P>::real_t* phi) {
    using S = typename Prec<P>::store_t;
    constexpr int N = phi_sites<P>();
    const S* gs = (const S*)g_part(c, state);
    const unsigned nb = row_blocks(c->geom);
    // a caller's state or fields buffer may be aligned to single values only
    if (N > 1 && (uintptr_t)gs % (N * sizeof(S)) == 0 && (uintptr_t)phi % (N * sizeof(*phi)) == 0)
        k_phi<P, I, N><<<(nb + N - 1) / N, kRowThreads, 0, c->stream>>>((int)c->geom.n, (I)c->geom.npad, gs, c->ref, phi,
                                                                        c->status);
    else
        k_phi<P, I, 1><<<nb, kRowThreads, 0, c->stream>>>((int)c->geom.n, (I)c->geom.npad, gs, c->ref, phi, c->status);
}

// mu from phi, and the chemical stress where the force is its divergence.
template <class R, class I>
void launch_mu(ld_ctx* c, const R* phi, R* mu) {
    const unsigned nb = row_blocks(c->geom);
    if (c->stress)
        k_stress<R, I><<<nb, kRowThreads, 0, c->stream>>>(row_geom(c->geom), (I)c->geom.npad, model_of<R>(c->prm), phi,
                                                          (R*)c->stress, mu);
    else
        k_mu<R><<<nb, kRowThreads, 0, c->stream>>>(row_geom(c->geom), model_of<R>(c->prm), phi, mu);
}

// phi and mu of a state (and the stress) into the context's scratch.
template <int P>
cudaError_t phi_mu_p(ld_ctx* c, const void* state) {
    using R = typename Prec<P>::real_t;
    if (offsets_fit_int(c)) {
        launch_phi<P, int>(c, state, (R*)c->phi);
        launch_mu<R, int>(c, (const R*)c->phi, (R*)c->mu);
    } else {
        launch_phi<P, long long>(c, state, (R*)c->phi);
        launch_mu<R, long long>(c, (const R*)c->phi, (R*)c->mu);
    }
    return cudaGetLastError();
}

// One step; phi and mu of the source state go to `fields` ([phi npad][mu
// npad]) when it is not null, else to the context's scratch.
template <int P, class I, int FORM, bool SR>
cudaError_t collide_rows(ld_ctx* c, const void* src, void* dst, void* fields) {
    using S = typename Prec<P>::store_t;
    using R = typename Prec<P>::real_t;
    R* phi = fields ? (R*)fields : (R*)c->phi;
    R* mu = fields ? (R*)fields + c->geom.npad : (R*)c->mu;
    launch_phi<P, I>(c, src, phi);
    if (!is_near(FORM)) launch_mu<R, I>(c, phi, mu);
    k_collide<P, I, FORM, SR><<<row_blocks(c->geom), kRowThreads, 0, c->stream>>>(
        row_geom(c->geom), (I)c->geom.npad, model_of<R>(c->prm), sr_stream(c->prm.seed, c->sr_step, c->geom.n),
        (const S*)f_part(c, src), (const S*)g_part(c, src), (S*)f_part(c, dst), (S*)g_part(c, dst), phi,
        is_near(FORM) ? nullptr : mu, c->ref, (const R*)c->stress, is_near(FORM) && fields ? mu : nullptr, c->status);
    return cudaGetLastError();
}

template <int P, int FORM, bool SR>
cudaError_t collide_r(ld_ctx* c, const void* src, void* dst, void* fields) {
    return offsets_fit_int(c) ? collide_rows<P, int, FORM, SR>(c, src, dst, fields)
                              : collide_rows<P, long long, FORM, SR>(c, src, dst, fields);
}

template <int P, bool SR>
cudaError_t collide_n(ld_ctx* c, const void* src, void* dst, void* fields) {
    if constexpr (sizeof(typename Prec<P>::real_t) == 4) {
        switch (collide_form<P>(c)) {
            case kNearMu: return collide_r<P, kNearMu, SR>(c, src, dst, fields);
            case kNearStress: return collide_r<P, kNearStress, SR>(c, src, dst, fields);
            case kFarStress:
                if constexpr (far_stress_apart<P>()) return collide_r<P, kFarStress, SR>(c, src, dst, fields);
        }
    }
    return collide_r<P, kFar, SR>(c, src, dst, fields);
}

template <int P>
cudaError_t collide_p(ld_ctx* c, const void* src, void* dst, void* fields) {
    if constexpr (Prec<P>::kDev) {
        if (c->prm.rounding == LD_ROUND_STOCHASTIC) return collide_n<P, true>(c, src, dst, fields);
    }
    return collide_n<P, false>(c, src, dst, fields);
}

template <int P>
cudaError_t macros_p(ld_ctx* c, double* rho, double* u, double* phi, double* gphi) {
    using S = typename Prec<P>::store_t;
    using R = typename Prec<P>::real_t;
    const Geom g = to_dev(c->geom);
    if (u || gphi) {
        const cudaError_t e = phi_mu_p<P>(c, c->dist[c->cur]);
        if (e != cudaSuccess) return e;
    }
    k_macros<P><<<blocks_for(g.n), kThreads, 0, c->stream>>>(
        MacrosArgs<P>{g, (const S*)f_of(c, c->cur), (const S*)g_of(c, c->cur), (const R*)c->phi, (const R*)c->mu,
                      (const R*)c->stress, c->ref, rho, u, phi, gphi, c->prm.stencil == LD_STENCIL_19});
    return cudaGetLastError();
}

template <int P>
cudaError_t totals_p(ld_ctx* c, double* out) {
    using S = typename Prec<P>::store_t;
    const Geom g = to_dev(c->geom);
    k_totals<P><<<kTotalsBlocks, kRedThreads, 0, c->stream>>>(g, (const S*)f_of(c, c->cur), (const S*)g_of(c, c->cur),
                                                           c->ref, c->partials);
    k_finalize<<<1, kRedBlocks, 0, c->stream>>>(c->partials, kTotalsBlocks, 5, out);
    return cudaGetLastError();
}

template <int P>
cudaError_t decode_p(ld_ctx* c, double* f, double* gout) {
    using S = typename Prec<P>::store_t;
    const Geom g = to_dev(c->geom);
    if (f) k_decode<P><<<blocks_for(g.n), kThreads, 0, c->stream>>>(g, (const S*)f_of(c, c->cur), c->ref, f);
    if (gout)
        k_decode<P><<<blocks_for(g.n), kThreads, 0, c->stream>>>(g, (const S*)g_of(c, c->cur), c->ref + Q, gout);
    return cudaGetLastError();
}

template <int P>
cudaError_t encode_p(ld_ctx* c, const double* f, const double* gin) {
    using S = typename Prec<P>::store_t;
    const Geom g = to_dev(c->geom);
    if (f) k_encode<P><<<blocks_for(g.n), kThreads, 0, c->stream>>>(g, f, c->ref, (S*)f_of(c, c->cur));
    if (gin) k_encode<P><<<blocks_for(g.n), kThreads, 0, c->stream>>>(g, gin, c->ref + Q, (S*)g_of(c, c->cur));
    return cudaGetLastError();
}


// Precision-independent launches.
cudaError_t default_refs(ld_ctx* c) {
    k_default_refs<<<1, 32, 0, c->stream>>>(c->prm.rho0, c->ref);
    return cudaGetLastError();
}

cudaError_t propagate_raw(ld_ctx* c, int reverse) {
    const Geom g = to_dev(c->geom);
    const void* src = c->dist[c->cur];
    void* dst = c->dist[1 - c->cur];
    const unsigned nb = blocks_for(g.n);
    switch (c->store_bytes) {
        case 8:
            k_propagate<unsigned long long><<<nb, kThreads, 0, c->stream>>>(g, reverse, (const unsigned long long*)src,
                                                                            (unsigned long long*)dst);
            break;
        case 4:
            k_propagate<unsigned int><<<nb, kThreads, 0, c->stream>>>(g, reverse, (const unsigned int*)src,
                                                                      (unsigned int*)dst);
            break;
        case 2:
            k_propagate<unsigned short><<<nb, kThreads, 0, c->stream>>>(g, reverse, (const unsigned short*)src,
                                                                        (unsigned short*)dst);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace
}  // namespace ld
