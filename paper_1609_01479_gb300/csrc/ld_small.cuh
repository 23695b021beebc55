// The step of a small lattice: one launch, each site collided by one thread,
// as many CTAs as the lattice gives.
//
// A lattice of a few hundred thousand sites lives in L2, and its step is bound
// by latency: the z-marching kernel (ld_fused.cuh) gives a 32^3 lattice 32 CTAs
// for 152 SMs, each of them eight planes of dependent phases, and the
// site-ordered launches of other sizes two or three launches a step. Here a CTA of 256
// threads owns a tile of 32 x 4 x 2 sites and runs three phases, each once:
//   1. all loads at once: the thread's own f and g, and the g of the tile's
//      2-site halo, summed to phi in shared memory;
//   2. mu over the tile and its 1-site halo;
//   3. force, collisions and push of the thread's site.
// The phi sums of the halo are repeated between CTAs (4.1 sites of g per site
// with the 7-point stencils, 5.8 with the 19-point ones, from L2), which costs
// bandwidth that a lattice of this size does not use. Any lattice size: tiles may reach past the lattice, and the
// halo wraps any number of times.
// Consecutive steps overlap their launches: each launch lets the next one
// start its CTAs at once (programmatic dependent launch), which compute their
// indices and then wait for the whole previous launch before they touch
// memory.
// The operations of every site are those of k_step_fused and k_collide, so the
// bits do not depend on the size (a lattice and its slabs may be on different
// sides of the line). FP32 only: the 16-bit forms' kernels for large lattices
// round their FP32 arithmetic differently (packed pairs, decoded values), and a
// third order for small ones would make a run's bits depend on its size.
#pragma once
#include "ld_async.cuh"
#include "ld_common.cuh"
#include "ld_fused.cuh"
#include "ld_internal.h"

namespace ld {
namespace {

constexpr int kSmX = 32, kSmY = 4, kSmZ = 2, kSmThreads = kSmX * kSmY * kSmZ;

__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Rows of the halo frame, (y, z) relative to the tile, whose phi the tile
// needs besides its own: 7-point forms reach two sites in total (28 rows),
// the 19-point ones the whole box (40 rows).
template <bool ISO>
__host__ __device__ constexpr int small_halo_rows() {
    return ISO ? (kSmY + 4) * (kSmZ + 4) - kSmY * kSmZ : 2 * kSmY + 2 * (kSmY + 2) + 4 * kSmZ;
}
template <bool ISO>
__device__ __forceinline__ void small_halo_row(int r, int& hy, int& hz) {
    if constexpr (ISO) {
        constexpr int H = kSmY + 4;
        if (r < 4 * H) {  // the four planes outside the tile
            const int p = r / H;
            hy = r % H - 2;
            hz = p < 2 ? p - 2 : kSmZ + p - 2;
        } else {
            const int q = r - 4 * H, e = q & 3;
            hz = q >> 2;
            hy = e < 2 ? e - 2 : kSmY + e - 2;
        }
    } else {
        constexpr int A = 2 * kSmY, B = 2 * (kSmY + 2);
        if (r < A) {
            hz = r < kSmY ? -2 : kSmZ + 1;
            hy = r % kSmY;
        } else if (r < A + B) {
            const int q = r - A;
            hz = q < kSmY + 2 ? -1 : kSmZ;
            hy = q % (kSmY + 2) - 1;
        } else {
            const int q = r - A - B, e = q & 3;
            hz = q >> 2;
            hy = e < 2 ? e - 2 : kSmY + e - 2;
        }
    }
}

// Periodic image of any coordinate.
__device__ __forceinline__ int wrap_any(int a, int n) {
    a %= n;
    return a < 0 ? a + n : a;
}

template <bool ISO>
__global__ void __launch_bounds__(kSmThreads, 2)
    k_step_small(Geom g, Model<float> m, const float* fs, const float* gs, float* fd, float* gd, float* phi_out,
                 float* mu_out, int* status) {
    // no __restrict__: the compiler may move loads it knows to be invariant
    // above the wait for the previous launch
    constexpr int PW = kSmX + 4, PH = kSmY + 4, PD = kSmZ + 4;
    constexpr int MW = kSmX + 2, MH = kSmY + 2, MD = kSmZ + 2;
    constexpr int kRows = small_halo_rows<ISO>(), kWarps = kSmThreads / 32;
    __shared__ float phis[PD][PH][PW];
    __shared__ float mus[MD][MH][MW];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = g.nx, ny = g.ny, nz = g.nz, plane = nx * ny;
    const int npad = (int)g.npad;  // 19 npad fits an int (launch_small)
    const int x0 = blockIdx.x * kSmX, y0 = blockIdx.y * kSmY, z0 = blockIdx.z * kSmZ;
    const int ty = warp % kSmY, tz = warp / kSmY;
    const int x = x0 + lane, y = y0 + ty, z = z0 + tz;
    const bool on = x < nx && y < ny && z < nz;
    const int s = on ? z * plane + y * nx + x : 0;
    // sites whose phi this thread forms: its column of every kWarps-th halo
    // row, and one of the four columns beside the tile
    constexpr int kMine = (kRows + kWarps - 1) / kWarps;
    int hs[kMine];
    const int wx = wrap_any(x, nx);
#pragma unroll
    for (int k = 0; k < kMine; ++k) {
        int hy = 0, hz = 0;
        const int r = warp + k * kWarps;
        if (r < kRows) small_halo_row<ISO>(r, hy, hz);
        hs[k] = wrap_any(z0 + hz, nz) * plane + wrap_any(y0 + hy, ny) * nx + wx;
    }
    constexpr int kSide = 4 * (kRows + kSmY * kSmZ);
    static_assert(kSide <= kSmThreads, "one side site per thread");
    int sy = 0, sz = 0, ss = 0;
    const int sx = (tid & 3) < 2 ? (tid & 3) - 2 : kSmX + (tid & 3) - 2;
    if (tid < kSide) {
        const int r = tid >> 2;
        if (r < kRows) {
            small_halo_row<ISO>(r, sy, sz);
        } else {
            sy = (r - kRows) % kSmY;
            sz = (r - kRows) / kSmY;
        }
        ss = wrap_any(z0 + sz, nz) * plane + wrap_any(y0 + sy, ny) * nx + wrap_any(x0 + sx, nx);
    }
    const int oxp = x + 1 == nx ? 1 - nx : 1, oxm = x == 0 ? nx - 1 : -1;
    const int oyp = y + 1 == ny ? (1 - ny) * nx : nx, oym = y == 0 ? (ny - 1) * nx : -nx;
    const int ozp = z + 1 == nz ? (1 - nz) * plane : plane, ozm = z == 0 ? (nz - 1) * plane : -plane;

    pdl_launch_next();
    pdl_wait_previous();
    // own g and f; tiles may reach past the lattice: such threads take the
    // wrapped site's phi (it may be another's halo) and collide nothing
    const int own = wrap_any(z, nz) * plane + wrap_any(y, ny) * nx + wx;
    const bool ook = site_ok(own, g.n, status);
    float gr[Q], fr[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) gr[i] = ook ? gs[i * npad + own] : 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) fr[i] = on && ook ? fs[i * npad + own] : 0.0f;
    auto phi_of = [&](int site) {
        float a = 0.0f;
        if (site_ok(site, g.n, status)) {
#pragma unroll
            for (int i = 0; i < Q; ++i) a += gs[i * npad + site];
        }
        return a;
    };
#pragma unroll
    for (int k = 0; k < kMine; ++k) {
        const int r = warp + k * kWarps;
        if (r < kRows) {
            int hy, hz;
            small_halo_row<ISO>(r, hy, hz);
            phis[hz + 2][hy + 2][lane + 2] = phi_of(hs[k]);
        }
    }
    if (tid < kSide) phis[sz + 2][sy + 2][sx + 2] = phi_of(ss);
    float ph = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) ph += gr[i];
    phis[tz + 2][ty + 2][lane + 2] = ph;
    __syncthreads();

    for (int idx = tid; idx < MW * MH * MD; idx += kSmThreads) {
        const int mx = idx % MW, r = idx / MW, my = r % MH, mz = r / MH;
        const bool edge_y = my == 0 || my == MH - 1, edge_z = mz == 0 || mz == MD - 1;
        if (!ISO && edge_y && edge_z) continue;  // its phi is not formed, and no force reads it
        const float c = phis[mz + 1][my + 1][mx + 1];
        float lap;
        if constexpr (ISO) {
            auto nb = [&](int i) { return phis[mz + 1 + cz(i)][my + 1 + cy(i)][mx + 1 + cx(i)]; };
            lap = lap19(c, nb);
        } else {
            const float nb = phis[mz + 1][my + 1][mx + 2] + phis[mz + 1][my + 1][mx] + phis[mz + 1][my + 2][mx + 1] +
                             phis[mz + 1][my][mx + 1] + phis[mz + 2][my + 1][mx + 1] + phis[mz][my + 1][mx + 1];
            lap = lap7(c, nb);
        }
        mus[mz][my][mx] = chem_potential_lap(c, lap, m);
    }
    __syncthreads();
    if (!on) return;

    const float muc = mus[tz + 1][ty + 1][lane + 1];
    float gmx, gmy, gmz;
    if constexpr (ISO) {
        auto nb = [&](int i) { return mus[tz + 1 + cz(i)][ty + 1 + cy(i)][lane + 1 + cx(i)]; };
        grad19(nb, gmx, gmy, gmz);
    } else {
        gmx = 0.5f * (mus[tz + 1][ty + 1][lane + 2] - mus[tz + 1][ty + 1][lane]);
        gmy = 0.5f * (mus[tz + 1][ty + 2][lane + 1] - mus[tz + 1][ty][lane + 1]);
        gmz = 0.5f * (mus[tz + 2][ty + 1][lane + 1] - mus[tz][ty + 1][lane + 1]);
    }
    const float Fx = -ph * gmx, Fy = -ph * gmy, Fz = -ph * gmz;
    if (phi_out && ook) {  // fields of the source state, for the adjoint
        phi_out[s] = ph;
        mu_out[s] = muc;
    }
    auto push = [&](float* dst, const float (&v)[Q]) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int d = s + (cx(i) > 0 ? oxp : (cx(i) < 0 ? oxm : 0)) + (cy(i) > 0 ? oyp : (cy(i) < 0 ? oym : 0)) +
                          (cz(i) > 0 ? ozp : (cz(i) < 0 ? ozm : 0));
            if (site_ok(d, g.n, status)) dst[i * npad + d] = v[i];
        }
    };
    float rho, jx, jy, jz, ux, uy, uz;
    moments_f(fr, rho, jx, jy, jz);
    guo_velocity(rho, jx, jy, jz, Fx, Fy, Fz, ux, uy, uz);
    collide_f(fr, rho, ux, uy, uz, Fx, Fy, Fz, m);
    push(fd, fr);
    collide_g(gr, ph, muc, ux, uy, uz, m);
    push(gd, gr);
}

inline cudaError_t launch_small(ld_ctx* c, const void* src, void* dst, void* fields) {
    const Geom g{c->geom.nx, c->geom.ny, c->geom.nz, c->geom.n, c->geom.npad};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((g.nx + kSmX - 1) / kSmX, (g.ny + kSmY - 1) / kSmY, (g.nz + kSmZ - 1) / kSmZ);
    cfg.blockDim = dim3(kSmThreads);
    cfg.stream = c->stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const auto kernel = c->prm.stencil == LD_STENCIL_19 ? k_step_small<true> : k_step_small<false>;
    return cudaLaunchKernelEx(&cfg, kernel, g, model_of<float>(c->prm), (const float*)f_part(c, src),
                              (const float*)g_part(c, src), (float*)f_part(c, dst), (float*)g_part(c, dst),
                              (float*)fields, fields ? (float*)fields + c->geom.npad : (float*)nullptr, c->status);
}

}  // namespace

// Lattices that LD_KERNEL_AUTO gives to k_step_small, by its tiles of 32 x 4 x 2
// sites: a tile costs about the same however many of its sites are the
// lattice's, so a lattice 4 sites wide pays for 8 times its own. Up to 304 tiles
// (two CTAs per SM) are one wave; beyond it the time grows by a wave of 3 to 5
// us, while the other kernels start from two launches (8.3 us, three with the
// 19-point stencils 12.4 to 14.4) or from the z-march's chunk (15 to 17 us) and
// stay there to some 30k to 130k sites. The lines lie where 223 measured
// lattices of 1k to 512k sites, 4 to 1000 wide, put them, us a step of this
// kernel and of the one AUTO takes otherwise:
//   row launches, 7-point   20 x 57 x 57, 435 tiles: 8.6, 10.3; 4 x 64 x 64, 512:
//     9.7, 8.3; 33 x 45 x 44, 528: 12.0, 10.3; 64 x 45 x 45, 552: 12.3, 12.4;
//     50 x 61 x 47, 768: 17.1, 14.4; 33 x 63 x 63, 1024: 20.0, 14.2; 4 x 128 x 128,
//     2048: 31, 10. From 448 tiles on it also depends on how full they are
//     (n/432): 31 x 65 x 65, 561: 12.2, 13.9; 60^3, 900: 19.7, 20.6.
//   row launches, 19-point  45^3, 552: 15.0, 16.5; 48 x 52 x 52, 676: 17.6, 18.6;
//     50 x 61 x 47, 768: 20.4, 18.5; 33 x 65 x 65, 1122: 25.9, 18.5
//   z-march, 7-point        32^3, 128: 5.9, 14.5; 96 x 96 x 24, 864: 19.5, 22.7;
//     64^3, 1024: 23.0, 22.7; 32 x 128 x 64, 1024: 22.3, 20.7; 19-point 96 x 96 x 24:
//     23.2, 24.7; 64^3: 26.6, 24.7
// The choice costs at most 10 % against the faster kernel on any of them and of
// 110 others, 0.1 to 0.2 % on average; by sites alone (up to 2^18) it cost up to
// a factor of 5.8, 7 % on average of the 110.
inline bool small_supported_impl(int nx, int ny, int nz, int stencil, bool tiled) {
    const long long n = (long long)nx * ny * nz;
    const long long tiles = (long long)((nx + kSmX - 1) / kSmX) * ((ny + kSmY - 1) / kSmY) * ((nz + kSmZ - 1) / kSmZ);
    if (tiled) return tiles <= 912;
    if (stencil == LD_STENCIL_19) return tiles <= 704;
    return tiles <= 448 || tiles <= 300 + n / 432;
}

}  // namespace ld
