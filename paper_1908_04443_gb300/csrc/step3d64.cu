// D3Q19 FP64 step and fields pass: bricks whose shape is chosen per grid.
//
// A CTA owns a w x h column and marches it through zc planes.  For lead plane zl it pulls (Eq. 3, Fig. 3)
// its nodes and their 1-node xy ring (2-node ring near solids) for density (Eq. 4) and psi (Eq. 6) into
// rings of planes, gives the wall cells of plane zl - 1 their virtual densities (Eqs. 16-17), and collides
// plane zl - 1 (zl - 2 near solids), whose distributions it pulls again.
// Bound by the FP64 pipe (fp64.cuh), as in 2D: a plane of 16 x 8 nodes keeps it busy for 20,000 clocks, so
// the second pull costs nothing beside it, and what counts is FP64 instructions and an equal share of
// them for every SM, with several bricks on each to hide one another's latency.  d3q19_fp64_brick weighs
// the halo's share (36 instructions a cell against 283 a node) against both.  A 64^3 step: 789 us in
// 32 x 4 x 32 bricks on 64 of 152 SMs with the general functions, 206 us here.
#include "fp64.cuh"
#include "kernels.h"
#include "lattice.cuh"
#include "pdl.cuh"
#include "tile_common.cuh"

namespace lbmwet {

namespace {

constexpr int NT = 128, RESIDENT = 4;       // threads (a column holds up to NT nodes), CTAs per SM
constexpr int MW = 32;                      // widest column (nodes); heights up to NT / width
// planes of the largest column (32 x 4; 16 x 8 and 8 x 16 are smaller), ring cells included
constexpr int PCELLS = 34 * 6, RCELLS = 36 * 8, YCELLS = 38 * 10;
static_assert(18 * 10 <= PCELLS && 20 * 12 <= RCELLS && 22 * 14 <= YCELLS, "16 x 8 columns");

struct Smem {
    double rho[4][RCELLS];
    double psi[5][PCELLS];
    uint8_t type[8][YCELLS];
};

template <int MODE, bool SOLID>
__device__ __forceinline__ void brick64(const double* __restrict__ fin, double* __restrict__ fout, const Geo& g,
                                        const Phys<double>& ph, int x0, int y0, int zb, int wl, int h, int zc,
                                        unsigned* err, double* __restrict__ rho_out, double* __restrict__ u_out, Smem& sm) {
    using L = D3Q19;
    constexpr int Q = 19, LAG = SOLID ? 2 : 1;
    const int nx = g.nx, ny = g.ny, nz = g.nz, N = g.N, nxy = nx * ny;
    const int tid = threadIdx.x, w = 1 << wl;
    const int we = min(w, nx - x0), he = min(h, ny - y0), ze = min(zb + zc, nz);
    const bool small = nx < MW + 8 || ny < NT / 8 + 8 || nz < 8;
    auto wx = [&](int v) { return small ? wrap_full(v, nx) : wrap1(v, nx); };
    auto wy = [&](int v) { return small ? wrap_full(v, ny) : wrap1(v, ny); };
    auto wz = [&](int v) { return small ? wrap_full(v, nz) : wrap1(v, nz); };
    // cells relative to the column's first node; pitches of the column's own width
    const int PX = w + 2, RX = w + 4, YX = w + 6;
    auto pix = [&](int cx, int cy) { return (cy + 1) * PX + cx + 1; };
    auto rix = [&](int cx, int cy) { return (cy + 2) * RX + cx + 2; };
    auto tix = [&](int cx, int cy) { return (cy + 3) * YX + cx + 3; };
    auto slot5 = [](int z) { return (z + 10) % 5; };

    auto load_types = [&](int z) {
        if constexpr (SOLID) {
            uint8_t* dst = sm.type[z & 7];
            const int gz = wz(z) * nxy;
            for (int i = tid; i < (he + 6) * YX; i += NT) {
                const int cx = i % YX - 3, cy = i / YX - 3;
                if (cx < we + 3) dst[i] = g.type[gz + wy(y0 + cy) * nx + wx(x0 + cx)];
            }
        }
    };
    auto type_at = [&](int z, int ti) -> uint8_t {
        if constexpr (!SOLID) return uint8_t(T_BULK);
        return sm.type[z & 7][ti];
    };
    auto pull = [&](double (&f)[Q], int cx, int cy, int z, uint8_t self) {
        const int gx = wx(x0 + cx), gy = wy(y0 + cy), gz = wz(z);
        const int col[3] = {wrap1(gx - 1, nx), gx, wrap1(gx + 1, nx)};
        const int row[3] = {wrap1(gy - 1, ny) * nx, gy * nx, wrap1(gy + 1, ny) * nx};
        const int pl[3] = {wrap1(gz - 1, nz) * nxy, gz * nxy, wrap1(gz + 1, nz) * nxy};
        if (!SOLID || (self & T_BULK)) {
#pragma unroll
            for (int a = 0; a < Q; ++a) f[a] = fin[a * N + pl[1 - L::ez(a)] + row[1 - L::ey(a)] + col[1 - L::ex(a)]];
        } else {
            const int ti = tix(cx, cy);
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const int ex = L::ex(a), ey = L::ey(a), ez = L::ez(a);
                const bool bb = (sm.type[(z - ez) & 7][ti - ex - ey * YX] & T_SOLID) != 0;
                f[a] = fin[bb ? L::opp(a) * N + pl[1] + row[1] + col[1]
                              : a * N + pl[1 - ez] + row[1 - ey] + col[1 - ex]];
            }
        }
    };
    // density and psi of cell (cx, cy) of plane z
    auto cell = [&](int cx, int cy, int z, bool want_psi) -> double {
        const uint8_t t = type_at(z, tix(cx, cy));
        double r = 0.0, psi = 0.0;
        if (!(t & T_SOLID)) {
            double v[Q];
            pull(v, cx, cy, z, t);
            r = density64(v);
            if (want_psi) psi = psi64(r, ph, err);
        }
        if (SOLID) sm.rho[z & 3][rix(cx, cy)] = r;
        if (want_psi) sm.psi[slot5(z)][pix(cx, cy)] = psi;
        return r;
    };

    const int lx = tid & (w - 1), ly = tid >> wl;
    const bool own = lx < we && ly < he;
    const int zlo = zb - LAG, zhi = ze + LAG - 1;
    for (int z = zlo - 3; z <= zlo + 1; ++z) load_types(z);
    if (SOLID) __syncthreads();
    double r0 = 0.0, r1 = 0.0, r2 = 0.0;   // own densities of planes zl, zl - 1, zl - 2
    for (int zl = zlo; zl <= zhi; ++zl) {
        // A. the lead plane: own node, then the ring from the last thread down
        r2 = r1;
        r1 = r0;
        if (own) r0 = cell(lx, ly, zl, true);
        for (int k = NT - 1 - tid; k < 2 * (we + 2) + 2 * he; k += NT) {
            int cx, cy;
            ring_cell(k, we + 2, he + 2, cx, cy);
            cell(cx - 1, cy - 1, zl, true);
        }
        if (SOLID) {
            for (int k = tid; k < 2 * (we + 4) + 2 * (he + 2); k += NT) {
                int cx, cy;
                ring_cell(k, we + 4, he + 4, cx, cy);
                cell(cx - 2, cy - 2, zl, false);
            }
            load_types(zl + 2);
        }
        __syncthreads();

        // B. wall cells of plane zl - 1 (the solid-fluid interaction scheme keeps psi = 0 on solids)
        const int zw = zl - 1;
        if (SOLID && ph.wall_kind != 2 && zw >= zb - 1) {
            for (int k = tid; k < (he + 2) * PX; k += NT) {
                const int cx = k % PX - 1, cy = k / PX - 1;
                if (cx > we || !(sm.type[zw & 7][tix(cx, cy)] & T_WALL)) continue;
                double rw;
                if (ph.wall_kind == 1) {
                    rw = ph.wall_param;
                } else {
                    // Eq. 17: weighted mean of the fluid neighbours' densities
                    double num = 0.0, den = 0.0;
#pragma unroll
                    for (int a = 1; a < Q; ++a) {
                        const int ex = L::ex(a), ey = L::ey(a), ez = L::ez(a);
                        if (!(sm.type[(zw + ez) & 7][tix(cx + ex, cy + ey)] & T_SOLID)) {
                            num += L::wf(a) * sm.rho[(zw + ez) & 3][rix(cx + ex, cy + ey)];
                            den += L::wf(a);
                        }
                    }
                    const double ave = num / den;
                    const double kap =
                        g.kappa_w ? g.kappa_w[g.wall_id[wz(zw) * nxy + wy(y0 + cy) * nx + wx(x0 + cx)]] : g.kappa;
                    // Eq. 16 (kappa >= 0: phi = 1 + kappa; kappa < 0: drho = -kappa) and the limiter
                    rw = kap >= 0.0 ? (1.0 + kap) * ave : ave + kap;
                    rw = rw > ph.rho_l ? ph.rho_l : rw;
                    rw = rw < ph.rho_g ? ph.rho_g : rw;
                }
                sm.psi[slot5(zw)][pix(cx, cy)] = psi64(rw, ph, err);
            }
            __syncthreads();
        }

        // C. collide plane zl - LAG
        const int z = zl - LAG;
        if (z >= zb && own) {
            const int gi = z * nxy + (y0 + ly) * nx + x0 + lx;
            const uint8_t t = type_at(z, tix(lx, ly));
            if (t & T_SOLID) {
                if (MODE == 1) {
                    if (rho_out) rho_out[gi] = 0.0;
                    if (u_out) u_out[gi] = u_out[N + gi] = u_out[2 * N + gi] = 0.0;
                }
            } else {
                double f[Q];
                pull(f, lx, ly, z, t);
                const double rho = SOLID ? r2 : r1;
                const int pc = pix(lx, ly);
                double d[9];
#pragma unroll
                for (int a = 1; a < Q; a += 2) {
                    const int off = L::ex(a) + L::ey(a) * PX, ez = L::ez(a);
                    d[a / 2] = dsub(sm.psi[slot5(z + ez)][pc + off], sm.psi[slot5(z - ez)][pc - off]);
                }
                const bool sf = SOLID && ph.wall_kind == 2 && !(t & T_BULK);
                double ax = 0.0, ay = 0.0, az = 0.0;
                if (sf) {
                    // Eq. 8: sum_a w_a s(x + e_a) e_a
#pragma unroll
                    for (int a = 1; a < Q; ++a) {
                        const int ex = L::ex(a), ey = L::ey(a), ez = L::ez(a);
                        if (sm.type[(z + ez) & 7][tix(lx + ex, ly + ey)] & T_SOLID) {
                            if (ex) ax += L::wf(a) * ex;
                            if (ey) ay += L::wf(a) * ey;
                            if (ez) az += L::wf(a) * ez;
                        }
                    }
                }
                if (!(rho > 0.0)) atomicOr(err, ERR_RHO);
                double ux, uy, uz;
                node3d64<MODE == 0>(f, rho, d, sm.psi[slot5(z)][pc], sf, ax, ay, az, ph, ux, uy, uz);
                if (MODE == 1) {
                    if (rho_out) rho_out[gi] = rho;
                    if (u_out) {
                        u_out[gi] = ux;
                        u_out[N + gi] = uy;
                        u_out[2 * N + gi] = uz;
                    }
                } else {
#pragma unroll
                    for (int a = 0; a < Q; ++a) fout[a * N + gi] = f[a];
                }
            }
        }
        // (the next lead plane writes psi and density slots that no collision or wall cell of this one
        // reads: psi of plane zl + 1 replaces zl - 4, density zl - 3; the types loaded above replace zl - 6)
    }
}

template <int MODE>
__global__ void __launch_bounds__(NT, RESIDENT)
    step3d64(const double* __restrict__ fin, double* __restrict__ fout, Geo g, const uint8_t* __restrict__ flags,
             Phys<double> ph, int wl, int h, int zc, unsigned* err, double* __restrict__ rho_out,
             double* __restrict__ u_out) {
    __shared__ Smem sm;
    const int x0 = int(blockIdx.x) << wl, y0 = int(blockIdx.y) * h, zb = int(blockIdx.z) * zc;
    const bool solid = flags[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] != 0;
    pdl_wait();
    if (solid)
        brick64<MODE, true>(fin, fout, g, ph, x0, y0, zb, wl, h, zc, err, rho_out, u_out, sm);
    else
        brick64<MODE, false>(fin, fout, g, ph, x0, y0, zb, wl, h, zc, err, rho_out, u_out, sm);
}

}  // namespace

// The shape with the least modelled time.  A brick costs the FP64 instructions of its warps (nodes and halo
// cells rounded up to warps, two halo planes) at 1.9 lane operations per clock.  With k bricks per SM the
// step takes about (1.12 k + 1) bricks: one alone leaves the pipe idle half the time (dependent chains,
// barriers), several fill it, and the last ones are the tail.  Fitted to 21 shapes on 40^3, 64^3 and 96 x 90
// x 100: it picks a shape within 5 % of the fastest on each (64^3: 221 to 236 us a step for 8 x 8 x 5, 16 x 8 x 3
// and 8 x 16 x 4; 32 x 4 x 16 takes 388 us).
void d3q19_fp64_brick(int nx, int ny, int nz, int sms, int* bw, int* bh, int* bz) {
    auto warps = [](int n) { return double((n + 31) / 32 * 32); };
    double best = 1e300;
    for (int w = 8; w <= MW; w *= 2)
        for (int h = 3 * NT / 4 / w; h <= NT / w; ++h)   // (3 or 4 warps of nodes)
            for (int z = 1; z <= nz; ++z) {
                const double n = double((nx + w - 1) / w) * ((ny + h - 1) / h) * ((nz + z - 1) / z);
                const double plane = 36.0 * (warps(w * h) + warps(2 * w + 2 * h + 4));
                const double brick = ((z + 2) * plane + z * 247.0 * warps(w * h)) / 1.9;
                const double cost = (1.12 * n / sms + 1.0) * brick;
                if (cost < best * 0.999) {
                    best = cost;
                    *bw = w;
                    *bh = h;
                    *bz = z;
                }
            }
}

cudaError_t launch_d3q19_fp64(int mode, const void* fin, void* fout, const Geo& g, const DevParams& p, double* rho,
                              double* u, cudaStream_t s) {
    int wl = 0;
    while ((1 << wl) < p.tile_w) ++wl;
    const dim3 grid((p.nx + p.tile_w - 1) / p.tile_w, (p.ny + p.tile_h - 1) / p.tile_h, (p.nz + p.tile_z - 1) / p.tile_z);
    const double* in = static_cast<const double*>(fin);
    if (mode == 0)
        return launch_pdl(step3d64<0>, grid, dim3(NT), 0, s, in, static_cast<double*>(fout), g, p.pair_solid,
                          make_phys<double>(p), wl, p.tile_h, p.tile_z, p.err, nullptr, nullptr);
    return launch_pdl(step3d64<1>, grid, dim3(NT), 0, s, in, nullptr, g, p.pair_solid, make_phys<double>(p), wl, p.tile_h,
                      p.tile_z, p.err, rho, u);
}

}  // namespace lbmwet
