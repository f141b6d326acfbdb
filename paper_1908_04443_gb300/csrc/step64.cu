// D2Q9 FP64 step and fields pass: tiles whose shape is chosen per grid.
//
// The phases are those of the scalar tile kernel (step.cu): node types of the tile + 3-node halo;
// pull (Eq. 3, Fig. 3), density (Eq. 4) and psi (Eq. 6) of the tile and its 1-node ring, the 2-node
// ring's densities near walls; virtual wall densities (Eqs. 16-17); force, velocity and collision.
// Bound by the FP64 pipe (fp64.cuh), so two things count: FP64 instructions per node, and that every SM
// has the same number of them.  A tile's ring costs 26 FP64 instructions a cell (density and psi)
// against 136 for an own node, so large tiles are cheaper (32 x 16: ring 20 % of the cells, +4 %) as long
// as there are many of them per SM; a grid with few nodes is cut into small tiles, about one per SM
// (d2q9_fp64_tile), since an SM works on a 32 x 8 tile for 17 us however idle the others are.
// Columns and rows of a tile beyond the grid's edge are skipped instead of wrapped.
// Integer work is free beside the FP64 pipe: shapes are run-time values and every neighbour wraps.
#include "fp64.cuh"
#include "kernels.h"
#include "lattice.cuh"
#include "pdl.cuh"
#include "tile_common.cuh"

namespace lbmwet {

namespace {

constexpr int NT = 256;                  // threads; tiles hold up to 2 NT nodes
constexpr int MW = 32, MH = 16;          // largest tile
constexpr int PXP = MW + 2, PYP = MH + 2;   // psi (1-node halo)
constexpr int RXP = MW + 4, RYP = MH + 4;   // density (2-node halo)
constexpr int YXP = MW + 6, YYP = MH + 6;   // types (3-node halo)

struct Smem64 {
    double rho[RYP * RXP];
    double psi[PYP * PXP];
    uint8_t type[YYP * YXP];
    short wall[PYP * PXP];
    int nwall;
};

// One tile of w x h nodes (w = 1 << wl) at (x0, y0) of the grid g (a BatchItem or PairGrid), reading
// g.f[parity].  MODE 0: step into g.f[parity ^ 1]; 1: fields.  SOLID: a solid node lies within the tile
// + 3 nodes.
template <int MODE, bool SOLID, class G>
__device__ __forceinline__ void body64(const G& g, int parity, const Phys<double>& ph, int x0, int y0, int wl, int h,
                                       unsigned* err, double* __restrict__ rho_out, double* __restrict__ u_out,
                                       Smem64& sm) {
    using L = D2Q9;
    constexpr int Q = 9;
    const int nx = g.nx, ny = g.ny, fp = g.fp, fs = g.fs;
    const double* __restrict__ fin = static_cast<const double*>(g.f[parity]);
    const int tid = threadIdx.x;
    const int we = min(1 << wl, nx - x0), he = min(h, ny - y0);   // the tile's nodes inside the grid
    const bool small = nx < MW + 8 || ny < MH + 8;
    auto wx = [&](int v) { return small ? wrap_full(v, nx) : wrap1(v, nx); };
    auto wy = [&](int v) { return small ? wrap_full(v, ny) : wrap1(v, ny); };
    // cells relative to the tile's first node
    auto tix = [](int cx, int cy) { return (cy + 3) * YXP + cx + 3; };
    auto rix = [](int cx, int cy) { return (cy + 2) * RXP + cx + 2; };
    auto pix = [](int cx, int cy) { return (cy + 1) * PXP + cx + 1; };

    if (tid == 0) sm.nwall = 0;
    bool has_wall = false;
    if constexpr (SOLID) {
        int seen = 0;
        for (int i = tid; i < (he + 6) * YXP; i += NT) {
            const int cx = i % YXP - 3, cy = i / YXP - 3;
            if (cx >= we + 3) continue;
            const uint8_t t = g.type[wy(y0 + cy) * nx + wx(x0 + cx)];
            sm.type[i] = t;
            if ((t & T_WALL) && cx >= -1 && cx <= we && cy >= -1 && cy <= he) seen = 1;
        }
        has_wall = __syncthreads_or(seen);
    }
    auto type_at = [&](int ti) -> uint8_t {
        if constexpr (!SOLID) return uint8_t(T_BULK);
        return sm.type[ti];
    };
    // pull of cell (cx, cy)
    auto pull = [&](double (&f)[Q], int cx, int cy, uint8_t self) {
        const int gx = wx(x0 + cx), gy = wy(y0 + cy);
        const int col[3] = {wrap1(gx - 1, nx), gx, wrap1(gx + 1, nx)};
        const int row[3] = {wrap1(gy - 1, ny) * fp, gy * fp, wrap1(gy + 1, ny) * fp};
        if (!SOLID || (self & T_BULK)) {
#pragma unroll
            for (int a = 0; a < Q; ++a) f[a] = fin[a * fs + row[1 - L::ey(a)] + col[1 - L::ex(a)]];
        } else {
            const int ti = tix(cx, cy);
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const bool bb = (sm.type[ti - L::ex(a) - L::ey(a) * YXP] & T_SOLID) != 0;
                f[a] = fin[bb ? L::opp(a) * fs + row[1] + col[1] : a * fs + row[1 - L::ey(a)] + col[1 - L::ex(a)]];
            }
        }
    };

    // 1. the thread's own nodes tid and tid + NT, kept in registers
    double f[2][Q], rho[2];
    bool fluid[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = tid + j * NT, lx = i & ((1 << wl) - 1), ly = i >> wl;
        fluid[j] = false;
        rho[j] = 0.0;
#pragma unroll
        for (int a = 0; a < Q; ++a) f[j][a] = 0.0;
        if (lx >= we || ly >= he) continue;
        const uint8_t t = type_at(tix(lx, ly));
        double psi = 0.0;
        if (!(t & T_SOLID)) {
            pull(f[j], lx, ly, t);
            rho[j] = density64(f[j]);
            psi = psi64(rho[j], ph, err);
            fluid[j] = true;
        } else if (t & T_WALL) {
            sm.wall[atomicAdd(&sm.nwall, 1)] = short(pix(lx, ly));
        }
        sm.psi[pix(lx, ly)] = psi;
        if (SOLID) sm.rho[rix(lx, ly)] = rho[j];
    }
    // the 1-node ring, from the last thread down: in a small tile they have no node of their own
    for (int k = NT - 1 - tid; k < 2 * (we + 2) + 2 * he; k += NT) {
        int cx, cy;
        ring_cell(k, we + 2, he + 2, cx, cy);
        --cx;
        --cy;
        const uint8_t t = type_at(tix(cx, cy));
        double r = 0.0, psi = 0.0;
        if (!(t & T_SOLID)) {
            double v[Q];
            pull(v, cx, cy, t);
            r = density64(v);
            psi = psi64(r, ph, err);
        } else if (t & T_WALL) {
            sm.wall[atomicAdd(&sm.nwall, 1)] = short(pix(cx, cy));
        }
        sm.psi[pix(cx, cy)] = psi;
        if (SOLID) sm.rho[rix(cx, cy)] = r;
    }
    // the 2-node ring's densities, where Eq. 17 needs them
    if (SOLID && has_wall) {
        for (int k = tid; k < 2 * (we + 4) + 2 * (he + 2); k += NT) {
            int cx, cy;
            ring_cell(k, we + 4, he + 4, cx, cy);
            cx -= 2;
            cy -= 2;
            const uint8_t t = sm.type[tix(cx, cy)];
            double r = 0.0;
            if (!(t & T_SOLID)) {
                double v[Q];
                pull(v, cx, cy, t);
                r = density64(v);
            }
            sm.rho[rix(cx, cy)] = r;
        }
    }
    __syncthreads();

    // 2. wall cells: virtual density and its psi (the solid-fluid interaction scheme keeps psi = 0)
    const int nwall = SOLID ? sm.nwall : 0;
    if (SOLID && nwall > 0 && ph.wall_kind != 2) {
        for (int k = tid; k < nwall; k += NT) {
            const int i = sm.wall[k], cx = i % PXP - 1, cy = i / PXP - 1;
            double rw;
            if (ph.wall_kind == 1) {
                rw = ph.wall_param;
            } else {
                // Eq. 17: weighted mean of the fluid neighbours' densities
                double num = 0.0, den = 0.0;
#pragma unroll
                for (int a = 1; a < Q; ++a) {
                    if (!(sm.type[tix(cx + L::ex(a), cy + L::ey(a))] & T_SOLID)) {
                        num += L::wf(a) * sm.rho[rix(cx + L::ex(a), cy + L::ey(a))];
                        den += L::wf(a);
                    }
                }
                const double ave = num / den;
                const int gw = wy(y0 + cy) * nx + wx(x0 + cx);
                if (ph.wall_kind == 3) {
                    // geometric formulation (Eqs. 10-15): crossings of the characteristic lines
                    rw = gf_wall_density(g.kappa_w + GF_STRIDE * g.wall_id[gw], ave,
                                         [&](int dx, int dy) { return sm.rho[rix(cx + dx, cy + dy)]; });
                } else {
                    const double kap = g.kappa_w ? g.kappa_w[g.wall_id[gw]] : g.kappa;
                    // Eq. 16 (kappa >= 0: phi = 1 + kappa; kappa < 0: drho = -kappa) and the limiter
                    const double raw = kap >= 0.0 ? (1.0 + kap) * ave : ave + kap;
                    rw = raw > ph.rho_l ? ph.rho_l : raw;
                    rw = rw < ph.rho_g ? ph.rho_g : rw;
                }
            }
            sm.psi[i] = psi64(rw, ph, err);
        }
        __syncthreads();
    }

    // 3. force, velocity and collision
    double* __restrict__ fout = static_cast<double*>(const_cast<void*>(g.f[parity ^ 1]));
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = tid + j * NT, lx = i & ((1 << wl) - 1), ly = i >> wl;
        if (lx >= we || ly >= he) continue;
        const int gx = x0 + lx, gy = y0 + ly, gi = gy * nx + gx, N = nx * ny;
        if (!fluid[j]) {
            if (MODE == 1) {
                if (rho_out) rho_out[gi] = 0.0;
                if (u_out) u_out[gi] = u_out[N + gi] = 0.0;
            }
            continue;
        }
        const int pc = pix(lx, ly);
        const bool sf = SOLID && ph.wall_kind == 2 && !(sm.type[tix(lx, ly)] & T_BULK);
        double ax = 0.0, ay = 0.0;
        if (sf) {
            // Eq. 8: sum_a w_a s(x + e_a) e_a
#pragma unroll
            for (int a = 1; a < Q; ++a) {
                const int ex = L::ex(a), ey = L::ey(a);
                if (sm.type[tix(lx + ex, ly + ey)] & T_SOLID) {
                    if (ex) ax += L::wf(a) * ex;
                    if (ey) ay += L::wf(a) * ey;
                }
            }
        }
        auto diff = [&](int off) { return dsub(sm.psi[pc + off], sm.psi[pc - off]); };
        if (!(rho[j] > 0.0)) atomicOr(err, ERR_RHO);
        double ux, uy;
        node2d64<MODE == 0>(f[j], rho[j], diff(1), diff(PXP), diff(PXP + 1), diff(PXP - 1), sm.psi[pc], sf, ax, ay, ph,
                            ux, uy);
        if (MODE == 1) {
            if (rho_out) rho_out[gi] = rho[j];
            if (u_out) {
                u_out[gi] = ux;
                u_out[N + gi] = uy;
            }
        } else {
            double* o = fout + gy * fp + gx;
#pragma unroll
            for (int a = 0; a < Q; ++a) o[a * fs] = f[j][a];
        }
    }
}

// One CTA per tile of one grid; flags: per tile, a solid node within the tile + 3 nodes.
template <int MODE>
__global__ void __launch_bounds__(NT, 2) step64(PairGrid g, const uint8_t* __restrict__ flags, Phys<double> ph, int wl,
                                                int h, unsigned* err, double* __restrict__ rho_out,
                                                double* __restrict__ u_out) {
    __shared__ Smem64 sm;
    const int x0 = int(blockIdx.x) << wl, y0 = int(blockIdx.y) * h;
    const bool solid = flags[blockIdx.y * gridDim.x + blockIdx.x] != 0;
    pdl_wait();
    if (solid)
        body64<MODE, true>(g, 0, ph, x0, y0, wl, h, err, rho_out, u_out, sm);
    else
        body64<MODE, false>(g, 0, ph, x0, y0, wl, h, err, rho_out, u_out, sm);
}

// One CTA per (instance, tile) record.
__global__ void __launch_bounds__(NT, 2) step64_batched(int parity, const BatchItem* __restrict__ items,
                                                        Phys<double> ph, int wl, int h, unsigned* err) {
    __shared__ Smem64 sm;
    const BatchItem& g = items[blockIdx.x];
    const bool solid = g.solid != 0;
    pdl_wait();
    if (solid) body64<0, true>(g, parity, ph, g.x0, g.y0, wl, h, err, nullptr, nullptr, sm);
    else body64<0, false>(g, parity, ph, g.x0, g.y0, wl, h, err, nullptr, nullptr, sm);
}

// The fields pass of several grids.
__global__ void __launch_bounds__(NT, 2) fields64_grids(const FieldGrid* __restrict__ tab, int n, Phys<double> ph) {
    __shared__ Smem64 sm;
    const int k = grid_of_tile(tab, n);
    const FieldGrid& q = tab[k];
    PairGrid g;
    g.nx = q.nx;
    g.ny = q.ny;
    g.N = q.nx * q.ny;
    g.fp = q.fp;
    g.fs = q.fs;
    g.type = q.type;
    g.wall_id = q.wall_id;
    g.kappa_w = q.kappa_w;
    g.kappa = q.kappa;
    g.f[0] = q.fin;
    g.f[1] = nullptr;
    const int tile = int(blockIdx.x) - q.tile0, ty = tile / q.tx, x0 = (tile - ty * q.tx) * q.tw, y0 = ty * q.th;
    const int wl = 31 - __clz(q.tw);
    if (q.tile_solid[tile]) body64<1, true>(g, 0, ph, x0, y0, wl, q.th, q.err, q.rho, q.u, sm);
    else body64<1, false>(g, 0, ph, x0, y0, wl, q.th, q.err, q.rho, q.u, sm);
}

}  // namespace

// The shape with the least modelled time.  A tile costs the FP64 instructions of its warps (own nodes and
// ring cells rounded up to warps) at 1.9 lane operations per clock and 1000 clocks of latency that its SM's
// other tiles do not hide; alone on its SM it takes 1.35 times that.  Up to two tiles per SM run at once, and
// the fullest SM decides; beyond that tiles are handed out as SMs get free and half a tile is the tail.
// Fitted to 14 shapes on 4 grids (100 x 100 to
// 1000 x 1000): it picks a shape within 5 % of the fastest on each, 8 x 10 (10.9 us a step) for 100 x 100,
// 32 x 12 for 300 x 350 (34.6 us; 32 x 16 takes 44.9), 16 x 14 for 600 x 400 (68 us; 32 x 16 takes 78.9).
void d2q9_fp64_tile(const int* nx, const int* ny, int ngrids, int sms, int* tw, int* th) {
    auto warps = [](int n) { return double((n + 31) / 32 * 32); };
    double best = 1e300;
    for (int w = 8; w <= MW; w *= 2)
        for (int h = 64 / w; h <= MH; ++h) {   // (at least two warps of nodes)
            long long n = 0;
            for (int i = 0; i < ngrids; ++i) n += (long long)((nx[i] + w - 1) / w) * ((ny[i] + h - 1) / h);
            const double tile = (136.0 * warps(w * h) + 26.0 * warps(2 * w + 2 * h + 4)) / 1.9 + 1000.0;
            const double rounds = n <= sms ? 1.35 : (n <= 2LL * sms ? 2.0 : double(n) / sms + 0.5);
            if (tile * rounds < best * 0.999) {
                best = tile * rounds;
                *tw = w;
                *th = h;
            }
        }
}

static int log2_of(int w) {
    int l = 0;
    while ((1 << l) < w) ++l;
    return l;
}

cudaError_t launch_d2q9_fp64(int mode, const void* fin, void* fout, const DevParams& p, double* rho, double* u,
                             cudaStream_t s) {
    const PairGrid g = pair_grid(fin, fout, p);
    const dim3 grid((p.nx + p.tile_w - 1) / p.tile_w, (p.ny + p.tile_h - 1) / p.tile_h, 1);
    if (mode == 0)
        return launch_pdl(step64<0>, grid, dim3(NT), 0, s, g, p.pair_solid, make_phys<double>(p), log2_of(p.tile_w), p.tile_h,
                          p.err, nullptr, nullptr);
    return launch_pdl(step64<1>, grid, dim3(NT), 0, s, g, p.pair_solid, make_phys<double>(p), log2_of(p.tile_w), p.tile_h,
                      p.err, rho, u);
}

cudaError_t launch_d2q9_fp64_batched(int parity, const DevParams& p, const BatchItem* items, int n_items, int tw, int th,
                                     cudaStream_t s) {
    if (n_items < 1) return cudaSuccess;
    return launch_pdl(step64_batched, dim3(n_items), dim3(NT), 0, s, parity, items, make_phys<double>(p), log2_of(tw), th,
                      p.err);
}

cudaError_t launch_d2q9_fp64_fields(const FieldGrid* grids, int ngrids, int total_tiles, const DevParams& p,
                                    cudaStream_t s) {
    if (ngrids < 1 || total_tiles < 1) return cudaSuccess;
    fields64_grids<<<total_tiles, NT, 0, s>>>(grids, ngrids, make_phys<double>(p));
    return cudaGetLastError();
}

}  // namespace lbmwet
