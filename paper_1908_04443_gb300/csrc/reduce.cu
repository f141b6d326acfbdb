// Observables reduction: total fluid mass, fluid density extremes (Fig. 11), maximum |u| (the
// spurious-current measure of Fig. 10) and the moments of the interface points used by a Kasa
// circle/sphere fit of the drop (contact angle).  Two launches: per-block partials with warp-shuffle
// tree reductions, then one block combining them.  All sums in double.
#include <cfloat>
#include <cmath>
#include <mutex>

#include "kernels.h"
#include "lattice.cuh"
#include "reduce.h"

namespace lbmwet {

namespace {

constexpr int RB = 256;   // threads per reduction block

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// A double's bits as an int64 in the same order as the doubles (finite values; -0 below +0): the
// sign-magnitude pattern of a negative value has its magnitude bits flipped.  The map is its own
// inverse.  Comparisons and extremes then run on the integer pipe: the FP64 pipe of this GPU issues
// under 2 operations per clock per SM, and the per-node compares would otherwise bound the pass.
__device__ __forceinline__ long long ord_bits(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffLL); }
__device__ __forceinline__ long long ord(double x) { return ord_bits(__double_as_longlong(x)); }

// the same extremes over a warp of values that are not NaN
__device__ __forceinline__ double warp_max_ord(double x) {
    long long v = ord(x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long t = __shfl_xor_sync(0xffffffffu, v, o);
        v = t > v ? t : v;
    }
    return __longlong_as_double(ord_bits(v));
}
__device__ __forceinline__ double warp_min_ord(double x) {
    long long v = ord(x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long t = __shfl_xor_sync(0xffffffffu, v, o);
        v = t < v ? t : v;
    }
    return __longlong_as_double(ord_bits(v));
}

// kind of each of the NRED slots: 0 sum, 1 max, 2 min
__device__ __forceinline__ int slot_kind(int k) { return k == 1 || k == 3 ? 1 : (k == 2 ? 2 : 0); }

// Combines the NRED slots of a block's threads: the mass (slot 0) and the extremes (1 .. 3) from v, the
// interface moments (4 .. 17) from v too or, with ACC, from the warps' sums in acc.  The FP64 pipe (1.7
// operations per clock per SM) would spend more on a warp's reduction of all 18 slots, 90
// instructions, than on its nodes; this way a warp without interface points issues 5, the extremes
// being compared on the integer pipe.
template <bool ACC>
__device__ void block_combine(double (&v)[ACC ? 4 : NRED], const double (*acc)[NRED - 4], double* out) {
    __shared__ double sh[RB / 32][NRED];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // (a NaN extreme, of an unstable state, is ignored as fmax and fmin do)
    const bool nan = __any_sync(0xffffffffu, v[1] != v[1] || v[2] != v[2] || v[3] != v[3]);
#pragma unroll
    for (int k = 0; k < (ACC ? 4 : NRED); ++k) {
        const int kind = slot_kind(k);
        double r;
        if (kind == 0) r = warp_sum(v[k]);
        else if (nan) r = kind == 1 ? warp_max(v[k]) : warp_min(v[k]);
        else r = kind == 1 ? warp_max_ord(v[k]) : warp_min_ord(v[k]);
        if (lane == 0) sh[w][k] = r;
    }
    if (ACC && lane < NRED - 4) sh[w][4 + lane] = acc[w][lane];
    __syncthreads();
    if (threadIdx.x < NRED) {
        const int k = threadIdx.x;
        const int kind = slot_kind(k);
        double r = sh[0][k];
        for (int i = 1; i < RB / 32; ++i) {
            const double x = sh[i][k];
            r = kind == 0 ? r + x : (kind == 1 ? fmax(r, x) : fmin(r, x));
        }
        out[k] = r;
    }
}

template <int K>
__device__ __forceinline__ void init_slots(double (&v)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.0;
    v[1] = -DBL_MAX;   // rho_max
    v[2] = DBL_MAX;    // rho_min
    v[3] = 0.0;        // max |u|^2
}

__device__ __forceinline__ int wrapp(int v, int n) { return v >= n ? v - n : v; }

// Block `blk` of `nblk` over one grid: its nodes blk * RB + threadIdx.x + k * nblk * RB, combined into
// partials[blk * NRED ..].  Latency bound: what counts is how many loads are in flight, so a thread
// keeps only the mass and the extremes in registers (the 14 moments of the few interface points took
// 28 more and left 2 blocks per SM).  Links that cross rho_mid go into a queue of the warp; 32 of them
// at a time are evaluated together, one per lane, and summed into the warp's 14 sums in shared memory.
// 24 grids of 600 x 400: 279 us with the moments in every thread, 150 us with the queue, 92 us with the
// moments summed link by link instead of by warp shuffles and without a division per node.
template <int DIM>
__device__ __forceinline__ void partial_block(const double* __restrict__ rho, const double* __restrict__ u,
                                              const uint8_t* __restrict__ type, int nx, int ny, int nz,
                                              double rho_mid, double hx, double hy, double hz, int blk, int nblk,
                                              double* __restrict__ partials) {
    constexpr int NM = NRED - 4;
    __shared__ double s_acc[RB / 32][NM];
    __shared__ double s_p[RB / 32][32][5];
    __shared__ unsigned s_q[RB / 32][128];   // queued links: 4 * node + axis (a grid holds fewer than 2^31 / 19 nodes)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long N = (long long)nx * ny * nz;
    // factors of moment k = (n, Sx, Sy, Sz, Sxx, Syy, Szz, Sxy, Sxz, Syz, Sx r2, Sy r2, Sz r2, S r2), four bits
    // each, moment 0 lowest
    const int ka = int((0x4442113210000ull >> (4 * (lane & 15))) & 15u), kb = int((0x43213323213210ull >> (4 * (lane & 15))) & 15u);
    if (lane < NM) s_acc[w][lane] = 0.0;
    __syncwarp();
    auto coords = [&](unsigned g, int& x, int& y, int& z) {   // (32-bit division)
        const unsigned q = g / unsigned(nx);
        x = int(g - q * unsigned(nx));
        if (DIM == 2) {
            y = int(q);
            z = 0;
        } else {
            z = int(q / unsigned(ny));
            y = int(q - unsigned(z) * unsigned(ny));
        }
    };
    auto next = [&](unsigned g, int x, int y, int z, int axis) -> long long {
        if (axis == 0) return (long long)g - x + wrapp(x + 1, nx);
        if (axis == 1) return ((long long)z * ny + wrapp(y + 1, ny)) * nx + x;
        return ((long long)wrapp(z + 1, nz) * ny + y) * nx + x;
    };
    // The first n queued links: each lane finds one crossing relative to the hint, then lane k < 14 adds
    // moment k of all of them, a product of two of (1, dx, dy, dz, r2), one FP64 instruction of the warp
    // per link (14 shuffle sums are 70, and most queues hold only a few links).
    auto flush = [&](int n) {
        __syncwarp();
        if (lane < n) {
            const unsigned e = s_q[w][lane], g = e >> 2, axis = e & 3u;
            int x, y, z;
            coords(g, x, y, z);
            const double r = rho[g], rn = rho[next(g, x, y, z, int(axis))];
            const double tt = (rho_mid - r) / (rn - r);
            double px = x, py = y, pz = z;
            if (axis == 0) px += tt;
            if (axis == 1) py += tt;
            if (axis == 2) pz += tt;
            // periodic image nearest to the hint, relative to the hint
            double dx = px - hx, dy = py - hy, dz = (DIM == 3) ? pz - hz : 0.0;
            auto nearest = [](double& d, int m) {   // (rint(d / m) is 0 within half a period)
                if (fabs(d) > 0.5 * m) d -= m * rint(d / m);
            };
            nearest(dx, nx);
            nearest(dy, ny);
            if (DIM == 3) nearest(dz, nz);
            double* p = s_p[w][lane];
            p[0] = 1.0;
            p[1] = dx;
            p[2] = dy;
            p[3] = dz;
            p[4] = dx * dx + dy * dy + dz * dz;
        }
        __syncwarp();
        if (lane < NM) {
            double a = s_acc[w][lane];
            for (int i = 0; i < n; ++i) a += s_p[w][i][ka] * s_p[w][i][kb];
            s_acc[w][lane] = a;
        }
        __syncwarp();
    };
    int qn = 0;   // links in the warp's queue (the same in every lane)
    double v[4];
    init_slots(v);
    // density extremes and the largest |u|^2 as ordered integers (see ord); u^2 >= +0, whose bits
    // are already in order
    long long kmax = ord(-DBL_MAX), kmin = ord(DBL_MAX), ku = 0;
    const long long kmid = ord(rho_mid);
    const long long base = blk * (long long)RB + w * 32;
    // the node's coordinates and their steps from one iteration to the next (no division per node)
    int x, y, z, sx, sy, sz;
    coords(unsigned(base + lane), x, y, z);
    coords(unsigned(nblk) * RB, sx, sy, sz);
    for (long long g0 = base; g0 < N; g0 += (long long)nblk * RB) {   // (uniform in the warp)
        const bool in = g0 + lane < N;
        const unsigned g = unsigned(g0 + lane);
        double r = 0.0, uc[DIM], rnb[DIM];
        uint8_t t = T_SOLID, tnb[DIM];
        // every load of the node and of its +x, +y (, +z) neighbours is issued before any branch, so
        // that they are in flight together rather than one dependent round trip after another (the
        // fields hold values at every node, solid ones included)
        if (in) {
            long long gn[DIM];
#pragma unroll
            for (int a = 0; a < DIM; ++a) gn[a] = next(g, x, y, z, a);
            t = type[g];
            r = rho[g];
#pragma unroll
            for (int c = 0; c < DIM; ++c) uc[c] = u[(long long)c * N + g];
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                tnb[a] = type[gn[a]];
                rnb[a] = rho[gn[a]];
            }
        } else {
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                tnb[a] = T_SOLID;
                rnb[a] = uc[a] = 0.0;
            }
        }
        x += sx;
        y += sy;
        z += sz;
        if (x >= nx) {
            x -= nx;
            ++y;
        }
        if (DIM == 3 && y >= ny) {
            y -= ny;
            ++z;
        }
        const bool fluid = !(t & T_SOLID);
        const long long kr = ord(r);
        if (fluid) {
            v[0] += r;
            kmax = kr > kmax ? kr : kmax;
            kmin = kr < kmin ? kr : kmin;
            double u2 = 0.0;
#pragma unroll
            for (int c = 0; c < DIM; ++c) u2 += uc[c] * uc[c];
            const long long k2 = __double_as_longlong(u2);
            ku = k2 > ku ? k2 : ku;
        }
        // links +x, +y (, +z) to a fluid neighbour away from walls whose densities lie on the two sides
        // of rho_mid (a link from r == rho_mid never does)
        const int side = (kr > kmid) - (kr < kmid);   // sign of r - rho_mid
        const bool src = fluid && !(t & T_NEARWALL) && side != 0;
#pragma unroll
        for (int axis = 0; axis < DIM; ++axis) {
            const long long kn = ord(rnb[axis]);
            const bool cross = src && !(tnb[axis] & (T_SOLID | T_NEARWALL)) && (side > 0 ? kn < kmid : kn > kmid);
            const unsigned m = __ballot_sync(0xffffffffu, cross);
            if (cross) s_q[w][qn + __popc(m & ((1u << lane) - 1u))] = 4u * g + unsigned(axis);
            qn += __popc(m);   // at most 31 + 32 DIM
        }
        // (the rest with the warp's last node; one call keeps one copy of the code)
        const bool last = g0 + (long long)nblk * RB >= N;
        while (qn >= 32 || (last && qn > 0)) {
            const int n = qn < 32 ? qn : 32;
            flush(n);
            qn -= n;
            unsigned e[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) e[k] = s_q[w][32 * (k + 1) + lane];
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 3; ++k) s_q[w][32 * k + lane] = e[k];
            __syncwarp();
        }
    }
    v[1] = __longlong_as_double(ord_bits(kmax));
    v[2] = __longlong_as_double(ord_bits(kmin));
    v[3] = __longlong_as_double(ku);
    block_combine<true>(v, s_acc, partials + (long long)blk * NRED);
}

template <int DIM>
__global__ void __launch_bounds__(RB, 4) reduce_partial(const double* __restrict__ rho, const double* __restrict__ u,
                                                     const uint8_t* __restrict__ type, int nx, int ny, int nz,
                                                     double rho_mid, double hx, double hy, double hz,
                                                     double* __restrict__ partials) {
    partial_block<DIM>(rho, u, type, nx, ny, nz, rho_mid, hx, hy, hz, blockIdx.x, gridDim.x, partials);
}

// One block combining nparts partials; err (optional): the grid's error word, stored after the NRED
// results
__device__ __forceinline__ void final_block(const double* __restrict__ partials, int nparts, double* __restrict__ out,
                                            const unsigned* __restrict__ err) {
    double v[NRED];
    init_slots(v);
    for (int i = threadIdx.x; i < nparts; i += RB) {
#pragma unroll
        for (int k = 0; k < NRED; ++k) {
            const double x = partials[(long long)i * NRED + k];
            const int kind = slot_kind(k);
            v[k] = kind == 0 ? v[k] + x : (kind == 1 ? fmax(v[k], x) : fmin(v[k], x));
        }
    }
    block_combine<false>(v, nullptr, out);
    if (err && threadIdx.x == 0) *reinterpret_cast<unsigned*>(out + NRED) = *err;
}

__global__ void __launch_bounds__(RB) reduce_final(const double* __restrict__ partials, int nparts, double* __restrict__ out,
                                                   const unsigned* __restrict__ err = nullptr) {
    final_block(partials, nparts, out, err);
}

// Several grids in one launch: grid k owns blocks [g[k].block0, g[k].block0 + g[k].nblk), which
// cover its nodes exactly as a launch of g[k].nblk blocks of its own would (same sums, same order).
template <int DIM>
__global__ void __launch_bounds__(RB, 4) reduce_partial_grids(const RedGrid* __restrict__ g, int ngrids) {
    int lo = 0, hi = ngrids - 1;
    while (lo < hi) {   // the last grid whose first block is at or before this one
        const int mid = (lo + hi + 1) >> 1;
        if (g[mid].block0 <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const RedGrid& r = g[lo];
    partial_block<DIM>(r.rho, r.u, r.type, r.nx, r.ny, r.nz, r.rho_mid, r.hint[0], r.hint[1], r.hint[2],
                       int(blockIdx.x) - r.block0, r.nblk, r.partials);
}

__global__ void __launch_bounds__(RB) reduce_final_grids(const RedGrid* __restrict__ g) {
    const RedGrid& r = g[blockIdx.x];
    final_block(r.partials, r.nblk, r.out, r.err);
}

// About 8 nodes per thread: each block ends with warp reductions of NRED doubles on the FP64 pipe,
// whose low rate makes one block per 256 nodes cost more than the nodes themselves on small grids.
int n_blocks(long long N) {
    long long b = (N + 8LL * RB - 1) / (8LL * RB);
    const long long cap = 152LL * 8;
    if (b > cap) b = cap;
    return int(b < 1 ? 1 : b);
}

}  // namespace

size_t reduce_partials_size(long long N) { return size_t(n_blocks(N)) * NRED; }

cudaError_t launch_reduce(int dim, const double* rho, const double* u, const uint8_t* type, int nx, int ny, int nz,
                          double rho_mid, const double* hint, double* partials, double* out, cudaStream_t s) {
    const long long N = (long long)nx * ny * nz;
    const int nb = n_blocks(N);
    if (dim == 2)
        reduce_partial<2><<<nb, RB, 0, s>>>(rho, u, type, nx, ny, nz, rho_mid, hint[0], hint[1], hint[2], partials);
    else
        reduce_partial<3><<<nb, RB, 0, s>>>(rho, u, type, nx, ny, nz, rho_mid, hint[0], hint[1], hint[2], partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    reduce_final<<<1, RB, 0, s>>>(partials, nb, out);
    return cudaGetLastError();
}

int reduce_blocks(long long N) { return n_blocks(N); }

cudaError_t launch_reduce_grids(int dim, const RedGrid* grids, int ngrids, int total_blocks, cudaStream_t s) {
    if (ngrids < 1) return cudaSuccess;
    if (dim == 2) reduce_partial_grids<2><<<total_blocks, RB, 0, s>>>(grids, ngrids);
    else reduce_partial_grids<3><<<total_blocks, RB, 0, s>>>(grids, ngrids);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    reduce_final_grids<<<ngrids, RB, 0, s>>>(grids);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Allocation-free variant of the observables reduction (no counterpart in the paper).
//
// For callers that must not call cudaMalloc - e.g. frameworks that route every device allocation
// through their own allocator and budget, or latency-sensitive loops where cudaMalloc's implicit
// device synchronisation is not acceptable - the same two kernels run with their per-block
// partials and final sums in this file-scope device array instead of handle-owned buffers.
//
// Capacity: STATIC_BLOCKS blocks of STATIC_NODES_PER_BLOCK nodes, i.e. grids of at most
// 4096 * 4096 = 16,777,216 nodes (256^3); larger grids are rejected.  The array (4096 * 18 + 18
// doubles, about 590 KB) is part of the module image, so every GPU that loads this library holds
// it until the process exits.  All calls share it and it keeps the last call's contents; every
// slot is written by the partial kernel before the final kernel reads it, so nothing needs
// clearing between calls.  Calls whose kernels overlap on the GPU (different streams, or
// different handles on one device without ordering) race on the array.
// ---------------------------------------------------------------------------------------------

namespace {

constexpr int STATIC_BLOCKS = 4096;
constexpr long long STATIC_NODES_PER_BLOCK = 4096;

static __device__ __align__(256) double g_static_scratch[STATIC_BLOCKS * NRED + NRED];

constexpr int MAX_DEVICES = 64;
double* g_static_ptr[MAX_DEVICES] = {nullptr};
std::mutex g_static_mutex;

}  // namespace

long long static_reduce_max_nodes() { return STATIC_BLOCKS * STATIC_NODES_PER_BLOCK; }

cudaError_t static_reduce_setup(int device, double** ptr) {
    if (device < 0 || device >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[device]) {
        // host code may not use the symbol itself as an address: ask the runtime for the device
        // address of this device's copy (the device must be current)
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return e;
        g_static_ptr[device] = static_cast<double*>(p);
    }
    *ptr = g_static_ptr[device];
    return cudaSuccess;
}

cudaError_t launch_reduce_static(int dim, const double* rho, const double* u, const uint8_t* type, int nx, int ny,
                                 int nz, double rho_mid, const double* hint, double* scratch, double* out_host,
                                 cudaStream_t s) {
    const long long N = (long long)nx * ny * nz;
    const long long nb = (N + STATIC_NODES_PER_BLOCK - 1) / STATIC_NODES_PER_BLOCK;
    if (nb < 1 || nb > STATIC_BLOCKS) return cudaErrorInvalidValue;
    double* partials = scratch;
    double* out = scratch + (long long)STATIC_BLOCKS * NRED;
    if (dim == 2)
        reduce_partial<2><<<int(nb), RB, 0, s>>>(rho, u, type, nx, ny, nz, rho_mid, hint[0], hint[1], hint[2], partials);
    else
        reduce_partial<3><<<int(nb), RB, 0, s>>>(rho, u, type, nx, ny, nz, rho_mid, hint[0], hint[1], hint[2], partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    reduce_final<<<1, RB, 0, s>>>(partials, int(nb), out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(out_host, out, sizeof(double) * NRED, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

}  // namespace lbmwet
