// k_cluster.cu -- all steps of a small 2D solve in one launch: a thread-block cluster holds every level in
// shared memory.
//
// A grid of a few thousand nodes gives an SM a node or two per thread, and one launch per step costs
// more than the step (2.2 us for a 64 x 64 grid even chained).  Here a cluster of kClusterCtas CTAs
// takes the grid's rows in equal shares; a CTA keeps its rows of every level, with one halo row
// either side, in shared memory in the level layout.  A step computes the CTA's rows (one node per
// thread and pass, the node function of k_direct, so the results are the same bits), writes the x
// ghost images, and writes its first and last row into the neighbours' halo rows over distributed
// shared memory; one cluster barrier ends the step.  The levels are read from and written back to
// global memory once per launch.
#include <cooperative_groups.h>

#include "k_direct.cuh"
#include "kernels.h"

namespace mmfd {

namespace cg = cooperative_groups;

namespace {

constexpr int kClusterCtas = 16;
constexpr int kClusterThreads = 512;
constexpr size_t kClusterSmem = 227 * 1024;

struct ClusterLevels {
    void* lev[3];
    void* out[3];
};

// Rows per CTA, and bytes of shared memory of a CTA holding nlev levels.
__host__ __device__ constexpr int cluster_rows(int ny) { return (ny + kClusterCtas - 1) / kClusterCtas; }

template <int LAT, int PDE, int LEVELS, int ST>
__global__ void __launch_bounds__(kClusterThreads) k_cluster(Geom g, const __grid_constant__ ClusterLevels gl, int cur,
                                                             const __grid_constant__ Coef<typename Storage<ST>::T> cf,
                                                             StepExtra ex, int nsteps) {
    using S = typename Storage<ST>::S;
    using T = typename Storage<ST>::T;
    constexpr int NF = pde_nf(PDE, LAT);
    constexpr int NLEV = LEVELS;   // level buffers: 2 or 3
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S* sm = reinterpret_cast<S*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int share = cluster_rows(g.ny);
    const int r0 = min(rank * share, g.ny), rows = min(share, g.ny - r0);
    const int active = (g.ny + share - 1) / share;   // CTAs with rows
    // the CTA's part of a level in the level layout: rows -1 .. share of its rows
    Geom gs = g;
    gs.ny = rows;
    gs.fs = (long long)(share + 2) * g.py;
    const long long lvl = gs.fs * NF;   // elements of one level

    chain_wait();
    // levels t and (three levels) t - dt, rows r0 - 1 .. r0 + rows with their ghosts
    for (int l = 0; l < NLEV - 1; ++l) {
        const int b = l == 0 ? cur : (cur + 2) % 3;
        const S* src = static_cast<const S*>(gl.lev[b]);
        for (int f = 0; f < NF; ++f) {
            const S* p = src + f * g.fs + (long long)r0 * g.py;
            S* q = sm + b * lvl + f * gs.fs;
            const int n = rows > 0 ? (rows + 2) * (int)g.py : 0;
            for (int i = threadIdx.x; i < n; i += kClusterThreads) q[i] = p[i];
        }
    }
    // the neighbours' memory: their copy of a row sits share + 2 rows apart at the same offsets
    const int up = rank + 1 == active ? 0 : rank + 1, dn = rank == 0 ? active - 1 : rank - 1;
    S* smu = reinterpret_cast<S*>(cluster.map_shared_rank(smem_raw, rows > 0 ? up : 0));
    S* smd = reinterpret_cast<S*>(cluster.map_shared_rank(smem_raw, rows > 0 ? dn : 0));
    const int dn_rows = min(share, g.ny - dn * share);   // rows of the CTA below
    cluster.sync();

    int c = cur;
    const int nodes = rows * g.nx;
    // the thread's first node and the way from one of its nodes to the next
    const int y0 = (int)threadIdx.x / g.nx, x0 = (int)threadIdx.x - y0 * g.nx;
    const int dy = kClusterThreads / g.nx, dx = kClusterThreads - dy * g.nx;
    for (int n = 0; n < nsteps; ++n) {
        const int pv = NLEV == 3 ? (c + 2) % 3 : c, nx_ = NLEV == 3 ? (c + 1) % 3 : 1 - c;
        const S* in0 = sm + c * lvl;
        const S* in1 = sm + pv * lvl;
        int x = x0, y = y0;
        for (int i = threadIdx.x; i < nodes; i += kClusterThreads, x += dx, y += dy) {
            if (x >= g.nx) {
                x -= g.nx;
                ++y;
            }
            T acc[NF];
            const long long at = gs.at(x, y, 0);
            direct_value<LAT, PDE, LEVELS, ST>(gs, in0, in1, cf, at, acc);
            const long long node = (long long)(r0 + y) * g.nx + x;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const unsigned rnd = ex.sr ? sr_bits(ex.seed, ex.step + n, node, f) : 0u;
                const S v = kpack<ST, PDE>(acc[f], cf.ref[f], rnd);
                const long long o = nx_ * lvl + f * gs.fs;
                auto put = [&](S* row) {   // row: the node's slot of some copy of its row
                    *row = v;
                    if (x < g.gx) row[g.nx] = v;
                    if (x >= g.nx - g.gx) row[-g.nx] = v;
                };
                put(sm + o + at);
                // first row: the halo row above the CTA below (dn); last row: below the CTA above (up)
                if (y == 0) put(smd + o + (long long)(dn_rows + 1) * g.py + g.ox + x);
                if (y == rows - 1) put(smu + o + g.ox + x);
            }
        }
        c = nx_;
        cluster.sync();
    }
    // the new level t and (three levels) t - dt back, with the ghost rows of the grid's edges
    for (int l = 0; l < NLEV - 1; ++l) {
        const int b = l == 0 ? c : (c + 2) % 3;
        for (int f = 0; f < NF; ++f) {
            S* p = static_cast<S*>(gl.out[b]) + f * g.fs;
            const S* q = sm + b * lvl + f * gs.fs;
            for (int i = threadIdx.x; i < rows * (int)g.py; i += kClusterThreads) {
                const int y = i / (int)g.py, x = i - y * (int)g.py;   // padded column
                if (x < g.ox - g.gx || x >= g.ox + g.nx + g.gx) continue;
                const S v = q[(y + 1) * g.py + x];
                p[(long long)(r0 + y + 1) * g.py + x] = v;
                if (r0 + y == 0) p[(long long)(g.ny + 1) * g.py + x] = v;
                if (r0 + y == g.ny - 1) p[x] = v;
            }
        }
    }
}

template <int LAT, int PDE, int LEVELS, int ST>
size_t smem_bytes(const Geom& g) {
    return (size_t)(cluster_rows(g.ny) + 2) * g.py * pde_nf(PDE, LAT) * LEVELS * sizeof(typename Storage<ST>::S);
}

template <int LAT, int PDE, int LEVELS, int ST>
cudaError_t launch(const ClusterArgs& a) {
    using T = typename Storage<ST>::T;
    auto kern = k_cluster<LAT, PDE, LEVELS, ST>;
    const size_t smem = smem_bytes<LAT, PDE, LEVELS, ST>(a.g);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kClusterCtas, 1, 1);
    cfg.blockDim = dim3(kClusterThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = a.stream;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kClusterCtas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // Whether the device schedules such a cluster: asked, and the attributes set, once on every device.
    static std::atomic<int> known[kMaxDevices];   // 0 not asked, 1 yes, 2 no
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    int fits = e == cudaSuccess && dev < kMaxDevices ? known[dev].load(std::memory_order_acquire) : 0;
    if (e == cudaSuccess && fits == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        int clusters = 0;
        cudaLaunchConfig_t top = cfg;
        top.dynamicSmemBytes = kClusterSmem;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kern, &top);
        fits = e == cudaSuccess && clusters > 0 ? 1 : 2;
        if (dev < kMaxDevices) known[dev].store(fits, std::memory_order_release);
    }
    if (e == cudaSuccess && fits == 2) return cudaErrorNotSupported;
    ClusterLevels gl;
    for (int i = 0; i < 3; ++i) {
        gl.lev[i] = a.lev[i];
        gl.out[i] = a.out[i];
    }
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kern, a.g, gl, a.cur, *static_cast<const Coef<T>*>(a.coef), a.ex, a.nsteps);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

template <int LAT, int PDE, int LEVELS, int ST>
ClusterFn pick(const Geom& g) {
    return smem_bytes<LAT, PDE, LEVELS, ST>(g) <= kClusterSmem ? launch<LAT, PDE, LEVELS, ST> : nullptr;
}
template <int LAT, int PDE, int LEVELS>
ClusterFn pick_st(int st, const Geom& g) {
    if (st == ST_F64) return pick<LAT, PDE, LEVELS, ST_F64>(g);
    if (st == ST_F32) return pick<LAT, PDE, LEVELS, ST_F32>(g);
    return pick<LAT, PDE, LEVELS, ST_BF16>(g);
}
template <int LAT, int PDE>
ClusterFn pick_lev(int levels, int st, const Geom& g) {
    return levels == 2 ? pick_st<LAT, PDE, 2>(st, g) : pick_st<LAT, PDE, 3>(st, g);
}

}  // namespace

ClusterFn find_cluster(int lat, int pde, int levels, int st, const Geom& g) {
    if (g.dim != 2 || g.nx < g.gx) return nullptr;
    // One cluster is 16 of 152 SMs, so it wins while a step's arithmetic stays below what launching over
    // all of them costs.  Per step, cluster
    // against one chained launch: LCDE FP32 64 x 64 0.54 us against 2.2, 100 x 120 0.73 against 2.1, but
    // 120 x 500 2.67 against 1.96; NSE 60 x 60 1.0 and 100 x 100 1.5 against 2.2, 125 x 146 2.4 against 2.3;
    // NCDE 100 x 120 2.0 against 2.2.  FP64 arithmetic (a sixtieth of the FP32 rate) moves the line to a
    // fifth for the LCDE, and the nonlinear PDEs' always belongs on all SMs.
    const long long nodes = (long long)g.nx * g.ny;
    const long long cost = (pde == PDE_LCDE ? 2 : pde == PDE_NCDE ? 3 : 5) * (levels - 1);
    if (st == ST_F64 && pde != PDE_LCDE) return nullptr;
    if (nodes * cost * (st == ST_F64 ? 5 : 1) > 65536) return nullptr;
    if (lat == LAT_D2Q5) return pde == PDE_LCDE ? pick_lev<LAT_D2Q5, PDE_LCDE>(levels, st, g) : nullptr;
    if (lat != LAT_D2Q9) return nullptr;
    if (pde == PDE_LCDE) return pick_lev<LAT_D2Q9, PDE_LCDE>(levels, st, g);
    if (pde == PDE_NCDE) return pick_lev<LAT_D2Q9, PDE_NCDE>(levels, st, g);
    return pick_lev<LAT_D2Q9, PDE_NSE>(levels, st, g);
}

}  // namespace mmfd
