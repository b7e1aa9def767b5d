// march3d_ring.cuh -- the plane ring of the class-form 3D marching kernels, refilled by the warps that read it.
//
// k_march3d keeps a producer warp; here the last warp through with a stage refills it.  These kernels'
// 16-row CTAs need the 128 registers a thread that 16 warps leave (17: 120), and their planes take
// long enough to compute that a refill a warp's skew later costs nothing.  The light linear kernel is
// the opposite case: without its producer cde3d_512 ran 243 us a step against 188.
#pragma once

#include "k_march3d.cuh"

namespace mmfd {

namespace {

// The sequence of input planes a CTA streams: its segments (tile, planes z0 .. z0 + nzs - 1), each with
// one halo plane on either side.  Items of H planes are dealt round-robin (H > 0); or (H < 0) each
// group of xs CTAs takes one balanced range of the (y tile, plane) pairs, y-tile-major, its CTAs the
// xs strips of the same range, so that the strips of a row advance plane by plane together and meet
// each other's halo columns in L2 (gridDim.x is a multiple of xs then).  (Counts of (y tile, plane)
// pairs fit an int: a level of more would not fit the device.)
struct PlaneCursor {
    int w, whi;              // items, or pairs, left
    int x0, y0, z0, np, i;   // segment, its input planes (0: no segment left), the next of them
};
template <int TY>
struct PlaneWalk {
    int xs, ys, nz, H, nitems;
    __device__ __forceinline__ PlaneWalk(const Geom& g, int H_, int nitems_)
        : xs((g.nx + 127) / 128), ys((g.ny + TY - 1) / TY), nz(g.nz), H(H_), nitems(nitems_) {}
    __device__ __forceinline__ void start(PlaneCursor& c) const {
        c.w = blockIdx.x;
        c.whi = nitems;
        if (H < 0) {
            const long long total = (long long)ys * nz;
            const long long groups = gridDim.x / xs, grp = blockIdx.x / xs;
            c.w = (int)(total * grp / groups);
            c.whi = (int)(total * (grp + 1) / groups);
        }
        next(c);
    }
    __device__ __forceinline__ void next(PlaneCursor& c) const {
        c.i = 0;
        c.np = 0;
        if (c.w >= c.whi) return;
        if (H > 0) {
            const int tiles = xs * ys, tile = c.w % tiles;
            c.x0 = tile % xs * 128;
            c.y0 = tile / xs * TY;
            c.z0 = c.w / tiles * H;
            c.np = min(H, nz - c.z0) + 2;
            c.w += gridDim.x;
        } else {
            c.x0 = (int)(blockIdx.x % xs) * 128;
            c.y0 = c.w / nz * TY;
            c.z0 = c.w % nz;
            c.np = min(nz - c.z0, c.whi - c.w) + 2;
            c.w += c.np - 2;
        }
    }
    __device__ __forceinline__ void advance(PlaneCursor& c) const {
        if (++c.i == c.np) next(c);
    }
};

// The plane ring of a 3D marching CTA of NWARP warps: NSTAGE stages of NIN boxes of BYTES bytes each, SLOT
// bytes apart, refilled in stream order by the last warp through with a stage.
template <int TY, int NWARP, int NIN, int NSTAGE, uint32_t BYTES, int SLOT>
struct PlaneRing {
    static constexpr int kHead = 128 * ((2 * NSTAGE * 8 + (int)sizeof(PlaneCursor) + 127) / 128);
    uint64_t* full;
    unsigned* done;      // warps through with each stage, counted on
    PlaneCursor* ld;     // the next plane to load
    unsigned char* ring;

    __device__ __forceinline__ explicit PlaneRing(unsigned char* smem_raw) {
        unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
        full = reinterpret_cast<uint64_t*>(smem);
        done = reinterpret_cast<unsigned*>(full + NSTAGE);
        ld = reinterpret_cast<PlaneCursor*>(full + 2 * NSTAGE);
        ring = smem + kHead;
    }
    __device__ __forceinline__ unsigned char* slot(int s, int q) const { return ring + (size_t)(s * NIN + q) * SLOT; }
    // one thread at a time: the next plane, if any is left, into stage s
    __device__ __forceinline__ void load_next(const TmapSet& maps, const PlaneWalk<TY>& walk, int s) const {
        PlaneCursor& c = *ld;
        if (c.np == 0) return;
        mbar_arrive_expect_tx(&full[s], NIN * BYTES);
#pragma unroll
        for (int q = 0; q < NIN; ++q) tma_load_3d(slot(s, q), &maps.m[q], &full[s], c.x0, c.y0, c.z0 + c.i);
        walk.advance(c);
    }
    // all threads, before the first use
    __device__ __forceinline__ void start(const TmapSet& maps, const PlaneWalk<TY>& walk) const {
        if (threadIdx.x == 0) {
#pragma unroll
            for (int s = 0; s < NSTAGE; ++s) {
                mbar_init(&full[s], 1);
                done[s] = 0;
            }
            fence_mbar_init();
#pragma unroll
            for (int q = 0; q < NIN; ++q) tma_prefetch_desc(&maps.m[q]);
            walk.start(*ld);
        }
        __syncthreads();
        chain_wait();
        if (threadIdx.x == 0)
            for (int s = 0; s < NSTAGE; ++s) load_next(maps, walk, s);
    }
    // a whole warp, when it has read stage s.  Refills happen one at a time and in order: a plane's last
    // warp counts after every warp has counted, and so refilled, the plane before.
    __device__ __forceinline__ void release(const TmapSet& maps, const PlaneWalk<TY>& walk, int s, int lane) const {
        __syncwarp();
        if (lane == 0) {
            __threadfence_block();
            if (atomicAdd_block(&done[s], 1u) % NWARP == NWARP - 1) {
                __threadfence_block();
                fence_proxy_async_smem();
                load_next(maps, walk, s);
            }
        }
    }
    // a warp whose wait ran out, at stage s with parity par: reports it and waits (bounded) for the copies
    // that may still land
    __device__ __forceinline__ void give_up(int* err, int s, uint32_t par, int lane) const {
        if (lane == 0) atomicExch(err, KERR_TMA_TIMEOUT);
        for (int k = 0; k < NSTAGE; ++k) {
            mbar_wait_bounded(&full[s], par);
            s = s + 1 == NSTAGE ? 0 : s + 1;
            if (s == 0) par ^= 1u;
        }
    }
};

template <int ST, int LEVELS, int NF, int TY, int NSTAGE>
constexpr size_t ring_smem() {
    return march3d_smem<ST, LEVELS, NF, TY, NSTAGE>() + 128;   // the load cursor
}

}  // namespace

}  // namespace mmfd
