// launch.cuh -- launching the kernels of a chain of dependent steps.
//
// A solve is a chain of short launches, each reading what the one before wrote.  A plain stream
// launch starts only after its predecessor has drained and its writes are flushed, and on this part
// consecutive short launches then start 4.1 us apart (and at multiples of 2.06 us above that).
// Launched as programmatic dependents, the next launch's CTAs are placed as soon as the last CTAs of the
// predecessor exit, set up their barriers, fetch their descriptors and wait on the device for its
// completion: 2.2 us per step of a 64 x 64 grid instead of 4.1, 7.3 instead of 10.3 on a 1024 x 1024
// NSE one.  The predecessor does not release its dependents early (griddepcontrol.launch_dependents
// right after its own wait): their CTAs then fill the free slots unevenly, and a launch that does
// not fill the GPU waits for its fullest SMs (1024 x 1024 NSE, three steps per launch: 20.8 us early
// against 15.8 at exit and 18.5 unchained).
//
// Rule every kernel launched this way keeps: chain_wait() before its first access to global memory
// that another kernel of the chain touches, reads and writes alike (it returns when the
// predecessor has completed and its writes are visible, and at once if there is none).  Such memory is
// read by plain loads through pointers that are not __restrict__: a read-only load (__ldg, or one the
// compiler derives from const __restrict__) is specified only for data that nothing writes while the
// kernel lives, and neither it nor an access to memory declared unaliased has to stay behind the
// wait's "memory" clobber.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <utility>

namespace mmfd {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Devices whose answers a launcher keeps (kernel attributes and occupancies belong to the device current
// at the call); on one beyond them it asks every time.
constexpr int kMaxDevices = 64;

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, bool chained,
                           A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    // (the error state is cleared as it is returned: left set, it would be taken for the next call's)
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

// CTAs of a kernel that an SM holds, the device's SMs and its L2 bytes.
struct Fit {
    int per_sm, sms;
    long long l2;
    int ctas() const { return per_sm * sms; }
};

// The Fit of `kern` at `threads` threads and `smem` bytes of dynamic shared memory a CTA on the current
// device, its shared memory limit raised on the way.  Asked once per device and kept in `known`, one word
// per device, so that concurrent host threads see either nothing or the whole answer.
template <typename... P>
cudaError_t fit_of(void (*kern)(P...), int threads, size_t smem, std::atomic<unsigned long long> (&known)[kMaxDevices], Fit* f) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    unsigned long long w = e == cudaSuccess && dev < kMaxDevices ? known[dev].load(std::memory_order_acquire) : 0;
    if (e == cudaSuccess && w == 0) {
        int per_sm = 0, sms = 0, l2 = 0;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e == cudaSuccess) {
            w = (unsigned long long)l2 << 32 | (unsigned long long)sms << 8 | (unsigned long long)(per_sm > 0 ? per_sm : 1);
            if (dev < kMaxDevices) known[dev].store(w, std::memory_order_release);
        }
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    *f = {(int)(w & 255), (int)(w >> 8 & 0xffffff), (long long)(w >> 32)};
    return cudaSuccess;
}

// Rows (planes) per work item of a marching launch: `tiles` columns of n rows are cut into equal segments
// of at least hmin and at most hmax rows, dealt round-robin to `slots` warps (CTAs), each segment
// streamed with `halo` further rows.  Picks the cut whose longest queue streams the fewest rows: for
// each number of rounds, the most segments that fit it.  (A rule on fill x h / (h + halo), which counted a
// last segment of two planes as a full one, took 85 planes per item at
// 512^3; the 3D LCDE step ran 193 us on it against 174, and 150 against 112 at 501 x 400 x 300.)
inline int march_height(long long tiles, int n, long long slots, int halo, int hmin, int hmax) {
    if (hmin > n) hmin = n;
    const long long smin = (n + hmax - 1) / hmax;   // segments of a column, at least
    const double work = (double)tiles * n / (double)slots;
    long long best = -1;
    int H = n < hmax ? n : hmax;
    for (long long r = (tiles * smin + slots - 1) / slots;; ++r) {
        const long long s = r * slots / tiles;
        const int h = (int)(s >= n ? 1 : (n + s - 1) / s);
        if (h < hmin && best >= 0) break;
        const int hh = h < hmin ? hmin : h;
        const long long rows = (tiles * ((n + hh - 1) / hh) + slots - 1) / slots * (hh + halo);
        if (best < 0 || rows < best) {
            best = rows;
            H = hh;
        }
        if (h <= hmin || work + (double)(r + 1) * halo >= (double)best) break;   // more rounds cannot be shorter
    }
    return H;
}

}  // namespace mmfd
