// k_util.cu -- layout conversion (dense user arrays <-> ghosted storage) and deterministic
// FP64 reductions (sum, max |v|, non-finite count, GRE of Sec. IV and max-norm).
#include <cuda_bf16.h>

#include <type_traits>

#include "kernels.h"
#include "stencil.cuh"

namespace mmfd {

namespace {

constexpr int kRedBlocks = 608;   // 4 x 152 SMs
constexpr int kRedThreads = 256;

// Value of a stored element: the reference plus the stored offset, formed in FP64 so that an
// FP32 / BF16 offset comes back exactly (FP64 levels hold values, ref 0).
template <int ST>
__device__ __forceinline__ double load_st(const void* base, long long i, double ref) {
    using Tr = Storage<ST>;
    return ref + (double)Tr::raw(static_cast<const typename Tr::S*>(base) + i);
}

// Four consecutive values of a dense FP64 / FP32 source row, 16-byte aligned.
__device__ __forceinline__ void ld4_src(const void* src, int dtype, long long i, double v[4]) {
    if (dtype == 0) {
        const double2 a = *reinterpret_cast<const double2*>(static_cast<const double*>(src) + i);
        const double2 b = *reinterpret_cast<const double2*>(static_cast<const double*>(src) + i + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
        const float4 a = *reinterpret_cast<const float4*>(static_cast<const float*>(src) + i);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    }
}

// Four consecutive stored values starting at a 16-byte aligned slot.
template <int ST>
__device__ __forceinline__ void ld4_st(const void* base, long long i, double ref, double v[4]) {
    using Tr = Storage<ST>;
    using S = typename Tr::S;
    const S* p = static_cast<const S*>(base) + i;
    if constexpr (ST == ST_F32) {
        // FP32 levels hold v - ref: the value is ref + stored, formed in FP64 (as load_st)
        const float4 a = *reinterpret_cast<const float4*>(p);
        v[0] = ref + (double)a.x; v[1] = ref + (double)a.y; v[2] = ref + (double)a.z; v[3] = ref + (double)a.w;
    } else if constexpr (ST == ST_F64) {
        const double2 a = *reinterpret_cast<const double2*>(p);
        const double2 b = *reinterpret_cast<const double2*>(p + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = ref + (double)Tr::raw(p + k);
    }
}

// ------------------------------------------------------------------ level <-> dense copies
// A copy walks rows (r = y + z ny) x column blocks: a CTA of 256 threads is tx column threads by
// 256 / tx rows, with tx the power of two that covers a row (host-chosen, at most 256), so that
// short rows still fill the CTA; every thread moves four columns of kCopyRows rows, all loads
// issued before the first store.  One launch covers every field (blockIdx.z) and, on the pack
// side, both levels a three-level start sets.  The copies are bound by HBM bytes.
//   VEC: the thread's four columns are neighbours and move as 16-byte vectors (nx a multiple of 4,
//        16-byte aligned dense buffers); otherwise they are tx apart and move one by one, each
//        access coalesced over the warp, so an odd nx costs no partial vectors.
//   F32: FP32 arithmetic for an FP32 dense buffer whose reference FP32 holds exactly.  Storing: the
//        exact difference of two FP32 values fits in FP64 unless their exponents are more than 29
//        apart, and then both forms round to the larger operand.  Reading: likewise for the sum
//        (a sum that FP64 cannot hold lies within 2^-5 ulp of its larger operand, not at a tie).
//        FP64 runs at a sixtieth of the FP32 rate on this part, so the FP64 forms are bound by
//        its conversions and adds.
constexpr int kCopyThreads = 256;
constexpr int kCopyRows = 4;

struct CopyArgs {
    const void* src[4];   // pack: dense fields; unpack: the level's fields
    void* dst[4];         // pack: the level's fields; unpack: dense fields
    void* dst2[4];        // pack: the same fields of a second level (or null)
    double ref[4];
    int dense_f32;        // element type of the dense side
    int tx;               // column threads per row
    long long r_lo, r_hi;
};

// v (columns x .. x+3, or the one column x) into one stored row, with its x ghost images.
template <int ST, bool VEC>
__device__ __forceinline__ void put_row(typename Storage<ST>::S* row, const Geom& g, int x,
                                        const typename Storage<ST>::S (&v)[VEC ? 4 : 1]) {
    if constexpr (!VEC) {
        row[x] = v[0];
    } else if constexpr (ST == ST_F32) {
        *reinterpret_cast<float4*>(row + x) = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (ST == ST_F64) {
        reinterpret_cast<double2*>(row + x)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2*>(row + x)[1] = make_double2(v[2], v[3]);
    } else {
        const unsigned lo = (unsigned)__bfloat16_as_ushort(v[0]) | ((unsigned)__bfloat16_as_ushort(v[1]) << 16);
        const unsigned hi = (unsigned)__bfloat16_as_ushort(v[2]) | ((unsigned)__bfloat16_as_ushort(v[3]) << 16);
        *reinterpret_cast<uint2*>(row + x) = make_uint2(lo, hi);
    }
#pragma unroll
    for (int k = 0; k < (VEC ? 4 : 1); ++k) {
        if (x + k < g.gx) row[x + k + g.nx] = v[k];
        if (x + k >= g.nx - g.gx) row[x + k - g.nx] = v[k];
    }
}

// The thread's column q of its four (VEC: the first column of the vector for q = 0).
template <bool VEC>
__device__ __forceinline__ int copy_col(int block, int lane_x, int tx, int q) {
    return VEC ? (block * tx + lane_x) * 4 : (block * 4 + q) * tx + lane_x;
}

// The stored values of the dense elements at .. (4 with VEC, else 1).
template <int ST, bool VEC, bool F32>
__device__ __forceinline__ void pack_values(const CopyArgs& a, int f, long long at, typename Storage<ST>::S* v) {
    using Tr = Storage<ST>;
    using T = typename Tr::T;
    const double ref = a.ref[f];
    if constexpr (F32) {
        const float rf = (float)ref;
        const float* p = static_cast<const float*>(a.src[f]) + at;
        if constexpr (VEC) {
            const float4 w = *reinterpret_cast<const float4*>(p);
            v[0] = Tr::pack_raw(w.x - rf, 0u);
            v[1] = Tr::pack_raw(w.y - rf, 0u);
            v[2] = Tr::pack_raw(w.z - rf, 0u);
            v[3] = Tr::pack_raw(w.w - rf, 0u);
        } else {
            v[0] = Tr::pack_raw(*p - rf, 0u);
        }
    } else {
        double w[VEC ? 4 : 1];
        if constexpr (VEC) ld4_src(a.src[f], a.dense_f32, at, w);
        else w[0] = a.dense_f32 ? (double)static_cast<const float*>(a.src[f])[at] : static_cast<const double*>(a.src[f])[at];
#pragma unroll
        for (int k = 0; k < (VEC ? 4 : 1); ++k) v[k] = Tr::pack_raw((T)(w[k] - ref), 0u);   // offset formed in FP64
    }
}

template <int ST, bool VEC, bool F32>
__global__ void __launch_bounds__(kCopyThreads) k_pack(Geom g, const __grid_constant__ CopyArgs a) {
    using S = typename Storage<ST>::S;
    static_assert(!(F32 && ST == ST_F64), "FP64 storage keeps the FP64 path");
    constexpr int NV = VEC ? 1 : 4;       // accesses per row
    constexpr int W = VEC ? 4 : 1;        // columns per access
    const int f = blockIdx.z;
    const int lx = threadIdx.x & (a.tx - 1);
    const int ly = threadIdx.x / a.tx, ty = kCopyThreads / a.tx;
    S* d = static_cast<S*>(a.dst[f]);
    S* d2 = static_cast<S*>(a.dst2[f]);
    for (long long rb = a.r_lo + (long long)blockIdx.y * (ty * kCopyRows); rb < a.r_hi;
         rb += (long long)gridDim.y * (ty * kCopyRows)) {
        S sv[kCopyRows][4];
#pragma unroll
        for (int i = 0; i < kCopyRows; ++i) {
            const long long r = rb + ly + i * ty;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int x = copy_col<VEC>(blockIdx.x, lx, a.tx, q);
                if (r < a.r_hi && x < g.nx) pack_values<ST, VEC, F32>(a, f, (r - a.r_lo) * g.nx + x, &sv[i][q]);
            }
        }
        bool edges = false;
#pragma unroll
        for (int i = 0; i < kCopyRows; ++i) {
            const long long r = rb + ly + i * ty;
            if (r >= a.r_hi) continue;
            const int y = g.dim == 3 ? (int)(r % g.ny) : (int)r;
            const int z = g.dim == 3 ? (int)(r / g.ny) : 0;
            edges = edges || y == 0 || y == g.ny - 1 || (g.dim == 3 && (z == 0 || z == g.nz - 1));
            S* row = d + g.at(0, y, z);
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int x = copy_col<VEC>(blockIdx.x, lx, a.tx, q);
                if (x >= g.nx) continue;
                S v[W];
#pragma unroll
                for (int k = 0; k < W; ++k) v[k] = sv[i][q + k];
                put_row<ST, VEC>(row, g, x, v);
                if (d2) put_row<ST, VEC>(d2 + (row - d), g, x, v);
            }
        }
        // The images of edge rows in the ghost rows and planes: few rows have any, and their values
        // are read again here, since carried along in the unrolled copy above the image stores took
        // 245 registers (one CTA per SM: 676 us for three 4095 x 4096 fields against 80).
        if (edges) {
#pragma unroll 1
            for (int i = 0; i < kCopyRows; ++i) {
                const long long r = rb + ly + i * ty;
                if (r >= a.r_hi) break;
                const int y = g.dim == 3 ? (int)(r % g.ny) : (int)r;
                const int z = g.dim == 3 ? (int)(r / g.ny) : 0;
#pragma unroll 1
                for (int m = 1; m < 9; ++m) {
                    const int my = m % 3, mz = m / 3;   // 0: the row / plane itself, 1: its low image, 2: its high one
                    if ((my == 1 && y != g.ny - 1) || (my == 2 && y != 0)) continue;
                    if (mz != 0 && (g.dim != 3 || (mz == 1 && z != g.nz - 1) || (mz == 2 && z != 0))) continue;
                    const long long at = g.at(0, my == 0 ? y : my == 1 ? -1 : g.ny, mz == 0 ? z : mz == 1 ? -1 : g.nz);
#pragma unroll 1
                    for (int q = 0; q < NV; ++q) {
                        const int x = copy_col<VEC>(blockIdx.x, lx, a.tx, q);
                        if (x >= g.nx) break;
                        S v[W];
                        pack_values<ST, VEC, F32>(a, f, (r - a.r_lo) * g.nx + x, v);
                        put_row<ST, VEC>(d + at, g, x, v);
                        if (d2) put_row<ST, VEC>(d2 + at, g, x, v);
                    }
                }
            }
        }
    }
}

// FP32 -> FP64, exact, without the FP64 pipe for normal numbers and zeros (its conversions run at
// the FP64 rate): the exponent is rebiased and the mantissa moved as integers.
__device__ __forceinline__ double widen(float v) {
    const unsigned b = __float_as_uint(v);
    const unsigned e = b & 0x7f800000u;
    if (e == 0x7f800000u || (e == 0u && (b & 0x007fffffu) != 0u)) return (double)v;   // inf, nan, subnormal
    const unsigned hi = e == 0u ? 0u : (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u);   // zero: +0, as 0 + v gives
    return __hiloint2double((int)hi, (int)(b << 29));
}

template <int ST, bool VEC, bool F32>
__global__ void __launch_bounds__(kCopyThreads) k_unpack(Geom g, const __grid_constant__ CopyArgs a) {
    using Tr = Storage<ST>;
    using S = typename Tr::S;
    using T = typename Tr::T;
    static_assert(!(F32 && ST == ST_F64), "FP64 storage keeps the FP64 path");
    constexpr int NV = VEC ? 1 : 4;
    const int f = blockIdx.z;
    const double ref = a.ref[f];
    const int lx = threadIdx.x & (a.tx - 1);
    const int ly = threadIdx.x / a.tx, ty = kCopyThreads / a.tx;
    const S* lev = static_cast<const S*>(a.src[f]);
    auto value = [&](T v) -> double {
        if constexpr (ST == ST_F64) return ref + v;
        else return ref == 0.0 ? widen(v) : ref + widen(v);
    };
    for (long long rb = a.r_lo + (long long)blockIdx.y * (ty * kCopyRows); rb < a.r_hi;
         rb += (long long)gridDim.y * (ty * kCopyRows)) {
        T v[kCopyRows][4];
#pragma unroll
        for (int i = 0; i < kCopyRows; ++i) {
            const long long r = rb + ly + i * ty;
            if (r >= a.r_hi) continue;
            const S* row = lev + (g.dim == 3 ? g.at(0, (int)(r % g.ny), (int)(r / g.ny)) : g.at(0, (int)r, 0));
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int x = copy_col<VEC>(blockIdx.x, lx, a.tx, q);
                if (x >= g.nx) continue;
                if constexpr (!VEC) {
                    v[i][q] = Tr::raw(row + x);
                } else if constexpr (ST == ST_F32) {
                    const float4 w = *reinterpret_cast<const float4*>(row + x);
                    v[i][0] = w.x; v[i][1] = w.y; v[i][2] = w.z; v[i][3] = w.w;
                } else if constexpr (ST == ST_F64) {
                    const double2 w0 = *reinterpret_cast<const double2*>(row + x);
                    const double2 w1 = *reinterpret_cast<const double2*>(row + x + 2);
                    v[i][0] = w0.x; v[i][1] = w0.y; v[i][2] = w1.x; v[i][3] = w1.y;
                } else {
                    const uint2 w = *reinterpret_cast<const uint2*>(row + x);
                    v[i][0] = __uint_as_float(w.x << 16); v[i][1] = __uint_as_float(w.x & 0xffff0000u);
                    v[i][2] = __uint_as_float(w.y << 16); v[i][3] = __uint_as_float(w.y & 0xffff0000u);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kCopyRows; ++i) {
            const long long r = rb + ly + i * ty;
            if (r >= a.r_hi) continue;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int x = copy_col<VEC>(blockIdx.x, lx, a.tx, q);
                if (x >= g.nx) continue;
                const long long at = (r - a.r_lo) * g.nx + x;
                if (a.dense_f32) {
                    float* o = static_cast<float*>(a.dst[f]) + at;
                    float w[VEC ? 4 : 1];
#pragma unroll
                    for (int k = 0; k < (VEC ? 4 : 1); ++k) {
                        if constexpr (F32) w[k] = __fadd_rn((float)ref, v[i][q + k]);
                        else w[k] = (float)(ref + (double)v[i][q + k]);
                    }
                    if constexpr (VEC) *reinterpret_cast<float4*>(o) = make_float4(w[0], w[1], w[2], w[3]);
                    else *o = w[0];
                } else {
                    double* o = static_cast<double*>(a.dst[f]) + at;
                    if constexpr (VEC) {
                        reinterpret_cast<double2*>(o)[0] = make_double2(value(v[i][0]), value(v[i][1]));
                        reinterpret_cast<double2*>(o)[1] = make_double2(value(v[i][2]), value(v[i][3]));
                    } else {
                        *o = value(v[i][q]);
                    }
                }
            }
        }
    }
}

// Rows [r_lo, r_hi) (r = y + z ny) of every field of a level to / from dense buffers in one launch
// (blockIdx.z = field): the halo-row exchange of a slab decomposition moves a few rows per step,
// so the launch count matters more than the bandwidth.
struct RowBufs {
    const void* src[4];
    void* dst[4];
    double ref[4];
};

template <int ST>
__global__ void k_rows_pack(Geom g, RowBufs b, int src_dtype, void* __restrict__ level, long long r_lo, long long r_hi) {
    using Tr = Storage<ST>;
    using S = typename Tr::S;
    using T = typename Tr::T;
    const int f = blockIdx.z;
    S* d = static_cast<S*>(level) + (size_t)f * g.fs;
    const double ref = b.ref[f];
    for (long long r = r_lo + blockIdx.y; r < r_hi; r += gridDim.y) {
        const int y = (int)(r % g.ny);
        const int z = (int)(r / g.ny);
        const long long base = (r - r_lo) * g.nx;
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < g.nx; x += gridDim.x * blockDim.x) {
            const long long i = base + x;
            const double v = src_dtype == 0 ? static_cast<const double*>(b.src[f])[i] : (double)static_cast<const float*>(b.src[f])[i];
            const S sv = Tr::pack_raw((T)(v - ref), 0u);
            if (g.dim == 3) store_with_ghosts<3>(d, g, x, y, z, sv);
            else store_with_ghosts<2>(d, g, x, y, z, sv);
        }
    }
}

template <int ST>
__global__ void k_rows_unpack(Geom g, RowBufs b, int dst_dtype, const void* __restrict__ level, long long r_lo,
                              long long r_hi) {
    const int f = blockIdx.z;
    const char* src = static_cast<const char*>(level) + (size_t)f * g.fs * g.es;
    const double ref = b.ref[f];
    for (long long r = r_lo + blockIdx.y; r < r_hi; r += gridDim.y) {
        const int y = (int)(r % g.ny);
        const int z = (int)(r / g.ny);
        const long long base = (r - r_lo) * g.nx;
        const long long sbase = g.at(0, y, z);
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < g.nx; x += gridDim.x * blockDim.x) {
            const double v = load_st<ST>(src, sbase + x, ref);
            if (dst_dtype == 0)
                static_cast<double*>(b.dst[f])[base + x] = v;
            else
                static_cast<float*>(b.dst[f])[base + x] = (float)v;
        }
    }
}

struct Acc4 {
    double a, b, c, d;
};

__device__ __forceinline__ Acc4 combine(int op, Acc4 x, Acc4 y) {
    if (op == 1) return {fmax(x.a, y.a), 0, 0, 0};
    if (op == 3) return {x.a + y.a, x.b + y.b, fmax(x.c, y.c), fmax(x.d, y.d)};
    return {x.a + y.a, 0, 0, 0};
}

// Fixed-order block reduction: block b covers rows b, b + nblocks, ... (row = y + z ny) and, in
// each row, columns threadIdx.x, + blockDim.x, ...; it reduces through shared memory in a fixed
// tree, so the result is bitwise reproducible.
// The operation is a template parameter (0 sum, 1 max |v|, 2 non-finite count, 3 error norms):
// with a run-time switch in the element loop every element paid for all four accumulators.
template <int ST, int OPT>
__global__ void __launch_bounds__(kRedThreads) k_reduce_parts(Geom g, const void* __restrict__ lev, double fref,
                                                              const void* __restrict__ ref, int ref_dtype,
                                                              Acc4* __restrict__ parts) {
    constexpr int op = OPT;
    __shared__ Acc4 sh[kRedThreads];
    const long long rows = (long long)g.ny * g.nz;
    Acc4 acc = {0, 0, 0, 0};
    constexpr int cop = op == 2 ? 0 : op;
    const bool vec = OPT != 3 && (g.nx & 3) == 0;
    for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
        const int y = (int)(r % g.ny);
        const int z = (int)(r / g.ny);
        const long long sbase = g.at(0, y, z);
        const long long dbase = r * g.nx;
        if (vec) {
            // four columns per thread per pass (the row starts on a 16-byte boundary)
            for (int x = threadIdx.x << 2; x < g.nx; x += blockDim.x << 2) {
                double v[4];
                ld4_st<ST>(lev, sbase + x, fref, v);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (OPT == 0) acc.a += v[k];
                    else if constexpr (OPT == 1) acc.a = fmax(acc.a, fabs(v[k]));
                    else if constexpr (OPT == 2) acc.a += isfinite(v[k]) ? 0.0 : 1.0;
                }
            }
            continue;
        }
        for (int x = threadIdx.x; x < g.nx; x += blockDim.x) {
            const double v = load_st<ST>(lev, sbase + x, fref);
            Acc4 e;
            if (op == 0) {
                e = {v, 0, 0, 0};
            } else if (op == 1) {
                e = {fabs(v), 0, 0, 0};
            } else if (op == 2) {
                e = {isfinite(v) ? 0.0 : 1.0, 0, 0, 0};
            } else {
                const long long i = dbase + x;
                const double rv = ref_dtype == 0 ? static_cast<const double*>(ref)[i] : (double)static_cast<const float*>(ref)[i];
                e = {fabs(v - rv), fabs(rv), fabs(v - rv), fabs(rv)};
                if (!isfinite(v)) e = {INFINITY, fabs(rv), INFINITY, fabs(rv)};
            }
            acc = combine(cop, acc, e);
        }
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = kRedThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = combine(cop, sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) parts[blockIdx.x] = sh[0];
}

__global__ void __launch_bounds__(kRedThreads) k_reduce_final(const Acc4* __restrict__ parts, int nparts, int op,
                                                              double* __restrict__ out) {
    __shared__ Acc4 sh[kRedThreads];
    Acc4 acc = {0, 0, 0, 0};
    const int cop = op == 2 ? 0 : op;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc = combine(cop, acc, parts[i]);
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = kRedThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = combine(cop, sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sh[0].a;
        out[1] = sh[0].b;
        out[2] = sh[0].c;
        out[3] = sh[0].d;
    }
}

// Launch shape of a copy: column threads per row and the grid.
dim3 copy_grid(const Geom& g, int nf, long long rows, int* tx) {
    int t = 8;
    while (t < kCopyThreads && t * 4 < g.nx) t *= 2;
    *tx = t;
    const int per = kCopyThreads / t * kCopyRows;
    const long long by = (rows + per - 1) / per;
    return dim3((unsigned)((g.nx + 4 * t - 1) / (4 * t)), (unsigned)(by < 65535 ? by : 65535), (unsigned)nf);
}

bool aligned16(const void* const* p, int nf) {
    for (int f = 0; f < nf; ++f)
        if (reinterpret_cast<uintptr_t>(p[f]) & 15) return false;
    return true;
}

// Whether FP32 arithmetic gives the FP64 form's result for every field (see the copies' F32).
bool copy_f32(int st, int dense_f32, const double* refs, int nf) {
    if (st == ST_F64 || !dense_f32) return false;
    for (int f = 0; f < nf; ++f)
        if ((double)(float)refs[f] != refs[f]) return false;
    return true;
}

}  // namespace

namespace {

// The boundary ring of a grid (nodes with x = 0 / nx - 1, y = 0 / ny - 1, and z = 0 / nz - 1 in
// 3D), enumerated face by face without repeats: in 3D the two z faces whole, then the two y faces
// between them, then the two x faces between those; in 2D the y faces and then the x faces.
__host__ __device__ inline long long ring_nodes(const Geom& g) {
    const long long zn = g.dim == 3 ? g.nz - 2 : 1;
    return (g.dim == 3 ? 2ll * g.nx * g.ny : 0ll) + 2ll * g.nx * zn + 2ll * (g.ny - 2) * zn;
}

template <typename E>
__global__ void k_ring_copy(Geom g, const E* __restrict__ src, E* __restrict__ dst, long long count) {
    const long long zn = g.dim == 3 ? g.nz - 2 : 1;
    const int z0 = g.dim == 3 ? 1 : 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        long long k = i;
        int x, y, z;
        const long long zface = g.dim == 3 ? (long long)g.nx * g.ny : 0;
        const long long yface = (long long)g.nx * zn;
        const long long xface = (long long)(g.ny - 2) * zn;
        if (k < 2 * zface) {
            z = k < zface ? 0 : g.nz - 1;
            const long long r = k % zface;
            x = (int)(r % g.nx);
            y = (int)(r / g.nx);
        } else if ((k -= 2 * zface) < 2 * yface) {
            y = k < yface ? 0 : g.ny - 1;
            const long long r = k % yface;
            x = (int)(r % g.nx);
            z = z0 + (int)(r / g.nx);
        } else {
            k -= 2 * yface;
            x = k < xface ? 0 : g.nx - 1;
            const long long r = k % xface;
            y = 1 + (int)(r % (g.ny - 2));
            z = z0 + (int)(r / (g.ny - 2));
        }
        const long long at = g.at(x, y, z);
        for (int f = 0; f < g.nf; ++f) dst[(long long)f * g.fs + at] = src[(long long)f * g.fs + at];
    }
}

}  // namespace

cudaError_t launch_ring_copy(const Geom& g, const void* src_level, void* dst_level, cudaStream_t s) {
    const long long count = ring_nodes(g);
    if (count <= 0) return cudaSuccess;
    const int blocks = (int)((count + 255) / 256 < 1184 ? (count + 255) / 256 : 1184);
    if (g.es == 8) k_ring_copy<unsigned long long><<<blocks, 256, 0, s>>>(g, static_cast<const unsigned long long*>(src_level), static_cast<unsigned long long*>(dst_level), count);
    else if (g.es == 4) k_ring_copy<unsigned int><<<blocks, 256, 0, s>>>(g, static_cast<const unsigned int*>(src_level), static_cast<unsigned int*>(dst_level), count);
    else k_ring_copy<unsigned short><<<blocks, 256, 0, s>>>(g, static_cast<const unsigned short*>(src_level), static_cast<unsigned short*>(dst_level), count);
    return cudaGetLastError();
}

cudaError_t launch_pack(const Geom& g, int st, const void* const* src, int nf, int src_dtype, void* level, void* level2,
                        int field0, const double* refs, cudaStream_t s) {
    if (nf < 1 || nf > 4) return cudaErrorInvalidValue;
    CopyArgs a{};
    for (int f = 0; f < nf; ++f) {
        const size_t at = (size_t)(field0 + f) * g.fs * g.es;
        a.src[f] = src[f];
        a.dst[f] = static_cast<char*>(level) + at;
        a.dst2[f] = level2 ? static_cast<char*>(level2) + at : nullptr;
        a.ref[f] = refs[f];
    }
    a.dense_f32 = src_dtype == 1 ? 1 : 0;   // 1: FP32 (MMFD_DT_F32)
    a.r_hi = (long long)g.ny * g.nz;
    const dim3 grid = copy_grid(g, nf, a.r_hi, &a.tx);
    const bool vec = (g.nx & 3) == 0 && aligned16(src, nf);
    const bool f32 = copy_f32(st, a.dense_f32, refs, nf);
#define MMFD_PACK(ST, F) \
    (vec ? k_pack<ST, true, F><<<grid, kCopyThreads, 0, s>>>(g, a) : k_pack<ST, false, F><<<grid, kCopyThreads, 0, s>>>(g, a))
    if (st == ST_F64) MMFD_PACK(ST_F64, false);
    else if (st == ST_F32 && f32) MMFD_PACK(ST_F32, true);
    else if (st == ST_F32) MMFD_PACK(ST_F32, false);
    else if (f32) MMFD_PACK(ST_BF16, true);
    else MMFD_PACK(ST_BF16, false);
#undef MMFD_PACK
    return cudaGetLastError();
}

cudaError_t launch_unpack(const Geom& g, int st, const void* level, int field0, int nf, const double* refs,
                          void* const* dst, int dst_dtype, cudaStream_t s) {
    if (nf < 1 || nf > 4) return cudaErrorInvalidValue;
    CopyArgs a{};
    for (int f = 0; f < nf; ++f) {
        a.src[f] = static_cast<const char*>(level) + (size_t)(field0 + f) * g.fs * g.es;
        a.dst[f] = dst[f];
        a.ref[f] = refs[f];
    }
    a.dense_f32 = dst_dtype == 1 ? 1 : 0;
    a.r_hi = (long long)g.ny * g.nz;
    const dim3 grid = copy_grid(g, nf, a.r_hi, &a.tx);
    const bool vec = (g.nx & 3) == 0 && aligned16(dst, nf);
    const bool f32 = copy_f32(st, a.dense_f32, refs, nf);
#define MMFD_UNPACK(ST, F) \
    (vec ? k_unpack<ST, true, F><<<grid, kCopyThreads, 0, s>>>(g, a) : k_unpack<ST, false, F><<<grid, kCopyThreads, 0, s>>>(g, a))
    if (st == ST_F64) MMFD_UNPACK(ST_F64, false);
    else if (st == ST_F32 && f32) MMFD_UNPACK(ST_F32, true);
    else if (st == ST_F32) MMFD_UNPACK(ST_F32, false);
    else if (f32) MMFD_UNPACK(ST_BF16, true);
    else MMFD_UNPACK(ST_BF16, false);
#undef MMFD_UNPACK
    return cudaGetLastError();
}

cudaError_t launch_rows(const Geom& g, int st, bool pack, const void* const* bufs, int nf, int dtype, void* level,
                        const double* refs, long long r_lo, long long r_hi, cudaStream_t s) {
    if (nf < 1 || nf > 4) return cudaErrorInvalidValue;
    if (r_hi <= r_lo) return cudaSuccess;
    RowBufs b{};
    for (int f = 0; f < nf; ++f) {
        if (pack) b.src[f] = bufs[f];
        else b.dst[f] = const_cast<void*>(bufs[f]);
        b.ref[f] = refs[f];
    }
    const long long rows = r_hi - r_lo;
    const dim3 blocks((unsigned)((g.nx + 255) / 256 < 64 ? (g.nx + 255) / 256 : 64),
                      (unsigned)(rows < 65535 ? rows : 65535), (unsigned)nf);
    if (pack) {
        if (st == ST_F64) k_rows_pack<ST_F64><<<blocks, 256, 0, s>>>(g, b, dtype, level, r_lo, r_hi);
        else if (st == ST_F32) k_rows_pack<ST_F32><<<blocks, 256, 0, s>>>(g, b, dtype, level, r_lo, r_hi);
        else k_rows_pack<ST_BF16><<<blocks, 256, 0, s>>>(g, b, dtype, level, r_lo, r_hi);
    } else {
        if (st == ST_F64) k_rows_unpack<ST_F64><<<blocks, 256, 0, s>>>(g, b, dtype, level, r_lo, r_hi);
        else if (st == ST_F32) k_rows_unpack<ST_F32><<<blocks, 256, 0, s>>>(g, b, dtype, level, r_lo, r_hi);
        else k_rows_unpack<ST_BF16><<<blocks, 256, 0, s>>>(g, b, dtype, level, r_lo, r_hi);
    }
    return cudaGetLastError();
}

int reduce_parts_needed() { return kRedBlocks * 4; }  // doubles (Acc4 per block)

cudaError_t launch_reduce(const Geom& g, int st, const void* level, int field, double fref, int op,
                          const void* ref, int ref_dtype, double* d_partials, int nparts, double* d_out,
                          cudaStream_t s) {
    (void)nparts;
    const char* lev = static_cast<const char*>(level) + (size_t)field * g.fs * g.es;
    Acc4* parts = reinterpret_cast<Acc4*>(d_partials);
    auto parts_kernel = [&](auto stc) -> void {
        constexpr int SC = decltype(stc)::value;
        switch (op) {
            case 0: k_reduce_parts<SC, 0><<<kRedBlocks, kRedThreads, 0, s>>>(g, lev, fref, ref, ref_dtype, parts); break;
            case 1: k_reduce_parts<SC, 1><<<kRedBlocks, kRedThreads, 0, s>>>(g, lev, fref, ref, ref_dtype, parts); break;
            case 2: k_reduce_parts<SC, 2><<<kRedBlocks, kRedThreads, 0, s>>>(g, lev, fref, ref, ref_dtype, parts); break;
            default: k_reduce_parts<SC, 3><<<kRedBlocks, kRedThreads, 0, s>>>(g, lev, fref, ref, ref_dtype, parts); break;
        }
    };
    if (st == ST_F64) parts_kernel(std::integral_constant<int, ST_F64>{});
    else if (st == ST_F32) parts_kernel(std::integral_constant<int, ST_F32>{});
    else parts_kernel(std::integral_constant<int, ST_BF16>{});
    k_reduce_final<<<1, kRedThreads, 0, s>>>(parts, kRedBlocks, op, d_out);
    return cudaGetLastError();
}

}  // namespace mmfd
