// kernels.h -- host-side entry points of the kernel families (type-erased launchers).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "mmfd_internal.h"

namespace mmfd {

// Up to 8 TMA tensor maps (nf fields x input levels), passed to a kernel as a grid constant.
struct TmapSet {
    CUtensorMap m[8];
};

// A launcher advances one (or `depth`) time level(s): reads level t (in0) and level t - dt
// (in1, three-level only) and writes level t + dt (out), all in the ghosted layout `g`.
// coef points at a Coef<double> or Coef<float> matching the storage type.
struct LaunchArgs {
    Geom g;
    const void* in0;
    const void* in1;
    void* out;
    const void* coef;
    StepExtra ex;
    cudaStream_t stream;
    int variant;          // kernel-shape variant chosen by the tuner (family specific)
    const TmapSet* maps;  // TMA descriptors of the input levels (march / blocked kernels)
    int H;                // rows (2D) or planes (3D) per CTA
    int* err;             // device error flag (bounded waits that ran out)
    const void* src[2];   // source levels t, t - dt (solvers with source terms; else null)
    const void* src_coef; // SrcCoef<double> or SrcCoef<float> matching the storage type
    double umom = 1.0;     // the NSE class kernels: factor of a uniform velocity in one step (Resolved::umom)
    const void* cls = nullptr; // NcdeClass<double> or NcdeClass<float> (the NCDE class kernels)
    bool chained = false; // a step of a chain on one stream: launched to overlap its predecessor's end (launch.cuh)
};
using LaunchFn = cudaError_t (*)(const LaunchArgs&);

// A launch advancing nsteps steps of a small 2D solve in one thread-block cluster: the level buffers
// lev[0 .. levels), level t in lev[cur]; afterwards level t + nsteps dt is in the buffer that as many
// single steps would leave it in, level t - dt (three levels) in that one's predecessor, and the
// other buffer is as it was.  An error (cudaErrorNotSupported if the device does not schedule the cluster)
// means that nothing was launched.
struct ClusterArgs {
    Geom g;
    void* lev[3];
    void* out[3];          // where the levels are written back, by the same indices: lev, or a spare buffer to time a launch
    int cur;
    const void* coef;
    StepExtra ex;          // step: that of the first new level
    int nsteps;
    cudaStream_t stream;
};
using ClusterFn = cudaError_t (*)(const ClusterArgs&);
// The cluster kernel of a solve, or null where one launch per step is the better choice.
ClusterFn find_cluster(int lat, int pde, int levels, int st, const Geom& g);

// One node per thread, neighbours read straight from the ghosted layout (any shape).
LaunchFn find_direct(int lat, int pde, int levels, int st);
// The same with source terms: src 1 (a source S, M_1F = 0 or S u folded) or 2 (S and M_1F fields).
LaunchFn find_direct_src(int lat, int pde, int levels, int st, int src);
// Row-marching 2D kernels fed by a TMA (cp.async.bulk.tensor) shared-memory ring.
LaunchFn find_march2d(int lat, int pde, int levels, int st);
// The same with source terms in the store epilogue (src as for find_direct_src; LCDE / NCDE).
LaunchFn find_march2d_src(int lat, int pde, int levels, int st, int src);
// Input rows per TMA box (stage) of the 2D marching kernel for this PDE; its tensor maps use
// boxes of 128 + 2 x 16 bytes by this many rows.
int march2d_rows_per_stage(int pde);
// 3D plane-marching kernels (z march, x-y tile staged in shared memory by TMA).
LaunchFn find_march3d(int lat, int pde, int levels, int st);
// Temporally blocked 2D kernel advancing `depth` levels per launch (two-level LCDE / NCDE;
// nullptr where unsupported) and the largest depth its ghost columns allow for storage st.
// It reads the level through the same 2-row-box tensor maps as k_march2d.
LaunchFn find_march2d_tb(int lat, int pde, int levels, int st, int depth);
int march2d_tb_max_depth(int st);
// The D2Q9 He-Luo NSE step in the lean streaming form (two levels), depth steps per launch: FP32 1 .. 3,
// FP64 1.
LaunchFn find_march2d_nse(int st, int depth);
// The temporally blocked one of these, FP32 / BF16 storage (depth 2 .. march2d_tb_nse_max_depth()).
LaunchFn find_march2d_tb_nse(int st, int depth);
int march2d_tb_nse_max_depth();
// The 2D theta-scheme kernels (FP32 / FP64 levels).  depth 0: the first pass of a step, from phi^n (in0)
// to rhs (written to src[0], stencil coef, a Coef block) and the first sweep's result (out, stencil
// src_coef, a SrcCoef block); depth >= 1: that many further sweeps (stencil coef, a Coef block; src[0] =
// rhs, its weight 1 / d in src_coef's W0[0]), up to march2d_tb_max_depth(st).  `end` picks the form with
// the rounding of single sweeps, for the last ones of a step (k_march2d_theta.cu).
LaunchFn find_march2d_theta(int lat, int st, int depth, bool end = false);
// The same with source terms in the store epilogue (src as for find_direct_src; LCDE / NCDE).
LaunchFn find_march3d_src(int lat, int pde, int levels, int st, int src);
// The 2D (D2Q9) and 3D (D3Q19) NCDE marching kernels in class form (NcdeClass, FP32 / FP64 storage, two or
// three levels; form = NCLS_GENERAL or NCLS_SHARED; nullptr elsewhere).  They take the tensor maps
// and launch arguments of find_march2d / find_march3d and LaunchArgs::cls.
LaunchFn find_march_ncde(int lat, int levels, int st, int form);
// Rows of the x-y tile a 3D march CTA stages per plane (the TMA box is 128+halo x rows+2 x 1).
int march3d_tile_rows(int pde);
// The 2D (D2Q9) and 3D (D3Q19) marching kernels in the lean He-Luo NSE form (lean = LEAN_STREAM
// or LEAN_GENERAL, see Coef::nA; FP32 / BF16 storage, two or three levels; FP64 for the two-level
// streaming form only; nullptr elsewhere).
// They take the same tensor maps and launch arguments as find_march2d / find_march3d, except that
// in 3D `rows` picks the CTA tile: march3d_tile_rows(PDE_NSE) rows at four CTAs per SM, or 16 rows
// at one CTA per SM (tensor-map boxes of rows + 2 rows either way; 2D ignores it).
LaunchFn find_march_lean(int lat, int levels, int st, int lean, int nx, int rows = 4);
// The D3Q19 He-Luo NSE step in the lean streaming form (two levels; FP32 with rows as for
// find_march_lean, FP64 with march3d_tile_rows(PDE_NSE) rows).
LaunchFn find_march3d_nse(int st, int rows);
// Tile rows a 3D lean solver of this grid runs with: 16 where the grid has enough 16-row tiles to
// fill the GPU with one CTA per SM, march3d_tile_rows(PDE_NSE) otherwise; force > 0 asks for the
// 16-row tiles and force < 0 for the narrow ones whatever the grid (for comparisons).
int march3d_lean_tile_rows(int nx, int ny, int nz, int force = 0);

// Encode a 2D / 3D tiled TMA descriptor over one field of a ghosted level buffer
// (box = boxw x 1 [x 1] elements).  Returns 0 on success.
// promote_l2 = false: no L2 promotion of the box's requests (only the box's own sectors are
// fetched), for kernels whose neighbouring CTAs do not read the surrounding bytes at about the
// same time.
int encode_field_map(CUtensorMap* m, void* field_base, int st, const Geom& g, int boxw, int boxh, int boxd,
                     bool promote_l2 = true);

// Utility kernels (k_util.cu).
// Dense buffers src[0 .. nf) of element type src_dtype (MMFD_DT_*) into fields field0 .. of a level
// (and of a second level of the same layout, if given), with their periodic ghost images; refs are
// the fields' storage references.  One launch.
cudaError_t launch_pack(const Geom& g, int st, const void* const* src, int nf, int src_dtype, void* level, void* level2,
                        int field0, const double* refs, cudaStream_t s);
// The reverse: fields field0 .. of a level into dense buffers.
cudaError_t launch_unpack(const Geom& g, int st, const void* level, int field0, int nf, const double* refs,
                          void* const* dst, int dst_dtype, cudaStream_t s);
// Rows [r_lo, r_hi) of all nf fields of a level to (pack) or from (unpack) nf dense buffers of
// element type dtype (MMFD_DT_*), one launch; refs are the fields' storage references.
cudaError_t launch_rows(const Geom& g, int st, bool pack, const void* const* bufs, int nf, int dtype, void* level,
                        const double* refs, long long r_lo, long long r_hi, cudaStream_t s);
// Copy the boundary ring (x = 0 / nx - 1, y = 0 / ny - 1, z = 0 / nz - 1 in 3D) of every field
// from one level buffer to another of the same layout and storage (Dirichlet boundaries).
cudaError_t launch_ring_copy(const Geom& g, const void* src_level, void* dst_level, cudaStream_t s);
// Deterministic FP64 reductions over the interior of one field: op 0 sum, 1 max|v|,
// 2 non-finite count; with ref != NULL: op 3 -> (sum |v - ref|, sum |ref|, max |v - ref|, max |ref|).
cudaError_t launch_reduce(const Geom& g, int st, const void* level, int field, double fref, int op,
                          const void* ref, int ref_dtype, double* d_partials, int nparts, double* d_out,
                          cudaStream_t s);
int reduce_parts_needed();

}  // namespace mmfd
