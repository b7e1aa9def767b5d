// k_march2d_nse.cu -- 2D He-Luo NSE steps, D2Q9, two levels, the lean streaming form
// (Coef::nA with streaming momentum) evaluated in class form on node pairs (nse_class.cuh).  One
// launch advances TT = 1, 2 or 3 time levels and reads / writes the stored level (rho, ux, uy) once.
//
// The layout of k_march2d_tb (the scalar blocked kernel) with three fields:
// - A warp owns items of one 128-column strip x H output rows. It streams the input rows
//   y0-TT .. y0+H+TT-1 of the three fields, two rows per stage, through its private TMA ring;
//   rows wrap periodically in y in the producer.
// - It keeps TT sets of row sums (Row2, 20 values per lane and level). An input row advances level
//   1's sums and yields a completed level-1 row, which advances level 2's; and so on -- a wavefront
//   of TT steps one row apart.  The one-step kernel is the same code with TT = 1, so the two round
//   alike.
// - Sums that cross into a neighbouring lane's columns come from that lane by shuffle at every
//   level, so no lane evaluates a halo node.  Strips overlap: lanes cover columns X0 .. X0+127
//   (X0 = 120 s - 8), lanes 1 .. 30 store.  At level t the first (last) t columns of lane 0 (31)
//   are wrong, which lane 1 (30) does not read for t < 4.
// - Columns within TT of the x edges are read from the ghost columns, which every writer keeps
//   current to the ghost depth.
//
// Bound by FP32 issue when blocked (46 instructions per node and step, the FMA pipe 64% busy), by DRAM with
// one step per launch.  4096^2 FP32: three steps per launch 34.1 us per step (the pushed form 39.1), one
// 75 us (77); FP64, bound by the FP64 rate, 1000 x 800 105 us (193).
// FP32 and FP64 storage; BF16 levels keep the pushed form and its rounding (k_march2d_tb_nse,
// k_march2d).
#define MMFD_PAIRED 1
#include "k_march2d.cuh"
#include "nse_class.cuh"

namespace mmfd {

namespace {

constexpr int kTbnStride = 120;   // output columns per strip
constexpr int kTbnLead = 8;       // lane 0's first column lies kTbnLead columns left of the strip's output

template <int ST, int TT, int NW, int NSTAGE>
__global__ void __launch_bounds__(NW * 32) k_march2d_nse(const __grid_constant__ TmapSet maps, Geom g,
                                                            void* outv, ClassCoef<typename Storage<ST>::T> cc, int H,
                                                            int nitems, int* err) {
    using Tr = Storage<ST>;
    using S = typename Tr::S;
    using T = typename Tr::T;
    constexpr int PDE = PDE_NSE;
    constexpr int NF = 3;
    constexpr int LN = 4;
    constexpr int ES = (int)sizeof(S);
    constexpr int ALIGN = 16 / ES;
    constexpr int COLS = 32 * LN;
    constexpr int BOXW = COLS + 2 * ALIGN;
    constexpr int RPS = 2;                                  // input rows per stage (box height)
    constexpr int ROWB = BOXW * ES;
    constexpr int SLOT = ((RPS * ROWB + 127) / 128) * 128;  // one field of one stage
    constexpr uint32_t kTx = (uint32_t)(NF * RPS * ROWB);
    constexpr size_t kRingBytes = (size_t)NSTAGE * NF * SLOT;
    static_assert(TT >= 1 && TT <= 3, "three fields: at most three levels in registers");
    static_assert(TT < LN, "the wrong columns of the edge lanes must not reach lanes 1 and 30");
    static_assert(TT <= ALIGN, "ghost columns of 16 bytes hold at most 16 / sizeof(S) levels");

    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem) + warp * NSTAGE;
    unsigned char* ring = smem + 128 * ((NW * NSTAGE * 8 + 127) / 128) + warp * kRingBytes;
    auto slot = [&](int s, int f) -> unsigned char* { return ring + (size_t)(s * NF + f) * SLOT; };

    const int strips = (g.nx + kTbnLead / 2 + kTbnStride - 1) / kTbnStride;
    const int wstride = gridDim.x * NW;
    const int wid = blockIdx.x * NW + warp;
    if (wid >= nitems) return;

    // producer (lane 0): the item's box column (padded coordinates) and first input row
    int p_item = wid, p_row = 0, p_rows = 0, p_xcol = 0, p_y = 0;
    auto p_load_item = [&]() {
        if (p_item < nitems) {
            const int seg = p_item / strips;
            p_xcol = (p_item - seg * strips) * kTbnStride - kTbnLead;
            p_y = seg * H - TT;
            p_rows = (min(H, g.ny - seg * H) + 2 * TT + RPS - 1) / RPS * RPS;
        }
    };
    p_load_item();
    int ps = 0;
    long long issued = 0;
    auto issue_next = [&]() {
        if (p_item >= nitems) return;
        const int y = p_y + p_row;
        const int yw = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);   // periodic in y
        mbar_arrive_expect_tx(&full[ps], kTx);
#pragma unroll
        for (int f = 0; f < NF; ++f) tma_load_2d(slot(ps, f), &maps.m[f], &full[ps], p_xcol, yw + 1);
        ++issued;
        ps = ps + 1 == NSTAGE ? 0 : ps + 1;
        p_row += RPS;
        if (p_row == p_rows) {
            p_item += wstride;
            p_row = 0;
            p_load_item();
        }
    };

    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < NSTAGE; ++s) mbar_init(&full[s], 1);
        fence_mbar_init();
#pragma unroll
        for (int f = 0; f < NF; ++f) tma_prefetch_desc(&maps.m[f]);
    }
    chain_wait();
    if (lane == 0)
        for (int k = 0; k < NSTAGE; ++k) issue_next();
    __syncwarp();

    Row2<T> acc[TT];   // level t's sums around its current input row
    S* out = static_cast<S*>(outv);
    int cs = 0;
    uint32_t cphase = 0;
    long long consumed = 0;
    bool failed = false;
    const bool store_lane = lane >= 1 && lane <= 30;

    // input row i of the item at (xb, y0): push it through the TT levels and store the completed
    // level-TT row y0 - 2 TT + i if it is one of the item's output rows
    EdgeStore<2, ST> es;
    auto cascade = [&](RowPk<T, NF>& row, int i, int xb, int y0, int hrows) {
#pragma unroll
        for (int t = 0; t < TT; ++t) class_row2d<T>(cc, row, acc[t]);
        const int yo = y0 - 2 * TT + i;
        if (i >= 2 * TT && i < hrows + 2 * TT) {   // warp-uniform; lanes 0 and 31 hold no output
            es.template put<NF>(out, g.fs, g, xb, yo, 0, [&](int f, S (&sv)[4]) {
                sv[0] = row.f[f][0].lo();
                sv[1] = row.f[f][0].hi();
                sv[2] = row.f[f][1].lo();
                sv[3] = row.f[f][1].hi();
            });
        }
    };

    auto load_row = [&](int s, int j, RowPk<T, NF>& row) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            T v4[4];
            lds4<ST, PDE>(slot(s, f) + (size_t)j * ROWB + (size_t)(ALIGN + lane * LN) * ES, T(0), v4);
            row.f[f][0] = Pk<T>::make(v4[0], v4[1]);
            row.f[f][1] = Pk<T>::make(v4[2], v4[3]);
        }
    };

    for (int item = wid; item < nitems && !failed; item += wstride) {
        const int seg = item / strips;
        const int x0 = (item - seg * strips) * kTbnStride - kTbnLead;
        const int y0 = seg * H;
        const int hrows = min(H, g.ny - y0);
        const int nrows = (hrows + 2 * TT + RPS - 1) / RPS * RPS;
        const int xb = x0 + lane * LN;
        es.init(g, xb, store_lane);
#pragma unroll
        for (int t = 0; t < TT; ++t) row2_clear(acc[t]);
        for (int i = 0; i < nrows; i += RPS) {
            const bool ok = mbar_wait_bounded(&full[cs], cphase);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            RowPk<T, NF> rawA, rawB;
            load_row(cs, 0, rawA);
            load_row(cs, 1, rawB);
            ++consumed;
            cs = cs + 1 == NSTAGE ? 0 : cs + 1;
            if (cs == 0) cphase ^= 1u;
            __syncwarp();
            if (lane == 0) {
                fence_proxy_async_smem();
                issue_next();
            }
            cascade(rawA, i, xb, y0, hrows);
            cascade(rawB, i + 1, xb, y0, hrows);
        }
    }
    if (failed && lane == 0) {
        atomicExch(err, KERR_TMA_TIMEOUT);
        for (long long k = consumed; k < issued; ++k) {
            const int s = (int)(k % NSTAGE);
            mbar_wait_bounded(&full[s], (uint32_t)((k / NSTAGE) & 1));
        }
    }
}

template <int ST, int NW, int NSTAGE>
constexpr size_t tbn_smem() {
    constexpr int ES = (int)sizeof(typename Storage<ST>::S);
    constexpr int SLOT = ((2 * (128 + 2 * (16 / ES)) * ES + 127) / 128) * 128;
    return 128 + 128 * ((NW * NSTAGE * 8 + 127) / 128) + (size_t)NW * NSTAGE * 3 * SLOT;
}

template <int ST, int TT>
cudaError_t launch_nse(const LaunchArgs& a) {
    using T = typename Storage<ST>::T;
    constexpr int NW = 4;
    constexpr int NSTAGE = 3;
    constexpr size_t smem = tbn_smem<ST, NW, NSTAGE>();
    auto kern = k_march2d_nse<ST, TT, NW, NSTAGE>;
    static std::atomic<unsigned long long> known[kMaxDevices];
    Fit fit;
    const cudaError_t e = fit_of(kern, NW * 32, smem, known, &fit);
    if (e != cudaSuccess) return e;
    const int resident = fit.ctas();
    const int strips = (a.g.nx + kTbnLead / 2 + kTbnStride - 1) / kTbnStride;
    int H = a.H;
    if (H <= 0) H = march_height(strips, a.g.ny, (long long)resident * NW, 2 * TT, TT == 1 ? 2 : 8, 512);
    const int nitems = strips * ((a.g.ny + H - 1) / H);
    const int blocks_needed = (nitems + NW - 1) / NW;
    const int grid = blocks_needed < resident ? blocks_needed : resident;
    return launch_chained(kern, grid, NW * 32, smem, a.stream, a.chained, *a.maps, a.g, a.out, class_coef<LAT_D2Q9, T>(*static_cast<const Coef<T>*>(a.coef), a.umom, 0), H,
                          nitems, a.err);
}

}  // namespace

LaunchFn find_march2d_nse(int st, int depth) {
    if (st == ST_F64) return depth == 1 ? launch_nse<ST_F64, 1> : nullptr;
    if (st == ST_F32)
        return depth == 1 ? launch_nse<ST_F32, 1> : depth == 2 ? launch_nse<ST_F32, 2> : depth == 3 ? launch_nse<ST_F32, 3> : nullptr;
    return nullptr;
}

}  // namespace mmfd
