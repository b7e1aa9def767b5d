// k_march3d_nse.cu -- 3D He-Luo NSE step, D3Q19, two levels, the lean streaming form (Coef::nA with
// streaming momentum) evaluated in class form on node pairs (nse_class.cuh).
//
// The tiles and the ring are k_march3d's.  Here a warp reads the three input rows its output row needs
// once per plane: its own row's nodes are evaluated towards their own row's outputs, those of the two
// neighbouring rows only towards the warp's row, and the x neighbours' sums come from the
// neighbouring lanes.  Lanes 0 and 31 evaluate the strip's halo columns, all lanes following.
//
// FP32 takes it for widths that are not a multiple of four and below 128 columns (find_march_lean): 250^3
// 161 us a step (the pushed form 301), 510 x 512^2 1110 (2062), 96^3 16.4 (k_direct 28.4).  136
// instructions per node; at 512^3 4.5 TB/s, waits on the planes and FP32 issue in equal parts.  FP64
// 144^3, bound by the FP64 rate, 1333 us (5300).
#define MMFD_PAIRED 1
#include "march3d_ring.cuh"
#include "nse_class.cuh"

namespace mmfd {

namespace {

template <int ST, int TY, int NSTAGE, int MINB>
__global__ void __launch_bounds__(TY * 32, MINB) k_march3d_nse(const __grid_constant__ TmapSet maps, Geom g,
                                                             void* outv, ClassNorm<typename Storage<ST>::T> cc,
                                                             int H, int nitems, int* err) {
    using Tr = Storage<ST>;
    using S = typename Tr::S;
    using T = typename Tr::T;
    constexpr int NF = 4, LN = 4;
    constexpr int ES = (int)sizeof(S);
    constexpr int ALIGN = 16 / ES;
    constexpr int COLS = 32 * LN;
    constexpr int BOXW = COLS + 2 * ALIGN;
    constexpr int BOXH = TY + 2;
    constexpr int ROWB = BOXW * ES;
    constexpr int SLOT = ((ROWB * BOXH + 127) / 128) * 128;

    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PlaneRing<TY, TY, NF, NSTAGE, (uint32_t)(BOXW * BOXH * ES), SLOT> ring(smem_raw);
    const PlaneWalk<TY> walk(g, H, nitems);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    ring.start(maps, walk);

    PlaneCursor rd;   // the plane being read
    walk.start(rd);
    Row3<T> acc;
    EdgeStore<3, ST> es;
    S* out = static_cast<S*>(outv);
    // the edge column: right of the strip's columns in lane 31, left of them in lane 0 (the other
    // lanes' values are not used), and the sign of its u_x
    const int ecol = lane == 0 ? ALIGN - 1 : lane == 31 ? ALIGN + COLS : ALIGN + lane * LN;
    const T esign = lane == 0 ? T(-1) : T(1);
    int cs = 0;
    uint32_t cpar = 0;
    bool failed = false;
    while (rd.np != 0) {
        const int xb = rd.x0 + lane * LN;
        const int y = rd.y0 + warp;
        const int i = rd.i, zo = rd.z0 + i - 2;
        if (i == 0) {
            es.init(g, xb, true);
            row3_clear(acc);
        }
        const bool ok = mbar_wait_bounded(&ring.full[cs], cpar);
        if (__any_sync(0xffffffffu, !ok)) {
            failed = true;
            break;
        }
        auto load_row = [&](int j, RowPk<T, NF>& row, T (&e)[4]) {
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const unsigned char* rowp = ring.slot(cs, f) + (size_t)(warp + j) * ROWB;
                T v4[4];
                lds4<ST, PDE_NSE>(rowp + (size_t)(ALIGN + lane * LN) * ES, T(0), v4);
                row.f[f][0] = Pk<T>::make(v4[0], v4[1]);
                row.f[f][1] = Pk<T>::make(v4[2], v4[3]);
                e[f] = Tr::raw(reinterpret_cast<const S*>(rowp) + ecol);
            }
            e[1] = rmul(e[1], esign);
        };
        Sides3<T> sd;
        {
            RowPk<T, NF> up, dn;
            T ue[4], de[4];
            load_row(2, up, ue);
            load_row(0, dn, de);
            class_sides3d<T>(cc, up, dn, ue, de, sd);
        }
        RowPk<T, NF> row;
        T e[4];
        load_row(1, row, e);
        ring.release(maps, walk, cs, lane);
        class_row3d<T>(cc, row, e, sd, lane, acc);
        cs = cs + 1 == NSTAGE ? 0 : cs + 1;
        if (cs == 0) cpar ^= 1u;
        walk.advance(rd);
        // plane zo of the row is complete
        if (i >= 2 && y < g.ny) {
            es.template put<NF>(out, g.fs, g, xb, y, zo, [&](int f, S (&sv)[4]) {
                sv[0] = row.f[f][0].lo();
                sv[1] = row.f[f][0].hi();
                sv[2] = row.f[f][1].lo();
                sv[3] = row.f[f][1].hi();
            });
        }
    }
    if (failed) ring.give_up(err, cs, cpar, lane);
}

template <int ST, int TY, int NSTAGE, int MINB>
cudaError_t launch(const LaunchArgs& a) {
    using T = typename Storage<ST>::T;
    constexpr size_t smem = ring_smem<ST, 2, 4, TY, NSTAGE>();
    constexpr int THREADS = TY * 32;
    auto kern = k_march3d_nse<ST, TY, NSTAGE, MINB>;
    static std::atomic<unsigned long long> known[kMaxDevices];
    Fit fit;
    const cudaError_t e = fit_of(kern, THREADS, smem, known, &fit);
    if (e != cudaSuccess) return e;
    const int resident = fit.ctas();
    int H = 0, nitems = 0, grid = 0;
    march3d_split(a.g, TY, a.H, resident, false, &H, &nitems, &grid);
    return launch_chained(kern, grid, THREADS, smem, a.stream, a.chained, *a.maps, a.g, a.out,
                          class_norm<T>(*static_cast<const Coef<T>*>(a.coef), a.umom, 0), H, nitems, a.err);
}

template <int ST, int TY, size_t BUDGET>
constexpr int stages() {
    return march3d_stages<LAT_D3Q19, PDE_NSE, 2, ST, TY, BUDGET>();
}

}  // namespace

LaunchFn find_march3d_nse(int st, int rows) {
    constexpr int W = kLeanWideRows, N = 4;
    if (st == ST_F64) return rows == N ? launch<ST_F64, N, stages<ST_F64, N, 98304>(), 2> : nullptr;
    if (st != ST_F32) return nullptr;
    if (rows == W) return launch<ST_F32, W, stages<ST_F32, W, kLeanWideRing>(), 1>;
    if (rows == N) return launch<ST_F32, N, stages<ST_F32, N, 49152>(), 4>;
    return nullptr;
}

}  // namespace mmfd
