// k_march_ncde.cu -- 2D (D2Q9) and 3D (D3Q19) NCDE steps in class form (ncde_class.cuh), FP32 and FP64
// storage, two or three levels.
//
// 2D: the layout of k_march2d_nse with one step per launch: a warp streams the rows of one 128-column
// strip through its TMA ring (120 output columns, lanes 1 .. 30), the row sums march in y, and
// the x neighbours' sums come by shuffle.
// 3D: the tiles, ring and refill of k_march3d_nse; a warp owns R output rows and evaluates each of
// its R + 2 input rows once per plane, lanes 0 and 31 also the strip's halo columns.
//
// Bound by FP32 (FP64) issue.  Shared flux, three levels: 2D 4096^2 FP32 42.5 us a step (the pushed form 74.6),
// 1024^2 5.8 us (10.6), FP64 151 us (389); 3D 96^3 FP32 13.4 us (22.9), 256^3 118 us (227), FP64 96^3 409 us
// (979).
#define MMFD_PAIRED 1
#include "march3d_ring.cuh"
#include "ncde_class.cuh"

namespace mmfd {

namespace {

constexpr int kNcStride = 120;   // output columns per 2D strip
constexpr int kNcLead = 8;       // lane 0's first column lies kNcLead columns left of the strip's output

template <int ST, int LEVELS, bool SHARED, int NW, int NSTAGE>
__global__ void __launch_bounds__(NW * 32) k_march2d_ncde(const __grid_constant__ TmapSet maps, Geom g, void* outv,
                                                          const __grid_constant__ NcdePk<typename Storage<ST>::T, 2, LEVELS - 1, SHARED> cc,
                                                          int H, int nitems, int* err) {
    using S = typename Storage<ST>::S;
    using T = typename Storage<ST>::T;
    using P = Pk<T>;
    constexpr int NL = LEVELS - 1;
    constexpr int LN = 4;
    constexpr int ES = (int)sizeof(S);
    constexpr int ALIGN = 16 / ES;
    constexpr int COLS = 32 * LN;
    constexpr int BOXW = COLS + 2 * ALIGN;
    constexpr int RPS = 2;
    constexpr int ROWB = BOXW * ES;
    constexpr int SLOT = ((RPS * ROWB + 127) / 128) * 128;
    constexpr uint32_t kTx = (uint32_t)(NL * RPS * ROWB);
    constexpr size_t kRingBytes = (size_t)NSTAGE * NL * SLOT;

    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem) + warp * NSTAGE;
    unsigned char* ring = smem + 128 * ((NW * NSTAGE * 8 + 127) / 128) + warp * kRingBytes;
    auto slot = [&](int s, int l) -> unsigned char* { return ring + (size_t)(s * NL + l) * SLOT; };

    const int strips = (g.nx + kNcLead / 2 + kNcStride - 1) / kNcStride;
    const int wstride = gridDim.x * NW;
    const int wid = blockIdx.x * NW + warp;
    if (wid >= nitems) return;

    // producer (lane 0): the item's box column (padded coordinates) and first padded row (y0 - 1)
    int p_item = wid, p_row = 0, p_rows = 0, p_xcol = 0, p_y = 0;
    auto p_load_item = [&]() {
        if (p_item < nitems) {
            const int seg = p_item / strips;
            p_xcol = (p_item - seg * strips) * kNcStride - kNcLead;
            p_y = seg * H;
            p_rows = (min(H, g.ny - seg * H) + 2 + RPS - 1) / RPS * RPS;
        }
    };
    p_load_item();
    int ps = 0;
    long long issued = 0;
    auto issue_next = [&]() {
        if (p_item >= nitems) return;
        mbar_arrive_expect_tx(&full[ps], kTx);
#pragma unroll
        for (int l = 0; l < NL; ++l) tma_load_2d(slot(ps, l), &maps.m[l], &full[ps], p_xcol, p_y + p_row);
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
        for (int l = 0; l < NL; ++l) tma_prefetch_desc(&maps.m[l]);
    }
    chain_wait();
    if (lane == 0)
        for (int k = 0; k < NSTAGE; ++k) issue_next();
    __syncwarp();

    // sums of the output rows around input row r: row r after its C group (c), row r + 1 after its N group (n)
    P sc[2], sn[2];
    S* out = static_cast<S*>(outv);
    int cs = 0;
    uint32_t cphase = 0;
    long long consumed = 0;
    bool failed = false;
    EdgeStore<2, ST> es;

    auto load_row = [&](int s, int j, P (&phi)[2][NL]) {
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            T v4[4];
            lds4<ST, PDE_NCDE>(slot(s, l) + (size_t)j * ROWB + (size_t)(ALIGN + lane * LN) * ES, T(0), v4);
            phi[0][l] = P::make(v4[0], v4[1]);
            phi[1][l] = P::make(v4[2], v4[3]);
        }
    };
    // take input row r; `done`: the completed output row r - 1
    auto advance = [&](const P (&phi)[2][NL], P (&done)[2]) {
        NcdeParts<P, 2> o[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) ncde_eval<SHARED, 2, NL, P, T>(cc, phi[h], o[h]);
        P L[2], R[2], s[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            L[h] = ncde_diag<SHARED, 0, 1, true, 1>(o[h]);
            R[h] = ncde_diag<SHARED, 0, 1, false, 1>(o[h]);
        }
        shift_sum<T>(L, R, s);
#pragma unroll
        for (int h = 0; h < 2; ++h) done[h] = padd(sc[h], padd(s[h], ncde_axis<SHARED, 1, 1>(o[h])));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            L[h] = ncde_axis<SHARED, 0, 1>(o[h]);
            R[h] = ncde_axis<SHARED, 0, -1>(o[h]);
        }
        shift_sum<T>(L, R, s);
#pragma unroll
        for (int h = 0; h < 2; ++h) sc[h] = padd(padd(o[h].ctr, sn[h]), s[h]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            L[h] = ncde_diag<SHARED, 0, 1, false, -1>(o[h]);
            R[h] = ncde_diag<SHARED, 0, 1, true, -1>(o[h]);
        }
        shift_sum<T>(L, R, s);
#pragma unroll
        for (int h = 0; h < 2; ++h) sn[h] = padd(s[h], ncde_axis<SHARED, 1, -1>(o[h]));
    };

    for (int item = wid; item < nitems && !failed; item += wstride) {
        const int seg = item / strips;
        const int x0 = (item - seg * strips) * kNcStride - kNcLead;
        const int y0 = seg * H;
        const int hrows = min(H, g.ny - y0);
        const int nrows = (hrows + 2 + RPS - 1) / RPS * RPS;
        const int xb = x0 + lane * LN;
        es.init(g, xb, lane >= 1 && lane <= 30);
#pragma unroll
        for (int h = 0; h < 2; ++h) sc[h] = sn[h] = P::fill(T(0));
        for (int i = 0; i < nrows; i += RPS) {
            const bool ok = mbar_wait_bounded(&full[cs], cphase);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            P a[2][NL], b[2][NL];
            load_row(cs, 0, a);
            load_row(cs, 1, b);
            ++consumed;
            cs = cs + 1 == NSTAGE ? 0 : cs + 1;
            if (cs == 0) cphase ^= 1u;
            __syncwarp();
            if (lane == 0) {
                fence_proxy_async_smem();
                issue_next();
            }
            P done[2];
            auto store = [&](int yo) {
                es.template put<1>(out, g.fs, g, xb, yo, 0, [&](int, S (&sv)[4]) {
                    sv[0] = done[0].lo();
                    sv[1] = done[0].hi();
                    sv[2] = done[1].lo();
                    sv[3] = done[1].hi();
                });
            };
            // input row i (y0 - 1 + i) completes output row y0 + i - 2
            advance(a, done);
            if (i >= 2) store(y0 + i - 2);
            advance(b, done);
            if (i >= 1 && i - 1 < hrows) store(y0 + i - 1);
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

template <int ST, int LEVELS, bool SHARED>
cudaError_t launch2(const LaunchArgs& a) {
    using T = typename Storage<ST>::T;
    constexpr int NW = 4;
    constexpr int NSTAGE = LEVELS == 2 ? 6 : 4;
    constexpr int ES = (int)sizeof(typename Storage<ST>::S);
    constexpr int SLOT = ((2 * (128 + 2 * (16 / ES)) * ES + 127) / 128) * 128;
    constexpr size_t smem = 128 + 128 * ((NW * NSTAGE * 8 + 127) / 128) + (size_t)NW * NSTAGE * (LEVELS - 1) * SLOT;
    auto kern = k_march2d_ncde<ST, LEVELS, SHARED, NW, NSTAGE>;
    static std::atomic<unsigned long long> known[kMaxDevices];
    Fit fit;
    const cudaError_t e = fit_of(kern, NW * 32, smem, known, &fit);
    if (e != cudaSuccess) return e;
    const int resident = fit.ctas();
    const int strips = (a.g.nx + kNcLead / 2 + kNcStride - 1) / kNcStride;
    int H = a.H;
    if (H <= 0) H = march_height(strips, a.g.ny, (long long)resident * NW, 2, 2, 256);
    const int nitems = strips * ((a.g.ny + H - 1) / H);
    const int blocks_needed = (nitems + NW - 1) / NW;
    const int grid = blocks_needed < resident ? blocks_needed : resident;
    return launch_chained(kern, grid, NW * 32, smem, a.stream, a.chained,
                          *a.maps, a.g, a.out, ncde_pk<T, 2, LEVELS - 1, SHARED>(*static_cast<const NcdeClass<T>*>(a.cls)),
                          H, nitems, a.err);
}

// ------------------------------------------------------------------ 3D

template <int ST, int LEVELS, bool SHARED, int TY, int R, int NSTAGE, int MINB>
__global__ void __launch_bounds__(TY / R * 32, MINB) k_march3d_ncde(const __grid_constant__ TmapSet maps, Geom g,
                                                                  void* outv,
                                                                  const __grid_constant__ NcdePk<typename Storage<ST>::T, 3, LEVELS - 1, SHARED> cc,
                                                                  int H, int nitems, int* err) {
    using S = typename Storage<ST>::S;
    using T = typename Storage<ST>::T;
    using P = Pk<T>;
    constexpr int NL = LEVELS - 1, LN = 4;
    constexpr int NWARP = TY / R;
    constexpr int ES = (int)sizeof(S);
    constexpr int ALIGN = 16 / ES;
    constexpr int COLS = 32 * LN;
    constexpr int BOXW = COLS + 2 * ALIGN;
    constexpr int BOXH = TY + 2;
    constexpr int ROWB = BOXW * ES;
    constexpr int SLOT = ((ROWB * BOXH + 127) / 128) * 128;

    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PlaneRing<TY, NWARP, NL, NSTAGE, (uint32_t)(BOXW * BOXH * ES), SLOT> ring(smem_raw);
    const PlaneWalk<TY> walk(g, H, nitems);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    ring.start(maps, walk);

    PlaneCursor rd;   // the plane being read
    walk.start(rd);
    // sums of the warp's output rows in plane z after its C group (c) and in plane z + 1 after its N group (n)
    P sc[R][2], sn[R][2];
    EdgeStore<3, ST> es;
    S* out = static_cast<S*>(outv);
    const bool mirrored = lane == 0;
    const int ecol = lane == 0 ? ALIGN - 1 : lane == 31 ? ALIGN + COLS : ALIGN + lane * LN;
    int cs = 0;
    uint32_t cpar = 0;
    bool failed = false;
    while (rd.np != 0) {
        const int xb = rd.x0 + lane * LN;
        const int y0 = rd.y0 + warp * R;
        const int i = rd.i, zo = rd.z0 + i - 2;
        if (i == 0) {
            es.init(g, xb, true);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) sc[r][h] = sn[r][h] = P::fill(T(0));
        }
        const bool ok = mbar_wait_bounded(&ring.full[cs], cpar);
        if (__any_sync(0xffffffffu, !ok)) {
            failed = true;
            break;
        }
        P res[R][2];
        // what the row before sends up (to y + 1), and the pending sums of the row before: its P and N
        // sums so far, its C group's left- and right-moving values and the rest of its C sum
        P uP[2], uL[2], uR[2], uE[2], uN[2], qP[2], qL[2], qR[2], qC[2], qN[2];
        T uh = T(0), qh = T(0);
        static_for<0, R + 2>([&](auto jc) {
            constexpr int J = decltype(jc)::value - 1;
            constexpr bool OWN = J >= 0 && J < R, UP = J + 1 < R, DN = J - 1 >= 0;
            NcdeParts<P, 3> o[2];
            NcdeParts<One<T>, 3> e;
            {
                P phi[2][NL];
                One<T> ep[NL];
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    const unsigned char* rowp = ring.slot(cs, l) + (size_t)(warp * R + J + 1) * ROWB;
                    T v4[4];
                    lds4<ST, PDE_NCDE>(rowp + (size_t)(ALIGN + lane * LN) * ES, T(0), v4);
                    phi[0][l] = P::make(v4[0], v4[1]);
                    phi[1][l] = P::make(v4[2], v4[3]);
                    ep[l].v = Storage<ST>::raw(reinterpret_cast<const S*>(rowp) + ecol);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) ncde_eval<SHARED, 3, NL, P, T>(cc, phi[h], o[h]);
                ncde_eval<SHARED, 3, NL, One<T>, T>(cc, ep, e);
            }
            if constexpr (DN) {
                // row J completes output row J - 1's inputs with what it sends down (to y - 1)
                P s[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    qL[h] = padd(qL[h], ncde_diag<SHARED, 0, 1, true, 1>(o[h]));
                    qR[h] = padd(qR[h], ncde_diag<SHARED, 0, 1, false, 1>(o[h]));
                }
                shift_sum_edge<T>(qL, qR, radd(qh, ncde_edge_diag<SHARED, 1, true>(e, mirrored)), lane, s);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    res[J - 1][h] = padd(sc[J - 1][h], padd(qP[h], ncde_diag<SHARED, 1, 2, true, 1>(o[h])));
                    sc[J - 1][h] = padd(padd(qC[h], ncde_axis<SHARED, 1, 1>(o[h])), padd(s[h], sn[J - 1][h]));
                    sn[J - 1][h] = padd(qN[h], ncde_diag<SHARED, 1, 2, false, -1>(o[h]));
                }
            }
            if constexpr (OWN) {
                P L[2], Rr[2], s[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    L[h] = ncde_diag<SHARED, 0, 2, true, 1>(o[h]);
                    Rr[h] = ncde_diag<SHARED, 0, 2, false, 1>(o[h]);
                }
                shift_sum_edge<T>(L, Rr, ncde_edge_diag<SHARED, 2, true>(e, mirrored), lane, s);
#pragma unroll
                for (int h = 0; h < 2; ++h) qP[h] = padd(padd(s[h], ncde_axis<SHARED, 2, 1>(o[h])), uP[h]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    L[h] = ncde_diag<SHARED, 0, 2, false, -1>(o[h]);
                    Rr[h] = ncde_diag<SHARED, 0, 2, true, -1>(o[h]);
                }
                shift_sum_edge<T>(L, Rr, ncde_edge_diag<SHARED, 2, false>(e, mirrored), lane, s);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    qN[h] = padd(padd(s[h], ncde_axis<SHARED, 2, -1>(o[h])), uN[h]);
                    qL[h] = padd(ncde_axis<SHARED, 0, 1>(o[h]), uL[h]);
                    qR[h] = padd(ncde_axis<SHARED, 0, -1>(o[h]), uR[h]);
                    qC[h] = padd(o[h].ctr, uE[h]);
                }
                qh = radd(ncde_edge_axis<SHARED>(e, mirrored), uh);
            }
            if constexpr (UP) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uE[h] = ncde_axis<SHARED, 1, -1>(o[h]);
                    uR[h] = ncde_diag<SHARED, 0, 1, true, -1>(o[h]);
                    uL[h] = ncde_diag<SHARED, 0, 1, false, -1>(o[h]);
                    uN[h] = ncde_diag<SHARED, 1, 2, true, -1>(o[h]);
                    uP[h] = ncde_diag<SHARED, 1, 2, false, 1>(o[h]);
                }
                uh = ncde_edge_diag<SHARED, 1, false>(e, mirrored);
            }
        });
        ring.release(maps, walk, cs, lane);
        cs = cs + 1 == NSTAGE ? 0 : cs + 1;
        if (cs == 0) cpar ^= 1u;
        walk.advance(rd);
        if (i >= 2) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (y0 + r >= g.ny) continue;
                es.template put<1>(out, g.fs, g, xb, y0 + r, zo, [&](int, S (&sv)[4]) {
                    sv[0] = res[r][0].lo();
                    sv[1] = res[r][0].hi();
                    sv[2] = res[r][1].lo();
                    sv[3] = res[r][1].hi();
                });
            }
        }
    }
    if (failed) ring.give_up(err, cs, cpar, lane);
}

template <int ST, int LEVELS, bool SHARED, int TY, int R, int MINB>
cudaError_t launch3(const LaunchArgs& a) {
    using T = typename Storage<ST>::T;
    constexpr int NSTAGE = march3d_stages<LAT_D3Q19, PDE_NCDE, LEVELS, ST, TY, 57344>();
    constexpr size_t smem = ring_smem<ST, LEVELS, 1, TY, NSTAGE>();
    constexpr int THREADS = TY / R * 32;
    auto kern = k_march3d_ncde<ST, LEVELS, SHARED, TY, R, NSTAGE, MINB>;
    static std::atomic<unsigned long long> known[kMaxDevices];
    Fit fit;
    const cudaError_t e = fit_of(kern, THREADS, smem, known, &fit);
    if (e != cudaSuccess) return e;
    const int resident = fit.ctas();
    int H = 0, nitems = 0, grid = 0;
    march3d_split(a.g, TY, a.H, resident, false, &H, &nitems, &grid);
    return launch_chained(kern, grid, THREADS, smem, a.stream, a.chained,
                          *a.maps, a.g, a.out, ncde_pk<T, 3, LEVELS - 1, SHARED>(*static_cast<const NcdeClass<T>*>(a.cls)),
                          H, nitems, a.err);
}

template <int ST, int LEVELS>
LaunchFn pick(int dim, bool shared) {
    constexpr int TY = tile_rows(PDE_NCDE);
    if (dim == 2) return shared ? launch2<ST, LEVELS, true> : launch2<ST, LEVELS, false>;
    return shared ? launch3<ST, LEVELS, true, TY, 1, 4> : launch3<ST, LEVELS, false, TY, 1, 4>;
}

}  // namespace

LaunchFn find_march_ncde(int lat, int levels, int st, int form) {
    const int dim = lat == LAT_D2Q9 ? 2 : lat == LAT_D3Q19 ? 3 : 0;
    if (dim == 0 || form == NCLS_NONE || st == ST_BF16) return nullptr;
    const bool shared = form == NCLS_SHARED;
    if (levels == 2) return st == ST_F32 ? pick<ST_F32, 2>(dim, shared) : pick<ST_F64, 2>(dim, shared);
    if (levels == 3) return st == ST_F32 ? pick<ST_F32, 3>(dim, shared) : pick<ST_F64, 3>(dim, shared);
    return nullptr;
}

}  // namespace mmfd
