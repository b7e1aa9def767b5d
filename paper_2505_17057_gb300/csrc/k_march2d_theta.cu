// k_march2d_theta.cu -- the 2D theta-scheme step (Eq. (GCN)) with fused Jacobi sweeps, FP32 and FP64 levels.
//
// A step solves (I - (1 - theta) L) x = r, r = (I + theta L) phi^n, by Jacobi sweeps
// x <- r / d + J x from x = phi^n (J: the sweep's stencil, no centre weight).  Two kernels:
//   k_theta_first  one pass over phi^n writes r and the first sweep's result: that is
//                  r / d + J phi^n, one more linear stencil of phi^n.
//   k_theta_sweeps TT further sweeps per launch, a wavefront of TT levels one row apart in registers as in
//                  k_march2d_tb.  The TT rows of r in use sit in a register window indexed by the row
//                  modulo four (four rows per pass over the loop, so no value moves), each fetched a row
//                  ahead of its use.  Two forms of a sweep:
//     - an output row's partial sum starts from its r / d, rounded once: no addition in the sweep, but every
//       term is then rounded at the full size of the sum;
//     - the last sweeps of a step (the launches that hold one of its last four) sum J x first and add r (1 / d)
//       at the end, as one fused operation: the rounding of the last sweeps is the step's error, that of
//       earlier ones shrinks with every sweep after them.  With the first form throughout, a step's error
//       against 64 bits was 1.1 to 2.2 times that of sweeps run one by one; with this rule the two agree.
// 4096^2 FP32, 17 sweeps, four per launch: 296 us a step (317 with the second form throughout); separate
// right-hand side pass, then sweeps adding the right-hand side at the store, 369 us.  Bound by FP32 issue in the sweeps, by DRAM in the first pass.
// A row's sums of rows r (c) and r + 1 (n) are chains of fused multiply-adds on the sum of the row
// before, with no accumulator copied from one role to the next.
#include "k_march2d.cuh"

namespace mmfd {

namespace {

constexpr int kThStride = 120;   // output columns per strip of the sweeps
constexpr int kThLead = 8;       // lane 0's first column lies kThLead columns left of the strip's output

// One input row (raw: the lane's four nodes and the two neighbouring ones) of the stencil (W0, Wp, Wm):
// completes the output row behind (out, from c), advances the input row's own sum (c, from n) and
// starts the row ahead's (n, from `start`).
template <int LAT, typename T>
__device__ __forceinline__ void stencil_row(const T& W0, const T (&Wp)[kMaxPair], const T (&Wm)[kMaxPair], const T (&raw)[6],
                                            const T (&start)[4], T (&c)[4], T (&n)[4], T (&out)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const T w = raw[k], m = raw[k + 1], e = raw[k + 2];
        T o = c[k], cc = n[k], nn = start[k];
        if constexpr (LAT == LAT_D2Q9) {
            // pairs: 0 x, 1 y, 2 (1, 1), 3 (-1, 1)
            o = rfma(Wp[2], e, rfma(Wp[1], m, rfma(Wp[3], w, o)));
            nn = rfma(Wm[3], e, rfma(Wm[1], m, rfma(Wm[2], w, nn)));
        } else {
            o = rfma(Wp[1], m, o);
            nn = rfma(Wm[1], m, nn);
        }
        cc = rfma(Wp[0], e, rfma(W0, m, rfma(Wm[0], w, cc)));
        out[k] = o;
        c[k] = cc;
        n[k] = nn;
    }
}

template <typename T>
struct Stencil {
    T W0, Wp[kMaxPair], Wm[kMaxPair];
};

// The per-warp row stream of both kernels: items of one strip x H rows, two rows per stage (as in
// k_march2d_tb); rows wrap periodically in y.
template <int ST>
struct RowBox {
    static constexpr int ES = (int)sizeof(typename Storage<ST>::S);
    static constexpr int ALIGN = 16 / ES;
    static constexpr int BOXW = 128 + 2 * ALIGN;
    static constexpr int ROWB = BOXW * ES;
    static constexpr int SLOT = ((2 * ROWB + 127) / 128) * 128;
    static constexpr int NSTAGE = 8192 / SLOT < 4 ? 4 : 8192 / SLOT;
    static constexpr size_t smem(int nw) { return 128 + 128 * ((nw * NSTAGE * 8 + 127) / 128) + (size_t)nw * NSTAGE * SLOT; }
};

// FIRST: k_theta_first (TT = 1; rhs is written, A its stencil, and B gives the first sweep's result);
// else the sweeps (rhs is read, B is J, jw is 1 / d; END: rhs is added at the end of a row's sum).
template <int LAT, int ST, int TT, bool FIRST, bool END, int NW>
__global__ void __launch_bounds__(NW * 32, ST == ST_F32 ? 4 : 1)
    k_theta(const __grid_constant__ TmapSet maps, Geom g, typename Storage<ST>::S* out,
            typename Storage<ST>::S* rhs, const __grid_constant__ Stencil<typename Storage<ST>::T> A,
            const __grid_constant__ Stencil<typename Storage<ST>::T> B, typename Storage<ST>::T jw, int H, int nitems, int* err) {
    using S = typename Storage<ST>::S;
    using T = typename Storage<ST>::T;
    using X = RowBox<ST>;
    constexpr int LN = 4;
    constexpr int NSTAGE = X::NSTAGE;
    constexpr int STRIDE = FIRST ? 128 : kThStride, LEAD = FIRST ? 0 : kThLead;
    static_assert(!FIRST || TT == 1, "the first sweep comes alone");
    static_assert(TT <= 4 && TT <= X::ALIGN, "the rhs window and the ghost columns hold at most that many levels");

    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem) + warp * NSTAGE;
    unsigned char* ring = smem + 128 * ((NW * NSTAGE * 8 + 127) / 128) + (size_t)warp * NSTAGE * X::SLOT;

    const int strips = (g.nx + LEAD / 2 + STRIDE - 1) / STRIDE;
    const int wstride = gridDim.x * NW;
    const int wid = blockIdx.x * NW + warp;
    if (wid >= nitems) return;

    // rows streamed per item: whole passes of four
    auto item_rows = [&](int y0) { return (min(H, g.ny - y0) + 2 * TT + 3) / 4 * 4; };
    int p_item = wid, p_row = 0, p_rows = 0, p_xcol = 0, p_y = 0;
    auto p_load_item = [&]() {
        if (p_item < nitems) {
            const int seg = p_item / strips;
            p_xcol = (p_item - seg * strips) * STRIDE - LEAD;
            p_y = seg * H - TT;
            p_rows = item_rows(seg * H);
        }
    };
    p_load_item();
    int ps = 0;
    long long issued = 0;
    auto issue_next = [&]() {
        if (p_item >= nitems) return;
        int y = p_y + p_row;
        y = y < 0 ? y + g.ny : y % g.ny;   // periodic in y
        mbar_arrive_expect_tx(&full[ps], 2 * X::ROWB);
        tma_load_2d(ring + (size_t)ps * X::SLOT, &maps.m[0], &full[ps], p_xcol, y + 1);
        ++issued;
        ps = ps + 1 == NSTAGE ? 0 : ps + 1;
        p_row += 2;
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
        tma_prefetch_desc(&maps.m[0]);
    }
    chain_wait();
    if (lane == 0)
        for (int k = 0; k < NSTAGE; ++k) issue_next();
    __syncwarp();

    T c[TT][LN], n[TT][LN];
    [[maybe_unused]] T ca[LN], na[LN];           // FIRST: the rhs's own sums
    [[maybe_unused]] T win[4][LN], next[LN];     // rhs rows by row modulo four, and the row after them
    EdgeStore<2, ST> es;
    int cs = 0;
    uint32_t cphase = 0;
    long long consumed = 0;
    bool failed = false;

    // the lane's four values of rhs row y, in bounds whatever the lane's columns: a lane outside the
    // row reads a neighbouring padded row (rows y = -1 and ny exist) into columns no output needs
    int ry = 0;   // the row to fetch next
    [[maybe_unused]] auto fetch = [&](int xb, T (&v)[LN]) {
        const S* p = rhs + g.at(0, ry, 0) + xb;
        if constexpr (sizeof(S) == 4) {
            const float4 q = *reinterpret_cast<const float4*>(p);
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        } else {
            const double2 q0 = *reinterpret_cast<const double2*>(p), q1 = *reinterpret_cast<const double2*>(p + 2);
            v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
        }
        ry = ry + 1 == g.ny ? 0 : ry + 1;
    };

    for (int item = wid; item < nitems && !failed; item += wstride) {
        const int seg = item / strips;
        const int xb = (item - seg * strips) * STRIDE - LEAD + lane * LN;
        const int y0 = seg * H;
        const int hrows = min(H, g.ny - y0);
        const int nrows = item_rows(y0);
        es.init(g, xb, FIRST || (lane >= 1 && lane <= 30));
#pragma unroll
        for (int t = 0; t < TT; ++t)
#pragma unroll
            for (int k = 0; k < LN; ++k) c[t][k] = n[t][k] = T(0);
        if constexpr (FIRST) {
#pragma unroll
            for (int k = 0; k < LN; ++k) ca[k] = na[k] = T(0);
        } else {
            // the first rows in use, by their place among the item's input rows: level 0 starts row i + 1 with
            // input row i, and completes (END) row i - 1; earlier rows feed no output
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int k = 0; k < LN; ++k) win[q][k] = T(0);
            ry = y0 - TT + (END ? 0 : 1);
            ry = ry < 0 ? ry + g.ny : ry % g.ny;
            if constexpr (!END) {
                fetch(xb, win[1]);
#pragma unroll
                for (int k = 0; k < LN; ++k) win[1][k] = rmul(jw, win[1][k]);
            }
            fetch(xb, next);
        }
        for (int i = 0; i < nrows && !failed; i += 4) {
            static_for<0, 2>([&](auto gc) {
                constexpr int G2 = decltype(gc)::value;
                if (failed) return;
                const bool ok = mbar_wait_bounded(&full[cs], cphase);
                if (__any_sync(0xffffffffu, !ok)) {
                    failed = true;
                    return;
                }
                T in[2][LN + 2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const unsigned char* row = ring + (size_t)cs * X::SLOT + j * X::ROWB;
                    T v4[4];
                    lds4<ST, PDE_LCDE>(row + (size_t)(X::ALIGN + lane * LN) * X::ES, T(0), v4);
                    in[j][0] = Storage<ST>::raw(reinterpret_cast<const S*>(row) + X::ALIGN + lane * LN - 1);
                    in[j][1] = v4[0];
                    in[j][2] = v4[1];
                    in[j][3] = v4[2];
                    in[j][4] = v4[3];
                    in[j][5] = Storage<ST>::raw(reinterpret_cast<const S*>(row) + X::ALIGN + lane * LN + LN);
                }
                ++consumed;
                cs = cs + 1 == NSTAGE ? 0 : cs + 1;
                if (cs == 0) cphase ^= 1u;
                __syncwarp();
                if (lane == 0) {
                    fence_proxy_async_smem();
                    issue_next();
                }
                static_for<0, 2>([&](auto jc) {
                    constexpr int J = 2 * G2 + decltype(jc)::value;   // input row i + J
                    T(&raw)[LN + 2] = in[decltype(jc)::value];
                    T o[LN];
                    const int yo = y0 - 2 * TT + i + J;
                    const bool stored = i + J >= 2 * TT && i + J < hrows + 2 * TT;   // warp-uniform
                    const T zero[LN] = {T(-0.0), T(-0.0), T(-0.0), T(-0.0)};
                    if constexpr (FIRST) {
                        T r[LN];
                        stencil_row<LAT, T>(A.W0, A.Wp, A.Wm, raw, zero, ca, na, r);
                        stencil_row<LAT, T>(B.W0, B.Wp, B.Wm, raw, zero, c[0], n[0], o);
                        if (stored) {
                            es.template put<1>(rhs, g.fs, g, xb, yo, 0, [&](int, S (&sv)[4]) {
#pragma unroll
                                for (int k = 0; k < 4; ++k) sv[k] = r[k];
                            });
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < TT; ++t) {
                            if (t > 0) {
                                raw[0] = __shfl_up_sync(0xffffffffu, raw[LN], 1);
                                raw[LN + 1] = __shfl_down_sync(0xffffffffu, raw[1], 1);
                            }
                            // level t takes row i + J - t, starts row i + J - t + 1 and completes row i + J - t - 1
                            if constexpr (END) {
                                stencil_row<LAT, T>(B.W0, B.Wp, B.Wm, raw, zero, c[t], n[t], o);
#pragma unroll
                                for (int k = 0; k < LN; ++k) o[k] = rfma(jw, win[(J - t + 7) & 3][k], o[k]);
                            } else {
                                stencil_row<LAT, T>(B.W0, B.Wp, B.Wm, raw, win[(J - t + 5) & 3], c[t], n[t], o);
                            }
#pragma unroll
                            for (int k = 0; k < LN; ++k) raw[1 + k] = o[k];
                        }
                        // the row that input row i + J + 1 starts (END: completes), and the fetch of the one after it
#pragma unroll
                        for (int k = 0; k < LN; ++k) win[(END ? J : J + 2) & 3][k] = END ? next[k] : rmul(jw, next[k]);
                        fetch(xb, next);
                    }
                    if (stored) {
                        es.template put<1>(out, g.fs, g, xb, yo, 0, [&](int, S (&sv)[4]) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) sv[k] = o[k];
                        });
                    }
                });
            });
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

// The level-t stencil of a Coef or SrcCoef block.
template <typename T, template <typename> class Block>
Stencil<T> stencil_of(const void* block) {
    const Block<T>& b = *static_cast<const Block<T>*>(block);
    Stencil<T> s;
    s.W0 = b.W0[0];
    for (int p = 0; p < kMaxPair; ++p) {
        s.Wp[p] = b.Wp[0][p];
        s.Wm[p] = b.Wm[0][p];
    }
    return s;
}

template <int LAT, int ST, int TT, bool FIRST, bool END>
cudaError_t launch(const LaunchArgs& a) {
    using T = typename Storage<ST>::T;
    using S = typename Storage<ST>::S;
    constexpr int NW = 4;
    constexpr size_t smem = RowBox<ST>::smem(NW);
    auto kern = k_theta<LAT, ST, TT, FIRST, END, NW>;
    static std::atomic<unsigned long long> known[kMaxDevices];
    Fit fit;
    const cudaError_t e = fit_of(kern, NW * 32, smem, known, &fit);
    if (e != cudaSuccess) return e;
    const int resident = fit.ctas();
    constexpr int STRIDE = FIRST ? 128 : kThStride, LEAD = FIRST ? 0 : kThLead;
    const int strips = (a.g.nx + LEAD / 2 + STRIDE - 1) / STRIDE;
    int H = a.H;
    if (H <= 0) H = march_height(strips, a.g.ny, (long long)resident * NW, 2 * TT + 1, FIRST ? 2 : 8, 512);
    const int nitems = strips * ((a.g.ny + H - 1) / H);
    const int blocks = (nitems + NW - 1) / NW;
    Stencil<T> A{}, B;
    T jw = T(0);
    if constexpr (FIRST) {
        A = stencil_of<T, Coef>(a.coef);
        B = stencil_of<T, SrcCoef>(a.src_coef);
    } else {
        B = stencil_of<T, Coef>(a.coef);
        jw = static_cast<const SrcCoef<T>*>(a.src_coef)->W0[0];
    }
    return launch_chained(kern, blocks < resident ? blocks : resident, NW * 32, smem, a.stream, a.chained, *a.maps, a.g,
                          static_cast<S*>(a.out), static_cast<S*>(const_cast<void*>(a.src[0])), A, B, jw, H, nitems, a.err);
}

template <int LAT, bool END>
LaunchFn pick(int st, int depth) {
    if (st == ST_F64)
        return depth == 1 ? launch<LAT, ST_F64, 1, false, END> : depth == 2 ? launch<LAT, ST_F64, 2, false, END> : nullptr;
    switch (depth) {
    case 1: return launch<LAT, ST_F32, 1, false, END>;
    case 2: return launch<LAT, ST_F32, 2, false, END>;
    case 3: return launch<LAT, ST_F32, 3, false, END>;
    case 4: return launch<LAT, ST_F32, 4, false, END>;
    }
    return nullptr;
}
template <int LAT>
LaunchFn pick_end(int st, int depth, bool end) {
    if (depth == 0) return st == ST_F64 ? launch<LAT, ST_F64, 1, true, false> : launch<LAT, ST_F32, 1, true, false>;
    return end ? pick<LAT, true>(st, depth) : pick<LAT, false>(st, depth);
}

}  // namespace

LaunchFn find_march2d_theta(int lat, int st, int depth, bool end) {
    if (st == ST_BF16) return nullptr;
    if (lat == LAT_D2Q5) return pick_end<LAT_D2Q5>(st, depth, end);
    if (lat == LAT_D2Q9) return pick_end<LAT_D2Q9>(st, depth, end);
    return nullptr;
}

}  // namespace mmfd
