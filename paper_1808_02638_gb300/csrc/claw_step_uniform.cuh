// claw_step_uniform.cuh -- the fused, persistent level-step in a uniform medium (rho0, K0).
//
// The skeleton is that of the cell-wise step (claw_step.cuh): persistent CTAs take the level's tiles,
// staged into shared memory by tensor bulk copies.  Two things differ:
//  * a tile is stepped in 64-bit fixed point (claw_fixed.cuh); the FP64 phases below take the tiles
//    whose states that does not fit, 8 rows at a time;
//  * everything a tile needs from global memory is fetched while the tile before it is computed:
//    its descriptors, its state (boxes with an odd nx or offset, which no bulk copy takes, by
//    asynchronous 8-byte copies of every cell), and the cells that its ghosts are pulled from (ring entries
//    into registers behind the first barrier, the values by asynchronous 8-byte copies behind the
//    strengths: into the frame of the next tile's buffer, which its bulk copy has filled by then, or,
//    with one buffer, into a side buffer).  Fetched when their tile began they cost 9 of 26 thousand
//    cycles of a 32 x 32 tile.
#pragma once

#include "claw_fixed.cuh"
#include "claw_reflux.cuh"
#include "claw_step.cuh"

namespace claw {

// Rows that the FP64 phases step at a time: 16 where that costs the kernel nothing, since the halo rows and the
// barriers then weigh less (2048^2, MC, every tile sent there, us a step by 8 and 16 rows: 32 x 32 tiles
// 516 and 474, 16 x 16 with 128 threads 544 and 491).  The others would lose a CTA per SM to the
// larger work arrays (32 x 16, two buffers) or spill under their register caps (32 x 16 with 352
// threads 236 and 299 in fixed point, 16 x 16 with 192 threads 255 and 273).
template <int TX, int TY, int NT, int STAGE> struct UniGeo {
    using G = Geo<TX, TY>;
    static constexpr int FP64_ROWS = TX == TY && NT != 192 ? 16 : 8;
    static constexpr int NF = 4 * (TX + TY + 4);             // cells of a staged tile's two-cell frame
    static constexpr int NI = (NF + NT - 1) / NT;            // ... of one thread
    static constexpr int FP64 = Geo<TX, FP64_ROWS>::NWORK, FIXED = fx::Strips<TX, TY, NT>::WORDS;
    static constexpr int WORK = ((FP64 > FIXED ? FP64 : FIXED) + 15) / 16 * 16;
    // q buffers, work arrays, side buffer of the pulled frame, two barriers (8-byte words)
    static constexpr int side(int pull) { return pull && STAGE == 2 ? 3 * NF : 0; }
    static constexpr size_t smem(int pull)
    {
        return (size_t)((STAGE == 2 ? 1 : 2) * G::QSTRIDE + WORK + side(pull) + 2) * 8;
    }
};

// ------------------------------------------------------------------------- the FP64 phases
// Steps the staged tile (planes qpl apart, rows SW = TX + 4) into q_new in rounds of ROWS rows;
// returns the error flags seen.  With a = 2 alpha and M = phi(theta) a:
//   x-normal update  dp = -(lx K/2) ap - (lx kap Z/4) bp,  du = -(lx c/2) au - (lx kap/4) bu
//   (dp also carries the centre term 2 kT D of the transverse update)
//   ap = A2_w + A1_e, au = A2_w - A1_e, bp = S_e - S_w, bu = P_e - P_w,  kap = c (1 - lx c)
//   x-fluctuation pressure into the cell D = (K/2) (ap + (1 - lx c) bp)
template <int LIM, int TX, int ROWS, int NT>
__device__ __noinline__ int uniform_tile_fp64(const StepArgs& A, const PatchDev& P, const double* sq, int qpl,
                                              double* work, int tx, int tile_ty, int x0, int tile_y0)
{
    using G = Geo<TX, ROWS>;
    constexpr int NPER = (TX * ROWS + NT - 1) / NT;
    double* A1x = work;                             // x-edge wave strengths, family 1 / 2
    double* A2x = A1x + G::XEW * G::XEH;
    double* B1y = A2x + G::XEW * G::XEH;            // y-edge wave strengths
    double* B2y = B1y + G::YEW * G::YEH;
    double* Sx = B2y + G::YEW * G::YEH;             // limited x-edges: M2 - M1
    double* Px = Sx + G::XLW * G::XLH;              //                  M1 + M2
    double* Sy = Px + G::XLW * G::XLH;
    double* Py = Sy + G::YLW * G::YLH;
    double* Dx = Py + G::YLW * G::YLH;              // x-fluctuation pressure into each cell
    double* Ey = Dx + G::DW * G::DH;                // y-fluctuation pressure into each cell
    __shared__ double s_k[12];
    const int tid = threadIdx.x;
    const bool second = A.order == 2;
    const bool trans = A.transverse != 0;
    const bool cw = A.transverse == 2 && A.order == 2;   // correction rides the transverse split
    const double c0 = A.c0, Z0 = A.Z0, iZ = A.iZ;
    const int W = P.nx + 4;
    const long long WH = (long long)W * (P.ny + 4);
    int flag = 0;
    if (tid == 0) {   // read behind the barrier that ends phase A
        const double dt = __ldg(A.dt + P.run) * P.dtscale;
        const double lx = dt * P.dxinv, ly = dt * P.dyinv;
        // the centre part 2 kT (D + E) of the transverse pressure update folds into the
        // normal-update coefficients (D = ap + kDx bp, E likewise); phase D adds the rest
        const double kapx = c0 * (1.0 - lx * c0), kapy = c0 * (1.0 - ly * c0);
        const double kDx = cw ? 1.0 - lx * c0 : 0.0, kDy = cw ? 1.0 - ly * c0 : 0.0;
        const double kT = trans ? 0.125 * lx * ly * c0 * A.K0 : 0.0;
        s_k[0] = fma(-0.5 * lx, A.K0, 2.0 * kT);              // cpa
        s_k[1] = fma(-0.25 * lx * kapx, Z0, 2.0 * kT * kDx);  // cpb
        s_k[2] = -0.5 * lx * c0;                              // cua
        s_k[3] = -0.25 * lx * kapx;                           // cub
        s_k[4] = fma(-0.5 * ly, A.K0, 2.0 * kT);              // cpay
        s_k[5] = fma(-0.25 * ly * kapy, Z0, 2.0 * kT * kDy);  // cpby
        s_k[6] = -0.5 * ly * c0;                              // cva
        s_k[7] = -0.25 * ly * kapy;                           // cvb
        s_k[8] = kDx;
        s_k[9] = kDy;
        s_k[10] = -kT;
        s_k[11] = trans ? 0.125 * lx * ly * c0 * c0 : 0.0;   // kU
    }
    for (int h0 = 0; h0 < tile_ty; h0 += ROWS) {
        const int ty = min(ROWS, tile_ty - h0), y0 = tile_y0 + h0;
        const double* sp = sq + h0 * G::SW;
        const double* su = sp + qpl;
        const double* sv = su + qpl;
        // ---------------------------------------------------------------- phase A: normal Riemann
        {   // x-edge a (between cells a-1 and a) on rows r in [-1, ty]
            const int w = tx + 3, n = (ty + 2) * w;
            for (int k = tid; k < n; k += NT) {
                const int r = k / w - 1, a = k - (r + 1) * w - 1;
                const int iR = (a + 2) + (r + 2) * G::SW;
                const double dp = sp[iR] - sp[iR - 1];
                const double du = su[iR] - su[iR - 1];
                A1x[(r + 1) * G::XEW + (a + 1)] = fma(-dp, iZ, du);   // 2 alpha: du -/+ dp / Z
                A2x[(r + 1) * G::XEW + (a + 1)] = fma(dp, iZ, du);
            }
        }
        {   // y-edge b (between rows b-1 and b) on columns c in [-1, tx]
            const int w = tx + 2, n = (ty + 3) * w;
            for (int k = tid; k < n; k += NT) {
                const int bb = k / w - 1, c = k - (bb + 1) * w - 1;
                const int iR = (c + 2) + (bb + 2) * G::SW;
                const double dp = sp[iR] - sp[iR - G::SW];
                const double dv = sv[iR] - sv[iR - G::SW];
                B1y[(bb + 1) * G::YEW + (c + 1)] = fma(-dp, iZ, dv);
                B2y[(bb + 1) * G::YEW + (c + 1)] = fma(dp, iZ, dv);
            }
        }
        __syncthreads();
        // ---------------------------------------------------------------- phase B: limiter
        if (second) {
            {
                const int w = tx + 1, n = (ty + 2) * w;
                for (int k = tid; k < n; k += NT) {
                    const int r = k / w - 1, a = k - (r + 1) * w;
                    const int e = (r + 1) * G::XEW + (a + 1);
                    const double m1 = Lim<LIM>::f(A1x[e], A1x[e + 1]);   // left-going: upwind edge a+1
                    const double m2 = Lim<LIM>::f(A2x[e], A2x[e - 1]);   // right-going: upwind edge a-1
                    Sx[(r + 1) * G::XLW + a] = m2 - m1;
                    Px[(r + 1) * G::XLW + a] = m1 + m2;
                }
            }
            {
                const int w = tx + 2, n = (ty + 1) * w;
                for (int k = tid; k < n; k += NT) {
                    const int bb = k / w, c = k - bb * w - 1;
                    const int e = (bb + 1) * G::YEW + (c + 1);
                    const double m1 = Lim<LIM>::f(B1y[e], B1y[e + G::YEW]);
                    const double m2 = Lim<LIM>::f(B2y[e], B2y[e - G::YEW]);
                    Sy[bb * G::YLW + (c + 1)] = m2 - m1;
                    Py[bb * G::YLW + (c + 1)] = m1 + m2;
                }
            }
            __syncthreads();
        }
        // ---------------------------------------------------------------- phase C: per-cell terms
        const double kDx = s_k[8], kDy = s_k[9];
        double dP[NPER], dU[NPER], dV[NPER];   // Q plus the normal updates
#pragma unroll
        for (int n = 0; n < NPER; ++n) {
            dP[n] = dU[n] = dV[n] = 0.0;
            const int ci = tid + n * NT;
            const int c = ci % TX, r = ci / TX;
            if (ci >= TX * ROWS || c >= tx || r >= ty) continue;
            const int iq = (c + 2) + (r + 2) * G::SW;
            const int ex = (r + 1) * G::XEW + (c + 1);
            const int ey = (r + 1) * G::YEW + (c + 1);
            const double apx = A2x[ex] + A1x[ex + 1], aux = A2x[ex] - A1x[ex + 1];
            const double apy = B2y[ey] + B1y[ey + G::YEW], avy = B2y[ey] - B1y[ey + G::YEW];
            double bpx = 0, bux = 0, bpy = 0, bvy = 0;
            if (second) {
                bpx = Sx[(r + 1) * G::XLW + c + 1] - Sx[(r + 1) * G::XLW + c];
                bux = Px[(r + 1) * G::XLW + c + 1] - Px[(r + 1) * G::XLW + c];
                bpy = Sy[(r + 1) * G::YLW + c + 1] - Sy[r * G::YLW + c + 1];
                bvy = Py[(r + 1) * G::YLW + c + 1] - Py[r * G::YLW + c + 1];
            }
            if (trans) {
                Dx[(r + 1) * G::DW + c] = fma(kDx, bpx, apx);
                Ey[r * G::EW + c + 1] = fma(kDy, bpy, apy);
            }
            dP[n] = fma(s_k[0], apx, fma(s_k[1], bpx, fma(s_k[4], apy, fma(s_k[5], bpy, sp[iq]))));
            dU[n] = fma(s_k[2], aux, fma(s_k[3], bux, su[iq]));
            dV[n] = fma(s_k[6], avy, fma(s_k[7], bvy, sv[iq]));
        }
        if (trans) {   // D on the ghost rows -1, ty and E on the ghost columns -1, tx
            const int n = 2 * (tx + ty);
            for (int k = tid; k < n; k += NT) {
                if (k < 2 * tx) {
                    const int c = k % tx, r = (k < tx) ? -1 : ty;
                    const int ex = (r + 1) * G::XEW + (c + 1);
                    const double bpx = second ? Sx[(r + 1) * G::XLW + c + 1] - Sx[(r + 1) * G::XLW + c] : 0.0;
                    Dx[(r + 1) * G::DW + c] = fma(kDx, bpx, A2x[ex] + A1x[ex + 1]);
                } else {
                    const int kk = k - 2 * tx;
                    const int r = kk % ty, c = (kk < ty) ? -1 : tx;
                    const int ey = (r + 1) * G::YEW + (c + 1);
                    const double bpy = second ? Sy[(r + 1) * G::YLW + c + 1] - Sy[r * G::YLW + c + 1] : 0.0;
                    Ey[r * G::EW + c + 1] = fma(kDy, bpy, B2y[ey] + B1y[ey + G::YEW]);
                }
            }
        }
        __syncthreads();
        // ---------------------------------------------------------------- phase D: update, store
        const double kT = s_k[10], kU = s_k[11];
        double* dst = A.qnew + P.qoff;
#pragma unroll
        for (int n = 0; n < NPER; ++n) {
            const int ci = tid + n * NT;
            const int c = ci % TX, r = ci / TX;
            if (ci >= TX * ROWS || c >= tx || r >= ty) continue;
            double p = dP[n], u = dU[n], v = dV[n];
            if (trans) {
                const double dn = Dx[(r + 2) * G::DW + c], ds = Dx[r * G::DW + c];
                const double ee = Ey[r * G::EW + c + 2], ew = Ey[r * G::EW + c];
                p = fma(kT, (dn + ds) + (ee + ew), p);   // kT holds -kT; 2 kT (dc + ec) is in p
                u = fma(kU, ee - ew, u);
                v = fma(kU, dn - ds, v);
            }
            if (not_finite(p) | not_finite(u) | not_finite(v)) flag |= ERR_NAN;
            const long long o = (long long)(y0 + r + 2) * W + (x0 + c + 2);
            dst[o] = p;
            dst[WH + o] = u;
            dst[2 * WH + o] = v;
        }
        __syncthreads();   // the work arrays are reused by the next rows or tile
    }
    return flag;
}

// ------------------------------------------------------------------------- the kernel
// STAGE: two buffers, filled by 0 asynchronous 8-byte copies, 1 tensor bulk copies; 2 tensor bulk copies into
// one (the next tile's copy is requested behind the first barrier, when the tile's state is in registers).
// PULL: 1 same-level and boundary ghosts are taken from their source cells; 2 those and the ghosts
// interpolated from the coarser level, evaluated in the step.
template <int LIM, int TX, int TY, int NT, int STAGE, int PULL>
__global__ void __launch_bounds__(NT, NT == 128 ? 4 : NT == 256 ? (TY == 16 ? 3 : 2) : NT == 352 ? 2 : NT == 192 ? 3 : 1)
    uniform_step_kernel(const __grid_constant__ StepArgs A)
{
    using U = UniGeo<TX, TY, NT, STAGE>;
    using G = Geo<TX, TY>;
    constexpr bool TWO = STAGE != 2;
    constexpr int NBUF = TWO ? 2 : 1;
    constexpr int NI = U::NI;
    if (A.step_grid && blockIdx.x >= A.step_grid) {   // a CTA beside those: no tiles, no shared memory
        if (PULL == 0 && A.nreflux && blockIdx.x >= A.reflux_grid)   // (reflux levels fill their ghosts)
            refl::run_jobs<LIM, NT>(A, A.reflux_grid, gridDim.x - A.reflux_grid);
        else
            fill_jobs<NT>(A);
        if (threadIdx.x == 0) finish_cta(A);
        return;
    }
    const int nstep = A.step_grid ? A.step_grid : (int)gridDim.x;   // the CTAs that step tiles
    extern __shared__ __align__(128) double smem[];
    double* qbuf = smem;                              // NBUF x QSTRIDE
    double* work = smem + NBUF * G::QSTRIDE;
    double* frame = work + U::WORK;                   // side buffer of the pulled ghosts: 3 planes of NF
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(frame + U::side(PULL));
    __shared__ PatchDev s_patch[2];                   // the tile's box, by tile parity
    __shared__ fx::Shared s_fx;
    __shared__ int s_flag;
    __shared__ int s_range[2];
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;

    // the CTA's tiles: strided by the grid, or a contiguous range of a column walk
    int t = blockIdx.x, t_end = A.ntiles;
    const int t_step = A.tcum ? 1 : nstep;
    if (A.tcum) {
        if (tid < 2) s_range[tid] = walk_start(A.tcum, A.ntiles, blockIdx.x + tid, nstep);
        __syncthreads();
        t = s_range[0];
        t_end = s_range[1];
    }
    const CUtensorMap* tmaps = reinterpret_cast<const CUtensorMap*>(A.tmaps);
    auto issue = [&](const TileDev& T, int b) {   // thread 0
        mbar_expect_tx(&bar[b], (unsigned)G::QBYTES);
        tma_load_3d(qbuf + b * G::QSTRIDE, &tmaps[T.patch], T.x0, T.y0, 0, &bar[b]);
    };
    static_assert(sizeof(PatchDev) % 8 == 0 && sizeof(PatchDev) / 8 <= 32, "a warp copies a PatchDev");
    TileDev T;
    if (t < t_end) T = A.tiles[t];
    if (tid == 0) {
        s_flag = 0;
        fx::init(s_fx, A.iZ);
        if (STAGE) {
            mbar_init(&bar[0], 1);
            mbar_init(&bar[1], 1);
            fence_barrier_init();
            if (t < t_end) issue(T, 0);
        }
    }
    if (wid == 1 && lane < (int)sizeof(PatchDev) / 8 && t < t_end)
        reinterpret_cast<long long*>(&s_patch[0])[lane] =
            __ldg(reinterpret_cast<const long long*>(A.patches + T.patch) + lane);
    __syncthreads();

    // a thread's cells of a tile's frame of width two: cell k of rows 0, 1, ty+2, ty+3, then of
    // columns 0, 1, tx+2, tx+3 of the rows between
    auto frame_cell = [&](int k, int tx, int ty, int& xs, int& ys) {
        const int w = tx + 4;
        if (k < 4 * w) {
            const int r = (k >= w) + (k >= 2 * w) + (k >= 3 * w);
            xs = k - r * w;
            ys = r < 2 ? r : ty + r;
        } else {
            const int kk = k - 4 * w, c = kk & 3;
            ys = 2 + (kk >> 2);
            xs = c < 2 ? c : tx + c;
        }
    };
    longlong2 ring[NI];   // entries of the next tile's frame cells (first: source or interpolated, -1 - j)
    int pulled[NI];       // 0: nothing, 1: interpolated (ring[i].x kept), 4 + wall flips: copied
    auto ring_load = [&](const TileDev& T, const PatchDev& P) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int k = tid + i * NT;
            pulled[i] = 0;
            if (P.ring < 0 || k >= 4 * (T.tx + T.ty + 4)) continue;
            int xs, ys;
            frame_cell(k, T.tx, T.ty, xs, ys);
            const int ri = ring_index(T.x0 + xs, T.y0 + ys, P.nx, P.ny);
            if (ri < 0) continue;
            ring[i] = __ldg(&A.ring[P.ring + ri]);
            pulled[i] = 1;
        }
    };
    // starts the copies for tile T; sq (two buffers): its staged state, already in place
    auto ring_fetch = [&](const TileDev& T, double* sq) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            if (!pulled[i]) continue;
            if (ring[i].x < 0) {   // interpolated from the coarser level: staged from the pool, or evaluated
                if (PULL != 2) pulled[i] = 0;
                continue;
            }
            const long long sp = ring[i].y & ((1LL << kRingFlagShift) - 1);
            const double* src = A.qold + ring[i].x;
            double* dst = frame + tid + i * NT;
            int plane = U::NF;
            if (TWO) {
                int xs, ys;
                frame_cell(tid + i * NT, T.tx, T.ty, xs, ys);
                dst = sq + xs + ys * G::SW;
                plane = G::QPL;
            }
            cp_async8(dst, src);
            cp_async8(dst + plane, src + sp);
            cp_async8(dst + 2 * plane, src + 2 * sp);
            pulled[i] = 4 + (int)(ring[i].y >> kRingFlagShift);
        }
    };
    auto ring_store = [&](const TileDev& T, const PatchDev& P, double* sq) {
        cp_async_wait_all();   // this thread's copies: it reads no other's
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            if (!pulled[i]) continue;
            int xs, ys;
            frame_cell(tid + i * NT, T.tx, T.ty, xs, ys);
            double* d = sq + xs + ys * G::SW;
            if (PULL == 2 && pulled[i] == 1) {
                const InterpCell C = A.interp[P.interp + (int)(-1 - ring[i].x)];
#pragma unroll
                for (int m = 0; m < 3; ++m) d[m * G::QPL] = interp_value(C, m, A.cold, A.cnew, A.tau);
                continue;
            }
            // wall sign flips as sign-bit xors
            if (TWO && pulled[i] == 4) continue;
            const double* f = TWO ? d : frame + tid + i * NT;
            constexpr int plane = TWO ? G::QPL : U::NF;
            const unsigned long long su = (unsigned long long)(pulled[i] & 1) << 63;
            const unsigned long long sv = (unsigned long long)((pulled[i] >> 1) & 1) << 63;
            d[0] = f[0];
            d[G::QPL] = __longlong_as_double((long long)((unsigned long long)__double_as_longlong(f[plane]) ^ su));
            d[2 * G::QPL] =
                __longlong_as_double((long long)((unsigned long long)__double_as_longlong(f[2 * plane]) ^ sv));
        }
        // these generic writes precede later bulk copies (async proxy) into the same buffer
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };
    // STAGE 0: starts the copies of a tile's state, ghost cells included
    auto stage_copy = [&](const TileDev& T, const PatchDev& P, double* sq) {
        const int w = T.tx + 4, h = T.ty + 4, n = 3 * h * w, m20 = (1 << 20) / w + 1, W = P.nx + 4;
        const long long WH = (long long)W * (P.ny + 4);
        const double* src = A.qold + P.qoff + (long long)T.y0 * W + T.x0;
        for (int k = tid; k < n; k += NT) {
            const int row = (k * m20) >> 20, col = k - row * w;   // k / w, exact for k w < 2^20
            const int m = (row >= h) + (row >= 2 * h), jj = row - m * h;
            cp_async8(sq + m * G::QPL + jj * G::SW + col, src + m * WH + (long long)jj * W + col);
        }
    };
    if (STAGE == 0 && t < t_end) {
        stage_copy(T, s_patch[0], qbuf);
        cp_async_wait_all();
        __syncthreads();   // the pulled cells go over staged ones
    }
    // a tile's barrier completes once per use of its buffer: every other tile with two buffers,
    // every tile with one
    auto landed = [&](int it) {
        return mbar_wait_bounded(&bar[STAGE == 1 ? it & 1 : 0], (unsigned)((STAGE == 1 ? it >> 1 : it) & 1),
                                 A.wait_polls);
    };
    bool late = false;   // the copy of this or (from strengths_done on) the next tile did not land in time
    if (PULL && t < t_end) {
        ring_load(T, s_patch[0]);
        late = STAGE == 1 && !landed(0);
        if (!late) ring_fetch(T, qbuf);
    }

    int my_flag = 0;
    int cur_run = -1;   // thread 0: the run whose speed the CTA has not reported yet
    auto flush = [&]() {
        if (cur_run >= 0 && A.c0 > 0.0)
            atomicMax(reinterpret_cast<unsigned long long*>(A.smax) + cur_run,
                      (unsigned long long)__double_as_longlong(A.c0));
    };
    int fx_run = -1, fx_set = 0;   // the run whose constants s_fx.run[fx_set] holds
    int it = 0;
    for (; t < t_end; t += t_step, ++it) {
        const int par = it & 1, b = TWO ? par : 0;
        const bool more = t + t_step < t_end;
        TileDev Tn;   // the next tile (used behind the first barrier of this one)
        if (more) Tn = A.tiles[t + t_step];
        const PatchDev& P = s_patch[par];
        double* sq = qbuf + b * G::QSTRIDE;
        if (P.run != fx_run) {
            fx_run = P.run;
            fx_set ^= 1;
            if (wid == NT / 32 - 1)   // read behind the tile's first barrier
                fx::init_run(s_fx, s_fx.run[fx_set], __ldg(A.dt + P.run) * P.dtscale, P.dxinv, P.dyinv, A.c0);
        }

        // ---------------------------------------------------------------- staged state
        if (STAGE && !(PULL && STAGE == 1)) late = !landed(it);
        if (STAGE == 0 && !PULL) cp_async_wait_all();   // (ring_store waits otherwise)
        if (PULL && !late) ring_store(T, P, sq);
        if (__syncthreads_or(late)) {   // the copy is late or lost: report and stop this CTA
            if (PULL) cp_async_wait_all();
            if (tid == 0) {
                atomicOr(A.err, ERR_TIMEOUT);
                // no copy may land in this CTA's shared memory after it exits: wait, with the full
                // bound, for this tile's own (the next one's is not requested yet)
                mbar_wait_bounded(&bar[b], (unsigned)((STAGE == 1 ? it >> 1 : it) & 1));
                finish_cta(A);   // keeps the completion count consistent
            }
            return;
        }
        // every thread is done with the previous tile: its buffer and its box's slot are free
        if (STAGE == 1 && tid == 0 && more) issue(Tn, par ^ 1);
        if (more && wid == 1) {
            if (lane < (int)sizeof(PatchDev) / 8)
                cp_async8(reinterpret_cast<long long*>(&s_patch[par ^ 1]) + lane,
                          reinterpret_cast<const long long*>(A.patches + Tn.patch) + lane);
        }

        // ---------------------------------------------------------------- the tile
        // the next tile's box has arrived behind the first barrier: warp 1 waits for it before
        auto jumps_done = [&]() {
            if (more && wid == 1) cp_async_wait_all();
        };
        auto begin = [&]() {
            if (STAGE == 2 && tid == 0 && more) issue(Tn, 0);
            if (STAGE == 0 && more) stage_copy(Tn, s_patch[par ^ 1], qbuf + (par ^ 1) * G::QSTRIDE);
            if (PULL && more) ring_load(Tn, s_patch[par ^ 1]);
        };
        auto strengths_done = [&]() {
            if (PULL && more && STAGE) {
                late = STAGE == 1 && !landed(it + 1);   // (requested when this tile began)
                if (!late) ring_fetch(Tn, qbuf + (par ^ 1) * G::QSTRIDE);
            }
            if (PULL && STAGE == 0) cp_async_wait_all();   // behind the second barrier the state is in place
        };
        auto limited_done = [&]() {
            if (PULL && more && STAGE == 0) ring_fetch(Tn, qbuf + (par ^ 1) * G::QSTRIDE);
        };
        const bool done = fx::step_tile<G, LIM, TX, TY, NT, STAGE == 2>(
            A, P, s_fx, s_fx.run[fx_set], par, sq, work, A.Z0, T.tx, T.ty, T.x0, T.y0, my_flag, jumps_done, begin,
            strengths_done, limited_done);
        if (!done) {
            my_flag |= uniform_tile_fp64<LIM, TX, U::FP64_ROWS, NT>(A, P, sq, G::QPL, work, T.tx, T.ty, T.x0, T.y0);
            begin();
            strengths_done();
            if (PULL && STAGE == 0) __syncthreads();
            limited_done();
        }
        if (tid == 0 && P.run != cur_run) {
            flush();
            cur_run = P.run;
        }
        if (more) T = Tn;
    }

    // ---------------------------------------------------------------- CFL and error flags
    if (tid == 0) flush();
    if (my_flag) atomicOr(&s_flag, my_flag);
    __syncthreads();
    if (tid == 0 && s_flag) atomicOr(A.err, s_flag);
    if (tid == 0) finish_cta(A);
}

template <int LIM, int TX, int TY, int NT, int STAGE, int PULL> StepKernel uniform_kernel_entry()
{
    StepKernel k;
    k.fn = uniform_step_kernel<LIM, TX, TY, NT, STAGE, PULL>;
    k.smem = UniGeo<TX, TY, NT, STAGE>::smem(PULL);
    k.nt = NT;
    return k;
}

// tile shapes x thread counts x stagings of one limiter (nt = 0: the default)
template <int LIM, int PULL> StepKernel uniform_kernel_select(int tx, int ty, int nt, int staging)
{
    if (tx == 32 && ty == 32 && (nt == 0 || nt == 256)) {
        if (staging == 2) return uniform_kernel_entry<LIM, 32, 32, 256, 2, PULL>();
        return staging ? uniform_kernel_entry<LIM, 32, 32, 256, 1, PULL>()
                       : uniform_kernel_entry<LIM, 32, 32, 256, 0, PULL>();
    }
    if (tx == 32 && ty == 16 && nt == 352)
        return staging ? uniform_kernel_entry<LIM, 32, 16, 352, 1, PULL>()
                       : uniform_kernel_entry<LIM, 32, 16, 352, 0, PULL>();
    if (tx == 16 && ty == 16 && nt == 192)
        return staging ? uniform_kernel_entry<LIM, 16, 16, 192, 1, PULL>()
                       : uniform_kernel_entry<LIM, 16, 16, 192, 0, PULL>();
    if (tx == 32 && ty == 32 && nt == 512)
        return staging ? uniform_kernel_entry<LIM, 32, 32, 512, 1, PULL>()
                       : uniform_kernel_entry<LIM, 32, 32, 512, 0, PULL>();
    if (tx == 32 && ty == 16 && (nt == 0 || nt == 256)) {
        if (staging == 2) return uniform_kernel_entry<LIM, 32, 16, 256, 2, PULL>();
        return staging ? uniform_kernel_entry<LIM, 32, 16, 256, 1, PULL>()
                       : uniform_kernel_entry<LIM, 32, 16, 256, 0, PULL>();
    }
    if (tx == 16 && ty == 16 && (nt == 0 || nt == 128))
        return staging ? uniform_kernel_entry<LIM, 16, 16, 128, 1, PULL>()
                       : uniform_kernel_entry<LIM, 16, 16, 128, 0, PULL>();
    return StepKernel{nullptr, 0, 0};
}

template <int PULL> StepKernel uniform_kernel_for(int lim, int tx, int ty, int nt, int staging)
{
    switch (lim) {
    case CLAW_LIM_NONE: return uniform_kernel_select<CLAW_LIM_NONE, PULL>(tx, ty, nt, staging);
    case CLAW_LIM_MINMOD: return uniform_kernel_select<CLAW_LIM_MINMOD, PULL>(tx, ty, nt, staging);
    case CLAW_LIM_SUPERBEE: return uniform_kernel_select<CLAW_LIM_SUPERBEE, PULL>(tx, ty, nt, staging);
    case CLAW_LIM_VANLEER: return uniform_kernel_select<CLAW_LIM_VANLEER, PULL>(tx, ty, nt, staging);
    case CLAW_LIM_MC: return uniform_kernel_select<CLAW_LIM_MC, PULL>(tx, ty, nt, staging);
    }
    return StepKernel{nullptr, 0, 0};
}

}  // namespace claw
