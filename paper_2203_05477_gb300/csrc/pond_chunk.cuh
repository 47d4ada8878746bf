// pond_chunk.cuh -- the fused step of D1Q4 grids: a warp per chunk of cells.
//
// A warp stages its chunk and two cells on each side (phi-bar-plus, one cell per lane), solves the
// chunk's faces and updates its cells from them; the faces at a chunk's ends are solved by both
// neighbours.  State and face frames are read from one set of buffers and written to the other,
// so no warp waits for another, and the next chunk's loads are issued before the current one is
// solved.  Face populations never reach memory: 112 bytes a cell (FP32) where the face and cell kernels
// move 224.  With a lane per face the chunk is 28 cells; with four lanes per face (pass1_quad) it is
// 7, which spreads a short grid over four times the warps.
//
// Measured (GB300, us a step; before: face and cell kernels): 4 M cells FP32 189 (338), at 72% of the
// issue slots with 16 warps per SM (128 registers; 96 would spill 376 B: 262); 200 cells FP32 12.7 (27,
// of which the serial step constants took 4), 400 cells FP64 57 (155).  Short grids are bound by
// the chain of passes of the faces at a shock.
#pragma once

#include "pond_kernels.cuh"

namespace pond {

// LPF lanes per face, WARPS warps per CTA, MINB CTAs per SM for the register budget
template <int LPF_, int WARPS_, int MINB_>
struct ChunkVariant {
    static constexpr bool CHUNK = true;
    static constexpr int LPF = LPF_, WARPS = WARPS_, MINB = MINB_, THREADS = 32 * WARPS_;
    static constexpr int CELLS = LPF_ == 1 ? 28 : 32 / LPF_ - 1, STAGED = CELLS + 4;
    static_assert(STAGED <= 32 && (CELLS + 1) * LPF_ <= 32, "a lane per staged cell, LPF per face");
};

// the stored state of a cell
template <typename R>
struct Cell1 {
    R rho, a2, a3, b0, b1, b2;
    typename FrameWords<R>::word u, T;
};

// cell i of the grid, ghosts resolved (mirror images with their odd orders and velocity reversed)
template <typename R>
__device__ __forceinline__ Cell1<R> load_cell1(const Params<1, R> &P, long long i, bool inside)
{
    Cell1<R> c;
    long long idx = i;
    int flip = 0;
    if (!inside) {
        const int side = resolve<1, R>(P, i, 0, &idx, &flip);
        if (side >= 0) {
            const double rho = P.inflow[side][0], T = P.inflow[side][3] / rho;
            c.rho = R(rho);
            c.a2 = c.a3 = c.b1 = c.b2 = R(0);
            c.b0 = R((P.Cv - 0.5) * rho * T);
            fr_store(c.u, P.inflow[side][1]);
            fr_store(c.T, T);
            return c;
        }
    }
    const long long n = P.nx;
    c.rho = P.sf[idx];
    c.a2 = P.sf[n + idx];
    c.a3 = P.sf[2 * n + idx];
    c.b0 = P.sg[idx];
    c.b1 = P.sg[n + idx];
    c.b2 = P.sg[2 * n + idx];
    c.u = P.sfr[idx];
    c.T = P.sfr[n + idx];
    if (flip) {
        c.a3 = -c.a3;
        c.b1 = -c.b1;
        c.u = fr_neg(c.u);
    }
    return c;
}

template <typename R, typename V>
__global__ void __launch_bounds__(V::THREADS, V::MINB)
chunk_step_kernel(const Params<1, R> P)
{
    using W = typename FrameWords<R>::word;
    constexpr int NC = V::CELLS, NW = V::WARPS, LPF = V::LPF;
    __shared__ StagedCell<1, R> tile[NW][V::STAGED];
    __shared__ R faceF[NW][NC + 1][4], faceG[NW][NC + 1][3];
    __shared__ R faceU[NW][NC + 1], faceT[NW][NC + 1];   // face frame: velocity relative to the chunk's reference, T
    // the raw state of the cell that each lane staged, parked across the face solves
    __shared__ R raw[NW][6][32];
    __shared__ W raww[NW][2][32];

    const Clock &K = *P.clock;
    const long long n = P.nx, nf = n + 1;
    if (!(K.dt > 0.0)) {
        // t_end reached: the state moves to the other buffers as it is
        for (long long i = (long long)blockIdx.x * V::THREADS + threadIdx.x; i < nf; i += (long long)gridDim.x * V::THREADS) {
            P.xfr_n[i] = P.xfr[i];
            P.xfr_n[nf + i] = P.xfr[nf + i];
            if (i >= n) continue;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                P.sf_n[k * n + i] = P.sf[k * n + i];
                P.sg_n[k * n + i] = P.sg[k * n + i];
            }
            P.sfr_n[i] = P.sfr[i];
            P.sfr_n[n + i] = P.sfr[n + i];
        }
        return;
    }
    const StepC<R> &KC = step_c<R>(K);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const R cp = KC.cp, ce = KC.ce;
    FaceCfg<R> cfg;
    cfg.h_dn = KC.h_dx;
    cfg.h_dt = R(0);
    cfg.Cv = P.Cv_r; cfg.tol = P.tol_r; cfg.wb = KC.wb; cfg.we = KC.we;
    cfg.limiter = P.limiter; cfg.max_iter = P.max_iter; cfg.fixed_iters = P.fixed_iters;
    unsigned int my_iters = 0, my_faces = 0, my_nonconv = 0, my_fallbacks = 0, my_nonphys = 0;
    R rate = R(0);
    StagedCell<1, R> *wt = tile[warp];
    const int f = lane / LPF;   // this lane's face
    const long long chunks = (n + NC - 1) / NC, stride = (long long)gridDim.x * NW;
    long long ci = (long long)blockIdx.x * NW + warp;
    Cell1<R> c{};
    W fu{}, fT{};
    auto load = [&](long long chunk) {
        const long long c0 = chunk * NC;
        const bool inside = c0 >= 2 && c0 + NC + 2 <= n;
        if (lane < V::STAGED) c = load_cell1<R>(P, c0 - 2 + lane, inside);
        const long long k = min(c0 + f, n);
        fu = P.xfr[k];
        fT = P.xfr[nf + k];
    };
    if (ci < chunks) load(ci);
    for (; ci < chunks; ci += stride) {
        const long long c0 = ci * NC;
        const int nc = int(min((long long)NC, n - c0));
        // reference velocity of the chunk: its first cell's
        W ref;
        if constexpr (sizeof(R) == 4) {
            ref.hi = __shfl_sync(0xffffffffu, c.u.hi, 2);
            ref.lo = __shfl_sync(0xffffffffu, c.u.lo, 2);
        } else {
            ref = __shfl_sync(0xffffffffu, c.u, 2);
        }
        if (lane < V::STAGED) {
            StagedCell<1, R> &o = wt[lane];
            const R T = R(fr_lead(c.T));
            o.A[0] = cp * c.rho + ce * c.rho;
            o.A[1] = R(0);
            o.A[2] = cp * c.a2;
            o.A[3] = cp * c.a3;
            o.B[0] = cp * c.b0 + ce * (P.Cvh_r * c.rho * T);
            o.B[1] = cp * c.b1;
            o.B[2] = cp * c.b2;
            o.du[0] = R(fr_rel(c.u, ref));
            o.T = T;
        }
        raw[warp][0][lane] = c.rho; raw[warp][1][lane] = c.a2; raw[warp][2][lane] = c.a3;
        raw[warp][3][lane] = c.b0; raw[warp][4][lane] = c.b1; raw[warp][5][lane] = c.b2;
        raww[warp][0][lane] = c.u; raww[warp][1][lane] = c.T;
        const W uref = fu;
        const R Tpred = R(fr_lead(fT));
        __syncwarp();
        if (ci + stride < chunks) load(ci + stride);
        // faces c0 .. c0 + nc: face k lies between cells k - 1 and k
        if (f <= nc) {
            const long long k = c0 + f;
            Stencil<1, R> cells;   // LL, L, R, RR at wt[f .. f + 3]
            cells.base = &wt[f + 2];
            cells.sn = 1;
            cells.st = 0;
            const R dref[1] = {R(fr_rel(uref, ref))}, uabs[1] = {R(fr_lead(uref))};
            FaceOut<1, R> o;
            solve_face<1, R, false, 0, true, 0, LPF>(cells, false, dref, uabs, Tpred, cfg, o);
            const bool writer = LPF == 1 || (lane & (LPF - 1)) == 0;
            const bool owned = writer && (f < nc || k == n);
            if (owned) {
                my_iters += o.iters;
                my_faces += 1;
                my_fallbacks += o.fallbacks;
                if (!o.done) ++my_nonconv;
            }
            if (o.have) {
                if (writer) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) faceF[warp][f][q] = o.F[q];
#pragma unroll
                    for (int q = 0; q < 3; ++q) faceG[warp][f][q] = o.G[q];
                    faceU[warp][f] = dref[0] + o.du[0];
                    faceT[warp][f] = o.T;
                }
                if (owned) {
                    P.xfr_n[k] = fr_add(uref, o.du[0]);
                    P.xfr_n[nf + k] = fr_word(o.T);
                }
            } else {
                const R nan = R(__int_as_float(0x7fc00000));
                if (writer) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) faceF[warp][f][q] = nan;
#pragma unroll
                    for (int q = 0; q < 3; ++q) faceG[warp][f][q] = nan;
                    faceU[warp][f] = dref[0];
                    faceT[warp][f] = nan;
                }
                if (owned) {
                    ++my_nonphys;
                    P.xfr_n[k] = uref;
                    fr_store(P.xfr_n[nf + k], double(nan));
                }
            }
        }
        __syncwarp();
        // lane l = 2 .. nc + 1 updates the cell it staged, between faces l - 2 and l - 1
        if (lane >= 2 && lane < nc + 2) {
            const int t = lane - 2;
            const long long i = c0 + t;
            const R rho = vload(&raw[warp][0][lane]), a2 = vload(&raw[warp][1][lane]), a3 = vload(&raw[warp][2][lane]);
            const R b0 = vload(&raw[warp][3][lane]), b1 = vload(&raw[warp][4][lane]), b2 = vload(&raw[warp][5][lane]);
            const W uc = vload_word(&raww[warp][0][lane]), Tc = vload_word(&raww[warp][1][lane]);
            const R Tcr = R(fr_lead(Tc)), duc = wt[lane].du[0], ca = KC.ca, cb = KC.cb;
            const R invTc = w_rcp<R>(Tcr), rsqTc = w_sqrt<R>(invTc), sqTc = Tcr * rsqTc;
            R H[4] = {ca * rho + cb * rho, R(0), ca * a2, ca * a3};
            R G[3] = {ca * b0 + cb * P.Cvh_r * rho * Tcr, ca * b1, ca * b2};
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const R dv[1] = {faceU[warp][t + side] - duc};
                add_face_flux<1, R>(faceF[warp][t + side], faceG[warp][t + side], dv, faceT[warp][t + side], Tcr, invTc, rsqTc, 0,
                                    side ? KC.dt_dx : -KC.dt_dx, sqTc, R(fr_lead(uc)), H, G);
            }
            R Ho[4], Go[3], du[1], dT;
            bool ok = cell_finish<1, R>(H, G, invTc, sqTc, P.Cv_r, Ho, Go, du, dT);
            const W un = fr_add(uc, du[0]), Tn = fr_add(Tc, Tcr * dT);
            const R unr = R(fr_lead(un)), Tnr = R(fr_lead(Tn));
            ok = ok && Tnr > R(0) && isfinite(Tnr);
            if (!ok) {
                ++my_nonphys;
                atomicCAS((unsigned long long *)&P.diag->first_bad, (unsigned long long)-1ll, (unsigned long long)i);
            }
            P.sf_n[i] = Ho[0];
            P.sf_n[n + i] = Ho[2];
            P.sf_n[2 * n + i] = Ho[3];
            P.sg_n[i] = Go[0];
            P.sg_n[n + i] = Go[1];
            P.sg_n[2 * n + i] = Go[2];
            P.sfr_n[i] = un;
            P.sfr_n[n + i] = Tn;
            if (ok) rate = max(rate, cell_rate_r<R>(&unr, Tnr, KC.inv_dx, KC.inv_dy, 1));
        }
        __syncwarp();   // the chunk's shared records are read before the next chunk restages them
    }
    my_iters = warp_sum_count(my_iters);
    my_faces = warp_sum_count(my_faces);
    my_nonconv = warp_sum_count(my_nonconv);
    my_fallbacks = warp_sum_count(my_fallbacks);
    my_nonphys = warp_sum_count(my_nonphys);
    if (lane == 0) {
        using U = unsigned long long;
        if (my_faces) { atomicAdd(&P.diag->face_iters, U(my_iters)); atomicAdd(&P.diag->face_solves, U(my_faces)); }
        if (my_nonconv) { atomicAdd(&P.diag->nonconv, U(my_nonconv)); atomicOr(&P.diag->flags, FLAG_NOT_CONVERGED); }
        if (my_fallbacks) atomicAdd(&P.diag->fallbacks, U(my_fallbacks));
        if (my_nonphys) { atomicAdd(&P.diag->nonphys, U(my_nonphys)); atomicOr(&P.diag->flags, FLAG_NONPHYSICAL); }
    }
    reduce_rate_and_advance(P.clock, double(rate), true);
}

}  // namespace pond
