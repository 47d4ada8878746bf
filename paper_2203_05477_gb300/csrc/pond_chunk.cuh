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
// FP32 steps are bit for bit those of the face and cell kernels (kRefFaces, Map1Written).
//
// Measured (GB300, us a step, before: face and cell kernels): FP32 4 M cells 201 (328), 200 000 cells 15.9
// (26.7), 200 cells 7.6 (12.9, of which the serial step constants took 4); 74% of the issue slots with 16 warps per SM
// (126 registers, no spills), 1240 thread instructions a cell.
// 400 cells FP64 57 (155).  Short grids are bound by the chain of passes of the faces at a shock.
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

// FP32 takes the reference velocity of a face from the first cell of its block of kRefFaces faces (the
// face kernel's tile), so that a face rounds the same in whichever chunk or kernel solves it: a
// shock makes a tube's FP32 result depend on every rounding.  A chunk whose faces lie in two
// blocks stages its cells relative to both.  FP64: the chunk's first cell.
constexpr int kRefFaces = 128;
template <typename R> __host__ __device__ constexpr int chunk_refs() { return sizeof(R) == 4 ? 2 : 1; }

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

// The update of a cell from its two faces (add_face_flux, cell_finish) in FP32 with the contractions
// written out (see Map1Written).  F, G, dv, Tb: the faces' populations, velocity less the cell's, and T.
struct CellUpdate1 {
    float Ho[4], Go[3], du[1], dT;
    bool ok;
    template <typename FACE>
    __device__ __forceinline__ CellUpdate1(const Cell1<float> &c, const StepC<float> &K, float Cv, float T, float un, float invT,
                                           float rsqT, float sqT, FACE &&face)
    {
        // a b + x y, the first product in the fused multiply-add
        auto fuse1 = [](float a, float b, float x, float y) { return fmaf(a, b, __fmul_rn(x, y)); };
        const float cvh = __fadd_rn(Cv, -0.5f), two = __fmul_rn(sqT, 2.f), three = __fmul_rn(sqT, 3.f);
        float H[4], G[3];
        H[0] = fuse1(K.cb, c.rho, K.ca, c.rho);
        H[1] = 0.f;
        G[0] = fuse1(__fmul_rn(__fmul_rn(K.cb, cvh), c.rho), T, K.ca, c.b0);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            float Fc[4], Gc[3], dv, Tb, F[4], Q[3];
            face(side, Fc, Gc, dv, Tb);
            const Map1Written<true> M(w_sqrt<float>(__fmul_rn(Tb, invT)), __fmul_rn(__fadd_rn(Tb, -T), invT), __fmul_rn(dv, rsqT));
            M.f(Fc, F);
            M.g(Gc, Q);
            const float m = side ? -K.dt_dx : K.dt_dx;
            const float v0 = fuse1(un, F[0], sqT, F[1]), v1 = fmaf(sqT, F[0], fuse1(un, F[1], sqT, F[2]));
            const float v2 = fmaf(two, F[1], fuse1(un, F[2], sqT, F[3])), v3 = fuse1(un, F[3], three, F[2]);
            const float w0 = fuse1(un, Q[0], sqT, Q[1]), w1 = fmaf(sqT, Q[0], fuse1(un, Q[1], sqT, Q[2])), w2 = fuse1(un, Q[2], two, Q[1]);
            H[0] = fmaf(m, v0, H[0]);
            H[1] = fmaf(m, v1, H[1]);
            H[2] = side ? fmaf(m, v2, H[2]) : fuse1(K.ca, c.a2, m, v2);
            H[3] = side ? fmaf(m, v3, H[3]) : fuse1(K.ca, c.a3, m, v3);
            G[0] = fmaf(m, w0, G[0]);
            G[1] = side ? fmaf(m, w1, G[1]) : fuse1(K.ca, c.b1, m, w1);
            G[2] = side ? fmaf(m, w2, G[2]) : fuse1(K.ca, c.b2, m, w2);
        }
        const float rsq = __fmul_rn(invT, sqT), rn = H[0];
        du[0] = __fmul_rn(__fmul_rn(sqT, H[1]), w_rcp<float>(rn));
        const float k2 = __fmul_rn(du[0], du[0]);
        dT = w_div<float>(fmaf(-__fmul_rn(__fmul_rn(0.5f, rn), k2), invT, fmaf(-cvh, rn, fuse1(0.5f, H[2], G[0], invT))), __fmul_rn(Cv, rn));
        ok = rn > 0.f && 1.f + dT > 0.f && isfinite(rn) && isfinite(dT);
        const float s2 = w_rcp<float>(__fadd_rn(1.f, dT)), s = w_sqrt<float>(s2);
        const Map1Written<false> M(s, __fmul_rn(-dT, s2), __fmul_rn(-du[0], __fmul_rn(rsq, s)));
        M.f(H, Ho);
        M.g(G, Go);
    }
};

template <typename R, typename V>
__global__ void __launch_bounds__(V::THREADS, V::MINB)
chunk_step_kernel(const Params<1, R> P)
{
    using W = typename FrameWords<R>::word;
    constexpr int NC = V::CELLS, NW = V::WARPS, LPF = V::LPF;
    constexpr int REFS = chunk_refs<R>();
    __shared__ StagedCell<1, R> tile[NW][REFS * V::STAGED];
    __shared__ R faceF[NW][NC + 1][4], faceG[NW][NC + 1][3];
    __shared__ W faceU[NW][NC + 1];   // face frame: velocity, T
    __shared__ R faceT[NW][NC + 1];
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
    W fu{}, fT{}, fref{};   // FP32: lanes 0 and 1 hold the reference velocities
    auto load = [&](long long chunk) {
        const long long c0 = chunk * NC;
        const bool inside = c0 >= 2 && c0 + NC + 2 <= n;
        if (lane < V::STAGED) c = load_cell1<R>(P, c0 - 2 + lane, inside);
        const long long k = min(c0 + f, n);
        fu = P.xfr[k];
        fT = P.xfr[nf + k];
        if (REFS == 2 && lane < 2) cell_velocity<1, R>(P, (c0 / kRefFaces + lane) * kRefFaces, 0, &fref);
    };
    if (ci < chunks) load(ci);
    for (; ci < chunks; ci += stride) {
        const long long c0 = ci * NC;
        const int nc = int(min((long long)NC, n - c0));
        W ref[REFS];
        if constexpr (REFS == 2) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                ref[q].hi = __shfl_sync(0xffffffffu, fref.hi, q);
                ref[q].lo = __shfl_sync(0xffffffffu, fref.lo, q);
            }
        } else {
            ref[0] = __shfl_sync(0xffffffffu, c.u, 2);
        }
        const bool two = REFS == 2 && (c0 + nc) / kRefFaces != c0 / kRefFaces;
        if (lane < V::STAGED) {
            StagedCell<1, R> o;
            o.A[0] = c.rho; o.A[1] = R(0); o.A[2] = c.a2; o.A[3] = c.a3;
            o.B[0] = c.b0; o.B[1] = c.b1; o.B[2] = c.b2;
            finish_bar_plus<1, R>(P, cp, ce, ref, &c.u, R(fr_lead(c.T)), o);
            wt[lane] = o;
            if (two) {
                o.du[0] = R(fr_rel(c.u, ref[REFS - 1]));
                wt[V::STAGED + lane] = o;
            }
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
            const int second = two && k / kRefFaces != c0 / kRefFaces ? 1 : 0;
            cells.base = &wt[second * V::STAGED + f + 2];
            cells.sn = 1;
            cells.st = 0;
            const R dref[1] = {R(fr_rel(uref, second ? ref[REFS - 1] : ref[0]))}, uabs[1] = {R(fr_lead(uref))};
            FaceOut<1, R> o;
            solve_face<1, R, false, 0, true, 0, LPF, sizeof(R) == 4>(cells, false, dref, uabs, Tpred, cfg, o);
            const bool writer = LPF == 1 || (lane & (LPF - 1)) == 0;
            const bool owned = writer && (f < nc || k == n);
            if (owned) {
                my_iters += o.iters;
                my_faces += 1;
                my_fallbacks += o.fallbacks;
                if (!o.done) ++my_nonconv;
            }
            if (o.have) {
                const W un = fr_add(uref, o.du[0]);
                if (writer) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) faceF[warp][f][q] = o.F[q];
#pragma unroll
                    for (int q = 0; q < 3; ++q) faceG[warp][f][q] = o.G[q];
                    faceU[warp][f] = un;
                    faceT[warp][f] = o.T;
                }
                if (owned) {
                    P.xfr_n[k] = un;
                    P.xfr_n[nf + k] = fr_word(o.T);
                }
            } else {
                const R nan = R(__int_as_float(0x7fc00000));
                if (writer) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) faceF[warp][f][q] = nan;
#pragma unroll
                    for (int q = 0; q < 3; ++q) faceG[warp][f][q] = nan;
                    faceU[warp][f] = uref;
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
            Cell1<R> o;
            o.rho = vload(&raw[warp][0][lane]); o.a2 = vload(&raw[warp][1][lane]); o.a3 = vload(&raw[warp][2][lane]);
            o.b0 = vload(&raw[warp][3][lane]); o.b1 = vload(&raw[warp][4][lane]); o.b2 = vload(&raw[warp][5][lane]);
            const W uc = vload_word(&raww[warp][0][lane]), Tc = vload_word(&raww[warp][1][lane]);
            const R Tcr = R(fr_lead(Tc)), Cv = P.Cv_r, ucr = R(fr_lead(uc));
            const R invTc = w_rcp<R>(Tcr), rsqTc = w_sqrt<R>(invTc), sqTc = Tcr * rsqTc;
            R Ho[4], Go[3], du[1], dT;
            bool ok;
            if constexpr (sizeof(R) == 4) {
                const CellUpdate1 q(o, KC, Cv, Tcr, ucr, invTc, rsqTc, sqTc, [&](int side, R *F, R *G, R &dv, R &Tb) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) F[k] = faceF[warp][t + side][k];
#pragma unroll
                    for (int k = 0; k < 3; ++k) G[k] = faceG[warp][t + side][k];
                    dv = R(fr_rel(faceU[warp][t + side], uc));
                    Tb = faceT[warp][t + side];
                });
#pragma unroll
                for (int k = 0; k < 4; ++k) Ho[k] = q.Ho[k];
#pragma unroll
                for (int k = 0; k < 3; ++k) Go[k] = q.Go[k];
                du[0] = q.du[0];
                dT = q.dT;
                ok = q.ok;
            } else {
                const R ca = KC.ca, cb = KC.cb;
                R H[4] = {ca * o.rho + cb * o.rho, R(0), ca * o.a2, ca * o.a3};
                R G[3] = {ca * o.b0 + cb * (Cv - R(0.5)) * o.rho * Tcr, ca * o.b1, ca * o.b2};
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    const R dv[1] = {R(fr_rel(faceU[warp][t + side], uc))};
                    add_face_flux<1, R>(faceF[warp][t + side], faceG[warp][t + side], dv, faceT[warp][t + side], Tcr, invTc, rsqTc, 0,
                                        side ? KC.dt_dx : -KC.dt_dx, sqTc, ucr, H, G);
                }
                ok = cell_finish<1, R>(H, G, invTc, sqTc, Cv, Ho, Go, du, dT);
            }
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
