// pond_sl2.cuh -- the semi-Lagrangian realization of Sec. III.A on D2Q16 grids.
//
// Four lanes per node, one for each x-node m of the lattice.  A CTA stages its TX x TY nodes and a halo
// of two (raw populations in each node's frame, as Hermite coefficients).  A corrector pass in
// frame lambda re-expresses the 24 nodes around the node in lambda (the regularized transformation,
// Sec. II.C), six by each lane, and leaves them in the node's part of shared memory as differences
// from the node's own coefficients; those enter the moments directly and only the differences are
// interpolated (the same result in exact arithmetic).  Lane m then takes the
// populations (m, n): their departure points share the x offset, so each of the five rows is
// collapsed along x at c_m and interpolated in x once for all n, and the four y-nodes, as even
// and odd parts, evaluate the rows and interpolate them in y.  The limiter of the reading in Sec. III.A
// needs the values at the 2 x 2 nearest nodes besides.  The moments are summed over the four
// lanes.  The converged populations are projected into the frame of their own moments, relaxed by BGK,
// and written to the other state buffer.
//
// Each node is re-expressed once a pass (a thread per node with a scratch of collapsed coefficients
// took 80 transformations for 24 nodes, and evaluated every population at 16 points), and a
// quarter of the pass is serial, which is what a small FP64 grid waits for.
//
// Measured (GB300, us a step; before: the thread per node): 500^2 FP32, two passes a node, 164 (329);
// 100^2 FP64, three passes, 516 (2316); 31 x 51 FP64 260 (2156).  FP32 issues 2000 instructions a warp and pass at
// 61% of the issue slots, with the shared-memory pipe at 63% (1024^2: 63% and 68%): a lane reads 240 words of
// the scratch a pass (320 before the writer formed the even and odd parts along x).  Two CTAs of
// 64 nodes fill the shared memory; one node's scratch is 1.6 KB.  FP64 is bound by its pipe.
#pragma once

#include "pond_sl.cuh"
#include "pond_vec.cuh"

namespace pond {

// Lagrange weights at offsets -1..2 of a point at th in [0, 1]
template <typename R>
__device__ __forceinline__ void sl_weights(R th, R *w)
{
    const R tm = th - R(1), t2 = th - R(2), tp = th + R(1);
    w[0] = -th * tm * t2 * R(1.0 / 6.0);
    w[1] = tp * tm * t2 * R(0.5);
    w[2] = -tp * th * t2 * R(0.5);
    w[3] = tp * th * tm * R(1.0 / 6.0);
}

// four words of shared memory in 16-byte accesses
__device__ __forceinline__ void sl2_load(const float *p, float *v)
{
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void sl2_load(const double *p, double *v)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void sl2_store(float *p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void sl2_store(double *p, double a, double b, double c, double d)
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(a, b);
    reinterpret_cast<double2 *>(p)[1] = make_double2(c, d);
}

// A node's scratch: 25 stencil nodes (the own one zero) of 16 words.  The even and odd parts along x
// are formed by the writer for both |c|, so a lane reads 12 words a stencil node:
//   0 .. 3, 4 .. 7   |c| = c_lo, c_hi: f 00 + 20, f 10 + 30, f 01 + 21, g 00 + 20 (odd: without the sign)
//   8 .. 11          f 11, f 02, f 12, f 03
//   12 .. 15         g 10, g 01, g 11, g 02
// The stride between nodes is an odd number of 16-byte words: eight neighbouring nodes' accesses fall
// in distinct banks (lane = 8 m + node).
template <typename R>
struct Sl2Scratch {
    static constexpr int NODE = 25 * 16 + int(16 / sizeof(R));
};

template <typename R, int TX_, int TY_, int MINB_>
struct Sl2Tile {
    static constexpr int TX = TX_, TY = TY_, MINB = MINB_, THREADS = 4 * TX * TY;
    static constexpr bool LAYERS = TY < 8;   // tile rows past 65 535 along gridDim.z
    static constexpr size_t scratch = size_t(TX) * TY * Sl2Scratch<R>::NODE * sizeof(R);
    static_assert(TX == 8, "a warp takes eight nodes of a row");
};

// a node's coefficients in the frame (dl, Tl)
template <typename R>
__device__ __forceinline__ void sl2_move(const StagedCell<2, R> *cp, const R *dl, R Tl, R invTl, R rsqTl, R *F, R *G)
{
    const StagedCell<2, R> c = fetch<2, R>(cp);   // 16-byte loads of the staged record
    const Move2<R> M(c.T, c.du[0], c.du[1], Tl, invTl, rsqTl, dl[0], dl[1]);
    M.f(c.A[0], c.A[3], c.A[4], c.A[5], c.A[6], c.A[7], c.A[8], c.A[9], F);   // staged f: zero first order
    M.g(c.B[0], c.B[1], c.B[2], c.B[3], c.B[4], c.B[5], G);
}

// f (orders 0..3 along y) and g (0..2) of a row at the four y-nodes
template <typename R>
__device__ __forceinline__ void sl2_nodes(const R *C, R *f, R *g)
{
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
        const int np = hi ? 3 : 2, nm = hi ? 0 : 1;
        const R c = R(node_c(np)), h2 = R(hen(2, np)), h3 = R(hen(3, np));
        const R E = vfma(h2, C[2], C[0]), O = vfma(h3, C[3], c * C[1]), Eg = vfma(h2, C[6], C[4]);
        f[np] = E + O;
        f[nm] = E - O;
        g[np] = vfma(c, C[5], Eg);
        g[nm] = vfma(-c, C[5], Eg);
    }
}

template <typename R, typename V>
__global__ void __launch_bounds__(V::THREADS, V::MINB)
sl2_kernel(const Params<2, R> P)
{
    using W = typename FrameWords<R>::word;
    constexpr int TX = V::TX, TY = V::TY, BX = TX + 4, BY = TY + 4;
    constexpr int NFC = NCoef<2, 3>::value, NGC = NCoef<2, 2>::value, NODE = Sl2Scratch<R>::NODE;
    __shared__ StagedCell<2, R> tile[BX * BY];
    __shared__ W utile[2];
    extern __shared__ __align__(16) unsigned char sl2_dyn[];
    const Clock &K = *P.clock;
    if (!(K.dt > 0.0)) return hold_state<2, R>(P, P.xf, P.xg, P.xfr);
    const StepC<R> &KC = step_c<R>(K);
    const long long n = P.ncell();
    // gridDim.y ends at 65 535 tile rows; FP64 tiles, of two nodes a row, go on along z, a row past the grid updating
    // nothing (in FP32, whose tiles are 8 high, the two more indices would spill: 500^2 163 -> 173 us a step)
    const long long i0 = (long long)blockIdx.x * TX;
    const long long j0 = (V::LAYERS ? (long long)blockIdx.z * gridDim.y + blockIdx.y : (long long)blockIdx.y) * TY;
    W ut[2];   // every thread reads it (the same words), so the staging needs no barrier before it
    cell_velocity<2, R>(P, i0, j0, ut);
    if (threadIdx.x < 2) utile[threadIdx.x] = threadIdx.x ? ut[1] : ut[0];
    for (int t = threadIdx.x; t < BX * BY; t += V::THREADS)
        load_cell_bar_plus<2, R>(P, i0 - 2 + t % BX, j0 - 2 + t / BX, R(1), R(0), ut, tile[t]);

    const int m = (threadIdx.x & 31) >> 3, tx = threadIdx.x & 7, ty = threadIdx.x >> 5;
    const long long i = i0 + tx, j = j0 + ty, c = j * P.nx + i;
    R *const node = reinterpret_cast<R *>(sl2_dyn) + (ty * TX + tx) * NODE;
    sl2_store(node + 12 * 16 + 4 * m, R(0), R(0), R(0), R(0));
    __syncthreads();
    unsigned long long my_iters = 0, my_nonconv = 0, my_fallbacks = 0, my_nonphys = 0;
    const bool active = i < P.nx && j < P.ny;
    auto cell = [&](int r, int col) -> const StagedCell<2, R> * { return &tile[(ty + r) * BX + tx + col]; };
    const R dt_dx = KC.dt_dx, dt_dy = KC.dt_dy;
    const R Cv = P.Cv_r, tolR = P.tol_r;
    const R uref[2] = {R(fr_lead(utile[0])), R(fr_lead(utile[1]))};
    const NodeTab<R> &tab = node_tab<R>();
    const R cm = tab.c[m], sgn = m >= 2 ? R(1) : R(-1);
    const int hi_m = m == 0 || m == 3 ? 4 : 0;
    R dl[2] = {cell(2, 2)->du[0], cell(2, 2)->du[1]}, Tl = cell(2, 2)->T;   // the node's own frame
    R keep_dl[2] = {dl[0], dl[1]}, keep_T = Tl, out_du[2] = {R(0), R(0)}, out_T = R(0), out_rho = R(0);
    R Phi[NFC], Psi[NGC];
    bool have = false, done = false, restarted = false, last_valid = false;
    int iters = 0, fallbacks = 0;
    // every lane of the warp takes part
    auto pass = [&](const R *dlp, R Tlp) {
        const R invTl = R(1) / Tlp, rsqTl = sqrt(invTl), sqTl = Tlp * rsqTl;
        sl2_move<R>(cell(2, 2), dlp, Tlp, invTl, rsqTl, Phi, Psi);
        __syncwarp();   // the scratch of the last pass has been read
#pragma unroll 3   // three nodes' loads and square roots in flight
        for (int u = 0; u < 6; ++u) {
            const int q = 4 * u + m, p = q + (q >= 12 ? 1 : 0), row = p / 5, col = p - 5 * row;
            R F[NFC], G[NGC];
            sl2_move<R>(cell(row, col), dlp, Tlp, invTl, rsqTl, F, G);
#pragma unroll
            for (int k = 0; k < NFC; ++k) F[k] -= Phi[k];
#pragma unroll
            for (int k = 0; k < NGC; ++k) G[k] -= Psi[k];
            R *o = node + p * 16;
#pragma unroll
            for (int hi = 0; hi < 2; ++hi) {
                const int np = hi ? 3 : 2;
                const R cc = R(node_c(np)), h2 = R(hen(2, np)), h3 = R(hen(3, np));
                sl2_store(o + 4 * hi, vfma(h2, F[3], F[0]), vfma(h3, F[6], cc * F[1]), vfma(h2, F[7], F[2]), vfma(h2, G[3], G[0]));
            }
            sl2_store(o + 8, F[4], F[5], F[8], F[9]);
            sl2_store(o + 12, G[1], G[2], G[4], G[5]);
        }
        __syncwarp();
        // departure points: distances in cells along x (this lane's c_m) and y
        const R dx = (sqTl * cm + uref[0] + dlp[0]) * dt_dx;
        const bool rx = dx > R(0);
        const R thx = rx ? R(1) - dx : -dx;
        R wx[4];
        sl_weights<R>(thx, wx);
        const R *const from = node + (rx ? 0 : 16), *const from_c = from + hi_m;
        // a row's differences collapsed along x at c_m: interpolated in x (X) and at the two
        // nearest nodes (C1, C2)
        auto row_of = [&](int row, R *X, R *C1, R *C2) {
#pragma unroll
            for (int s = 0; s < 7; ++s) X[s] = R(0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                R a[4], b[4], g[4], C[7];
                sl2_load(from_c + (row * 5 + k) * 16, a);
                sl2_load(from + (row * 5 + k) * 16 + 8, b);
                sl2_load(from + (row * 5 + k) * 16 + 12, g);
                C[0] = vfma(sgn, a[1], a[0]);
                C[1] = vfma(cm, b[0], a[2]);
                C[2] = vfma(cm, b[2], b[1]);
                C[3] = b[3];
                C[4] = vfma(cm, g[0], a[3]);
                C[5] = vfma(cm, g[2], g[1]);
                C[6] = g[3];
#pragma unroll
                for (int s = 0; s < 7; ++s) {
                    X[s] = vfma(wx[k], C[s], X[s]);
                    if (k == 1) C1[s] = C[s];
                    if (k == 2) C2[s] = C[s];
                }
            }
        };
        // The y offsets.  Departing downwards (dy > 0) a population uses rows 0 .. 3, else 1 .. 4: every one
        // uses rows 1 .. 3 and one of rows 0 and 4; the nearest rows are 2 and one of 1 and 3.
        R wE[4], w1[4], w2[4], w3[4], thy[4];
        bool ry[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const R dy = (sqTl * R(node_c(k)) + uref[1] + dlp[1]) * dt_dy;
            ry[k] = dy > R(0);
            thy[k] = ry[k] ? R(1) - dy : -dy;
            R w[4];
            sl_weights<R>(thy[k], w);
            wE[k] = ry[k] ? w[0] : w[3];
            w1[k] = ry[k] ? w[1] : w[0];
            w2[k] = ry[k] ? w[2] : w[1];
            w3[k] = ry[k] ? w[3] : w[2];
        }
        R pf[4], pg[4], f1[4], g1[4], f2[4], g2[4], X[7], C1[7], C2[7];
        row_of(0, X, C1, C2);
        sl2_nodes<R>(X, pf, pg);
        row_of(4, X, C1, C2);
        sl2_nodes<R>(X, f1, g1);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            pf[k] = wE[k] * (ry[k] ? pf[k] : f1[k]);
            pg[k] = wE[k] * (ry[k] ? pg[k] : g1[k]);
        }
        // the nearest nodes of rows 1 and 3 (af, ag at the left one, bf, bg at the right one)
        R af[4], ag[4], bf[4], bg[4];
        row_of(1, X, C1, C2);
        sl2_nodes<R>(C1, af, ag);
        sl2_nodes<R>(C2, bf, bg);
        sl2_nodes<R>(X, f1, g1);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            pf[k] = vfma(w1[k], f1[k], pf[k]);
            pg[k] = vfma(w1[k], g1[k], pg[k]);
        }
        row_of(3, X, C1, C2);
        sl2_nodes<R>(C1, f1, g1);
        sl2_nodes<R>(C2, f2, g2);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            af[k] = ry[k] ? af[k] : f1[k];
            ag[k] = ry[k] ? ag[k] : g1[k];
            bf[k] = ry[k] ? bf[k] : f2[k];
            bg[k] = ry[k] ? bg[k] : g2[k];
        }
        sl2_nodes<R>(X, f1, g1);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            pf[k] = vfma(w3[k], f1[k], pf[k]);
            pg[k] = vfma(w3[k], g1[k], pg[k]);
        }
        row_of(2, X, C1, C2);
        sl2_nodes<R>(X, f1, g1);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            pf[k] = vfma(w2[k], f1[k], pf[k]);
            pg[k] = vfma(w2[k], g1[k], pg[k]);
        }
        sl2_nodes<R>(C1, f1, g1);
        sl2_nodes<R>(C2, f2, g2);
        // bicubic, or the bilinear one of the 2 x 2 nearest values when it leaves their range
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const R wa = ry[k] ? R(1) - thy[k] : thy[k], wb = ry[k] ? thy[k] : R(1) - thy[k];
            auto limited = [&](R p, R a, R b, R d, R e) {
                const R lo = min(min(a, b), min(d, e)), hi = max(max(a, b), max(d, e));
                const R bi = wa * ((R(1) - thx) * a + thx * b) + wb * ((R(1) - thx) * d + thx * e);
                return p < lo || p > hi ? bi : p;
            };
            pf[k] = limited(pf[k], af[k], bf[k], f1[k], f2[k]);
            pg[k] = limited(pg[k], ag[k], bg[k], g1[k], g2[k]);
        }
        // Moments along y, then of all lanes' c_m.  Each lane stops by its own copy of them and moves its
        // stencil nodes into its own frame, so the copies must agree to the last bit: the product is rounded
        // before the exchange (contracted into the sum, each lane would round the other one's).
        R S[4] = {R(0), R(0), R(0), R(0)}, SG[3] = {R(0), R(0), R(0)};
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {
            const int np = hi ? 3 : 2, nm = hi ? 0 : 1;
            const R s = pf[np] + pf[nm], d = pf[np] - pf[nm], sg = pg[np] + pg[nm], dg = pg[np] - pg[nm];
            const R v0 = R(node_w(np)), v1 = R(node_w(np) * he(1, np)), v2 = R(node_w(np) * he(2, np)), v3 = R(node_w(np) * he(3, np));
            S[0] = vfma(v0, s, S[0]); S[1] = vfma(v1, d, S[1]); S[2] = vfma(v2, s, S[2]); S[3] = vfma(v3, d, S[3]);
            SG[0] = vfma(v0, sg, SG[0]); SG[1] = vfma(v1, dg, SG[1]); SG[2] = vfma(v2, sg, SG[2]);
        }
        auto over_lanes = [&](R a, R b) {
            R v = vmul_rn(a, b);
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            return v + __shfl_xor_sync(0xffffffffu, v, 16);
        };
#pragma unroll
        for (int r = 0; r <= 3; ++r) {
            const R w = tab.whe[m][r];
#pragma unroll
            for (int s = 0; r + s <= 3; ++s) Phi[hidx(r, s)] += over_lanes(w, S[s]);
#pragma unroll
            for (int s = 0; r + s <= 2; ++s) Psi[hidx(r, s)] += over_lanes(w, SG[s]);
        }
    };
    bool running = active;
    for (int k = 0; k < P.max_iter && __any_sync(0xffffffffu, running); ++k) {
        // a node that has stopped goes along in its last valid pass's frame, which gives
        // the same moments again
        R fdl[2] = {running ? dl[0] : keep_dl[0], running ? dl[1] : keep_dl[1]};
        pass(fdl, running ? Tl : keep_T);
        if (!running) continue;
        R rho1, du[2], T1;
        const bool ok = pass_frame<2, R>(Phi, Psi, Tl, Cv, rho1, du, T1);
        iters = k + 1;
        if (!ok) {
            ++fallbacks;
            last_valid = false;
            running = !restarted;
            if (!restarted) {
                // restart once from the frame of the pooled conserved moments of the stencil
                restarted = true;
                R r = R(0), mo[2] = {R(0), R(0)}, e = R(0);
#pragma unroll 1
                for (int q = 0; q < 25; ++q) {
                    const StagedCell<2, R> *sc = cell(q / 5, q % 5);
                    const R rc = sc->A[0];
                    r += rc;
                    mo[0] += rc * sc->du[0];
                    mo[1] += rc * sc->du[1];
                    e += rc * (Cv * sc->T + R(0.5) * (sc->du[0] * sc->du[0] + sc->du[1] * sc->du[1]));
                }
                r *= R(1.0 / 25.0); mo[0] *= R(1.0 / 25.0); mo[1] *= R(1.0 / 25.0); e *= R(1.0 / 25.0);
                dl[0] = mo[0] / r;
                dl[1] = mo[1] / r;
                Tl = (e - R(0.5) * (mo[0] * mo[0] + mo[1] * mo[1]) / r) / (Cv * r);
            }
            continue;
        }
        have = true;
        last_valid = true;
        keep_dl[0] = dl[0]; keep_dl[1] = dl[1]; keep_T = Tl;
        out_du[0] = du[0]; out_du[1] = du[1]; out_T = T1; out_rho = rho1;
        if (P.fixed_iters > 0) done = iters >= P.fixed_iters;
        else done = fabs(T1 - Tl) <= tolR * Tl && fabs(du[0]) <= tolR * sqrt(Tl) && fabs(du[1]) <= tolR * sqrt(Tl);
        running = !done;
        dl[0] += du[0];
        dl[1] += du[1];
        Tl = T1;
    }
    // a last pass that defined no frame: recompute the last valid one
    if (__any_sync(0xffffffffu, have && !last_valid)) pass(keep_dl, keep_T);
    double rate = 0.0;
    if (active && m == 0) {   // the node's first lane has the rest
        my_iters = iters;
        my_nonconv = done ? 0 : 1;
        my_fallbacks = fallbacks;
        W un[2] = {utile[0], utile[1]}, Tn;
        R A[NFC], B[NGC];
        bool ok = have;
        if (have) {
            // the pre-collision populations in the frame of their own moments, then BGK
            const R invT = R(1) / out_T;
            Move2<R> M(keep_T, R(0), R(0), out_T, invT, sqrt(invT), out_du[0], out_du[1]);
            M.s = sqrt(keep_T * invT);
            M.s3 = M.s2 * M.s;
            M.f_full(Phi, A);
            M.g(Psi[0], Psi[1], Psi[2], Psi[3], Psi[4], Psi[5], B);
            const R twob = KC.cb;  // 2 beta = 2 dt / (2 tau + dt)
            const R keep = R(1) - twob;
#pragma unroll
            for (int k = 0; k < NFC; ++k) A[k] = keep * A[k];
#pragma unroll
            for (int k = 0; k < NGC; ++k) B[k] = keep * B[k];
            A[0] += twob * out_rho;
            B[0] += twob * P.Cvh_r * out_rho * out_T;
#pragma unroll
            for (int a = 0; a < 2; ++a) un[a] = fr_add(utile[a], keep_dl[a] + out_du[a]);
            Tn = fr_word(out_T);
            ok = out_rho > R(0) && out_T > R(0) && isfinite(out_rho) && isfinite(out_T);
        }
        if (!ok) {
            ++my_nonphys;
            const R nan = R(__int_as_float(0x7fc00000));
#pragma unroll
            for (int k = 0; k < NFC; ++k) A[k] = nan;
#pragma unroll
            for (int k = 0; k < NGC; ++k) B[k] = nan;
            Tn = fr_word(nan);
            atomicCAS((unsigned long long *)&P.diag->first_bad, (unsigned long long)-1ll, (unsigned long long)c);
        }
        // the new state goes to the other buffer (held in the face planes, plane stride n)
#pragma unroll
        for (int k = 0; k < NFC; ++k) {
            const int pl = fplane<2>(k);
            if (pl >= 0) P.xf[pl * n + c] = A[k];
        }
#pragma unroll
        for (int k = 0; k < NGC; ++k) P.xg[k * n + c] = B[k];
        P.xfr[c] = un[0];
        P.xfr[n + c] = un[1];
        P.xfr[2 * n + c] = Tn;
        if (ok) {
            const R unr[2] = {R(fr_lead(un[0])), R(fr_lead(un[1]))};
            rate = cell_rate<R>(unr, out_T, KC.inv_dx, KC.inv_dy, 2);
        }
    }
    sl_diag_and_advance<R>(P.diag, P.clock, active && m == 0, my_iters, my_nonconv, my_fallbacks, my_nonphys, rate);
}

}  // namespace pond
