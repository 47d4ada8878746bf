// pond3.cuh -- the finite-volume step on D3Q64 grids: the tensor product of the D1Q4 rule
// (Table I) in three dimensions, the extension the paper names as future work (Sec. V,
// with the slow-moment count q = 20 of Sec. II.C for D = 3).
//
// The arithmetic is that of the D1Q4/D2Q16 kernels with a third axis.  A population set is
// held through its Hermite coefficients A_rst = sum_i f_i He_r(c_ix) He_s(c_iy) He_t(c_iz)
// (r + s + t <= 3 for f: 20 coefficients; <= 2 for g: 10), and the regularized change of
// frame (Sec. II.C) is the product of three one-dimensional lower-triangular maps.
//
// Data layout (structure of arrays, x fastest, then y):
//   cell state : f coefficients in the cell's own frame without the three (zero) first-order
//                ones (17 planes), g coefficients (10 planes), frame (ux, uy, uz, T) as
//                frame words (FP64, or float-float pairs with FP32 populations);
//   faces      : per axis, the face populations' coefficients in the face frame (20 + 10
//                planes) and that frame (4 words), which also seeds the next step's corrector.
// x-face (i, j, k) lies between cells (i-1, j, k) and (i, j, k), i = 0..nx, and likewise for
// y- and z-faces.
//
// Per step (Sec. III.B.4): face3_kernel (steps 2a-2b for the faces of all three axes), then
// cell3_kernel (step 3 fused with step 1 of the next step and the CFL time step).
#pragma once

#include "pond_kernels.cuh"

namespace pond {

// ------------------------------------------------------------ coefficient packing

// index of A_rst in the packed array: blocks of order n = r + s + t; inside a block the
// pairs (s, t) by j = s + t, then t: 000 | 100 010 001 | 200 110 101 020 011 002 | ...
__host__ __device__ constexpr int h3idx(int r, int s, int t)
{
    return (r + s + t) * (r + s + t + 1) * (r + s + t + 2) / 6 + (s + t) * (s + t + 1) / 2 + t;
}
// (s, t) index once the first axis is collapsed
__host__ __device__ constexpr int h2st(int s, int t) { return (s + t) * (s + t + 1) / 2 + t; }
template <int N>
struct NC3 {
    static constexpr int value = (N + 1) * (N + 2) * (N + 3) / 6;
};
constexpr int kNF3 = NC3<3>::value, kNG3 = NC3<2>::value, kNFS3 = kNF3 - 3;

// orders (r, s, t) of packed index k, in closed form (block n = r + s + t, then j = s + t, then t)
__host__ __device__ constexpr int h3n(int k) { return (k >= 1) + (k >= 4) + (k >= 10); }
__host__ __device__ constexpr int h3rem(int k) { return k - h3n(k) * (h3n(k) + 1) * (h3n(k) + 2) / 6; }
__host__ __device__ constexpr int h3j(int k) { return (h3rem(k) >= 1) + (h3rem(k) >= 3) + (h3rem(k) >= 6); }
__host__ __device__ constexpr int h3t(int k) { return h3rem(k) - h3j(k) * (h3j(k) + 1) / 2; }
__host__ __device__ constexpr int h3s(int k) { return h3j(k) - h3t(k); }
__host__ __device__ constexpr int h3r(int k) { return h3n(k) - h3j(k); }

// stored f plane of coefficient k (-1: a first-order one, zero in the cell's own frame)
__host__ __device__ constexpr int fplane3(int k) { return k == 0 ? 0 : (k <= 3 ? -1 : k - 3); }

// out_rst = sum_{p<=r} X(r,p) sum_{q<=s} Y(s,q) sum_{w<=t} Z(t,w) in_pqw, r + s + t <= N.
// Z1: the first-order inputs are known to be zero (coefficients in the frame of their own
// first moment); their terms are skipped, and so are the intermediates they alone feed
// (B_100 = B_010 = 0 after the z stage, C_100 = 0 after the y stage).
template <int N, typename R, bool Z1 = false>
__device__ __forceinline__ void shift_scale_3d(const R *in, const Map1<R> &X, const Map1<R> &Y, const Map1<R> &Z, R *out)
{
    R B[NC3<N>::value], C[NC3<N>::value];
#pragma unroll
    for (int p = 0; p <= N; ++p)
#pragma unroll
        for (int q = 0; p + q <= N; ++q)
#pragma unroll
            for (int t = 0; p + q + t <= N; ++t) {
                R acc = R(0);
#pragma unroll
                for (int w = 0; w <= t; ++w)
                    if (!(Z1 && p + q + w == 1)) acc += Z.get(t, w) * in[h3idx(p, q, w)];
                B[h3idx(p, q, t)] = acc;
            }
#pragma unroll
    for (int p = 0; p <= N; ++p)
#pragma unroll
        for (int s = 0; p + s <= N; ++s)
#pragma unroll
            for (int t = 0; p + s + t <= N; ++t) {
                R acc = R(0);
#pragma unroll
                for (int q = 0; q <= s; ++q)
                    if (!(Z1 && t == 0 && p + q == 1)) acc += Y.get(s, q) * B[h3idx(p, q, t)];
                C[h3idx(p, s, t)] = acc;
            }
#pragma unroll
    for (int r = 0; r <= N; ++r)
#pragma unroll
        for (int s = 0; r + s <= N; ++s)
#pragma unroll
            for (int t = 0; r + s + t <= N; ++t) {
                R acc = R(0);
#pragma unroll
                for (int p = 0; p <= r; ++p)
                    if (!(Z1 && p == 1 && s == 0 && t == 0)) acc += X.get(r, p) * C[h3idx(p, s, t)];
                out[h3idx(r, s, t)] = acc;
            }
}

// Faces work in face axes (normal, first tangential, second tangential), the tangential
// axes being the other two in increasing order: x-face (x, y, z), y-face (y, x, z),
// z-face (z, x, y).
// lab index of face-axis orders (r, s, t)
__host__ __device__ __forceinline__ int lab_of_face(int dir, int r, int s, int t)
{
    return dir == 0 ? h3idx(r, s, t) : (dir == 1 ? h3idx(s, r, t) : h3idx(s, t, r));
}
// lab index of face-axis coefficient k, per face axis (a warp-uniform constant-bank read)
struct FacePerm {
    signed char k[3][kNF3];
};
__host__ __device__ constexpr FacePerm make_face_perm()
{
    FacePerm P{};
    for (int d = 0; d < 3; ++d)
        for (int r = 0; r <= 3; ++r)
            for (int s = 0; r + s <= 3; ++s)
                for (int t = 0; r + s + t <= 3; ++t)
                    P.k[d][h3idx(r, s, t)] = (signed char)(d == 0 ? h3idx(r, s, t) : (d == 1 ? h3idx(s, r, t) : h3idx(s, t, r)));
    return P;
}
static __constant__ FacePerm kFacePerm = make_face_perm();

// ------------------------------------------------------------------ parameters

template <typename R>
struct Params3 {
    using W = typename FrameWords<R>::word;
    long long nx, ny, nz;
    double dx, dy, dz;
    int bc[6];                        // x-lo, x-hi, y-lo, y-hi, z-lo, z-hi
    double gamma, Cv, tau;
    R Cv_r, Cvh_r, tol_r;             // Cv, Cv - 3/2 and tol in the working precision
    int limiter;
    int max_iter, fixed_iters;
    R *sf;                            // [17][ncell]
    R *sg;                            // [10][ncell]
    W *sfr;                           // [4][ncell]
    R *ff[3], *fg[3];                 // per face axis: [20][nf], [10][nf]
    W *ffr[3];                        // [4][nf]
    Clock *clock;
    Diag *diag;
    // list of the faces that the face kernel leaves to its tail (room for every face)
    TailList *tail;
    unsigned long long *tail_items;
    int tail_at;                      // a warp with at most this many unfinished faces lists them
    int sms;                          // SMs of the device (grid of the tail kernel)
    __host__ __device__ long long ncell() const { return nx * ny * nz; }
    __host__ __device__ long long nf(int a) const
    {
        return a == 0 ? (nx + 1) * ny * nz : (a == 1 ? nx * (ny + 1) * nz : nx * ny * (nz + 1));
    }
    __host__ __device__ long long fidx(int a, long long i, long long j, long long k) const
    {
        return a == 0 ? (k * ny + j) * (nx + 1) + i : (a == 1 ? (k * (ny + 1) + j) * nx + i : (k * ny + j) * nx + i);
    }
};

// Ghost-cell rules along each axis (two layers): wrap-around, copy of the nearest cell, or
// the mirror image across a reflective wall (ghost -k mirrors cell k-1, ghost n-1+k mirrors
// cell n-k).  *flip receives the axes (bit a) across which the cell is a mirror image.
template <typename R>
__device__ __forceinline__ long long resolve3(const Params3<R> &P, long long i, long long j, long long k, int *flip)
{
    long long c[3] = {i, j, k};
    const long long n[3] = {P.nx, P.ny, P.nz};
    int fl = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (c[a] >= 0 && c[a] < n[a]) continue;
        const int b = c[a] < 0 ? P.bc[2 * a] : P.bc[2 * a + 1];   // selects: no run-time indexed parameter
        if (b == BC_REFLECTIVE) {
            c[a] = c[a] < 0 ? -1 - c[a] : 2 * n[a] - 1 - c[a];
            c[a] = clampll(c[a], 0, n[a] - 1);
            fl |= 1 << a;
        } else {
            c[a] = b == BC_PERIODIC ? wrapll(c[a], n[a]) : clampll(c[a], 0, n[a] - 1);
        }
    }
    *flip = fl;
    return (c[2] * P.ny + c[1]) * P.nx + c[0];
}

__host__ __device__ constexpr bool mirror_odd3(int k, int flip)
{
    return (((flip & 1) && (h3r(k) & 1)) != 0) != (((flip & 2) && (h3s(k) & 1)) != 0) != (((flip & 4) && (h3t(k) & 1)) != 0);
}

template <typename R>
struct StagedCell3 {
    R A[kNF3];
    R B[kNG3];
    R du[3];   // frame velocity relative to the tile reference (lab axes)
    R T;
};

template <typename R>
__device__ __forceinline__ void cell_velocity3(const Params3<R> &P, long long i, long long j, long long k,
                                               typename FrameWords<R>::word *u)
{
    int flip = 0;
    const long long idx = resolve3(P, i, j, k, &flip);
    const long long n = P.ncell();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = P.sfr[a * n + idx];
        if (flip & (1 << a)) u[a] = fr_neg(u[a]);
    }
}

// phi-bar-plus (Eq. Fbarplus) of cell (i, j, k), ghosts resolved: cp phi~ + ce phi^eq
template <typename R>
__device__ __forceinline__ void load_cell3(const Params3<R> &P, long long i, long long j, long long k, R cp, R ce,
                                           const typename FrameWords<R>::word *utile, StagedCell3<R> &c)
{
    using W = typename FrameWords<R>::word;
    int flip = 0;
    const long long idx = resolve3(P, i, j, k, &flip);
    const long long n = P.ncell();
#pragma unroll
    for (int q = 0; q < kNF3; ++q) {
        const int pl = fplane3(q);
        const R v = pl < 0 ? R(0) : P.sf[pl * n + idx];
        c.A[q] = mirror_odd3(q, flip) ? -v : v;
    }
#pragma unroll
    for (int q = 0; q < kNG3; ++q) {
        const R v = P.sg[q * n + idx];
        c.B[q] = mirror_odd3(q, flip) ? -v : v;
    }
    W u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = P.sfr[a * n + idx];
        if (flip & (1 << a)) u[a] = fr_neg(u[a]);
        c.du[a] = R(fr_rel(u[a], utile[a]));
    }
    const R T = R(fr_lead(P.sfr[3 * n + idx]));
    const R r = c.A[0];
    c.A[0] = cp * r + ce * r;
#pragma unroll
    for (int q = 1; q < kNF3; ++q) c.A[q] = cp * c.A[q];
    c.B[0] = cp * c.B[0] + ce * (P.Cvh_r * r * T);
#pragma unroll
    for (int q = 1; q < kNG3; ++q) c.B[q] = cp * c.B[q];
    c.T = T;
}

// ---------------------------------------------------------------- cell update

// -scale * H[v_a phi] of one face of axis A added to the cell's moments (H: f, G: g): the
// face populations re-expressed in the cell frame (Eq. fluxEq), times v_a = sqrt(T) c_a + u_a
// by c He_r(c) = He_{r+1}(c) + r He_{r-1}(c) along axis A (He_4 vanishes on the nodes).
template <typename R, int A>
__device__ __forceinline__ void add_face_flux3(const R *Fc, const R *Gc, const R *dv, R Tb, R Tc, R invTc, R rsqTc, R scale,
                                               R sqTc, R un, R *H, R *G)
{
    const R s = sqrt(Tb * invTc), e = (Tb - Tc) * invTc;
    Map1<R> X(s, e, dv[0] * rsqTc), Y(s, e, dv[1] * rsqTc), Z(s, e, dv[2] * rsqTc);
    R Fp[kNF3], Gp[kNG3];
    shift_scale_3d<3, R>(Fc, X, Y, Z, Fp);
    shift_scale_3d<2, R>(Gc, X, Y, Z, Gp);
#pragma unroll
    for (int k = 0; k < kNF3; ++k) {
        const int o[3] = {h3r(k), h3s(k), h3t(k)};
        R v = un * Fp[k];
        if (o[0] + o[1] + o[2] + 1 <= 3)
            v += sqTc * Fp[h3idx(o[0] + (A == 0), o[1] + (A == 1), o[2] + (A == 2))];
        if (o[A] >= 1) v += sqTc * R(o[A]) * Fp[h3idx(o[0] - (A == 0), o[1] - (A == 1), o[2] - (A == 2))];
        H[k] -= scale * v;
    }
#pragma unroll
    for (int k = 0; k < kNG3; ++k) {
        const int o[3] = {h3r(k), h3s(k), h3t(k)};
        R v = un * Gp[k];
        if (o[0] + o[1] + o[2] + 1 <= 2)
            v += sqTc * Gp[h3idx(o[0] + (A == 0), o[1] + (A == 1), o[2] + (A == 2))];
        if (o[A] >= 1) v += sqTc * R(o[A]) * Gp[h3idx(o[0] - (A == 0), o[1] - (A == 1), o[2] - (A == 2))];
        G[k] -= scale * v;
    }
}

template <typename R, int A>
__device__ __forceinline__ void cell_face_flux3(const Params3<R> &P, long long f, R scale, const typename FrameWords<R>::word *uc,
                                                R Tcr, R invTc, R rsqTc, R sqTc, R *H, R *G)
{
    const long long nf = P.nf(A);
    R Fc[kNF3], Gc[kNG3], dv[3];
#pragma unroll
    for (int q = 0; q < kNF3; ++q) Fc[q] = P.ff[A][q * nf + f];
#pragma unroll
    for (int q = 0; q < kNG3; ++q) Gc[q] = P.fg[A][q * nf + f];
#pragma unroll
    for (int a = 0; a < 3; ++a) dv[a] = R(fr_rel(P.ffr[A][a * nf + f], uc[a]));
    const R Tb = R(fr_lead(P.ffr[A][3 * nf + f]));
    add_face_flux3<R, A>(Fc, Gc, dv, Tb, Tcr, invTc, rsqTc, scale, sqTc, R(fr_lead(uc[A])), H, G);
}

template <typename R>
__device__ __forceinline__ double cell_rate3(const R *u, R T, const StepC<R> &KC)
{
    const R c = sqrt(T) * R(kCHi);
    R r = (fabs(u[0]) + c) * KC.inv_dx;
    r = max(r, (fabs(u[1]) + c) * KC.inv_dy);
    r = max(r, (fabs(u[2]) + c) * KC.inv_dz);
    return double(r);
}

// Step 3 of Sec. III.B.4 (Eqs. fluxEq, FinalUpdateDUGKS) through the six faces, fused with
// step 1 of the next step (the new co-moving frame from the conserved moments and the Grad
// projection into it) and the CFL reduction.
template <typename R, int THREADS = 128>
__global__ void __launch_bounds__(THREADS)
cell3_kernel(const Params3<R> P)
{
    const Clock &K = *P.clock;
    if (!(K.dt > 0.0)) return;
    const long long n = P.ncell();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double rate = 0.0;
    using W = typename FrameWords<R>::word;
    const StepC<R> &KC = step_c<R>(K);
    if (c < n) {
        const long long i = c % P.nx, j = (c / P.nx) % P.ny, k = c / (P.nx * P.ny);
        W uc[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) uc[a] = P.sfr[a * n + c];
        const W Tc = P.sfr[3 * n + c];
        const R rho = P.sf[c];
        const R ca = KC.ca, cb = KC.cb, Cv = P.Cv_r;
        const R Tcr = R(fr_lead(Tc));
        const R invTc = R(1) / Tcr, rsqTc = sqrt(invTc), sqTc = Tcr * rsqTc;
        R H[kNF3], G[kNG3];
#pragma unroll
        for (int q = 0; q < kNF3; ++q) {
            const int pl = fplane3(q);
            H[q] = pl < 0 ? R(0) : ca * P.sf[pl * n + c];
        }
        H[0] += cb * rho;
#pragma unroll
        for (int q = 0; q < kNG3; ++q) G[q] = ca * P.sg[q * n + c];
        G[0] += cb * (Cv - R(1.5)) * rho * Tcr;
        const R sx = KC.dt_dx, sy = KC.dt_dy, sz = KC.dt_dz;
        cell_face_flux3<R, 0>(P, P.fidx(0, i, j, k), -sx, uc, Tcr, invTc, rsqTc, sqTc, H, G);
        cell_face_flux3<R, 0>(P, P.fidx(0, i + 1, j, k), sx, uc, Tcr, invTc, rsqTc, sqTc, H, G);
        cell_face_flux3<R, 1>(P, P.fidx(1, i, j, k), -sy, uc, Tcr, invTc, rsqTc, sqTc, H, G);
        cell_face_flux3<R, 1>(P, P.fidx(1, i, j + 1, k), sy, uc, Tcr, invTc, rsqTc, sqTc, H, G);
        cell_face_flux3<R, 2>(P, P.fidx(2, i, j, k), -sz, uc, Tcr, invTc, rsqTc, sqTc, H, G);
        cell_face_flux3<R, 2>(P, P.fidx(2, i, j, k + 1), sz, uc, Tcr, invTc, rsqTc, sqTc, H, G);
        // the new frame from the conserved moments (increments relative to the old frame)
        const R rn = H[0], irn = R(1) / rn;
        R du[3];
        du[0] = sqTc * H[h3idx(1, 0, 0)] * irn;
        du[1] = sqTc * H[h3idx(0, 1, 0)] * irn;
        du[2] = sqTc * H[h3idx(0, 0, 1)] * irn;
        const R k2 = du[0] * du[0] + du[1] * du[1] + du[2] * du[2];
        const R trH = H[h3idx(2, 0, 0)] + H[h3idx(0, 2, 0)] + H[h3idx(0, 0, 2)];
        const R dT = (R(0.5) * trH + G[0] * invTc - (Cv - R(1.5)) * rn - R(0.5) * rn * k2 * invTc) / (Cv * rn);
        bool ok = rn > R(0) && R(1) + dT > R(0) && isfinite(double(rn)) && isfinite(double(dT));
        const R s2 = R(1) / (R(1) + dT);
        const R sc = sqrt(s2), e = -dT * s2, rsqn = rsqTc * sc;
        Map1<R> X(sc, e, -du[0] * rsqn), Y(sc, e, -du[1] * rsqn), Z(sc, e, -du[2] * rsqn);
        R Ho[kNF3], Go[kNG3];
        shift_scale_3d<3, R>(H, X, Y, Z, Ho);
        shift_scale_3d<2, R>(G, X, Y, Z, Go);
        W un[3];
        R unr[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            un[a] = fr_add(uc[a], du[a]);
            unr[a] = R(fr_lead(un[a]));
        }
        const W Tn = fr_add(Tc, Tcr * dT);
        const R Tnr = R(fr_lead(Tn));
        ok = ok && Tnr > R(0) && isfinite(Tnr);
        if (!ok) {
            atomicOr(&P.diag->flags, FLAG_NONPHYSICAL);
            atomicAdd(&P.diag->nonphys, 1ull);
            atomicCAS((unsigned long long *)&P.diag->first_bad, (unsigned long long)-1ll, (unsigned long long)c);
        }
#pragma unroll
        for (int q = 0; q < kNF3; ++q) {
            const int pl = fplane3(q);
            if (pl >= 0) P.sf[pl * n + c] = Ho[q];
        }
#pragma unroll
        for (int q = 0; q < kNG3; ++q) P.sg[q * n + c] = Go[q];
#pragma unroll
        for (int a = 0; a < 3; ++a) P.sfr[a * n + c] = un[a];
        P.sfr[3 * n + c] = Tn;
        rate = ok ? cell_rate3<R>(unr, Tnr, KC) : 0.0;
    }
    reduce_rate_and_advance(P.clock, rate, true);
}

// ------------------------------------------------------- initial condition, read-back

// equilibria of Eqs. (feqPond), (geqPond) in each cell's frame from primitive fields
template <typename R>
__global__ void init_cells3_kernel(const Params3<R> P, const double *rho, const double *ux, const double *uy,
                                   const double *uz, const double *p)
{
    const long long n = P.ncell();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double rate = 0.0;
    if (c < n) {
        const double r = rho[c], T = p[c] / r;
        const double u[3] = {ux[c], uy[c], uz[c]};
        P.sf[c] = R(r);
#pragma unroll
        for (int q = 1; q < kNFS3; ++q) P.sf[q * n + c] = R(0);
        P.sg[c] = R((P.Cv - 1.5) * r * T);
#pragma unroll
        for (int q = 1; q < kNG3; ++q) P.sg[q * n + c] = R(0);
#pragma unroll
        for (int a = 0; a < 3; ++a) fr_store(P.sfr[a * n + c], u[a]);
        fr_store(P.sfr[3 * n + c], T);
        const bool ok = r > 0.0 && T > 0.0 && isfinite(r) && isfinite(T);
        if (!ok) {
            atomicOr(&P.diag->flags, FLAG_NONPHYSICAL);
            atomicAdd(&P.diag->nonphys, 1ull);
            atomicCAS((unsigned long long *)&P.diag->first_bad, (unsigned long long)-1ll, (unsigned long long)c);
        }
        const double cm = sqrt(T) * kCHi;
        rate = ok ? fmax(fmax((fabs(u[0]) + cm) / P.dx, (fabs(u[1]) + cm) / P.dy), (fabs(u[2]) + cm) / P.dz) : 0.0;
    }
    reduce_rate_and_advance(P.clock, rate, false);
}

template <typename R>
__device__ __forceinline__ void cell_conserved3(const Params3<R> &P, long long i, long long j, long long k, double &r,
                                                double *m, double &E)
{
    int flip = 0;
    const long long idx = resolve3(P, i, j, k, &flip);
    const long long n = P.ncell();
    r = double(P.sf[idx]);
    const double T = fr_value(P.sfr[3 * n + idx]);
    double k2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double u = fr_value(P.sfr[a * n + idx]);
        if (flip & (1 << a)) u = -u;
        m[a] = r * u;
        k2 += u * u;
    }
    E = r * (P.Cv * T + 0.5 * k2);
}

// face predictor before the first step: the frame of the pooled moments of the two cells
template <typename R>
__global__ void init_faces3_kernel(const Params3<R> P)
{
    const long long n0 = P.nf(0), n1 = P.nf(1), n2 = P.nf(2);
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n0 + n1 + n2) return;
    const int dir = t < n0 ? 0 : (t < n0 + n1 ? 1 : 2);
    const long long f = t - (dir == 0 ? 0 : (dir == 1 ? n0 : n0 + n1));
    const long long ex = P.nx + (dir == 0), ey = P.ny + (dir == 1);
    const long long i = f % ex, j = (f / ex) % ey, k = f / (ex * ey);
    double ra, ma[3], Ea, rb, mb[3], Eb;
    cell_conserved3<R>(P, i - (dir == 0), j - (dir == 1), k - (dir == 2), ra, ma, Ea);
    cell_conserved3<R>(P, i, j, k, rb, mb, Eb);
    const double r = 0.5 * (ra + rb), E = 0.5 * (Ea + Eb);
    double k2 = 0.0;
    typename FrameWords<R>::word *Frm = P.ffr[dir];
    const long long nf = P.nf(dir);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double m = 0.5 * (ma[a] + mb[a]);
        fr_store(Frm[a * nf + f], m / r);
        k2 += m * m;
    }
    fr_store(Frm[3 * nf + f], (E - 0.5 * k2 / r) / (P.Cv * r));
}

template <typename R>
__global__ void conserved3_kernel(const Params3<R> P, double *rho, double *mx, double *my, double *mz, double *E)
{
    const long long n = P.ncell();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    double r, m[3], e;
    cell_conserved3<R>(P, c % P.nx, (c / P.nx) % P.ny, c / (P.nx * P.ny), r, m, e);
    if (rho) rho[c] = r;
    if (mx) mx[c] = m[0];
    if (my) my[c] = m[1];
    if (mz) mz[c] = m[2];
    if (E) E[c] = e;
}

// stored state as full coefficient arrays [cells][20], [cells][10] and frames [cells][4]
template <typename R>
__global__ void export_state3_kernel(const Params3<R> P, double *cf, double *cg, double *fr)
{
    const long long n = P.ncell();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
#pragma unroll
    for (int q = 0; q < kNF3; ++q) {
        const int pl = fplane3(q);
        cf[c * kNF3 + q] = pl < 0 ? 0.0 : double(P.sf[pl * n + c]);
    }
#pragma unroll
    for (int q = 0; q < kNG3; ++q) cg[c * kNG3 + q] = double(P.sg[q * n + c]);
#pragma unroll
    for (int a = 0; a <= 3; ++a) fr[c * 4 + a] = fr_value(P.sfr[a * n + c]);
}

}  // namespace pond
