// pond_face3.cuh -- the face predictor-corrector of Sec. III.B.3 on D3Q64 grids.
//
// Arithmetic bounds this kernel (64 populations of f and g, three limited slopes each: about
// 9000 operations a face and pass), as in two dimensions (pond_face2.cuh), and it is laid out the
// same way for the fewest of them:
//   - The normal nodes are taken by their upwind side; a side's nodes share the upwind cell and
//     its six neighbours, so a pass changes the frame of 18 cells (node by node it was 28),
//     each in shift form (Move3: 90 operations against about 230 for the maps and their products).
//   - Slopes come from differences formed once in Hermite space.  The three directions
//     (normal, first and second tangential) are three sweeps of the same rolled code; a sweep
//     keeps its two differences in a per-thread scratch in shared memory, collapses them along the
//     normal at each node of the side, then along the first tangent, and evaluates them at
//     the second tangent's nodes in pairs +-c.  The upwind population is never evaluated: its
//     moments over the tangential nodes are its own collapsed coefficients.
//   - f rides in lane x and g in lane y of packed FP32x2 instructions for the orders both have,
//     where the multiplier is a node constant; the changes of frame are scalar (a packed
//     multiply-add with three different register pairs costs more than two scalar ones).
//   - Nearly every face converges in its first pass, but those at shocks take up to max_iter.  A warp
//     goes on with passes only while more than tail_at (tail3_faces) of its faces need it; the others go to a
//     list in device memory that a second kernel works off, a warp per face, two populations per
//     lane, spread over the whole chip (face3_tail_kernel): such a face is a chain of up to 15
//     passes, and the few tiles at a shock hold most of them.
//
// Reciprocals, square roots and quotients are the IEEE ones in FP32 too: the hardware's approximations gain 3.5%
// (64^3 0.71 ms) and cost accuracy, over 30 explosions and smooth flows an error against 64 bits 1.01 times that of the
// node-by-node kernel, where it is 0.93 times with these.
//
// Measured (GB300, ms a step's faces, before: the node-by-node kernel this one replaces): FP32 explosion
// 64^3 0.74 (1.76), FP64 explosion 25 x 23 x 21 2.2 (15.3).  FP32 issues 61% of the slots with 12 warps
// per SM (167 registers, no spills; the tail 51 to 56%), the rest are dependent-instruction waits and the barrier;
// FP64 is bound by its pipe (57% busy in the first pass, 65% in the tail).
#pragma once

#include "pond3.cuh"
#include "pond_vec.cuh"
#include "pond_face2.cuh"

namespace pond {

// ------------------------------------------------------------ staged cells

// A staged cell: f 000 and 111, g 000, T, then per lab axis a (others b < c) nine words: f 2a, f 3a,
// g 1a, g 2a, u_a, f 2a1b, f 2a1c, f 1b1c, g 1b1c.  A face reads the axes' groups in face order
// (normal, first, second tangent).  31 words: neighbouring threads' cells fall in distinct banks.
constexpr int kCell3 = 31;
template <typename R>
struct FaceAxes3 {
    int n, t1, t2;   // word offsets of the three axes' groups
    int w1, w2;      // 1 where the normal comes second among the other axes of t1 (t2)
    __device__ __forceinline__ explicit FaceAxes3(int dir)
        : n(4 + 9 * dir), t1(4 + 9 * (dir == 0 ? 1 : 0)), t2(4 + 9 * (dir == 2 ? 1 : 2)), w1(dir == 2 ? 1 : 0), w2(dir == 0 ? 0 : 1)
    {
    }
};
template <typename R>
__device__ __forceinline__ void store_cell3(const Params3<R> &P, long long i, long long j, long long k, R cp, R ce,
                                            const typename FrameWords<R>::word *ut, R *o)
{
    StagedCell3<R> c;
    load_cell3<R>(P, i, j, k, cp, ce, ut, c);
    o[0] = c.A[0];
    o[1] = c.A[h3idx(1, 1, 1)];
    o[2] = c.B[0];
    o[3] = c.T;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        R *g = o + 4 + 9 * a;
        const int b = a == 0 ? 1 : 0, d = a == 2 ? 1 : 2;
        auto h = [&](int na, int nb, int nd) {
            int r[3] = {0, 0, 0};
            r[a] = na;
            r[b] = nb;
            r[d] = nd;
            return h3idx(r[0], r[1], r[2]);
        };
        g[0] = c.A[h(2, 0, 0)];
        g[1] = c.A[h(3, 0, 0)];
        g[2] = c.B[h(1, 0, 0)];
        g[3] = c.B[h(2, 0, 0)];
        g[4] = c.du[a];
        g[5] = c.A[h(2, 1, 0)];
        g[6] = c.A[h(2, 0, 1)];
        g[7] = c.A[h(0, 1, 1)];
        g[8] = c.B[h(0, 1, 1)];
    }
}

// the change of frame in shift form (pond_vec.cuh), three axes
template <typename R>
struct Move3 {
    R s, e, d[3], s2, s3;
    __device__ __forceinline__ Move3(R Tc, const R *u, R Tl, R invTl, R rsqTl, const R *l)
    {
        s = sqrt(Tc * invTl);
        e = (Tc - Tl) * invTl;
#pragma unroll
        for (int a = 0; a < 3; ++a) d[a] = (u[a] - l[a]) * rsqTl;
        s2 = e + R(1);
        s3 = s2 * s;
    }
    // first order zero: F[20] in h3idx order from A000, A2 and A3 per axis, A11 per excluded axis,
    // A21[a][b] (twice a, once b) and A111
    __device__ __forceinline__ void f(R A0, const R *A2, const R *A3, const R *A11, const R (*A21)[3], R A111, R *F) const
    {
        R F1[3], q[3], F2[3], a11[3], F11[3];
        const R e0 = e * A0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            F1[a] = d[a] * A0;
            q[a] = vfma(s2, A2[a], e0);
            F2[a] = vfma(d[a], F1[a], q[a]);
            a11[a] = s2 * A11[a];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) F11[a] = vfma(d[(a + 1) % 3], F1[(a + 2) % 3], a11[a]);
        put(A0, F1, F2, F11, F);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            F[h3idx(a == 0 ? 3 : 0, a == 1 ? 3 : 0, a == 2 ? 3 : 0)] = vfma(s3, A3[a], d[a] * vfma(R(2), q[a], F2[a]));
#pragma unroll
            for (int b = 0; b < 3; ++b)
                if (b != a)
                    F[i21(a, b)] = vfma(s3, A21[a][b], vfma(d[a] + d[a], a11[3 - a - b], d[b] * F2[a]));
        }
        F[h3idx(1, 1, 1)] = vfma(s3, A111, vfma(d[2], a11[2], vfma(d[1], a11[1], d[0] * F11[0])));
    }
    // the same for coefficients with a first order, in h3idx order
    __device__ __forceinline__ void f_full(const R *A, R *F) const
    {
        R F1[3], q[3], F2[3], a11[3], F11[3], a1[3], ex[3];
        const R e0 = e * A[0];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            a1[a] = s * A[1 + a];
            F1[a] = vfma(d[a], A[0], a1[a]);
            q[a] = vfma(s2, A[i2(a)], e0);
            F2[a] = vfma(d[a], F1[a] + a1[a], q[a]);
            a11[a] = s2 * A[i11(a)];
            ex[a] = vfma(d[a], d[a], e);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int b = (a + 1) % 3, c = (a + 2) % 3;
            F11[a] = vfma(d[b], F1[c], vfma(d[c], a1[b], a11[a]));
        }
        put(A[0], F1, F2, F11, F);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int k3 = h3idx(a == 0 ? 3 : 0, a == 1 ? 3 : 0, a == 2 ? 3 : 0);
            F[k3] = vfma(s3, A[k3], vfma(R(3) * e, a1[a], d[a] * vfma(d[a], a1[a], vfma(R(2), q[a], F2[a]))));
#pragma unroll
            for (int b = 0; b < 3; ++b)
                if (b != a)
                    F[i21(a, b)] = vfma(s3, A[i21(a, b)],
                                        vfma(d[a] + d[a], a11[3 - a - b], vfma(ex[a], a1[b], d[b] * F2[a])));
        }
        F[h3idx(1, 1, 1)] = vfma(s3, A[h3idx(1, 1, 1)], vfma(d[2], a11[2], vfma(d[1], vfma(d[2], a1[0], a11[1]), d[0] * F11[0])));
    }
    // G[10] from B000, B1 and B2 per axis, B11 per excluded axis
    __device__ __forceinline__ void g(R B0, const R *B1, const R *B2, const R *B11, R *G) const
    {
        R b1[3], G1[3], G2[3], G11[3];
        const R e0 = e * B0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            b1[a] = s * B1[a];
            G1[a] = vfma(d[a], B0, b1[a]);
            G2[a] = vfma(d[a], G1[a] + b1[a], vfma(s2, B2[a], e0));
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int b = (a + 1) % 3, c = (a + 2) % 3;
            G11[a] = vfma(s2, B11[a], vfma(d[c], b1[b], d[b] * G1[c]));
        }
        put(B0, G1, G2, G11, G);
    }
    __host__ __device__ static constexpr int i2(int a) { return h3idx(a == 0 ? 2 : 0, a == 1 ? 2 : 0, a == 2 ? 2 : 0); }
    __host__ __device__ static constexpr int i11(int a) { return h3idx(a == 0 ? 0 : 1, a == 1 ? 0 : 1, a == 2 ? 0 : 1); }   // a excluded
    __host__ __device__ static constexpr int i21(int a, int b)
    {
        return h3idx(a == 0 ? 2 : (b == 0 ? 1 : 0), a == 1 ? 2 : (b == 1 ? 1 : 0), a == 2 ? 2 : (b == 2 ? 1 : 0));
    }
    __device__ __forceinline__ static void put(R A0, const R *F1, const R *F2, const R *F11, R *F)
    {
        F[0] = A0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            F[1 + a] = F1[a];
            F[i2(a)] = F2[a];
            F[i11(a)] = F11[a];
        }
    }
};

// a staged cell in the pass frame, face axes
template <typename R>
__device__ __forceinline__ void move_cell3(const R *c, const FaceAxes3<R> &ax, R Tl, R invTl, R rsqTl, const R *l, R *F, R *G)
{
    const R *cn = c + ax.n, *c1 = c + ax.t1, *c2 = c + ax.t2;
    const R u[3] = {cn[4], c1[4], c2[4]};
    const Move3<R> M(c[3], u, Tl, invTl, rsqTl, l);
    const R A2[3] = {cn[0], c1[0], c2[0]}, A3[3] = {cn[1], c1[1], c2[1]}, A11[3] = {cn[7], c1[7], c2[7]};
    const R A21[3][3] = {{R(0), cn[5], cn[6]}, {c1[5 + ax.w1], R(0), c1[6 - ax.w1]}, {c2[5 + ax.w2], c2[6 - ax.w2], R(0)}};
    M.f(c[0], A2, A3, A11, A21, c[1], F);
    const R B1[3] = {cn[2], c1[2], c2[2]}, B2[3] = {cn[3], c1[3], c2[3]}, B11[3] = {cn[8], c1[8], c2[8]};
    M.g(c[2], B1, B2, B11, G);
}

// Per-thread scratch of NT threads in shared memory, slot-major in 16-byte slots; volatile, so
// that nothing kept here stays in registers too
template <typename R, int NT>
struct Scratch3 {
    static constexpr int PER = 16 / int(sizeof(R));
    unsigned int addr;
    __device__ __forceinline__ void put(int slot, const R *x) const
    {
        union { R r[PER]; float4 f; } u;
#pragma unroll
        for (int k = 0; k < PER; ++k) u.r[k] = x[k];
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr + slot * (NT * 16)), "f"(u.f.x), "f"(u.f.y),
                     "f"(u.f.z), "f"(u.f.w) : "memory");
    }
    __device__ __forceinline__ void get(int slot, R *x) const
    {
        union { R r[PER]; float4 f; } u;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(u.f.x), "=f"(u.f.y), "=f"(u.f.z), "=f"(u.f.w)
                     : "r"(addr + slot * (NT * 16)) : "memory");
#pragma unroll
        for (int k = 0; k < PER; ++k) x[k] = u.r[k];
    }
};
// words of the scratch: two differences of 30 coefficients (f and g alternating for the orders
// both have, then f's third order)
constexpr int kScr3 = 60;

// normal collapse at node constants h[1..3]: the (f, g) pairs of orders s + t <= 2 and f's third
// order, from the 30 words of a difference (f_k, g_k for k < 10, then f_10 .. f_19)
template <typename R>
__device__ __forceinline__ void collapse3(const R *w, R h1, R h2, R h3, FG<R> *Q, R *T)
{
    auto p = [&](int k) { return fg(w[2 * k], w[2 * k + 1]); };
    auto f3 = [&](int r, int s, int t) { return w[10 + h3idx(r, s, t)]; };
    Q[0] = fgfma(p(h3idx(2, 0, 0)), h2, fgfma(p(h3idx(1, 0, 0)), h1, p(0)));
    add_f(Q[0], f3(3, 0, 0), h3);
    Q[1] = fgfma(p(h3idx(1, 1, 0)), h1, p(h3idx(0, 1, 0)));
    add_f(Q[1], f3(2, 1, 0), h2);
    Q[2] = fgfma(p(h3idx(1, 0, 1)), h1, p(h3idx(0, 0, 1)));
    add_f(Q[2], f3(2, 0, 1), h2);
    Q[3] = p(h3idx(0, 2, 0));
    add_f(Q[3], f3(1, 2, 0), h1);
    Q[4] = p(h3idx(0, 1, 1));
    add_f(Q[4], f3(1, 1, 1), h1);
    Q[5] = p(h3idx(0, 0, 2));
    add_f(Q[5], f3(1, 0, 2), h1);
    T[0] = f3(0, 3, 0);
    T[1] = f3(0, 2, 1);
    T[2] = f3(0, 1, 2);
    T[3] = f3(0, 0, 3);
}

// limited slopes of two differences (collapsed along the normal) at the first tangent's node n
// and the four nodes of the second, times off[p] if by_p, and their moments along the second
// tangent: S (f, g) for the orders 0..2, S3 f's third
template <typename R>
__device__ __forceinline__ void slopes3(const FG<R> *QA, const R *TA, const FG<R> *QB, const R *TB, R h1, R h2, R h3,
                                        int limiter, bool by_p, const R *off, FG<R> *S, R &S3)
{
    const R k3 = R(0x1.a20bd700c2c3dp-2);   // sqrt(6)/6: He_3(c)/6 = -+ c sqrt(6)/6 at c_lo, c_hi
    auto along1 = [&](const FG<R> *Q, const R *T, FG<R> *C, R &C3) {
        C[0] = fgfma(Q[3], h2, fgfma(Q[1], h1, Q[0]));
        add_f(C[0], T[0], h3);
        C[1] = fgfma(Q[4], h1, Q[2]);
        add_f(C[1], T[1], h2);
        C[2] = Q[5];
        add_f(C[2], T[2], h1);
        C3 = T[3] * k3;
    };
    FG<R> A[3], B[3];
    R A3, B3;
    along1(QA, TA, A, A3);
    along1(QB, TB, B, B3);
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
        const int np = hi ? 3 : 2, nm = hi ? 0 : 1;   // nodes +c, -c
        const R c = R(node_c(np)), e2 = R(hen(2, np)), sg = hi ? R(1) : R(-1);
        const FG<R> EA = fgfma(A[2], e2, A[0]), EB = fgfma(B[2], e2, B[0]);
        FG<R> OA = A[1], OB = B[1];
        add_f(OA, A3, sg);
        add_f(OB, B3, sg);
        const FG<R> ap = fgfma(OA, c, EA), am = fgfma(OA, -c, EA), bp = fgfma(OB, c, EB), bm = fgfma(OB, -c, EB);
        FG<R> p, m;
        if (limiter == 1) {
            p = vminmod(ap, bp);
            m = vminmod(am, bm);
        } else {
            p = vanleer_half(ap, bp);
            m = vanleer_half(am, bm);
        }
        if (by_p) {
            p = p * off[np];
            m = m * off[nm];
        }
        const FG<R> s = p + m, d = p - m;
        const R w0 = R(node_w(np)), w1 = R(node_w(np) * he(1, np)), w2 = R(node_w(np) * he(2, np)), w3 = R(node_w(np) * he(3, np));
        if (hi == 0) {
            S[0] = s * w0;
            S[1] = d * w1;
            S[2] = s * w2;
            S3 = fpart(d) * w3;
        } else {
            S[0] = fgfma(s, w0, S[0]);
            S[1] = fgfma(d, w1, S[1]);
            S[2] = fgfma(s, w2, S[2]);
            S3 = vfma(fpart(d), w3, S3);
        }
    }
}

// Phi_rst += w_r X_st (f, r + s + t <= 3), Psi_rst (g, <= 2), from moments over the tangential nodes
template <typename R>
__device__ __forceinline__ void add_moments3(const R *w, const FG<R> *Q, const R *T, R *Phi, R *Psi)
{
#pragma unroll
    for (int r = 0; r <= 3; ++r)
#pragma unroll
        for (int s = 0; r + s <= 3; ++s)
#pragma unroll
            for (int t = 0; r + s + t <= 3; ++t) {
                const int st = h2st(s, t), k = h3idx(r, s, t);
                if (st < 6) {
                    Phi[k] = vfma(w[r], fpart(Q[st]), Phi[k]);
                    if (r + s + t <= 2) Psi[k] = vfma(w[r], gpart(Q[st]), Psi[k]);
                } else {
                    Phi[k] = vfma(w[r], T[st - 6], Phi[k]);
                }
            }
}

// One corrector pass of a face: base is cell R of its stencil in the staged box, st[3] the strides
// (in cells) of the face axes, l the frame velocity relative to the tile reference, ua the
// absolute one, h[3] the half steps over the cell sizes.
template <typename R, typename SCR>
__device__ __forceinline__ void pass3(const R *base, const FaceAxes3<R> &ax, const int *st, const R *l, R Tl, const R *ua,
                                      const R *h, int limiter, const SCR &scr, R *Phi, R *Psi)
{
    const NodeTab<R> &tab = node_tab<R>();
    const R invTl = R(1) / Tl, rsqTl = sqrt(invTl), sqTl = Tl * rsqTl;
    // departure offsets with the limiter's factor (2 for van Leer, 1 for minmod)
    const R sc = limiter == 1 ? R(1) : R(2);
#pragma unroll
    for (int k = 0; k < kNF3; ++k) Phi[k] = R(0);
#pragma unroll
    for (int k = 0; k < kNG3; ++k) Psi[k] = R(0);
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {   // 0: the nodes upwind of the right cell, 1: of the left
        unsigned mine = 0u;
#pragma unroll
        for (int m = 0; m < 4; ++m) mine |= (vfma(sqTl, R(node_c(m)), ua[0]) > R(0)) == (side == 1) ? 1u << m : 0u;
        if (mine == 0u) continue;
        const R *up = base - (side ? st[0] : 0) * kCell3;
#pragma unroll 1
        for (int sweep = 0; sweep < 3; ++sweep) {
            {
                R UF[kNF3], UG[kNG3];
                move_cell3<R>(up, ax, Tl, invTl, rsqTl, l, UF, UG);
                if (sweep == 0) {
                    // the upwind cell's own moments: its collapsed coefficients
                    R w[30];
#pragma unroll
                    for (int k = 0; k < 10; ++k) { w[2 * k] = UF[k]; w[2 * k + 1] = UG[k]; w[20 + k] = UF[10 + k]; }
#pragma unroll 1
                    for (int m = 0; m < 4; ++m) {
                        if (!((mine >> m) & 1u)) continue;
                        FG<R> Q[6];
                        R T[4];
                        collapse3<R>(w, tab.hen[m][1], tab.hen[m][2], tab.hen[m][3], Q, T);
                        add_moments3<R>(tab.whe[m], Q, T, Phi, Psi);
                    }
                }
                // upwind minus below, above minus upwind, into the scratch
                const int d = sweep == 0 ? st[0] : (sweep == 1 ? st[1] : st[2]);
#pragma unroll 1
                for (int q = 0; q < 2; ++q) {
                    R F[kNF3], G[kNG3], w[30];
                    move_cell3<R>(up + (q ? d : -d) * kCell3, ax, Tl, invTl, rsqTl, l, F, G);
                    const R sg = q ? R(-1) : R(1);
#pragma unroll
                    for (int k = 0; k < 10; ++k) {
                        w[2 * k] = sg * (UF[k] - F[k]);
                        w[2 * k + 1] = sg * (UG[k] - G[k]);
                        w[20 + k] = sg * (UF[10 + k] - F[10 + k]);
                    }
                    // 30 words are 7.5 slots of four: the halves meet in the middle slot in FP32
                    if constexpr (SCR::PER == 4) {
#pragma unroll
                        for (int k = 0; k < 7; ++k) scr.put(8 * q + k, w + 4 * k);
                        const R tail[4] = {w[28], w[29], R(0), R(0)};
                        scr.put(8 * q + 7, tail);
                    } else {
#pragma unroll
                        for (int k = 0; k < 15; ++k) scr.put(16 * q + k, w + 2 * k);
                    }
                }
            }
#pragma unroll 1
            for (int m = 0; m < 4; ++m) {
                if (!((mine >> m) & 1u)) continue;
                FG<R> QA[6], QB[6], Q[6];
                R TA[4], TB[4], T[4];
                {
                    const R h1 = tab.hen[m][1], h2 = tab.hen[m][2], h3 = tab.hen[m][3];
                    R w[32];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        constexpr int NS = 32 / SCR::PER;
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (SCR::PER == 4 || k < 15) scr.get(NS * q + k, w + SCR::PER * k);
                        if (q == 0) collapse3<R>(w, h1, h2, h3, QA, TA);
                        else collapse3<R>(w, h1, h2, h3, QB, TB);
                    }
                }
#pragma unroll
                for (int k = 0; k < 6; ++k) Q[k] = fg(R(0), R(0));
#pragma unroll
                for (int k = 0; k < 4; ++k) T[k] = R(0);
                R off[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) off[p] = -vfma(sqTl, R(node_c(p)), ua[2]) * (h[2] * sc);
#pragma unroll 1
                for (int n = 0; n < 4; ++n) {
                    FG<R> S[3];
                    R S3;
                    slopes3<R>(QA, TA, QB, TB, tab.hen[n][1], tab.hen[n][2], tab.hen[n][3], limiter, sweep == 2, off, S, S3);
                    // moments along the first tangent; its departure offset scales the weights of sweep 1
                    const R o1 = sweep == 1 ? -vfma(sqTl, tab.c[n], ua[1]) * (h[1] * sc) : R(1);
                    const R w0 = tab.whe[n][0] * o1, w1 = tab.whe[n][1] * o1, w2 = tab.whe[n][2] * o1, w3 = tab.whe[n][3] * o1;
                    Q[0] = fgfma(S[0], w0, Q[0]);
                    Q[1] = fgfma(S[0], w1, Q[1]);
                    Q[3] = fgfma(S[0], w2, Q[3]);
                    Q[2] = fgfma(S[1], w0, Q[2]);
                    Q[4] = fgfma(S[1], w1, Q[4]);
                    Q[5] = fgfma(S[2], w0, Q[5]);
                    T[0] = vfma(fpart(S[0]), w3, T[0]);
                    T[1] = vfma(fpart(S[1]), w2, T[1]);
                    T[2] = vfma(fpart(S[2]), w1, T[2]);
                    T[3] = vfma(S3, w0, T[3]);
                }
                // the departure offset along the normal scales the weights of sweep 0
                const R on = sweep == 0 ? sc * ((side ? R(0.5) : R(-0.5)) - vfma(sqTl, tab.c[m], ua[0]) * h[0]) : R(1);
                R w[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) w[r] = tab.whe[m][r] * on;
                add_moments3<R>(w, Q, T, Phi, Psi);
            }
        }
    }
}

// the frame of a pass's moments relative to the pass frame
template <typename R>
__device__ __forceinline__ bool moments_frame3(const R *p, const R *g, R Tl, R sq, R Cv, R &rho, R *du, R &T1)
{
    // p: 000, 100, 010, 001, 200, 020, 002
    rho = p[0];
    R k2 = R(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        du[a] = sq * p[1 + a] / rho;
        k2 = vfma(du[a], du[a], k2);
    }
    const R tr = vfma(R(3), rho, p[4] + p[5] + p[6]);
    T1 = (vfma(R(0.5) * Tl, tr, g[0]) - R(0.5) * rho * k2) / (Cv * rho);
    return T1 > R(0) && isfinite(T1) && isfinite(rho) && isfinite(du[0]) && isfinite(du[1]) && isfinite(du[2]);
}

// Eq. (FluxTransf) in the frame that a face's last moments define (face axes)
template <typename R>
__device__ __forceinline__ void face_populations3(const R *Phi, const R *Psi, R Tl, R rho, const R *du, R T1, R wb, R we,
                                                  R Cvh, R *Fo, R *Go)
{
    const R invT = R(1) / T1, zero[3] = {R(0), R(0), R(0)}, u[3] = {-du[0], -du[1], -du[2]};
    const Move3<R> M(Tl, u, T1, invT, sqrt(invT), zero);
    M.f_full(Phi, Fo);
    const R B1[3] = {Psi[1], Psi[2], Psi[3]}, B2[3] = {Psi[4], Psi[7], Psi[9]}, B11[3] = {Psi[8], Psi[6], Psi[5]};
    M.g(Psi[0], B1, B2, B11, Go);
    Fo[0] = vfma(wb, Fo[0], we * rho);
    Go[0] = vfma(wb, Go[0], we * Cvh * rho * T1);
#pragma unroll
    for (int k = 1; k < kNF3; ++k) Fo[k] = wb * Fo[k];
#pragma unroll
    for (int k = 1; k < kNG3; ++k) Go[k] = wb * Go[k];
}

// Tiles: TX x TY x TZ cells per CTA, one thread per face of each axis (whole warps per axis), the
// box [i0-2, i0+TX] x [j0-2, j0+TY] x [k0-2, k0+TZ] staged in dynamic shared memory, then the
// scratch.
template <typename R, int TX_, int TY_, int TZ_, int MINB_>
struct Face3Tile {
    static constexpr int TX = TX_, TY = TY_, TZ = TZ_, NF = TX * TY * TZ;
    static constexpr int THREADS = 3 * NF, MINB = MINB_;
    static constexpr int BX = TX + 3, BY = TY + 3, BZ = TZ + 3;
    static constexpr int SLOTS = 64 / (16 / int(sizeof(R)));
    static constexpr size_t tile_bytes = (sizeof(R) * kCell3 * BX * BY * BZ + 15) / 16 * 16;
    static constexpr size_t smem = tile_bytes + size_t(SLOTS) * 16 * THREADS;
    static_assert(NF % 32 == 0, "whole warps per face axis");
    static_assert(smem <= 227 * 1024, "the tile and scratch fit one CTA's shared memory");
};

// A warp with at most this many unfinished faces hands them over.  A pass of the warp costs about as
// much as 7 (FP32) or 15 (FP64) passes of a warp per face, but the list runs in parallel: us a launch for
// 12 / 20 / 31, FP32: explosion 64^3 812 / 714 / 705, smooth flow 64^3 1242 / 1314 / 1408; for 15 / 24 / 31,
// FP64: explosion 64^3 24.0 / 22.8 / 23.2 ms, smooth flow 48^3 28.6 / 28.9 / 31.7 ms.  An FP64 grid of at most
// three warps of faces per sub-partition hands over everything after the first pass (32): a pass of
// a warp is a chain of 9000 FP64 instructions of 64 cycles there, 285 us (explosion 25 x 23 x 21: 5.6 ms
// at 20, 3.7 at 31, 2.2 at 32); with a fixed number of passes the faces stay together anyway.
template <typename R>
inline int tail3_faces(long long faces, int sms, int fixed_iters)
{
    return sizeof(R) == 8 && fixed_iters == 0 && faces <= 32ll * 12 * sms ? 32 : 20;
}
// R words of a warp in the tail kernel: the 12 stencil cells as staged, the same in the pass frame, and
// 32 moments
constexpr int kTailCell3 = 31, kTailWords3 = 12 * kCell3 + 12 * kTailCell3 + 32, kTailThreads3 = 128;
// (of a listed face the passes so far, its next frame and its last valid one wait in its own output
// planes)

// the sum over the warp of each of c[0..31]; lane q returns that of c[q]
template <typename R>
__device__ __forceinline__ R reduce32(R *c, int q)
{
#pragma unroll
    for (int half = 16; half >= 1; half >>= 1) {
        const bool upper = (q & half) != 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (k >= half) continue;
            const R keep = upper ? c[k + half] : c[k], send = upper ? c[k] : c[k + half];
            c[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
        }
    }
    return c[0];
}

// offset of stencil slot s along the face axes: 0 LL, 1 L, 2 R, 3 RR; 4 L-, 5 L+, 6 R-, 7 R+ along the
// first tangent; 8 .. 11 along the second
__device__ __forceinline__ void slot_offset3(int s, int &on, int &o1, int &o2)
{
    on = s < 4 ? s - 2 : (((s - 4) & 3) >> 1) - 1;
    const int sg = s < 4 ? 0 : ((s & 1) ? 1 : -1);
    o1 = s < 8 ? sg : 0;
    o2 = s < 8 ? 0 : sg;
}

// Works off the list of unfinished faces, a warp per face: lane q holds stencil cell q (< 12) and
// evaluates the populations (m, n, +-c) with m = q / 8, n = q / 2 % 4 and c = c_lo (q even) or c_hi.
// The last CTA empties the list for the next step.
template <typename R>
__global__ void __launch_bounds__(kTailThreads3, 3)
face3_tail_kernel(const Params3<R> P)
{
    using W = typename FrameWords<R>::word;
    __shared__ __align__(16) R words[kTailThreads3 / 32][kTailWords3];
    const unsigned full = 0xffffffffu;
    const int q = threadIdx.x & 31, m = q >> 3, n = (q >> 1) & 3, np = (q & 1) ? 3 : 2;
    R *raw = words[threadIdx.x >> 5], *cells = raw + 12 * kCell3, *mom = cells + 12 * kTailCell3;
    const StepC<R> &KC = step_c<R>(*P.clock);
    const NodeTab<R> &tab = node_tab<R>();
    const R Cv = P.Cv_r, tol = P.tol_r;
    R basis[10], weight[10];   // over (r, s), r + s <= 3, in hidx order
#pragma unroll
    for (int r = 0; r <= 3; ++r)
#pragma unroll
        for (int s = 0; r + s <= 3; ++s) {
            basis[hidx(r, s)] = tab.hen[m][r] * tab.hen[n][s];
            weight[hidx(r, s)] = tab.whe[m][r] * tab.whe[n][s];
        }
    const R cp_ = tab.c[np], e2 = tab.hen[np][2], e3 = tab.hen[np][3];
    FaceCount fc{0, 0, 0, 0};
    const unsigned int count = P.tail->n;
    for (;;) {
        unsigned int item = 0;
        if (q == 0) item = atomicAdd(&P.tail->next, 1u);
        item = __shfl_sync(full, item, 0);
        if (item >= count) break;
        const unsigned long long it = P.tail_items[item];
        const int dir = int((it >> kTailDirShift) & 3ull);
        const long long f = (long long)(it & ((1ull << kTailDirShift) - 1));
        const long long nf = P.nf(dir), sx = P.nx + (dir == 0), sy = P.ny + (dir == 1);
        const long long fi = f % sx, fj = (f / sx) % sy, fk = f / (sx * sy);
        R *Fout = dir == 0 ? P.ff[0] : (dir == 1 ? P.ff[1] : P.ff[2]), *Gout = dir == 0 ? P.fg[0] : (dir == 1 ? P.fg[1] : P.fg[2]);
        W *Frm = dir == 0 ? P.ffr[0] : (dir == 1 ? P.ffr[1] : P.ffr[2]);
        const FaceAxes3<R> ax(dir);
        const R h[3] = {dir == 0 ? KC.h_dx : (dir == 1 ? KC.h_dy : KC.h_dz), dir == 0 ? KC.h_dy : KC.h_dx, dir == 2 ? KC.h_dy : KC.h_dz};
        // velocities are taken relative to the face's base frame here (in the tiles: to the tile's)
        const W ref[3] = {Frm[f], Frm[nf + f], Frm[2 * nf + f]};
        const R ba[3] = {R(fr_lead(dir == 0 ? ref[0] : (dir == 1 ? ref[1] : ref[2]))), R(fr_lead(dir == 0 ? ref[1] : ref[0])),
                         R(fr_lead(dir == 2 ? ref[1] : ref[2]))};
        R d[3], v[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            d[a] = Fout[a * nf + f];
            v[a] = Fout[(3 + a) * nf + f];
        }
        R Tl = Fout[6 * nf + f], vT = Fout[7 * nf + f];
        int iters = int(Fout[8 * nf + f]);
        bool bad = (it & kTailBad) != 0;
        int fallbacks = bad ? 1 : 0;
        bool have = !bad || iters > 1, done = false, restarted = false, redo = false;
        __syncwarp();
        if (q < 12) {
            int on, o1, o2;
            slot_offset3(q, on, o1, o2);
            store_cell3<R>(P, fi + (dir == 0 ? on : o1), fj + (dir == 1 ? on : (dir == 0 ? o1 : o2)), fk + (dir == 2 ? on : o2), KC.cp,
                           KC.ce, ref, raw + q * kCell3);
        }
        __syncwarp();
        R rho, du[3], T1;
        for (;;) {
            if (bad) {
                bad = false;
                if (!restarted && iters < P.max_iter) {
                    // once: the frame of the pooled conserved moments of the twelve stencil cells
                    restarted = true;
                    R r = R(0), mo[3] = {R(0), R(0), R(0)}, e = R(0);
#pragma unroll 1
                    for (int s = 0; s < 12; ++s) {
                        const R *c = raw + s * kCell3;
                        const R rc = c[0], x[3] = {c[ax.n + 4], c[ax.t1 + 4], c[ax.t2 + 4]};
                        r += rc;
                        R v2 = R(0);
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            mo[a] += rc * x[a];
                            v2 += x[a] * x[a];
                        }
                        e += rc * (Cv * c[3] + R(0.5) * v2);
                    }
                    r /= R(12);
                    e /= R(12);
                    R k2 = R(0);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        mo[a] /= R(12);
                        d[a] = mo[a] / r;
                        k2 += mo[a] * mo[a];
                    }
                    Tl = (e - R(0.5) * k2 / r) / (Cv * r);
                } else {
                    // stopped by a pass without a frame: the last valid one over again, if any
                    redo = true;
#pragma unroll
                    for (int a = 0; a < 3; ++a) d[a] = v[a];
                    Tl = vT;
                }
            }
            // ---- the pass
            const R invTl = R(1) / Tl, rsqTl = sqrt(invTl), sqTl = Tl * rsqTl, sq = sqrt(Tl);
            __syncwarp();
            if (q < 12) {
                R F[kNF3], G[kNG3];
                move_cell3<R>(raw + q * kCell3, ax, Tl, invTl, rsqTl, d, F, G);
                R *o = cells + q * kTailCell3;
#pragma unroll
                for (int k = 0; k < kNF3; ++k) o[k] = F[k];
#pragma unroll
                for (int k = 0; k < kNG3; ++k) o[20 + k] = G[k];
            }
            __syncwarp();
            const R un = vfma(sqTl, tab.c[m], ba[0] + d[0]), u1 = vfma(sqTl, tab.c[n], ba[1] + d[1]);
            const bool left = un > R(0);
            // populations (m, n, +c) and (m, n, -c) of a moved cell, f and g
            auto eval = [&](int s, FG<R> &p, FG<R> &mi) {
                const R *c = cells + s * kTailCell3;
                R C[4] = {c[0], c[h3idx(0, 0, 1)], c[h3idx(0, 0, 2)], c[h3idx(0, 0, 3)]};
                R D[3] = {c[20], c[20 + h3idx(0, 0, 1)], c[20 + h3idx(0, 0, 2)]};
#pragma unroll
                for (int r = 0; r <= 3; ++r)
#pragma unroll
                    for (int s2 = 0; r + s2 <= 3; ++s2) {
                        if (r + s2 == 0) continue;
#pragma unroll
                        for (int t2 = 0; r + s2 + t2 <= 3; ++t2) {
                            C[t2] = vfma(c[h3idx(r, s2, t2)], basis[hidx(r, s2)], C[t2]);
                            if (r + s2 + t2 <= 2) D[t2] = vfma(c[20 + h3idx(r, s2, t2)], basis[hidx(r, s2)], D[t2]);
                        }
                    }
                const R E = vfma(C[2], e2, C[0]), O = vfma(C[3], e3, cp_ * C[1]), Eg = vfma(D[2], e2, D[0]);
                p = fg(E + O, vfma(cp_, D[1], Eg));
                mi = fg(E - O, vfma(-cp_, D[1], Eg));
            };
            FG<R> up, um, lp, lm, hp, hm;
            eval(left ? 1 : 2, up, um);
            FG<R> rp = up, rm = um;
            const R sc = P.limiter == 1 ? R(1) : R(2);
            auto slope = [&](FG<R> a, FG<R> c) { return P.limiter == 1 ? vminmod(a, c) : vanleer_half(a, c); };
            auto add_slope = [&](int lo, int hi, R offp, R offm) {
                eval(lo, lp, lm);
                eval(hi, hp, hm);
                rp = fgfma(slope(up - lp, hp - up), offp, rp);
                rm = fgfma(slope(um - lm, hm - um), offm, rm);
            };
            const R on = sc * ((left ? R(0.5) : R(-0.5)) - un * h[0]), o1 = -u1 * (h[1] * sc), k2 = -(h[2] * sc);
            add_slope(left ? 0 : 1, left ? 2 : 3, on, on);
            add_slope(left ? 4 : 6, left ? 5 : 7, o1, o1);
            add_slope(left ? 8 : 10, left ? 9 : 11, vfma(sqTl, cp_, ba[2] + d[2]) * k2, vfma(sqTl, -cp_, ba[2] + d[2]) * k2);
            {
                const FG<R> s = rp + rm, dd = rp - rm;
                const FG<R> v0 = s * tab.whe[np][0], v1 = dd * tab.whe[np][1], v2 = s * tab.whe[np][2];
                const R v3 = fpart(dd) * tab.whe[np][3];
                R c[32];
#pragma unroll
                for (int r = 0; r <= 3; ++r)
#pragma unroll
                    for (int s2 = 0; r + s2 <= 3; ++s2)
#pragma unroll
                        for (int t2 = 0; r + s2 + t2 <= 3; ++t2) {
                            const int k = h3idx(r, s2, t2);
                            const R w = weight[hidx(r, s2)];
                            c[k] = w * (t2 == 0 ? fpart(v0) : (t2 == 1 ? fpart(v1) : (t2 == 2 ? fpart(v2) : v3)));
                            if (r + s2 + t2 <= 2) c[20 + k] = w * (t2 == 0 ? gpart(v0) : (t2 == 1 ? gpart(v1) : gpart(v2)));
                        }
                c[30] = c[31] = R(0);
                mom[q] = reduce32(c, q);
            }
            __syncwarp();
            const R p[7] = {mom[0], mom[1], mom[2], mom[3], mom[4], mom[7], mom[9]};
            const bool ok = moments_frame3<R>(p, mom + 20, Tl, sq, Cv, rho, du, T1);
            if (redo) break;
            ++iters;
            if (ok) {
                have = true;
#pragma unroll
                for (int a = 0; a < 3; ++a) v[a] = d[a];
                vT = Tl;
                if (P.fixed_iters > 0) {
                    done = iters >= P.fixed_iters;
                } else {
                    const R s = tol * sq;
                    done = fabs(T1 - Tl) <= tol * Tl && fabs(du[0]) <= s && fabs(du[1]) <= s && fabs(du[2]) <= s;
                }
                if (done || iters >= P.max_iter) break;
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] += du[a];
                Tl = T1;
            } else {
                ++fallbacks;
                bad = true;
                if (!have && (restarted || iters >= P.max_iter)) break;
            }
        }
        // ---- the face's result
        R out = R(__longlong_as_double(0x7ff8000000000000ll));
        if (have) {
            R Phi[kNF3], Psi[kNG3], Fo[kNF3], Go[kNG3];
#pragma unroll
            for (int k = 0; k < kNF3; ++k) Phi[k] = mom[k];
#pragma unroll
            for (int k = 0; k < kNG3; ++k) Psi[k] = mom[20 + k];
            face_populations3<R>(Phi, Psi, Tl, rho, du, T1, KC.wb, KC.we, P.Cvh_r, Fo, Go);
            __syncwarp();
            if (q == 0) {
#pragma unroll
                for (int k = 0; k < kNF3; ++k) mom[k] = Fo[k];
#pragma unroll
                for (int k = 0; k < kNG3; ++k) mom[20 + k] = Go[k];
                const R dn = d[0] + du[0], d1 = d[1] + du[1], d2 = d[2] + du[2];
                const R dl[3] = {dir == 0 ? dn : d1, dir == 1 ? dn : (dir == 0 ? d1 : d2), dir == 2 ? dn : d2};
#pragma unroll
                for (int a = 0; a < 3; ++a) Frm[a * nf + f] = fr_add(ref[a], dl[a]);
                Frm[3 * nf + f] = fr_word(T1);
            }
            __syncwarp();
            out = mom[q];
        } else if (q == 0) {
            fr_store(Frm[3 * nf + f], double(out));
        }
        if (q < 20) Fout[kFacePerm.k[dir][q] * nf + f] = out;
        else if (q < 30) Gout[kFacePerm.k[dir][q - 20] * nf + f] = out;
        if (q == 0) {
            fc.iters += iters;
            fc.fallbacks += fallbacks;
            fc.nonconv += done ? 0 : 1;
            fc.nonphys += have ? 0 : 1;
        }
    }
    if (q == 0 && fc.iters) count_faces(P.diag, fc, 0);
    __syncthreads();
    if (threadIdx.x == 0) {
        // every CTA has taken its last ticket: empty the list
        if (atomicAdd(&P.tail->ctas, 1u) == gridDim.x - 1) {
            P.tail->n = 0u;
            P.tail->next = 0u;
            P.tail->ctas = 0u;
        }
    }
}

// The face kernel of a step, the faces of all three axes.  The rules of the corrector are those of the
// D2Q16 kernel (convergence, one restart from the pooled moments of the stencil, the last valid
// pass); the warp's own passes only ever go forward, the tail does the rest.
template <typename R, typename TL>
__global__ void __launch_bounds__(TL::THREADS, TL::MINB)
face3_kernel(const Params3<R> P)
{
    constexpr int TX = TL::TX, TY = TL::TY, TZ = TL::TZ, BX = TL::BX, BY = TL::BY, BZ = TL::BZ, NT = TL::THREADS;
    using W = typename FrameWords<R>::word;
    using Scr = Scratch3<R, NT>;
    extern __shared__ __align__(16) unsigned char f3_dyn[];
    R *tile = reinterpret_cast<R *>(f3_dyn);
    unsigned char *scratch = f3_dyn + TL::tile_bytes;
    const Scr scr{(unsigned)__cvta_generic_to_shared(scratch) + threadIdx.x * 16u};
    const Clock &K = *P.clock;
    const double step_dt = K.dt;   // 0: t_end reached, the step is a no-op (tested after the staging loads)
    const StepC<R> &KC = step_c<R>(K);
    const long long i0 = (long long)blockIdx.x * TX, j0 = (long long)blockIdx.y * TY, k0 = (long long)blockIdx.z * TZ;
    const int dir = threadIdx.x / TL::NF, tl = threadIdx.x - dir * TL::NF;
    const int tx = tl % TX, ty = (tl / TX) % TY, tz = tl / (TX * TY);
    const long long fi = i0 + tx, fj = j0 + ty, fk = k0 + tz;
    const bool active = fi < P.nx + (dir == 0) && fj < P.ny + (dir == 1) && fk < P.nz + (dir == 2);
    const long long nf = P.nf(dir), f = active ? P.fidx(dir, fi, fj, fk) : 0;
    // selects: a run-time index into the parameter arrays would copy them to local memory
    W *Frm = dir == 0 ? P.ffr[0] : (dir == 1 ? P.ffr[1] : P.ffr[2]);
    W uref[3], Tpw;   // the predictor frame, loaded before the staging so that the loads overlap
#pragma unroll
    for (int a = 0; a < 3; ++a) uref[a] = active ? Frm[a * nf + f] : fr_word(R(0));
    Tpw = active ? Frm[3 * nf + f] : fr_word(R(1));
    W ut[3];
    cell_velocity3<R>(P, i0, j0, k0, ut);
    for (int t = threadIdx.x; t < BX * BY * BZ; t += NT) {
        const int bx = t % BX, by = (t / BX) % BY, bz = t / (BX * BY);
        store_cell3<R>(P, i0 - 2 + bx, j0 - 2 + by, k0 - 2 + bz, KC.cp, KC.ce, ut, tile + t * kCell3);
    }
    if (!(step_dt > 0.0)) return;   // the same value in every thread
    __syncthreads();

    const R *base = tile + (((tz + 2) * BY + ty + 2) * BX + tx + 2) * kCell3;
    const int sx = 1, sy = BX, sz = BX * BY;
    const int st[3] = {dir == 0 ? sx : (dir == 1 ? sy : sz), dir == 0 ? sy : sx, dir == 2 ? sy : sz};
    const FaceAxes3<R> ax(dir);
    const R h[3] = {dir == 0 ? KC.h_dx : (dir == 1 ? KC.h_dy : KC.h_dz), dir == 0 ? KC.h_dy : KC.h_dx, dir == 2 ? KC.h_dy : KC.h_dz};
    const R Cv = P.Cv_r, tol = P.tol_r;
    R b[3], ba[3], d[3] = {R(0), R(0), R(0)}, v[3] = {R(0), R(0), R(0)}, Tl = R(fr_lead(Tpw)), vT = Tl;
    {
        // the base frame in face axes (selects: no run-time indexed array)
        const W un = dir == 0 ? uref[0] : (dir == 1 ? uref[1] : uref[2]), u1 = dir == 0 ? uref[1] : uref[0], u2 = dir == 2 ? uref[1] : uref[2];
        const W tn = dir == 0 ? ut[0] : (dir == 1 ? ut[1] : ut[2]), t1 = dir == 0 ? ut[1] : ut[0], t2 = dir == 2 ? ut[1] : ut[2];
        b[0] = R(fr_rel(un, tn));
        b[1] = R(fr_rel(u1, t1));
        b[2] = R(fr_rel(u2, t2));
        ba[0] = R(fr_lead(un));
        ba[1] = R(fr_lead(u1));
        ba[2] = R(fr_lead(u2));
    }
    bool run = active, done = false;
    bool bad = false;   // the last pass defined no frame
    int iters = 0;
    R Phi[kNF3], Psi[kNG3], rho, du[3], T1, pd[3], pT;
    for (;;) {
        const R l[3] = {b[0] + d[0], b[1] + d[1], b[2] + d[2]}, ua[3] = {ba[0] + d[0], ba[1] + d[1], ba[2] + d[2]};
        pass3<R, Scr>(base, ax, st, l, Tl, ua, h, P.limiter, scr, Phi, Psi);
        const R sq = sqrt(Tl), p[7] = {Phi[0], Phi[1], Phi[2], Phi[3], Phi[4], Phi[7], Phi[9]};
        const bool ok = moments_frame3<R>(p, Psi, Tl, sq, Cv, rho, du, T1);
        pT = Tl;
#pragma unroll
        for (int a = 0; a < 3; ++a) pd[a] = d[a];
        if (run) {
            ++iters;
            if (ok) {
#pragma unroll
                for (int a = 0; a < 3; ++a) v[a] = d[a];
                vT = Tl;
                if (P.fixed_iters > 0) {
                    done = iters >= P.fixed_iters;
                } else {
                    const R s = tol * sq;
                    done = fabs(T1 - Tl) <= tol * Tl && fabs(du[0]) <= s && fabs(du[1]) <= s && fabs(du[2]) <= s;
                }
                run = !done && iters < P.max_iter;
                if (run) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) d[a] += du[a];
                    Tl = T1;
                }
            } else {
                run = false;
                bad = true;
            }
        }
        if (__popc(__ballot_sync(0xffffffffu, run)) <= P.tail_at) break;
    }
    R *Fout = dir == 0 ? P.ff[0] : (dir == 1 ? P.ff[1] : P.ff[2]), *Gout = dir == 0 ? P.fg[0] : (dir == 1 ? P.fg[1] : P.fg[2]);
    // faces for the tail: their frames into their own output planes, then a place in the list
    const bool listed = run || bad;
    const unsigned int lists = __ballot_sync(0xffffffffu, listed);
    if (lists) {
        unsigned int at = 0;
        if ((threadIdx.x & 31) == 0) at = atomicAdd(&P.tail->n, __popc(lists));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(lists & ((1u << (threadIdx.x & 31)) - 1u));
        if (listed) {
            const R c[9] = {d[0], d[1], d[2], v[0], v[1], v[2], Tl, vT, R(iters)};
#pragma unroll
            for (int k = 0; k < 9; ++k) Fout[k * nf + f] = c[k];
            P.tail_items[at] = (unsigned long long)f | (unsigned long long)dir << kTailDirShift | (bad ? kTailBad : 0ull);
        }
    }
    FaceCount fc{0, 0, 0, 0};
    if (active && !listed) {
        fc.iters = iters;
        fc.nonconv = done ? 0 : 1;
        R Fo[kNF3], Go[kNG3];
        face_populations3<R>(Phi, Psi, pT, rho, du, T1, KC.wb, KC.we, P.Cvh_r, Fo, Go);
#pragma unroll
        for (int k = 0; k < kNF3; ++k) (Fout + kFacePerm.k[dir][k] * nf)[f] = Fo[k];
#pragma unroll
        for (int k = 0; k < kNG3; ++k) (Gout + kFacePerm.k[dir][k] * nf)[f] = Go[k];
        const R dn = pd[0] + du[0], d1 = pd[1] + du[1], d2 = pd[2] + du[2];
        const R dl[3] = {dir == 0 ? dn : d1, dir == 1 ? dn : (dir == 0 ? d1 : d2), dir == 2 ? dn : d2};
#pragma unroll
        for (int a = 0; a < 3; ++a) Frm[a * nf + f] = fr_add(Frm[a * nf + f], dl[a]);
        Frm[3 * nf + f] = fr_word(T1);
    }
    fc.iters = warp_sum_count(fc.iters);
    fc.nonconv = warp_sum_count(fc.nonconv);
    const unsigned int n_act = __popc(__ballot_sync(0xffffffffu, active));
    if ((threadIdx.x & 31) == 0 && n_act) count_faces(P.diag, fc, n_act);
}

}  // namespace pond
