// pond_face2.cuh -- the face predictor-corrector of Sec. III.B.3 on D2Q16 grids.
//
// The arithmetic bounds this kernel (about 2000 operations a face and pass against 300 bytes),
// so it is laid out for the fewest instructions per face:
//   - FP32: a thread solves two faces, one per lane of the packed FP32x2 instructions
//     (pond_vec.cuh): the faces (i, j) and (i, j + TY/2) of its tile.  The staged box holds the
//     cells in the same pairs, so a 16-byte shared-memory load brings two coefficients of both.
//     FP64: one face per thread; the FP64 pipe (1/64 of the FP32 rate) is the bound there.
//   - The normal nodes are taken by their upwind side.  All nodes of a side read the same
//     neighbours of the same upwind cell, so a side takes 5 changes of frame and a pass 10 at
//     most (node by node it was 14).
//   - Everything but the limiter is linear, so the one-sided differences are formed once in
//     Hermite space, and the upwind population itself never has to be evaluated: its moments
//     over the tangential nodes are its own coefficients.
//   - The tangential nodes come in pairs +-c, evaluated and summed as even and odd parts.
//   - A side is done in two sweeps over its nodes, the normal slopes and then the tangential ones
//     with the upwind terms, by one rolled loop: the instruction caches hold all of it, and no
//     more than two cells' coefficients are live at once (the upwind cell waits in a per-thread
//     scratch in shared memory).
//
// Nearly every face converges in its first pass, but the faces at shocks take up to max_iter, a
// few per warp, and would keep whole warps (and, at small sizes, the whole launch) waiting.
// So a warp goes on pass by pass only while more than coop_faces of its faces need it; the
// others go to a list that is worked off with 16 lanes per face, one lane per population: the whole
// grid's, by a kernel of its own (lane_tail_kernel), or with the learned predictor the CTA's (coop_tail).
//
// Measured (GB300, us a launch; before: the best of the node-by-node tiles, that is 8 x 8 with
// shared scratch in FP32 and 8 x 8 in FP64, and the 32 x 4 tile that was the default): FP32 quadrants
// 1024^2 280 (328, default 446), shocked interface 1001 x 253 with minmod 93 (130, 186); FP64
// quadrants 256^2 981 (3208), all with the tail kernel.  FP32 issues 143 M instructions where the node-by-node tile issued 252 M,
// at 49% of the issue slots with 12 warps per SM: a packed multiply-add with three different
// register pairs takes four cycles of the register file (two with a repeated operand), the
// dependent-instruction waits come next (1.6 of 6 cycles), then the loads around the pass; 168 registers
// spill 72 B.  Four CTAs
// per SM would need 128 registers and spill 212 B (397 us at 8 x 16 cells); two leave the loads
// exposed (318 us).
#pragma once

#include <type_traits>

#include "pond_kernels.cuh"
#include "pond_vec.cuh"

namespace pond {

// Tile variants: TX x TY cells per CTA, each thread one group of lanes (two x- or two y-faces
// in FP32, one in FP64), MINB CTAs per SM for the register budget.
template <int TX_, int TY_, int MINB_>
struct LaneVariant {
    static constexpr int TX = TX_, TY = TY_, MINB = MINB_;
    static constexpr bool LANES = true;
};
template <typename R, typename V>
__host__ __device__ constexpr int lane_threads() { return 2 * V::TX * V::TY / VecOf<R>::lanes; }

// A staged cell (FP32: the pair (i, j), (i, j + TY/2)): phi-bar-plus coefficients of f and g,
// velocity relative to the tile reference, T, in three groups of six words: those symmetric
// in the axes (f 00 11, g 00 11, T), those along x (f 20 30 21, g 10 20, u_x) and the same along
// y.  A face reads its stencil normal first: the y-faces read the second and third groups
// exchanged, so one staged box serves both directions.  144 bytes: nine 16-byte loads, and
// eight neighbouring threads' loads fall in distinct bank groups.
template <typename V>
struct __align__(16) LaneCell {
    V sym[6], ax[2][6];
};
// words of a fetched cell: symmetric group, normal group, tangential group
enum { C_A00, C_A11, C_B00, C_B11, C_T, C_PAD, C_A20, C_A30, C_A21, C_B10, C_B20, C_UN,
       C_A02, C_A03, C_A12, C_B01, C_B02, C_UT };
template <typename V>
struct LaneWords {
    V w[18];
};
template <typename V>
__device__ __forceinline__ LaneWords<V> fetch_lane(const LaneCell<V> *p, int dir)
{
    union {
        LaneWords<V> c;
        float4 v[9];
    } u;
    const float4 *src = reinterpret_cast<const float4 *>(p);
    const float4 *sn = src + 3 * dir, *st = src - 3 * dir;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u.v[k] = src[k];
        u.v[3 + k] = sn[3 + k];
        u.v[6 + k] = st[6 + k];
    }
    return u.c;
}

// Per-thread scratch in shared memory, 16-byte slots, thread-minor (a warp's accesses are
// contiguous).  Volatile accesses, so that nothing kept here stays in registers too.
template <typename V, int NT>
struct LaneScratch {
    unsigned int addr;   // this thread's slot 0
    __device__ __forceinline__ void put(int slot, V a, V b) const
    {
        union { V v[2]; float4 f; } u;
        u.v[0] = a;
        u.v[1] = b;
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr + slot * (NT * 16)), "f"(u.f.x), "f"(u.f.y),
                     "f"(u.f.z), "f"(u.f.w) : "memory");
    }
    __device__ __forceinline__ void get(int slot, V &a, V &b) const
    {
        union { V v[2]; float4 f; } u;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(u.f.x), "=f"(u.f.y), "=f"(u.f.z), "=f"(u.f.w)
                     : "r"(addr + slot * (NT * 16)) : "memory");
        a = u.v[0];
        b = u.v[1];
    }
    // a cell's coefficients, f (10) and g (6), in slots base .. base + 7
    __device__ __forceinline__ void store(int base, const V *F, const V *G) const
    {
#pragma unroll
        for (int k = 0; k < 5; ++k) put(base + k, F[2 * k], F[2 * k + 1]);
#pragma unroll
        for (int k = 0; k < 3; ++k) put(base + 5 + k, G[2 * k], G[2 * k + 1]);
    }
    __device__ __forceinline__ void load(int base, V *F, V *G) const
    {
#pragma unroll
        for (int k = 0; k < 5; ++k) get(base + k, F[2 * k], F[2 * k + 1]);
#pragma unroll
        for (int k = 0; k < 3; ++k) get(base + 5 + k, G[2 * k], G[2 * k + 1]);
    }
};

// node tables with every entry in both lanes
template <typename V>
struct LaneTab {
    V hen[4][4], whe[4][4], c[4];
};
template <typename V> __host__ __device__ constexpr LaneTab<V> make_lane_tab();
template <>
__host__ __device__ constexpr LaneTab<double> make_lane_tab<double>()
{
    LaneTab<double> t{};
    for (int m = 0; m < 4; ++m) {
        t.c[m] = node_c(m);
        for (int k = 0; k < 4; ++k) {
            t.hen[m][k] = hen(k, m);
            t.whe[m][k] = node_w(m) * he(k, m);
        }
    }
    return t;
}
template <>
__host__ __device__ constexpr LaneTab<Lane2> make_lane_tab<Lane2>()
{
    LaneTab<Lane2> t{};
    const LaneTab<double> d = make_lane_tab<double>();
    for (int m = 0; m < 4; ++m) {
        t.c[m].v.x = t.c[m].v.y = float(d.c[m]);
        for (int k = 0; k < 4; ++k) {
            t.hen[m][k].v.x = t.hen[m][k].v.y = float(d.hen[m][k]);
            t.whe[m][k].v.x = t.whe[m][k].v.y = float(d.whe[m][k]);
        }
    }
    return t;
}
static __constant__ LaneTab<double> kLaneTabD = make_lane_tab<double>();
static __constant__ LaneTab<Lane2> kLaneTabF = make_lane_tab<Lane2>();
template <typename V> __device__ __forceinline__ const LaneTab<V> &lane_tab();
template <> __device__ __forceinline__ const LaneTab<double> &lane_tab<double>() { return kLaneTabD; }
template <> __device__ __forceinline__ const LaneTab<Lane2> &lane_tab<Lane2>() { return kLaneTabF; }

// column collapse at normal node m: C_b = sum_a A_ab He_a(c_m)/a!, f (10 -> 4) and g (6 -> 3)
template <typename V>
__device__ __forceinline__ void collapse(const V *F, const V *G, V h1, V h2, V h3, V *C, V *D)
{
    C[0] = vfma(F[hidx(3, 0)], h3, vfma(F[hidx(2, 0)], h2, vfma(F[hidx(1, 0)], h1, F[0])));
    C[1] = vfma(F[hidx(2, 1)], h2, vfma(F[hidx(1, 1)], h1, F[hidx(0, 1)]));
    C[2] = vfma(F[hidx(1, 2)], h1, F[hidx(0, 2)]);
    C[3] = F[hidx(0, 3)];
    D[0] = vfma(G[hidx(2, 0)], h2, vfma(G[hidx(1, 0)], h1, G[0]));
    D[1] = vfma(G[hidx(1, 1)], h1, G[hidx(0, 1)]);
    D[2] = G[hidx(0, 2)];
}

// Limited slopes of the one-sided differences a and b (collapsed coefficients) at the four
// tangential nodes, times off[n] if tang, and their moments along the tangent: S (f, orders
// 0..3), SG (g, 0..2).  The nodes come as +-c_lo and +-c_hi: a value there is the even part
// plus or minus the odd part, and the moments need their sums and differences.
template <typename V>
__device__ __forceinline__ void slope_moments(const V *Ca, const V *Da, const V *Cb, const V *Db, int limiter, bool tang,
                                              const V *off, V *S, V *SG)
{
    // He_3(c)/6 = -+ c sqrt(6)/6 at c_lo, c_hi
    const V k3 = vset<V>(0x1.a20bd700c2c3dp-2);
    const V a3 = k3 * Ca[3], b3 = k3 * Cb[3];
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
        const int np = hi ? 3 : 2, nm = hi ? 0 : 1;   // nodes +c, -c
        const V c = vset<V>(node_c(np)), mc = vset<V>(node_c(nm)), h2 = vset<V>(hen(2, np));
        const V Ea = vfma(Ca[2], h2, Ca[0]), Eb = vfma(Cb[2], h2, Cb[0]);
        const V Oa = hi ? Ca[1] + a3 : Ca[1] - a3, Ob = hi ? Cb[1] + b3 : Cb[1] - b3;
        const V fap = vfma(c, Oa, Ea), fam = vfma(mc, Oa, Ea), fbp = vfma(c, Ob, Eb), fbm = vfma(mc, Ob, Eb);
        const V Ga = vfma(Da[2], h2, Da[0]), Gb = vfma(Db[2], h2, Db[0]);
        const V gap = vfma(c, Da[1], Ga), gam = vfma(mc, Da[1], Ga), gbp = vfma(c, Db[1], Gb), gbm = vfma(mc, Db[1], Gb);
        V fp, fm, gp, gm;
        if (limiter == 1) {
            fp = vminmod(fap, fbp); fm = vminmod(fam, fbm);
            gp = vminmod(gap, gbp); gm = vminmod(gam, gbm);
        } else {
            fp = vanleer_half(fap, fbp); fm = vanleer_half(fam, fbm);
            gp = vanleer_half(gap, gbp); gm = vanleer_half(gam, gbm);
        }
        if (tang) {
            fp = fp * off[np]; fm = fm * off[nm];
            gp = gp * off[np]; gm = gm * off[nm];
        }
        const V sf = fp + fm, df = fp - fm, sg = gp + gm, dg = gp - gm;
        const V w0 = vset<V>(node_w(np)), w1 = vset<V>(node_w(np) * he(1, np)), w2 = vset<V>(node_w(np) * he(2, np)),
                w3 = vset<V>(node_w(np) * he(3, np));
        if (hi == 0) {
            S[0] = w0 * sf; S[1] = w1 * df; S[2] = w2 * sf; S[3] = w3 * df;
            SG[0] = w0 * sg; SG[1] = w1 * dg; SG[2] = w2 * sg;
        } else {
            S[0] = vfma(w0, sf, S[0]); S[1] = vfma(w1, df, S[1]); S[2] = vfma(w2, sf, S[2]); S[3] = vfma(w3, df, S[3]);
            SG[0] = vfma(w0, sg, SG[0]); SG[1] = vfma(w1, dg, SG[1]); SG[2] = vfma(w2, sg, SG[2]);
        }
    }
}

// Phi_ab += w_a S_b (f, a + b <= 3), Psi_ab += w_a SG_b (g, <= 2)
template <typename V>
__device__ __forceinline__ void add_moments(const V *w, const V *S, const V *SG, V *Phi, V *Psi)
{
#pragma unroll
    for (int a = 0; a <= 3; ++a)
#pragma unroll
        for (int b = 0; a + b <= 3; ++b) {
            Phi[hidx(a, b)] = vfma(w[a], S[b], Phi[hidx(a, b)]);
            if (a + b <= 2) Psi[hidx(a, b)] = vfma(w[a], SG[b], Psi[hidx(a, b)]);
        }
}

// the lanes for which node m does not belong to the side in hand contribute nothing
template <typename V>
__device__ __forceinline__ void mask_lanes(const unsigned *mine, int m, V *S, V *SG)
{
    if constexpr (!std::is_same<V, double>::value) {
        const bool a = (mine[0] >> m) & 1u, b = (mine[1] >> m) & 1u;
        if (a != b) {
            const int off = a ? 1 : 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) vput(S[k], off, 0.f);
#pragma unroll
            for (int k = 0; k < 3; ++k) vput(SG[k], off, 0.f);
        }
    }
}

// slots of the per-thread scratch: the side's upwind cell in the pass frame, the offsets of the
// normal and tangential nodes, and what a face carries from pass to pass (base frame, next and
// last valid frame; the base frame's words)
enum { S_U = 0, S_OFFN = 8, S_OFFT = 10, S_BN = 12, S_BT = 13, S_DL = 14, S_T = 15, S_LAST = 16, S_REF = 17, S_SLOTS = 19 };

// One corrector pass at the faces of a thread: base is cell R of the stencil in the staged
// box, sn and st the strides of the normal and tangential axes; (ln, lt) the frame velocity
// relative to the tile reference, Tl its temperature, un and ut the absolute velocity.
// Phi: f moments (hidx order), Psi: g.
template <typename V, typename SCR>
__device__ __forceinline__ void lane_pass(const LaneCell<V> *base, int dir, int sn, int st, V ln, V lt, V Tl, V un, V ut,
                                          V h_dn, V h_dt, int limiter, const SCR &scr, V *Phi, V *Psi)
{
    constexpr int L = std::is_same<V, double>::value ? 1 : 2;
    const LaneTab<V> &tab = lane_tab<V>();
    const V invTl = vrcp(Tl), rsqTl = vsqrt(invTl);
    auto move = [&](const LaneCell<V> *p, V *F, V *G) {
        const LaneWords<V> c = fetch_lane<V>(p, dir);
        const Move2<V> M(c.w[C_T], c.w[C_UN], c.w[C_UT], Tl, invTl, rsqTl, ln, lt);
        M.f(c.w[C_A00], c.w[C_A20], c.w[C_A11], c.w[C_A02], c.w[C_A30], c.w[C_A21], c.w[C_A12], c.w[C_A03], F);
        M.g(c.w[C_B00], c.w[C_B10], c.w[C_B01], c.w[C_B20], c.w[C_B11], c.w[C_B02], G);
    };
    unsigned left[L];   // the nodes upwind of the left cell, per lane (bit m)
    {
        const V sqTl = Tl * rsqTl;
        // departure offsets in cells, with the limiter's factor (2 for van Leer, 1 for minmod):
        // v h along the normal (the upwind centre's half cell is added with the side), -v h along
        // the tangent
        const V sc = vset<V>(limiter == 1 ? 1.0 : 2.0);
        const V kn = sc * h_dn, kt = vset<V>(0.0) - sc * h_dt;
        V on[4], ot[4];
#pragma unroll
        for (int l = 0; l < L; ++l) left[l] = 0u;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const V vn = vfma(sqTl, vset<V>(node_c(m)), un);
#pragma unroll
            for (int l = 0; l < L; ++l) left[l] |= vget(vn, l) > 0 ? 1u << m : 0u;
            on[m] = vn * kn;
            ot[m] = vfma(sqTl, vset<V>(node_c(m)), ut) * kt;
        }
        scr.put(S_OFFN, on[0], on[1]);
        scr.put(S_OFFN + 1, on[2], on[3]);
        scr.put(S_OFFT, ot[0], ot[1]);
        scr.put(S_OFFT + 1, ot[2], ot[3]);
    }
#pragma unroll
    for (int k = 0; k < 10; ++k) Phi[k] = vset<V>(0.0);
#pragma unroll
    for (int k = 0; k < 6; ++k) Psi[k] = vset<V>(0.0);
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {   // 0: the nodes upwind of the right cell, 1: of the left
        unsigned mine[L], any = 0u;
#pragma unroll
        for (int l = 0; l < L; ++l) {
            mine[l] = side ? left[l] : ~left[l] & 15u;
            any |= mine[l];
        }
        if (any == 0u) continue;
        const LaneCell<V> *up = side ? base - sn : base;
        {
            V UF[10], UG[6];
            move(up, UF, UG);
            scr.store(S_U, UF, UG);
        }
        // The sweep along the normal, then the one along the tangent (with the upwind cell's own
        // moments): the same code on the neighbours one stride below and above the upwind cell.
#pragma unroll 1
        for (int tang = 0; tang < 2; ++tang) {
            const int d = tang ? st : sn;
            V AF[10], AG[6], BF[10], BG[6];   // upwind minus below, above minus upwind
            move(up - d, AF, AG);
            move(up + d, BF, BG);
            {
                V UF[10], UG[6];
                scr.load(S_U, UF, UG);
#pragma unroll
                for (int k = 0; k < 10; ++k) { AF[k] = UF[k] - AF[k]; BF[k] = BF[k] - UF[k]; }
#pragma unroll
                for (int k = 0; k < 6; ++k) { AG[k] = UG[k] - AG[k]; BG[k] = BG[k] - UG[k]; }
            }
#pragma unroll 1
            for (int m = 0; m < 4; ++m) {
                if (!((any >> m) & 1u)) continue;
                const V h1 = tab.hen[m][1], h2 = tab.hen[m][2], h3 = tab.hen[m][3];
                V Ca[4], Da[3], Cb[4], Db[3], S[4], SG[3], offt[4], w[4];
                collapse(AF, AG, h1, h2, h3, Ca, Da);
                collapse(BF, BG, h1, h2, h3, Cb, Db);
                scr.get(S_OFFT, offt[0], offt[1]);
                scr.get(S_OFFT + 1, offt[2], offt[3]);
                slope_moments<V>(Ca, Da, Cb, Db, limiter, tang, offt, S, SG);
                if (tang) {
                    V UF[10], UG[6];
                    scr.load(S_U, UF, UG);
                    collapse(UF, UG, h1, h2, h3, Ca, Da);
#pragma unroll
                    for (int b = 0; b < 4; ++b) S[b] = S[b] + Ca[b];
#pragma unroll
                    for (int b = 0; b < 3; ++b) SG[b] = SG[b] + Da[b];
#pragma unroll
                    for (int a = 0; a < 4; ++a) w[a] = tab.whe[m][a];
                } else {
                    // times the departure offset along the normal, from the upwind centre
                    const double half = limiter == 1 ? 0.5 : 1.0;
                    V o0, o1;
                    scr.get(S_OFFN + (m >> 1), o0, o1);
                    const V off = vset<V>(side ? half : -half) - ((m & 1) ? o1 : o0);
#pragma unroll
                    for (int a = 0; a < 4; ++a) w[a] = tab.whe[m][a] * off;
                }
                mask_lanes<V>(mine, m, S, SG);
                add_moments(w, S, SG, Phi, Psi);
            }
        }
    }
}

// ------------------------------------------------------------ 16 lanes per face

// A pass by 16 lanes: R words of a group's part of shared memory (8 moved cells of 16 coefficients, f then
// g, padded against bank conflicts, and the 16 moments).  A pass reads 80 words a lane, and its latency is
// what a small grid with a shock waits for: in FP32 a cell moves in 16-byte accesses (interface 80 x 229
// 47.0 -> 43.9 us a launch, quadrants 49 x 583 86 -> 83.5; in FP64 it makes no difference).
template <typename R> __host__ __device__ constexpr int coop_cell() { return sizeof(R) == 4 ? 20 : 17; }
template <typename R> __host__ __device__ constexpr int coop_words() { return 8 * coop_cell<R>() + 16; }
__device__ __forceinline__ void coop_put(float *o, const float *F, const float *G)
{
    float4 *v = reinterpret_cast<float4 *>(o);
    v[0] = make_float4(F[0], F[1], F[2], F[3]);
    v[1] = make_float4(F[4], F[5], F[6], F[7]);
    v[2] = make_float4(F[8], F[9], G[0], G[1]);
    v[3] = make_float4(G[2], G[3], G[4], G[5]);
}
__device__ __forceinline__ void coop_put(double *o, const double *F, const double *G)
{
#pragma unroll
    for (int k = 0; k < 10; ++k) o[k] = F[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) o[10 + k] = G[k];
}
__device__ __forceinline__ void coop_get(const float *o, float *c)
{
    const float4 *v = reinterpret_cast<const float4 *>(o);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 x = v[k];
        c[4 * k] = x.x; c[4 * k + 1] = x.y; c[4 * k + 2] = x.z; c[4 * k + 3] = x.w;
    }
}
// Without the predictor the faces that their warps leave go to a list of the whole grid, which
// lane_tail_kernel works off, instead of to the CTA's own.
template <typename R, int MODE>
__host__ __device__ constexpr bool chip_tail() { return MODE == FACE_PLAIN; }
constexpr int kTailThreads = 128;
template <typename R> constexpr int tail_ctas() { return sizeof(R) == 8 ? 2 : 4; }

// A warp with at most this many unfinished faces hands them over.  FP32 (64 faces a warp), us a launch with
// the tail for 12 / 24 / 40 / 63: quadrants 64^2 108 / 57 / 38 / 35, 49 x 583 98 / 63 / 50 / 48, 1024^2 293 / 277 /
// 280 / 280, interface 1001 x 253 104 / 97 / 93 / 92, smooth 300^2 (two passes everywhere) 53 / 54 / 54 / 62; to
// the CTA's own list 12 (1024^2 302 / 290 / 289 for 6 / 12 / 20).  FP64 (32 faces): a pass takes 64 cycles per
// instruction however few lanes need it, so more go over, and all of them where the whole chip takes
// them (49 x 583 / 64^2 / 256^2: 884 / 495 / 994 for 20, 718 / 375 / 969 for 31; smooth 300^2 2241 and 2266).
// Smooth FP32 flows, two passes everywhere, pay for the list and are ahead of the node-by-node kernel all the
// same (us a step, cells included): 40^2 26 (27), 100^2 28 (28), 200 x 150 32 (35), 300^2 60 (75), 1024^2 488 (702).
template <typename R, int MODE>
__host__ __device__ constexpr int coop_faces() { return sizeof(R) == 4 ? (chip_tail<R, MODE>() ? 40 : 12) : (chip_tail<R, MODE>() ? 31 : 20); }
// how a face came to the list: to be passed again from its next frame, or after a pass that
// defined no frame (COOP_BAD), or after a learned prediction that did not hold (COOP_FAIL)
enum { COOP_BAD = 1, COOP_FAIL = 2, COOP_LEARNED = 4 };
struct CoopItem {
    int face, iters;   // thread | lane << 8 | COOP_* << 16; passes so far
};

// stencil slot s (0 LL, 1 L, 2 R, 3 RR, 4 L-t, 5 L+t, 6 R-t, 7 R+t) as an offset in the staged box
__device__ __forceinline__ int slot_cell(int s, int sn, int st)
{
    const int on = s < 4 ? s - 2 : (s < 6 ? -1 : 0), ot = s < 4 ? 0 : ((s & 1) ? 1 : -1);
    return on * sn + ot * st;
}

// The sum over 16 lanes of each of c[0..15]; lane q returns the sum of c[q] (q in the lane's low
// four bits; both halves of the warp at once)
template <typename R>
__device__ __forceinline__ R reduce16(R *c, int q)
{
#pragma unroll
    for (int half = 8; half >= 1; half >>= 1) {
        const bool upper = (q & half) != 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k >= half) continue;
            const R keep = upper ? c[k + half] : c[k], send = upper ? c[k] : c[k + half];
            c[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
        }
    }
    return c[0];
}

// the moments of the face populations of a finished face (hidx order, face axes) in the frame
// they define: Eq. (FluxTransf), phi = (2 tau phibar + h phi^eq)/(2 tau + h) with the exact
// co-moving equilibria there
template <typename V>
__device__ __forceinline__ void face_populations(const V *Phi, const V *Psi, V Tl, V rho, V du_n, V du_t, V T1, V wb, V we,
                                                 V Cvh, V *Fo, V *Go)
{
    const V zero = vset<V>(0.0), invT = vrcp(T1);
    const Move2<V> M(Tl, zero - du_n, zero - du_t, T1, invT, vsqrt(invT), zero, zero);
    M.f_full(Phi, Fo);
    M.g(Psi[0], Psi[1], Psi[2], Psi[3], Psi[4], Psi[5], Go);
    Fo[0] = vfma(wb, Fo[0], we * rho);
    Go[0] = vfma(wb, Go[0], we * Cvh * rho * T1);
#pragma unroll
    for (int k = 1; k < 10; ++k) Fo[k] = wb * Fo[k];
#pragma unroll
    for (int k = 1; k < 6; ++k) Go[k] = wb * Go[k];
}

// the frame of a pass's moments relative to the pass frame (Eqs. correctorfieldsrhoDUGKS-TDUGKS)
template <typename V>
__device__ __forceinline__ void moments_frame(V rho, V p10, V p01, V p20, V p02, V g0, V Tl, V sq, V Cv, V &du_n, V &du_t, V &T1)
{
    const V half = vset<V>(0.5), ir = vrcp(rho);
    du_n = sq * p10 * ir;
    du_t = sq * p01 * ir;
    const V k2 = vfma(du_n, du_n, du_t * du_t);
    const V tr = vfma(vset<V>(2.0), rho, p20 + p02);
    T1 = (vfma(half * Tl, tr, g0) - half * rho * k2) * vrcp(Cv * rho);
}

struct FaceCount {
    unsigned int iters, nonconv, fallbacks, nonphys;
};

// a warp's or a thread's counts of faces into the diagnostics
__device__ __forceinline__ void count_faces(Diag *diag, const FaceCount &fc, unsigned int solves)
{
    using U = unsigned long long;
    atomicAdd(&diag->face_iters, U(fc.iters));
    if (solves) atomicAdd(&diag->face_solves, U(solves));
    if (fc.nonconv) { atomicAdd(&diag->nonconv, U(fc.nonconv)); atomicOr(&diag->flags, FLAG_NOT_CONVERGED); }
    if (fc.fallbacks) atomicAdd(&diag->fallbacks, U(fc.fallbacks));
    if (fc.nonphys) { atomicAdd(&diag->nonphys, U(fc.nonphys)); atomicOr(&diag->flags, FLAG_NONPHYSICAL); }
}

// plane of coefficient k (hidx order, normal first) of a y-face
__host__ __device__ constexpr int lane_plane_y(int k)
{
    const int t[10] = {0, 2, 1, 5, 4, 3, 9, 8, 7, 6};
    return t[k];
}

// Population (m, n) of the lane reconstructed from the stencil cells in the pass frame (cells), and the
// 16 moments of the group's populations, one per lane; every lane of the warp calls it
template <typename R>
__device__ __forceinline__ R coop_moments(const R *cells, int q, const R *basis, const R *weight, R un, R utn, R h_dn, R h_dt, int limiter)
{
    const bool left = un > R(0);
    auto eval = [&](int s, R &f, R &g) {
        const R *c = cells + s * coop_cell<R>();
        R w[16];
        if constexpr (sizeof(R) == 4) {
            coop_get(c, w);
            c = w;
        }
        f = c[0];
        g = c[10];
#pragma unroll
        for (int k = 1; k < 10; ++k) f = vfma(c[k], basis[k], f);
#pragma unroll
        for (int k = 1; k < 6; ++k) g = vfma(c[10 + k], basis[k], g);
    };
    R fu, gu, fl, gl, fh, gh, fm, gm, fp, gp;
    eval(left ? 1 : 2, fu, gu);
    eval(left ? 0 : 1, fl, gl);
    eval(left ? 2 : 3, fh, gh);
    eval(left ? 4 : 6, fm, gm);
    eval(left ? 5 : 7, fp, gp);
    R offn = (left ? R(0.5) : R(-0.5)) - un * h_dn, offt = -utn * h_dt;
    if (limiter == 1) {
        fu = vfma(offt, vminmod(fu - fm, fp - fu), vfma(offn, vminmod(fu - fl, fh - fu), fu));
        gu = vfma(offt, vminmod(gu - gm, gp - gu), vfma(offn, vminmod(gu - gl, gh - gu), gu));
    } else {
        offn *= R(2);
        offt *= R(2);
        fu = vfma(offt, vanleer_half(fu - fm, fp - fu), vfma(offn, vanleer_half(fu - fl, fh - fu), fu));
        gu = vfma(offt, vanleer_half(gu - gm, gp - gu), vfma(offn, vanleer_half(gu - gl, gh - gu), gu));
    }
    R c[16];
#pragma unroll
    for (int k = 0; k < 10; ++k) c[k] = weight[k] * fu;
#pragma unroll
    for (int k = 0; k < 6; ++k) c[10 + k] = weight[k] * gu;
    return reduce16(c, q);
}

// Works off the CTA's list of unfinished faces, 16 lanes per face.  Lane q of a group moves
// stencil cell q (< 8) into the pass frame and evaluates population (m, n) = (q / 4, q % 4) of
// the five cells it needs; the moments are summed across the group.  The rules of the corrector
// are those of lane_face_kernel.
template <typename R, int MODE, typename VT>
__device__ __forceinline__ void coop_tail(const Params<2, R> &P, const typename FrameWords<R>::word *ut,
                                          const LaneCell<typename VecOf<R>::type> *tile, unsigned char *scratch,
                                          const CoopItem *items, int count, int *next, FaceCount &fc)
{
    using W = typename FrameWords<R>::word;
    using Cell = LaneCell<typename VecOf<R>::type>;
    constexpr int L = VecOf<R>::lanes, TX = VT::TX, TH = VT::TY / L, BX = TX + 3, NT = lane_threads<R, VT>();
    constexpr bool LEARNED = MODE == FACE_LEARNED;
    const unsigned full = 0xffffffffu;
    const int q = threadIdx.x & 15, lead = threadIdx.x & 16, m = q >> 2, n = q & 3;
    R *cells = reinterpret_cast<R *>(scratch) + (threadIdx.x >> 4) * coop_words<R>(), *mom = cells + 8 * coop_cell<R>();
    const StepC<R> &KC = step_c<R>(*P.clock);
    const NodeTab<R> &tab = node_tab<R>();
    const R Cv = P.Cv_r, tol = P.tol_r, cm = tab.c[m], cn = tab.c[n];
    // He_a(c_m) He_b(c_n)/(a! b!) and w_m w_n He_a(c_m) He_b(c_n), a + b <= 3
    R basis[10], weight[10];
#pragma unroll
    for (int a = 0; a <= 3; ++a)
#pragma unroll
        for (int b = 0; a + b <= 3; ++b) {
            basis[hidx(a, b)] = tab.hen[m][a] * tab.hen[n][b];
            weight[hidx(a, b)] = tab.whe[m][a] * tab.whe[n][b];
        }
    // the face in hand
    int dir = 0, l = 0, iters = 0, tot_iters = 0, fallbacks = 0, tot_fallbacks = 0, flags = 0;
    long long fidx = 0, nf = 0;
    const Cell *base = tile + 2 * BX + 2;   // (a group without a face passes over a cell inside the box)
    R bn = R(0), bna = R(0), bt = R(0), bta = R(0), dn = R(0), dt = R(0), Tl = R(1), vn = R(0), vt = R(0), vT = R(1);
    bool live = false, have = false, done = false, restarted = false, redo = false;
    W *Frm = P.xfr;
    long long ptile = 0;
    auto take = [&]() {
        int item = 0;
        if (q == 0) item = atomicAdd(next, 1);
        item = __shfl_sync(lead ? 0xffff0000u : 0x0000ffffu, item, lead);
        live = item < count;
        if (!live) return;
        const CoopItem it = items[item];
        const int t = it.face & 255;
        l = (it.face >> 8) & 1;
        flags = it.face >> 16;
        iters = it.iters;
        tot_iters = tot_fallbacks = 0;
        fallbacks = (flags & COOP_BAD) ? 1 : 0;
        have = !(flags & COOP_BAD) || iters > 1;
        done = restarted = redo = false;
        dir = t >= TX * TH ? 1 : 0;
        const int tid = t - dir * TX * TH, tx = tid % TX, ty = tid / TX;
        const long long fi = (long long)blockIdx.x * TX + tx, fj = (long long)blockIdx.y * VT::TY + ty + l * TH;
        nf = dir == 0 ? P.nxf() : P.nyf();
        fidx = fj * (dir == 0 ? P.nx + 1 : P.nx) + fi;
        Frm = dir == 0 ? P.xfr : P.yfr;
        if constexpr (LEARNED) ptile = (fj / kPredTileY) * ((P.nx + 1 + kPredTileX - 1) / kPredTileX) + fi / kPredTileX;
        base = &tile[(ty + 2) * BX + tx + 2];
        auto word = [&](int slot, int second) {
            return reinterpret_cast<const R *>(scratch + (size_t(slot) * NT + t) * 16)[second * L + l];
        };
        bn = word(S_BN, 0); bna = word(S_BN, 1);
        bt = word(S_BT, 0); bta = word(S_BT, 1);
        dn = word(S_DL, 0); dt = word(S_DL, 1);
        Tl = word(S_T, 0); vT = word(S_T, 1);
        vn = word(S_LAST, 0); vt = word(S_LAST, 1);
    };
    take();
    for (;;) {
        __syncwarp();
        if (!__any_sync(full, live)) break;
        const int sn = dir == 0 ? 1 : BX, st = dir == 0 ? BX : 1;
        if (live && (flags & (COOP_BAD | COOP_FAIL))) {
            if (LEARNED && (flags & COOP_FAIL)) {
                // the prediction did not hold: solve from the previous half step's frame
                tot_iters += iters;
                tot_fallbacks += fallbacks;
                const W u0 = Frm[fidx], u1 = Frm[nf + fidx];
                bn = R(fr_rel(dir ? u1 : u0, dir ? ut[1] : ut[0]));
                bt = R(fr_rel(dir ? u0 : u1, dir ? ut[0] : ut[1]));
                bna = R(fr_lead(dir ? u1 : u0));
                bta = R(fr_lead(dir ? u0 : u1));
                Tl = R(fr_lead(Frm[2 * nf + fidx]));
                dn = dt = R(0);
                iters = fallbacks = 0;
                have = done = restarted = false;
                flags = 0;
            } else {
                flags &= ~COOP_BAD;
                if (!restarted && iters < P.max_iter) {
                    // once: the frame of the pooled conserved moments of the eight stencil cells
                    restarted = true;
                    R r = R(0), mn = R(0), mt = R(0), e = R(0);
#pragma unroll 1
                    for (int s = 0; s < 8; ++s) {
                        const Cell *c = base + slot_cell(s, sn, st);
                        const R rc = vget(c->sym[0], l), u = vget(c->ax[dir][5], l) - bn, w = vget(c->ax[1 - dir][5], l) - bt;
                        r += rc;
                        mn += rc * u;
                        mt += rc * w;
                        e += rc * (Cv * vget(c->sym[4], l) + R(0.5) * (u * u + w * w));
                    }
                    r /= R(8); mn /= R(8); mt /= R(8); e /= R(8);
                    dn = mn / r;
                    dt = mt / r;
                    Tl = (e - R(0.5) * (mn * mn + mt * mt) / r) / (Cv * r);
                } else {
                    // stopped by a pass without a frame: the last valid one over again, if any
                    redo = true;
                    dn = vn;
                    dt = vt;
                    Tl = vT;
                }
            }
        }
        // ---- the pass
        const R invTl = vrcp(Tl), rsqTl = vsqrt(invTl), sqTl = Tl * rsqTl, sq = vsqrt(Tl);
        if (q < 8) {
            const R *c = reinterpret_cast<const R *>(base + slot_cell(q, sn, st)) + l;
            const R *cx = c + (1 + dir) * 6 * L, *cy = c + (2 - dir) * 6 * L;   // normal and tangential groups
            const Move2<R> M(c[4 * L], cx[5 * L], cy[5 * L], Tl, invTl, rsqTl, bn + dn, bt + dt);
            R F[10], G[6];
            M.f(c[0], cx[0], c[L], cy[0], cx[L], cx[2 * L], cy[2 * L], cy[L], F);
            M.g(c[2 * L], cx[3 * L], cy[3 * L], cx[4 * L], c[3 * L], cy[4 * L], G);
            coop_put(cells + q * coop_cell<R>(), F, G);
        }
        __syncwarp();
        const R un = vfma(sqTl, cm, bna + dn), utn = vfma(sqTl, cn, bta + dt);
        mom[q] = coop_moments<R>(cells, q, basis, weight, un, utn, dir ? KC.h_dy : KC.h_dx, dir ? KC.h_dx : KC.h_dy, P.limiter);
        __syncwarp();
        R rho = mom[0], du_n, du_t, T1;
        moments_frame<R>(rho, mom[1], mom[2], mom[3], mom[5], mom[10], Tl, sq, Cv, du_n, du_t, T1);
        if (!live) continue;
        bool finished = redo;
        if (!redo) {
            ++iters;
            const bool ok = T1 > R(0) && isfinite(T1) && isfinite(rho) && isfinite(du_n) && isfinite(du_t);
            if (ok) {
                have = true;
                vn = dn;
                vt = dt;
                vT = Tl;
                if (P.fixed_iters > 0) done = iters >= P.fixed_iters;
                else done = fabs(T1 - Tl) <= tol * Tl && fabs(du_n) <= tol * sq && fabs(du_t) <= tol * sq;
                finished = done || iters >= P.max_iter;
                if (LEARNED && (flags & COOP_LEARNED) && finished && !(done && fallbacks == 0)) {
                    finished = false;
                    flags |= COOP_FAIL;
                } else if (!finished) {
                    dn += du_n;
                    dt += du_t;
                    Tl = T1;
                }
            } else {
                ++fallbacks;
                if (LEARNED && (flags & COOP_LEARNED) && (restarted || iters >= P.max_iter)) flags |= COOP_FAIL;
                else if (!have && (restarted || iters >= P.max_iter)) finished = true;
                else flags |= COOP_BAD;
            }
        }
        if (!finished) continue;
        // ---- the face's result
        R *Fout = dir == 0 ? P.xf : P.yf, *Gout = dir == 0 ? P.xg : P.yg;
        const unsigned half = lead ? 0xffff0000u : 0x0000ffffu;
        R v = R(__longlong_as_double(0x7ff8000000000000ll));
        if (have) {
            R Phi[10], Psi[6], Fo[10], Go[6];
#pragma unroll
            for (int k = 0; k < 10; ++k) Phi[k] = mom[k];
#pragma unroll
            for (int k = 0; k < 6; ++k) Psi[k] = mom[10 + k];
            face_populations<R>(Phi, Psi, Tl, rho, du_n, du_t, T1, KC.wb, KC.we, P.Cvh_r, Fo, Go);
            __syncwarp(half);
            if (q == 0) {
#pragma unroll
                for (int k = 0; k < 10; ++k) mom[k] = Fo[k];
#pragma unroll
                for (int k = 0; k < 6; ++k) mom[10 + k] = Go[k];
                W b0 = Frm[fidx], b1 = Frm[nf + fidx];
                if constexpr (LEARNED) {
                    if (flags & COOP_LEARNED) {
                        const W *Lrm = dir == 0 ? P.xlr : P.ylr;
                        b0 = Lrm[fidx];
                        b1 = Lrm[nf + fidx];
                    }
                }
                const R fn = dn + du_n, ft = dt + du_t;
                Frm[fidx] = fr_add(b0, dir ? ft : fn);
                Frm[nf + fidx] = fr_add(b1, dir ? fn : ft);
                Frm[2 * nf + fidx] = fr_word(T1);
            }
            __syncwarp(half);
            v = mom[q];
        } else if (q == 0) {
            fr_store(Frm[2 * nf + fidx], double(v));
        }
        {
            const int k = q < 10 ? q : q - 10;
            int pl = k;
            if (dir) pl = k == 0 || k == 4 ? k : (k < 3 ? 3 - k : (k < 6 ? 8 - k : 15 - k));   // axes exchanged
            (q < 10 ? Fout : Gout)[pl * nf + fidx] = v;
        }
        if (q == 0) {
            tot_iters += iters;
            tot_fallbacks += fallbacks;
            fc.iters += tot_iters;
            fc.fallbacks += tot_fallbacks;
            fc.nonconv += done ? 0 : 1;
            fc.nonphys += have ? 0 : 1;
            if constexpr (LEARNED) {
                if (P.use_learned) {   // the face took more than one pass
                    const unsigned int nx = (unsigned int)P.clock->steps + 1u;
                    P.pred_active[(nx & 1u) * pred_tiles(P) + ptile] = nx;
                }
            }
        }
        take();
    }
}

// ------------------------------------------------------------ the face kernel of a step

// phi-bar-plus of cell idx (inside the grid) as lane l of a staged pair; 32-bit plane offsets
template <typename R, typename V>
__device__ __forceinline__ void stage_inside(const Params<2, R> &P, unsigned int idx, R cp, R ce,
                                             const typename FrameWords<R>::word *ut, int l, LaneCell<V> &c)
{
    const long long n = P.ncell();
    R f[8], g[6];
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = (P.sf + k * n)[idx];
#pragma unroll
    for (int k = 0; k < 6; ++k) g[k] = (P.sg + k * n)[idx];
    const auto u0 = P.sfr[idx], u1 = (P.sfr + n)[idx], T_ = (P.sfr + 2 * n)[idx];
    const R T = R(fr_lead(T_)), r = f[0];
    vput(c.sym[0], l, cp * r + ce * r);
    vput(c.ax[0][0], l, cp * f[1]); vput(c.sym[1], l, cp * f[2]); vput(c.ax[1][0], l, cp * f[3]);
    vput(c.ax[0][1], l, cp * f[4]); vput(c.ax[0][2], l, cp * f[5]); vput(c.ax[1][2], l, cp * f[6]); vput(c.ax[1][1], l, cp * f[7]);
    vput(c.sym[2], l, cp * g[0] + ce * (P.Cvh_r * r * T));
    vput(c.ax[0][3], l, cp * g[1]); vput(c.ax[1][3], l, cp * g[2]);
    vput(c.ax[0][4], l, cp * g[3]); vput(c.sym[3], l, cp * g[4]); vput(c.ax[1][4], l, cp * g[5]);
    vput(c.sym[4], l, T); vput(c.sym[5], l, R(0));
    vput(c.ax[0][5], l, R(fr_rel(u0, ut[0]))); vput(c.ax[1][5], l, R(fr_rel(u1, ut[1])));
}
// the same with the ghost rules
template <typename R, typename V>
__device__ __forceinline__ void stage_any(const Params<2, R> &P, long long i, long long j, R cp, R ce,
                                          const typename FrameWords<R>::word *ut, int l, LaneCell<V> &c)
{
    StagedCell<2, R> q;
    load_cell_bar_plus<2, R>(P, i, j, cp, ce, ut, q);
    vput(c.sym[0], l, q.A[0]); vput(c.sym[1], l, q.A[hidx(1, 1)]);
    vput(c.sym[2], l, q.B[0]); vput(c.sym[3], l, q.B[hidx(1, 1)]);
    vput(c.sym[4], l, q.T); vput(c.sym[5], l, R(0));
    vput(c.ax[0][0], l, q.A[hidx(2, 0)]); vput(c.ax[1][0], l, q.A[hidx(0, 2)]);
    vput(c.ax[0][1], l, q.A[hidx(3, 0)]); vput(c.ax[1][1], l, q.A[hidx(0, 3)]);
    vput(c.ax[0][2], l, q.A[hidx(2, 1)]); vput(c.ax[1][2], l, q.A[hidx(1, 2)]);
    vput(c.ax[0][3], l, q.B[hidx(1, 0)]); vput(c.ax[1][3], l, q.B[hidx(0, 1)]);
    vput(c.ax[0][4], l, q.B[hidx(2, 0)]); vput(c.ax[1][4], l, q.B[hidx(0, 2)]);
    vput(c.ax[0][5], l, q.du[0]); vput(c.ax[1][5], l, q.du[1]);
}

// Per face the rules of the corrector are those of solve_face (pond_kernels.cuh): passes run until
// the frame converges; a pass whose moments define no frame restarts the corrector once from the
// pooled moments of the stencil, then stops it at the last pass that did.  With the learned
// predictor a face starts from its prediction and, unless that converges without a restart,
// again from the previous half step's frame.  The warp's own passes only ever go forward;
// whatever else happens to a face (and what few faces are left) goes to coop_tail.  A face that is
// done keeps its last frame while the warp goes on, so its moments stay what they were.
template <typename R, int MODE, typename VT>
__global__ void __launch_bounds__(lane_threads<R, VT>(), VT::MINB)
lane_face_kernel(const Params<2, R> P)
{
    using V = typename VecOf<R>::type;
    using W = typename FrameWords<R>::word;
    constexpr int L = VecOf<R>::lanes;
    constexpr bool LEARNED = MODE == FACE_LEARNED, CHIP = chip_tail<R, MODE>();
    constexpr int TX = VT::TX, TY = VT::TY, TH = TY / L;   // TH rows of threads; lane l is TH rows up
    constexpr int BX = TX + 3, BH = TH + 3, NT = lane_threads<R, VT>();
    static_assert(TY % L == 0 && (TX * TH) % 32 == 0 && NT <= 256, "whole warps per face direction");
    extern __shared__ __align__(16) unsigned char lane_smem[];   // the staged box, then the scratch
    LaneCell<V> *tile = reinterpret_cast<LaneCell<V> *>(lane_smem);
    unsigned char *scratch = lane_smem + sizeof(LaneCell<V>) * BH * BX;
    using Scr = LaneScratch<V, NT>;
    const Scr scr{(unsigned)__cvta_generic_to_shared(scratch) + threadIdx.x * 16u};
    __shared__ CoopItem items[CHIP ? 1 : NT * L];
    __shared__ int n_items, next_item;
    if (threadIdx.x == 0) n_items = next_item = 0;
    unsigned int n_act = 0;   // faces finished by the warp itself, or listed for the grid's tail

    const Clock &K = *P.clock;
    const double step_dt = K.dt;   // 0: t_end reached, the step is a no-op (tested after the staging loads)
    const StepC<R> &KC = step_c<R>(K);
    const R cp = KC.cp, ce = KC.ce;
    const long long i0 = (long long)blockIdx.x * TX, j0 = (long long)blockIdx.y * TY;

    // the faces of this thread
    const int dir = threadIdx.x >= TX * TH ? 1 : 0;
    const int tid = threadIdx.x - dir * TX * TH, tx = tid % TX, ty = tid / TX;
    const long long fi = i0 + tx;
    const long long nf = dir == 0 ? P.nxf() : P.nyf();
    W *Frm = dir == 0 ? P.xfr : P.yfr;
    auto face = [&](int l) { return (j0 + ty + l * TH) * (dir == 0 ? P.nx + 1 : P.nx) + fi; };
    bool active[L];
    W uref[L][2], Tpw[L];   // the predictor frame, loaded before the staging so that the loads overlap
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const long long fj = j0 + ty + l * TH;
        active[l] = dir == 0 ? fi <= P.nx && fj < P.ny : fi < P.nx && fj <= P.ny;
#pragma unroll
        for (int a = 0; a < 2; ++a) uref[l][a] = active[l] ? Frm[a * nf + face(l)] : fr_word(R(0));
        Tpw[l] = active[l] ? Frm[2 * nf + face(l)] : fr_word(R(1));
    }
    W ut[2];   // reference velocity of the tile (staged velocities are differences from it)
    cell_velocity<2, R>(P, i0, j0, ut);
    // box [i0-2, i0+TX] x [j0-2, j0+TY]; without ghosts (and with 32-bit offsets) in the interior
    const bool inside = i0 >= 2 && i0 + TX < P.nx && j0 >= 2 && j0 + TY < P.ny && P.ncell() < (1ll << 31);
    for (int s = threadIdx.x; s < BX * BH; s += NT) {
        const int bx = s % BX, by = s / BX;
        LaneCell<V> c;
        if (inside) {
            const unsigned int at = (unsigned int)((j0 - 2 + by) * P.nx + i0 - 2 + bx);
#pragma unroll
            for (int l = 0; l < L; ++l) stage_inside<R, V>(P, at + l * TH * (unsigned int)P.nx, cp, ce, ut, l, c);
        } else {
#pragma unroll
            for (int l = 0; l < L; ++l) stage_any<R, V>(P, i0 - 2 + bx, j0 - 2 + by + l * TH, cp, ce, ut, l, c);
        }
        tile[s] = c;
    }
    if (!(step_dt > 0.0)) return;   // the same value in every thread
    __syncthreads();

    const LaneCell<V> *base = &tile[(ty + 2) * BX + tx + 2];
    const int sn = dir == 0 ? 1 : BX, st = dir == 0 ? BX : 1;
    const R Cv = P.Cv_r, tol = P.tol_r;
    auto pred_tile = [&](int l) {
        return ((j0 + ty + l * TH) / kPredTileY) * ((P.nx + 1 + kPredTileX - 1) / kPredTileX) + fi / kPredTileX;
    };

    // What a face carries from pass to pass waits in the scratch: the base frame (S_BN, S_BT: normal
    // and tangential velocity, relative to the tile reference and absolute), the frame of the next
    // pass relative to it (S_DL, S_T) and that of the last valid pass (S_LAST, S_T).
    bool run[L], done[L], learned[L];
    int iters[L];
    {
        V bn, bna, bt, bta, T0;
        W base_w[L][2];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            run[l] = active[l];
            done[l] = learned[l] = false;
            iters[l] = 0;
            W u[2] = {uref[l][0], uref[l][1]};
            R T = R(fr_lead(Tpw[l]));
            if constexpr (LEARNED) {
                // the learned prediction of the face, if the predictor ran there and made one
                const unsigned int step = (unsigned int)K.steps;
                if (active[l] && P.use_learned && P.pred_active[(step & 1u) * pred_tiles(P) + pred_tile(l)] == step) {
                    const W *Lrm = dir == 0 ? P.xlr : P.ylr;
                    const R lT = R(fr_lead(Lrm[2 * nf + face(l)]));
                    if (lT > R(0) && isfinite(lT)) {
                        learned[l] = true;
                        u[0] = Lrm[face(l)];
                        u[1] = Lrm[nf + face(l)];
                        T = lT;
                    }
                }
            }
            base_w[l][0] = u[0];
            base_w[l][1] = u[1];
            vput(bn, l, R(fr_rel(dir ? u[1] : u[0], dir ? ut[1] : ut[0])));
            vput(bt, l, R(fr_rel(dir ? u[0] : u[1], dir ? ut[0] : ut[1])));
            vput(bna, l, R(fr_lead(dir ? u[1] : u[0])));
            vput(bta, l, R(fr_lead(dir ? u[0] : u[1])));
            vput(T0, l, T);
        }
        scr.put(S_BN, bn, bna);
        scr.put(S_BT, bt, bta);
        scr.put(S_DL, vset<V>(0.0), vset<V>(0.0));
        scr.put(S_T, T0, T0);
        scr.put(S_LAST, vset<V>(0.0), vset<V>(0.0));
        W *ref = reinterpret_cast<W *>(scratch + (S_REF * NT + threadIdx.x) * 16);   // lane l: slot S_REF + l
#pragma unroll
        for (int l = 0; l < L; ++l) {
            ref[l * NT * (16 / int(sizeof(W)))] = base_w[l][0];
            ref[l * NT * (16 / int(sizeof(W))) + 1] = base_w[l][1];
        }
    }
    V Phi[10], Psi[6], rho, du_n, du_t, T1, dn, dt, Tl;
    for (;;) {
        {
            V rn, un, rt, utg, vT;
            scr.get(S_BN, rn, un);
            scr.get(S_BT, rt, utg);
            scr.get(S_DL, dn, dt);
            scr.get(S_T, Tl, vT);
            lane_pass<V>(base, dir, sn, st, rn + dn, rt + dt, Tl, un + dn, utg + dt, vbc(dir ? KC.h_dy : KC.h_dx),
                         vbc(dir ? KC.h_dx : KC.h_dy), P.limiter, scr, Phi, Psi);
        }
        V vT, vn, vt;
        scr.get(S_T, Tl, vT);
        scr.get(S_DL, dn, dt);
        scr.get(S_LAST, vn, vt);
        const V sq = vsqrt(Tl);
        rho = Phi[0];
        moments_frame<V>(rho, Phi[1], Phi[2], Phi[3], Phi[5], Psi[0], Tl, sq, vbc(Cv), du_n, du_t, T1);
        V nn = dn, nt = dt, nT = Tl;   // the next pass's frame
        int flags[L];                  // COOP_* of a face that leaves for the list, else -1
#pragma unroll
        for (int l = 0; l < L; ++l) {
            flags[l] = -1;
            if (!run[l]) continue;
            const R T = vget(T1, l), T0 = vget(Tl, l), r1 = vget(rho, l), dun = vget(du_n, l), dut = vget(du_t, l);
            ++iters[l];
            const bool ok = T > R(0) && isfinite(T) && isfinite(r1) && isfinite(dun) && isfinite(dut);
            if (ok) {
                if (P.fixed_iters > 0) {
                    done[l] = iters[l] >= P.fixed_iters;
                } else {
                    const R s = tol * vget(sq, l);
                    done[l] = fabs(T - T0) <= tol * T0 && fabs(dun) <= s && fabs(dut) <= s;
                }
                vput(vn, l, vget(dn, l));
                vput(vt, l, vget(dt, l));
                vput(vT, l, T0);
                run[l] = !done[l] && iters[l] < P.max_iter;
                if (run[l]) {
                    vput(nn, l, vget(dn, l) + dun);
                    vput(nt, l, vget(dt, l) + dut);
                    vput(nT, l, T);
                } else if (LEARNED && learned[l] && !done[l]) {
                    flags[l] = COOP_FAIL | COOP_LEARNED;
                }
            } else {
                run[l] = false;
                flags[l] = COOP_BAD | (LEARNED && learned[l] ? COOP_LEARNED : 0);
            }
        }
        unsigned left_over = __popc(__ballot_sync(0xffffffffu, run[0]));
        if constexpr (L > 1) left_over += __popc(__ballot_sync(0xffffffffu, run[L - 1]));
        const bool go_on = left_over > coop_faces<R, MODE>();
        bool store = go_on;
#pragma unroll
        for (int l = 0; l < L; ++l) {
            if (!go_on && run[l]) flags[l] = LEARNED && learned[l] ? COOP_LEARNED : 0;
            if (flags[l] < 0) continue;
            store = true;
            active[l] = false;   // finished by the tail
            if constexpr (!CHIP) items[atomicAdd(&n_items, 1)] = {int(threadIdx.x) | (l << 8) | (flags[l] << 16), iters[l]};
        }
        if constexpr (CHIP) {
            // the face's frames go into its own output planes, then it takes a place in the list
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const unsigned lists = __ballot_sync(0xffffffffu, flags[l] >= 0);
                if (!lists) continue;
                unsigned at = 0;
                if ((threadIdx.x & 31) == 0) at = atomicAdd(&P.tail->n, __popc(lists));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(lists & ((1u << (threadIdx.x & 31)) - 1u));
                if (flags[l] >= 0) {
                    const long long f = face(l);
                    R *o = (dir == 0 ? P.xf : P.yf) + f;
                    o[0] = vget(nn, l); o[nf] = vget(nt, l); o[2 * nf] = vget(vn, l); o[3 * nf] = vget(vt, l);
                    o[4 * nf] = vget(nT, l); o[5 * nf] = vget(vT, l); o[6 * nf] = R(iters[l]);
                    P.tail_items()[at] = (unsigned long long)f | (unsigned long long)dir << kTailDirShift | (flags[l] & COOP_BAD ? kTailBad : 0ull);
                    ++n_act;
                }
            }
        }
        if (store) {
            scr.put(S_DL, nn, nt);
            scr.put(S_T, nT, vT);
            scr.put(S_LAST, vn, vt);
        }
        if (!go_on) break;
    }
    FaceCount fc{0, 0, 0, 0};
    bool write = false;
#pragma unroll
    for (int l = 0; l < L; ++l) {
        if (!active[l]) continue;
        write = true;
        ++n_act;
        fc.iters += iters[l];
        fc.nonconv += done[l] ? 0 : 1;
        if constexpr (LEARNED) {
            if (P.use_learned && (iters[l] > 1 || learned[l])) {
                const unsigned int next = (unsigned int)K.steps + 1u;
                P.pred_active[(next & 1u) * pred_tiles(P) + pred_tile(l)] = next;
            }
        }
    }
    if (write) {
        V Fo[10], Go[6];
        face_populations<V>(Phi, Psi, Tl, rho, du_n, du_t, T1, vbc(KC.wb), vbc(KC.we), vbc(P.Cvh_r), Fo, Go);
        const V fn = dn + du_n, ft = dt + du_t;   // the face frame, relative to the base frame
        R *Fout = dir == 0 ? P.xf : P.yf, *Gout = dir == 0 ? P.xg : P.yg;
#pragma unroll
        for (int l = 0; l < L; ++l) {
            if (!active[l]) continue;
            const long long f = face(l);
#pragma unroll
            for (int k = 0; k < 10; ++k) (Fout + (dir ? lane_plane_y(k) : k) * nf)[f] = vget(Fo[k], l);
#pragma unroll
            for (int k = 0; k < 6; ++k) (Gout + (dir ? lane_plane_y(k) : k) * nf)[f] = vget(Go[k], l);
            const W *b = reinterpret_cast<const W *>(scratch + ((S_REF + l) * NT + threadIdx.x) * 16);   // the base frame
            Frm[f] = fr_add(b[0], vget(dir ? ft : fn, l));
            Frm[nf + f] = fr_add(b[1], vget(dir ? fn : ft, l));
            Frm[2 * nf + f] = fr_word(vget(T1, l));
        }
    }
    int count = 0;
    if constexpr (!CHIP) {
        __syncthreads();
        count = n_items;
        if (count > 0) coop_tail<R, MODE, VT>(P, ut, tile, scratch, items, count, &next_item, fc);
    }
    fc.iters = warp_sum_count(fc.iters);
    fc.nonconv = warp_sum_count(fc.nonconv);
    fc.fallbacks = warp_sum_count(fc.fallbacks);
    fc.nonphys = warp_sum_count(fc.nonphys);
    if (threadIdx.x == 0) n_act += count;
    n_act = warp_sum_count(n_act);
    if ((threadIdx.x & 31) == 0 && (n_act || fc.iters)) count_faces(P.diag, fc, n_act);
}

// Works off the grid's list of unfinished faces, 16 lanes per face and two faces a warp: the form
// of coop_tail, with lane q < 8 holding stencil cell q in registers and velocities relative to the face's
// own predictor frame.  Faces that take many passes lie together (a shock crosses a few tiles), so a CTA's
// own list keeps a few SMs busy while the others are done: the grid's list spreads them over the
// chip.  Measured (GB300, us a launch of face and tail; before: each CTA its own list): FP64 quadrants 256^2 981
// (1310), 64^2 367 (1007), 49 x 583 724 (1117), interface 401 x 201 1074 (1388), smooth 300^2 2292 (2222); FP32
// quadrants 64^2 36 (81), 49 x 583 46 (76), 300^2 55 (107), 1024^2 280 (290), interface 1001 x 253 93 (110).
// Two CTAs per SM in FP64 (three: 5% slower), four in FP32 (two: 7% slower at 1024^2).  Two warps a face, f and g
// apart, halve the chain of a pass but cost twice the issue: FP64 850 at 49 x 583, 1105 at 256^2.
template <typename R>
__global__ void __launch_bounds__(kTailThreads)
lane_tail_kernel(const Params<2, R> P)
{
    using W = typename FrameWords<R>::word;
    __shared__ __align__(16) R words[kTailThreads / 16][coop_words<R>()];
    const unsigned full = 0xffffffffu;
    const int q = threadIdx.x & 15, lead = threadIdx.x & 16, m = q >> 2, n = q & 3;
    R *cells = words[threadIdx.x >> 4], *mom = cells + 8 * coop_cell<R>();
    // The first face of a group goes by its place (the groups of different CTAs first), the others by a
    // ticket: a CTA without a face leaves at once, and a short list costs no atomics.
    const unsigned int count = P.tail->n, groups = gridDim.x * (kTailThreads / 16);
    if (blockIdx.x >= count) return;
    const StepC<R> &KC = step_c<R>(*P.clock);
    const NodeTab<R> &tab = node_tab<R>();
    const R Cv = P.Cv_r, tol = P.tol_r, cm = tab.c[m], cn = tab.c[n];
    R basis[10], weight[10];   // as in coop_tail
#pragma unroll
    for (int a = 0; a <= 3; ++a)
#pragma unroll
        for (int b = 0; a + b <= 3; ++b) {
            basis[hidx(a, b)] = tab.hen[m][a] * tab.hen[n][b];
            weight[hidx(a, b)] = tab.whe[m][a] * tab.whe[n][b];
        }
    FaceCount fc{0, 0, 0, 0};
    int dir = 0, iters = 0, fallbacks = 0;
    long long f = 0, nf = 0;
    LaneCell<R> cell{};
    cell.sym[4] = R(1);   // (a group without a face passes over a cell at rest)
    W ref[2] = {};
    R una = R(0), uta = R(0), dn = R(0), dt = R(0), Tl = R(1), vn = R(0), vt = R(0), vT = R(1);
    bool live = false, have = false, done = false, restarted = false, redo = false, bad = false;
    auto take = [&](unsigned int item) {
        live = item < count;
        if (!live) return;
        const unsigned long long it = P.tail_items()[item];
        dir = int(it >> kTailDirShift) & 1;
        f = (long long)(it & ((1ull << kTailDirShift) - 1));
        bad = (it & kTailBad) != 0;
        nf = dir == 0 ? P.nxf() : P.nyf();
        const long long w = dir == 0 ? P.nx + 1 : P.nx, fj = f / w, fi = f - fj * w;
        const R *o = (dir == 0 ? P.xf : P.yf) + f;
        dn = o[0]; dt = o[nf]; vn = o[2 * nf]; vt = o[3 * nf]; Tl = o[4 * nf]; vT = o[5 * nf];
        iters = int(o[6 * nf]);
        fallbacks = bad ? 1 : 0;
        have = !bad || iters > 1;
        done = restarted = redo = false;
        const W *Frm = dir == 0 ? P.xfr : P.yfr;
        ref[0] = Frm[f];
        ref[1] = Frm[nf + f];
        una = R(fr_lead(dir ? ref[1] : ref[0]));
        uta = R(fr_lead(dir ? ref[0] : ref[1]));
        if (q < 8) {
            const int on = q < 4 ? q - 2 : (q < 6 ? -1 : 0), ot = q < 4 ? 0 : ((q & 1) ? 1 : -1);
            stage_any<R, R>(P, fi + (dir ? ot : on), fj + (dir ? on : ot), KC.cp, KC.ce, ref, 0, cell);
            // in face axes
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const R x = cell.ax[0][k], y = cell.ax[1][k];
                cell.ax[0][k] = dir ? y : x;
                cell.ax[1][k] = dir ? x : y;
            }
        }
    };
    take((threadIdx.x >> 4) * gridDim.x + blockIdx.x);
    for (;;) {
        __syncwarp();
        if (!__any_sync(full, live)) break;
        // once: the frame of the pooled conserved moments of the eight stencil cells (every lane sums)
        R r = cell.sym[0], mn = r * cell.ax[0][5], mt = r * cell.ax[1][5];
        R e = r * (Cv * cell.sym[4] + R(0.5) * (cell.ax[0][5] * cell.ax[0][5] + cell.ax[1][5] * cell.ax[1][5]));
        if (__any_sync(full, live && bad)) {
#pragma unroll
            for (int s = 1; s < 8; s <<= 1) {
                r += __shfl_xor_sync(full, r, s);
                mn += __shfl_xor_sync(full, mn, s);
                mt += __shfl_xor_sync(full, mt, s);
                e += __shfl_xor_sync(full, e, s);
            }
            const int from = lead;   // the sums of lanes 0 .. 7 of the group
            r = __shfl_sync(full, r, from) * R(0.125);
            mn = __shfl_sync(full, mn, from) * R(0.125);
            mt = __shfl_sync(full, mt, from) * R(0.125);
            e = __shfl_sync(full, e, from) * R(0.125);
        }
        if (live && bad) {
            bad = false;
            if (!restarted && iters < P.max_iter) {
                restarted = true;
                dn = mn / r;
                dt = mt / r;
                Tl = (e - R(0.5) * (mn * mn + mt * mt) / r) / (Cv * r);
            } else {
                // stopped by a pass without a frame: the last valid one over again, if any
                redo = true;
                dn = vn;
                dt = vt;
                Tl = vT;
            }
        }
        // ---- the pass
        const R invTl = vrcp(Tl), rsqTl = vsqrt(invTl), sqTl = Tl * rsqTl, sq = vsqrt(Tl);
        if (q < 8) {
            const R *cx = cell.ax[0], *cy = cell.ax[1];
            const Move2<R> M(cell.sym[4], cx[5], cy[5], Tl, invTl, rsqTl, dn, dt);
            R F[10], G[6];
            M.f(cell.sym[0], cx[0], cell.sym[1], cy[0], cx[1], cx[2], cy[2], cy[1], F);
            M.g(cell.sym[2], cx[3], cy[3], cx[4], cell.sym[3], cy[4], G);
            coop_put(cells + q * coop_cell<R>(), F, G);
        }
        __syncwarp();
        mom[q] = coop_moments<R>(cells, q, basis, weight, vfma(sqTl, cm, una + dn), vfma(sqTl, cn, uta + dt),
                                 dir ? KC.h_dy : KC.h_dx, dir ? KC.h_dx : KC.h_dy, P.limiter);
        __syncwarp();
        R rho = mom[0], du_n, du_t, T1;
        moments_frame<R>(rho, mom[1], mom[2], mom[3], mom[5], mom[10], Tl, sq, Cv, du_n, du_t, T1);
        if (!live) continue;
        bool finished = redo;
        if (!redo) {
            ++iters;
            const bool ok = T1 > R(0) && isfinite(T1) && isfinite(rho) && isfinite(du_n) && isfinite(du_t);
            if (ok) {
                have = true;
                vn = dn;
                vt = dt;
                vT = Tl;
                if (P.fixed_iters > 0) done = iters >= P.fixed_iters;
                else done = fabs(T1 - Tl) <= tol * Tl && fabs(du_n) <= tol * sq && fabs(du_t) <= tol * sq;
                finished = done || iters >= P.max_iter;
                if (!finished) {
                    dn += du_n;
                    dt += du_t;
                    Tl = T1;
                }
            } else {
                ++fallbacks;
                if (!have && (restarted || iters >= P.max_iter)) finished = true;
                else bad = true;
            }
        }
        if (!finished) continue;
        // ---- the face's result
        R *Fout = dir == 0 ? P.xf : P.yf, *Gout = dir == 0 ? P.xg : P.yg;
        W *Frm = dir == 0 ? P.xfr : P.yfr;
        const unsigned half = lead ? 0xffff0000u : 0x0000ffffu;
        R v = R(__longlong_as_double(0x7ff8000000000000ll));
        if (have) {
            R Phi[10], Psi[6], Fo[10], Go[6];
#pragma unroll
            for (int k = 0; k < 10; ++k) Phi[k] = mom[k];
#pragma unroll
            for (int k = 0; k < 6; ++k) Psi[k] = mom[10 + k];
            face_populations<R>(Phi, Psi, Tl, rho, du_n, du_t, T1, KC.wb, KC.we, P.Cvh_r, Fo, Go);
            __syncwarp(half);
            if (q == 0) {
#pragma unroll
                for (int k = 0; k < 10; ++k) mom[k] = Fo[k];
#pragma unroll
                for (int k = 0; k < 6; ++k) mom[10 + k] = Go[k];
                const R fn = dn + du_n, ft = dt + du_t;
                Frm[f] = fr_add(ref[0], dir ? ft : fn);
                Frm[nf + f] = fr_add(ref[1], dir ? fn : ft);
                Frm[2 * nf + f] = fr_word(T1);
            }
            __syncwarp(half);
            v = mom[q];
        } else if (q == 0) {
            fr_store(Frm[2 * nf + f], double(v));
        }
        const int k = q < 10 ? q : q - 10;
        int pl = k;
        if (dir) pl = k == 0 || k == 4 ? k : (k < 3 ? 3 - k : (k < 6 ? 8 - k : 15 - k));   // axes exchanged
        (q < 10 ? Fout : Gout)[pl * nf + f] = v;
        if (q == 0) {
            fc.iters += iters;
            fc.fallbacks += fallbacks;
            fc.nonconv += done ? 0 : 1;
            fc.nonphys += have ? 0 : 1;
        }
        unsigned int item = 0;
        if (q == 0) item = groups + atomicAdd(&P.tail->next, 1u);
        take(__shfl_sync(half, item, lead));
    }
    if (q == 0 && fc.iters) count_faces(P.diag, fc, 0);
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&P.tail->ctas, 1u) == min(gridDim.x, count) - 1) {
        // every CTA with a face has taken its last ticket: empty the list
        P.tail->n = 0u;
        P.tail->next = 0u;
        P.tail->ctas = 0u;
    }
}

template <typename R, typename VT>
constexpr size_t lane_smem_bytes()
{
    constexpr int TH = VT::TY / VecOf<R>::lanes;
    return sizeof(LaneCell<typename VecOf<R>::type>) * (VT::TX + 3) * (TH + 3) + size_t(S_SLOTS) * 16 * lane_threads<R, VT>();
}

}  // namespace pond
