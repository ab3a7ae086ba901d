// btdf_pair.cu - two time steps in one pass over the lattice (Algorithm 1
// twice, NF = 1), bitwise the results of two single steps.
//
// A single step reads and writes every population once: 72 bytes a node in
// FP32, which bounds it on lattices beyond L2 and, through L2, on smaller ones.
// Nothing in the scheme needs the intermediate state in memory: a node's
// second step needs the first step's result on its eight neighbours only.
// pair_kernel keeps that result in shared memory, so a pair of steps moves what a
// single one moves.  Measured, us a step, single -> pair: 8192 x 4096 with 400
// bodies FP32 343 -> 231, FP16 220 -> 209; 1600 x 800 with one body FP32
// 14.8 -> 11.5, FP16 13.3 -> 10.7; 1601 x 1601 BF16 with the convective outlet
// 28.2 -> 20.5; 128 lattices in a batch FP32 395 -> 239.
//
// The marker forces of the second step are needed before the pass that would
// produce the state they are interpolated from.  ib_pair_kernel redoes the
// first step on the (S + 2)^2 nodes around each marker's support: 25 node
// updates a marker for the 3-point delta, 0.2% of a 1600 x 800 lattice with
// 126 markers and 2% of 8192 x 4096 with 25 200.
//
// Kernels per two steps: ib_force (marker forces of the first step), ib_pair
// (those of the second, and the first step's spread over the band nodes),
// spread (the second step's), pair (both collisions, streamings and force
// histories).  Each is a programmatic dependent of the one before; tiles of the
// pair kernel off the band wait for none of them.  What is on the chain's path is
// kept short: the kernels after ib_force have loaded everything but the forces
// (state, tables, the first terms of every spread) before they wait.  With those
// loads after the wait, entry by entry, a pair on 160 x 80 with the 3-point delta took
// 12.7 us, now 9.4; with the 4-point cosine, whose 36 patch nodes take a warp two
// rounds, it takes 11.9 (two single steps 12.2).
#include "btdf_internal.cuh"
#include "btdf_device.cuh"
#include "btdf_collide.cuh"

#include <algorithm>

namespace btdf {
namespace {

// Two FP32 values in a 64-bit register, and the packed operations on them (two
// IEEE round-to-nearest operations each).  Held as 64-bit values throughout:
// with float2 the compiler re-pairs operands with moves.
using P2 = unsigned long long;
__device__ __forceinline__ P2 pk(float x, float y) {
    P2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ P2 pk(float x) { return pk(x, x); }
__device__ __forceinline__ float2 unpk(P2 v) {
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(v));
    return o;
}
__device__ __forceinline__ P2 padd(P2 a, P2 b) {
    P2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ P2 pmul(P2 a, P2 b) {
    P2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ P2 pfma(P2 a, P2 b, P2 c) {
    P2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// e_a . (x, y) of a pair; nx, ny are -x, -y (a != 0).
__device__ __forceinline__ P2 pdot(int a, P2 x, P2 y, P2 nx, P2 ny) {
    const P2 sx = ex(a) > 0 ? x : nx, sy = ey(a) > 0 ? y : ny;
    return ex(a) == 0 ? sy : (ey(a) == 0 ? sx : padd(sx, sy));
}

// Constants of the collision as register pairs, by the population's class: e_x
// for the first two (the reference velocity lies along x), the weight for the
// third.
struct PairConst {
    P2 c1[3], kr[3], wom[3], omop, m1, urx2, nurx, c45, one, m15;
    __device__ __forceinline__ explicit PairConst(const LatticeParams& p) {
        const int ax[3] = {3, 0, 1}, aw[3] = {0, 1, 5};
#pragma unroll
        for (int k = 0; k < 3; k++) {
            c1[k] = pk(p.c1[ax[k]]);
            kr[k] = pk(p.kr[ax[k]]);
            wom[k] = pk(p.wom[aw[k]]);
        }
        omop = pk(p.one_m_omega);
        m1 = pk(-1.0f);
        urx2 = pk(2.0f * p.urx);
        nurx = pk(-p.urx);
        c45 = pk(4.5f);
        one = pk(1.0f);
        m15 = pk(-1.5f);
    }
};

// collide_nodes() for two nodes in packed operations, in place, forced or not:
// operation for operation the same values (the reference velocity lies along x
// and e_0 = 0: their zero terms are left out).  scale is the stored value of a
// unit deviation.
template <bool kForced>
__device__ __forceinline__ void collide_pair(P2& f0, P2& f1, P2& f2_, P2& f3, P2& f4, P2& f5, P2& f6, P2& f7, P2& f8,
                                             const LatticeParams& p, const PairConst& k, P2 Fx, P2 Fy, float scale) {
    P2* const f[9] = {&f0, &f1, &f2_, &f3, &f4, &f5, &f6, &f7, &f8};
    auto sub = [&](P2 a, P2 b) { return pfma(b, k.m1, a); };
    P2 d = padd(padd(padd(f0, f1), padd(f2_, f3)), padd(padd(f4, f5), padd(f6, f7)));
    d = padd(d, f8);
    P2 jx = padd(padd(sub(f1, f3), sub(f5, f6)), sub(f8, f7));
    P2 jy = sub(padd(sub(f2_, f4), padd(f5, f6)), padd(f7, f8));
    if (scale != 1.0f) {
        const P2 s = pk(1.0f / scale);
        d = pmul(d, s);
        jx = pmul(jx, s);
        jy = pmul(jy, s);
    }
    const P2 rho = padd(k.one, d);
    const float2 rs = unpk(rho);
    const P2 inv = pk(__fdividef(1.0f, rs.x), __fdividef(1.0f, rs.y));
    P2 U = pmul(pfma(d, k.nurx, jx), inv);
    P2 V = pmul(jy, inv);
    P2 uF = 0, nFx = 0, nFy = 0;
    if (kForced) {
        Fx = padd(Fx, pk(p.gx));
        Fy = padd(Fy, pk(p.gy));
        U = pfma(pmul(pk(0.5f), Fx), inv, U);
        V = pfma(pmul(pk(0.5f), Fy), inv, V);
        uF = pfma(padd(pk(p.urx), U), Fx, pmul(V, Fy));
        uF = pmul(pk(-3.0f), uF);
        nFx = pmul(Fx, k.m1);
        nFy = pmul(Fy, k.m1);
    }
    const P2 nU = pmul(U, k.m1), nV = pmul(V, k.m1);
    // -1.5 (2 U_r.du + du^2)
    P2 t = pfma(U, U, pmul(V, V));
    t = pfma(k.urx2, U, t);
    const P2 P = pmul(k.m15, t);
#pragma unroll
    for (int a = 0; a < 9; a++) {
        const int cx = ex(a) + 1, cw = a == 0 ? 0 : a < 5 ? 1 : 2;
        const P2 ed = a == 0 ? 0 : pdot(a, U, V, nU, nV);
        const P2 pdiff = a == 0 ? P : pfma(ed, pfma(k.c45, ed, k.c1[cx]), P);
        const P2 deqw = pfma(rho, pdiff, pmul(k.kr[cx], d));
        P2 r = pfma(k.wom[cw], deqw, pmul(k.omop, *f[a]));
        if (kForced) {
            P2 g = uF;
            if (a != 0) {
                const P2 eu = padd(pk(p.eur[a]), ed);
                g = pfma(pdot(a, Fx, Fy, nFx, nFy), pfma(pk(9.0f), eu, pk(3.0f)), uF);
            }
            r = pfma(pk(p.wg[a]), g, r);
        }
        *f[a] = r;
    }
}
template <bool kForced, int NP>
__device__ __forceinline__ void collide_pairs(P2 (&f)[9][NP], const LatticeParams& p, const PairConst& k,
                                              const P2 (&Fx)[NP], const P2 (&Fy)[NP], float scale) {
#pragma unroll
    for (int j = 0; j < NP; j++)
        collide_pair<kForced>(f[0][j], f[1][j], f[2][j], f[3][j], f[4][j], f[5][j], f[6][j], f[7][j], f[8][j], p, k,
                              Fx[j], Fy[j], scale);
}

// NPL neighbouring populations of one direction, as stored: packed FP32 pairs, or
// 16-bit pairs (four of them: pair_npl).
template <typename T, int NPL> struct Vec {
    static_assert(NPL == 4, "16-bit storage takes 4 nodes per lane");
    static constexpr int NP = NPL / 2;
    unsigned w[NP];
    static __device__ __forceinline__ float2 to2(unsigned v) {
        if constexpr (Raw<T>::kScale != 1.0f) return Raw<__half>::to2(v);
        else return Io16<__nv_bfloat16, __nv_bfloat162>::to2(v);
    }
    __device__ __forceinline__ void load(const T* p) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
        w[0] = v.x;
        w[1] = v.y;
    }
    __device__ __forceinline__ void loads(const T* p) {   // shared memory
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x;
        w[1] = v.y;
    }
    __device__ __forceinline__ void store(T* p) const {
        *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
    }
    __device__ __forceinline__ P2 get(int j) const {
        const float2 f = to2(w[j]);
        return pk(f.x, f.y);
    }
    __device__ __forceinline__ void set(int j, P2 o) {
        const float2 f = unpk(o);
        if constexpr (Raw<T>::kScale != 1.0f) w[j] = Raw<__half>::from2(f.x, f.y);
        else w[j] = Io16<__nv_bfloat16, __nv_bfloat162>::from2(f.x, f.y);
    }
    __device__ __forceinline__ void scalars(const T (&t)[NPL]) {
#pragma unroll
        for (int j = 0; j < NP; j++)
            w[j] = (unsigned)*reinterpret_cast<const unsigned short*>(&t[2 * j]) |
                   (unsigned)*reinterpret_cast<const unsigned short*>(&t[2 * j + 1]) << 16;
    }
    // the values one node to the left / right of each (lane 0's first / lane
    // 31's last is left undefined)
    __device__ __forceinline__ Vec left() const {
        Vec o;
        const unsigned prev = __shfl_up_sync(kFull, w[NP - 1], 1);
#pragma unroll
        for (int j = 0; j < NP; j++) o.w[j] = __byte_perm(j == 0 ? prev : w[j - 1], w[j], 0x5432);
        return o;
    }
    __device__ __forceinline__ Vec right() const {
        Vec o;
        const unsigned next = __shfl_down_sync(kFull, w[0], 1);
#pragma unroll
        for (int j = 0; j < NP; j++) o.w[j] = __byte_perm(w[j], j == NP - 1 ? next : w[j + 1], 0x5432);
        return o;
    }
};
template <int NPL> struct Vec<float, NPL> {
    static constexpr int NP = NPL / 2;
    P2 w[NP];
    __device__ __forceinline__ void load(const float* p) {
        if constexpr (NPL == 4) {
            const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
            w[0] = v.x;
            w[1] = v.y;
        } else {
            w[0] = __ldg(reinterpret_cast<const P2*>(p));
        }
    }
    __device__ __forceinline__ void loads(const float* p) {   // shared memory
        if constexpr (NPL == 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
            w[0] = v.x;
            w[1] = v.y;
        } else {
            w[0] = *reinterpret_cast<const P2*>(p);
        }
    }
    __device__ __forceinline__ void store(float* p) const {
        if constexpr (NPL == 4) *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(w[0], w[1]);
        else *reinterpret_cast<P2*>(p) = w[0];
    }
    __device__ __forceinline__ void scalars(const float (&t)[NPL]) {
#pragma unroll
        for (int j = 0; j < NP; j++) w[j] = pk(t[2 * j], t[2 * j + 1]);
    }
    __device__ __forceinline__ P2 get(int j) const { return w[j]; }
    __device__ __forceinline__ void set(int j, P2 o) { w[j] = o; }
    __device__ __forceinline__ Vec left() const {
        Vec o;
        float prev = __shfl_up_sync(kFull, unpk(w[NP - 1]).y, 1);
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const float2 f = unpk(w[j]);
            o.w[j] = pk(prev, f.x);
            prev = f.y;
        }
        return o;
    }
    __device__ __forceinline__ Vec right() const {
        Vec o;
        float next = __shfl_down_sync(kFull, unpk(w[0]).x, 1);
#pragma unroll
        for (int j = NP - 1; j >= 0; j--) {
            const float2 f = unpk(w[j]);
            o.w[j] = pk(f.y, next);
            next = f.x;
        }
        return o;
    }
};

// A tile of 30 * NPL columns x TH rows per block.  First step: the block's warps
// pull the TH + 2 rows of 32 * NPL columns around the tile from memory, collide
// them and leave the results, rounded to the storage type, in shared memory.
// Second step: they pull the tile's rows from there, collide and store them.  A
// warp takes a row at a time, NPL consecutive nodes per lane; the outer two lanes
// hold the columns beside the tile.
//
// What bounds it: instructions, FP32 nearly as much the traffic.  On 8192 x 4096 FP32
// it moves 2.42 GB a pair at 5.2 TB/s (0.78 of the measured copy rate), FP16 half the
// bytes in nearly the same time; under ncu on 4096 x 2048 the issue slots are 52%
// (FP32) and 62% (FP16) busy and DRAM 62% and 32%, with 273 and 297 warp instructions
// per 64 nodes and step, halo included.  The register caps cost spills, of boundary
// code for the most part: 164 bytes a thread in FP32 with 4 nodes per lane, 64 with 2,
// 24 in FP16, 156 in BF16; in the batch, whose constants come from shared memory, 448,
// 164, 236 and 444.  Small tiles, although their halo costs 14-20% more node
// updates, keep the register count low and 3 to 5 blocks an SM resident, so that one block's
// barrier and loads hide behind the others: tiles of 14 rows with two blocks an SM
// took 235 to 265 us a step on 8192 x 4096.
// A form that walks down the rows with the first step's rows in registers
// (128-168 registers, 3-4 warps a scheduler) stayed at 245-255 us there and made
// a chain of a small lattice's rows (14.4 us at 1600 x 800).
template <typename T, int NPL, int TH>
struct PairTile {
    static constexpr int NP = NPL / 2, W = 32 * NPL, RN = TH + 2;
    static constexpr size_t kShared = sizeof(T) * 9 * RN * W;
};

// Boundary rules of row y on the lane's post-streaming nodes x0 ..: the constant
// of the populations that come back from a bounce-back wall; the inlet node from
// the node beside it, the outlet node from the node before it, which may be the
// lane below's last (old: the convective outlet's previous column; keep: write
// the new one).  As in the single steps, inner nodes take the wall's constant with
// one rounding, row ends (g; those of a periodic lattice too) with two; in FP16,
// whose constant is rounded before it is scaled, all nodes take it with two.
// One population at a time: arrays of the lane's nodes would raise the register
// count of the whole kernel.
template <typename T, int NPL>
__device__ __forceinline__ void pair_boundaries(P2 (&fp)[9][NPL / 2], const LatticeParams& p, int x0, int y, bool ends,
                                                const float* old, bool keep) {
    constexpr int NP = NPL / 2;
    constexpr float up = Raw<T>::kScale, down = 1.0f / Raw<T>::kScale;
    const int nx = p.nx, ny = p.ny;
    const bool perx = p.bcx == kBcxPeriodic;
    float f[9][NPL], g[9][NPL];
#pragma unroll
    for (int a = 0; a < 9; a++)
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const float2 v = unpk(fp[a][j]);
            f[a][2 * j] = g[a][2 * j] = v.x;
            f[a][2 * j + 1] = g[a][2 * j + 1] = v.y;
        }
    if (p.bcy == kBcyNoslip && (y == 0 || y == ny - 1)) {
#pragma unroll
        for (int a = 0; a < 9; a++)
            if ((ey(a) > 0 && y == 0) || (ey(a) < 0 && y == ny - 1)) {
                const float w = -6.0f * wt(a) * up, add = __fmul_rn(w, p.eur[a]);
#pragma unroll
                for (int i = 0; i < NPL; i++) {
                    g[a][i] = __fadd_rn(f[a][i], add);
                    const int x = x0 + i;
                    const bool end = perx && (x == -1 || x == 0 || x == nx - 1 || x == nx);
                    f[a][i] = end || up != 1.0f ? g[a][i] : __fmaf_rn(w, p.eur[a], f[a][i]);
                }
            }
    }
    if (ends && !perx) {
        if (x0 == 0) {
            float f1[9], fe[9];
#pragma unroll
            for (int a = 0; a < 9; a++) f1[a] = __fmul_rn(g[a][1], down);   // a product of its own: not contracted
            inlet_from(f1, p, fe);
#pragma unroll
            for (int a = 0; a < 9; a++) f[a][0] = fe[a] * up;
        }
        const int i = nx - 1 - x0;
        // Nine lanes load the previous column's populations, for the one lane that
        // holds the outlet node: loaded there one by one, between the stores of the new
        // column, a lattice of 160 x 80 without bodies took 4.4 us a step (3.8 singly),
        // now 2.2; 1601 x 1601 FP32 with one body 23.7, now 21.9.
        const int lane = (int)threadIdx.x & 31;
        const bool here = old != nullptr && i >= 0 && i < NPL;
        const unsigned who = __ballot_sync(kFull, here);
        const float* src = (const float*)__shfl_sync(kFull, (unsigned long long)old, who ? __ffs(who) - 1 : 0);
        const float olds = who != 0u && lane < 9 ? src[lane * ny + y] : 0.f;
#pragma unroll
        for (int a = 0; a < 9; a++) {
            float v = __shfl_up_sync(kFull, g[a][NPL - 1], 1);
#pragma unroll
            for (int m = 1; m < NPL; m++)
                if (m == i) v = g[a][m - 1];
            const float o = __shfl_sync(kFull, olds, a);
            if (here) {
                const float w = __fmaf_rn(p.uc_new, v * down, __fmul_rn(p.uc_old, o));
                if (keep) p.outlet_out[a * ny + y] = w;
                v = w * up;
            }
#pragma unroll
            for (int m = 0; m < NPL; m++)
                if (m == i) f[a][m] = v;
        }
    }
#pragma unroll
    for (int a = 0; a < 9; a++)
#pragma unroll
        for (int j = 0; j < NP; j++) fp[a][j] = pk(f[a][2 * j], f[a][2 * j + 1]);
}

// Spread forces on the lane's nodes: the x, then the y components of a band
// row's 32 * NPL nodes.
template <int NPL>
__device__ __forceinline__ void pair_spread(const float* fb, int band, int lane, P2 (&Fx)[NPL / 2], P2 (&Fy)[NPL / 2]) {
    const P2* s = reinterpret_cast<const P2*>(fb + (size_t)band * (64 * NPL)) + NPL / 2 * lane;
#pragma unroll
    for (int j = 0; j < NPL / 2; j++) {
        Fx[j] = __ldcg(s + j);
        Fy[j] = __ldcg(s + 16 * NPL + j);
    }
}

// Two steps of the tile of strip s from row y0 on, of the lattice p whose
// populations are gin / gout; the other arguments are PairForces'.
template <typename T, int NPL, int NW, int TH>
__device__ __forceinline__ void pair_tile(const T* __restrict__ gin, T* __restrict__ gout, const LatticeParams& p,
                                          const unsigned (&kin)[9], const int* strip_row, int nstrip, const float* fb1,
                                          const float* fb2, int s, int y0, T* tile) {
    using C = PairTile<T, NPL, TH>;
    constexpr int NP = NPL / 2;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int ny = p.ny, nx = p.nx, xs = s * pair_own(NPL) - NPL;
    const bool pery = p.bcy == kBcyPeriodic, perx = p.bcx == kBcxPeriodic, noslip = p.bcy == kBcyNoslip;
    const int x0 = xs + NPL * lane;
    const int x0c = min(max(x0, 0), p.nxp - NPL);
    const bool own = lane > 0 && lane < 31 && x0 < nx;
    const bool ends = xs <= 0 || xs + 32 * NPL >= nx;   // the tile holds a row end
    const T* const cin = gin + x0c;
    T* const cout = gout + x0c;
    const int* const srow = strip_row != nullptr ? strip_row + s : nullptr;
    const bool uniform_force = p.gx != 0.f || p.gy != 0.f;
    const PairConst k(p);

#pragma unroll 1
    for (int j = warp; j < C::RN; j += NW) {
        const int r = y0 - 1 + j;
        int rr = r;
        if (pery) rr = r < 0 ? r + ny : r >= ny ? r - ny : r;
        if (rr < 0 || rr >= ny) continue;   // beyond a wall, or past the periodic halo
        Vec<T, NPL> v[9];
        const bool inner = rr > 0 && rr < ny - 1;
        if (inner) {
            const T* row = cin + (long long)(rr - 1) * p.rs;
#pragma unroll
            for (int a = 0; a < 9; a++) v[a].load(row + kin[a]);   // one multiply-add a population
        } else {
#pragma unroll
            for (int a = 0; a < 9; a++) {
                int pa, sy, dx;
                float unused;
                y_source(a, rr, p, pa, sy, dx, unused);
                v[a].load(cin + (long long)sy * p.rs + p.poff[pa]);
            }
        }
        if (perx && ends && (x0 < 0 || x0 + NPL > nx)) {
            // the columns beside a periodic lattice wrap, node by node
#pragma unroll
            for (int a = 0; a < 9; a++) {
                int pa, sy, dx;
                float unused;
                y_source(a, rr, p, pa, sy, dx, unused);
                const T* row = gin + (long long)sy * p.rs + p.poff[pa];
                T t[NPL];
#pragma unroll
                for (int i = 0; i < NPL; i++) t[i] = __ldg(row + ((x0 + i) % nx + nx) % nx);
                v[a].scalars(t);
            }
        }
        const int band = srow != nullptr ? __ldg(srow + rr * nstrip) : -1;
        P2 f[9][NP];
#pragma unroll
        for (int a = 0; a < 9; a++) {
            Vec<T, NPL> u = ex(a) > 0 ? v[a].left() : ex(a) < 0 ? v[a].right() : v[a];
            if (ex(a) != 0 && ey(a) != 0 && noslip && !inner && (ey(a) > 0 ? rr == 0 : rr == ny - 1)) u = v[a];
#pragma unroll
            for (int i = 0; i < NP; i++) f[a][i] = u.get(i);
        }
        if ((ends && !perx) || (noslip && !inner))
            pair_boundaries<T, NPL>(f, p, x0, rr, ends, p.outlet, own && j > 0 && j <= TH && r < ny);
        T* const trow = tile + j * C::W + NPL * lane;
        P2 Fx[NP] = {}, Fy[NP] = {};
        if (uniform_force || band >= 0) {
            if (band >= 0) {
                cudaGridDependencySynchronize();
                pair_spread<NPL>(fb1, band, lane, Fx, Fy);
            }
            collide_pairs<true, NP>(f, p, k, Fx, Fy, Raw<T>::kScale);
        } else {
            collide_pairs<false, NP>(f, p, k, Fx, Fy, Raw<T>::kScale);
        }
#pragma unroll
        for (int a = 0; a < 9; a++) {
            Vec<T, NPL> o;
#pragma unroll
            for (int i = 0; i < NP; i++) o.set(i, f[a][i]);
            o.store(trow + a * (C::RN * C::W));
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int j = warp; j < TH; j += NW) {
        const int y = y0 + j;
        if (y >= ny) break;
        const int band = srow != nullptr ? __ldg(srow + y * nstrip) : -1;
        const T* const trow = tile + (j + 1) * C::W + NPL * lane;
        const bool inner = pery || (y > 0 && y < ny - 1);
        P2 f[9][NP];
#pragma unroll
        for (int a = 0; a < 9; a++) {
            Vec<T, NPL> v;
            v.loads(trow + a * (C::RN * C::W) - ey(a) * C::W);
            Vec<T, NPL> u = ex(a) > 0 ? v.left() : ex(a) < 0 ? v.right() : v;
#pragma unroll
            for (int i = 0; i < NP; i++) f[a][i] = u.get(i);
        }
        if (!inner) {
            // populations from beyond a wall: the row's own mirrored (free-slip)
            // or opposite ones (bounce-back, unshifted)
#pragma unroll
            for (int a = 0; a < 9; a++) {
                if (ey(a) == 0 || (ey(a) > 0 ? y != 0 : y != ny - 1)) continue;
                Vec<T, NPL> v;
                v.loads(trow + (noslip ? opposite(a) : mirror_y(a)) * (C::RN * C::W));
                Vec<T, NPL> u = ex(a) > 0 ? v.left() : ex(a) < 0 ? v.right() : v;
                if (noslip) u = v;
#pragma unroll
                for (int i = 0; i < NP; i++) f[a][i] = u.get(i);
            }
        }
        if ((ends && !perx) || (noslip && !inner))
            pair_boundaries<T, NPL>(f, p, x0, y, ends, p.outlet != nullptr && own ? p.outlet_out : nullptr, own);
        T* const row = cout + (long long)y * p.rs;
        P2 Fx[NP] = {}, Fy[NP] = {};
        if (uniform_force || band >= 0) {
            if (band >= 0) pair_spread<NPL>(fb2, band, lane, Fx, Fy);
            collide_pairs<true, NP>(f, p, k, Fx, Fy, Raw<T>::kScale);
        } else {
            collide_pairs<false, NP>(f, p, k, Fx, Fy, Raw<T>::kScale);
        }
        if (own) {
#pragma unroll
            for (int a = 0; a < 9; a++) {
                Vec<T, NPL> o;
#pragma unroll
                for (int i = 0; i < NP; i++) o.set(i, f[a][i]);
                o.store(row + p.poff[a]);
            }
        }
    }
}

// Last of the reduction blocks: the step counter.
__device__ __forceinline__ void pair_finish(unsigned long long* counter, unsigned long long step, unsigned* done,
                                            int nred) {
    __syncthreads();
    if (threadIdx.x == 0 && counter != nullptr) {
        __threadfence();
        if (atomicAdd(done, 1u) == (unsigned)nred - 1u) {
            *counter = step + 2ull;
            *done = 0u;
        }
    }
}

template <typename T, int NPL, int NW, int TH, int MINB>
__global__ void __launch_bounds__(32 * NW, MINB)
pair_kernel(const T* __restrict__ gin, T* __restrict__ gout, const __grid_constant__ LatticeParams p,
            const __grid_constant__ PairForces q, int nred) {
    cudaTriggerProgrammaticLaunchCompletion();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // The first nred blocks reduce the body forces of both steps while the
    // others work; the last of them to finish advances the step counter.
    if ((int)blockIdx.x < nred) {
        if (p.nbody > 0) cudaGridDependencySynchronize();
        const unsigned long long step = p.step != nullptr ? *p.step : 0ull;
        const int half = NW / 2, w = (int)threadIdx.x >> 5;
        // a ring of one step keeps the second step's forces only
        if (w < half && p.hist_len > 1) body_forces(p, q.F1, step, blockIdx.x * half + w, nred * half);
        if (w >= half && w < 2 * half) body_forces(p, p.F, step + 1ull, blockIdx.x * half + w - half, nred * half);
        pair_finish(p.step, step, q.done, nred);
        return;
    }
    const int b = (int)blockIdx.x - nred;
    const int c = b / q.nstrip, s = b - c * q.nstrip;
    pair_tile<T, NPL, NW, TH>(gin, gout, p, q.kin, q.strip_row, q.nstrip, q.fb1, q.fb2, s, c * TH,
                              reinterpret_cast<T*>(smem_raw));
}

// Batched form: the tiles of all lattices in one launch; a block copies its
// lattice's description to shared memory first.
template <typename T, int NPL, int NW, int TH, int MINB>
__global__ void __launch_bounds__(32 * NW, MINB)
pair_batch_kernel(const T* __restrict__ gin, T* __restrict__ gout, const __grid_constant__ PairBatch b,
                  const __grid_constant__ PairForces q, int nred) {
    cudaTriggerProgrammaticLaunchCompletion();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if ((int)blockIdx.x < nred) {
        if (b.nbody > 0) cudaGridDependencySynchronize();
        const unsigned long long step = *b.step;
        const int half = NW / 2, w = (int)threadIdx.x >> 5;
        if (w < half && b.hist_len > 1)   // as in pair_kernel
            body_forces(b.nbody, b.body_rng, 2, b.body_scale, b.hist, b.hist_len, q.F1, step, blockIdx.x * half + w,
                        nred * half);
        if (w >= half && w < 2 * half)
            body_forces(b.nbody, b.body_rng, 2, b.body_scale, b.hist, b.hist_len, b.F2, step + 1ull,
                        blockIdx.x * half + w - half, nred * half);
        pair_finish(b.step, step, q.done, nred);
        return;
    }
    __shared__ __align__(16) LatticeParams sp;
    __shared__ __align__(16) PairLattice sl;
    const int4 t = __ldg(b.tile + ((int)blockIdx.x - nred));
    {
        const int* a = reinterpret_cast<const int*>(b.descs + t.x);
        const int* c = reinterpret_cast<const int*>(b.lat + t.x);
        for (int i = threadIdx.x; i < (int)(sizeof(LatticeParams) / 4); i += 32 * NW)
            reinterpret_cast<int*>(&sp)[i] = __ldg(a + i);
        for (int i = threadIdx.x; i < (int)(sizeof(PairLattice) / 4); i += 32 * NW)
            reinterpret_cast<int*>(&sl)[i] = __ldg(c + i);
    }
    __syncthreads();
    pair_tile<T, NPL, NW, TH>(gin + sl.off, gout + sl.off, sp, sl.kin, sl.strip_row, sl.nstrip, q.fb1, q.fb2, t.y, t.z,
                              reinterpret_cast<T*>(smem_raw));
}

// Spread (Eq. 15) of the forces F, one thread per band node of a strip that has
// terms: nodes[t] = (slot in fb, first term, end of terms).
__device__ __forceinline__ void spread_node(const CsrEntry* csr, const float2* F, const PairForces& q, float* fb,
                                            int t) {
    int4 n = make_int4(0, 0, 0, 0);
    SpreadTerms terms;
    if (t < q.nnode) n = __ldg(q.nodes + t);
    terms.load(csr, n.y, n.z);
    cudaGridDependencySynchronize();
    if (t >= q.nnode) return;
    float fx, fy;
    terms.sum(csr, F, fx, fy);
    fb[n.x] = fx;
    fb[n.x + 32 * q.npl] = fy;
}

__global__ void __launch_bounds__(128) spread_kernel(const CsrEntry* csr, const float2* F, PairForces q) {
    // Its dependent may start at once: this grid starts after ib_force's wait for
    // the previous pair (ib_pair_kernel launches it the same way).
    cudaTriggerProgrammaticLaunchCompletion();
    spread_node(csr, F, q, q.fb2, (int)(blockIdx.x * blockDim.x + threadIdx.x));
}

// Forces of the second step, one warp per marker.  The lanes redo the first
// step on the (S + 2)^2 nodes around the marker's support (the forces F1 of
// that step come from ib_force_kernel) into shared memory; then the lanes of
// the support nodes pull from there and interpolate like ib_force_kernel.  The
// caller makes sure that no support is clipped or touches an inlet or outlet
// column, so no row-end rule applies to a support node.
constexpr int kIbPairThreads = 128;

template <typename T, int S>
__device__ __forceinline__ void ib_pair_marker(const T* __restrict__ g, const LatticeParams& p, const IbParams& q,
                                               const float2* F1, long long m, float (*patch)[(S + 2) * (S + 2)]) {
    constexpr int P = S + 2;
    const int lane = threadIdx.x & 31;
    const Marker* mk = q.mk + m;
    const MarkerAux ax = q.aux[m];
    const int xa = __ldg(&mk->xs[0]), ya = __ldg(&mk->ys[0]);
    const bool act = lane < S * S;
    const float w = act ? __ldg(&mk->w[lane]) : 0.f;
    // Everything but the forces F1 is there before ib_force has finished: the
    // state g (ib_force let this grid start after its wait for it) and the tables.
    constexpr int R = (P * P + 31) / 32;
    float f[R][9][1];
    SpreadTerms terms[R];
    bool valid[R], band[R];
#pragma unroll
    for (int k = 0; k < R; k++) {
        const int e = lane + 32 * k;
        const int j = e / P, i = e - j * P;
        // support columns are consecutive up to a periodic wrap
        int x = xa + i - 1, y = ya + j - 1;
        if (p.bcx == kBcxPeriodic) x = ((x % p.nx) + p.nx) % p.nx;
        if (p.bcy == kBcyPeriodic) y = ((y % p.ny) + p.ny) % p.ny;
        valid[k] = e < P * P && x >= 0 && x < p.nx && y >= 0 && y < p.ny;
        band[k] = false;
        terms[k].load(p.csr, 0, 0);
        if (!valid[k]) continue;
        float d[9];
        gather_node<T>(g, p, true, x, y, d);
#pragma unroll
        for (int a = 0; a < 9; a++) f[k][a][0] = d[a] * Raw<T>::kScale;
        // the LBM kernels add a bounce-back wall's constant with one rounding
        // on inner columns (not in FP16: pair_boundaries)
        if (Raw<T>::kScale == 1.0f && p.bcy == kBcyNoslip && (y == 0 || y == p.ny - 1) && x > 0 && x < p.nx - 1) {
#pragma unroll
            for (int a = 0; a < 9; a++)
                if ((ey(a) > 0 && y == 0) || (ey(a) < 0 && y == p.ny - 1)) {
                    const float v = Io<T>::ld1(g + p.poff[opposite(a)] + (unsigned)y * p.rs + (unsigned)x);
                    f[k][a][0] = __fmaf_rn(-6.0f * wt(a), p.eur[a], v);
                }
        }
        const int seg = __ldg(p.seg_index + y * p.nseg + x / kSeg);
        if (seg >= 0) {
            const int* ptr = p.seg_ptr + (long long)seg * (kSeg + 1) + (x % kSeg);
            terms[k].load(p.csr, __ldg(ptr), __ldg(ptr + 1));
            band[k] = true;
        }
    }
    cudaGridDependencySynchronize();
#pragma unroll
    for (int k = 0; k < R; k++) {
        if (!valid[k]) continue;
        const int e = lane + 32 * k;
        float Fx[1], Fy[1];
        terms[k].sum(p.csr, F1, Fx[0], Fy[0]);
        const bool forced = band[k] || p.gx != 0.f || p.gy != 0.f;
        collide_nodes<T, 1>(f[k], p, Fx, Fy, forced, []() {}, [&](int a, const float (&o)[1]) {
            T st;
            Raw<T>::template stv<1>(&st, o);
            patch[a][e] = Io<T>::ld1s(&st);
        });
    }
    __syncwarp();
    float wr = 0.f, wu = 0.f, wv = 0.f;
    if (act && w != 0.f) {
        const int sj = lane / S, si = lane - sj * S;
        int y = ya + sj;
        if (p.bcy == kBcyPeriodic && y >= p.ny) y -= p.ny;
        float d[9];
#pragma unroll
        for (int a = 0; a < 9; a++) {
            int pa, sy, dx;
            float add;
            y_source(a, y, p, pa, sy, dx, add);
            const bool wall = p.bcy != kBcyPeriodic && y - ey(a) != sy;
            const int row = wall ? sj + 1 : sj + 1 - ey(a);
            d[a] = patch[pa][row * P + si + 1 + dx] + add;
        }
        const Moments mo = moments(d, p.urx, p.ury);
        wr = w * mo.drho;
        wu = w * mo.dux;
        wv = w * mo.duy;
    }
    constexpr int G = Group<S>::G;
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
        wr += __shfl_xor_sync(kFull, wr, off);
        wu += __shfl_xor_sync(kFull, wu, off);
        wv += __shfl_xor_sync(kFull, wv, off);
    }
    if (lane == 0) {
        const float rl = ax.wsum + wr;
        const float dFx = 2.0f * rl * (ax.ubx_rel - wu);
        const float dFy = 2.0f * rl * (ax.uby_rel - wv);
        q.F_out[m] = make_float2(0.f + dFx, 0.f + dFy);
        q.Us[m] = make_float2(p.urx * ax.wsum + wu, p.ury * ax.wsum + wv);
        q.rhol[m] = rl;
        if (!(rl > 0.f) || !isfinite(dFx) || !isfinite(dFy)) atomicOr(q.status, kStatusUnstable);
    }
}

template <typename T, int S>
__global__ void __launch_bounds__(kIbPairThreads)
ib_pair_kernel(const T* __restrict__ g, LatticeParams p, IbParams q, PairForces r, int mblocks) {
    constexpr int W = kIbPairThreads / 32;
    __shared__ float patch[W][9][(S + 2) * (S + 2)];
    // ib_force, whose dependent this is, has waited for the previous pair of
    // steps before letting this grid start, so everything after it may start too:
    // the pair kernel's warps off the band need nothing else.
    cudaTriggerProgrammaticLaunchCompletion();
    if ((int)blockIdx.x >= mblocks) {   // the first step's spread
        spread_node(p.csr, r.F1, r, r.fb1, ((int)blockIdx.x - mblocks) * kIbPairThreads + (int)threadIdx.x);
        return;
    }
    const int warp = threadIdx.x >> 5;
    const long long m = (long long)blockIdx.x * W + warp;
    if (m >= q.nmark) return;   // whole warps
    ib_pair_marker<T, S>(g, p, q, r.F1, m, patch[warp]);
}

// Batched form: MarkerAux.body holds the marker's lattice.
template <typename T, int S>
__global__ void __launch_bounds__(kIbPairThreads)
ib_pair_batch_kernel(const T* __restrict__ g, const LatticeParams* __restrict__ descs,
                     const unsigned long long* __restrict__ case_off, IbParams q, PairForces r,
                     const CsrEntry* csr, int mblocks) {
    constexpr int W = kIbPairThreads / 32;
    __shared__ float patch[W][9][(S + 2) * (S + 2)];
    cudaTriggerProgrammaticLaunchCompletion();   // as in ib_pair_kernel
    if ((int)blockIdx.x >= mblocks) {
        spread_node(csr, r.F1, r, r.fb1, ((int)blockIdx.x - mblocks) * kIbPairThreads + (int)threadIdx.x);
        return;
    }
    const int warp = threadIdx.x >> 5;
    const long long m = (long long)blockIdx.x * W + warp;
    if (m >= q.nmark) return;
    const int c = q.aux[m].body;
    ib_pair_marker<T, S>(g + case_off[c], descs[c], q, r.F1, m, patch[warp]);
}

cudaLaunchConfig_t config(unsigned grid, unsigned threads, bool pdl, cudaLaunchAttribute* attr, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cfg;
}

template <typename T, int NPL, int NW, int TH, int MINB>
cudaError_t pair_tn(const void* gin, void* gout, const LatticeParams& p, const PairForces& q, bool pdl,
                    cudaStream_t st) {
    using C = PairTile<T, NPL, TH>;
    auto kern = pair_kernel<T, NPL, NW, TH, MINB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kShared);
    if (e != cudaSuccess) return e;
    const long long nchunk = (p.ny + TH - 1) / TH;
    const int nred = std::min(16, std::max(1, (p.nbody + 2 * NW - 1) / (2 * NW)));
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = config((unsigned)(q.nstrip * nchunk + nred), 32 * NW, pdl, attr, st);
    cfg.dynamicSmemBytes = C::kShared;
    return cudaLaunchKernelEx(&cfg, kern, (const T*)gin, (T*)gout, p, q, nred);
}

template <typename T>
cudaError_t ib_pair_t(int width, const void* g, const LatticeParams& p, const IbParams& q, const PairForces& r,
                      bool pdl, cudaStream_t st) {
    constexpr int W = kIbPairThreads / 32;
    const int mb = (q.nmark + W - 1) / W;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg =
        config((unsigned)(mb + (r.nnode + kIbPairThreads - 1) / kIbPairThreads), kIbPairThreads, pdl, attr, st);
    switch (width) {
    case 2: return cudaLaunchKernelEx(&cfg, ib_pair_kernel<T, 2>, (const T*)g, p, q, r, mb);
    case 3: return cudaLaunchKernelEx(&cfg, ib_pair_kernel<T, 3>, (const T*)g, p, q, r, mb);
    case 4: return cudaLaunchKernelEx(&cfg, ib_pair_kernel<T, 4>, (const T*)g, p, q, r, mb);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Nodes per lane.  FP32 below 2^22 nodes: 2, with 40 warps an SM in tiles of 60 x 6
// (11.5 us a step at 1600 x 800 against 12.2 with 4); above, where fewer
// instructions per node count for more, 4, with 27 warps in tiles of 120 x 7
// (232 us at 8192 x 4096 against 243), unless its strips leave many columns unused
// (128 x 65536: 139 us with 4, 105 with 2, 110 singly).  16-bit storage: 4 (2 took
// 11.4 us at 1600 x 800, now 10.7, and 239 at 8192 x 4096 against 209).  Also measured
// with 4: tiles of 120 x 6 with four blocks an SM (FP32 234, FP16 207 at 8192 x 4096,
// 11.3 at 1600 x 800), 120 x 8 with three (240, 209, 11.4).
int pair_npl(int storage, int bcx, int nx, int ny) {
    if (storage != kStoreF32 || pair_needs_4(bcx, nx)) return 4;
    return (long long)nx * ny >= (1ll << 22) && pair_wide(pair_columns(nx, 2), pair_columns(nx, 4)) ? 4 : 2;
}
int pair_tile_rows(int npl) { return npl == 2 ? 6 : 7; }

// A pair halves the launches and the traffic but goes through the columns of whole
// strips and their halo.  Where those are 1.4 times the single steps' or more (1.5:
// 122 to 128 columns FP32, 241 to 256 16-bit; 2: 122 to 128 16-bit, 121 FP32) that
// decides, except on small lattices, where the launches do, and for FP32 beyond L2,
// where the traffic does.  Pair over single time, without bodies, at 2^16, 2^18, 2^20
// and 2^22 nodes: 128 columns FP32 0.66, 1.06, 1.01, 0.85, FP16 0.57, 1.12, 1.26, 1.28;
// 244 FP16 0.56, 0.98, 1.14, 1.15; 121 FP32 -, 1.22, 1.31, 1.14; with one body later:
// 128 FP16 0.59, 0.78, 1.25.  Below 1.4 pairs were never slower (364 FP16 1.05).
bool pairs_pay(int storage, bool bodies, double nodes, double pair, double single) {
    const double waste = pair / single;
    if (waste < 1.4) return true;
    auto below = [&](int log2) { return nodes < 0.75 * (1 << log2); };   // 3/4: sizes just below a power count as it
    if (storage != kStoreF32) return waste < 1.9 ? below(20) : below(bodies ? 19 : 18);
    if (waste >= 1.9 && single >= 128.0) return below(bodies ? 18 : 17);
    return below(bodies ? 19 : 18) || nodes >= 1.5 * (1 << 20);
}

namespace {

template <typename T>
cudaError_t pair_t(const void* gin, void* gout, const LatticeParams& p, const PairForces& q, bool pdl, cudaStream_t st) {
    if constexpr (sizeof(T) == 4)
        if (q.npl == 2) return pair_tn<T, 2, 8, 6, 5>(gin, gout, p, q, pdl, st);
    return pair_tn<T, 4, 9, 7, 3>(gin, gout, p, q, pdl, st);
}

template <typename T, int NPL, int NW, int TH, int MINB>
cudaError_t pair_batch_tn(const void* gin, void* gout, const PairBatch& b, const PairForces& q, bool pdl,
                          cudaStream_t st) {
    using C = PairTile<T, NPL, TH>;
    auto kern = pair_batch_kernel<T, NPL, NW, TH, MINB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kShared);
    if (e != cudaSuccess) return e;
    const int nred = std::min(16, std::max(1, (b.nbody + 2 * NW - 1) / (2 * NW)));
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = config((unsigned)(b.ntile + nred), 32 * NW, pdl, attr, st);
    cfg.dynamicSmemBytes = C::kShared;
    return cudaLaunchKernelEx(&cfg, kern, (const T*)gin, (T*)gout, b, q, nred);
}

template <typename T>
cudaError_t pair_batch_t(const void* gin, void* gout, const PairBatch& b, const PairForces& q, bool pdl,
                         cudaStream_t st) {
    if constexpr (sizeof(T) == 4)
        if (q.npl == 2) return pair_batch_tn<T, 2, 8, 6, 5>(gin, gout, b, q, pdl, st);
    return pair_batch_tn<T, 4, 9, 7, 3>(gin, gout, b, q, pdl, st);
}

template <typename T>
cudaError_t ib_pair_batch_t(int width, const void* g, const LatticeParams* descs, const unsigned long long* off,
                            const IbParams& q, const PairForces& r, const CsrEntry* csr, bool pdl, cudaStream_t st) {
    constexpr int W = kIbPairThreads / 32;
    const int mb = (q.nmark + W - 1) / W;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg =
        config((unsigned)(mb + (r.nnode + kIbPairThreads - 1) / kIbPairThreads), kIbPairThreads, pdl, attr, st);
    switch (width) {
    case 2: return cudaLaunchKernelEx(&cfg, ib_pair_batch_kernel<T, 2>, (const T*)g, descs, off, q, r, csr, mb);
    case 3: return cudaLaunchKernelEx(&cfg, ib_pair_batch_kernel<T, 3>, (const T*)g, descs, off, q, r, csr, mb);
    case 4: return cudaLaunchKernelEx(&cfg, ib_pair_batch_kernel<T, 4>, (const T*)g, descs, off, q, r, csr, mb);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t spread_second(const CsrEntry* csr, const float2* F, const PairForces& r, bool pdl, cudaStream_t st) {
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = config((unsigned)((r.nnode + 127) / 128), 128, pdl, attr, st);
    return cudaLaunchKernelEx(&cfg, spread_kernel, csr, F, r);
}

}  // namespace

cudaError_t launch_pair_batch(int storage, const void* gin, void* gout, const PairBatch& b, const PairForces& q,
                              bool pdl, cudaStream_t st) {
    switch (storage) {
    case kStoreF32: return pair_batch_t<float>(gin, gout, b, q, pdl, st);
    case kStoreF16: return pair_batch_t<__half>(gin, gout, b, q, pdl, st);
    case kStoreBF16: return pair_batch_t<__nv_bfloat16>(gin, gout, b, q, pdl, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_ib_pair_batch(int storage, int width, const void* g, const LatticeParams* descs,
                                 const unsigned long long* case_off, const IbParams& q, const PairForces& r,
                                 const CsrEntry* csr, bool pdl, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    switch (storage) {
    case kStoreF32: e = ib_pair_batch_t<float>(width, g, descs, case_off, q, r, csr, pdl, st); break;
    case kStoreF16: e = ib_pair_batch_t<__half>(width, g, descs, case_off, q, r, csr, pdl, st); break;
    case kStoreBF16: e = ib_pair_batch_t<__nv_bfloat16>(width, g, descs, case_off, q, r, csr, pdl, st); break;
    }
    return e != cudaSuccess ? e : spread_second(csr, q.F_out, r, pdl, st);
}

cudaError_t launch_pair(int storage, const void* gin, void* gout, const LatticeParams& p, const PairForces& q, bool pdl,
                        cudaStream_t st) {
    switch (storage) {
    case kStoreF32: return pair_t<float>(gin, gout, p, q, pdl, st);
    case kStoreF16: return pair_t<__half>(gin, gout, p, q, pdl, st);
    case kStoreBF16: return pair_t<__nv_bfloat16>(gin, gout, p, q, pdl, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_ib_pair(int storage, int width, const void* g, const LatticeParams& p, const IbParams& q,
                           const PairForces& r, bool pdl, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    switch (storage) {
    case kStoreF32: e = ib_pair_t<float>(width, g, p, q, r, pdl, st); break;
    case kStoreF16: e = ib_pair_t<__half>(width, g, p, q, r, pdl, st); break;
    case kStoreBF16: e = ib_pair_t<__nv_bfloat16>(width, g, p, q, r, pdl, st); break;
    }
    return e != cudaSuccess ? e : spread_second(p.csr, q.F_out, r, pdl, st);
}

}  // namespace btdf
