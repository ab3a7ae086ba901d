// btdf_collide.cuh - the collision of a lane's nodes (moments, velocity
// correction, BGK with the Guo term), shared by every forward kernel, so that
// all of them round alike.
#pragma once

#include "btdf_device.cuh"

namespace btdf {
namespace {

// Spread force (Eq. 15) of the terms b .. e-1.  The first kTerms of them are
// loaded ahead (no kernel of a step writes them), so that only the loads of the
// forces, all at once, follow the wait for the kernel that writes those.
constexpr int kTerms = 8;
struct SpreadTerms {
    CsrEntry c[kTerms];
    int b, e;
    __device__ __forceinline__ void load(const CsrEntry* csr, int b_, int e_) {
        b = b_;
        e = e_;
#pragma unroll
        for (int k = 0; k < kTerms; k++) {
            c[k] = CsrEntry{0, 0.f};
            if (b + k < e) c[k] = csr[b + k];
        }
    }
    __device__ __forceinline__ void sum(const CsrEntry* csr, const float2* F, float& sx, float& sy) const {
        float2 f[kTerms];
#pragma unroll
        for (int k = 0; k < kTerms; k++) f[k] = b + k < e ? F[c[k].marker] : make_float2(0.f, 0.f);
        sx = 0.f;
        sy = 0.f;
#pragma unroll
        for (int k = 0; k < kTerms; k++)
            if (b + k < e) {
                sx = __fmaf_rn(c[k].w, f[k].x, sx);
                sy = __fmaf_rn(c[k].w, f[k].y, sy);
            }
        for (int k = b + kTerms; k < e; k++) {
            const CsrEntry t = csr[k];
            const float2 v = F[t.marker];
            sx = __fmaf_rn(t.w, v.x, sx);
            sy = __fmaf_rn(t.w, v.y, sy);
        }
    }
};

// Forces on the bodies (Eq. 27) in step `step` from its Lagrangian forces, in
// FP64, into the history ring, by warp `warp` of `nwarps`; body b's markers are
// ptr[b * stride] .. ptr[b * stride + 1] - 1.  FP64 arithmetic is slow on this
// part and, on small lattices, this reduction is on the step's critical path:
// one warp per body and no work for absent bodies.
__device__ __forceinline__ void body_forces(int nbody, const int* ptr, int stride, const double* scale, double2* hist,
                                            int hist_len, const float2* Fl, unsigned long long step, int warp,
                                            int nwarps) {
    const int lane = threadIdx.x & 31;
    const long long slot = (long long)(step % (unsigned long long)(hist_len > 0 ? hist_len : 1)) * nbody;
    for (int b = warp; b < nbody; b += nwarps) {
        double sx = 0.0, sy = 0.0;
        for (int k = ptr[b * stride] + lane; k < ptr[b * stride + 1]; k += 32) {
            const float2 F = Fl[k];
            sx += (double)F.x;
            sy += (double)F.y;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            sx += __shfl_xor_sync(kFull, sx, off);
            sy += __shfl_xor_sync(kFull, sy, off);
        }
        if (lane == 0) {
            const double sc = scale[b];
            hist[slot + b] = make_double2(-sx * sc, -sy * sc);
        }
    }
}
__device__ __forceinline__ void body_forces(const LatticeParams& p, const float2* Fl, unsigned long long step,
                                            int warp, int nwarps) {
    body_forces(p.nbody, p.body_ptr, 1, p.body_scale, p.hist, p.hist_len, Fl, step, warp, nwarps);
}

// f holds the post-streaming deviations of NPL nodes at their stored scale,
// (Fx, Fy) the force density of the spread (Eq. 15), without the uniform body
// force; forced: any of them, or the uniform force, is not zero.  Calls
// begin() between the moments and the collision, then store(a, o) with the NPL
// post-collision values of population a (stored scale), one population after
// the other.
template <typename T, int NPL, typename Begin, typename Store>
__device__ __forceinline__ void collide_nodes(const float (&f)[9][NPL], const LatticeParams& p,
                                              float (&Fx)[NPL], float (&Fy)[NPL], bool forced,
                                              Begin&& begin, Store&& store) {
    // Moments (Eqs. 9-10) and the velocity correction u = u* + f / (2 rho)
    // (Eq. 11), as deviations from the reference state.
    float drho[NPL], rho[NPL], du[NPL], dv[NPL], pd0[NPL], uF[NPL], inv[NPL];
    if constexpr (NPL % 2 == 0) {
        // node pairs through the packed FP32x2 instructions
#pragma unroll
        for (int j = 0; j < NPL; j += 2) {
            float2 d[9];
#pragma unroll
            for (int a = 0; a < 9; a++) d[a] = make_float2(f[a][j], f[a][j + 1]);
            const Moments2 m = moments2(d, p.urx, p.ury, 1.0f / Raw<T>::kScale);
            drho[j] = m.drho.x; drho[j + 1] = m.drho.y;
            rho[j] = m.rho.x; rho[j + 1] = m.rho.y;
            inv[j] = m.inv.x; inv[j + 1] = m.inv.y;
            du[j] = m.dux.x; du[j + 1] = m.dux.y;
            dv[j] = m.duy.x; dv[j + 1] = m.duy.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NPL; i++) {
            float d[9];
#pragma unroll
            for (int a = 0; a < 9; a++) d[a] = f[a][i];
            const Moments m = moments(d, p.urx, p.ury, 1.0f / Raw<T>::kScale);
            drho[i] = m.drho;
            rho[i] = m.rho;
            inv[i] = m.inv;
            du[i] = m.dux;
            dv[i] = m.duy;
        }
    }
#pragma unroll
    for (int i = 0; i < NPL; i++) {
        uF[i] = 0.0f;
        if (forced) {
            Fx[i] += p.gx;
            Fy[i] += p.gy;
            du[i] = __fmaf_rn(__fmul_rn(0.5f, Fx[i]), inv[i], du[i]);
            dv[i] = __fmaf_rn(__fmul_rn(0.5f, Fy[i]), inv[i], dv[i]);
            uF[i] = __fmaf_rn(p.urx + du[i], Fx[i], __fmul_rn(p.ury + dv[i], Fy[i]));
        }
    }
    // 1.5 (2 U_r.du + du^2), the velocity part shared by all populations
    auto velocity_term = [&]() {
#pragma unroll
        for (int i = 0; i < NPL; i++) {
            float t = __fmaf_rn(du[i], du[i], __fmul_rn(dv[i], dv[i]));
            t = __fmaf_rn(2.0f * p.urx, du[i], t);
            t = __fmaf_rn(2.0f * p.ury, dv[i], t);
            pd0[i] = __fmul_rn(1.5f, t);
        }
    };

    begin();
    // Collision (Eqs. 5-7), one population at a time, in the form
    //   d_eq / w = drho (1 + P(U_r)) + rho (P(u) - P(U_r))
    //   P(u) - P(U_r) = ed (3 + 9 e.U_r + 4.5 ed) - 1.5 (2 U_r.du + du^2),  ed = e.du
    //   d' = (1 - 1/tau) d + (w / tau) d_eq / w
    //        + (1 - 1/(2 tau)) w [e.F (3 + 9 e.u) - 3 u.F]
    if (NPL % 2 == 0 && !forced) {
        constexpr int NP = NPL / 2 > 0 ? NPL / 2 : 1;
        float2 U[NP], V[NP], nU[NP], nV[NP], D[NP], R[NP], P[NP];
#pragma unroll
        for (int j = 0; j < NP; j++) {
            U[j] = make_float2(du[2 * j], du[2 * j + 1]);
            V[j] = make_float2(dv[2 * j], dv[2 * j + 1]);
            nU[j] = mul2(U[j], f2(-1.0f));
            nV[j] = mul2(V[j], f2(-1.0f));
            D[j] = make_float2(drho[2 * j], drho[2 * j + 1]);
            R[j] = make_float2(rho[2 * j], rho[2 * j + 1]);
            // -pd0 of velocity_term for the pair (-1.5 t is exactly -(1.5 t))
            float2 t = fma2(U[j], U[j], mul2(V[j], V[j]));
            t = fma2(f2(2.0f * p.urx), U[j], t);
            t = fma2(f2(2.0f * p.ury), V[j], t);
            P[j] = mul2(f2(-1.5f), t);
        }
#pragma unroll
        for (int a = 0; a < 9; a++) {
            float o[NPL];
#pragma unroll
            for (int j = 0; j < NP; j++) {
                const float2 ed = edot2(a, U[j], V[j], nU[j], nV[j]);
                const float2 pdiff = fma2(ed, fma2(f2(4.5f), ed, p.c1p[a]), P[j]);
                const float2 deqw = fma2(R[j], pdiff, mul2(p.krp[a], D[j]));
                const float2 r = fma2(p.womp[a], deqw, mul2(p.omop, make_float2(f[a][2 * j], f[a][2 * j + 1])));
                o[2 * j] = r.x;
                o[2 * j + 1] = r.y;
            }
            store(a, o);
        }
    } else if (!forced) {
        velocity_term();
#pragma unroll
        for (int a = 0; a < 9; a++) {
            float o[NPL];
#pragma unroll
            for (int i = 0; i < NPL; i++) {
                const float ed = edot(a, du[i], dv[i]);
                const float pdiff = __fmaf_rn(ed, __fmaf_rn(4.5f, ed, p.c1[a]), -pd0[i]);
                const float deqw = __fmaf_rn(rho[i], pdiff, __fmul_rn(p.kr[a], drho[i]));
                o[i] = __fmaf_rn(p.wom[a], deqw, __fmul_rn(p.one_m_omega, f[a][i]));
            }
            store(a, o);
        }
    } else {
        velocity_term();
#pragma unroll
        for (int a = 0; a < 9; a++) {
            float o[NPL];
#pragma unroll
            for (int i = 0; i < NPL; i++) {
                const float ed = edot(a, du[i], dv[i]);
                const float pdiff = __fmaf_rn(ed, __fmaf_rn(4.5f, ed, p.c1[a]), -pd0[i]);
                const float deqw = __fmaf_rn(rho[i], pdiff, __fmul_rn(p.kr[a], drho[i]));
                float r = __fmaf_rn(p.wom[a], deqw, __fmul_rn(p.one_m_omega, f[a][i]));
                const float eF = edot(a, Fx[i], Fy[i]);
                const float eu = p.eur[a] + ed;
                const float g = __fmaf_rn(eF, __fmaf_rn(9.0f, eu, 3.0f), __fmul_rn(-3.0f, uF[i]));
                o[i] = __fmaf_rn(p.wg[a], g, r);
            }
            store(a, o);
        }
    }
}

}  // namespace
}  // namespace btdf
