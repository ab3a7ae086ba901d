// btdf_adjoint.cu - discrete adjoint of one BTDF-IB/LBM time step (FP32
// storage, NF = 1).
//
// The forward step n maps the post-collision state g^n to g^{n+1}:
//   f = Pull(g^n) with the boundary rules,
//   rho_e, u*_e from f at the support nodes (Eqs. 9-10),
//   rho_l = sum_e W_le rho_e,  U*_l = sum_e W_le u*_e            (Eq. 14),
//   F_l = 2 rho_l (U_b - U*_l)                                    (Eq. 20),
//   F(x) = sum_l c_l W_lx F_l + body force,  c_l = drs_l ds_l      (Eq. 15),
//   g^{n+1}(x) = BGK collision of f(x) with the Guo term of F(x)   (Eqs. 5-7, 11),
// and the objective collects sum_l dJ/dF_l . F_l.  Given
// lam = dJ/dg^{n+1} the two kernels below form gbar = dJ/dg^n and
// accumulate dJ/dX_l, dJ/dY_l and the inlet part of dJ/dU_in:
//   (A) marker-parallel: adjoint of the force law and of spreading and
//       interpolation with respect to the forces and the marker positions.  It
//       needs dJ/dF(x) at the support nodes only and forms it there itself, so
//       it comes first and stays small;
//   (B) node-parallel: adjoint of the collision, of the interpolation (at the
//       nodes that markers cover) and of the inlet and outlet rules (folded
//       into columns 1 and nx-2), then the transpose of the pull.
// The pull reads every stored population at most once, so its adjoint is a
// scatter with a unique writer per entry: plain vector stores, and zeros where
// the pull reads nothing.
#include "btdf_internal.cuh"
#include "btdf_device.cuh"

namespace btdf {
namespace {

constexpr int kAdjThreads = 128;
constexpr int kAdjIbThreads = 64;

// Node force of the step at (x, y) (Eq. 15 plus the uniform body force) and the
// range of its spread terms.
__device__ __forceinline__ void node_force(const LatticeParams& p, int x, int y, float& Fx, float& Fy, int& b,
                                           int& e) {
    Fx = 0.f;
    Fy = 0.f;
    b = e = 0;
    if (p.seg_index != nullptr) {
        const int seg = __ldg(p.seg_index + y * p.nseg + x / kSeg);
        if (seg >= 0) {
            const int* ptr = p.seg_ptr + (long long)seg * (kSeg + 1) + (x % kSeg);
            b = __ldg(ptr);
            e = __ldg(ptr + 1);
            for (int k = b; k < e; k++) {
                const CsrEntry c = p.csr[k];
                const float2 F = p.F[c.marker];
                Fx = __fmaf_rn(c.w, F.x, Fx);
                Fy = __fmaf_rn(c.w, F.y, Fy);
            }
        }
    }
    Fx += p.gx;
    Fy += p.gy;
}

// Adjoint of the collision (Eqs. 5-7 with Eq. 11) at one node.  With full
// populations f, rho = sum f, m = rho u = sum e f + F/2 and B = 1 - omega/2:
//   g'_a = (1 - omega) f_a + omega w_a [rho + 3 e.m + (4.5 (e.m)^2 - 1.5 m.m) / rho]
//          + B w_a [3 e.F - 3 m.F / rho + 9 (e.m)(e.F) / rho].
// Given lam_a = dJ/dg'_a returns fb_b = dJ/df_b and (Fbx, Fby) = dJ/dF.
__device__ __forceinline__ void adj_collide(const LatticeParams& p, const float d[9], float Fx, float Fy,
                            const float lam[9], float fb[9], float& Fbx, float& Fby) {
    float rho = 0.f, jx = 0.f, jy = 0.f;
#pragma unroll
    for (int a = 0; a < 9; a++) {
        const float fa = d[a] + wt(a) * (1.0f + eq_part(a, p.urx, p.ury));   // full population
        rho += fa;
        jx += ex(a) * fa;
        jy += ey(a) * fa;
    }
    const float om = p.omega, B = 1.0f - 0.5f * om;
    const float mx = jx + 0.5f * Fx, my = jy + 0.5f * Fy;
    const float ir = 1.0f / rho, ir2 = ir * ir;
    const float m2 = mx * mx + my * my, mF = mx * Fx + my * Fy;
    float rb = 0.f, mbx = 0.f, mby = 0.f, Fex = 0.f, Fey = 0.f;
#pragma unroll
    for (int a = 0; a < 9; a++) {
        const float l = lam[a] * wt(a);
        const float em = ex(a) * mx + ey(a) * my, eF = ex(a) * Fx + ey(a) * Fy;
        // d/drho
        rb += l * (om * (1.0f - (4.5f * em * em - 1.5f * m2) * ir2) + B * (3.0f * mF - 9.0f * em * eF) * ir2);
        // d/dm
        const float cm = om * (3.0f + 9.0f * em * ir) + B * 9.0f * eF * ir;
        mbx += l * (cm * ex(a) - (om * 3.0f * mx + B * 3.0f * Fx) * ir);
        mby += l * (cm * ey(a) - (om * 3.0f * my + B * 3.0f * Fy) * ir);
        // d/dF at fixed m
        const float ce = B * (3.0f + 9.0f * em * ir);
        Fex += l * (ce * ex(a) - B * 3.0f * mx * ir);
        Fey += l * (ce * ey(a) - B * 3.0f * my * ir);
    }
#pragma unroll
    for (int b = 0; b < 9; b++) fb[b] = (1.0f - om) * lam[b] + rb + ex(b) * mbx + ey(b) * mby;
    Fbx = Fex + 0.5f * mbx;   // m depends on F through F/2
    Fby = Fey + 0.5f * mby;
}

// (A) marker-parallel, G lanes per marker (one per support node).  The
// interpolation is recomputed from g^n and dJ/dF(e) at the support nodes from
// lam; then
//   dJ/dF_l   = c_l sum_e W_le dJ/dF(e) + (objective weight of F_l),
//   dJ/dU*_l  = -2 rho_l dJ/dF_l,   dJ/drho_l = 2 (U_b - U*_l) . dJ/dF_l,
// and, W_le depending on the marker position through delta(x_e - X) delta(y_e - Y),
//   dJ/dX_l  += sum_e dW_le/dX_l [dJ/dU*_l . u*_e + dJ/drho_l rho_e + c_l F_l . dJ/dF(e)]
// (the same with Y).  dJ/drho_l and dJ/dU*_l go to (B) through mbar.
template <int S>
__global__ void __launch_bounds__(kAdjIbThreads)
adj_ib_kernel(const float* __restrict__ g, const float* __restrict__ lam, LatticeParams p, AdjParams q, int pull) {
    constexpr int G = Group<S>::G;
    const long long m = ib_marker_index<float, S>();
    const int lane = threadIdx.x & 31;
    const int li = lane % G;
    const bool valid = m < q.nmark;
    const long long mm = valid ? m : 0;
    const MarkerAux ax = q.aux[mm];
    const AdjMarker am = q.am[mm];
    const float c = q.cscale[mm];
    const float2 ow = q.objw[mm];
    float w = 0.f, dwx = 0.f, dwy = 0.f, rho = 1.f, dux = 0.f, duy = 0.f, drho = 0.f;
    float Fex = 0.f, Fey = 0.f;
    int x = 0, y = 0;
    if (valid && li < S * S) {
        const int xi = li % S, yi = li / S;
        const Marker* mk = q.mk + mm;
        w = __ldg(&mk->w[li]);
        dwx = am.dwx[xi] * am.wy[yi];
        dwy = am.wx[xi] * am.dwy[yi];
        x = __ldg(&mk->xs[xi]);
        y = __ldg(&mk->ys[yi]);
    }
    // lam and g come from the kernel before; the dependent grid (B) may start
    // once it has finished
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    if (w != 0.f || dwx != 0.f || dwy != 0.f) {
        float d[9], l[9], fb[9];
#pragma unroll
        for (int a = 0; a < 9; a++) l[a] = lam[p.poff[a] + (unsigned)y * p.rs + (unsigned)x];
        gather_node<float>(g, p, pull != 0, x, y, d);
        const Moments mo = moments(d, p.urx, p.ury);
        rho = mo.rho;
        drho = mo.drho;
        dux = mo.dux;
        duy = mo.duy;
        if (__ldg(p.seg_index + y * p.nseg + x / kSeg) >= 0) {
            float Fx, Fy;
            int b, e;
            node_force(p, x, y, Fx, Fy, b, e);
            adj_collide(p, d, Fx, Fy, l, fb, Fex, Fey);
        }
    }
    float sr = w * drho, su = w * dux, sv = w * duy, sfx = w * Fex, sfy = w * Fey;
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
        sr += __shfl_xor_sync(kFull, sr, off);
        su += __shfl_xor_sync(kFull, su, off);
        sv += __shfl_xor_sync(kFull, sv, off);
        sfx += __shfl_xor_sync(kFull, sfx, off);
        sfy += __shfl_xor_sync(kFull, sfy, off);
    }
    const float rl = ax.wsum + sr;                              // rho_l
    const float vx = ax.ubx_rel - su, vy = ax.uby_rel - sv;     // U_b - U*_l
    const float Flx = 2.0f * rl * vx, Fly = 2.0f * rl * vy;     // F_l
    const float Fbx = c * sfx + ow.x, Fby = c * sfy + ow.y;     // dJ/dF_l
    const float ubx = -2.0f * rl * Fbx, uby = -2.0f * rl * Fby; // dJ/dU*_l
    const float rb = 2.0f * (vx * Fbx + vy * Fby);              // dJ/drho_l
    const float h = ubx * (p.urx + dux) + uby * (p.ury + duy) + rb * rho + c * (Flx * Fex + Fly * Fey);
    float gX = dwx * h, gY = dwy * h;
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
        gX += __shfl_xor_sync(kFull, gX, off);
        gY += __shfl_xor_sync(kFull, gY, off);
    }
    if (valid && li == 0) {
        q.dJdX[mm] += (double)gX;
        q.dJdY[mm] += (double)gY;
        q.mbar[mm] = make_float4(rb, ubx, uby, 0.f);
    }
}

// (B) one warp per row segment of 60 nodes, two per lane; the outer lanes hold
// the nodes beside it, whose dJ/df the transposed shift along x brings in.
//
// What bounds it: latency.  72 bytes a node read and 36 written (g, lam, gbar) are
// 35 MB on 800 x 400, in L2.  One thread per node with run-time boundary cases,
// scalar loads, a zeroed buffer and a second kernel for the band nodes took 47 us
// a reverse step there (recomputation included), a 500-step window with its
// gradients 34.9 ms; this form takes 20.6 ms.
constexpr int kAdjNpl = 2;
constexpr int kAdjOwn = 30 * kAdjNpl;

__global__ void __launch_bounds__(kAdjThreads)
adj_node_kernel(const float* __restrict__ g, const float* __restrict__ lam, float* __restrict__ gbar,
                const __grid_constant__ LatticeParams p, const __grid_constant__ AdjParams q, int pull, int nstrip) {
    cudaTriggerProgrammaticLaunchCompletion();   // the next step's first kernel waits for this grid
    constexpr int N = kAdjNpl;
    const int lane = threadIdx.x & 31;
    const int u = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int y = u / nstrip, s = u - y * nstrip;
    const int nx = p.nx, ny = p.ny;
    if (y >= ny) return;   // whole warps
    const bool perx = p.bcx == kBcxPeriodic, noslip = p.bcy == kBcyNoslip;
    const bool inout = pull && !perx;
    const int xs = s * kAdjOwn - N, x0 = xs + N * lane;
    const int x0c = min(max(x0, 0), p.nxp - N);
    const bool own = lane > 0 && lane < 31 && x0 < nx;
    const bool ends = xs <= 0 || xs + 32 * N >= nx;
    const bool wraps = perx && ends && (x0 < 0 || x0 + N > nx);
    int xc[N];   // the nodes' columns, wrapped under periodic x
#pragma unroll
    for (int i = 0; i < N; i++) xc[i] = perx ? ((x0 + i) % nx + nx) % nx : x0 + i;

    // dJ/dg' at the nodes and the post-streaming state there
    float l[N][9], f[N][9];
    float2 raw[9];
    const bool inner = y > 0 && y < ny - 1;
#pragma unroll
    for (int a = 0; a < 9; a++) {
        int pa = a, sy = y, dx = 0;
        if (pull) {
            sy = y - ey(a);
            if (!inner) {
                float unused;
                y_source(a, y, p, pa, sy, dx, unused);
            }
        }
        const float* src = g + (p.poff[pa] + (unsigned)sy * p.rs);
        const float* lrow = lam + (p.poff[a] + (unsigned)y * p.rs);
        float2 v = *reinterpret_cast<const float2*>(src + x0c), m = *reinterpret_cast<const float2*>(lrow + x0c);
        if (wraps) {
            v = make_float2(src[xc[0]], src[xc[1]]);
            m = make_float2(lrow[xc[0]], lrow[xc[1]]);
        }
        raw[a] = v;
        l[0][a] = m.x;
        l[1][a] = m.y;
    }
#pragma unroll
    for (int a = 0; a < 9; a++) {
        float2 v = raw[a];
        const bool wall = !inner && (ey(a) > 0 ? y == 0 : ey(a) < 0 && y == ny - 1) && noslip;
        if (pull && ex(a) > 0) {
            const float prev = __shfl_up_sync(kFull, v.y, 1);
            if (!wall) v = make_float2(prev, v.x);
        } else if (pull && ex(a) < 0) {
            const float next = __shfl_down_sync(kFull, v.x, 1);
            if (!wall) v = make_float2(v.y, next);
        }
        if (pull && wall) {
            const float add = __fmul_rn(-6.0f * wt(a), p.eur[a]);
            v = make_float2(__fadd_rn(v.x, add), __fadd_rn(v.y, add));
        }
        f[0][a] = v.x;
        f[1][a] = v.y;
    }
    float f1[9];   // the state of column 1 beside an inlet node
#pragma unroll
    for (int a = 0; a < 9; a++) f1[a] = f[1][a];
    if (inout && ends) {
        // inlet node from column 1, outlet node copied from column nx - 2
        if (x0 == 0) inlet_from(f1, p, f[0]);
        const int i = nx - 1 - x0;
#pragma unroll
        for (int a = 0; a < 9; a++) {
            const float v = __shfl_up_sync(kFull, f[1][a], 1);
            if (i == 0) f[0][a] = v;
            if (i == 1) f[1][a] = f[0][a];
        }
    }

    float fb[N][9];
    int tb[N], te[N];   // spread terms of the nodes
#pragma unroll
    for (int i = 0; i < N; i++) {
        float Fx = p.gx, Fy = p.gy, Fbx, Fby;
        tb[i] = te[i] = 0;
        if (xc[i] >= 0 && xc[i] < nx) node_force(p, xc[i], y, Fx, Fy, tb[i], te[i]);
        adj_collide(p, f[i], Fx, Fy, l[i], fb[i], Fbx, Fby);
    }
    if (inout && ends) {
        if (x0 == 0) {
            // Inlet by non-equilibrium extrapolation from column 1 (post-stream
            // f1, pre-force u1 = J1 / rho1):
            //   f_a(0) = f1_a + w_a [rho1 P_a(U_in) - 3 e.J1 - (4.5 (e.J1)^2 - 1.5 J1.J1) / rho1].
            float r1 = 0.f, jx = 0.f, jy = 0.f;
#pragma unroll
            for (int a = 0; a < 9; a++) {
                const float fa = f1[a] + wt(a) * (1.0f + eq_part(a, p.urx, p.ury));
                r1 += fa;
                jx += ex(a) * fa;
                jy += ey(a) * fa;
            }
            const float ir = 1.0f / r1, U = p.u_in;
            const float j2 = jx * jx + jy * jy;
            float sb = 0.f, sjx = 0.f, sjy = 0.f, dU = 0.f;
#pragma unroll
            for (int a = 0; a < 9; a++) {
                const float lw = fb[0][a] * wt(a);
                const float ej = ex(a) * jx + ey(a) * jy;
                const float PU = 3.0f * ex(a) * U + 4.5f * ex(a) * ex(a) * U * U - 1.5f * U * U;
                sb += lw * (PU + (4.5f * ej * ej - 1.5f * j2) * ir * ir);       // d/drho1
                const float cj = 3.0f + 9.0f * ej * ir;
                sjx += lw * (cj * ex(a) - 3.0f * jx * ir);                        // d/dJ1
                sjy += lw * (cj * ey(a) - 3.0f * jy * ir);
                dU += lw * r1 * (3.0f * ex(a) + 9.0f * ex(a) * ex(a) * U - 3.0f * U);   // d/dU_in
            }
#pragma unroll
            for (int b = 0; b < 9; b++) fb[1][b] += fb[0][b] + sb - (ex(b) * sjx + ey(b) * sjy);
            atomicAdd(q.dU, (double)dU);
        }
        const int i = nx - 2 - x0;   // f(nx-1) = f(nx-2)
#pragma unroll
        for (int b = 0; b < 9; b++) {
            const float next = __shfl_down_sync(kFull, fb[0][b], 1);
            if (i == 1) fb[1][b] += next;
            if (i == 0) fb[0][b] += fb[1][b];
        }
    }
    // adjoint of the interpolation at the nodes that markers cover (rho = sum f,
    // u* = sum e f / rho, so d/df_b = rho_bar + (e_b - u*) . U*_bar / rho)
    if (__any_sync(kFull, te[0] > tb[0] || te[1] > tb[1])) {
        cudaGridDependencySynchronize();
#pragma unroll
        for (int i = 0; i < N; i++) {
            if (te[i] <= tb[i]) continue;
            float rb = 0.f, ubx = 0.f, uby = 0.f;
            for (int k = tb[i]; k < te[i]; k++) {
                const CsrEntry c = p.csr[k];
                const float W = c.w / q.cscale[c.marker];
                const float4 mb = q.mbar[c.marker];
                rb = __fmaf_rn(W, mb.x, rb);
                ubx = __fmaf_rn(W, mb.y, ubx);
                uby = __fmaf_rn(W, mb.z, uby);
            }
            const Moments mo = moments(f[i], p.urx, p.ury);
            const float ux = p.urx + mo.dux, uy = p.ury + mo.duy;
            const float jbx = ubx * mo.inv, jby = uby * mo.inv;
            const float rbar = rb - (ux * ubx + uy * uby) * mo.inv;
#pragma unroll
            for (int b = 0; b < 9; b++) fb[i][b] += rbar + ex(b) * jbx + ey(b) * jby;
        }
    }
    // transpose of the pull: stored entry (pa, x', sy) <- fb_a(x' - dx)
#pragma unroll
    for (int a = 0; a < 9; a++) {
        int pa = a, sy = y, dx = 0;
        if (pull) {
            sy = y - ey(a);
            dx = -ex(a);
            if (!inner) {
                float unused;
                y_source(a, y, p, pa, sy, dx, unused);
            }
        }
        float2 v = make_float2(fb[0][a], fb[1][a]);
        int t0 = x0;   // the node the first value comes from
        if (ex(a) > 0) {
            const float next = __shfl_down_sync(kFull, v.x, 1);
            if (dx != 0) {
                v = make_float2(v.y, next);
                t0 = x0 + 1;
            }
        } else if (ex(a) < 0) {
            const float prev = __shfl_up_sync(kFull, v.y, 1);
            if (dx != 0) {
                v = make_float2(prev, v.x);
                t0 = x0 - 1;
            }
        }
        if (inout) {   // nodes 0 and nx - 1 pull nothing of their own
            if (t0 < 1 || t0 > nx - 2) v.x = 0.f;
            if (t0 + 1 < 1 || t0 + 1 > nx - 2) v.y = 0.f;
        }
        if (own) *reinterpret_cast<float2*>(gbar + (p.poff[pa] + (unsigned)sy * p.rs + (unsigned)x0c)) = v;
    }
}

template <typename K, typename... A>
cudaError_t launch_pdl(K kern, long long threads, int block, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((threads + block - 1) / block));
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace

// Both kernels are programmatic dependents: (A) waits for the step before, whose
// lam it reads, and only then lets (B) start; (B)'s warps off the markers'
// supports wait for nothing.
cudaError_t launch_adjoint_step(const float* g, const float* lam, float* gbar, const LatticeParams& p,
                                const AdjParams& q, int width, bool pull, cudaStream_t st) {
    const int pl = pull ? 1 : 0;
    const int G = width * width <= 4 ? 4 : 16;
    const long long lanes = ((long long)q.nmark + 32 / G - 1) / (32 / G) * 32;
    cudaError_t e;
    switch (width) {
    case 2: e = launch_pdl(adj_ib_kernel<2>, lanes, kAdjIbThreads, st, g, lam, p, q, pl); break;
    case 3: e = launch_pdl(adj_ib_kernel<3>, lanes, kAdjIbThreads, st, g, lam, p, q, pl); break;
    case 4: e = launch_pdl(adj_ib_kernel<4>, lanes, kAdjIbThreads, st, g, lam, p, q, pl); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int nstrip = (p.nx + kAdjOwn - 1) / kAdjOwn;
    return launch_pdl(adj_node_kernel, 32ll * nstrip * p.ny, kAdjThreads, st, g, lam, gbar, p, q, pl, nstrip);
}

}  // namespace btdf
