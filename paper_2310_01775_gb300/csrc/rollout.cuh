// Device bodies of the relaxed block-pushing simulation (Sec. III-B; Algorithm
// 1 "simulate plans" and the gradient of log rho): the relaxation, the contact
// forces and their derivatives.  block_team.cuh builds the rollout and its
// reverse sweep from them.
//
// Physics (all choices restate the paper's model class: kinematic pushers,
// spring-damper penalty contact, smoothed Coulomb friction, semi-implicit
// Euler):
//   pusher c = (object o = c/4, side s = c%4), sides N,E,S,W with outward
//   normals (0,1),(1,0),(0,-1),(-1,0); it starts touching side s at
//   tangential offset `off` and moves `dist` along the inward normal over T
//   substeps; during substep j (0-based) its centre is p0 + (j+1)*delta,
//   delta = -R(yaw_o) n_s * dist/T, its velocity delta/dt;
//   every pusher acts on every block with weight z_{k,c};
//   disk/box contact: delta = r - sd, f_n = max(0, k*delta - c*v_n),
//   smoothed Coulomb tangential force mu_c*f_n*w_t/sqrt(|w_t|^2+eps_t^2);
//   box/box: the 8 corners of each pair tested against the other box;
//   ground: -mu*m*g*v/sqrt(|v|^2+eps_v^2), -mu*m*g*r_eff*w/sqrt(w^2+eps_w^2).
#pragma once

#include <cfloat>
#include <cstdint>

#include "stamp_internal.cuh"

namespace stamp {
namespace rollout {

template <int NB>
struct Dims {
    static constexpr int M = 4 * NB;              // choices per action
    static constexpr int P = M + 2;               // parameters per action
    static constexpr int S = 6 * NB;              // state floats per particle
};

template <int NB>
struct Blocks {
    float x[NB], y[NB], ph[NB], vx[NB], vy[NB], om[NB];
};

// sin/cos of a yaw (full-accuracy sincosf: the hardware approximation's
// ~4e-7 absolute error measurably degrades parity through the contact
// dynamics).
__device__ __forceinline__ void yaw_sincos(float x, float* s, float* c) { sincosf(x, s, c); }

__device__ __forceinline__ void side_normal(int s, float& nx, float& ny) {
    nx = (s == 1) ? 1.f : (s == 3) ? -1.f : 0.f;
    ny = (s == 0) ? 1.f : (s == 2) ? -1.f : 0.f;
}

// Relaxed action parameters of action k for particle row `th`
// (Eq. gamma_map: softmax((a+g)/tau), or one-hot argmax when hard).
template <int NB>
__device__ __forceinline__ void relax_action(const SimConst& sc, const float* th, int k, int i,
                                             uint64_t gkey, bool noise, bool hard,
                                             float (&z)[Dims<NB>::M], float& uu, float& vv) {
    constexpr int M = Dims<NB>::M, P = Dims<NB>::P;
    const float* a = th + k * P;
#pragma unroll
    for (int c = 0; c < M; ++c) {
        float v = a[c];
        if (noise) {
            const float u = u23(sm64(gkey, (uint64_t)((i * sc.H + k) * M + c)));
            v += -logf(-logf(u));
        }
        z[c] = v;
    }
    if (hard) {
        int best = 0;
        float bv = z[0];
#pragma unroll
        for (int c = 1; c < M; ++c)
            if (z[c] > bv) { bv = z[c]; best = c; }
#pragma unroll
        for (int c = 0; c < M; ++c) z[c] = (c == best) ? 1.f : 0.f;
    } else {
        float mx = z[0] * sc.inv_tau;
#pragma unroll
        for (int c = 1; c < M; ++c) mx = fmaxf(mx, z[c] * sc.inv_tau);
        float sum = 0.f;
#pragma unroll
        for (int c = 0; c < M; ++c) { z[c] = expf(z[c] * sc.inv_tau - mx); sum += z[c]; }
        const float inv = 1.f / sum;
#pragma unroll
        for (int c = 0; c < M; ++c) z[c] *= inv;
    }
    uu = a[M];
    vv = a[M + 1];
}

// a b + c d with the first product fused.  Where a sum has two products, the
// compiler may fuse either, and picks by context: written out, every kernel
// and team width rounds alike (the dynamics amplify a last bit).
__device__ __forceinline__ float dot2(float a, float b, float c, float d) {
    return fmaf(a, b, __fmul_rn(c, d));
}

__device__ __forceinline__ float sigmoidf_(float v) { return 1.f / (1.f + expf(-v)); }

// ------------------------------- forces -------------------------------------
// A pusher centre (corner) at offset (dx, dy) from a block centre farther
// than the block's reach cannot touch it: the contact tests below return no
// contact there, so callers may skip them.
__device__ __forceinline__ bool out_of_reach(float dx, float dy, float reach2) {
    return dot2(dx, dx, dy, dy) > reach2;
}

// Corner k (position, velocity) of one box against square B: force on the
// corner's owner (B receives the opposite at the same point).
__device__ __forceinline__ void corner_box(const SimConst& sc, float kx, float ky, float kvx,
                                           float kvy, float bx, float by, float cph, float sph,
                                           float vx, float vy, float om, float& fx, float& fy) {
    fx = fy = 0.f;
    const float dx = kx - bx, dy = ky - by;
    if (out_of_reach(dx, dy, sc.corner_reach2)) return;   // no contact
    const float lx = dot2(cph, dx, sph, dy), ly = dot2(cph, dy, -sph, dx);
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    if (!(qx < 0.f && qy < 0.f)) return;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool xa = qx >= qy;
    const float nlx = xa ? sx : 0.f, nly = xa ? 0.f : sy;
    const float delta = -(xa ? qx : qy);
    const float nx = dot2(cph, nlx, -sph, nly), ny = dot2(sph, nlx, cph, nly);
    const float wx = kvx - fmaf(-om, dy, vx), wy = kvy - fmaf(om, dx, vy);
    const float vn = dot2(wx, nx, wy, ny);
    const float fn = dot2(sc.k, delta, -sc.c, vn);
    if (!(fn > 0.f)) return;
    const float tx = fmaf(-vn, nx, wx), ty = fmaf(-vn, ny, wy);
    const float gt = sc.mu_c * fn * rsqrtf(dot2(tx, tx, ty, ty) + sc.eps_t2);
    fx = dot2(fn, nx, -gt, tx);
    fy = dot2(fn, ny, -gt, ty);
}

// State row of one particle: per block (x, y), (ph, vx), (vy, om).
template <int NB>
__device__ __forceinline__ void load_state(const float2* src, Blocks<NB>& s) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const float2 p = src[3 * b], q = src[3 * b + 1], r = src[3 * b + 2];
        s.x[b] = p.x; s.y[b] = p.y;
        s.ph[b] = q.x; s.vx[b] = q.y;
        s.vy[b] = r.x; s.om[b] = r.y;
    }
}

__device__ __forceinline__ float wrapf(float e) { return atan2f(sinf(e), cosf(e)); }

// ------------------------------ adjoint pieces -------------------------------
// VJP of one corner test.  gO*/gB*: adjoints of the owner's / other box's
// force and torque.  Returns the adjoints of both boxes' states.
struct CornerGrad {
    float ox, oy, oph, ovx, ovy, oom, bx, by, bph, bvx, bvy, bom;
};
__device__ __forceinline__ CornerGrad corner_vjp(const SimConst& sc, float xo, float yo,
                                                 float co, float so, float vxo, float vyo,
                                                 float omo, float xb, float yb, float cb,
                                                 float sb, float vxb, float vyb, float omb,
                                                 float clx, float cly, float gOx, float gOy,
                                                 float gOT, float gBx, float gBy, float gBT) {
    CornerGrad g = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float rlx = dot2(co, clx, -so, cly), rly = dot2(so, clx, co, cly);
    const float kx = xo + rlx, ky = yo + rly;
    const float kvx = fmaf(-omo, rly, vxo), kvy = fmaf(omo, rlx, vyo);
    const float dx = kx - xb, dy = ky - yb;
    if (out_of_reach(dx, dy, sc.corner_reach2)) return g;   // no contact
    const float lx = dot2(cb, dx, sb, dy), ly = dot2(cb, dy, -sb, dx);
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    if (!(qx < 0.f && qy < 0.f)) return g;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool xa = qx >= qy;
    const float nlx = xa ? sx : 0.f, nly = xa ? 0.f : sy;
    const float delta = -(xa ? qx : qy);
    const float nx = dot2(cb, nlx, -sb, nly), ny = dot2(sb, nlx, cb, nly);
    const float wx = kvx - fmaf(-omb, dy, vxb), wy = kvy - fmaf(omb, dx, vyb);
    const float vn = dot2(wx, nx, wy, ny);
    const float fn = dot2(sc.k, delta, -sc.c, vn);
    if (!(fn > 0.f)) return g;
    const float tx = fmaf(-vn, nx, wx), ty = fmaf(-vn, ny, wy);
    const float iden = rsqrtf(dot2(tx, tx, ty, ty) + sc.eps_t2);
    const float gt = sc.mu_c * fn * iden;
    const float fx = dot2(fn, nx, -gt, tx), fy = dot2(fn, ny, -gt, ty);
    // owner: +f, torque rl x f; other: -f, torque -(d x f)
    const float afx = fmaf(gBT, dy, fmaf(-gOT, rly, gOx - gBx));
    const float afy = fmaf(-gBT, dx, fmaf(gOT, rlx, gOy - gBy));
    // f = fn n - gt t
    float afn = dot2(afx, nx, afy, ny);
    const float agt = -dot2(afx, tx, afy, ty);
    afn = fmaf(agt * sc.mu_c, iden, afn);
    const float aden = -agt * gt * iden;
    const float atx = dot2(aden * tx, iden, -afx, gt), aty = dot2(aden * ty, iden, -afy, gt);
    float avn = -dot2(atx, nx, aty, ny);
    float anx = dot2(afx, fn, -atx, vn), any = dot2(afy, fn, -aty, vn);
    const float adelta = sc.k * afn;
    avn = fmaf(-sc.c, afn, avn);
    const float awx = fmaf(avn, nx, atx), awy = fmaf(avn, ny, aty);
    anx = fmaf(avn, wx, anx);
    any = fmaf(avn, wy, any);
    // w = kv - vb - omb x d:  wx = kvx - vxb + omb dy, wy = kvy - vyb - omb dx
    const float akvx = awx, akvy = awy;
    g.bvx = -awx; g.bvy = -awy;
    g.bom = dot2(awx, dy, -awy, dx);
    // n = R_b nl (nl constant)
    float acb = dot2(anx, nlx, any, nly);
    float asb = dot2(any, nlx, -anx, nly);
    // delta = -(q on the axis), q = |l| - hs
    const float aqx = xa ? -adelta : 0.f, aqy = xa ? 0.f : -adelta;
    const float alx = aqx * sx, aly = aqy * sy;
    const float adx = dot2(-awy, omb, -gBT, fy) + dot2(cb, alx, -sb, aly);
    const float ady = dot2(awx, omb, gBT, fx) + dot2(sb, alx, cb, aly);
    acb += dot2(alx, dx, aly, dy);
    asb += dot2(alx, dy, -aly, dx);
    // d = k - b
    g.bx = -adx; g.by = -ady;
    // kv = vo + omo x rl
    g.ovx = akvx; g.ovy = akvy;
    g.oom = dot2(akvy, rlx, -akvx, rly);
    // k = o + rl
    g.ox = adx; g.oy = ady;
    const float arlx = dot2(akvy, omo, gOT, fy) + adx;
    const float arly = dot2(-akvx, omo, -gOT, fx) + ady;
    const float aco = dot2(arlx, clx, arly, cly), aso = dot2(arly, clx, -arlx, cly);
    g.oph = dot2(co, aso, -so, aco);
    g.bph = dot2(cb, asb, -sb, acb);
    return g;
}

// The reverse sweep's shared memory per team: C states (before each substep of
// the current segment) when C > 1; teams sit seg_stride<NB>(C) float2 apart to spread
// them over banks.
template <int NB>
__host__ __device__ constexpr int seg_stride(int C) { return C * (Dims<NB>::S / 2) + 1; }

}  // namespace rollout
}  // namespace stamp
