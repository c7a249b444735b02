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

__device__ __forceinline__ float sigmoidf_(float v) { return 1.f / (1.f + expf(-v)); }

// ------------------------------- forces -------------------------------------
// A pusher centre (corner) at offset (dx, dy) from a block centre farther
// than the block's reach cannot touch it: the contact tests below return no
// contact there, so callers may skip them.
__device__ __forceinline__ bool out_of_reach(float dx, float dy, float reach2) {
    return dx * dx + dy * dy > reach2;
}

// Force and torque on a square block (centre b, yaw via cph/sph, velocity v,
// omega) from a kinematic disk pusher at p moving with vp (unweighted).
__device__ __forceinline__ void disk_box(const SimConst& sc, float px, float py, float vpx,
                                         float vpy, float bx, float by, float cph, float sph,
                                         float vx, float vy, float om, float& fx, float& fy,
                                         float& tq) {
    fx = fy = tq = 0.f;
    const float dx = px - bx, dy = py - by;
    const float lx = cph * dx + sph * dy, ly = -sph * dx + cph * dy;
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    // outside: normalised clamped offset; inside: the axis of the larger q
    // (selects, not branches: both are cheap and the chain stays straight)
    const bool outside = qx > 0.f || qy > 0.f;
    const float mx = fmaxf(qx, 0.f), my = fmaxf(qy, 0.f);
    const float il = rsqrtf(fmaxf(mx * mx + my * my, 1e-30f));
    const bool xa = qx >= qy;
    const float sd = outside ? (mx * mx + my * my) * il : fmaxf(qx, qy);
    const float nlx = outside ? sx * mx * il : (xa ? sx : 0.f);
    const float nly = outside ? sy * my * il : (xa ? 0.f : sy);
    const float delta = sc.r - sd;
    if (!(delta > 0.f)) return;
    const float nx = cph * nlx - sph * nly, ny = sph * nlx + cph * nly;
    const float rx = px - sc.r * nx - bx, ry = py - sc.r * ny - by;
    const float wx = vpx - (vx - om * ry), wy = vpy - (vy + om * rx);
    const float vn = wx * nx + wy * ny;
    const float fn = sc.k * delta - sc.c * vn;
    if (!(fn > 0.f)) return;
    const float tx = wx - vn * nx, ty = wy - vn * ny;
    const float gt = sc.mu_c * fn * rsqrtf(tx * tx + ty * ty + sc.eps_t2);
    fx = -fn * nx + gt * tx;
    fy = -fn * ny + gt * ty;
    tq = rx * fy - ry * fx;
}

// Corner k (position, velocity) of one box against square B: force on the
// corner's owner (B receives the opposite at the same point).
__device__ __forceinline__ void corner_box(const SimConst& sc, float kx, float ky, float kvx,
                                           float kvy, float bx, float by, float cph, float sph,
                                           float vx, float vy, float om, float& fx, float& fy) {
    fx = fy = 0.f;
    const float dx = kx - bx, dy = ky - by;
    if (dx * dx + dy * dy > sc.corner_reach2) return;   // out of reach: no contact
    const float lx = cph * dx + sph * dy, ly = -sph * dx + cph * dy;
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    if (!(qx < 0.f && qy < 0.f)) return;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool xa = qx >= qy;
    const float nlx = xa ? sx : 0.f, nly = xa ? 0.f : sy;
    const float delta = -(xa ? qx : qy);
    const float nx = cph * nlx - sph * nly, ny = sph * nlx + cph * nly;
    const float wx = kvx - (vx - om * dy), wy = kvy - (vy + om * dx);
    const float vn = wx * nx + wy * ny;
    const float fn = sc.k * delta - sc.c * vn;
    if (!(fn > 0.f)) return;
    const float tx = wx - vn * nx, ty = wy - vn * ny;
    const float gt = sc.mu_c * fn * rsqrtf(tx * tx + ty * ty + sc.eps_t2);
    fx = fn * nx - gt * tx;
    fy = fn * ny - gt * ty;
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
// VJP of disk_box for the weighted force (w*f, w*torque).  Inputs gFx, gFy,
// gT: adjoints of the block's force and torque.  Outputs are overwritten.
struct DiskGrad {
    float px, py, vpx, vpy, bx, by, ph, vx, vy, om, w;
};
__device__ __forceinline__ DiskGrad disk_box_vjp(const SimConst& sc, float px, float py,
                                                 float vpx, float vpy, float bx, float by,
                                                 float cph, float sph, float vx, float vy,
                                                 float om, float w, float gFx, float gFy,
                                                 float gT) {
    DiskGrad g = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float dx = px - bx, dy = py - by;
    const float lx = cph * dx + sph * dy, ly = -sph * dx + cph * dy;
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool outside = qx > 0.f || qy > 0.f;
    const bool xa = qx >= qy;
    const float mx = fmaxf(qx, 0.f), my = fmaxf(qy, 0.f);
    const float il = rsqrtf(fmaxf(mx * mx + my * my, 1e-30f));
    const float ln = (mx * mx + my * my) * il;
    const float sd = outside ? ln : fmaxf(qx, qy);
    const float nlx = outside ? sx * mx * il : (xa ? sx : 0.f);
    const float nly = outside ? sy * my * il : (xa ? 0.f : sy);
    const float delta = sc.r - sd;
    if (!(delta > 0.f)) return g;
    const float nx = cph * nlx - sph * nly, ny = sph * nlx + cph * nly;
    const float rx = px - sc.r * nx - bx, ry = py - sc.r * ny - by;
    const float wx = vpx - (vx - om * ry), wy = vpy - (vy + om * rx);
    const float vn = wx * nx + wy * ny;
    const float fn = sc.k * delta - sc.c * vn;
    if (!(fn > 0.f)) return g;
    const float tx = wx - vn * nx, ty = wy - vn * ny;
    const float iden = rsqrtf(tx * tx + ty * ty + sc.eps_t2);
    const float gt = sc.mu_c * fn * iden;
    const float fx = -fn * nx + gt * tx, fy = -fn * ny + gt * ty;
    // torque T = rx*(w fy) - ry*(w fx)
    const float aFx = gFx - gT * ry, aFy = gFy + gT * rx;
    float arx = gT * (w * fy), ary = -gT * (w * fx);
    g.w = aFx * fx + aFy * fy;
    const float afx = w * aFx, afy = w * aFy;
    // f = -fn n + gt t
    float afn = -(afx * nx + afy * ny);
    float anx = -afx * fn, any = -afy * fn;
    const float agt = afx * tx + afy * ty;
    float atx = afx * gt, aty = afy * gt;
    // gt = mu_c fn / den, den = sqrt(|t|^2 + eps^2)
    afn += agt * sc.mu_c * iden;
    const float aden = -agt * gt * iden;
    atx += aden * tx * iden;
    aty += aden * ty * iden;
    // t = w - vn n
    float awx = atx, awy = aty;
    float avn = -(atx * nx + aty * ny);
    anx -= atx * vn;
    any -= aty * vn;
    // fn = k delta - c vn
    const float adelta = sc.k * afn;
    avn -= sc.c * afn;
    // vn = w . n
    awx += avn * nx;
    awy += avn * ny;
    anx += avn * wx;
    any += avn * wy;
    // w = vp - v - om x r:  wx = vpx - vx + om ry, wy = vpy - vy - om rx
    g.vpx = awx; g.vpy = awy;
    g.vx = -awx; g.vy = -awy;
    g.om = awx * ry - awy * rx;
    ary += awx * om;
    arx -= awy * om;
    // r = p - r_p n - b
    g.px = arx; g.py = ary;
    anx -= sc.r * arx;
    any -= sc.r * ary;
    g.bx = -arx; g.by = -ary;
    // n = R nl
    const float anlx = cph * anx + sph * any;
    const float anly = -sph * anx + cph * any;
    float acph = anx * nlx + any * nly;
    float asph = -anx * nly + any * nlx;
    // delta = r - sd
    const float asd = -adelta;
    // outside: through the normalised clamped offset; inside: the chosen axis
    const float aln = asd - (anlx * nlx + anly * nly) * il;
    const float amx = (sx * anlx + aln * mx) * il, amy = (sy * anly + aln * my) * il;
    const float aqx = outside ? (qx > 0.f ? amx : 0.f) : (xa ? asd : 0.f);
    const float aqy = outside ? (qy > 0.f ? amy : 0.f) : (xa ? 0.f : asd);
    const float alx = aqx * sx, aly = aqy * sy;
    const float adx = cph * alx - sph * aly, ady = sph * alx + cph * aly;
    acph += alx * dx + aly * dy;
    asph += alx * dy - aly * dx;
    g.px += adx; g.py += ady;
    g.bx -= adx; g.by -= ady;
    g.ph = -sph * acph + cph * asph;
    return g;
}

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
    const float rlx = co * clx - so * cly, rly = so * clx + co * cly;
    const float kx = xo + rlx, ky = yo + rly;
    const float kvx = vxo - omo * rly, kvy = vyo + omo * rlx;
    const float dx = kx - xb, dy = ky - yb;
    if (dx * dx + dy * dy > sc.corner_reach2) return g;   // out of reach: no contact
    const float lx = cb * dx + sb * dy, ly = -sb * dx + cb * dy;
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    if (!(qx < 0.f && qy < 0.f)) return g;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool xa = qx >= qy;
    const float nlx = xa ? sx : 0.f, nly = xa ? 0.f : sy;
    const float delta = -(xa ? qx : qy);
    const float nx = cb * nlx - sb * nly, ny = sb * nlx + cb * nly;
    const float wx = kvx - (vxb - omb * dy), wy = kvy - (vyb + omb * dx);
    const float vn = wx * nx + wy * ny;
    const float fn = sc.k * delta - sc.c * vn;
    if (!(fn > 0.f)) return g;
    const float tx = wx - vn * nx, ty = wy - vn * ny;
    const float iden = rsqrtf(tx * tx + ty * ty + sc.eps_t2);
    const float gt = sc.mu_c * fn * iden;
    const float fx = fn * nx - gt * tx, fy = fn * ny - gt * ty;
    // owner: +f, torque rl x f; other: -f, torque -(d x f)
    const float afx = gOx - gBx - gOT * rly + gBT * dy;
    const float afy = gOy - gBy + gOT * rlx - gBT * dx;
    float arlx = gOT * fy, arly = -gOT * fx;
    float adx = -gBT * fy, ady = gBT * fx;
    // f = fn n - gt t
    float afn = afx * nx + afy * ny;
    float anx = afx * fn, any = afy * fn;
    const float agt = -(afx * tx + afy * ty);
    float atx = -afx * gt, aty = -afy * gt;
    afn += agt * sc.mu_c * iden;
    const float aden = -agt * gt * iden;
    atx += aden * tx * iden;
    aty += aden * ty * iden;
    float awx = atx, awy = aty;
    float avn = -(atx * nx + aty * ny);
    anx -= atx * vn;
    any -= aty * vn;
    const float adelta = sc.k * afn;
    avn -= sc.c * afn;
    awx += avn * nx;
    awy += avn * ny;
    anx += avn * wx;
    any += avn * wy;
    // w = kv - vb - omb x d:  wx = kvx - vxb + omb dy, wy = kvy - vyb - omb dx
    const float akvx = awx, akvy = awy;
    g.bvx = -awx; g.bvy = -awy;
    g.bom = awx * dy - awy * dx;
    ady += awx * omb;
    adx -= awy * omb;
    // n = R_b nl (nl constant)
    float acb = anx * nlx + any * nly;
    float asb = -anx * nly + any * nlx;
    // delta = -(q on the axis), q = |l| - hs
    const float aqx = xa ? -adelta : 0.f, aqy = xa ? 0.f : -adelta;
    const float alx = aqx * sx, aly = aqy * sy;
    adx += cb * alx - sb * aly;
    ady += sb * alx + cb * aly;
    acb += alx * dx + aly * dy;
    asb += alx * dy - aly * dx;
    // d = k - b
    float akx = adx, aky = ady;
    g.bx = -adx; g.by = -ady;
    // kv = vo + omo x rl
    g.ovx = akvx; g.ovy = akvy;
    g.oom = -akvx * rly + akvy * rlx;
    arly -= akvx * omo;
    arlx += akvy * omo;
    // k = o + rl
    g.ox = akx; g.oy = aky;
    arlx += akx;
    arly += aky;
    const float aco = arlx * clx + arly * cly, aso = -arlx * cly + arly * clx;
    g.oph = -so * aco + co * aso;
    g.bph = -sb * acb + cb * asb;
    return g;
}

// The reverse sweep's shared memory per team: C states (before each substep of
// the current segment) when C > 1; teams sit seg_stride<NB>(C) float2 apart to spread
// them over banks.
template <int NB>
__host__ __device__ constexpr int seg_stride(int C) { return C * (Dims<NB>::S / 2) + 1; }

}  // namespace rollout
}  // namespace stamp
