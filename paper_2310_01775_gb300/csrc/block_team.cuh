// Rollout and reverse sweep with a group of QL lanes (1, 2 or 4) per block.
//
// A particle's team has QL lanes per block (the groups padded to 1, 2 or 4:
// with three blocks the last group idles).  Lane (b, r) holds the state of
// block b only, and K = 4/QL sides of it: the pushers placed on those sides
// and the corners of the same numbers.
//   - The contact of a pusher with its own block, in force through most of a
//     push, is K straight-line copies per lane on data the lane already
//     holds: no selection of block data by a runtime index, no loop over
//     items, no branch (the early outs became selects), so the K chains
//     overlap.
//   - Yaw sine/cosine, ground friction and integration run once per block
//     (on its QL lanes), not once per lane and block.
//   - A block's forces are summed over its lanes in log2(QL) butterfly steps.
//   - The other pairs (a pusher or corner of block b against block t != b)
//     are NB - 1 tests on the centre of block t, fetched by shuffle; one warp
//     vote skips everything else unless some pair is in reach.
// What bounds a rollout of a few thousand particles is the serial chain of a
// substep (one or two warps per scheduler), so the layout is chosen for few
// dependent instructions in it; with more particles it is the instruction
// count, where fewer lanes per block (less repeated friction, trigonometry
// and butterflies) win.
//
// Measured on GB300, three blocks, N = 2048, H = 6, T = 100, C = 25, softer
// contact (us, forward + reverse sweep): 512 + 815 with every state on every
// lane and all pairs dealt round-robin over 8 lanes; 155 + 279 here with QL = 2.
// Four blocks, N = 613, H = 5, both together: 1184 on scenes whose blocks stay apart,
// up to 1464 where they meet, against 278 and up to 726 (QL = 4).
//
// The results' bits do not depend on QL, nor on the number of particles that a
// width is picked by: every value that belongs to a side of a block (a contact's
// force, what it sends to another block, an adjoint) is rounded by itself and a
// block's four are added as (f0 + f1) + (f2 + f3), whatever lanes hold them; sums
// of two products say which one is fused (dot2).
#pragma once

#include "rollout.cuh"

namespace stamp {
namespace rollout {

// Padded block groups of a team, and its lanes.
__host__ __device__ constexpr int team_groups(int nb) { return nb <= 2 ? nb : 4; }
__host__ __device__ constexpr int team_lanes(int nb, int ql) { return team_groups(nb) * ql; }

struct One {   // one block's state (or its adjoint)
    float x, y, ph, vx, vy, om;
};
template <int K>
struct Own {   // this lane's pushers: start centres, displacements per substep, weights
    float p0x[K], p0y[K], dx[K], dy[K], w[K];
};

constexpr unsigned kAll = 0xffffffffu;

template <int NB, int QL>
struct Quad {
    static constexpr int K = 4 / QL, L = team_lanes(NB, QL);
    int base;        // warp lane of the team's lane 0
    int l;           // lane in the team
    int b, r;        // block; lane of the block (its sides are K r .. K r + K - 1)
    bool live;       // b < NB
    int to[NB];      // to[d]: warp lane of (b + d mod NB, r)
    int from[NB];    // from[d]: warp lane of (b - d mod NB, r)
    __device__ __forceinline__ int side(int j) const { return QL == 1 ? j : K * r + j; }
    __device__ __forceinline__ int choice(int j) const { return 4 * b + side(j); }
};
template <int NB, int QL>
__device__ __forceinline__ Quad<NB, QL> make_quad() {
    Quad<NB, QL> q;
    const int lane = threadIdx.x & 31;
    q.l = lane & (Quad<NB, QL>::L - 1);
    q.base = lane - q.l;
    q.b = q.l / QL;
    q.r = q.l % QL;
    q.live = q.b < NB;
#pragma unroll
    for (int d = 0; d < NB; ++d) {
        int t = q.b + d, f = q.b - d;
        t -= t >= NB ? NB : 0;
        f += f < 0 ? NB : 0;
        q.to[d] = q.live ? q.base + QL * t + q.r : lane;
        q.from[d] = q.live ? q.base + QL * f + q.r : lane;
    }
    return q;
}
// Corner s of a block, in its frame (units of the half side).
__device__ __forceinline__ void corner_of(int s, float& ex, float& ey) {
    ex = (s == 0 || s == 3) ? 1.f : -1.f;
    ey = s < 2 ? 1.f : -1.f;
}

// Sum of a lane's K values, then over the block's QL lanes: (v0 + v1) + (v2 + v3).
template <int QL>
__device__ __forceinline__ float block_sum(const float (&v)[4 / QL]) {
    float t;
    if constexpr (QL == 4) t = v[0];
    else if constexpr (QL == 2) t = __fadd_rn(v[0], v[1]);
    else t = __fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3]));
#pragma unroll
    for (int o = 1; o < QL; o <<= 1) t += __shfl_xor_sync(kAll, t, o);
    return t;
}
// Sum over the block's QL lanes.
template <int QL>
__device__ __forceinline__ float lanes_sum(float t) {
#pragma unroll
    for (int o = 1; o < QL; o <<= 1) t += __shfl_xor_sync(kAll, t, o);
    return t;
}
__device__ __forceinline__ float from_lane(float v, int lane) { return __shfl_sync(kAll, v, lane); }
// Choice c's value of a per-lane array of K (c compile-time after unrolling).
template <int NB, int QL>
__device__ __forceinline__ float choice_value(const Quad<NB, QL>& q, const float (&v)[4 / QL], int c) {
    constexpr int K = 4 / QL;
    return from_lane(v[c % K], q.base + c / K);
}

// Coordinate c of block b's row of a pose table, without dynamic indexing.
template <int NB>
__device__ __forceinline__ float pose_of(const float (&p)[kMaxBlocks][3], int b, int c) {
    float r = p[0][c];
#pragma unroll
    for (int i = 1; i < NB; ++i) r = (b == i) ? p[i][c] : r;
    return r;
}

// The lane's choice weights of action k (Eq. gamma_map: softmax((a+g)/tau),
// or one-hot argmax when hard), one logit per lane and side; maxima, sums and
// ties are taken in choice order.
template <int NB, int QL>
__device__ __forceinline__ void relax_lane(const SimConst& sc, const Quad<NB, QL>& q, const float* th,
                                           int k, int i, uint64_t gkey, bool noise, bool hard,
                                           float (&z)[4 / QL], float& uu, float& vv) {
    constexpr int M = Dims<NB>::M, P = Dims<NB>::P, K = 4 / QL;
    const float* a = th + k * P;
    float v[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        v[j] = 0.f;
        if (q.live) {
            v[j] = a[q.choice(j)];
            if (noise) {
                const float u = u23(sm64(gkey, (uint64_t)((i * sc.H + k) * M + q.choice(j))));
                v[j] += -logf(-logf(u));
            }
        }
    }
    uu = a[M];
    vv = a[M + 1];
    if (hard) {
        int best = 0;
        float bv = choice_value(q, v, 0);
#pragma unroll
        for (int c = 1; c < M; ++c) {
            const float x = choice_value(q, v, c);
            if (x > bv) { bv = x; best = c; }
        }
#pragma unroll
        for (int j = 0; j < K; ++j) z[j] = q.choice(j) == best ? 1.f : 0.f;
        return;
    }
    float t[K];
#pragma unroll
    for (int j = 0; j < K; ++j) t[j] = v[j] * sc.inv_tau;
    float mx = choice_value(q, t, 0);
#pragma unroll
    for (int c = 1; c < M; ++c) mx = fmaxf(mx, choice_value(q, t, c));
#pragma unroll
    for (int j = 0; j < K; ++j) t[j] = expf(v[j] * sc.inv_tau - mx);
    float sum = 0.f;
#pragma unroll
    for (int c = 0; c < M; ++c) sum += choice_value(q, t, c);
    const float inv = 1.f / sum;
#pragma unroll
    for (int j = 0; j < K; ++j) z[j] = q.live ? t[j] * inv : 0.f;
}

// The lane's pushers on the sides of its block, from the block's pose at the action start.
template <int NB, int QL>
__device__ __forceinline__ void place(const SimConst& sc, const Quad<NB, QL>& q, const One& p, float off,
                                      float dist, Own<4 / QL>& o) {
    const float step = dist / (float)sc.T;
    float cph, sph;
    yaw_sincos(p.ph, &sph, &cph);
#pragma unroll
    for (int j = 0; j < 4 / QL; ++j) {
        float nx, ny;
        side_normal(q.side(j), nx, ny);
        const float tx = -ny, ty = nx;
        const float lx = nx * (sc.hs + sc.r) + tx * off;
        const float ly = ny * (sc.hs + sc.r) + ty * off;
        o.p0x[j] = p.x + cph * lx - sph * ly;
        o.p0y[j] = p.y + sph * lx + cph * ly;
        o.dx[j] = -(cph * nx - sph * ny) * step;
        o.dy[j] = -(sph * nx + cph * ny) * step;
    }
}

// Force and torque on a square block (centre b, yaw via cph/sph, velocity v,
// omega) from a kinematic disk pusher at p (unweighted).  (ddx, ddy): the
// pusher's displacement per substep; the relative velocity takes displacement/dt
// in one fused multiply-add.  A pusher's own block: out of contact the results are
// selected to zero, so the chain has no branch.  kEarly (another block, already
// behind a branch): return there.
template <bool kEarly = false>
__device__ __forceinline__ void disk_box(const SimConst& sc, float px, float py, float ddx,
                                              float ddy, float bx, float by, float cph, float sph,
                                              float vx, float vy, float om, float& fx, float& fy,
                                              float& tq) {
    const float dx = px - bx, dy = py - by;
    const float lx = dot2(cph, dx, sph, dy), ly = dot2(cph, dy, -sph, dx);
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool outside = qx > 0.f || qy > 0.f;
    const float mx = fmaxf(qx, 0.f), my = fmaxf(qy, 0.f);
    const float m2 = dot2(mx, mx, my, my);
    const float il = rsqrtf(fmaxf(m2, 1e-30f));
    const bool xa = qx >= qy;
    const float sd = outside ? m2 * il : fmaxf(qx, qy);
    const float nlx = outside ? sx * mx * il : (xa ? sx : 0.f);
    const float nly = outside ? sy * my * il : (xa ? 0.f : sy);
    const float delta = sc.r - sd;
    if (kEarly) {
        fx = fy = tq = 0.f;
        if (!(delta > 0.f)) return;
    }
    const float nx = dot2(cph, nlx, -sph, nly), ny = dot2(sph, nlx, cph, nly);
    const float rx = px - sc.r * nx - bx, ry = py - sc.r * ny - by;
    const float wx = fmaf(ddx, sc.inv_dt, -(vx - om * ry)), wy = fmaf(ddy, sc.inv_dt, -(vy + om * rx));
    const float vn = dot2(wx, nx, wy, ny);
    const float fn = dot2(sc.k, delta, -sc.c, vn);
    const bool hit = delta > 0.f && fn > 0.f;
    if (kEarly && !hit) return;
    const float tx = wx - vn * nx, ty = wy - vn * ny;
    const float gt = sc.mu_c * fn * rsqrtf(dot2(tx, tx, ty, ty) + sc.eps_t2);
    const float gx = dot2(gt, tx, -fn, nx), gy = dot2(gt, ty, -fn, ny);
    fx = hit ? gx : 0.f;
    fy = hit ? gy : 0.f;
    tq = hit ? dot2(rx, gy, -ry, gx) : 0.f;
}

// Pairs (this lane's pusher or corner j, block b + d) in reach: bits
// 2 (K (d-1) + j) and the next.  (px, py): pusher centres; (kx, ky): corners.
template <int NB, int QL>
__device__ __forceinline__ unsigned near_pairs(const SimConst& sc, const Quad<NB, QL>& q, const One& s,
                                               const float (&px)[4 / QL], const float (&py)[4 / QL],
                                               const float (&kx)[4 / QL], const float (&ky)[4 / QL]) {
    constexpr int K = 4 / QL;
    unsigned near = 0u;
#pragma unroll
    for (int d = 1; d < NB; ++d) {
        const float tx = from_lane(s.x, q.to[d]), ty = from_lane(s.y, q.to[d]);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const unsigned bit = 1u << (2 * (K * (d - 1) + j));
            if (!out_of_reach(px[j] - tx, py[j] - ty, sc.disk_reach2)) near |= bit;
            if (!out_of_reach(kx[j] - tx, ky[j] - ty, sc.corner_reach2)) near |= 2u * bit;
        }
    }
    return q.live ? near : 0u;
}

// Pusher centres (and, with other blocks about, corners) during substep j1.
template <int NB, int QL>
__device__ __forceinline__ void points(const SimConst& sc, const Quad<NB, QL>& q, const One& s, float cs,
                                       float sn, const Own<4 / QL>& o, float j1, float (&px)[4 / QL],
                                       float (&py)[4 / QL], float (&rlx)[4 / QL], float (&rly)[4 / QL],
                                       float (&kx)[4 / QL], float (&ky)[4 / QL]) {
#pragma unroll
    for (int j = 0; j < 4 / QL; ++j) {
        px[j] = o.p0x[j] + j1 * o.dx[j];
        py[j] = o.p0y[j] + j1 * o.dy[j];
        if constexpr (NB > 1) {
            float ex, ey;
            corner_of(q.side(j), ex, ey);
            const float clx = ex * sc.hs, cly = ey * sc.hs;
            rlx[j] = dot2(cs, clx, -sn, cly);
            rly[j] = dot2(sn, clx, cs, cly);
            kx[j] = s.x + rlx[j];
            ky[j] = s.y + rly[j];
        }
    }
}

// Warp lanes of the other block at distance d (1 <= d < NB, runtime).
template <int NB, int QL>
__device__ __forceinline__ void partner(const Quad<NB, QL>& q, int d, int& to, int& from) {
    to = q.to[NB > 1 ? 1 : 0];
    from = q.from[NB > 1 ? 1 : 0];
#pragma unroll
    for (int e = 2; e < NB; ++e) {
        to = d == e ? q.to[e] : to;
        from = d == e ? q.from[e] : from;
    }
}

// One substep of every block of the team (forces, ground friction, semi-implicit Euler).
template <int NB, int QL>
__device__ __forceinline__ void block_substep(const SimConst& sc, const Quad<NB, QL>& q, One& s, float cs,
                                              float sn, const Own<4 / QL>& o, float j1) {
    constexpr int K = 4 / QL;
    float px[K], py[K], rlx[K], rly[K], kx[K], ky[K];
    points(sc, q, s, cs, sn, o, j1, px, py, rlx, rly, kx, ky);
    unsigned near = 0u;
    if constexpr (NB > 1) near = near_pairs(sc, q, s, px, py, kx, ky);
    float Fx[K], Fy[K], Tq[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        float fx, fy, tq;
        disk_box(sc, px[j], py[j], o.dx[j], o.dy[j], s.x, s.y, cs, sn, s.vx, s.vy, s.om, fx, fy, tq);
        Fx[j] = __fmul_rn(o.w[j], fx);
        Fy[j] = __fmul_rn(o.w[j], fy);
        Tq[j] = __fmul_rn(o.w[j], tq);
    }
    float Ix = 0.f, Iy = 0.f, It = 0.f;   // forces of the other blocks' pushers and corners
    if constexpr (NB > 1) {
        if (__any_sync(kAll, near)) {
#pragma unroll 1
            for (int d = 1; d < NB; ++d) {
                const unsigned nd = (near >> (2 * K * (d - 1))) & ((1u << (2 * K)) - 1u);
                if (!__any_sync(kAll, nd)) continue;
                int to, from;
                partner(q, d, to, from);
                const float bx = from_lane(s.x, to), by = from_lane(s.y, to);
                const float bc = from_lane(cs, to), bs = from_lane(sn, to);
                const float bvx = from_lane(s.vx, to), bvy = from_lane(s.vy, to);
                const float bom = from_lane(s.om, to);
                float Rx[K], Ry[K], Rt[K];   // each side's, on block b + d
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    float fx, fy, tq;
                    Rx[j] = Ry[j] = Rt[j] = 0.f;
                    if (nd & (1u << (2 * j))) {
                        disk_box<true>(sc, px[j], py[j], o.dx[j], o.dy[j], bx, by, bc, bs, bvx, bvy, bom, fx,
                                       fy, tq);
                        Rx[j] = __fmul_rn(o.w[j], fx);
                        Ry[j] = __fmul_rn(o.w[j], fy);
                        Rt[j] = __fmul_rn(o.w[j], tq);
                    }
                    if (nd & (2u << (2 * j))) {
                        const float kvx = fmaf(-s.om, rly[j], s.vx), kvy = fmaf(s.om, rlx[j], s.vy);
                        corner_box(sc, kx[j], ky[j], kvx, kvy, bx, by, bc, bs, bvx, bvy, bom, fx, fy);
                        Fx[j] += fx;
                        Fy[j] += fy;
                        Tq[j] += dot2(rlx[j], fy, -rly[j], fx);
                        Rx[j] -= fx;
                        Ry[j] -= fy;
                        Rt[j] -= dot2(kx[j] - bx, fy, -(ky[j] - by), fx);
                    }
                }
                Ix += from_lane(block_sum<QL>(Rx), from);
                Iy += from_lane(block_sum<QL>(Ry), from);
                It += from_lane(block_sum<QL>(Rt), from);
            }
        }
    }
    float fx = block_sum<QL>(Fx), fy = block_sum<QL>(Fy), tq = block_sum<QL>(Tq);
    if constexpr (NB > 1) {
        fx += Ix;
        fy += Iy;
        tq += It;
    }
    const float isv = rsqrtf(dot2(s.vx, s.vx, s.vy, s.vy) + sc.eps_v2);
    const float iso = rsqrtf(s.om * s.om + sc.eps_w2);
    const float gx = fx - sc.fric_lin * s.vx * isv;
    const float gy = fy - sc.fric_lin * s.vy * isv;
    const float gq = tq - sc.fric_ang * s.om * iso;
    s.vx += sc.dt * (gx * sc.inv_m);
    s.vy += sc.dt * (gy * sc.inv_m);
    s.om += sc.dt * (gq * sc.inv_I);
    s.x += sc.dt * s.vx;
    s.y += sc.dt * s.vy;
    s.ph += sc.dt * s.om;
}

// A team's state row (NB x 3 float2): the block's lanes store its three
// chunks (the last one repeatedly where lanes are left over: a branch would
// split the warp); every lane loads its block's chunks.  on: false for shadow
// teams and for lanes without a block.
template <int NB, int QL>
__device__ __forceinline__ void store_one(float2* row, const Quad<NB, QL>& q, const One& s, bool on) {
    float2* p = row + 3 * q.b;
    const float2 v0 = make_float2(s.x, s.y), v1 = make_float2(s.ph, s.vx), v2 = make_float2(s.vy, s.om);
    if constexpr (QL == 4) {
        const float2 v = q.r == 0 ? v0 : q.r == 1 ? v1 : v2;
        if (on) p[q.r < 2 ? q.r : 2] = v;
    } else if constexpr (QL == 2) {
        const float2 v = q.r == 0 ? v0 : v1;
        if (on) p[q.r] = v;
        if (on) p[2] = v2;
    } else if (on) {
        p[0] = v0;
        p[1] = v1;
        p[2] = v2;
    }
}
template <int NB, int QL, bool kL2 = false>
__device__ __forceinline__ One load_one(const float2* row, const Quad<NB, QL>& q) {
    const float2* p = row + 3 * (q.live ? q.b : 0);
    const float2 a = kL2 ? __ldcg(p) : p[0], b = kL2 ? __ldcg(p + 1) : p[1], c = kL2 ? __ldcg(p + 2) : p[2];
    return One{a.x, a.y, b.x, b.y, c.x, c.y};
}

// One team's forward rollout of particle i (on = false: a surplus team that
// shadows particle i and stores nothing).  kRows false: checkpoints (C > 1) and
// results only, in a loop without a store (one block, N = 1024, H = 4, C = 25: 92
// -> 78 us; the same choice inside one kernel cost the other side 2 to 6%).
template <int NB, int QL, bool kRows = true>
__device__ __forceinline__ void fwd_block_team(const SimConst& sc, const RolloutArgs& a, int i,
                                               bool on) {
    constexpr int S = Dims<NB>::S;
    const Quad<NB, QL> q = make_quad<NB, QL>();
    const bool put = on && q.live;
    const float* th = a.theta + (size_t)i * sc.D;
    const bool noise = a.iter >= 0;
    const uint64_t gkey = noise ? sm64(sm64(a.seed, kStreamGumbel), (uint64_t)a.iter) : 0ull;
    One s{pose_of<NB>(sc.init, q.b, 0), pose_of<NB>(sc.init, q.b, 1), pose_of<NB>(sc.init, q.b, 2),
          0.f, 0.f, 0.f};
    if (a.init_states && q.live) {   // per-particle start poses (transition sampling)
        const float* p0 = a.init_states + (size_t)i * 3 * NB + 3 * q.b;
        s.x = p0[0];
        s.y = p0[1];
        s.ph = p0[2];
    }
    float dsum = 0.f;
    const size_t ck2 = (size_t)a.N * (S / 2);   // float2 per checkpoint
    float2* row = reinterpret_cast<float2*>(a.tape + (size_t)i * S);
    // The state before every substep goes to the reverse sweep's rows: the tape
    // itself at interval 1, `full` beside the checkpoints otherwise.  Storing
    // them costs the forward 5 us of 160 (three blocks, N = 2048, H = 6, T =
    // 100); rebuilding them from the checkpoints in a launch of its own took 130.
    const bool every = sc.C == 1;
    float2* frow = every ? row : reinterpret_cast<float2*>(a.full) + (size_t)i * (S / 2);
    const bool rows = put && (every || a.full != nullptr);
    for (int k = 0; k < sc.H; ++k) {
        float uu, vv;
        Own<4 / QL> o;
        relax_lane(sc, q, th, k, i + a.particle0, gkey, noise, a.hard != 0, o.w, uu, vv);
        const float off = sc.off_max * tanhf(uu);
        const float dist = sc.dist_max * sigmoidf_(vv);
        dsum += dist * dist;
        place(sc, q, s, off, dist, o);
        if constexpr (!kRows) {
            for (int j = 1; j <= sc.T;) {
                store_one(row, q, s, put);
                row += ck2;
                for (const int end = j + sc.C; j < end; ++j) {
                    float cs, sn;
                    yaw_sincos(s.ph, &sn, &cs);
                    block_substep(sc, q, s, cs, sn, o, (float)j);
                }
            }
            continue;
        }
        int left = every ? -1 : 0;   // substeps to the next checkpoint
        for (int j = 1; j <= sc.T; ++j) {
            if (left == 0) {
                store_one(row, q, s, put);
                row += ck2;
                left = sc.C;
            }
            --left;
            float cs, sn;
            yaw_sincos(s.ph, &sn, &cs);
            store_one(frow, q, s, rows);
            frow += ck2;
            block_substep(sc, q, s, cs, sn, o, (float)j);
        }
    }
    if constexpr (kRows) store_one(frow, q, s, rows);
    if (!every) store_one(row, q, s, put);

    const float ex = s.x - pose_of<NB>(sc.goal, q.b, 0), ey = s.y - pose_of<NB>(sc.goal, q.b, 1);
    const float ew = wrapf(s.ph - pose_of<NB>(sc.goal, q.b, 2));
    const float term = fmaf(sc.w_yaw * ew, ew, dot2(ex, ex, ey, ey));
    float cost = sc.w_push * dsum;
#pragma unroll
    for (int b = 0; b < NB; ++b) cost += from_lane(term, q.base + QL * b);
    if (on && q.l == 0) {
        if (a.cost) a.cost[i] = cost;
        if (a.stats_min) atomicMin(a.stats_min, __float_as_uint(cost));
    }
    if (a.final_state) store_one(reinterpret_cast<float2*>(a.final_state + (size_t)i * S), q, s, put);
}

// ------------------------------ reverse sweep --------------------------------
// VJP of disk_box for the weighted force (w f, w torque).  gFx, gFy, gT: adjoints
// of the block's force and torque.  The block's position and velocity adjoints
// are the negatives of the pusher's.  Out of contact: the incoming adjoints are
// selected to zero, or (kEarly) all zero at once.
struct DiskAdj {
    float px, py, vpx, vpy, ph, om, w;
};
template <bool kEarly = false>
__device__ __forceinline__ DiskAdj disk_box_vjp(const SimConst& sc, float px, float py, float ddx,
                                                float ddy, float bx, float by, float cph, float sph,
                                                float vx, float vy, float om, float w, float gFx,
                                                float gFy, float gT) {
    const float dx = px - bx, dy = py - by;
    const float lx = dot2(cph, dx, sph, dy), ly = dot2(cph, dy, -sph, dx);
    const float qx = fabsf(lx) - sc.hs, qy = fabsf(ly) - sc.hs;
    const float sx = lx >= 0.f ? 1.f : -1.f, sy = ly >= 0.f ? 1.f : -1.f;
    const bool outside = qx > 0.f || qy > 0.f;
    const bool xa = qx >= qy;
    const float mx = fmaxf(qx, 0.f), my = fmaxf(qy, 0.f);
    const float m2 = dot2(mx, mx, my, my);
    const float il = rsqrtf(fmaxf(m2, 1e-30f));
    const float ln = m2 * il;
    const float sd = outside ? ln : fmaxf(qx, qy);
    const float nlx = outside ? sx * mx * il : (xa ? sx : 0.f);
    const float nly = outside ? sy * my * il : (xa ? 0.f : sy);
    const float delta = sc.r - sd;
    if (kEarly && !(delta > 0.f)) return DiskAdj{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float nx = dot2(cph, nlx, -sph, nly), ny = dot2(sph, nlx, cph, nly);
    const float rx = px - sc.r * nx - bx, ry = py - sc.r * ny - by;
    const float wx = fmaf(ddx, sc.inv_dt, -(vx - om * ry)), wy = fmaf(ddy, sc.inv_dt, -(vy + om * rx));
    const float vn = dot2(wx, nx, wy, ny);
    const float fn = dot2(sc.k, delta, -sc.c, vn);
    const bool hit = delta > 0.f && fn > 0.f;
    if (kEarly && !hit) return DiskAdj{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    gFx = hit ? gFx : 0.f;
    gFy = hit ? gFy : 0.f;
    gT = hit ? gT : 0.f;
    const float tx = wx - vn * nx, ty = wy - vn * ny;
    const float iden = rsqrtf(dot2(tx, tx, ty, ty) + sc.eps_t2);
    const float gt = sc.mu_c * fn * iden;
    const float fx = dot2(gt, tx, -fn, nx), fy = dot2(gt, ty, -fn, ny);
    DiskAdj g;
    // torque T = rx*(w fy) - ry*(w fx)
    const float aFx = gFx - gT * ry, aFy = gFy + gT * rx;
    g.w = dot2(aFx, fx, aFy, fy);
    const float afx = w * aFx, afy = w * aFy;
    // f = -fn n + gt t
    float afn = -dot2(afx, nx, afy, ny);
    const float agt = dot2(afx, tx, afy, ty);
    // gt = mu_c fn / den, den = sqrt(|t|^2 + eps^2)
    afn = fmaf(agt * sc.mu_c, iden, afn);
    const float aden = -agt * gt * iden;
    const float atx = dot2(afx, gt, aden * tx, iden), aty = dot2(afy, gt, aden * ty, iden);
    // t = w - vn n
    float avn = -dot2(atx, nx, aty, ny);
    float anx = dot2(-afx, fn, -atx, vn), any = dot2(-afy, fn, -aty, vn);
    // fn = k delta - c vn
    const float adelta = sc.k * afn;
    avn = fmaf(-sc.c, afn, avn);
    // vn = w . n
    const float awx = fmaf(avn, nx, atx), awy = fmaf(avn, ny, aty);
    anx = fmaf(avn, wx, anx);
    any = fmaf(avn, wy, any);
    // w = vp - v - om x r:  wx = vpx - vx + om ry, wy = vpy - vy - om rx
    g.vpx = awx;
    g.vpy = awy;
    g.om = dot2(awx, ry, -awy, rx);
    const float arx = dot2(gT, w * fy, -awy, om), ary = dot2(awx, om, -gT, w * fx);
    // r = p - r_p n - b
    anx = fmaf(-sc.r, arx, anx);
    any = fmaf(-sc.r, ary, any);
    // n = R nl
    const float anlx = dot2(cph, anx, sph, any);
    const float anly = dot2(cph, any, -sph, anx);
    float acph = dot2(anx, nlx, any, nly);
    float asph = dot2(any, nlx, -anx, nly);
    // delta = r - sd
    const float asd = -adelta;
    // outside: through the normalised clamped offset; inside: the chosen axis
    const float aln = fmaf(-dot2(anlx, nlx, anly, nly), il, asd);
    const float amx = dot2(sx, anlx, aln, mx) * il, amy = dot2(sy, anly, aln, my) * il;
    const float aqx = outside ? (qx > 0.f ? amx : 0.f) : (xa ? asd : 0.f);
    const float aqy = outside ? (qy > 0.f ? amy : 0.f) : (xa ? 0.f : asd);
    const float alx = aqx * sx, aly = aqy * sy;
    const float adx = dot2(cph, alx, -sph, aly), ady = dot2(sph, alx, cph, aly);
    acph += dot2(alx, dx, aly, dy);
    asph += dot2(alx, dy, -aly, dx);
    g.px = arx + adx;
    g.py = ary + ady;
    g.ph = dot2(cph, asph, -sph, acph);
    return g;
}

template <int K>
struct OwnAcc {   // adjoints of the lane's pushers
    float p0x[K], p0y[K], dx[K], dy[K], w[K];
};

template <int K>
struct Sides {   // adjoints of a block's state, by the side they come through
    float x[K], y[K], ph[K], vx[K], vy[K], om[K];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < K; ++j) x[j] = y[j] = ph[j] = vx[j] = vy[j] = om[j] = 0.f;
    }
};

// Reverse of block_substep: `a` is the adjoint of the block's state after
// the substep on entry, before it on exit.
template <int NB, int QL>
__device__ __forceinline__ void block_substep_vjp(const SimConst& sc, const Quad<NB, QL>& q, const One& s,
                                                  float cs, float sn, const Own<4 / QL>& o,
                                                  OwnAcc<4 / QL>& acc, float j1, One& a) {
    constexpr int K = 4 / QL;
    float px[K], py[K], rlx[K], rly[K], kx[K], ky[K];
    points(sc, q, s, cs, sn, o, j1, px, py, rlx, rly, kx, ky);
    unsigned near = 0u;
    if constexpr (NB > 1) near = near_pairs(sc, q, s, px, py, kx, ky);
    // v1 = v + dt F/m ; p1 = p + dt v1 (likewise for the yaw)
    const float av1x = a.vx + sc.dt * a.x;
    const float av1y = a.vy + sc.dt * a.y;
    const float aw1 = a.om + sc.dt * a.ph;
    const float aFx = av1x * (sc.dt * sc.inv_m);
    const float aFy = av1y * (sc.dt * sc.inv_m);
    const float aT = aw1 * (sc.dt * sc.inv_I);
    // ground friction F = -fl v/sv, T = -fa om/so
    const float isv = rsqrtf(dot2(s.vx, s.vx, s.vy, s.vy) + sc.eps_v2);
    const float iso = rsqrtf(s.om * s.om + sc.eps_w2);
    const float dotv = dot2(aFx, s.vx, aFy, s.vy) * (isv * isv * isv);
    a.vx = fmaf(-sc.fric_lin, dot2(aFx, isv, -s.vx, dotv), av1x);
    a.vy = fmaf(-sc.fric_lin, dot2(aFy, isv, -s.vy, dotv), av1y);
    a.om = aw1 - sc.fric_ang * aT * sc.eps_w2 * (iso * iso * iso);

    float dpx[K], dpy[K], dph[K], dvx[K], dvy[K], dom[K];   // own contacts (position, velocity negated)
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const DiskAdj g = disk_box_vjp(sc, px[j], py[j], o.dx[j], o.dy[j], s.x, s.y, cs, sn, s.vx,
                                            s.vy, s.om, o.w[j], aFx, aFy, aT);
        acc.p0x[j] += g.px;
        acc.p0y[j] += g.py;
        acc.dx[j] += dot2(j1, g.px, g.vpx, sc.inv_dt);
        acc.dy[j] += dot2(j1, g.py, g.vpy, sc.inv_dt);
        acc.w[j] += g.w;
        dpx[j] = g.px; dpy[j] = g.py; dph[j] = g.ph;
        dvx[j] = g.vpx; dvy[j] = g.vpy; dom[j] = g.om;
    }
    One in{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // from the pairs with other blocks
    if constexpr (NB > 1) {
        if (__any_sync(kAll, near)) {
            Sides<K> c;   // to this block, from its corners
            c.clear();
#pragma unroll 1
            for (int d = 1; d < NB; ++d) {
                const unsigned nd = (near >> (2 * K * (d - 1))) & ((1u << (2 * K)) - 1u);
                if (!__any_sync(kAll, nd)) continue;
                int to, from;
                partner(q, d, to, from);
                const float bx = from_lane(s.x, to), by = from_lane(s.y, to);
                const float bc = from_lane(cs, to), bs = from_lane(sn, to);
                const float bvx = from_lane(s.vx, to), bvy = from_lane(s.vy, to);
                const float bom = from_lane(s.om, to);
                const float bFx = from_lane(aFx, to), bFy = from_lane(aFy, to), bT = from_lane(aT, to);
                Sides<K> r;   // to block b + d
                r.clear();
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    if (nd & (1u << (2 * j))) {
                        const DiskAdj h = disk_box_vjp<true>(sc, px[j], py[j], o.dx[j], o.dy[j], bx, by, bc, bs,
                                                             bvx, bvy, bom, o.w[j], bFx, bFy, bT);
                        acc.p0x[j] += h.px;
                        acc.p0y[j] += h.py;
                        acc.dx[j] += dot2(j1, h.px, h.vpx, sc.inv_dt);
                        acc.dy[j] += dot2(j1, h.py, h.vpy, sc.inv_dt);
                        acc.w[j] += h.w;
                        r.x[j] = -h.px; r.y[j] = -h.py; r.ph[j] = h.ph;
                        r.vx[j] = -h.vpx; r.vy[j] = -h.vpy; r.om[j] = h.om;
                    }
                    if (nd & (2u << (2 * j))) {
                        float ex, ey;
                        corner_of(q.side(j), ex, ey);
                        const CornerGrad h = corner_vjp(sc, s.x, s.y, cs, sn, s.vx, s.vy, s.om, bx, by, bc,
                                                        bs, bvx, bvy, bom, ex * sc.hs, ey * sc.hs, aFx,
                                                        aFy, aT, bFx, bFy, bT);
                        c.x[j] += h.ox; c.y[j] += h.oy; c.ph[j] += h.oph;
                        c.vx[j] += h.ovx; c.vy[j] += h.ovy; c.om[j] += h.oom;
                        r.x[j] += h.bx; r.y[j] += h.by; r.ph[j] += h.bph;
                        r.vx[j] += h.bvx; r.vy[j] += h.bvy; r.om[j] += h.bom;
                    }
                }
                in.x += from_lane(block_sum<QL>(r.x), from);
                in.y += from_lane(block_sum<QL>(r.y), from);
                in.ph += from_lane(block_sum<QL>(r.ph), from);
                in.vx += from_lane(block_sum<QL>(r.vx), from);
                in.vy += from_lane(block_sum<QL>(r.vy), from);
                in.om += from_lane(block_sum<QL>(r.om), from);
            }
            in.x += block_sum<QL>(c.x);
            in.y += block_sum<QL>(c.y);
            in.ph += block_sum<QL>(c.ph);
            in.vx += block_sum<QL>(c.vx);
            in.vy += block_sum<QL>(c.vy);
            in.om += block_sum<QL>(c.om);
        }
    }
    a.x += in.x - block_sum<QL>(dpx);
    a.y += in.y - block_sum<QL>(dpy);
    a.ph += block_sum<QL>(dph) + in.ph;
    a.vx += in.vx - block_sum<QL>(dvx);
    a.vy += in.vy - block_sum<QL>(dvy);
    a.om += block_sum<QL>(dom) + in.om;
}

// One team's reverse sweep of particle i over its tape.  seg: the team's
// shared memory (the C states of a segment) when C > 1.  kL2: read the tape
// through L2 only (a forward of the same launch wrote it).
template <int NB, int QL, bool kL2 = false>
__device__ __forceinline__ void adj_block_team(const SimConst& sc, const RolloutArgs& a, int i, bool on,
                                               float2* seg) {
    constexpr int M = Dims<NB>::M, P = Dims<NB>::P, S = Dims<NB>::S, K = 4 / QL, L = Quad<NB, QL>::L;
    const Quad<NB, QL> q = make_quad<NB, QL>();
    const float* th = a.theta + (size_t)i * sc.D;
    float* gr = a.grad + (size_t)i * sc.D;
    const bool noise = a.iter >= 0;
    const bool hard = a.hard != 0;
    const uint64_t gkey = noise ? sm64(sm64(a.seed, kStreamGumbel), (uint64_t)a.iter) : 0ull;
    const size_t ck2 = (size_t)a.N * (S / 2);   // float2 per checkpoint
    const float2* tape_i = reinterpret_cast<const float2*>(a.tape + (size_t)i * S);
    One s = load_one<NB, QL, kL2>(tape_i + (size_t)sc.n_ckpt * ck2, q);
    // C = sum |p - g|^2 + w_yaw wrap(yaw - yaw_g)^2 (+ push term, below)
    One adj{2.f * (s.x - pose_of<NB>(sc.goal, q.b, 0)), 2.f * (s.y - pose_of<NB>(sc.goal, q.b, 1)),
            2.f * sc.w_yaw * wrapf(s.ph - pose_of<NB>(sc.goal, q.b, 2)), 0.f, 0.f, 0.f};
    const int segs = sc.T / sc.C;
    bool bad = false;
    for (int k = sc.H - 1; k >= 0; --k) {
        const One s0 = load_one<NB, QL, kL2>(tape_i + (size_t)(k * segs) * ck2, q);
        float uu, vv;
        Own<K> o;
        relax_lane(sc, q, th, k, i + a.particle0, gkey, noise, hard, o.w, uu, vv);
        const float tu = tanhf(uu);
        const float off = sc.off_max * tu;
        const float sg = sigmoidf_(vv);
        const float dist = sc.dist_max * sg;
        place(sc, q, s0, off, dist, o);
        OwnAcc<K> acc;
#pragma unroll
        for (int j = 0; j < K; ++j) acc.p0x[j] = acc.p0y[j] = acc.dx[j] = acc.dy[j] = acc.w[j] = 0.f;
        // three checkpoints in flight (an L2 or DRAM read outlasts a substep),
        // and the next one's sine and cosine beside this one's chain
        const float2* row = tape_i + (size_t)(k * segs + segs - 1) * ck2;
        One n1 = load_one<NB, QL, kL2>(row, q), n2 = n1, n3 = n1;
        if (segs > 1) n2 = load_one<NB, QL, kL2>(row - ck2, q);
        if (segs > 2) n3 = load_one<NB, QL, kL2>(row - 2 * ck2, q);
        float ncs, nsn;
        yaw_sincos(n1.ph, &nsn, &ncs);
        for (int sgi = segs - 1; sgi >= 0; --sgi) {
            s = n1;
            float cs = ncs, sn = nsn;
            n1 = n2;
            n2 = n3;
            if (sgi > 2) n3 = load_one<NB, QL, kL2>(row - 3 * ck2, q);
            row -= ck2;
            if (sc.C == 1) {   // every state is on the tape: nothing to recompute
                yaw_sincos(n1.ph, &nsn, &ncs);
                block_substep_vjp(sc, q, s, cs, sn, o, acc, (float)(sgi + 1), adj);
                continue;
            }
            // recompute the segment forward, keeping the state before each substep
            for (int jj = 0; jj < sc.C; ++jj) {
                store_one(seg + jj * (S / 2), q, s, q.live);
                if (jj + 1 < sc.C) {
                    yaw_sincos(s.ph, &sn, &cs);
                    block_substep(sc, q, s, cs, sn, o, (float)(sgi * sc.C + jj + 1));
                }
            }
            __syncwarp();
            for (int jj = sc.C - 1; jj >= 0; --jj) {
                s = load_one<NB, QL>(seg + jj * (S / 2), q);
                yaw_sincos(s.ph, &sn, &cs);
                block_substep_vjp(sc, q, s, cs, sn, o, acc, (float)(sgi * sc.C + jj + 1), adj);
            }
            __syncwarp();
        }

        // Action start: p0 = pos + R(yaw) (n (hs+r) + t off), delta = -R(yaw) n dist/T.
        const float step = dist / (float)sc.T;
        float cph, sph;
        yaw_sincos(s0.ph, &sph, &cph);
        float dph[K], doff[K], ddist[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
            float nx, ny;
            side_normal(q.side(j), nx, ny);
            const float tx = -ny, ty = nx;
            const float lx = nx * (sc.hs + sc.r) + tx * off;
            const float ly = ny * (sc.hs + sc.r) + ty * off;
            // d(R v)/dyaw = (-s vx - c vy, c vx - s vy)
            const float dRl_x = dot2(-sph, lx, -cph, ly), dRl_y = dot2(cph, lx, -sph, ly);
            const float dRn_x = -sph * nx - cph * ny, dRn_y = cph * nx - sph * ny;
            dph[j] = fmaf(-dot2(acc.dx[j], dRn_x, acc.dy[j], dRn_y), step,
                          dot2(acc.p0x[j], dRl_x, acc.p0y[j], dRl_y));
            // local offset adjoint R^T ap0, projected on t
            const float alx = dot2(cph, acc.p0x[j], sph, acc.p0y[j]);
            const float aly = dot2(cph, acc.p0y[j], -sph, acc.p0x[j]);
            const float ux = -(cph * nx - sph * ny), uy = -(sph * nx + cph * ny);
            doff[j] = q.live ? alx * tx + aly * ty : 0.f;
            ddist[j] = q.live ? dot2(acc.dx[j], ux, acc.dy[j], uy) / (float)sc.T : 0.f;
        }
        float aoff = block_sum<QL>(doff), adist = block_sum<QL>(ddist);
#pragma unroll
        for (int w = QL; w < L; w <<= 1) {
            aoff += __shfl_xor_sync(kAll, aoff, w);
            adist += __shfl_xor_sync(kAll, adist, w);
        }
        adj.x += block_sum<QL>(acc.p0x);
        adj.y += block_sum<QL>(acc.p0y);
        adj.ph += block_sum<QL>(dph);
        adist += 2.f * sc.w_push * dist;
        // softmax((a+g)/tau) backward; the one-hot of the hard map has no gradient
        float zaz = 0.f;
#pragma unroll
        for (int c = 0; c < M; ++c) zaz += choice_value(q, o.w, c) * choice_value(q, acc.w, c);
        if (on) {
            if (q.live) {
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const float gv = hard ? 0.f : -(o.w[j] * (acc.w[j] - zaz) * sc.inv_tau);
                    gr[k * P + q.choice(j)] = gv;
                    bad |= !isfinite(gv);
                }
            }
            if (q.l == 0) {
                const float go = -(aoff * sc.off_max * (1.f - tu * tu));
                const float gd = -(adist * sc.dist_max * sg * (1.f - sg));
                gr[k * P + M] = go;
                gr[k * P + M + 1] = gd;
                bad |= !isfinite(go) || !isfinite(gd);
            }
        }
    }
    // A reverse sweep that overflowed float32 (exploding gradient through the
    // contact dynamics) gives the particle a zero gradient, and is counted.
    const unsigned bads = (__ballot_sync(kAll, bad) >> q.base) & ((1u << L) - 1u);
    __syncwarp();   // the team's gradient stores come before these
    if (on && bads) {
        for (int d = q.l; d < sc.D; d += L) gr[d] = 0.f;
        if (q.l == 0 && a.dropped) atomicAdd(a.dropped, 1ull);
    }
}

}  // namespace rollout
}  // namespace stamp
