// sph_boids.cuh -- the boid rules of one boid, for the kernels that run them:
// the rules' own launch and the force pass (sph_physics.cu), whose boid warps
// run them straight after the fluid force on their boid.
#pragma once

#include "sph_internal.cuh"

namespace sphk {

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

__device__ __forceinline__ int warp_sum_i(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// The rules of the boid at sorted boid slot s, by one warp (all 32 lanes call
// it).  fluid_force(b): F_b of boid b, asked of lane 0 alone.
template <class F>
__device__ __forceinline__ void boid_rules_warp(const BoidArgs& a, const Scenes& sc, int s, int lane, F&& fluid_force)
{
    const float4* __restrict__ bpos_s = a.bpos_s;
    const float4* __restrict__ bvel_s = a.bvel_s;
    const StepConst& c = sc.c[scene_of(sc.bbase, sc.S, (unsigned)s)];
    const float4 pb = bpos_s[s];
    const float4 vb = bvel_s[s];
    const int b = id_of(pb);
    float cl[3] = {0.f, 0.f, 0.f};  // separation: sum of d (1 - |d|/r_sep), d = p_b - p_j
    float vs[3] = {0.f, 0.f, 0.f};  // alignment: sum of v_j
    float ps[3] = {0.f, 0.f, 0.f};  // cohesion: sum of (p_j - p_b)
    int nv = 0;
    // boid j at pj with velocity vj (vj is used only within r_vis)
    auto take = [&](const float4& pj, const float4& vj) {
        const float dx = __fsub_rn(pj.x, pb.x);
        const float dy_ = __fsub_rn(pj.y, pb.y);
        const float dz_ = __fsub_rn(pj.z, pb.z);
        const float r2 = pair_r2(dx, dy_, dz_);
        if (r2 < c.rs2) {
            float w = 1.0f - sqrtf(r2) / c.rs;
            w = fminf(fmaxf(w, 0.0f), 1.0f);
            cl[0] -= dx * w;
            cl[1] -= dy_ * w;
            cl[2] -= dz_ * w;
        }
        if (r2 < c.rv2) {
            vs[0] += vj.x;
            vs[1] += vj.y;
            vs[2] += vj.z;
            ps[0] += dx;
            ps[1] += dy_;
            ps[2] += dz_;
            ++nv;
        }
    };
    // the lanes fetch the walk's rows together (a row after another, their
    // start loads were most of a small school's time), then take each in turn
    WarpRows rows(c.gb, c.wb, a.bstart + c.cb_base, pb.x, pb.y, pb.z);
    for (int bt = 0; 32 * bt < rows.nrows; ++bt) {
        const int n = rows.batch(bt);
        for (int k = 0; k < n; ++k) {
            unsigned s0, s1;
            rows.row(k, s0, s1);
            // lane l takes slots s0 + l, s0 + l + 32, ... in that order, two
            // at a time so that both candidates' loads are in flight together
            unsigned j = s0 + lane;
            for (; j + 32 < s1; j += 64) {
                const float4 pa = bpos_s[j], va = bvel_s[j];
                const float4 pc = bpos_s[j + 32], vc = bvel_s[j + 32];
                if (j != (unsigned)s) take(pa, va);
                if (j + 32 != (unsigned)s) take(pc, vc);
            }
            if (j < s1 && j != (unsigned)s) take(bpos_s[j], bvel_s[j]);
        }
    }
    // obstacle avoidance: the obstacle-grid cells whose centre lies within
    // the visual range (the float32 predicate of the boid pairs), their mean
    // normals weighted obst_near within the protection range; the lanes take
    // the cells of the box of obst_reach cells around the boid's own
    float ob[3] = {0.f, 0.f, 0.f};
    int nob = 0;
    if (c.obst_on) {
        bool cl3 = false;
        int lo[3], n3[3];
        const float pp[3] = {pb.x, pb.y, pb.z};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int cc = cell_coord(pp[a], c.gb.minf[a], c.gb.inv_d, c.gb.dim[a], &cl3);
            lo[a] = max(cc - c.obst_reach, 0);
            n3[a] = min(cc + c.obst_reach, c.gb.dim[a] - 1) - lo[a] + 1;
        }
        const int total = n3[0] * n3[1] * n3[2];
        const float d = c.wb.d;
        for (int k = lane; k < total; k += 32) {
            const int ix = lo[0] + k % n3[0], iy = lo[1] + (k / n3[0]) % n3[1], iz = lo[2] + k / (n3[0] * n3[1]);
            const float4 g = __ldg(a.obst + c.cb_base + ix + c.gb.dim[0] * (iy + c.gb.dim[1] * iz));
            if (g.w == 0.0f) continue;
            const float cx = __fadd_rn(__fmul_rn((float)ix + 0.5f, d), c.gb.minf[0]);
            const float cy = __fadd_rn(__fmul_rn((float)iy + 0.5f, d), c.gb.minf[1]);
            const float cz = __fadd_rn(__fmul_rn((float)iz + 0.5f, d), c.gb.minf[2]);
            const float r2 = pair_r2(__fsub_rn(cx, pb.x), __fsub_rn(cy, pb.y), __fsub_rn(cz, pb.z));
            if (r2 < c.rv2) {
                const float w = r2 < c.rs2 ? c.obst_near : 1.0f;
                ob[0] = fmaf(w, g.x, ob[0]);
                ob[1] = fmaf(w, g.y, ob[1]);
                ob[2] = fmaf(w, g.z, ob[2]);
                ++nob;
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cl[a] = warp_sum(cl[a]);
        vs[a] = warp_sum(vs[a]);
        ps[a] = warp_sum(ps[a]);
        ob[a] = warp_sum(ob[a]);
    }
    nv = warp_sum_i(nv);
    nob = warp_sum_i(nob);
    if (lane != 0) return;

    float v[3] = {vb.x, vb.y, vb.z};
    const float p[3] = {pb.x, pb.y, pb.z};
    // 1. separation
#pragma unroll
    for (int a = 0; a < 3; ++a) v[a] = fmaf(c.w_sep, cl[a], v[a]);
    if (nv > 0) {
        const float inv_n = 1.0f / (float)nv;
        // 2. alignment towards the mean velocity of the visible boids
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fmaf(c.w_align, vs[a] * inv_n - v[a], v[a]);
        // 3. cohesion towards their mean position
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fmaf(c.w_coh, ps[a] * inv_n, v[a]);
    }
    // 4. fluid -> boid coupling: v += sph_factor dt F_b; literal coupling:
    // the attached particle is integrated like every particle (F_b plus
    // gravity) and v += sph_factor v_att (the paper's velocity update)
    const float4 f = fluid_force(b);
    float vatt[3] = {0.f, 0.f, 0.f};
    if (c.literal) {
        const float4 va = a.vel_s[a.slot_of_boid[b]];
        vatt[0] = fmaf(c.dt, f.x + c.grav[0], va.x);
        vatt[1] = fmaf(c.dt, f.y + c.grav[1], va.y);
        vatt[2] = fmaf(c.dt, f.z + c.grav[2], va.z);
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fmaf(c.sph_factor, vatt[a], v[a]);
    } else {
        v[0] = fmaf(c.sph_dt, f.x, v[0]);
        v[1] = fmaf(c.sph_dt, f.y, v[1]);
        v[2] = fmaf(c.sph_dt, f.z, v[2]);
    }
    // 4b. obstacle avoidance: v += w_obst * (weighted mean of the cells' normals)
    if (nob > 0) {
        const float g = c.w_obst / (float)nob;
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fmaf(g, ob[a], v[a]);
    }
    // 5. edge avoidance
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (p[a] < c.box_min[a]) v[a] += c.edge_turn;
        if (p[a] > c.box_max[a]) v[a] -= c.edge_turn;
    }
    // 6. speed limit
    const float sp = sqrtf(fmaf(v[2], v[2], fmaf(v[1], v[1], v[0] * v[0])));
    float scale = 1.0f;
    if (sp > c.v_max) scale = c.v_max / sp;
    else if (sp > 0.0f && sp < c.v_min) scale = c.v_min / sp;
#pragma unroll
    for (int a = 0; a < 3; ++a) v[a] *= scale;
    // 7. position update
    float x[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = fmaf(v[a], c.dt, p[a]);
    if (!(isfinite(x[0]) && isfinite(x[1]) && isfinite(x[2]))) atomicOr(a.err, SPH_DEV_NONFINITE);

    const float4 np = make_float4(x[0], x[1], x[2], pb.w);
    const float4 nvel = make_float4(v[0], v[1], v[2], 0.0f);
    a.bpos[b] = np;
    a.bvel[b] = nvel;
    // the attached particle follows the boid into the next step: its
    // position, and its velocity (force coupling) or its own (literal)
    const int slot = a.slot_of_boid[b];
    a.pos_next[slot] = np;
    a.vel_next[slot] = c.literal ? make_float4(vatt[0], vatt[1], vatt[2], 0.0f) : nvel;
    // a boid outside the tank bins its particle into the nearest cell of the
    // grid (no fluid is there); that is the method's state, not an anomaly
    bool cl2 = false;
    const unsigned k = (unsigned)c.c_base + cell_key(c.g, x[0], x[1], x[2], &cl2);
    a.key[slot] = k;
    a.rank[slot] = atomicAdd(&a.count[k], 1u);
}

}  // namespace sphk
