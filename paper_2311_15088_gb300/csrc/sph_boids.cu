// sph_boids.cu -- the boid half of the step: boid-grid keys and the boid
// rules with the fluid coupling, one warp per boid.
//
// Paper: section "Underwater Agent Behaviors" (Boid Space spatial hash, Boid
// Grid) and section "Boid Motion and Agent Fluid Interaction": separation
// inside protect_range, alignment and cohesion inside visible_range, edge
// avoidance, speed limit, position update, and the fluid -> boid coupling
// through sph_factor.  The boid also moves its attached particle, which
// pushes the fluid in the next step (the paper attaches particles[id] to
// boids[id]).
//
// Every boid reads the start-of-step snapshot (sorted copies), so the result
// does not depend on the order boids are processed in.  Lanes stride over
// the candidates of the boid cells within r_vis (WarpRows) and the warp
// sums with a fixed butterfly, so the float32 result is deterministic.
#include "sph_boids.cuh"

namespace sphk {

__global__ void __launch_bounds__(256)
k_boid_keys(const float4* __restrict__ bpos, Scenes sc, unsigned* __restrict__ bkey,
            unsigned* __restrict__ brank, unsigned* __restrict__ bcount)
{
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    bool clamped = false;
    if (b < sc.nb_all) {
        const StepConst& c = sc.c[scene_of(sc.bbase, sc.S, (unsigned)b)];
        float4 p = bpos[b];
        const unsigned k = (unsigned)c.cb_base + cell_key(c.gb, p.x, p.y, p.z, &clamped);
        bkey[b] = k;
        brank[b] = count_in_cell(bcount, k);
    }
}

cudaError_t launch_boid_keys(const float4* bpos, const Scenes& sc, unsigned* bkey, unsigned* brank,
                             unsigned* bcount, cudaStream_t s, long long* launches)
{
    if (sc.nb_all <= 0) return cudaSuccess;
    k_boid_keys<<<(sc.nb_all + 255) / 256, 256, 0, s>>>(bpos, sc, bkey, brank, bcount);
    ++*launches;
    return cudaGetLastError();
}

// The whole boid binning (keys, order by cell then id, cell starts, sorted
// copies) in one launch, for at most BIN_BOIDS boids and BIN_CELLS cells:
// every block puts all the boids' (key, id) values into shared memory, and
// a thread counts those below its own value, that of a boid (its sorted slot)
// or of a cell's first place (the cell's start).  Replaces seven short launches;
// 1,024 boids take 4 us (one block ranking them all took 37).
constexpr int BIN_BOIDS = 1024, BIN_CELLS = 8192, BIN_THREADS = 128;

__global__ void __launch_bounds__(BIN_THREADS)
k_boid_bin_small(const float4* __restrict__ bpos, const float4* __restrict__ bvel, Scenes sc, int nbcells,
                 float4* __restrict__ bpos_s, float4* __restrict__ bvel_s, unsigned* __restrict__ bstart)
{
    __shared__ __align__(16) unsigned s_val[BIN_BOIDS];
    static_assert(BIN_CELLS * BIN_BOIDS <= 0x7fffffff, "a value is key * BIN_BOIDS + id");
    const int nb = sc.nb_all, padded = (nb + 3) & ~3;
    for (int b = threadIdx.x; b < padded; b += BIN_THREADS) {
        unsigned v = 0xffffffffu;  // padding: above every value
        if (b < nb) {
            const StepConst& c = sc.c[scene_of(sc.bbase, sc.S, (unsigned)b)];
            const float4 p = bpos[b];
            bool clamped = false;
            v = ((unsigned)c.cb_base + cell_key(c.gb, p.x, p.y, p.z, &clamped)) * BIN_BOIDS + (unsigned)b;
        }
        s_val[b] = v;
    }
    __syncthreads();
    const int t = blockIdx.x * BIN_THREADS + threadIdx.x;  // a boid, then the cells' starts
    if (t > nb + nbcells) return;
    const unsigned mine = t < nb ? s_val[t] : (unsigned)(t - nb) * BIN_BOIDS;
    unsigned r = 0;
    for (int q = 0; q < padded; q += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(s_val + q);
        r += (o.x < mine) + (o.y < mine) + (o.z < mine) + (o.w < mine);
    }
    if (t < nb) {
        bpos_s[r] = bpos[t];
        bvel_s[r] = bvel[t];
    } else {
        bstart[t - nb] = r;
    }
}

bool boid_bin_is_small(const Scenes& sc, int nbcells) { return sc.nb_all <= BIN_BOIDS && nbcells < BIN_CELLS; }

cudaError_t launch_boid_bin_small(const float4* bpos, const float4* bvel, const Scenes& sc, int nbcells,
                                  float4* bpos_s, float4* bvel_s, unsigned* bstart, cudaStream_t s,
                                  long long* launches)
{
    k_boid_bin_small<<<(sc.nb_all + nbcells + BIN_THREADS) / BIN_THREADS, BIN_THREADS, 0, s>>>(
        bpos, bvel, sc, nbcells, bpos_s, bvel_s, bstart);
    ++*launches;
    return cudaGetLastError();
}

constexpr int BOID_WARPS = 8;

__global__ void __launch_bounds__(BOID_WARPS * 32)
k_boid_rules(BoidArgs a, Scenes sc)
{
    const int s = blockIdx.x * BOID_WARPS + (threadIdx.x >> 5);
    if (s < sc.nb_all)  // whole warps
        boid_rules_warp(a, sc, s, threadIdx.x & 31, [&](int b) { return a.fb[b]; });
}

cudaError_t launch_boid_rules(const BoidArgs& a, const Scenes& sc, cudaStream_t s, long long* launches)
{
    if (sc.nb_all <= 0) return cudaSuccess;
    k_boid_rules<<<(sc.nb_all + BOID_WARPS - 1) / BOID_WARPS, BOID_WARPS * 32, 0, s>>>(a, sc);
    ++*launches;
    return cudaGetLastError();
}

// ------------------------------------------------------------ obstacles

// The obstacle grid (section "Boid Motion and Agent Fluid Interaction": the
// normals of the obstacles' meshes are attributed to the cells of an
// obstacle grid; analytic spheres and boxes stand in for the meshes): a
// thread per boid-grid cell.  An obstacle counts in a cell when its signed
// distance at the cell's centre is within half a cell diagonal (float32, in
// this fixed order); it adds its outward unit normal at the surface point
// nearest the centre (a box from inside: the normal of its nearest face,
// the lowest axis on ties).  The cell keeps their mean and count.
__global__ void __launch_bounds__(256)
k_obstacle_grid(StepConst c, const float* __restrict__ shapes, int n_sphere, int n_box, float half_diag,
                float4* __restrict__ grid)
{
    const int cell = blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= c.gb.ncells) return;
    const int ix = cell % c.gb.dim[0], iy = (cell / c.gb.dim[0]) % c.gb.dim[1],
              iz = cell / (c.gb.dim[0] * c.gb.dim[1]);
    const float d = c.wb.d;
    const float x[3] = {__fadd_rn(__fmul_rn((float)ix + 0.5f, d), c.gb.minf[0]),
                        __fadd_rn(__fmul_rn((float)iy + 0.5f, d), c.gb.minf[1]),
                        __fadd_rn(__fmul_rn((float)iz + 0.5f, d), c.gb.minf[2])};
    float sum[3] = {0.f, 0.f, 0.f};
    int cnt = 0;
    for (int k = 0; k < n_sphere; ++k) {
        const float* S = shapes + 4 * k;
        const float dx = __fsub_rn(x[0], S[0]), dy = __fsub_rn(x[1], S[1]), dz = __fsub_rn(x[2], S[2]);
        const float q2 = pair_r2(dx, dy, dz);
        const float dist = __fsub_rn(sqrtf(q2), S[3]);
        if (!(fabsf(dist) <= half_diag) || !(q2 > 0.0f)) continue;
        const float inv = 1.0f / sqrtf(q2);
        sum[0] += dx * inv;
        sum[1] += dy * inv;
        sum[2] += dz * inv;
        ++cnt;
    }
    for (int k = 0; k < n_box; ++k) {
        const float* B = shapes + 4 * n_sphere + 6 * k;
        float q[3], m[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            q[a] = fmaxf(__fsub_rn(B[a], x[a]), __fsub_rn(x[a], B[3 + a]));
            m[a] = fmaxf(q[a], 0.0f);
        }
        const bool outside = q[0] > 0.0f || q[1] > 0.0f || q[2] > 0.0f;
        const float dist = outside ? sqrtf(pair_r2(m[0], m[1], m[2])) : fmaxf(q[0], fmaxf(q[1], q[2]));
        if (!(fabsf(dist) <= half_diag)) continue;
        float n[3] = {0.f, 0.f, 0.f};
        if (outside) {
#pragma unroll
            for (int a = 0; a < 3; ++a) n[a] = x[a] > B[3 + a] ? m[a] : (x[a] < B[a] ? -m[a] : 0.0f);
            const float inv = 1.0f / dist;
#pragma unroll
            for (int a = 0; a < 3; ++a) n[a] *= inv;
        } else {
            int ax = 0;
            if (q[1] > q[ax]) ax = 1;
            if (q[2] > q[ax]) ax = 2;
            n[ax] = __fsub_rn(x[ax], B[3 + ax]) >= __fsub_rn(B[ax], x[ax]) ? 1.0f : -1.0f;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) sum[a] += n[a];
        ++cnt;
    }
    const float inv = cnt ? 1.0f / (float)cnt : 0.0f;
    grid[cell] = make_float4(sum[0] * inv, sum[1] * inv, sum[2] * inv, (float)cnt);
}

cudaError_t launch_obstacle_grid(const StepConst& c, const float* shapes, int n_sphere, int n_box, float half_diag,
                                 float4* grid, cudaStream_t s, long long* launches)
{
    if (c.gb.ncells <= 0) return cudaSuccess;
    k_obstacle_grid<<<(c.gb.ncells + 255) / 256, 256, 0, s>>>(c, shapes, n_sphere, n_box, half_diag,
                                                             grid + c.cb_base);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace sphk
