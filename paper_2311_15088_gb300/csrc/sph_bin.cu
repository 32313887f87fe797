// sph_bin.cu -- uniform-grid binning of the step: cell keys with the
// cells' histogram, exclusive scan of the cell counts, scatter and a per-cell
// sort by particle id fused with the gather of the SoA state.
//
// Paper: section "Neighborhood Search" (get_cell, hash) and section
// "Neighbor Search with Sorting" (set_particle_count, prefix sum,
// count_sort_particle_index).  The paper's atomic rank makes the order
// inside a cell nondeterministic; here every cell is re-sorted by particle
// id so that the sorted order, and with it every float32 summation order,
// is a pure function of the state.
#include "sph_internal.cuh"

namespace sphk {

// ------------------------------------------------------------------ keys

struct Box {
    float box_min[3], box_max[3];
};

__global__ void __launch_bounds__(256)
k_keys(const float4* __restrict__ pos, int n, GridDesc g, Box box, unsigned* __restrict__ key,
       unsigned* __restrict__ rank, unsigned* __restrict__ count, unsigned* __restrict__ err)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool active = i < n;
    unsigned k = 0;
    bool clamped = false;
    if (active) {
        float4 p = pos[i];
        bool cl = false;
        k = cell_key(g, p.x, p.y, p.z, &cl);
        key[i] = k;
        clamped = outside_box(box, p.x, p.y, p.z);
    }
    if (active) rank[i] = count_in_cell(count, k);
    if (__any_sync(FULL, clamped) && (threadIdx.x & 31) == 0) atomicOr(err, SPH_DEV_CLAMPED);
}

cudaError_t launch_keys(const float4* pos, int n, const GridDesc& g, const float box_min[3], const float box_max[3],
                        unsigned* key, unsigned* rank, unsigned* count, unsigned* err, cudaStream_t s,
                        long long* launches)
{
    if (n <= 0) return cudaSuccess;
    Box box;
    for (int a = 0; a < 3; ++a) {
        box.box_min[a] = box_min[a];
        box.box_max[a] = box_max[a];
    }
    k_keys<<<(n + 255) / 256, 256, 0, s>>>(pos, n, g, box, key, rank, count, err);
    ++*launches;
    return cudaGetLastError();
}

// Keys of every scene's particles: the thread of storage slot i finds its
// scene and emits the global key c_base + hash(get_cell(p)).
__global__ void __launch_bounds__(256)
k_scene_keys(const float4* __restrict__ pos, Scenes sc, unsigned* __restrict__ key,
             unsigned* __restrict__ rank, unsigned* __restrict__ count, unsigned* __restrict__ err)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool active = i < sc.n_all;
    unsigned k = 0;
    bool clamped = false;
    if (active) {
        const StepConst& c = sc.c[scene_of(sc.pbase, sc.S, (unsigned)i)];
        float4 p = pos[i];
        bool cl = false;
        k = (unsigned)c.c_base + cell_key(c.g, p.x, p.y, p.z, &cl);
        key[i] = k;
        // boid-attached particles follow their boids, which may leave the tank
        clamped = id_of(p) >= sc.nb_all && outside_box(c, p.x, p.y, p.z);
    }
    if (active) rank[i] = count_in_cell(count, k);
    if (__any_sync(FULL, clamped) && (threadIdx.x & 31) == 0) atomicOr(err, SPH_DEV_CLAMPED);
}

cudaError_t launch_scene_keys(const float4* pos, const Scenes& sc, unsigned* key, unsigned* rank,
                              unsigned* count, unsigned* err, cudaStream_t s, long long* launches)
{
    if (sc.n_all <= 0) return cudaSuccess;
    k_scene_keys<<<(sc.n_all + 255) / 256, 256, 0, s>>>(pos, sc, key, rank, count, err);
    ++*launches;
    return cudaGetLastError();
}

// ------------------------------------------------------------------ scan

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 16;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

int scan_parts(int n) { return (n + SCAN_TILE - 1) / SCAN_TILE; }

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned* prefix_out, unsigned* sh_warp)
{
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned w = lane < (SCAN_THREADS / 32) ? sh_warp[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        if (lane < (SCAN_THREADS / 32)) sh_warp[lane] = w;  // inclusive warp totals
    }
    __syncthreads();
    unsigned total = sh_warp[SCAN_THREADS / 32 - 1];
    unsigned warp_base = warp ? sh_warp[warp - 1] : 0u;
    *prefix_out = warp_base + x - v;
    __syncthreads();
    return total;
}

__global__ void __launch_bounds__(SCAN_THREADS)
k_scan_reduce(const unsigned* __restrict__ in, int n, unsigned* __restrict__ part)
{
    __shared__ unsigned sh_warp[SCAN_THREADS / 32];
    int base = blockIdx.x * SCAN_TILE;
    unsigned sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        int idx = base + k * SCAN_THREADS + threadIdx.x;
        if (idx < n) sum += in[idx];
    }
    unsigned dummy;
    unsigned total = block_exclusive_scan(sum, &dummy, sh_warp);
    if (threadIdx.x == 0) part[blockIdx.x] = total;
}

// One block: exclusive scan of the tile totals in place (grids of so many
// tiles that adding up those before it would hold every block).  1024 values
// per round: a shuffle scan in each warp, then of the 32 warp totals by the
// first warp.
__global__ void __launch_bounds__(1024) k_scan_parts(unsigned* __restrict__ part, int nparts)
{
    __shared__ unsigned sh_w[32];
    __shared__ unsigned carry_sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned carry = 0;
    for (int base = 0; base < nparts; base += 1024) {
        const int idx = base + threadIdx.x;
        const unsigned v = idx < nparts ? part[idx] : 0u;
        unsigned x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sh_w[warp] = x;
        __syncthreads();
        if (warp == 0) {
            unsigned w = sh_w[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(FULL, w, o);
                if (lane >= o) w += y;
            }
            sh_w[lane] = w;  // inclusive warp totals
            if (lane == 31) carry_sh = w;
        }
        __syncthreads();
        const unsigned incl = x + (warp ? sh_w[warp - 1] : 0u);
        if (idx < nparts) part[idx] = carry + incl - v;
        carry += carry_sh;
        __syncthreads();
    }
}

// Element e of a tile lives at sh[e + e / 32]: one padding word per 32
// keeps both the coalesced phase (thread t, elements k * 256 + t) and the
// per-thread phase (thread t, elements 16 t .. 16 t + 15) free of bank
// conflicts (without it the second phase is a 16-way conflict).
__device__ __forceinline__ int scan_pad(int e) { return e + (e >> 5); }

// out[i] = the counts before i, out[n] = their total.  SUM: part holds the
// tiles' totals and each block adds up those before its own (otherwise part
// is already scanned).  zero: the counts are reset for the next histogram
// (each is read by its own block alone).
template <bool SUM>
__global__ void __launch_bounds__(SCAN_THREADS)
k_scan_tiles(unsigned* __restrict__ in, int n, const unsigned* __restrict__ part, unsigned* __restrict__ out, int zero)
{
    __shared__ unsigned sh[SCAN_TILE + SCAN_TILE / 32];
    __shared__ unsigned sh_warp[SCAN_THREADS / 32];
    int base = blockIdx.x * SCAN_TILE;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        int idx = base + k * SCAN_THREADS + threadIdx.x;
        sh[scan_pad(k * SCAN_THREADS + threadIdx.x)] = idx < n ? in[idx] : 0u;
    }
    unsigned before = 0;
    if (SUM) {
        for (int k = threadIdx.x; k < (int)blockIdx.x; k += SCAN_THREADS) before += __ldg(part + k);
        unsigned dummy;
        before = block_exclusive_scan(before, &dummy, sh_warp);
    } else {
        before = __ldg(part + blockIdx.x);
    }
    __syncthreads();
    if (zero) {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            int idx = base + k * SCAN_THREADS + threadIdx.x;
            if (idx < n) in[idx] = 0u;
        }
    }
    unsigned local[SCAN_ITEMS];
    unsigned sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        local[k] = sh[scan_pad(threadIdx.x * SCAN_ITEMS + k)];
        sum += local[k];
    }
    unsigned prefix;
    const unsigned total = block_exclusive_scan(sum, &prefix, sh_warp);
    prefix += before;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        sh[scan_pad(threadIdx.x * SCAN_ITEMS + k)] = prefix;
        prefix += local[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        int idx = base + k * SCAN_THREADS + threadIdx.x;
        if (idx < n) out[idx] = sh[scan_pad(k * SCAN_THREADS + threadIdx.x)];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = before + total;
}

// Two launches up to this many tiles (33.5M cells; the large tank's grid has
// 1,430): a block adds up to 32 totals per thread.  As three launches and a
// fourth for the grand total the scan was a quarter of a small step's chain.
// A step of 2,000 particles in grids of 1,500, 6,000 and 8,191 tiles takes 32,
// 89 and 114 us (80, 134 and 165 with the four), of 9,000, with three, 122 (169).
constexpr int SCAN_SUM_MAX = 8192;

cudaError_t launch_scan(unsigned* counts, int n, unsigned* part, unsigned* start, bool zero, cudaStream_t s,
                        long long* launches)
{
    if (n <= 0) return cudaSuccess;
    int np = scan_parts(n);
    k_scan_reduce<<<np, SCAN_THREADS, 0, s>>>(counts, n, part);
    if (np <= SCAN_SUM_MAX) {
        k_scan_tiles<true><<<np, SCAN_THREADS, 0, s>>>(counts, n, part, start, zero);
        *launches += 2;
    } else {
        k_scan_parts<<<1, 1024, 0, s>>>(part, np);
        k_scan_tiles<false><<<np, SCAN_THREADS, 0, s>>>(counts, n, part, start, zero);
        *launches += 3;
    }
    return cudaGetLastError();
}

// --------------------------------------------------------------- scatter

__global__ void __launch_bounds__(256)
k_scatter(const unsigned* __restrict__ key, const unsigned* __restrict__ rank,
          const unsigned* __restrict__ start, int n, int* __restrict__ tmp)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) tmp[start[key[i]] + rank[i]] = i;
}

// The same, also placing each particle's id (pos.w) beside its index:
// tmp_id[start[key] + rank] = id, so that the per-cell sort ranks a cell's
// particles from one contiguous run of ids.
__global__ void __launch_bounds__(256)
k_scatter_ids(const unsigned* __restrict__ key, const unsigned* __restrict__ rank,
              const unsigned* __restrict__ start, const float4* __restrict__ pos, int n, int* __restrict__ tmp,
              int* __restrict__ tmp_id)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned dst = start[key[i]] + rank[i];
    tmp[dst] = i;
    tmp_id[dst] = id_of(pos[i]);
}

cudaError_t launch_scatter_ids(const unsigned* key, const unsigned* rank, const unsigned* start, const float4* pos,
                               int n, int* tmp, int* tmp_id, cudaStream_t s, long long* launches)
{
    if (n <= 0) return cudaSuccess;
    k_scatter_ids<<<(n + 255) / 256, 256, 0, s>>>(key, rank, start, pos, n, tmp, tmp_id);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_scatter(const unsigned* key, const unsigned* rank, const unsigned* start, int n,
                           int* tmp, cudaStream_t s, long long* launches)
{
    if (n <= 0) return cudaSuccess;
    k_scatter<<<(n + 255) / 256, 256, 0, s>>>(key, rank, start, n, tmp);
    ++*launches;
    return cudaGetLastError();
}

// ------------------------------------------------ per-cell sort + gather

// One thread per sorted slot: the thread of slot s takes the storage index
// tmp[s] of its cell, ranks its id tmp_id[s] against the cell's other ids (a
// contiguous run of tmp_id, read by its threads together) and moves pos/vel
// to start[c] + rank, also writing x, y, z to the SoA copy (soa, soa_st
// floats per axis; may be NULL; hide: attached particles and positions that
// are not finite stand at HIDDEN there; the unpaired slot behind an odd number
// of particles is finite).  The attached particle of boid b records its sorted
// slot in slot_of_boid[b].  A cell of n entries costs n comparisons per
// entry; the entries are spread over the chip.  Read id by id, a crowded
// cell's pass waited for every 128-byte line in turn (its warps reach each new
// line together), so a warp passes the ids of a cell of more than SORT_STREAM
// entries through shared memory, 32 at a time, the next 64 on their way
// meanwhile.  One cell of 2,000, 16,000 and 40,000 entries, us: by a block's
// bitonic sort (which ranked the last by counting) 34, 213 and 66,000, read id
// by id 38, 265 and 661, now 20, 114 and 378; the large tank's boids 26 -> 17.  Lines of 32 to 256 entries give the same times.  The
// shared memory is kept small: with 128 ids a warp the tank's particles, which
// need none of it, took 59 instead of 58 (57 without the branch).
constexpr int SORT_STREAM = 128;

__global__ void __launch_bounds__(256)
k_cellsort_slots(const unsigned* __restrict__ start, const unsigned* __restrict__ key, int n,
                 const int* __restrict__ tmp, const int* __restrict__ tmp_id, const float4* __restrict__ pos_in,
                 const float4* __restrict__ vel_in, float4* __restrict__ pos_out,
                 float4* __restrict__ vel_out, float* __restrict__ soa, size_t soa_st, int hide, int nb,
                 int* __restrict__ slot_of_boid)
{
    __shared__ __align__(16) int s_ids[256 / 32][32];
    const int s = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool active = s < n;
    int src = 0, nc = 0, id = 0;
    unsigned s0 = 0;
    if (active) {
        src = tmp[s];
        const unsigned c = key[src];
        s0 = start[c];
        nc = (int)(start[c + 1] - s0);
        id = tmp_id[s];
    }
    const bool crowded = nc > SORT_STREAM;
    int r = 0;
    if (!crowded)
        for (int k = 0; k < nc; ++k) r += __ldg(tmp_id + s0 + k) < id;
    // the crowded cells of the warp's slots, one after another
    for (unsigned todo = __ballot_sync(FULL, crowded); todo;) {
        const int lead = __ffs((int)todo) - 1;
        const unsigned c0 = __shfl_sync(FULL, s0, lead), c1 = c0 + (unsigned)__shfl_sync(FULL, nc, lead);
        int* ids = s_ids[threadIdx.x >> 5];
        // past the cell: above every id
        auto fetch = [&](unsigned k) { return k < c1 ? __ldg(tmp_id + k) : 0x7fffffff; };
        int below = 0;
        int next = fetch(c0 + lane), next2 = fetch(c0 + 32 + lane);
        for (unsigned k = c0; k < c1; k += 32) {
            __syncwarp();  // the 32 before are read
            ids[lane] = next;
            __syncwarp();
            next = next2;
            next2 = fetch(k + 64 + lane);
#pragma unroll
            for (int q = 0; q < 32; q += 4) {
                const int4 o = *reinterpret_cast<const int4*>(ids + q);
                below += (o.x < id) + (o.y < id) + (o.z < id) + (o.w < id);
            }
        }
        const bool mine = crowded && s0 == c0;
        if (mine) r = below;
        todo &= ~__ballot_sync(FULL, mine);
    }
    if (!active) return;
    const unsigned dst = s0 + (unsigned)r;
    const float4 p = pos_in[src];
    pos_out[dst] = p;
    vel_out[dst] = vel_in[src];
    if (soa) {
        const bool away = hide && (id < nb || !(fabsf(p.x) < HIDDEN && fabsf(p.y) < HIDDEN && fabsf(p.z) < HIDDEN));
        soa[dst] = away ? HIDDEN : p.x;
        soa[soa_st + dst] = away ? 0.0f : p.y;
        soa[2 * soa_st + dst] = away ? 0.0f : p.z;
        if (s == n - 1 && (n & 1)) soa[n] = soa[soa_st + n] = soa[2 * soa_st + n] = 0.0f;
    }
    if (id < nb && slot_of_boid) slot_of_boid[id] = (int)dst;
}

cudaError_t launch_cellsort_slots(const unsigned* start, const unsigned* key, int n, const int* tmp,
                                  const int* tmp_id, const float4* pos_in, const float4* vel_in,
                                  float4* pos_out, float4* vel_out, float* soa, bool hide, int nb,
                                  int* slot_of_boid, cudaStream_t s, long long* launches)
{
    if (n <= 0) return cudaSuccess;
    k_cellsort_slots<<<(n + 255) / 256, 256, 0, s>>>(start, key, n, tmp, tmp_id, pos_in, vel_in, pos_out, vel_out,
                                                     soa, soa_stride((size_t)n), hide, nb, slot_of_boid);
    ++*launches;
    return cudaGetLastError();
}

// Key of every sorted slot, recovered from cell_start (warp per cell).
__global__ void __launch_bounds__(256)
k_slot_keys(const unsigned* __restrict__ start, int ncells, unsigned* __restrict__ slot_key)
{
    // (a grid of more than 2^27 cells has more threads than 32 bits count)
    const int c = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    int lane = threadIdx.x & 31;
    if (c >= ncells) return;
    for (unsigned s = start[c] + lane; s < start[c + 1]; s += 32) slot_key[s] = (unsigned)c;
}

cudaError_t launch_slot_keys(const unsigned* start, int ncells, unsigned* slot_key, cudaStream_t s,
                             long long* launches)
{
    if (ncells <= 0) return cudaSuccess;
    k_slot_keys<<<(ncells + 7) / 8, 256, 0, s>>>(start, ncells, slot_key);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace sphk
