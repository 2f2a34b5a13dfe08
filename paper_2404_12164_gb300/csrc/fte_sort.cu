// Spatial ordering of the alive particles: a counting sort by grid bucket (the
// lower corner of the interpolation stencil, radial index in pairs, and the sign
// of mu), so
// that consecutive entries of the order list - and so the lanes of a warp - read
// the same cache lines of the background.  Dead particles are left out, which
// also compacts the work list.  Performance only: each particle's trajectory does not depend on the order.
#include "fte_kernels.cuh"

namespace fte {


// Bucket of a point: the lower corner (i0, j0, k0) of its interpolation stencil -
// the first of the records the step gathers - with i0 taken in pairs, so that the
// particles of one bucket read the same corner records (a bucket by the cell
// holding the point would mix up to 3 x 2 x 2 different stencils).  The index
// arithmetic follows locate / locate_amr.
__device__ __forceinline__ int bucket_of(const GridK& g, float x, float y, float z)
{
    const float rho2 = x * x + y * y;
    const float r = sqrtf(rho2 + z * z);
    const float th = atan2f(sqrtf(rho2), z);
    float ph = atan2f(y, x);
    if (ph < 0.f) ph += kTwoPi;
    const float xr = g.radial ? logf(r / g.r_min) * g.inv_dr : (r - g.r_min) * g.inv_dr;
    const float xt = (th - g.th_min) * g.inv_dth;
    const float xp = ph * g.inv_dph;
    if (g.amr) {      // AMR: leaf, then the stencil corner on its padded lattice (0 .. B)
        const float ur = g.radial ? logf(r / g.r_min) * g.inv_lnr : (r - g.r_min) * g.inv_lnr;
        const float ut = (th - g.th_min) * g.inv_thspan;
        const float up = ph * (1.f / kTwoPi);
        const int f0 = min(max((int)floorf(ur * (float)g.nf0), 0), g.nf0 - 1);
        const int f1 = min(max((int)floorf(ut * (float)g.nf1), 0), g.nf1 - 1);
        int f2 = (int)floorf(up * (float)g.nf2);
        if (f2 < 0) f2 += g.nf2;
        if (f2 >= g.nf2) f2 -= g.nf2;
        const int leaf = min(max(__ldg(g.table + ((long long)f2 * g.nf1 + f1) * g.nf0 + f0), 0), g.amr_leaves - 1);
        const int4 lf = __ldg(g.leaves + leaf);
        const float s = (float)(1 << lf.x);
        const int B = g.B;
        const int ii = min(max((int)floorf(xr * s - 0.5f) - (lf.y * B - 1), 0), B);
        const int jj = min(max((int)floorf(xt * s - 0.5f) - (lf.z * B - 1), 0), B);
        const int kk = min(max((int)floorf(xp * s - 0.5f) - (lf.w * B - 1), 0), B);
        return ((leaf * (B + 1) + kk) * (B + 1) + jj) * ((B + 2) >> 1) + (ii >> 1);
    }
    const int i = min(max((int)floorf(xr - 0.5f), 0), g.nr - 2);
    const int j = min(max((int)floorf(xt - 0.5f), 0), g.nth - 2);
    int k = (int)floorf(xp - 0.5f);
    if (k < 0) k += g.nph;
    k = min(max(k, 0), g.nph - 1);
    const int nrb = (g.nr + 1) >> 1;
    return (k * g.nth + j) * nrb + (i >> 1);
}

// Within a bucket the particles are grouped by the sign of the pitch-angle cosine
// (kMuBins equal bins of mu): particles moving the same way along the field stay
// together for longer (mu changes on the scattering time, many reorderings apart),
// so the lanes of a warp keep sharing records through the launch.  Two bins
// measured best: four halve the particles per bucket for a smaller gain.
constexpr int kMuBins = 2;

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

__global__ void __launch_bounds__(256) key_kernel(const SortArgs a)
{
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    int key = -1, rank = 0;
    if (a.steps ? a.steps[i] > a.steps_min : a.status[i] == FTE_ALIVE) {
        int mb = 0;
        if (a.mu) mb = min(max((int)((a.mu[i] + 1.f) * (0.5f * kMuBins)), 0), kMuBins - 1);
        key = bucket_of(a.g, a.x[i], a.y[i], a.z[i]) * kMuBins + mb;
        rank = (int)atomicAdd(a.hist + key, 1u);
        if (rank == 0) a.tiles[key / kScanTile] = 1u;
    }
    a.key[i] = key;
    a.rank[i] = rank;
}

// Bucket counts -> first entry of every bucket in the order list, in one pass over the tiles of
// kScanTile buckets that hold particles: each block scans its tile and takes the tile's place in
// the list from the running total hist[nb] (buckets stay in order within a tile; which tile comes
// first does not matter to any result).  Most tiles are empty - the particles sit in a few per
// cent of the grid - so a tile's flag, set by its first particle, spares reading it, and before the
// next reordering only the flagged tiles are zeroed again.  The whole histogram (22 MB on a 512 x
// 60 x 180 grid, 0.2 GB on 11,296 AMR leaves) used to be cleared, read, and read and written once
// per reordering, in a clear and three scan launches: 38 us for the 22 MB against 9 us now, 0.24 ms
// against 24 us for the 0.2 GB (1e6 particles over 4 days 580 -> 543 ms, 3e5 in BF16 25.8 -> 23.7
// ms, 9e4 on 3-level AMR, 90 steps, 2.0 -> 1.0 ms).  The work counters of the step kernel that
// follows are reset here too.
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned* sh, unsigned* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    unsigned off = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) {
        const unsigned t = sh[w];
        if (w < wid) off += t;
        sum += t;
    }
    *total = sum;
    return off + x - v;
}

__global__ void __launch_bounds__(kScanThreads) scan_kernel(unsigned* hist, int nb, const unsigned* tiles,
                                                            unsigned long long* fetch, int n_fetch)
{
    __shared__ unsigned sh[kScanThreads / 32], s_base;
    if (blockIdx.x == 0)
        for (int q = threadIdx.x; q < n_fetch; q += kScanThreads) fetch[q] = 0ULL;
    if (tiles[blockIdx.x] == 0u) return;
    const long long base = (long long)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    unsigned v[kScanItems];
    unsigned sum = 0;
    const bool whole = base + kScanItems <= nb;     // base is a multiple of 16 entries: 16-byte accesses
    uint4* h4 = reinterpret_cast<uint4*>(hist + base);
    if (whole) {
#pragma unroll
        for (int q = 0; q < kScanItems / 4; ++q) {
            const uint4 t = h4[q];
            v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) v[q] = (base + q < nb) ? hist[base + q] : 0u;
    }
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) sum += v[q];
    unsigned total;
    const unsigned ex = block_exclusive_scan(sum, sh, &total);
    if (threadIdx.x == 0) s_base = atomicAdd(hist + nb, total);
    __syncthreads();
    unsigned run = s_base + ex;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        const unsigned t = v[q];
        v[q] = run;
        run += t;
    }
    if (whole) {
#pragma unroll
        for (int q = 0; q < kScanItems / 4; ++q)
            h4[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < kScanItems; ++q)
            if (base + q < nb) hist[base + q] = v[q];
    }
}

// Zeroes the flagged tiles and their flags, and the total.
__global__ void __launch_bounds__(kScanThreads) clear_kernel(unsigned* hist, int nb, unsigned* tiles)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) hist[nb] = 0u;
    if (tiles[blockIdx.x] == 0u) return;
    const long long base = (long long)blockIdx.x * kScanTile;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        const long long b = base + q * kScanThreads + threadIdx.x;
        if (b < nb) hist[b] = 0u;
    }
    __syncthreads();                  // every thread has read the flag
    if (threadIdx.x == 0) tiles[blockIdx.x] = 0u;
}

__global__ void __launch_bounds__(256) scatter_kernel(const SortArgs a)
{
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const int key = a.key[i];
    if (key >= 0) a.order[a.hist[key] + (unsigned)a.rank[i]] = (uint32_t)i;
}

int sort_buckets(const GridK& g)
{
    if (g.amr) return g.amr_leaves * (g.B + 1) * (g.B + 1) * ((g.B + 2) >> 1) * kMuBins;
    return g.nph * g.nth * ((g.nr + 1) >> 1) * kMuBins;
}

size_t sort_scratch_bytes(const GridK& g, unsigned long long n)
{
    const long long nb = sort_buckets(g);
    const long long ntiles = (nb + kScanTile - 1) / kScanTile;
    size_t b = 0;
    b += ((size_t)(nb + 1) * 4 + 255) & ~(size_t)255;        // hist / offsets
    b += ((size_t)(ntiles + 1) * 4 + 255) & ~(size_t)255;    // tile sums
    b += 3 * (((size_t)n * 4 + 255) & ~(size_t)255);         // key, rank, order
    return b;
}

void sort_carve(const GridK& g, unsigned long long n, char* p, SortArgs* a)
{
    const long long nb = sort_buckets(g);
    const long long ntiles = (nb + kScanTile - 1) / kScanTile;
    a->hist = (unsigned*)p; p += ((size_t)(nb + 1) * 4 + 255) & ~(size_t)255;
    a->tiles = (unsigned*)p; p += ((size_t)(ntiles + 1) * 4 + 255) & ~(size_t)255;
    a->key = (int*)p; p += ((size_t)n * 4 + 255) & ~(size_t)255;
    a->rank = (int*)p; p += ((size_t)n * 4 + 255) & ~(size_t)255;
    a->order = (uint32_t*)p;
    a->nb = (int)nb;
    a->ntiles = (int)ntiles;
}

cudaError_t launch_sort(const SortArgs& a, bool first, unsigned long long* fetch, int n_fetch, cudaStream_t s)
{
    if (first) {        // the workspace holds anything: histogram, total and flags lie side by side
        const cudaError_t e = cudaMemsetAsync(a.hist, 0, (char*)(a.tiles + a.ntiles) - (char*)a.hist, s);
        if (e != cudaSuccess) return e;
    } else {
        clear_kernel<<<a.ntiles, kScanThreads, 0, s>>>(a.hist, a.nb, a.tiles);
    }
    const unsigned blocks = (unsigned)((a.n + 255) / 256);
    if (blocks) key_kernel<<<blocks, 256, 0, s>>>(a);
    scan_kernel<<<a.ntiles, kScanThreads, 0, s>>>(a.hist, a.nb, a.tiles, fetch, n_fetch);
    if (blocks) scatter_kernel<<<blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace fte
