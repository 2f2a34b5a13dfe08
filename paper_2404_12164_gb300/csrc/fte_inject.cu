// Injection kernel (Sec. 2.3, Eq. 7): counter-based draws (tag 1: pitch-angle
// cosine and energy; tag 2: position attempt a), volume-uniform positions
// (optionally in a band of spiral phase) with optional div V < 0 acceptance on
// the stored cell values, weight 1 or 1/r^2.
//
// One thread owns one particle.  With the acceptance test a particle takes as many
// attempts as its draws need (about 8 on average where the compressions fill an eighth
// of the box, 35 for the slowest of 32), each with a dependent read of a random cell:
// run one after another per thread, the whole warp waits for its slowest lane
// (1e6 particles 747 us, and 90-130 us even for a few hundred).  So the warp shares the
// attempts: as long as more than 16 particles have none accepted yet, each makes its own on
// its lane; once at most 16, 8, .. 1 are left, a round evaluates 2, 4, .. 32 consecutive
// attempts of each, and each particle takes its first accepted attempt, which is the one
// it would have stopped at alone.  (With an exchange between the lanes in the rounds of one
// attempt too, a region where few attempts or none succeed was slower than one thread per
// particle: 1e6 particles, 100 attempts, none accepted 755 us alone, 1086 with the exchange,
// 795 as it is; 8 attempts between two looks at the warp, with 1, 4 and 16: 830, 808, 790.)
// The sets of an ensemble go in one launch (each on blocks of its own), and the ledger gets
// one atomic add per block instead of one per warp: all of them go to the same two addresses.
// Measured before -> after: 1e6 particles 747 -> 324 us, 1e5 158 -> 57 us, 3e3 129 -> 35 us, 64
// sets of 4e6 particles together 8.4 -> 1.3 ms.
#include "fte_kernels.cuh"

namespace fte {

constexpr int kInjThreads = 256;
constexpr int kInjWarps = kInjThreads / 32;
constexpr int kInjAlone = 8;      // attempts of a lane between two looks at the warp

__device__ __forceinline__ double warp_sum_f64(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ unsigned warp_sum_u32(unsigned v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Position attempt t of particle pid: (r, th, ph), and whether the cell there is accepted.
// r13, dr3: r1^3 and r2^3 - r1^3; c1, dc: cos(th1) and cos(th2) - cos(th1).
__device__ __forceinline__ bool attempt(const GridK& g, const InjectSet& a, float r13, float dr3, float c1, float dc,
                                        int t, uint32_t pid, uint2 key, float& r, float& th, float& ph)
{
    const uint4 q = philox4x32_10(make_uint4((uint32_t)t, pid, 2u, 0u), key);
    r = cbrtf(r13 + u01(q.x) * dr3);
    th = acosf(c1 + u01(q.y) * dc);
    ph = a.ph1 + u01(q.z) * (a.ph2 - a.ph1);
    if (a.spiral != 0.f) ph -= a.spiral * (r - a.spiral_rb);   // spiral phase -> longitude
    if (!a.use_divv) return true;
    float phw = fmodf(ph, kTwoPi);
    if (phw < 0.f) phw += kTwoPi;
    long long ri;
    if (g.amr) {
        int ci, cj, ck;
        const int leaf = amr_containing(g, r, th, phw, ci, cj, ck);
        ri = (long long)a.divv_snap * g.snap_recs + (((long long)leaf * g.P + ck + 1) * g.P + cj + 1) * g.P + ci + 1;
    } else {
        const float xr = g.radial ? logf(r / g.r_min) * g.inv_dr : (r - g.r_min) * g.inv_dr;
        const float xt = (th - g.th_min) * g.inv_dth;
        const float xp = phw * g.inv_dph;
        const int ci = min(max((int)floorf(xr), 0), g.nr - 1);
        const int cj = min(max((int)floorf(xt), 0), g.nth - 1);
        int ck = (int)floorf(xp) % g.nph;
        if (ck < 0) ck += g.nph;
        ri = (long long)a.divv_snap * g.snap_recs + ((long long)ck * g.nth + cj) * g.nr + ci;
    }
    float g00, g11, g22;
    // the cell's own fields lead its record in either layout
    if (g.dtype == FTE_F32) {
        const float* rec = g.fields + ri * (g.pair ? kPairRec : FTE_REC);
        g00 = __ldg(rec + 6); g11 = __ldg(rec + 10); g22 = __ldg(rec + 14);
    } else {
        // stored value times its field scale, rounded once
        const uint32_t* rec = g.hfields + ri * ((g.pair ? kPairHRec : FTE_HREC) / 2);
        const uint32_t w3 = __ldg(rec + 3), w5 = __ldg(rec + 5), w7 = __ldg(rec + 7);
        const bool bf = g.dtype == FTE_BF16;
        g00 = __fmul_rn(bf ? h_lo<FTE_BF16>(w3) : h_lo<FTE_F16>(w3), __ldg(g.scale + 6));
        g11 = __fmul_rn(bf ? h_lo<FTE_BF16>(w5) : h_lo<FTE_F16>(w5), __ldg(g.scale + 10));
        g22 = __fmul_rn(bf ? h_lo<FTE_BF16>(w7) : h_lo<FTE_F16>(w7), __ldg(g.scale + 14));
    }
    const float s01 = __fadd_rn(g00, g11);
    const float tr = __fadd_rn(s01, g22);
    return tr < a.divv_max;
}

template <int NS>
__global__ void __launch_bounds__(kInjThreads) inject_kernel(const InjectArgs<NS> k)
{
    __shared__ float s_c[4];                      // cos(th1), cos(th2); e1^(1-gamma), e2^(1-gamma)
    __shared__ unsigned char s_own[kInjWarps][32];
    __shared__ double s_w[kInjWarps];
    __shared__ unsigned s_n[kInjWarps][2];
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    // the block's set: the last one that starts at or before this block
    int s = 0;
    if (NS > 1) {
        int hi = k.n_sets - 1;
        while (s < hi) {
            const int mid = (s + hi + 1) >> 1;
            if (k.set[mid].block0 <= blockIdx.x) s = mid; else hi = mid - 1;
        }
    }
    const InjectSet& a = k.set[s];
    if (threadIdx.x < 2) {
        if (a.region == 1) s_c[threadIdx.x] = cosf(threadIdx.x ? a.th2 : a.th1);
        if (a.energy == 1) s_c[2 + threadIdx.x] = powf(threadIdx.x ? a.e2 : a.e1, 1.f - a.gamma);
    }
    __syncthreads();
    const unsigned long long i = (unsigned long long)(blockIdx.x - a.block0) * kInjThreads + threadIdx.x;
    const bool mine = i < a.n;
    const uint32_t pid = a.id_base + (uint32_t)i;
    const uint2 key = make_uint2(a.seed, a.set_id);
    float r = a.r, th = a.th, ph = a.ph;
    bool ok = mine;
    if (a.region == 1) {
        const float r13 = a.r1 * a.r1 * a.r1, dr3 = a.r2 * a.r2 * a.r2 - r13, c1 = s_c[0], dc = s_c[1] - c1;
        ok = false;
        int t0 = 0;                               // attempts made by every particle still pending
        unsigned pend = __ballot_sync(0xffffffffu, mine);
        while (__popc(pend) > 16 && t0 < a.max_tries) {
            const int e = a.max_tries - t0 < kInjAlone ? a.max_tries : t0 + kInjAlone;
            for (int t = t0; t < e && mine && !ok; ++t) ok = attempt(k.g, a, r13, dr3, c1, dc, t, pid, key, r, th, ph);
            pend = __ballot_sync(0xffffffffu, mine && !ok);
            t0 = e;
        }
        while (pend != 0u && t0 < a.max_tries) {
            const int u = __popc(pend);
            const AttemptRound round(u, t0, a.max_tries);
            const int g = round.width;
            const bool waits = (pend >> lane) & 1u;
            const int rank = __popc(pend & ((1u << lane) - 1u));
            if (waits) s_own[wid][rank] = (unsigned char)lane;
            __syncwarp();
            const int q = (int)lane / g, j = (int)lane % g;
            const bool works = q < u && j < round.made;
            const unsigned owner = works ? s_own[wid][q] : lane;
            __syncwarp();                         // read by every lane before the next round's stores
            const uint32_t opid = pid - lane + owner;     // ids are consecutive within the warp
            float tr = 0.f, tth = 0.f, tph = 0.f;
            bool hit = false;
            if (works) hit = attempt(k.g, a, r13, dr3, c1, dc, t0 + j, opid, key, tr, tth, tph);
            const unsigned hits = __ballot_sync(0xffffffffu, hit);
            const unsigned seg = waits ? (hits >> (rank * g)) & (g == 32 ? 0xffffffffu : (1u << g) - 1u) : 0u;
            // the accepted attempt, or the last one of a particle that runs out of attempts
            const int src = waits ? rank * g + (seg ? __ffs(seg) - 1 : round.made - 1) : (int)lane;
            const float fr = __shfl_sync(0xffffffffu, tr, src);
            const float fth = __shfl_sync(0xffffffffu, tth, src);
            const float fph = __shfl_sync(0xffffffffu, tph, src);
            if (waits) { r = fr; th = fth; ph = fph; }
            if (seg) ok = true;
            pend = __ballot_sync(0xffffffffu, waits && !seg);
            t0 += round.made;
        }
    }
    double wsum = 0.0;
    unsigned nok = 0, nfail = 0;
    if (mine) {
        const unsigned long long idx = a.offset + i;
        const uint4 d = philox4x32_10(make_uint4(0u, pid, 1u, 0u), key);
        const float mu = a.mu_mode ? a.mu0 : u11(d.x);
        float E;
        if (a.energy == 0) {
            E = a.e0;
        } else if (fabsf(a.gamma - 1.f) < 1e-6f) {
            E = a.e1 * powf(a.e2 / a.e1, u01(d.y));
        } else {
            const float g1 = 1.f - a.gamma;
            const float lo = s_c[2], hi = s_c[3];
            E = powf(lo + u01(d.y) * (hi - lo), 1.f / g1);
        }
        const float T = E / kMc2;
        const float p = sqrtf(T * (T + 2.f));
        float sp, cp, st, ct;
        sincosf(ph, &sp, &cp);
        sincosf(th, &st, &ct);
        k.x[idx] = r * st * cp;
        k.y[idx] = r * st * sp;
        k.z[idx] = r * ct;
        k.mu[idx] = mu;
        k.p[idx] = p;
        k.id[idx] = pid;
        const float w = a.weight ? 1.f / (r * r) : 1.f;
        k.w[idx] = ok ? w : 0.f;
        k.status[idx] = ok ? FTE_ALIVE : FTE_INJ_FAIL;
        if (ok) { wsum = (double)w; nok = 1; } else nfail = 1;
    }
    wsum = warp_sum_f64(wsum);
    nok = warp_sum_u32(nok);
    nfail = warp_sum_u32(nfail);
    if (lane == 0) { s_w[wid] = wsum; s_n[wid][0] = nok; s_n[wid][1] = nfail; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < kInjWarps; ++q) { wsum += s_w[q]; nok += s_n[q][0]; nfail += s_n[q][1]; }
        if (nok) {
            atomicAdd(&k.ledger_w[0], wsum);
            atomicAdd(&k.ledger_n[0], (unsigned long long)nok);
        }
        if (nfail) atomicAdd(&k.ledger_n[5], (unsigned long long)nfail);
    }
}

template <int NS>
cudaError_t launch_inject(InjectArgs<NS>& a, cudaStream_t s)
{
    unsigned long long blocks = 0;
    for (int q = 0; q < a.n_sets; ++q) {
        a.set[q].block0 = (unsigned)blocks;
        blocks += (a.set[q].n + kInjThreads - 1) / kInjThreads;
    }
    if (blocks) inject_kernel<NS><<<(unsigned)blocks, kInjThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template cudaError_t launch_inject<1>(InjectArgs<1>&, cudaStream_t);
template cudaError_t launch_inject<FTE_MAX_SETS>(InjectArgs<FTE_MAX_SETS>&, cudaStream_t);

}  // namespace fte
