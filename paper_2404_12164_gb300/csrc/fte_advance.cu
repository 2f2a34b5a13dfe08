// Transport kernels: the per-particle step loop with the fused occupancy tally,
// the reduction of the blocks' step counts, the FP64 per-step time
// table, the D_mumu normalisation integral and the intensity output.
#include "fte_step.cuh"

namespace fte {

// single-set kernels without cross-field diffusion are compiled for exactly the two blocks of
// 256 threads per SM that they get: told so, the compiler uses all 128 registers and keeps more
// record loads in flight (left to itself it took 104 - 110; 1e6 particles over 4 days of
// snapshots 603 -> 577 ms, 1e4 Parker particles 14.8 -> 13.2 ms; 28 - 56 bytes of spills, about
// one spilled load per step of 876 instructions).  The cross-field builds use
// 128 anyway and measured 2 % faster left alone.
constexpr int kMinBlocks = 512 / kThreads;

template <int DT, int MODE, int LAY, int SHAPE>
static const void* single_dt(int kperp)
{
    return kperp ? (const void*)advance_kernel<true, DT, MODE, kThreads, LAY>
                 : (const void*)advance_kernel<false, DT, MODE, kThreads, LAY, kMinBlocks, kOptAny, SHAPE>;
}

template <int MODE, int LAY>
static const void* single_fn(int kperp, int dtype)
{
    constexpr int shape = MODE == kModeSingle ? kShapeNormals : kShapeLoop;
    if (dtype == FTE_BF16) return single_dt<FTE_BF16, MODE, LAY, shape>(kperp);
    if (dtype == FTE_F16) return single_dt<FTE_F16, MODE, LAY, shape>(kperp);
    return single_dt<FTE_F32, MODE, LAY, shape>(kperp);
}

// the builds of block AMR (global tally, no cross-field diffusion), 128 registers and 16 warps per
// SM: FP32 records 4 blocks of 128 threads, 16-bit records 2 blocks of 256.  With the options
// fixed and the shorter step 16 warps overtook the register-limited builds that ran before (FP32,
// 1e7 particles x 320 steps: 145 ms with 20 warps at 102 registers, 136 with 16, 157 with 12 at
// 168; BF16, 24 warps at 85 registers and 250 bytes of spills against 16: 3e6 particles x 192
// steps 25.0 and 25.1 ms, 1e5 particles 1.40 and 1.30 ms).
constexpr int kDenseBlocks = 512 / kThreads;
constexpr int kAmr32Threads = 128;
constexpr int kAmr32Blocks = 4;
template <int LAY, int OPT = kOptAny, int SHAPE = kShapeLoop>
static const void* dense_fn(int dtype)
{
    if (dtype == FTE_BF16)
        return (const void*)advance_kernel<false, FTE_BF16, kModeSingleGlobal, kThreads, LAY, kDenseBlocks, OPT, SHAPE>;
    if (dtype == FTE_F16)
        return (const void*)advance_kernel<false, FTE_F16, kModeSingleGlobal, kThreads, LAY, kDenseBlocks, OPT, SHAPE>;
    return (const void*)advance_kernel<false, FTE_F32, kModeSingleGlobal, kAmr32Threads, LAY, kAmr32Blocks, OPT, SHAPE>;
}

// FP32 records, 5 blocks of 128 threads, 20 warps per SM at 96 registers, 64 - 80 bytes of spills
// (see advance_opt)
template <int LAY>
static const void* warps_fn()
{
    return (const void*)advance_kernel<false, FTE_F32, kModeSingleGlobal, kAmr32Threads, LAY, 5>;
}

// near: the build with the reach test of the observers (kShapeNear)
template <int DT>
static const void* linear_dt(bool near)
{
    constexpr int shape = kShapeUnroll | kShapeNormals;
    return near ? (const void*)advance_kernel<false, DT, kModeSingleGlobal, kThreads, kLayCell, kMinBlocks, kOptLinear,
                                              shape | kShapeNear>
                : (const void*)advance_kernel<false, DT, kModeSingleGlobal, kThreads, kLayCell, kMinBlocks, kOptLinear,
                                              shape>;
}

static const void* linear_fn(int dtype, bool near)
{
    if (dtype == FTE_BF16) return linear_dt<FTE_BF16>(near);
    if (dtype == FTE_F16) return linear_dt<FTE_F16>(near);
    return linear_dt<FTE_F32>(near);
}

static bool dense_variant(int kperp, int mode, int amr)
{
    return mode == kModeSingleGlobal && !kperp && amr;
}

int advance_opt(const GridK& g, const ParamsK& prm, int kperp, int mode, bool ordered, unsigned long long n, int sms)
{
    // FP32 block AMR with linear r, not reordered, more than 8 warps of particles per SM: the general
    // kernel in the build of 20 warps per SM.  Its 16-warp build, the faster one everywhere else, falls
    // behind there (per launch of 192 - 384 steps, 16 against 20 warps: 1e6 particles 37.2 and 32.2 ms,
    // in pair records 41.4 and 28.4; 3e5 15.4 and 12.9; 1.2e5 9.9 and 8.1; 6e4 5.3 and 4.3; but 2e4
    // 2.9 and 3.9; reordered, 1.2e5: 3.0 and 3.6).  Logarithmic r and 16-bit records do not show it.
    if (mode == kModeSingleGlobal && !kperp && g.amr > 0 && !g.radial && g.dtype == FTE_F32 && !ordered &&
        n > (unsigned long long)sms * 256)
        return kOptAnyWarps;
    const bool common = prm.dmumu == 0 && !prm.use_rig && prm.p_update == 0 && prm.dvdt_term;
    if (!common || kperp || g.pair || !global_tally(mode)) return kOptAny;
    if (g.amr > 0) return g.radial && mode == kModeSingleGlobal ? kOptAmrLog : kOptAny;
    return g.radial ? kOptAny : kOptLinear;
}

int advance_threads(int kperp, int dtype, int mode, int amr)
{
    return single_set(mode) && dense_variant(kperp, mode, amr) && dtype == FTE_F32 ? kAmr32Threads : kThreads;
}

// the single-set kernels come in one variant per record layout (pair: 1) and tally
// mode, for block AMR in a register-limited build, and for the common options (advance_opt)
// in one with these fixed
static const void* advance_fn(int kperp, int dtype, int mode, int nt, int pair, int amr, int opt, bool near = true)
{
    if (!single_set(mode)) return advance_fn_batched(kperp, dtype, mode, nt, pair, opt, near);
    if (nt != advance_threads(kperp, dtype, mode, amr)) return nullptr;
    if (opt == kOptAnyWarps) return pair ? warps_fn<kLayPair>() : warps_fn<kLayCell>();
    if (opt == kOptAmrLog)
        return near ? dense_fn<kLayCell, kOptAmrLog, kShapeNear>(dtype) : dense_fn<kLayCell, kOptAmrLog>(dtype);
    if (opt == kOptLinear) return linear_fn(dtype, near);
    if (dense_variant(kperp, mode, amr)) return pair ? dense_fn<kLayPair>(dtype) : dense_fn<kLayCell>(dtype);
    if (mode == kModeSingleGlobal)
        return pair ? single_fn<kModeSingleGlobal, kLayPair>(kperp, dtype)
                    : single_fn<kModeSingleGlobal, kLayCell>(kperp, dtype);
    return pair ? single_fn<kModeSingle, kLayPair>(kperp, dtype) : single_fn<kModeSingle, kLayCell>(kperp, dtype);
}

cudaError_t advance_occupancy(int kperp, int dtype, int mode, int nt, int pair, int amr, int opt, size_t smem,
                              int* blocks_per_sm)
{
    const void* fn = advance_fn(kperp, dtype, mode, nt, pair, amr, opt);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, nt, smem);
}

cudaError_t launch_advance(const AdvanceArgs& a, const BatchArgs& b, int kperp, int mode, int nt, int opt, int blocks,
                           size_t smem, cudaStream_t s)
{
    // reordered, or at most one particle per thread (see kShapeNear)
    const bool near = a.order || a.n_particles <= (unsigned long long)blocks * nt;
    if (!single_set(mode)) return launch_advance_batched(a, b, kperp, mode, nt, opt, near, blocks, smem, s);
    const void* fn = advance_fn(kperp, a.g.dtype, mode, nt, a.g.pair, a.g.amr > 0, opt, near);
    if (!fn) return cudaErrorInvalidValue;
    void* args[] = {(void*)&a, (void*)&b};
    // The global-tally kernels share nothing within a block, so blocks only decide how warps
    // spread over the SMs.  A pool that is not reordered goes in blocks of one warp: 1e4 particles
    // in blocks of 256 occupy 40 of 152 SMs with 8 warps each, in blocks of 32 every SM with 2, and
    // a step's latency falls with the warps it shares an SM with (1e4 particles x 8640 steps 19.1
    // -> 17.4 ms, 2000 x 200 0.54 -> 0.50 ms); 1.3e5 particles, two per thread, are 254 blocks of
    // 256, two on 102 SMs and one on 50.  A reordered pool launches one wave in blocks of 64: when
    // few particles are left alive and the surplus blocks leave at once (see advance_kernel), those
    // that stay are spread as evenly (1e6 particles over 4 days, 4.6e4 alive at the end: 543 ms in
    // blocks of 256, 531 of 128, 530 of 64, 528 of 32; 1.2e5 with cross-field diffusion 929 -> 910
    // us).  A block of the shared-memory tally carries a count of every bin and stays as it is.
    if (mode == kModeSingleGlobal) {
        const int small = a.order ? 64 : 32;
        const unsigned long long need = (a.n_particles + small - 1) / small,
                                 given = (unsigned long long)blocks * (nt / small);
        blocks = (int)(a.order || need >= given ? given : need);
        nt = small;
    }
    return cudaLaunchKernel(fn, dim3(blocks), dim3(nt), args, smem, s);
}

// ---------------------------------------------------------------------------
// Quantization of an FP32 background to 16-bit storage with per-field scales:
// (1) largest |value| per field (atomic max of the non-negative float bits),
// (2) zero scales become 1, (3) each record is encoded as the round-to-nearest-
// even of (value / scale), the quotient correctly rounded in FP32.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) maxabs_kernel(const float* __restrict__ f, long long nrec,
                                                     unsigned* hdr)
{
    float m[FTE_NFIELD];
#pragma unroll
    for (int k = 0; k < FTE_NFIELD; ++k) m[k] = 0.f;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < nrec;
         r += (long long)gridDim.x * blockDim.x) {
        float a[FTE_REC];
#pragma unroll
        for (int q = 0; q < FTE_REC / 8; ++q) ldg8(f + r * FTE_REC + 8 * q, a + 8 * q);
#pragma unroll
        for (int k = 0; k < FTE_NFIELD; ++k) m[k] = fmaxf(m[k], fabsf(a[k]));
    }
#pragma unroll
    for (int k = 0; k < FTE_NFIELD; ++k) {
        float v = m[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
        if ((threadIdx.x & 31) == 0 && v > 0.f) atomicMax(hdr + k, __float_as_uint(v));
    }
}

__global__ void scale_final_kernel(float* hdr)
{
    const int k = threadIdx.x;
    if (k < FTE_HHDR) hdr[k] = (k < FTE_NFIELD) ? (hdr[k] > 0.f ? hdr[k] : 1.f) : 0.f;
}

template <int DT>
__device__ __forceinline__ uint32_t encode16(float v)
{
    if (DT == FTE_BF16) return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v));
    return (uint32_t)__half_as_ushort(__float2half_rn(v));
}

// 16-bit records: cell layout (18 values, padded to FTE_HREC) or pair layout
// (the cell's 18 values, then those of its upper r-neighbour - zero at the end of
// an r-row of `row` cells - padded to kPairHRec).
template <int DT, bool PAIR>
__global__ void __launch_bounds__(256) encode_kernel(const float* __restrict__ f, long long nrec, int row,
                                                     const float* __restrict__ hdr, uint32_t* out)
{
    constexpr int kWords = (PAIR ? kPairHRec : FTE_HREC) / 2;
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrec) return;
    uint32_t w[kWords];
#pragma unroll
    for (int k = 0; k < kWords; ++k) w[k] = 0u;
    const bool hi_in_row = (r % row) != row - 1;
#pragma unroll
    for (int c = 0; c < (PAIR ? 2 : 1); ++c) {
        if (c == 1 && !hi_in_row) break;
        float a[FTE_REC];
#pragma unroll
        for (int q = 0; q < FTE_REC / 8; ++q) ldg8(f + (r + c) * FTE_REC + 8 * q, a + 8 * q);
#pragma unroll
        for (int k = 0; k < FTE_NFIELD; ++k) {
            const uint32_t h = encode16<DT>(__fdiv_rn(a[k], __ldg(hdr + k)));
            const int slot = c * FTE_NFIELD + k;
            w[slot >> 1] |= (slot & 1) ? (h << 16) : h;
        }
    }
    uint4* o = reinterpret_cast<uint4*>(out + r * kWords);
#pragma unroll
    for (int q = 0; q < kWords / 4; ++q) o[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// FP32 pair records from FP32 cell records.
__global__ void __launch_bounds__(256) pair_f32_kernel(const float* __restrict__ f, long long nrec, int row,
                                                       float* out)
{
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrec) return;
    float a[kPairRec];
#pragma unroll
    for (int k = 0; k < kPairRec; ++k) a[k] = 0.f;
    float b[FTE_REC];
#pragma unroll
    for (int q = 0; q < FTE_REC / 8; ++q) ldg8(f + r * FTE_REC + 8 * q, b + 8 * q);
#pragma unroll
    for (int k = 0; k < FTE_NFIELD; ++k) a[k] = b[k];
    if ((r % row) != row - 1) {
#pragma unroll
        for (int q = 0; q < FTE_REC / 8; ++q) ldg8(f + (r + 1) * FTE_REC + 8 * q, b + 8 * q);
#pragma unroll
        for (int k = 0; k < FTE_NFIELD; ++k) a[FTE_NFIELD + k] = b[k];
    }
    float4* o = reinterpret_cast<float4*>(out + r * kPairRec);
#pragma unroll
    for (int q = 0; q < kPairRec / 4; ++q) o[q] = make_float4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]);
}

// Per-field scales of FP32 cell records: `first` zeroes the header, each call
// folds nrec records into the running maxima, `last` turns them into scales.
cudaError_t launch_scales(const float* f32, long long nrec, float* hdr, bool first, bool last, cudaStream_t s)
{
    if (first) {
        const cudaError_t e = cudaMemsetAsync(hdr, 0, FTE_HHDR * sizeof(float), s);
        if (e != cudaSuccess) return e;
    }
    if (nrec > 0) maxabs_kernel<<<1216, 256, 0, s>>>(f32, nrec, reinterpret_cast<unsigned*>(hdr));
    if (last) scale_final_kernel<<<1, 32, 0, s>>>(hdr);
    return cudaGetLastError();
}

// FP32 cell records into pair and/or 16-bit records (16-bit: with the scales
// already in `hdr`), nrec records starting at `out_recs`.
cudaError_t launch_convert(const float* f32, long long nrec, int row, int dtype, int pair, const float* hdr,
                           void* out_recs, cudaStream_t s)
{
    const long long blocks = (nrec + 255) / 256;
    if (nrec <= 0) return cudaSuccess;
    if (dtype == FTE_F32) {
        if (!pair) return cudaErrorInvalidValue;
        pair_f32_kernel<<<(unsigned)blocks, 256, 0, s>>>(f32, nrec, row, reinterpret_cast<float*>(out_recs));
        return cudaGetLastError();
    }
    uint32_t* recs = reinterpret_cast<uint32_t*>(out_recs);
#define FTE_ENC(D, P) encode_kernel<D, P><<<(unsigned)blocks, 256, 0, s>>>(f32, nrec, row, hdr, recs)
    if (dtype == FTE_BF16) { if (pair) FTE_ENC(FTE_BF16, true); else FTE_ENC(FTE_BF16, false); }
    else { if (pair) FTE_ENC(FTE_F16, true); else FTE_ENC(FTE_F16, false); }
#undef FTE_ENC
    return cudaGetLastError();
}

cudaError_t launch_quantize(const float* f32, long long nrec, int row, int dtype, int pair, void* out,
                            cudaStream_t s)
{
    if (dtype == FTE_F32) return launch_convert(f32, nrec, row, dtype, pair, nullptr, out, s);
    float* hdr = reinterpret_cast<float*>(out);
    const cudaError_t e = launch_scales(f32, nrec, hdr, true, true, s);
    if (e != cudaSuccess) return e;
    return launch_convert(f32, nrec, row, dtype, pair, hdr, reinterpret_cast<char*>(out) + FTE_HHDR * sizeof(float), s);
}

// ---------------------------------------------------------------------------
// Sum of the blocks' step counts into the tally: each bin's blocks are summed by 8 warps.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) reduce_kernel(const unsigned* __restrict__ part, int nblk, int nbins,
                                                     unsigned long long* C)
{
    __shared__ unsigned long long rc[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int b = blockIdx.x * 32 + lane;
    unsigned long long c = 0;
    if (b < nbins)
        for (int k = wid; k < nblk; k += 8) c += part[(size_t)k * nbins + b];
    rc[wid][lane] = c;
    __syncthreads();
    if (wid == 0 && b < nbins) {
        for (int k = 1; k < 8; ++k) c += rc[k][lane];
        C[b] += c;
    }
}

cudaError_t launch_reduce(const unsigned* part, int nblk, int nbins, unsigned long long* C, cudaStream_t s)
{
    reduce_kernel<<<(nbins + 31) / 32, 256, 0, s>>>(part, nblk, nbins, C);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Per-step time table in FP64: t_n = t0 + n dt, bracketing snapshots and the
// time weight, and the time bin of every observer (rounded operations, no
// contraction, so that edges fall exactly where the definition puts them).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void step_table_entry(const StepTableArgs& a, long long k)
{
    const long long n = a.n0 + k;
    const double t = __dadd_rn(a.t0, __dmul_rn((double)n, a.dt));
    StepEntry e;
    e.s0 = 0; e.s1 = 0; e.wt = 0.f; e.two = 0;
    if (a.n_snap > 1) {
        const double tau = __ddiv_rn(__dsub_rn(t, a.t_snap0), a.dt_snap);
        // u0, u1: the snapshots in time order (periodic sequences unwrapped)
        long long u0 = 0, u1 = 0;
        if (a.periodic) {
            const double kf = floor(tau);
            u0 = (long long)kf;
            u1 = u0 + 1;
            e.wt = (float)(tau - kf);
            e.two = 1;
        } else if (tau < 0.0) {
            u0 = u1 = 0;
        } else if (tau >= (double)(a.n_snap - 1)) {
            u0 = u1 = a.n_snap - 1;
        } else {
            const double kf = floor(tau);
            u0 = (long long)kf;
            u1 = u0 + 1;
            e.wt = (float)(tau - kf);
            e.two = 1;
        }
        // storage slot: the snapshot itself, or its place in the ring
        const long long m = a.ring > 0 ? a.ring : a.n_snap;
        e.s0 = (int)(((u0 % m) + m) % m);
        e.s1 = (int)(((u1 % m) + m) % m);
    }
    for (int o = 0; o < FTE_MAX_OBS; ++o) {
        short it = -1;
        if (o < a.n_obs) {
            const ObsTime& ot = a.ot[o];
            const double f = floor(__ddiv_rn(__dmul_rn(__dsub_rn(t, ot.t_lo), (double)ot.nt),
                                             __dsub_rn(ot.t_hi, ot.t_lo)));
            if (f >= 0.0 && f < (double)ot.nt) it = (short)f;
        }
        e.it[o] = it;
    }
    a.tab[k] = e;
}

// ---------------------------------------------------------------------------
// Normalisation of D_mumu from lambda_par: I (quasi-linear) or J (Eq. 5), by
// composite Simpson in FP64 after mu = s^3; 1 for the isotropic form, one set per
// blockIdx.y.  The nodes are summed in trees of 256 and the trees' sums in order.
// A tree is spread over four blocks by node index mod 4 (its last two levels, which
// add the four residue classes, come in the second kernel): 16,385 FP64 powers on 260
// blocks of 64 threads keep every SM's slow FP64 unit busy (6.8 us), where 65 blocks of
// 256 ran on 65 SMs (11.4 us).
// ---------------------------------------------------------------------------
constexpr int kNormIntervals = 16384;
constexpr int kNormTree = 256;
constexpr int kNormTrees = kNormIntervals / kNormTree + 1;   // nodes 0 .. kNormIntervals
constexpr int kNormSplit = 4;
constexpr int kNormThreads = kNormTree / kNormSplit;
static_assert(kNormTrees * kNormSplit <= kNormPartials, "norm partials");

template <int NS>
struct NormArgs {
    int model;
    double q[NS], H[NS], eps[NS];
    double* part;                 // [set][kNormPartials]
};

template <int NS>
__global__ void __launch_bounds__(kNormThreads) norm_partial_kernel(const NormArgs<NS> a)
{
    __shared__ double upper[32];
    const int s = NS > 1 ? blockIdx.y : 0;
    const int tree = blockIdx.x / kNormSplit, c = blockIdx.x % kNormSplit, u = threadIdx.x;
    const int i = tree * kNormTree + u * kNormSplit + c;
    double f = 0.0;
    if (a.model != 2 && i <= kNormIntervals) {
        const double h = 1.0 / kNormIntervals;
        const double x = i * h;
        const double m = x * x * x;
        const double den = (a.model == 0) ? pow(m, a.q[s] - 1.0) + a.H[s] : m / (1.0 + m) + a.eps[s];
        const double wgt = (i == 0 || i == kNormIntervals) ? 1.0 : ((i & 1) ? 4.0 : 2.0);
        f = wgt * 3.0 * x * x * (1.0 - m * m) / den;
    }
    // the tree's levels above the four residue classes: node t adds node t + 128, 64, .. 4
    if (u >= 32) upper[u - 32] = f;
    __syncthreads();
    if (u >= 32) return;
    f += upper[u];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f += __shfl_down_sync(0xffffffffu, f, o);
    if (u == 0) a.part[(size_t)s * kNormPartials + blockIdx.x] = f;
}

// What the step kernels read besides the particles: the step table (blocks 0 .. table_blocks - 1)
// and the normalisation integrals from their partial sums (one further block), in one launch
// (5.3 us; 5.4 + 4.1 us in two).
__global__ void __launch_bounds__(256) setup_kernel(const StepTableArgs a, int table_blocks, int model, int n_sets,
                                                    const double* part, double* out)
{
    if ((int)blockIdx.x < table_blocks) {
        const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (k < a.count) step_table_entry(a, k);
        return;
    }
    __shared__ double tree[FTE_MAX_SETS * kNormTrees];
    for (int k = threadIdx.x; k < n_sets * kNormTrees; k += blockDim.x) {
        const double* p = part + (size_t)(k / kNormTrees) * kNormPartials + (k % kNormTrees) * kNormSplit;
        tree[k] = (p[0] + p[2]) + (p[1] + p[3]);       // the last two levels of the tree
    }
    __syncthreads();
    if ((int)threadIdx.x < n_sets) {
        double acc = 0.0;
        for (int b = 0; b < kNormTrees; ++b) acc += tree[threadIdx.x * kNormTrees + b];
        out[threadIdx.x] = (model == 2) ? 1.0 : acc / (3.0 * kNormIntervals);
    }
}

static cudaError_t launch_second(const StepTableArgs* ta, int model, int n_sets, const double* part, double* out,
                                 cudaStream_t s)
{
    StepTableArgs none = {};
    if (!ta) ta = &none;
    const int tb = (int)((ta->count + 255) / 256), blocks = tb + (n_sets > 0 ? 1 : 0);
    if (blocks > 0) setup_kernel<<<blocks, 256, 0, s>>>(*ta, tb, model, n_sets, part, out);
    return cudaGetLastError();
}

cudaError_t launch_step_table(const StepTableArgs& a, cudaStream_t s)
{
    return launch_second(&a, 2, 0, nullptr, nullptr, s);
}

cudaError_t launch_setup(int model, double q, double H, double eps, double* out, double* part,
                         const StepTableArgs* ta, cudaStream_t s)
{
    const NormArgs<1> a = {model, {q}, {H}, {eps}, part};
    norm_partial_kernel<1><<<kNormTrees * kNormSplit, kNormThreads, 0, s>>>(a);
    return launch_second(ta, model, 1, part, out, s);
}

cudaError_t launch_setup_sets(int model, const NormSets& ns, int n_sets, double* out, double* part,
                              const StepTableArgs* ta, cudaStream_t s)
{
    NormArgs<FTE_MAX_SETS> a;
    a.model = model;
    a.part = part;
    for (int k = 0; k < FTE_MAX_SETS; ++k) { a.q[k] = ns.q[k]; a.H[k] = ns.H[k]; a.eps[k] = ns.eps[k]; }
    norm_partial_kernel<FTE_MAX_SETS><<<dim3(kNormTrees * kNormSplit, n_sets), kNormThreads, 0, s>>>(a);
    return launch_second(ta, model, n_sets, part, out, s);
}

// ---------------------------------------------------------------------------
// Zeroes up to six arrays of 8-byte values in one launch (the tally and its ledger: 3 us instead
// of six clears of about 1.5 us each).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) zero_kernel(const ZeroArgs a)
{
    const size_t step = (size_t)gridDim.x * blockDim.x, first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
#pragma unroll
    for (int k = 0; k < 6; ++k)
        for (size_t i = first; i < a.n[k]; i += step) a.p[k][i] = 0ULL;
}

cudaError_t launch_zero(const ZeroArgs& a, cudaStream_t s)
{
    size_t most = 1;
    for (int k = 0; k < 6; ++k) most = a.n[k] > most ? a.n[k] : most;
    const size_t blocks = (most + 1023) / 1024;
    zero_kernel<<<(unsigned)(blocks < 1216 ? blocks : 1216), 256, 0, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Tally output for one observer: S, S2, C (as doubles) or the intensity
// j = S v(E_c) / (4 pi V_obs dt_bin dE).
// ---------------------------------------------------------------------------
// v(E_c) / (4 pi V dt dE) of energy row ie: the factor from the occupancy sum to the
// intensity.  Ring observers: V of one longitude bin, dt the whole time window.
__device__ double intensity_factor(const ObsOut& ob, int ie)
{
    const double pi = 3.141592653589793;
    double vol;
    if (ob.kind == 0) {
        const double lo = ob.r - ob.dr, hi = ob.r + ob.dr;
        vol = 4.0 * pi / 3.0 * (hi * hi * hi - lo * lo * lo);
    } else if (ob.kind == 1) {
        const double lo = ob.r - ob.dr, hi = ob.r + ob.dr;
        vol = (hi * hi * hi - lo * lo * lo) / 3.0 * (cos(ob.th - ob.dth) - cos(ob.th + ob.dth))
              * 2.0 * ob.dph;
    } else if (ob.kind == 3) {
        const double lo = ob.r - ob.dr, hi = ob.r + ob.dr;
        vol = (hi * hi * hi - lo * lo * lo) / 3.0 * (cos(ob.th - ob.dth) - cos(ob.th + ob.dth))
              * 2.0 * pi / ob.nt;
    } else {
        vol = 2.0 * ob.dr;
    }
    const double e0 = ob.e_lo * pow(ob.e_hi / ob.e_lo, (double)ie / ob.ne);
    const double e1 = ob.e_lo * pow(ob.e_hi / ob.e_lo, (double)(ie + 1) / ob.ne);
    const double ec = sqrt(e0 * e1);
    const double T = ec / 938.27208816;
    const double pm = sqrt(T * (T + 2.0));
    const double v = (299792458.0 / 1.495978707e11) * pm / sqrt(1.0 + pm * pm);
    const double dtb = ob.kind == 3 ? ob.t_hi - ob.t_lo : (ob.t_hi - ob.t_lo) / ob.nt;
    return v / (4.0 * pi * vol * dtb * (e1 - e0));
}

__global__ void tally_out_kernel(const double* S, const double* S2, const unsigned long long* C,
                                 const ObsOut ob, int kind, double* out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ob.ne * ob.nt) return;
    const int b = ob.off + k;
    if (kind == FTE_TALLY_S) { out[k] = S[b]; return; }
    if (kind == FTE_TALLY_S2) { out[k] = S2[b]; return; }
    if (kind == FTE_TALLY_C) { out[k] = (double)C[b]; return; }
    out[k] = S[b] * intensity_factor(ob, k / ob.nt);
}

// Green's function -> time-dependent source (Sec. 2.3): out[e][k] = dt_bin *
// sum_{m <= k} src[m] X[e][k - m], X = S or the intensity; src NULL = 1.
__global__ void convolve_kernel(const double* S, const ObsOut ob, int kind, const double* src, double* out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ob.ne * ob.nt) return;
    const int ie = k / ob.nt, it = k - ie * ob.nt;
    const double* row = S + ob.off + (size_t)ie * ob.nt;
    double acc = 0.0;
    for (int m = 0; m <= it; ++m) acc += (src ? src[m] : 1.0) * row[it - m];
    const double dtb = (ob.t_hi - ob.t_lo) / ob.nt;
    out[k] = dtb * acc * (kind == FTE_TALLY_INTENSITY ? intensity_factor(ob, ie) : 1.0);
}

cudaError_t launch_convolve(const double* S, const ObsOut& ob, int kind, const double* src, double* out,
                            cudaStream_t s)
{
    const int n = ob.ne * ob.nt;
    convolve_kernel<<<(n + 127) / 128, 128, 0, s>>>(S, ob, kind, src, out);
    return cudaGetLastError();
}

cudaError_t launch_tally_out(const double* S, const double* S2, const unsigned long long* C,
                             const ObsOut& ob, int kind, double* out, cudaStream_t s)
{
    const int n = ob.ne * ob.nt;
    tally_out_kernel<<<(n + 255) / 256, 256, 0, s>>>(S, S2, C, ob, kind, out);
    return cudaGetLastError();
}

}  // namespace fte
