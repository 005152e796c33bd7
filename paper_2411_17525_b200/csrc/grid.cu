// Grid fit of Algorithm 2 ("CLVQ(n, p), computed once"), run as Lloyd's batch
// iteration on caller-provided samples of N(0, I_p): the assignment step is the
// encoder's exhaustive nearest-point rule, the update a segmented mean.
#include "common.cuh"

namespace higgs {

namespace {

constexpr int kFitThreads = 1024;
constexpr int kMaxFitBlocks = 1024;
constexpr int kNear = 32;              // centres in a cell's neighbour list
constexpr int kNearRow = 40;           // ... which is 80 bytes in shared memory: the lists of a warp's cells spread over the banks
constexpr int kLaneScans = 160;        // more listed scans than this in a batch: one per lane instead of one per warp
constexpr int kMinNearCentres = 65;    // grids with lists: below, a scan is no longer than a list or two ...
constexpr int kMaxNearCentres = 512;   // ... above, building the lists costs as much as the scans they save
constexpr int kMaxSharedSums = 1024;   // coordinates whose changes a block collects in shared memory first
constexpr int kQueueRounds = 4;        // samples a lane tests before the block scans those that need it
constexpr int64_t kAdaptSamples = 1 << 20;   // sets from which on the fit decides by measured work whether bounds pay

struct GridWs {
    float* centres;               // [n][p]
    long long* delta;             // [3][n][p] changes of the cells' sums, fixed point
    int32_t* delta_cnt;           // [3][n]    changes of the cells' sizes
    double* err;                  // [kMaxFitBlocks] squared error of a block's samples; before the fit the range of the samples, as uint2
    unsigned long long* bar;      // [2] grid barrier: arrivals (low half), blocks with a changed assignment (high half)
    unsigned long long* work;     // [3] scans of an iteration in steps of a warp (three in turn)
    int32_t* flags;               // [0] done, [1] iterations, [2] the samples are left to plain_fit_kernel, [3] a barrier ran out
    uint16_t* near_idx;           // [kMaxNearCentres][kNear] neighbour lists
    float* excl;                  // [kMaxNearCentres]
    int32_t* assign;              // [m]
    float* lower;                 // [m]
};

__host__ __device__ inline size_t up256(size_t v) { return (v + 255) / 256 * 256; }

GridWs carve(void* ws, int p, int n, int64_t m) {
    uint8_t* b = static_cast<uint8_t*>(ws);
    GridWs w;
    w.centres = reinterpret_cast<float*>(b); b += up256(sizeof(float) * n * p);
    w.delta = reinterpret_cast<long long*>(b); b += up256(sizeof(long long) * 3 * n * p);
    w.delta_cnt = reinterpret_cast<int32_t*>(b); b += up256(sizeof(int32_t) * 3 * n);
    w.err = reinterpret_cast<double*>(b); b += up256(sizeof(double) * kMaxFitBlocks);
    w.bar = reinterpret_cast<unsigned long long*>(b);
    w.flags = reinterpret_cast<int32_t*>(b + 16);
    w.work = reinterpret_cast<unsigned long long*>(b + 64); b += 256;
    w.near_idx = reinterpret_cast<uint16_t*>(b); b += sizeof(uint16_t) * kMaxNearCentres * kNear;
    w.excl = reinterpret_cast<float*>(b); b += sizeof(float) * kMaxNearCentres;
    w.assign = reinterpret_cast<int32_t*>(b); b += up256(sizeof(int32_t) * (size_t)m);
    w.lower = reinterpret_cast<float*>(b);
    return w;
}

// Also the bits of the largest |coordinate| among a block's samples.
constexpr int kRangeThreads = 256;
__global__ void __launch_bounds__(kRangeThreads) grid_init_kernel(GridWs w, const float* __restrict__ samples, int p, int n, int64_t m) {
    __shared__ unsigned s_top[kRangeThreads / 32];
    const int64_t first = (int64_t)blockIdx.x * kRangeThreads + threadIdx.x, step = (int64_t)gridDim.x * kRangeThreads;
    for (int64_t i = first; i < (int64_t)3 * n * p; i += step) w.delta[i] = 0;
    for (int64_t i = first; i < 3 * n; i += step) w.delta_cnt[i] = 0;
    for (int64_t i = first; i < n * p; i += step) w.centres[i] = samples[i];       // (the result if a barrier runs out)
    if (first < 2) w.bar[first] = 0;
    if (first < 8) w.flags[first] = 0;
    if (first < 3) w.work[first] = 0;
    unsigned top = 0u;
    for (int64_t i = first; i < m; i += step) {
        w.assign[i] = -1;
        for (int k = 0; k < p; ++k) top = max(top, __float_as_uint(fabsf(samples[i * p + k])));
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) s_top[threadIdx.x >> 5] = top;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kRangeThreads / 32; ++i) top = max(top, s_top[i]);
        reinterpret_cast<uint2*>(w.err)[blockIdx.x] = make_uint2(top, 0u);
    }
}

// The scale of the fixed-point sums, 2^shift: m times the largest |coordinate|, below 2^(exponent - 126), stays below 2^62.
__device__ __forceinline__ int sum_shift(unsigned top, int64_t m) { return 62 - (m > 1 ? 64 - __clzll(m - 1) : 0) - (max((int)(top >> 23), 1) - 126); }
__device__ __forceinline__ double power_of_two(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// The largest |coordinate| over all blocks (slots at most kFitThreads, one per thread of a block of 32 warps at most).
__device__ __forceinline__ uint2 range_of(const GridWs& w, int slots) {
    __shared__ unsigned s_top, s_rounded;
    if (threadIdx.x == 0) s_top = s_rounded = 0u;
    __syncthreads();
    unsigned top = 0u, rounded = 0u;
    for (int i = threadIdx.x; i < slots; i += blockDim.x) {
        const uint2 r = reinterpret_cast<const uint2*>(w.err)[i];
        top = max(top, r.x);
        rounded += r.y;
    }
    top = __reduce_max_sync(0xffffffffu, top);
    rounded = __reduce_add_sync(0xffffffffu, rounded);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&s_top, top);
        atomicAdd(&s_rounded, rounded);
    }
    __syncthreads();
    return make_uint2(s_top, s_rounded);
}

// The number of a block's samples with a coordinate that the fixed-point sums round.  (Same grid as grid_init_kernel; a block
// writes only the second half of its slot.)
__global__ void __launch_bounds__(kRangeThreads) grid_range_kernel(GridWs w, const float* __restrict__ samples, int p, int64_t m, int slots) {
    const double scale = power_of_two(sum_shift(range_of(w, slots).x, m));
    unsigned rounded = 0u;
    for (int64_t i = (int64_t)blockIdx.x * kRangeThreads + threadIdx.x; i < m; i += (int64_t)gridDim.x * kRangeThreads) {
        bool exact = true;
        for (int k = 0; k < p; ++k) {
            const double v = (double)samples[i * p + k] * scale;
            exact = exact && rint(v) == v;
        }
        rounded += exact ? 0u : 1u;
    }
    __shared__ unsigned s_count;
    if (threadIdx.x == 0) s_count = 0u;
    __syncthreads();
    rounded = __reduce_add_sync(0xffffffffu, rounded);
    if ((threadIdx.x & 31) == 0 && rounded) atomicAdd(&s_count, rounded);
    __syncthreads();
    if (threadIdx.x == 0) reinterpret_cast<uint2*>(w.err)[blockIdx.x].y = s_count;
}

// Whether a sample set is left to plain_fit_kernel: more than one sample in 32 would be rounded (an outlier of 2^16 among 2^18
// samples of N(0, I) rounds those below 2^-5, one in 40; a coordinate of 2^(23 - shift) or more is exact, so a mean beyond that is
// off by half an ulp at most), or squares and their sums may leave the normal fp32 range, on which the bounds rely.
__device__ __forceinline__ bool range_unsuited(uint2 range, int64_t m) {
    return (range.x >> 23) >= 127 + 61 || (range.x >> 23) < 127 - 40 || range.y > (unsigned)(m >> 5);
}

// Every block is resident (a cooperative launch, or one block), so the blocks can meet at a barrier: a counter in the
// workspace that every block's first thread adds to and then polls, with a limit on the polls - a barrier that runs out
// raises the grid-fit status word and the fit's own flag, and every block leaves.  The same addition counts the blocks that report `changed`.
// Two counters take turns (barrier number `no` uses no % 2), so a block that reads late cannot see the next barrier's.
__device__ int g_grid_status = 0;
constexpr unsigned kGridBarrierLimit = 1u << 22;

// returns whether any block reported a change in this barrier; *ok = false if it ran out.  RUN_OUT (a test): one arrival more is
// waited for than there are blocks, for a short time.
template <bool RUN_OUT>
__device__ __forceinline__ bool grid_barrier(const GridWs& w, int no, bool changed, unsigned& seen, bool* ok) {
    __shared__ unsigned s_high;
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long* counter = w.bar + (no & 1);
        const unsigned target = (unsigned)(no / 2 + 1) * (gridDim.x + (RUN_OUT ? 1u : 0u));
        __threadfence();
        atomicAdd(counter, 1ull | (changed ? 1ull << 32 : 0ull));
        unsigned it = 0;
        unsigned long long v;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(counter) : "memory");
            if ((unsigned)v >= target || ++it > (RUN_OUT ? 1u << 10 : kGridBarrierLimit)) break;
        }
        __threadfence();
        s_high = (unsigned)(v >> 32);
        s_ok = (unsigned)v >= target;
        if ((unsigned)v < target) {
            atomicExch(&g_grid_status, (int)HIGGS_ERR_TIMEOUT);
            w.flags[3] = 1;
        }
    }
    __syncthreads();
    *ok = s_ok != 0;
    const bool any = s_high != seen;
    seen = s_high;
    return any;
}

// fp32 squared distance, plain sum of (x_k - c_k)^2 in coordinate order: the encoder's rule
template <int P>
__device__ __forceinline__ float centre_distance(const float (&x)[P], const float* c) {
    float d = 0.f;
#pragma unroll
    for (int k = 0; k < P; ++k) {
        const float e = x[k] - c[k];
        d = k == 0 ? e * e : fmaf(e, e, d);
    }
    return d;
}

// The nearest of all centres; centre 0 when no distance compares below infinity.
template <int P>
__device__ __forceinline__ int nearest_centre(const float (&x)[P], const float* sc, int n, float& best) {
    int bi = 0;
    best = INFINITY;
#pragma unroll 4
    for (int q = 0; q < n; ++q) {
        const float d = centre_distance<P>(x, sc + q * P);
        if (d < best) { best = d; bi = q; }
    }
    return bi;
}

// What grid_finalize_kernel reads: this block's share of the squared error, and from block 0 the rest.
__device__ __forceinline__ void write_result(const GridWs& w, const float* sc, int coords, double err, bool done, int it, double* s_err) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) err += __shfl_xor_sync(0xffffffffu, err, k);
    if ((tid & 31) == 0) s_err[tid >> 5] = err;
    __syncthreads();
    if (tid == 0) {
        double total = 0.0;
        for (int i = 0; i < kFitThreads / 32; ++i) total += s_err[i];
        w.err[blockIdx.x] = total;
        if (blockIdx.x == 0) { w.flags[0] = done ? 1 : 0; w.flags[1] = it; }
    }
    if (blockIdx.x == 0)
        for (int i = tid; i < coords; i += kFitThreads) w.centres[i] = sc[i];
}

// The iteration as it stands, without bounds and with fp64 sums over all samples, for the sample sets that grid_fit_kernel leaves
// untouched (it is launched after that kernel every time; a kernel of its own because a call in there takes registers from the
// other path: 2 % of its time).  The sums of an iteration are in w.delta (as doubles), three buffers in turn as there.
template <int P, bool RUN_OUT>
__global__ void __launch_bounds__(kFitThreads, 1) plain_fit_kernel(GridWs w, const float* __restrict__ samples, int n, int64_t m, int max_iters) {
    if (!w.flags[2]) return;
    extern __shared__ __align__(16) unsigned char grid_smem[];
    double* block_sums = reinterpret_cast<double*>(grid_smem);         // [n][P]
    float* sc = reinterpret_cast<float*>(block_sums + (size_t)n * P);  // [n][P]
    int* block_cnt = reinterpret_cast<int*>(sc + (size_t)n * P);       // [n]
    __shared__ double s_err[kFitThreads / 32];
    const int tid = threadIdx.x, blocks = (int)gridDim.x;
    const int64_t first = ((int64_t)(tid >> 5) * blocks + blockIdx.x) * 32 + (tid & 31), step = (int64_t)blocks * kFitThreads;
    unsigned seen[2] = {0u, 0u};
    double err = 0.0;
    int it = 0;
    bool done = false, ok;
    for (int i = tid; i < n * P; i += kFitThreads) sc[i] = samples[i];
    for (; it < max_iters; ++it) {
        for (int i = tid; i < n * P; i += kFitThreads) block_sums[i] = 0.0;
        for (int i = tid; i < n; i += kFitThreads) block_cnt[i] = 0;
        __syncthreads();
        err = 0.0;
        int changed = 0;
        for (int64_t i = first; i < m; i += step) {
            float x[P], best;
#pragma unroll
            for (int k = 0; k < P; ++k) x[k] = samples[i * P + k];
            const int to = nearest_centre<P>(x, sc, n, best);
            if (w.assign[i] != to) { w.assign[i] = to; changed = 1; }
            err += (double)best;
#pragma unroll
            for (int k = 0; k < P; ++k) atomicAdd(&block_sums[to * P + k], (double)x[k]);
            atomicAdd(&block_cnt[to], 1);
        }
        const bool block_changed = __syncthreads_or(changed) != 0;
        double* sums = reinterpret_cast<double*>(w.delta) + (size_t)(it % 3) * n * P;
        int32_t* cnt = w.delta_cnt + (size_t)(it % 3) * n;
        for (int i = tid; i < n * P; i += kFitThreads)
            if (block_cnt[i / P]) atomicAdd(&sums[i], block_sums[i]);
        for (int i = tid; i < n; i += kFitThreads)
            if (block_cnt[i]) atomicAdd(&cnt[i], block_cnt[i]);
        const bool any = grid_barrier<RUN_OUT>(w, it, block_changed, seen[it & 1], &ok);
        if (!ok) return;
        if (!any) { done = true; ++it; break; }
        for (int i = tid; i < n * P; i += kFitThreads) {
            const int size = __ldcg(&cnt[i / P]);
            if (size > 0) sc[i] = (float)(__ldcg(&sums[i]) / (double)size);      // (an empty cell keeps its centre)
        }
        if (blockIdx.x == 0) {
            const int old = (it + 2) % 3;
            for (int i = tid; i < n * P; i += kFitThreads) w.delta[(size_t)old * n * P + i] = 0;
            for (int i = tid; i < n; i += kFitThreads) w.delta_cnt[(size_t)old * n + i] = 0;
        }
        __syncthreads();
    }
    write_result(w, sc, n * P, err, done, it, s_err);
}

__host__ __device__ inline bool fit_lists(int n) { return n >= kMinNearCentres && n <= kMaxNearCentres; }
inline size_t fit_smem(int p, int n) {
    return (size_t)n * p * (sizeof(long long) + sizeof(float)) + (size_t)n * sizeof(int) +
           (n * p <= kMaxSharedSums ? (size_t)n * p * 8 + (size_t)n * 4 : 0) + (fit_lists(n) ? (size_t)n * (kNearRow * 2 + 20) + 16 : 0);
}

// The whole iteration in ONE cooperatively launched kernel, one barrier per iteration.
//   * Assignment.  A sample keeps its cell without a scan while a lower bound on its distance to every OTHER centre
//     exceeds its distance to its own (Hamerly, "Making k-means even faster", 2010).  The bound is the second-best
//     distance at the last scan minus what the centres have moved since; the movements add up in a running total M, and
//     a bound is stored once, as bound + M.  Bounds are rounded down, distances up, by more than fp32 rounding of the
//     squared distances (a few 2^-24 relative), so a skipped scan could not have ended differently - same centre, lowest
//     index on ties.  The largest movement is that of a few outer centres with few samples, so for grids of 65 to 512
//     points every cell a has a list of the up to 32 centres nearest to its own, and M counts only their movements: a
//     centre outside the list is at least D_a from centre a, so it is no rival while the sample is nearer than D_a / 2
//     to a, with D_a reduced by twice the movement of any centre since the lists were built.  A scan then covers the
//     list.  When that movement exceeds 0.15 of the smallest D_a the lists are built anew.
//     The samples that need a scan go through a queue of the block, so that its warps share them evenly, a warp scanning
//     one at a time; many scans are done one per lane.
//   * Update.  Only samples that changed cell touch the sums.  The sums are 64-bit fixed point, scaled so that m times the
//     largest |coordinate| stays below 2^62: for N(0, I) samples all but the tiniest coordinates are represented
//     exactly, and integer sums do not depend on the order of the atomics.  (Sample sets that this does not suit go to
//     plain_fit_kernel.)  Every block adds the iteration's changes to
//     its own copy of the sums and computes the new centres itself, so no second barrier is needed.  Three buffers take
//     turns: the changes of iteration i are read after its barrier; block 0 clears those of i - 1, which every block has
//     read before it arrived there, for iteration i + 2.
//   * Large sets (ADAPT) are bound by the scans, not by latency, and bounds then have to pay for themselves: keeping the second-best
//     distance makes a scan 1.3 times as long, and while the centres still move much, or without lists, most samples are scanned all the
//     same.  The fit starts with four iterations of plain scans (one with lists of a sixth of the centres); then one that sets the bounds, then bounded ones, whose scans are
//     counted.  When they cost more than 0.85 of scanning everything, plain iterations follow, 8, 16, 32, 64, and another try.  (2^24 samples,
//     30 iterations, plain scans with fp64 sums / bounds always / this, in ms: p = 2, n = 16 9.3 / 7.5 / 4.8, n = 64 11.1 / 17.3 / 11.2, n = 65
//     11.5 / 13.0 / 11.4, n = 256 34.8 / 14.9 / 15.1, n = 600 84.9 / 88.6 / 75.8.  Below 2^20 samples bounds are ahead from the start.)
// Bound: latency - per iteration about 2.5 us of barrier, 2 us of update, 2.5 us to test the samples and 1 to 2 us of scans.
// p = 2, n = 256, 2^18 samples: 37 -> 9 us per iteration (before: every sample scanned all centres every time, sums by
// fp64 atomics in shared memory, two barriers).  One barrier and movement bounds without lists: 12.4 us.
template <int P, bool RUN_OUT, bool ADAPT>
__global__ void __launch_bounds__(kFitThreads, 1) grid_fit_kernel(GridWs w, const float* __restrict__ samples, int n, int64_t m, int slots, int max_iters) {
    extern __shared__ __align__(16) unsigned char grid_smem[];
    const bool shared_sums = n * P <= kMaxSharedSums, lists = fit_lists(n);
    long long* sums = reinterpret_cast<long long*>(grid_smem);         // [n][P]
    float* sc = reinterpret_cast<float*>(sums + (size_t)n * P);        // [n][P]
    int* cnt = reinterpret_cast<int*>(sc + (size_t)n * P);             // [n]
    unsigned* d_lo = reinterpret_cast<unsigned*>(cnt + n);             // [n][P] this block's changes: low and high halves, sizes
    unsigned* d_hi = d_lo + (shared_sums ? n * P : 0);
    int* d_cnt = reinterpret_cast<int*>(d_hi + (shared_sums ? n * P : 0));
    float* excl = reinterpret_cast<float*>(d_cnt + (shared_sums ? n : 0));      // [n] D_a when the lists were built
    float* near_moved = excl + n;                                      // [n] M of a cell
    float* went = near_moved + n;                                      // [n] the centre's movement in this iteration
    float* old_reach = went + n;                                       // [n] D_a of the lists before, now
    float* old_moved = old_reach + n;                                  // [n] M with the lists before
    uint16_t* near_idx = reinterpret_cast<uint16_t*>((reinterpret_cast<uintptr_t>(old_moved + n) + 15) & ~(uintptr_t)15);  // [n][kNearRow], padded with the cell itself
    __shared__ unsigned s_move[2], s_min_excl;
    __shared__ uint16_t s_queue[kQueueRounds * kFitThreads];            // samples to scan: place in the batch, bit 15 = by list
    __shared__ int s_queued[2];
    __shared__ double s_err[kFitThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, blocks = (int)gridDim.x;
    const int64_t chunks = (m + 31) / 32, chunk0 = (int64_t)warp * blocks + blockIdx.x, chunk_step = (int64_t)blocks * (kFitThreads / 32);

    for (int i = tid; i < n * P; i += kFitThreads) {
        sc[i] = samples[i];
        sums[i] = 0;
        if (shared_sums) d_lo[i] = d_hi[i] = 0u;
    }
    for (int i = tid; i < n; i += kFitThreads) {
        cnt[i] = 0;
        if (shared_sums) d_cnt[i] = 0;
    }
    if (tid < 2) s_move[tid] = 0u;
    if (tid < 2) s_queued[tid] = 0;
    int qi = 0;
    const uint2 range = range_of(w, slots);
    if (range_unsuited(range, m)) {
        if (blockIdx.x == 0 && tid == 0) w.flags[2] = 1;
        return;
    }
    const int shift = sum_shift(range.x, m);
    const double scale = power_of_two(shift), unscale = power_of_two(-shift);
    int barrier_no = 0;
    unsigned seen[2] = {0u, 0u};
    bool ok;

    // scanning one sample: n steps of its lane, or ceil(n / 32) steps and a reduction of the whole warp
    const int scan_all = max(1, 9 * n / (9 * ((n + 31) / 32) + 45));
    float moved = 0.f, moved_at_build = 0.f;    // sum over the iterations of the largest movement of any centre
    bool fresh = lists && !ADAPT;               // the lists have to be (have just been) built
    int plain_left = lists && n >= 192 ? 1 : 4, plain_next = 8;         // ADAPT: plain iterations until bounds are set, and after the next futile try
    bool set_bounds = false;                    // ADAPT: this iteration scans everything and sets the bounds
    unsigned work = 0u;                         // ADAPT: this warp's scans
    double err = 0.0;
    int it = 0;
    bool done = false;
    for (; it < max_iters; ++it) {
        if (fresh) {
            // one warp per centre, the centres spread over the blocks: the largest set of at most kNear nearest centres that a
            // threshold can cut off (bisection over the bits of the squared distance)
            for (int a = warp * blocks + (int)blockIdx.x; a < n; a += blocks * (kFitThreads / 32)) {
                float x[P], d[kMaxNearCentres / 32];
#pragma unroll
                for (int k = 0; k < P; ++k) x[k] = sc[a * P + k];
#pragma unroll
                for (int j = 0; j < kMaxNearCentres / 32; ++j)
                    d[j] = 32 * j + lane < n ? centre_distance<P>(x, sc + (32 * j + lane) * P) : INFINITY;
                unsigned lo = 0u, hi = 0x7f800000u;
                for (int round = 0; round < 16; ++round) {
                    const unsigned mid = (lo + hi) >> 1;
                    int c = 0;
#pragma unroll
                    for (int j = 0; j < kMaxNearCentres / 32; ++j) c += __float_as_uint(d[j]) < mid ? 1 : 0;
                    if (__reduce_add_sync(0xffffffffu, c) <= kNear) lo = mid; else hi = mid;
                }
                int c = 0;
                unsigned out = 0x7f800000u;
#pragma unroll
                for (int j = 0; j < kMaxNearCentres / 32; ++j) {
                    const bool in = __float_as_uint(d[j]) < lo;
                    const unsigned mask = __ballot_sync(0xffffffffu, in);
                    if (in) w.near_idx[a * kNear + c + __popc(mask & ((1u << lane) - 1u))] = (uint16_t)(32 * j + lane);
                    else out = min(out, __float_as_uint(d[j]));
                    c += __popc(mask);
                }
                if (lane >= c) w.near_idx[a * kNear + lane] = (uint16_t)a;
                out = __reduce_min_sync(0xffffffffu, out);
                if (lane == 0) w.excl[a] = __fsqrt_rd(__fmul_rd(__uint_as_float(out), 0.999996f));
            }
            if (tid == 0) s_min_excl = 0x7f800000u;
            grid_barrier<RUN_OUT>(w, barrier_no, false, seen[barrier_no & 1], &ok);
            ++barrier_no;
            if (!ok) return;
            for (int i = tid; i < n * kNear / 8; i += kFitThreads)
                *reinterpret_cast<uint4*>(near_idx + (i >> 2) * kNearRow + (i & 3) * 8) = __ldcg(reinterpret_cast<const uint4*>(w.near_idx) + i);
            for (int i = tid; i < n; i += kFitThreads) {
                const float e = __ldcg(&w.excl[i]);
                old_reach[i] = __fsub_rd(excl[i], 2.f * __fsub_ru(moved, moved_at_build));
                old_moved[i] = near_moved[i];
                excl[i] = e;
                near_moved[i] = 0.f;
                atomicMin(&s_min_excl, __float_as_uint(e));
            }
            moved_at_build = moved;
            __syncthreads();
        }
        const float since_build = __fsub_ru(moved, moved_at_build);
        const int buf = it % 3;
        const bool last = it == max_iters - 1;
        long long* delta = w.delta + (size_t)buf * n * P;
        int32_t* delta_cnt = w.delta_cnt + (size_t)buf * n;
        int changed = 0;
        auto add_coord = [&](int cell, int k, long long v) {
            if (shared_sums) {                  // (two native 32-bit atomics; a 64-bit one would be a loop)
                const unsigned vl = (unsigned)v;
                const unsigned carry = atomicAdd(&d_lo[cell * P + k], vl) > ~vl ? 1u : 0u;
                atomicAdd(&d_hi[cell * P + k], (unsigned)(v >> 32) + carry);
            } else {
                atomicAdd(reinterpret_cast<unsigned long long*>(&delta[cell * P + k]), (unsigned long long)v);
            }
        };
        auto move = [&](int64_t i, const float (&x)[P], int a, int to) {
            w.assign[i] = to;
            changed = 1;
#pragma unroll
            for (int k = 0; k < P; ++k) {
                const long long v = __double2ll_rn((double)x[k] * scale);
                add_coord(to, k, v);
                if (a >= 0) add_coord(a, k, -v);
            }
            int32_t* dc = shared_sums ? d_cnt : delta_cnt;
            atomicAdd(&dc[to], 1);
            if (a >= 0) atomicAdd(&dc[a], -1);
        };
        // the outcome of a scan: the bound on every other centre, and the cell if it changed
        auto settle = [&](int64_t i, const float (&x)[P], int a, int to, float second) {
            w.lower[i] = __fadd_rd(second, lists ? near_moved[to] : moved);
            if (to != a) move(i, x, a, to);
        };
        const bool plain = ADAPT && plain_left > 0;
        if (plain) {
            for (int64_t c = chunk0; c < chunks; c += chunk_step) {
                const int64_t i = c * 32 + lane;
                if (i >= m) continue;
                float x[P], best;
#pragma unroll
                for (int k = 0; k < P; ++k) x[k] = samples[i * P + k];
                const int a = w.assign[i], to = nearest_centre<P>(x, sc, n, best);
                if (to != a) move(i, x, a, to);
                if (last) err += (double)best;
            }
        }
        for (int64_t batch = 0; !plain && batch * chunk_step < chunks; batch += kQueueRounds) {
            for (int r = 0; r < kQueueRounds; ++r) {
                const int64_t c = chunk0 + (batch + r) * chunk_step;
                if (c >= chunks) break;
                const int64_t i = c * 32 + lane;
                const bool valid = i < m;
                float x[P];
#pragma unroll
                for (int k = 0; k < P; ++k) x[k] = valid ? samples[i * P + k] : 0.f;
                const int a = valid ? w.assign[i] : 0;
                const float lower = valid ? w.lower[i] : 0.f;           // (not yet written in the first iteration, and not used)
                bool need = valid && (ADAPT ? set_bounds : a < 0), listed = false;
                float best = 0.f;
                if (valid && (ADAPT ? !set_bounds : a >= 0)) {
                    best = centre_distance<P>(x, sc + a * P);
                    const float u = __fsqrt_ru(__fmul_ru(best, 1.000004f));
                    if (lists) {
                        listed = u < 0.5f * __fsub_rd(excl[a], 2.f * since_build);
                        float bound = __fsub_rd(lower, fresh ? old_moved[a] : near_moved[a]);
                        // the new list may hold centres whose movements M has not counted: those were outside the old list
                        if (fresh) bound = fminf(bound, __fsub_rd(old_reach[a], u));
                        need = !listed || !(u < bound);
                        if (fresh && !need) w.lower[i] = bound;         // (M of the new lists starts at 0)
                    } else {
                        need = !(u < __fsub_rd(lower, moved));
                    }
                }
                const unsigned todo = __ballot_sync(0xffffffffu, need), by_list = __ballot_sync(0xffffffffu, need && listed);
                if (__popc(todo & ~by_list) >= scan_all) {
                    float b = INFINITY, s2 = INFINITY;
                    int bi = 0;
#pragma unroll 4
                    for (int q = 0; q < n; ++q) {
                        const float d = centre_distance<P>(x, sc + q * P);
                        s2 = fminf(s2, fmaxf(b, d));
                        if (d < b) { b = d; bi = q; }
                    }
                    if (need) {
                        best = b;
                        settle(i, x, a, bi, __fsqrt_rd(__fmul_rd(s2, 0.999996f)));
                    }
                    if (ADAPT) work += (unsigned)n + (unsigned)n / 4u;
                    if (last && valid) err += (double)best;
                } else {
                    if (ADAPT) work += 10u + (unsigned)__popc(by_list) * 3u + (unsigned)__popc(todo & ~by_list) * ((unsigned)n / 32u + 8u);
                    int at = 0;
                    if (lane == 0 && todo) at = atomicAdd(&s_queued[qi], __popc(todo));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (need) s_queue[at + __popc(todo & ((1u << lane) - 1u))] = (uint16_t)((r * kFitThreads + tid) | (listed ? 0x8000u : 0u));
                    if (last && valid && !need) err += (double)best;
                }
            }
            __syncthreads();
            const int queued = s_queued[qi];
            qi ^= 1;
            if (tid == 0) s_queued[qi] = 0;            // (every thread has read it before this barrier)
            auto sample_of = [&](unsigned place) {
                return ((int64_t)((place >> 5) & 31) * blocks + blockIdx.x + (batch + place / kFitThreads) * chunk_step) * 32 + (place & 31);
            };
            const bool by_lane = queued > kLaneScans;
            if (by_lane) {
                for (int e = tid; e < queued; e += kFitThreads) {
                    const unsigned entry = s_queue[e];
                    if (!(entry & 0x8000u)) continue;
                    const int64_t i = sample_of(entry & 0x7fffu);
                    float x[P];
#pragma unroll
                    for (int k = 0; k < P; ++k) x[k] = samples[i * P + k];
                    const int a = w.assign[i];
                    const float u = __fsqrt_ru(__fmul_ru(centre_distance<P>(x, sc + a * P), 1.000004f));
                    float b = INFINITY, s2 = INFINITY;
                    int bi = 0;
#pragma unroll
                    for (int g = 0; g < kNear / 8; ++g) {
                        const uint4 idx = *reinterpret_cast<const uint4*>(near_idx + a * kNearRow + g * 8);
                        const unsigned v[4] = {idx.x, idx.y, idx.z, idx.w};
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const int q = (int)((v[k >> 1] >> (16 * (k & 1))) & 0xffffu);
                            const float d = centre_distance<P>(x, sc + q * P);
                            if (q != bi || b == INFINITY) s2 = fminf(s2, fmaxf(b, d));      // (the padding repeats the cell itself)
                            if (d < b || (d == b && q < bi)) { b = d; bi = q; }
                        }
                    }
                    settle(i, x, a, bi, fminf(__fsqrt_rd(__fmul_rd(s2, 0.999996f)), __fsub_rd(__fsub_rd(excl[a], 2.f * since_build), u)));
                    if (last) err += (double)b;
                }
            }
            for (int e = warp; e < queued; e += kFitThreads / 32) {
                const unsigned entry = s_queue[e];
                const bool listed = (entry & 0x8000u) != 0;
                if (listed && by_lane) continue;
                const int64_t i = sample_of(entry & 0x7fffu);
                float y[P];
#pragma unroll
                for (int k = 0; k < P; ++k) y[k] = samples[i * P + k];
                const int a = w.assign[i];
                float b = INFINITY, s2 = INFINITY, beyond = INFINITY;       // beyond: a bound on the distance to centres outside the list
                int bi = 0x7fffffff;
                if (listed) {
                    bi = near_idx[a * kNearRow + lane];
                    b = centre_distance<P>(y, sc + bi * P);
                    beyond = __fsub_rd(__fsub_rd(excl[a], 2.f * since_build), __fsqrt_ru(__fmul_ru(centre_distance<P>(y, sc + a * P), 1.000004f)));
                } else {
#pragma unroll 4
                    for (int q = lane; q < n; q += 32) {
                        const float d = centre_distance<P>(y, sc + q * P);
                        s2 = fminf(s2, fmaxf(b, d));
                        if (d < b) { b = d; bi = q; }
                    }
                }
                const unsigned wb = __reduce_min_sync(0xffffffffu, __float_as_uint(b));        // (not negative: ordered as integers)
                int to = (int)__reduce_min_sync(0xffffffffu, __float_as_uint(b) == wb ? (unsigned)bi : 0x7fffffffu);
                if (to >= n) to = 0;               // no distance compared below infinity (NaN, or squares that overflow): index 0, as a plain scan
                const unsigned ws = __reduce_min_sync(0xffffffffu, __float_as_uint(bi == to ? s2 : b));
                if (lane == 0) {
                    settle(i, y, a, to, fminf(__fsqrt_rd(__fmul_rd(__uint_as_float(ws), 0.999996f)), beyond));
                    if (last) err += (double)__uint_as_float(wb);
                }
            }
            if ((batch + kQueueRounds) * chunk_step < chunks) __syncthreads();      // (the queue is written again)
        }
        if (ADAPT && !plain) {
            if (lane == 0) atomicAdd(&w.work[buf], (unsigned long long)work);
            work = 0u;
        }
        const bool block_changed = __syncthreads_or(changed) != 0;
        if (shared_sums && block_changed) {
            for (int q = tid; q < n * P; q += kFitThreads) {
                const unsigned long long v = (unsigned long long)d_lo[q] | ((unsigned long long)d_hi[q] << 32);
                if (v) { atomicAdd(reinterpret_cast<unsigned long long*>(&delta[q]), v); d_lo[q] = d_hi[q] = 0u; }
            }
            for (int q = tid; q < n; q += kFitThreads)
                if (d_cnt[q]) { atomicAdd(&delta_cnt[q], d_cnt[q]); d_cnt[q] = 0; }
        }
        const bool any = grid_barrier<RUN_OUT>(w, barrier_no, block_changed, seen[barrier_no & 1], &ok);
        ++barrier_no;
        if (!ok) return;
        if (!any) { done = true; ++it; break; }          // no assignment changed: a fixed point
        for (int q = tid; q < n; q += kFitThreads) {
            const int size = cnt[q] + __ldcg(&delta_cnt[q]);
            cnt[q] = size;
            float go2 = 0.f;
#pragma unroll
            for (int k = 0; k < P; ++k) {
                const long long s = sums[q * P + k] + __ldcg(&delta[q * P + k]);
                sums[q * P + k] = s;
                if (size > 0) {                                                 // (an empty cell keeps its centre)
                    const float c = (float)((double)s * unscale / (double)size), go = c - sc[q * P + k];
                    sc[q * P + k] = c;
                    go2 = __fmaf_ru(go, go, go2);
                }
            }
            const float step = go2 > 0.f ? __fmul_ru(__fsqrt_ru(go2), 1.000001f) : 0.f;
            if (step > 0.f) atomicMax(&s_move[it & 1], __float_as_uint(step));
            if (lists) went[q] = step;
        }
        if (blockIdx.x == 0) {
            const int old = (it + 2) % 3;
            for (int i = tid; i < n * P; i += kFitThreads) w.delta[(size_t)old * n * P + i] = 0;
            for (int i = tid; i < n; i += kFitThreads) w.delta_cnt[(size_t)old * n + i] = 0;
            if (ADAPT && tid == 0) w.work[old] = 0;
        }
        __syncthreads();
        moved = __fadd_ru(moved, __uint_as_float(s_move[it & 1]));
        if (tid == 0) s_move[(it + 1) & 1] = 0u;       // (last read before the barrier of this iteration)
        if (ADAPT) {
            const bool tried = !plain && !set_bounds;
            set_bounds = plain && --plain_left == 0;
            if (tried && __ldcg(&w.work[buf]) * 20 > (unsigned long long)chunks * (unsigned)n * 17) {
                plain_left = plain_next;
                plain_next = min(2 * plain_next, 64);
            }
        }
        if (ADAPT && (plain || plain_left > 0)) {
            fresh = lists && set_bounds;
        } else if (lists) {
            fresh = __fsub_ru(moved, moved_at_build) > 0.15f * __uint_as_float(s_min_excl);
            // four threads per cell: the largest movement among its list
            for (int q = tid; q < ((4 * n + 31) & ~31); q += kFitThreads) {
                const int a = min(q >> 2, n - 1);
                const uint4 idx = *reinterpret_cast<const uint4*>(near_idx + a * kNearRow + (q & 3) * 8);
                const unsigned v[4] = {idx.x, idx.y, idx.z, idx.w};
                float far = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) far = fmaxf(far, fmaxf(went[v[k] & 0xffffu], went[v[k] >> 16]));
                far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, 1));
                far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, 2));
                if (q < 4 * n && (q & 3) == 0) near_moved[a] = __fadd_ru(near_moved[a], far);
            }
            __syncthreads();
        }
    }
    if (done && it < max_iters) {                       // (otherwise the last assignment step has added the errors up)
        for (int64_t c = chunk0; c < chunks; c += chunk_step) {
            const int64_t i = c * 32 + lane;
            if (i >= m) continue;
            float x[P];
#pragma unroll
            for (int k = 0; k < P; ++k) x[k] = samples[i * P + k];
            err += (double)centre_distance<P>(x, sc + w.assign[i] * P);
        }
    }
    write_result(w, sc, n * P, err, done, it, s_err);
}

__global__ void __launch_bounds__(256) grid_finalize_kernel(GridWs w, int p, int n, int64_t m, int fit_blocks, int plain_blocks, float* __restrict__ grid_out,
                                                            float* __restrict__ mse_out, int32_t* __restrict__ iters_out) {
    // lexicographic sort by rank counting, one warp per centre (coordinate 0 first; equal points keep their index order)
    const int lane = threadIdx.x & 31, c = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (c < n) {
        int rank = 0;
        for (int o = lane; o < n; o += 32) {
            int cmp = 0;                                   // sign of (centre o) - (centre c)
            for (int k = 0; k < p && cmp == 0; ++k) {
                const float a = w.centres[c * p + k], b = w.centres[o * p + k];
                cmp = b < a ? -1 : (b > a ? 1 : 0);
            }
            rank += (cmp < 0 || (cmp == 0 && o < c)) ? 1 : 0;
        }
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (lane < p) grid_out[rank * p + lane] = w.centres[c * p + lane];
    }
    if (c == 0) {
        const int blocks = w.flags[2] ? plain_blocks : fit_blocks;
        double e = 0.0;
        for (int i = lane; i < blocks; i += 32) e += w.err[i];
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) e += __shfl_xor_sync(0xffffffffu, e, k);
        if (lane == 0) {
            const bool ran_out = w.flags[3] != 0;
            if (mse_out) *mse_out = ran_out ? NAN : (float)(e / ((double)m * p));
            if (iters_out) *iters_out = ran_out ? -1 : w.flags[0] ? w.flags[1] : -w.flags[1];
        }
    }
}

// ---- constrained (uniform) grid, Section 4.3 "Constrained HIGGS" ------------------------------------------
// n equally spaced levels (k - (n-1)/2) * step, symmetric about 0 (the Gaussian is); the step minimises the expected
// squared error of rounding N(0,1):  MSE(step) = sum over cells of  M2 - 2 c M1 + c^2 P  with the cell's probability
// P, first moment M1 = phi(a) - phi(b) and second moment M2 = P + a phi(a) - b phi(b)  (a, b the cell's thresholds,
// the outer cells unbounded).  One block; thread i owns cell i; golden-section search on the step in fp64.
__device__ __forceinline__ double d_phi(double x) { return 0.3989422804014327 * exp(-0.5 * x * x); }
__device__ __forceinline__ double d_Phi(double x) { return 0.5 * erfc(-x * 0.7071067811865476); }

__device__ double uniform_mse_block(int n, double step, double* red) {
    double term = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double c = ((double)i - 0.5 * (double)(n - 1)) * step;
        const bool lo_inf = i == 0, hi_inf = i == n - 1;
        const double a = c - 0.5 * step, b = c + 0.5 * step;
        const double Pa = lo_inf ? 0.0 : d_Phi(a), Pb = hi_inf ? 1.0 : d_Phi(b);
        const double fa = lo_inf ? 0.0 : d_phi(a), fb = hi_inf ? 0.0 : d_phi(b);
        const double P = Pb - Pa, M1 = fa - fb, M2 = P + (lo_inf ? 0.0 : a * fa) - (hi_inf ? 0.0 : b * fb);
        term += M2 - 2.0 * c * M1 + c * c * P;
    }
    red[threadIdx.x] = term;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    const double v = red[0];
    __syncthreads();
    return v;
}

__global__ void __launch_bounds__(256) uniform_grid_kernel(int n, float* __restrict__ grid_out, float* __restrict__ step_out,
                                                           float* __restrict__ mse_out) {
    __shared__ double red[256];
    double lo = 1e-4, hi = 8.0 / n + 2.0;
    const double r = 0.6180339887498949;
    double a = hi - r * (hi - lo), b = lo + r * (hi - lo);
    double fa = uniform_mse_block(n, a, red), fb = uniform_mse_block(n, b, red);
    for (int it = 0; it < 120; ++it) {         // every thread follows the same path: the values are block-uniform
        if (fa < fb) {
            hi = b; b = a; fb = fa;
            a = hi - r * (hi - lo);
            fa = uniform_mse_block(n, a, red);
        } else {
            lo = a; a = b; fa = fb;
            b = lo + r * (hi - lo);
            fb = uniform_mse_block(n, b, red);
        }
    }
    const double step = 0.5 * (lo + hi);
    const double mse = uniform_mse_block(n, step, red);
    for (int i = threadIdx.x; i < n; i += blockDim.x) grid_out[i] = (float)(((double)i - 0.5 * (double)(n - 1)) * step);
    if (threadIdx.x == 0) {
        if (step_out) *step_out = (float)step;
        if (mse_out) *mse_out = (float)mse;
    }
}

}  // namespace

int launch_uniform_grid(int n, float* grid_out, float* step_out, float* mse_out, cudaStream_t st) {
    uniform_grid_kernel<<<1, 256, 0, st>>>(n, grid_out, step_out, mse_out);
    return cuda_status(cudaGetLastError());
}

size_t make_grid_workspace(int p, int n, int64_t m) {
    return up256(sizeof(float) * n * p) + up256(sizeof(long long) * 3 * n * p) + up256(sizeof(int32_t) * 3 * n) +
           up256(sizeof(double) * kMaxFitBlocks) + 256 + (sizeof(uint16_t) * kNear + sizeof(float)) * kMaxNearCentres +
           up256(sizeof(int32_t) * (size_t)m) + up256(sizeof(float) * (size_t)m);
}

static int sm_count_of_device() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) v = 1;
    return v;
}

// One cooperative launch for the whole iteration, a block per SM (fewer when there are fewer than 32 samples for each).  Where fewer
// are resident (a context that owns a part of the SMs), half as many are tried until they are; the last resort is one ordinary
// block, whose barriers are trivial.
template <typename... Args>
static int launch_resident(void (*kernel)(Args...), int* blocks, size_t smem, cudaStream_t st, Args... args) {
    void* ptrs[] = {&args...};
    for (; *blocks > 1; *blocks /= 2) {
        if (cudaLaunchCooperativeKernel((const void*)kernel, dim3((unsigned)*blocks), dim3(kFitThreads), ptrs, smem, st) == cudaSuccess) return HIGGS_OK;
        (void)cudaGetLastError();
    }
    kernel<<<1, kFitThreads, smem, st>>>(args...);
    return cuda_status(cudaGetLastError());
}

template <int P, bool RUN_OUT, bool ADAPT>
static int launch_fit(GridWs w, const float* samples, int n, int64_t m, int slots, int max_iters, int crowd, int (&blocks_out)[2], cudaStream_t st) {
    constexpr size_t kMaxSmem = (P * (sizeof(long long) + sizeof(float)) + sizeof(int)) * kMaxGridPoints;     // (n = 4096: no lists)
    static int state[64] = {0};           // 1 = cooperative launch possible, 2 = not, -1 = failed
    const int how = device_once(state, [] {
        int dev = 0, coop = 0, v = 0;
        if (cudaFuncSetAttribute(grid_fit_kernel<P, RUN_OUT, ADAPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxSmem > 73728 ? kMaxSmem : 73728)) != cudaSuccess ||
            cudaFuncSetAttribute(plain_fit_kernel<P, RUN_OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess)
            return -1;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, grid_fit_kernel<P, RUN_OUT, ADAPT>, kFitThreads, kMaxSmem) != cudaSuccess || v < 1)
            return 2;
        return 1;
    });
    if (how < 0) return HIGGS_ERR_CUDA;
    int64_t blocks = how == 1 ? (m + 31) / 32 : 1;
    if (blocks > sm_count_of_device()) blocks = sm_count_of_device();
    if (blocks > kMaxFitBlocks) blocks = kMaxFitBlocks;
    blocks_out[0] = blocks_out[1] = (int)blocks * crowd;
    const int rc = launch_resident(grid_fit_kernel<P, RUN_OUT, ADAPT>, &blocks_out[0], fit_smem(P, n), st, w, samples, n, m, slots, max_iters);
    if (rc != HIGGS_OK) return rc;
    return launch_resident(plain_fit_kernel<P, RUN_OUT>, &blocks_out[1], (size_t)n * (P * (sizeof(double) + sizeof(float)) + sizeof(int)), st, w, samples, n, m, max_iters);
}

int launch_make_grid(int p, int n, const float* samples, int64_t m, int max_iters, float* grid_out, float* mse_out,
                     int32_t* iters_out, void* ws, cudaStream_t st, FitTest test) {
    GridWs w = carve(ws, p, n, m);
    const int64_t most = (m + kRangeThreads - 1) / kRangeThreads;
    const int slots = (int)(most < kMaxFitBlocks ? most : kMaxFitBlocks);
    grid_init_kernel<<<(unsigned)slots, kRangeThreads, 0, st>>>(w, samples, p, n, m);
    grid_range_kernel<<<(unsigned)slots, kRangeThreads, 0, st>>>(w, samples, p, m, slots);
    int blocks[2] = {0, 0}, rc = HIGGS_ERR_UNSUPPORTED;
    const int crowd = test == FitTest::kTooManyBlocks ? 4 : 1;
    switch (4 * p + (test == FitTest::kRunOut ? 1 : test == FitTest::kAdapt || m >= kAdaptSamples ? 2 : 0)) {
        case 4: rc = launch_fit<1, false, false>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 5: rc = launch_fit<1, true, false>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 6: rc = launch_fit<1, false, true>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 8: rc = launch_fit<2, false, false>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 9: rc = launch_fit<2, true, false>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 10: rc = launch_fit<2, false, true>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 12: rc = launch_fit<3, false, false>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 14: rc = launch_fit<3, false, true>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 16: rc = launch_fit<4, false, false>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
        case 18: rc = launch_fit<4, false, true>(w, samples, n, m, slots, max_iters, crowd, blocks, st); break;
    }
    if (rc != HIGGS_OK) return rc;
    grid_finalize_kernel<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(w, p, n, m, blocks[0], blocks[1], grid_out, mse_out, iters_out);
    return cuda_status(cudaGetLastError());
}

int read_grid_status(int clear) {
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_grid_status, sizeof(int)) != cudaSuccess) return HIGGS_ERR_CUDA;
    if (clear && v != 0) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_grid_status, &zero, sizeof(int)) != cudaSuccess) return HIGGS_ERR_CUDA;
    }
    return v;
}

}  // namespace higgs
