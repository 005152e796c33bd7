// Dequantisation to the original space (Appendix F, "Dequantization"): for every (row, group)
//   r = scale * G[codes]  (the layer in the rotated space),   w^ = diag(sign) (H / sqrt(g)) r,
// and the layer's relative error t^2 (Section 5, "Measuring Grid Parameters").  Both read the packed stream directly.
#include "common.cuh"

namespace higgs {

namespace {

constexpr int kDqWarps = 8;            // a block takes one row tile (16 rows) x one group per turn; warp w rows w and w + 8

// The table indices of rows w (low halves) and w + 8 of one (row tile, group), as this lane needs them after
// fwht1024_to_columns: lane c*8 + e holds elements c*256 + j*8 + e, j = 0..31, i.e. pair (e >> 1) of every second
// 4-pair step of the 64-input blocks 4c .. 4c + 3.  In every packed format the indices of one such pair position for
// the two rows are one contiguous run of packed lane L = 4 w + (e >> 1): the lanes of a warp read whole 64-byte runs.
template <int FMT>
struct ColumnCodes {
    static constexpr bool SIX = FMT == 1, NIB = FMT == 2, B8 = FMT == 3;
    uint32_t w[SIX ? 12 : NIB ? 8 : B8 ? 32 : 16];
    __device__ __forceinline__ void load(const uint8_t* __restrict__ packed, int64_t first_block, int warp, int lane) {
        const int c = lane >> 3, L = warp * 4 + ((lane & 7) >> 1);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int64_t blk = first_block + 4 * c + jj;
            if (SIX) {
                if (jj & 1) continue;                                    // a super-block covers blocks jj and jj + 1
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) {
                    const uint2 q = __ldg(reinterpret_cast<const uint2*>(packed + (blk >> 1) * 768 + pl * 256 + L * 8));
                    w[jj * 3 + pl] = q.x;
                    w[jj * 3 + 3 + pl] = q.y;
                }
            } else if (NIB) {
                const uint2 q = __ldg(reinterpret_cast<const uint2*>(packed + blk * 256 + L * 8));
                w[jj * 2] = q.x; w[jj * 2 + 1] = q.y;
            } else {
#pragma unroll
                for (int h = 0; h < (B8 ? 2 : 1); ++h) {
                    const uint4 q = __ldg(reinterpret_cast<const uint4*>(packed + blk * (B8 ? 1024 : 512) + h * 512 + L * 16));
                    uint32_t* o = w + jj * (B8 ? 8 : 4) + h * 4;
                    o[0] = q.x; o[1] = q.y; o[2] = q.z; o[3] = q.w;
                }
            }
        }
    }
    // table row of element j (jj = j >> 3, m = (j & 7) >> 1, ah = j & 1) for row half rh; see the slot layout in quantize.cu
    __device__ __forceinline__ uint32_t index(int j, int rh, int lane) const {
        const int jj = j >> 3, m = (j & 7) >> 1, ah = j & 1, a = rh + 2 * ah;
        if (SIX) {
            const uint32_t lo = (w[jj * 3 + (m >> 1)] >> (8 * a + 4 * (m & 1))) & 15u;
            return lo | (((w[jj * 3 + 2] >> (8 * a + 2 * m)) & 3u) << 4);
        }
        if (NIB) return (w[jj * 2 + ((j & 7) >> 2)] >> (8 * (j & 3) + 4 * rh)) & 15u;
        if (B8) return (w[jj * 8 + (j & 7)] >> (16 * rh + 8 * (lane & 1))) & 255u;
        return (w[jj * 4 + m] >> (8 * a)) & 255u;
    }
};

// Lookup table in shared memory: row idx holds, 16 times over, the two coordinates an index stands for (one p = 2 code
// or two p = 1 codes; 8-bit scalar codes: the value, twice), so that lane l reads word l of its row - the coordinate of
// its parity - and the 32 lookups of a warp never meet in a bank.
template <int FMT>
__device__ __forceinline__ void fill_pair_table(float* table, const float* __restrict__ grid, int p, int n, int bits) {
    constexpr int ROWS = FMT == 1 ? 64 : FMT == 2 ? 16 : 256;
    for (int i = threadIdx.x; i < ROWS * 32; i += blockDim.x) {
        const int idx = i >> 5, k = i & 1;
        table[i] = FMT == 3 ? grid[idx] : p == 2 ? grid[2 * idx + k] : grid[(idx >> (k * bits)) & (n - 1)];
    }
}

template <typename OutT>
__device__ __forceinline__ void store_row(OutT* __restrict__ dst, int lane, const float (&v)[32]);
template <>
__device__ __forceinline__ void store_row<float>(float* __restrict__ dst, int lane, const float (&v)[32]) {
#pragma unroll
    for (int c = 0; c < 8; ++c)
        *reinterpret_cast<float4*>(dst + (c >> 1) * 256 + lane * 8 + (c & 1) * 4) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
}
template <>
__device__ __forceinline__ void store_row<__nv_bfloat16>(__nv_bfloat16* __restrict__ dst, int lane, const float (&v)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t w4[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[c * 8 + 2 * e], v[c * 8 + 2 * e + 1]);
            w4[e] = *reinterpret_cast<const uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(dst + c * 256 + lane * 8) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
    }
}

// ERROR = false: W_out[row][k] = the dequantised matrix.  ERROR = true: the two sums of t^2 = ||W^ - W||^2 / ||W||^2,
// taken in the rotated space (the transform is orthonormal): W is rotated as the encoder rotates it and compared with
// scale * G[code].  A block writes its pair of partial sums; launch_layer_error's second kernel adds them in block order.
// Bound: instruction issue (75-79 % of the slots with scalar arithmetic, 810 instructions per row and group of which 360 the
// transform; most of it works on fp32 pairs now), next to 2 or 4 + b/8 bytes per weight from HBM.  14336 x 4096 bf16 at 4 bits: error
// 185 + 47 us (canonical codes unpacked to memory byte by byte, then one warp per row and group adding to two global
// doubles) -> 63 -> 57 us with pairs (3 bits 68 -> 60), dequantised 56 -> 52; the 147 MB it reads take 22 us.
template <int FMT, typename T, bool ERROR>
__global__ void __launch_bounds__(kDqWarps * 32, 2) packed_rows_kernel(const uint8_t* __restrict__ packed, const __half* __restrict__ scales,
                                                                       const float* __restrict__ grid, int p, int n, int bits,
                                                                       const T* __restrict__ W, T* __restrict__ W_out, int64_t N,
                                                                       int64_t K, uint64_t xi, double* __restrict__ partials) {
    extern __shared__ __align__(16) float dq_smem[];
    constexpr int ROWS = FMT == 1 ? 64 : FMT == 2 ? 16 : 256;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* ex = dq_smem + ROWS * 32 + warp * kFwhtExchange;
    if (ERROR) pdl_trigger();          // (the kernel that adds the partial sums waits for this one's end on the SM)
    fill_pair_table<FMT>(dq_smem, grid, p, n, bits);
    __syncthreads();
    const float* table_lane = dq_smem + lane;
    const int64_t groups = K / kGroup, kblocks = K / kBlockK, turns = (N / kRowTile) * groups;
    int64_t rt = (int64_t)blockIdx.x / groups, gi = (int64_t)blockIdx.x % groups;
    const int64_t step_tiles = (int64_t)gridDim.x / groups, step_groups = (int64_t)gridDim.x % groups;
    double num = 0.0, den = 0.0;
    for (int64_t turn = blockIdx.x; turn < turns; turn += gridDim.x, rt += step_tiles, gi += step_groups) {
        if (gi >= groups) { gi -= groups; ++rt; }
        ColumnCodes<FMT> codes;
        codes.load(packed, rt * kblocks + gi * 16, warp, lane);
        const __half* sc = scales + (rt * groups + gi) * kRowTile + warp;
        const float scale[2] = {__half2float(sc[0]), __half2float(sc[8])};
        const uint32_t sign = lane_sign_bits(xi, gi * kGroup, lane);
        RawGroup<T> raw[2];
        if (ERROR) {
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) raw[rh].load(W + (rt * 16 + warp + 8 * rh) * K + gi * kGroup, lane);
        }
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            float v[32];
            if (ERROR) {
                uint64_t dsum2 = pair_of(0.f, 0.f), nsum2 = dsum2;
#pragma unroll
                for (int t = 0; t < 16; ++t) {
                    raw[rh].get_signed(t, sign, v[2 * t], v[2 * t + 1]);
                    const uint64_t x = pair_of(v[2 * t], v[2 * t + 1]);
                    dsum2 = fma2(x, x, dsum2);
                }
                fwht1024_to_columns(v, ex, lane);
                const uint64_t scale2 = pair_of(scale[rh], scale[rh]), to_unit = pair_of(-0.03125f, -0.03125f);
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    const uint64_t g = pair_of(table_lane[codes.index(j, rh, lane) * 32], table_lane[codes.index(j + 1, rh, lane) * 32]);
                    const uint64_t d = fma2(scale2, g, mul2(pair_of(v[j], v[j + 1]), to_unit));
                    nsum2 = fma2(d, d, nsum2);
                }
                float dsum, nsum, odd;
                unpair(dsum2, dsum, odd);
                dsum += odd;
                unpair(nsum2, nsum, odd);
                nsum += odd;
#pragma unroll
                for (int m = 16; m > 0; m >>= 1) {
                    nsum += __shfl_xor_sync(0xffffffffu, nsum, m);
                    dsum += __shfl_xor_sync(0xffffffffu, dsum, m);
                }
                num += (double)nsum;
                den += (double)dsum;
            } else {
                const float s = scale[rh] * 0.03125f;          // H / sqrt(1024)
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = s * table_lane[codes.index(j, rh, lane) * 32];
                fwht1024_from_columns(v, ex, lane);
#pragma unroll
                for (int r = 0; r < 32; ++r) v[r] = with_sign(v[r], sign, r);
                store_row<T>(W_out + (rt * 16 + warp + 8 * rh) * K + gi * kGroup, lane, v);
            }
        }
    }
    if (ERROR) {
        __syncthreads();                                       // (the table and exchange buffers are free: reuse them)
        double* red = reinterpret_cast<double*>(dq_smem);
        if (lane == 0) { red[2 * warp] = num; red[2 * warp + 1] = den; }
        __syncthreads();
        if (threadIdx.x < 2) {
            double s = 0.0;
            for (int w = 0; w < kDqWarps; ++w) s += red[2 * w + threadIdx.x];
            partials[2 * blockIdx.x + threadIdx.x] = s;
        }
    }
}

__global__ void __launch_bounds__(64) error_total_kernel(const double* partials, int blocks, double* __restrict__ sums) {
    __shared__ double total[2];
    const int which = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
    pdl_wait();
    for (int i = lane; i < blocks; i += 32) s += __ldcg(&partials[2 * i + which]);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    if (lane == 0) { total[which] = s; sums[which] = s; }
    __syncthreads();
    if (threadIdx.x == 0) sums[2] = total[1] > 0.0 ? total[0] / total[1] : 0.0;
}

int sm_count() {
    static int cached[64] = {0};
    return device_once(cached, [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0)
            v = 148;
        return v;
    });
}

template <int FMT, typename T, bool ERROR>
int launch_rows(const higgs_desc& d, const void* packed, const void* scales, const float* grid, const void* W, void* W_out,
                double* partials, int* blocks_out, cudaStream_t st) {
    constexpr int ROWS = FMT == 1 ? 64 : FMT == 2 ? 16 : 256;
    constexpr int smem = (ROWS * 32 + kDqWarps * kFwhtExchange) * (int)sizeof(float);
    static int per_sm[64] = {0};
    const int resident = device_once(per_sm, [] {
        int b = 0;
        if (cudaFuncSetAttribute(packed_rows_kernel<FMT, T, ERROR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, packed_rows_kernel<FMT, T, ERROR>, kDqWarps * 32, smem) != cudaSuccess || b < 1)
            return -1;
        return b;
    });
    if (resident < 1) return HIGGS_ERR_CUDA;
    const int64_t turns = (d.N / kRowTile) * (d.K / kGroup);
    int64_t blocks = (int64_t)resident * sm_count();
    if (ERROR && blocks > kErrorPartials) blocks = kErrorPartials;
    if (blocks > turns) blocks = turns;
    if (blocks_out) *blocks_out = (int)blocks;
    packed_rows_kernel<FMT, T, ERROR><<<(unsigned)blocks, kDqWarps * 32, smem, st>>>(
        static_cast<const uint8_t*>(packed), static_cast<const __half*>(scales), grid, d.p, d.n, code_bits(d.n), static_cast<const T*>(W),
        static_cast<T*>(W_out), d.N, d.K, d.rht_seed, partials);
    return cuda_status(cudaGetLastError());
}

template <typename T, bool ERROR>
int launch_format(const higgs_desc& d, const void* packed, const void* scales, const float* grid, const void* W, void* W_out,
                  double* partials, int* blocks, cudaStream_t st) {
    switch (format_of(d.p, d.n)) {
        case Format::kByteLut: return launch_rows<0, T, ERROR>(d, packed, scales, grid, W, W_out, partials, blocks, st);
        case Format::kSixBit: return launch_rows<1, T, ERROR>(d, packed, scales, grid, W, W_out, partials, blocks, st);
        case Format::kNibble: return launch_rows<2, T, ERROR>(d, packed, scales, grid, W, W_out, partials, blocks, st);
        case Format::kByte8: return launch_rows<3, T, ERROR>(d, packed, scales, grid, W, W_out, partials, blocks, st);
        default: return HIGGS_ERR_UNSUPPORTED;
    }
}

}  // namespace

int launch_layer_error(const higgs_desc& d, const void* packed, const void* scales, const float* grid, const void* W,
                       int w_dtype, double* sums, double* partials, cudaStream_t st) {
    int blocks = 0;
    const int rc = w_dtype == HIGGS_F32 ? launch_format<float, true>(d, packed, scales, grid, W, nullptr, partials, &blocks, st)
                                        : launch_format<__nv_bfloat16, true>(d, packed, scales, grid, W, nullptr, partials, &blocks, st);
    if (rc != HIGGS_OK) return rc;
    return cuda_status(launch_pdl(error_total_kernel, dim3(1), dim3(64), 0, st, static_cast<const double*>(partials), blocks, sums));
}

int launch_dequantize(const higgs_desc& d, const void* packed, const void* scales, const float* grid, void* W_out,
                      int w_dtype, cudaStream_t st) {
    return w_dtype == HIGGS_F32 ? launch_format<float, false>(d, packed, scales, grid, nullptr, W_out, nullptr, nullptr, st)
                                : launch_format<__nv_bfloat16, false>(d, packed, scales, grid, nullptr, W_out, nullptr, nullptr, st);
}

}  // namespace higgs
