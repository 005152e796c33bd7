// Randomised Hadamard transform kernels (Algorithm 1's RandomHadamardTransform and
// Appendix F's rotation of the activations).
#include "common.cuh"

namespace higgs {

namespace {

// Loads the 32 values of this lane (see fwht1024_warp for the mapping) from a
// row-major source of bf16 or fp32.
template <typename T>
__device__ __forceinline__ void load_group(const T* __restrict__ src, int lane, float (&v)[32]);

template <>
__device__ __forceinline__ void load_group<__nv_bfloat16>(const __nv_bfloat16* __restrict__ src, int lane,
                                                          float (&v)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint4 q = __ldg(reinterpret_cast<const uint4*>(src + c * 256 + lane * 8));
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[c * 8 + 2 * e] = __uint_as_float(w[e] << 16);
            v[c * 8 + 2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
        }
    }
}

template <>
__device__ __forceinline__ void load_group<float>(const float* __restrict__ src, int lane, float (&v)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float4 a = __ldg(reinterpret_cast<const float4*>(src + c * 256 + lane * 8));
        float4 b = __ldg(reinterpret_cast<const float4*>(src + c * 256 + lane * 8 + 4));
        v[c * 8 + 0] = a.x; v[c * 8 + 1] = a.y; v[c * 8 + 2] = a.z; v[c * 8 + 3] = a.w;
        v[c * 8 + 4] = b.x; v[c * 8 + 5] = b.y; v[c * 8 + 6] = b.z; v[c * 8 + 7] = b.w;
    }
}

// x+ = (H/32) diag(sign) x, written as fp16 in "fragment order": inside every block of 64 inputs the 32 input pairs are
// permuted so that the eight pairs one lane of the product kernel needs as m16n8k16 B-fragment registers (steps
// m = 0..3, halves h = 0..1 of its column pair t) are 32 contiguous bytes: position t*8 + m*2 + h holds pair 8m + t + 4h.
//
// One warp per (token, group), one block each.  The transform stands between two dependent product launches, so what
// counts is when it can start: a product kernel leaves shared memory (kRotationReserve) and registers for a few of
// these small blocks, which are therefore on the SMs and waiting - code fetched, signs computed - when the product
// before them ends; the next product's blocks take the SMs over as they become free, and build their tables and fetch
// their first weights while the rotation runs.  As blocks of four warps, which found no room, it added 4.4 us to a
// 4096 x 4096 product with four tokens (8.8 against 4.3 us on rotated activations); now 1.3.
// Lane l reads inputs 32 l .. + 31: bits 0 to 4 of the input index are butterflies in registers (two fp32 operations
// an instruction), bit 5 is a shuffle; the pairs are then exchanged through shared memory, 2 KB at a time, so that
// lane P holds pair P of the sixteen 64-input blocks and bits 6 to 9 are in registers too.  (The same sums, bit for
// bit, as the rotation fused into the product kernel.)
// Threads also clear `zero_ptr` (the fp32 accumulation target of a K-split product) so that no separate memset launch
// is needed.
__global__ void __launch_bounds__(32) rht_activations_kernel(const __nv_bfloat16* x, __half* __restrict__ xdag,
                                                             int64_t B, int64_t K, uint64_t xi,
                                                             float* __restrict__ zero_ptr, size_t zero_floats) {
    __shared__ __align__(16) uint8_t ex[2048];
    const int lane = threadIdx.x;
    const int64_t groups = K / kGroup;
    pdl_trigger();     // the product kernel may start its table build and weight prefetch now
    const int64_t b = blockIdx.x / groups, k0 = blockIdx.x % groups * kGroup;
    const uint64_t word = sign_word(xi, ((uint64_t)k0 >> 6) + (uint64_t)(lane >> 1));
    const uint32_t signs = (uint32_t)(word >> (32 * (lane & 1)));
    const __nv_bfloat16* src = x + b * K + k0 + lane * 32;
    if (b < B) {       // into L2 already now: a line the previous kernel is still going to write is written there
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src + 16));
    }
    pdl_wait();        // x may be the previous kernel's output; the buffers written below may still be read by it
    for (size_t i = (size_t)blockIdx.x * 32 + lane; i < zero_floats; i += (size_t)gridDim.x * 32) zero_ptr[i] = 0.0f;
    if (b >= B) return;                                      // (blocks beyond the transform work only clear)
    uint64_t q[16];
    {
        uint4 raw[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) raw[c] = __ldcg(reinterpret_cast<const uint4*>(src) + c);
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const uint4 r = raw[t >> 2];
            uint32_t w = (t & 3) == 0 ? r.x : (t & 3) == 1 ? r.y : (t & 3) == 2 ? r.z : r.w;
            // the signs of elements 2t, 2t + 1: one multiply puts both bits on the two sign positions
            w ^= (((signs >> (8 * (t >> 2))) & 0xffu) * ((1u << (15 - 2 * (t & 3))) + (1u << (30 - 2 * (t & 3))))) & 0x80008000u;
            const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xffff0000u);
            q[t] = pair_of(lo + hi, lo - hi);                // bit 0
        }
    }
    pair_stages(q);                                          // bits 1 to 4
    {
        const float sgn = (lane & 1) ? -1.0f : 1.0f;
        const uint64_t sgn2 = pair_of(sgn, sgn);
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            float lo, hi;
            unpair(q[t], lo, hi);
            q[t] = fma2(q[t], sgn2, pair_of(__shfl_xor_sync(0xffffffffu, lo, 1), __shfl_xor_sync(0xffffffffu, hi, 1)));
        }
    }
    // row r of the buffer: the 16 pairs of lane r (then of lane 16 + r) as eight 16-byte chunks, permuted by r % 8: no
    // bank conflicts on either side
    uint64_t o[16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1) __syncwarp();
        if ((lane >> 4) == h) {
            const int r = lane & 15;
#pragma unroll
            for (int j = 0; j < 8; ++j) *reinterpret_cast<ulonglong2*>(ex + r * 128 + ((j ^ (r & 7)) << 4)) = make_ulonglong2(q[2 * j], q[2 * j + 1]);
        }
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int r = 2 * s + (lane >> 4), k = lane & 15;
            o[8 * h + s] = *reinterpret_cast<const uint64_t*>(ex + r * 128 + (((k >> 1) ^ (r & 7)) << 4) + (k & 1) * 8);
        }
    }
    pair_stages<2>(o);                                       // bits 6 and 7
    // bits 8 and 9: the sums in the order in which the product kernel's fused rotation adds up its four warps' parts
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const uint64_t a = add2(o[s], o[s + 4]), b2 = sub2(o[s], o[s + 4]);
        const uint64_t c = add2(a, o[s + 8]), d = add2(b2, o[s + 8]), e = sub2(a, o[s + 8]), f = sub2(b2, o[s + 8]);
        o[s] = add2(c, o[s + 12]);
        o[s + 4] = sub2(d, o[s + 12]);
        o[s + 8] = sub2(e, o[s + 12]);
        o[s + 12] = add2(f, o[s + 12]);
    }
    uint32_t* dst = reinterpret_cast<uint32_t*>(xdag + b * K + k0) + (lane & 3) * 8 + (lane >> 3) * 2 + ((lane >> 2) & 1);
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        float lo, hi;
        unpair(o[s], lo, hi);
        const __half2 v = __floats2half2_rn(lo * 0.03125f, hi * 0.03125f);
        dst[s * 32] = *reinterpret_cast<const uint32_t*>(&v);
    }
}

// The same with four warps per (token, group), for layers that leave SMs free: there a block needs no room beside a product block,
// and what counts is how long one group takes.  Chains of one layer, one warp / four warps in us: 2048x1024 with 12 tokens
// 4.1 / 3.6, 256x8192 with one 3.2 / 3.05, 512x3072 with two 3.4 / 3.15; where a block finds no free SM: 2560x1024 with three 3.8 /
// 4.1, 4096x4096 with four 5.7 / 8.8.
__global__ void __launch_bounds__(128) rht_activations_wide_kernel(const __nv_bfloat16* x, __half* __restrict__ xdag, int64_t B, int64_t K,
                                                                   uint64_t xi, float* __restrict__ zero_ptr, size_t zero_floats) {
    __shared__ __align__(16) float ex[4][256];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const unsigned groups = (unsigned)(K / kGroup), gi = blockIdx.x % groups;
    pdl_trigger();
    const int64_t b = blockIdx.x / groups, k0 = (int64_t)gi * kGroup + q * 256 + lane * 8;       // this lane's 8 consecutive inputs
    pdl_wait();
    for (size_t i = (size_t)blockIdx.x * 128 + threadIdx.x; i < zero_floats; i += (size_t)gridDim.x * 128) zero_ptr[i] = 0.0f;
    if (b >= B) return;
    float o[8];
    rotate_by_four_warps<true>(x + b * K + k0, xi, k0, ex, q, lane, o);
    // this lane holds pairs 4 j + i (i = 0..3, j = lane % 8) of 64-input block q*4 + lane/8 of the group, i.e.
    // m = j >> 1, h = j & 1, t = i  ->  position i*8 + j
    uint32_t* blk = reinterpret_cast<uint32_t*>(xdag + b * K + (int64_t)gi * kGroup) + (q * 4 + (lane >> 3)) * 32;
    const int j = lane & 7;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __half2 hh = __floats2half2_rn(o[2 * e] * 0.03125f, o[2 * e + 1] * 0.03125f);
        blk[e * 8 + j] = *reinterpret_cast<const uint32_t*>(&hh);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) rht_debug_kernel(const T* __restrict__ x, float* __restrict__ out,
                                                        int64_t rows, int64_t K, uint64_t xi, float mul) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t groups = K / kGroup;
    if (warp >= rows * groups) return;
    const int64_t b = warp / groups, gi = warp % groups;
    float v[32];
    load_group<T>(x + b * K + gi * kGroup, lane, v);
    apply_signs1024(v, xi, gi * kGroup, lane);
    fwht1024_warp(v, lane);
    float* dst = out + b * K + gi * kGroup;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        *reinterpret_cast<float4*>(dst + c * 256 + lane * 8) =
            make_float4(v[c * 8] * mul, v[c * 8 + 1] * mul, v[c * 8 + 2] * mul, v[c * 8 + 3] * mul);
        *reinterpret_cast<float4*>(dst + c * 256 + lane * 8 + 4) =
            make_float4(v[c * 8 + 4] * mul, v[c * 8 + 5] * mul, v[c * 8 + 6] * mul, v[c * 8 + 7] * mul);
    }
}

}  // namespace

int launch_rht_activations(const higgs_desc& d, const void* x, int64_t B, __half* xdag, float* zero_ptr,
                           size_t zero_floats, cudaStream_t st) {
    int64_t blocks = B * (d.K / kGroup);
    // (a block of four warps finds an SM of its own beside the product's blocks; above 16 tokens several products follow: 1040x2048 with
    // 32 8.4 / 9.3)
    const bool wide = B <= 16 && linear_leaves_sms(d, B, blocks);
    const int threads = wide ? 128 : 32;
    if (zero_floats) {
        int64_t zb = (int64_t)((zero_floats + threads * 8 - 1) / (threads * 8));
        if (zb > 1184) zb = 1184;
        if (zb > blocks) blocks = zb;
    }
    if (wide)
        return cuda_status(launch_pdl(rht_activations_wide_kernel, dim3((unsigned)blocks), dim3(128), 0, st,
                                      static_cast<const __nv_bfloat16*>(x), xdag, B, d.K, d.rht_seed, zero_ptr, zero_floats));
    return cuda_status(launch_pdl(rht_activations_kernel, dim3((unsigned)blocks), dim3(32), 0, st,
                                  static_cast<const __nv_bfloat16*>(x), xdag, B, d.K, d.rht_seed, zero_ptr, zero_floats));
}

int launch_rht_debug(const higgs_desc& d, const void* x, int x_dtype, int64_t rows, float* out, int normalised,
                     cudaStream_t st) {
    const int64_t warps = rows * (d.K / kGroup);
    if (warps == 0) return HIGGS_OK;
    const unsigned blocks = (unsigned)((warps + 7) / 8);
    const float mul = normalised ? 0.03125f : 1.0f;
    if (x_dtype == HIGGS_BF16)
        rht_debug_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(x), out, rows, d.K,
                                                               d.rht_seed, mul);
    else if (x_dtype == HIGGS_F32)
        rht_debug_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(x), out, rows, d.K, d.rht_seed, mul);
    else
        return HIGGS_ERR_UNSUPPORTED;
    return cuda_status(cudaGetLastError());
}

}  // namespace higgs
