// FP32 sketches as two FP16 planes for the FP32-accuracy product.
//
// A row of FP32 sums x is written as hi + lo / 2048 with hi and lo in FP16 after a
// power-of-two scale 2^-e that brings the row's largest magnitude into [2^14, 2^15):
//   hi = RN16(x 2^-e),   lo = RN16((x 2^-e - hi) 2048)      (the difference is exact)
// so x 2^-e = hi + lo / 2048 to 2^-24 of x for every |x| >= 2^-28 of the row's
// largest (below that, to 2^-36 of the scale's unit).  3xTF32 keeps 22 bits of x
// (both of its planes lose bits by truncation), and the FP16 tensor rate is twice
// the TF32 one.
//
// Rows that the format does not suit are counted on the device: a largest magnitude
// that is not finite or lies outside [2^-40, 2^60], or more than a 64th of the
// nonzeros below 2^-28 of the largest.  One such row raises *flag; the FP16 product
// then returns at once and the TF32 planes are made from the same sums in place
// (tf32_planes_kernel), so that these operands keep the accuracy they had.
//
// The split is memory-bound: 2 x 8192 rows of 8192 sums, 4 bytes read (twice, the
// second time from L1/L2) and 4 written each, take 165 us (6.5 TB/s) on GB300.
#include <cuda_fp16.h>

#include "common.cuh"

namespace osk {

namespace {

constexpr uint32_t kAmaxLo = 0x2b800000u;   // 2^-40
constexpr uint32_t kAmaxHi = 0x5d800000u;   // 2^60

__global__ void __launch_bounds__(256) split_f16_kernel(SplitSide a, SplitSide b, int64_t ld, int32_t blk,
                                                        BlockList kept, unsigned int *__restrict__ flag) {
    const bool right = blockIdx.x >= (uint64_t)a.rows;
    const SplitSide s = right ? b : a;
    const int64_t r = right ? (int64_t)blockIdx.x - a.rows : (int64_t)blockIdx.x;
    const float *x = s.sums + r * ld;
    __half *hi = reinterpret_cast<__half *>(s.sums + s.rows * ld) + r * ld;   // planes follow the sums
    __half *lo = hi + s.rows * ld;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = blk / 4, total = kept.count * per;   // 16-byte pieces
    __shared__ uint32_t red[8];
    __shared__ int2 cnt[8];
    auto piece = [&](int q) -> int64_t {
        const int t = q / per;
        return (int64_t)kept.idx[t] * blk + 4 * (q - t * per);
    };
    // the row's largest magnitude (as bits: NaN above Inf above every finite value)
    uint32_t am = 0;
#pragma unroll 4
    for (int q = tid; q < total; q += 256) {
        const uint4 u = *reinterpret_cast<const uint4 *>(x + piece(q));
        am = max(max(am, u.x & 0x7fffffffu), max(u.y & 0x7fffffffu, max(u.z & 0x7fffffffu, u.w & 0x7fffffffu)));
    }
    am = __reduce_max_sync(0xffffffffu, am);
    if (lane == 0) red[warp] = am;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) am = max(am, red[w]);
    if (am != 0 && (am < kAmaxLo || am > kAmaxHi)) {
        if (tid == 0) *flag = 1u;
        return;
    }
    const int e = am ? (int)(am >> 23) - 127 - 14 : 0;
    const float down = __uint_as_float((uint32_t)(127 - e) << 23);   // 2^-e, exact
    int nz = 0, small = 0;
#pragma unroll 4
    for (int q = tid; q < total; q += 256) {
        const int64_t c = piece(q);
        const float4 u = *reinterpret_cast<const float4 *>(x + c);
        const float v[4] = {u.x * down, u.y * down, u.z * down, u.w * down};
        __half h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            h[k] = __float2half_rn(v[k]);
            l[k] = __float2half_rn((v[k] - __half2float(h[k])) * 2048.f);
            nz += v[k] != 0.f;
            small += v[k] != 0.f && fabsf(v[k]) < 0x1p-13f;
        }
        *reinterpret_cast<uint2 *>(hi + c) = *reinterpret_cast<const uint2 *>(h);
        *reinterpret_cast<uint2 *>(lo + c) = *reinterpret_cast<const uint2 *>(l);
    }
    nz = __reduce_add_sync(0xffffffffu, nz);
    small = __reduce_add_sync(0xffffffffu, small);
    if (lane == 0) cnt[warp] = make_int2(nz, small);
    __syncthreads();
    if (tid == 0) {
        int n = 0, t = 0;
        for (int w = 0; w < 8; ++w) n += cnt[w].x, t += cnt[w].y;
        if ((int64_t)t * 64 > n) *flag = 1u;
        s.scale[r] = __uint_as_float((uint32_t)(127 + e) << 23);   // 2^e
    }
}

// The sums as the two TF32 planes (hi in place, lo over the FP16 planes), when *flag is set.
__global__ void __launch_bounds__(256) tf32_planes_kernel(SplitSide a, SplitSide b, int64_t ld, int32_t blk,
                                                          BlockList kept, const unsigned int *__restrict__ flag) {
    if (*flag == 0u) return;
    const int per = blk / 4, total = kept.count * per;
    for (int64_t row = blockIdx.x; row < a.rows + b.rows; row += gridDim.x) {
        const SplitSide &s = row < a.rows ? a : b;
        float *x = s.sums + (row < a.rows ? row : row - a.rows) * ld;
        float *y = x + s.rows * ld;
        for (int q = threadIdx.x; q < total; q += 256) {
            const int t = q / per;
            const int64_t c = (int64_t)kept.idx[t] * blk + 4 * (q - t * per);
            const float4 u = *reinterpret_cast<const float4 *>(x + c);
            auto top = [](float v) { return __uint_as_float(__float_as_uint(v) & 0xffffe000u); };
            const float4 h = make_float4(top(u.x), top(u.y), top(u.z), top(u.w));
            *reinterpret_cast<float4 *>(x + c) = h;
            *reinterpret_cast<float4 *>(y + c) = make_float4(u.x - h.x, u.y - h.y, u.z - h.z, u.w - h.w);
        }
    }
}

}  // namespace

os_status launch_split_f16(const SplitSide &a, const SplitSide &b, int64_t ld, int32_t blk, const BlockList &kept,
                           unsigned int *flag, cudaStream_t st) {
    OSK_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(unsigned int), st));
    split_f16_kernel<<<(unsigned)(a.rows + b.rows), 256, 0, st>>>(a, b, ld, blk, kept, flag);
    return check_launch();
}

os_status launch_tf32_planes(const SplitSide &a, const SplitSide &b, int64_t ld, int32_t blk, const BlockList &kept,
                             const unsigned int *flag, cudaStream_t st) {
    const int64_t rows = a.rows + b.rows;
    tf32_planes_kernel<<<(unsigned)(rows < 152 * 8 ? rows : 152 * 8), 256, 0, st>>>(a, b, ld, blk, kept, flag);
    return check_launch();
}

}  // namespace osk
