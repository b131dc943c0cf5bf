// FP32 sketches as two FP16 planes for the FP32-accuracy product.
//
// A row of FP32 sums x is written as hi + lo / 4096 with hi and lo in FP16 after a
// power-of-two scale 2^-e that brings the row's largest magnitude into [2^14, 2^15):
//   hi = RN16(x 2^-e),   lo = RN16((x 2^-e - hi) 4096)      (the difference is exact)
// so hi + lo / 4096 is x 2^-e to 2^-23 of it (hi leaves at most 2^-11, of which lo keeps 11
// bits) and, where FP16 runs out of exponents, to 2^-37: 2^-21 of x at 2^-16, that is 2^-30
// of the row's largest, where lo holds up to 2^-9 of x, so that the dropped lo.lo is 2^-20 of
// its term (2^-22 of ordinary ones).  3xTF32 holds x to 2^-20 and drops 2^-20 (its planes
// keep 11 bits each by truncation), and the FP16 tensor rate is twice the TF32 one.
//
// Below that line the planes would be off by any share of x.  How few such entries a row
// has says nothing about what they contribute (C consists of them where the other operand
// is zero beside them), so none is left to the planes: they get zeros there, the entries
// are listed, and correct_kernel adds their products to C in FP32.  Sums of random signs
// have one by chance in every few products of 2^27 sums, sums whose columns are scaled over
// six decades (an interior-point matrix) about one in 10^4; operands with more than the
// list may take (launch_split_f16's `most`) raise the flag, and so does a row whose largest magnitude is not finite or
// lies outside [2^-60, 2^80].  The FP16 product then returns at once and the TF32 planes
// are made from the same sums in place, so these operands get the 3xTF32 product.
//
// The split is memory-bound: 2 x 8192 rows of 8192 sums, 4 bytes read (twice, the
// second time from L1/L2) and 4 written each, take 165 us (6.5 TB/s) on GB300.
#include <cuda_fp16.h>

#include "common.cuh"

namespace osk {

namespace {

// A row's largest magnitude: between these, a sum of products of scaled values (2^-50 ..
// 2^48) times one side's scale stays a normal number before the other's is applied.
constexpr uint32_t kAmaxLo = 0x21800000u;   // 2^-60
constexpr uint32_t kAmaxHi = 0x67800000u;   // 2^80
constexpr float kHeldFrom = 0x1p-16f;       // scaled magnitudes from here on are left to the planes

// Whether a scaled sum is left to the list.
__device__ __forceinline__ bool listed(float v) { return v != 0.f && fabsf(v) < kHeldFrom; }

__global__ void __launch_bounds__(256) split_f16_kernel(SplitSide a, SplitSide b, int64_t ld, int32_t blk,
                                                        BlockList kept, SplitCtl *__restrict__ ctl, unsigned int most) {
    const bool right = blockIdx.x >= (uint64_t)a.rows;
    const SplitSide s = right ? b : a;
    const int64_t r = right ? (int64_t)blockIdx.x - a.rows : (int64_t)blockIdx.x;
    const float *x = s.sums + r * ld;
    __half *hi = reinterpret_cast<__half *>(s.sums + s.rows * ld) + r * ld;   // planes follow the sums
    __half *lo = hi + s.rows * ld;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = blk / 4, total = kept.count * per;   // 16-byte pieces
    __shared__ uint32_t red[8];
    __shared__ int cnt[8];
    __shared__ unsigned int at;
    auto piece = [&](int q) -> int64_t {
        const int t = q / per;
        return (int64_t)kept.idx[t] * blk + 4 * (q - t * per);
    };
    // another row has raised the flag: nothing of this pass will be used
    if (__syncthreads_or(tid == 0 && *(volatile unsigned int *)&ctl->flag != 0u)) return;
    // the row's largest magnitude (as bits: NaN above Inf above every finite value)
    uint32_t am = 0;
#pragma unroll 4
    for (int q = tid; q < total; q += 256) {
        const uint4 u = *reinterpret_cast<const uint4 *>(x + piece(q));
        am = max(am, max(u.x & 0x7fffffffu, u.y & 0x7fffffffu));
        am = max(am, max(u.z & 0x7fffffffu, u.w & 0x7fffffffu));
    }
    am = __reduce_max_sync(0xffffffffu, am);
    if (lane == 0) red[warp] = am;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) am = max(am, red[w]);
    if (am != 0 && (am < kAmaxLo || am > kAmaxHi)) {
        if (tid == 0) ctl->flag = 1u;
        return;
    }
    const int e = am ? (int)(am >> 23) - 127 - 14 : 0;
    const float down = __uint_as_float((uint32_t)(127 - e) << 23);   // 2^-e, exact
    int small = 0;
#pragma unroll 4
    for (int q = tid; q < total; q += 256) {
        const int64_t c = piece(q);
        const float4 u = *reinterpret_cast<const float4 *>(x + c);
        const float v[4] = {u.x * down, u.y * down, u.z * down, u.w * down};
        __half h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float p = fabsf(v[k]) < kHeldFrom ? 0.f : v[k];
            h[k] = __float2half_rn(p);
            l[k] = __float2half_rn((p - __half2float(h[k])) * 4096.f);
            small += p != v[k];
        }
        *reinterpret_cast<uint2 *>(hi + c) = *reinterpret_cast<const uint2 *>(h);
        *reinterpret_cast<uint2 *>(lo + c) = *reinterpret_cast<const uint2 *>(l);
    }
    if (tid == 0) s.scale[r] = __uint_as_float((uint32_t)(127 + e) << 23);   // 2^e
    small = __reduce_add_sync(0xffffffffu, small);
    if (lane == 0) cnt[warp] = small;
    __syncthreads();
    int n = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) n += cnt[w];
    if (n == 0) return;
    // the row's entries for the list: consecutive, by ascending column
    if (tid == 0) {
        at = n <= kSplitLostRow ? atomicAdd(&ctl->lost, (unsigned int)n) : most;
        if (at + n > most) ctl->flag = 1u;
    }
    __syncthreads();
    unsigned int base = at;
    if (base + n > most) return;
    for (int q0 = 0; q0 < total; q0 += 256) {
        const int q = q0 + tid;
        const int64_t c = q < total ? piece(q) : 0;
        const float4 u = q < total ? *reinterpret_cast<const float4 *>(x + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float v[4] = {u.x * down, u.y * down, u.z * down, u.w * down};
        int mine = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) mine += listed(v[k]);
        int inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        __syncthreads();   // cnt has been read
        if (lane == 31) cnt[warp] = inc;
        __syncthreads();
        unsigned int pos = base + inc - mine;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) pos += cnt[w];
            base += cnt[w];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (listed(v[k])) ctl->entry[pos++] = make_uint2((uint32_t)r | (right ? 0x80000000u : 0u), (uint32_t)(c + k));
    }
}

// After the FP16 product: with the flag set, the sums as the two TF32 planes (hi in
// place, lo over the FP16 planes) for the 3xTF32 product that follows; else the products
// of the listed entries, added to C: those of A with all of B, those of B with what the
// planes hold of A.  Tiles of 128 x 128 of C, one owner each: first the entries of A in
// its rows (thread = column), then those of B in its columns (thread = row).  The entries
// of one row are consecutive and ascending in the list and no two rows meet in an
// element, so the sums do not depend on the order in which the rows entered it.  Nothing
// listed: two loads.  A chain of loads per entry is what it waits for, so eight entries are
// taken at a time (2000 entries beside a 4160 x 8192 x 4160 product 92 us, one at a time
// 467: 1.1e-5 us per element of C that an entry adds to, kListedUs).
constexpr int kTile = 128, kBatch = 8;

__global__ void __launch_bounds__(kTile) correct_kernel(SplitSide a, SplitSide b, int64_t ld, int32_t blk,
                                                        BlockList kept, const SplitCtl *__restrict__ ctl, float alpha,
                                                        float *__restrict__ C, int64_t ldc, int64_t l) {
    if (ctl->flag != 0u) {
        const int per = blk / 4, total = kept.count * per;
        for (int64_t row = blockIdx.x; row < a.rows + b.rows; row += gridDim.x) {
            const SplitSide &s = row < a.rows ? a : b;
            float *x = s.sums + (row < a.rows ? row : row - a.rows) * ld;
            float *y = x + s.rows * ld;
#pragma unroll 2
            for (int q = threadIdx.x; q < total; q += kTile) {
                const int t = q / per;
                const int64_t c = (int64_t)kept.idx[t] * blk + 4 * (q - t * per);
                const float4 u = *reinterpret_cast<const float4 *>(x + c);
                auto top = [](float v) { return __uint_as_float(__float_as_uint(v) & 0xffffe000u); };
                const float4 h = make_float4(top(u.x), top(u.y), top(u.z), top(u.w));
                *reinterpret_cast<float4 *>(x + c) = h;
                *reinterpret_cast<float4 *>(y + c) = make_float4(u.x - h.x, u.y - h.y, u.z - h.z, u.w - h.w);
            }
        }
        return;
    }
    const int lost = (int)ctl->lost;
    if (lost == 0) return;
    const int lane = threadIdx.x & 31;
    const bool sym = b.rows == 0;   // B is A: its entries count on both sides
    const SplitSide &bs = sym ? a : b;
    // the listed entries of one side whose row lies in [from, from + kTile), a batch at a
    // time: apply(rows, columns, count)
    auto each = [&](bool of_b, int64_t from, auto apply) {
        const uint32_t side = of_b && !sym ? 1u : 0u;
        for (int i0 = 0; i0 < lost; i0 += 32) {
            const uint2 e = i0 + lane < lost ? ctl->entry[i0 + lane] : make_uint2(0u, 0u);
            const int64_t row = e.x & 0x7fffffffu;
            uint32_t in = __ballot_sync(0xffffffffu, i0 + lane < lost && e.x >> 31 == side && row >= from && row < from + kTile);
            while (in) {
                int64_t r[kBatch], c[kBatch];
                int n = 0;
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const int at = in ? __ffs((int)in) - 1 : 0;
                    r[k] = __shfl_sync(0xffffffffu, e.x, at) & 0x7fffffffu;
                    c[k] = __shfl_sync(0xffffffffu, e.y, at);
                    n += in != 0u;
                    in &= in - 1u;
                }
                apply(r, c, n);
            }
        }
    };
    // C at(r) += x y for each of the batch, one load and store per run of equal r
    auto add = [&](const int64_t (&r)[kBatch], int n, const float (&x)[kBatch], const float (&y)[kBatch], auto at) {
        float old[kBatch], acc = 0.f;
#pragma unroll
        for (int k = 0; k < kBatch; ++k) old[k] = k < n && (k == 0 || r[k] != r[k - 1]) ? *at(r[k]) : 0.f;
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            if (k >= n) break;
            if (k == 0 || r[k] != r[k - 1]) acc = old[k];
            acc = fmaf(alpha * x[k], y[k], acc);
            if (k + 1 == n || k + 1 == kBatch || r[k + 1 < kBatch ? k + 1 : k] != r[k]) *at(r[k]) = acc;
        }
    };
    const int64_t tm = (a.rows + kTile - 1) / kTile, tn = (l + kTile - 1) / kTile;
    for (int64_t t = blockIdx.x; t < tm * tn; t += gridDim.x) {
        const int64_t r0 = t / tn * kTile, s0 = (t - t / tn * tn) * kTile;
        const int64_t col = s0 + threadIdx.x, row = r0 + threadIdx.x;
        each(false, r0, [&](const int64_t (&r)[kBatch], const int64_t (&c)[kBatch], int n) {
            if (col >= l) return;
            float x[kBatch], y[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                x[k] = k < n ? a.sums[r[k] * ld + c[k]] : 0.f;
                y[k] = k < n ? bs.sums[col * ld + c[k]] : 0.f;
            }
            add(r, n, x, y, [&](int64_t q) { return C + q * ldc + col; });
        });
        __syncthreads();   // the rows above may hold elements of the columns below
        each(true, s0, [&](const int64_t (&s)[kBatch], const int64_t (&c)[kBatch], int n) {
            if (row >= a.rows) return;
            const float down = 1.f / a.scale[row];
            float x[kBatch], y[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                x[k] = k < n ? a.sums[row * ld + c[k]] : 0.f;
                if (listed(x[k] * down)) x[k] = 0.f;   // added above
                y[k] = k < n ? bs.sums[s[k] * ld + c[k]] : 0.f;
            }
            add(s, n, x, y, [&](int64_t q) { return C + row * ldc + q; });
        });
        __syncthreads();
    }
}

}  // namespace

os_status launch_split_f16(const SplitSide &a, const SplitSide &b, int64_t ld, int32_t blk, const BlockList &kept,
                           SplitCtl *ctl, unsigned int most, cudaStream_t st) {
    OSK_CUDA_TRY(cudaMemsetAsync(ctl, 0, offsetof(SplitCtl, entry), st));
    split_f16_kernel<<<(unsigned)(a.rows + b.rows), 256, 0, st>>>(a, b, ld, blk, kept, ctl, most < kSplitLost ? most : kSplitLost);
    return check_launch();
}

os_status launch_split_correct(const SplitSide &a, const SplitSide &b, int64_t ld, int32_t blk, const BlockList &kept,
                               const SplitCtl *ctl, float alpha, float *C, int64_t ldc, int64_t l, cudaStream_t st) {
    const int64_t rows = a.rows + b.rows;
    correct_kernel<<<(unsigned)(rows < 152 * 16 ? rows : 152 * 16), kTile, 0, st>>>(a, b, ld, blk, kept, ctl, alpha, C, ldc,
                                                                                   l);
    return check_launch();
}

}  // namespace osk
