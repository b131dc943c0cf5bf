// Sketch kernels: A~ = A S and B~ = S^T B (Alg. 5, Alg. 4 step 3), plus the
// adjoint gathers used by the backward pass.
//
// One gather kernel serves both sides.  It reads a matrix X whose rows are
// indexed by the sketched dimension i (n rows) and whose "free" dimension f
// runs along the other axis, and writes Y^T[f, q] for q = j*b + c:
//
//     Y^T[f, j*b + c] = sum_{i in bucket c of block j} sigma_j(i) * s_i * X[i, f]
//
// Right sketch: X = B (n x l), Y^T = B~^T (l x z).  Left sketch: X = A^T,
// Y^T = A~ (m x z).
//
// The gather reads X in strips of W free indices (W = 128 for FP32, 256 for
// BF16): strip s holds X[0..n-1, Ws .. Ws+W-1], and a random row of it is one
// 512-byte piece, 16 bytes per lane of a warp.  The left operand (and a BF16
// right operand whose rows are not 16-byte aligned) is first packed strip-major into the workspace, n contiguous
// rows of 128 elements per strip, zero-padded past the free extent; packing
// the left operand is the transpose it needs anyway.  An FP32 right operand
// is gathered in place: in 128-wide strips when its rows are 16-byte aligned,
// else in 124-wide strips whose row pieces start d = 0..3 elements into a
// 16-byte granule (lane c loads granule c; the sums are kept per class d and
// realigned with one shuffle per bucket), or packed when that costs less
// (more than 6 blocks gathered).  Whole 512-byte pieces keep the address
// translations of the random row accesses cheap; 128-byte pieces spread over
// a 4 GB matrix ran at a quarter to a half of the L2 gather rate on GB300.
//
// A gather CTA owns 16 consecutive sketched columns q (32 for FP8 output;
// whole buckets of one block) and one strip.  Each warp walks the bucket-CSR of its buckets
// (indices ascending inside a bucket, the same order in every run: no
// atomics, bitwise reproducible) and gathers row pieces with 16-byte loads,
// accumulating in FP32.  The (16 or 32)-column x 128-row tile is transposed through
// shared memory so that Y^T rows are written contiguously.  CTAs of one strip
// are adjacent in launch order, so a strip stays in L2 while all of its
// buckets are gathered.  For FP8 output the four CTAs that own the quarters of
// one 128-column scale slice form a thread-block cluster and combine their
// per-row maxima through distributed shared memory.
#include <cooperative_groups.h>
#include <cstdint>
#include <cstdlib>
#include <type_traits>

#include "common.cuh"

namespace osk {

namespace {

constexpr int kWarps = 8;
constexpr int kStrip = 128;   // free indices per FP32 strip (the in-place right sketch)

// Free indices per packed strip of an element type: 16 bytes per lane of a warp
// (128 FP32, 256 BF16), so every gathered row piece is 512 bytes.
template <typename T>
__host__ __device__ constexpr int strip_of() {
    return 32 * (16 / (int)sizeof(T));
}

// VW consecutive elements of the free dimension per lane (strip = 32*VW).
template <typename InT, int VW, bool kAligned>
struct Loader {
    __device__ __forceinline__ static void load(const InT *p, float (&v)[VW]) {
        if constexpr (kAligned && std::is_same<InT, float>::value && VW == 4) {
            const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
            v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
        } else if constexpr (kAligned && std::is_same<InT, float>::value && VW == 2) {
            const float2 t = __ldg(reinterpret_cast<const float2 *>(p));
            v[0] = t.x; v[1] = t.y;
        } else if constexpr (kAligned && std::is_same<InT, __nv_bfloat16>::value && VW == 4) {
            const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
            const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
            v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
        } else if constexpr (kAligned && std::is_same<InT, __nv_bfloat16>::value && VW == 2) {
            const unsigned u = __ldg(reinterpret_cast<const unsigned *>(p));
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u));
            v[0] = a.x; v[1] = a.y;
        } else {
#pragma unroll
            for (int k = 0; k < VW; ++k) v[k] = to_f32(p[k]);
        }
    }
    // 16 raw bytes (VW = 16 / sizeof(InT)) now, converted when they are summed
    using Raw = uint4;
    __device__ __forceinline__ static Raw load_raw(const InT *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
    __device__ __forceinline__ static void unpack(const Raw &u, float (&v)[VW]) {
        if constexpr (std::is_same<InT, float>::value) {
            static_assert(VW == 4, "four FP32 per 16 bytes");
            v[0] = __uint_as_float(u.x); v[1] = __uint_as_float(u.y);
            v[2] = __uint_as_float(u.z); v[3] = __uint_as_float(u.w);
        } else {
            static_assert(VW == 8, "eight BF16 per 16 bytes");
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[q]));
                v[2 * q] = f.x;
                v[2 * q + 1] = f.y;
            }
        }
    }
    __device__ __forceinline__ static float to_f32(float x) { return x; }
    __device__ __forceinline__ static float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
    __device__ __forceinline__ static float load1(const InT *p) { return to_f32(p[0]); }
};

// Two FP32 values in a 64-bit register, for the packed FP32 multiply-add (each half
// rounded as fmaf does).  Kept packed from load to flush: packing around every
// instruction costs more moves than it saves.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(f32x2 &acc, f32x2 w, f32x2 x) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(w), "l"(x));
}
// The 16 raw bytes of a row piece as pairs of FP32.
template <typename InT> struct Pairs;
template <> struct Pairs<float> {
    static constexpr int N = 2;
    __device__ __forceinline__ static f32x2 get(const uint4 &u, int k) {
        return k == 0 ? pack2(__uint_as_float(u.x), __uint_as_float(u.y))
                      : pack2(__uint_as_float(u.z), __uint_as_float(u.w));
    }
};
template <> struct Pairs<__nv_bfloat16> {
    static constexpr int N = 4;
    __device__ __forceinline__ static f32x2 get(const uint4 &u, int k) {
        const uint32_t w = k == 0 ? u.x : k == 1 ? u.y : k == 2 ? u.z : u.w;
        return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
};

// Sixteen bytes of zeros: the row segment that padding entries of the bucket
// lists point at, so the gather loop needs no predication.
__device__ __align__(16) float g_zero_row[8];

// A gather CTA's (block, tile) and strip: in launch order, or (tpb < 0, -tpb tiles per
// block) with the first block of the next strip dealt out between the other blocks of
// this one, tile by tile.
__device__ __forceinline__ int2 mixed_place(int tpb, int count, int64_t &strip) {
    const uint32_t K = count, T = tpb < 0 ? -tpb : tpb, per = K * T;
    uint32_t at = blockIdx.x, tile = 0, bt = 0;
    strip = blockIdx.y;
    if (tpb > 0) {
        bt = at / T;
        return make_int2(bt, at - bt * T);
    }
    at += blockIdx.y * gridDim.x;
    if (at < T) {
        strip = 0;
        return make_int2(0, at);
    }
    at -= T;
    strip = at / per;
    at -= (uint32_t)strip * per;
    const bool last = strip + 1 == gridDim.y;
    tile = at / (last ? K - 1 : K);
    bt = last ? 1 + at - tile * (K - 1) : at - tile * K;
    strip += bt == 0;
    return make_int2(bt, tile);
}

// Lane layout: lane = slot * SUBS + sub (SUBS = 32 / SLOTS lanes per member;
// the launches use SLOTS = 1, one member per warp load).  With SLOTS > 1 the
// slots of a warp gather different members of one bucket at once (bucket lists
// are padded to a multiple of 4).  Lane `sub` holds the 16 bytes at elements
// VW*sub .. VW*sub+VW-1 of the strip (VW = 4 FP32 or 8 BF16).
// A warp owns QT/8 consecutive buckets and streams their (contiguous) padded
// member list 32 entries at a time, keeping 8 independent 16-byte loads per
// lane in flight and prefetching the next 32 entries.  Slot s accumulates
// members s, s+SLOTS, ... of a bucket in ascending order and the partial sums
// are combined by a fixed butterfly (one chain when SLOTS = 1): a fixed order,
// so the results are bitwise reproducible.
template <typename InT, typename OutT, int QT, bool kScale, int SLOTS, bool kMis>
__global__ void __launch_bounds__(kWarps * 32, kMis ? 3 : 4)
sketch_gather_kernel(const InT *__restrict__ X, int64_t strip_stride, int64_t ldx, int64_t F,
                     const uint32_t *__restrict__ pperm, const uint32_t *__restrict__ poffs,
                     int64_t pstride, int32_t b, int32_t z, const float *__restrict__ wts,
                     OutT *__restrict__ Yt, int64_t ldy, float *__restrict__ scales,
                     int64_t lds, BlockList blocks, int32_t tiles_per_block, int64_t plane_elems,
                     const uint64_t *__restrict__ dmask) {
    constexpr int SUBS = 32 / SLOTS;     // lanes per member
    constexpr int VW = 16 / (int)sizeof(InT);   // free indices per lane: 16 bytes
    constexpr int TF = VW * SUBS;        // free indices per tile row (one strip)
    constexpr int TFO = kMis ? TF - 4 : TF;   // free indices written per CTA
    constexpr int PITCH = TF + 1;        // odd pitch: conflict-free column reads
    constexpr int NC = kMis ? 4 : 1;     // accumulator sets: one per misalignment class
    // BF16 rows and misaligned ones are bound by instructions: packed FP32 multiply-adds
    // and no padding test before a bucket's last batch.  BF16 keeps its accumulators
    // packed; for the four sets of misaligned rows that was slower (95 against 86 us
    // for 20011 x 1777, 6 blocks), and aligned FP32 rows, bound by L2, lose with
    // either (1.68 -> 1.81 ms on the square product's left operand).
    constexpr bool kPacked = sizeof(InT) == 2;
    constexpr bool kFewer = kMis || kPacked;
    static_assert(!kMis || (std::is_same<InT, float>::value && SLOTS == 1), "misaligned rows: FP32, one member per load");
    constexpr int G = 2 * SLOTS;         // groups of 4 members per batch: 8 loads per lane in flight
    constexpr int QPW = QT / kWarps;     // buckets per warp
    static_assert(QT == 8 || QT == 16 || QT == 32 || QT == 128, "tile of 8, 16, 32 or 128 sketched columns");
    static_assert(SLOTS == 1 || SLOTS == 2 || SLOTS == 4, "1, 2 or 4 members per warp load");
    extern __shared__ float4 smem_tile[];
    float *tile = reinterpret_cast<float *>(smem_tile);   // [QT][PITCH]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = lane / SUBS, sub = lane % SUBS;
    // FP32 rows with scales may run in the mixed order of mixed_place (FP8 tiles have to
    // stay in launch order: clusters of four; aligned rows without scales lose 0.5 - 10 %
    // to the longer prologue, whose registers they do not have).
    constexpr bool kMixable = kScale && !kMis && sizeof(InT) == 4 && sizeof(OutT) != 1;
    int2 place = make_int2(0, 0);            // block and tile
    int64_t place_y = 0;
    if constexpr (kMixable) place = mixed_place(tiles_per_block, blocks.count, place_y);
    const int bt = kMixable ? place.x : blockIdx.x / tiles_per_block;
    const int jblk = blocks.idx[bt];
    // q0: first sketched column of this CTA, inside one of the listed blocks
    const int q0 = kMixable ? jblk * b + place.y * QT : jblk * b + (blockIdx.x - bt * tiles_per_block) * QT;
    const int qend = min(z, jblk * b + b);
    // a packed operand (rows as wide as a strip): strips last to first, since the last
    // ones packed are still in L2 (1 - 2 % of the left sketches of 20011 - 32768 rows;
    // in-place operands lose as much that way)
    const int64_t strip = kMixable ? (ldx == TF ? gridDim.y - 1 - place_y : place_y)
                                   : (ldx == TF ? gridDim.y - 1 - blockIdx.y : blockIdx.y);
    const int64_t f0 = strip * TFO;
    // a block mask read at run time: CTAs of blocks it does not keep have nothing to do
    if (dmask && !((__ldg(dmask) >> jblk) & 1ull)) return;
    using L = Loader<InT, VW, true>;

    const int nb = min(QPW, qend - q0 - warp * QPW);   // buckets owned by this warp
    if (nb > 0) {
        const int cb = q0 - jblk * b + warp * QPW;        // first bucket (within the block)
        const uint32_t *pl = pperm + (int64_t)jblk * pstride;
        const float *wl = kScale ? wts + (int64_t)jblk * pstride : nullptr;
        // group boundaries of the warp's buckets: lane t holds poffs[cb + t] / 4
        const uint32_t gbl = lane <= nb ? __ldg(poffs + (int64_t)jblk * (b + 1) + cb + lane) >> 2 : 0u;
        const uint32_t gend = __shfl_sync(0xffffffffu, gbl, nb);
        // row i of the strip at xbase + i * row_bytes: one wide multiply-add per member
        const uint64_t xbase = reinterpret_cast<uint64_t>(X + strip * strip_stride + VW * sub);
        const uint32_t row_bytes = (uint32_t)(ldx * (int64_t)sizeof(InT));
        const uint64_t zrow = reinterpret_cast<uint64_t>(g_zero_row);

        // 32 entries starting at group g (past the warp's last group: padding)
        auto load_entries = [&](uint32_t g) -> uint32_t {
            const uint32_t pos = 4 * g + lane;
            return pos < 4 * gend ? __ldg(pl + pos) : kPadEntry;
        };
        // the signed scales sigma_j(i) s_i of the same 32 entries (scaled sketches)
        auto load_weights = [&](uint32_t g) -> float {
            if constexpr (!kScale) return 1.f;
            const uint32_t pos = 4 * g + lane;
            return pos < 4 * gend ? __ldg(wl + pos) : 0.f;
        };
        // GG groups (4*GG members) of the current bucket, entries in lanes 0 .. 4*GG-1
        // of e, their signed scales in the same lanes of w.  Only a bucket's last group
        // holds padding: the batches before it skip the test for it.
        auto batch = [&](auto gg, auto padded, uint32_t e, float w, auto *acc) {
            constexpr int GG = decltype(gg)::value;
            constexpr bool kPadded = decltype(padded)::value;
            constexpr int KS = 4 * GG / SLOTS;            // member loads per lane
            uint4 v[KS];
            float wgt[KS];
            uint32_t cls = 0;                             // 4 x misalignment class of member k: bits 2k+2, 2k+3
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                const uint32_t ent = __shfl_sync(0xffffffffu, e, k * SLOTS + slot);
                // +-1 from the sign bit (or the signed scale); padding reads the zero row
                // (a signed scale is fetched when the row is added: eight fewer live registers)
                if constexpr (!kScale) wgt[k] = __uint_as_float(0x3f800000u | (ent & kSignBit));
                uint64_t addr = (uint64_t)(ent & kIndexMask) * row_bytes + xbase;
                if constexpr (kMis) {
                    // The row piece starts d = 0..3 elements into a 16-byte granule
                    // (the same d on every lane); lane c loads granule c from there:
                    // the 32 granules cover the strip's 124 elements and end inside
                    // the row (the launch keeps 128 elements of every strip in it).
                    cls |= ((uint32_t)addr & 12u) << (2 * k);
                    addr &= ~uint64_t(15);
                }
                v[k] = L::load_raw(reinterpret_cast<const InT *>(!kPadded || ent != kPadEntry ? addr : zrow));
            }
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                if constexpr (kScale) wgt[k] = __shfl_sync(0xffffffffu, w, k * SLOTS + slot);
                if constexpr (kPacked) {
                    constexpr int N = Pairs<InT>::N;
                    const f32x2 w2 = pack2(wgt[k], wgt[k]);
#pragma unroll
                    for (int q = 0; q < N; ++q) fma2(acc[q], w2, Pairs<InT>::get(v[k], q));
                } else if constexpr (kMis) {
                    // one accumulator set per class (a warp-uniform branch)
                    float x[VW];
                    L::unpack(v[k], x);
                    const f32x2 w2 = pack2(wgt[k], wgt[k]);
                    auto add = [&](float *a) {
#pragma unroll
                        for (int w = 0; w < VW; w += 2) {
                            f32x2 t = pack2(a[w], a[w + 1]);
                            fma2(t, w2, pack2(x[w], x[w + 1]));
                            unpack2(t, a[w], a[w + 1]);
                        }
                    };
                    const uint32_t d = (cls >> (2 * k)) & 12u;
                    if (d == 0u) add(acc);
                    else if (d == 4u) add(acc + VW);
                    else if (d == 8u) add(acc + 2 * VW);
                    else add(acc + 3 * VW);
                } else {
                    float x[VW];
                    L::unpack(v[k], x);
#pragma unroll
                    for (int w = 0; w < VW; ++w) acc[w] = fmaf(wgt[k], x[w], acc[w]);
                }
            }
        };
        auto flush = [&](int t, const float *acc) {
            float out[VW];
            if constexpr (kMis) {
                // class d holds element 4*sub + w - d of the strip in lane sub, slot w:
                // free index 4*sub + w is slot w + d of this lane, or slot w + d - 4
                // of the next lane; the classes are added in the order 0, 1, 2, 3
                float nx[NC * VW];
#pragma unroll
                for (int d = 1; d < NC; ++d)
#pragma unroll
                    for (int w = 0; w < d; ++w) nx[d * VW + w] = __shfl_down_sync(0xffffffffu, acc[d * VW + w], 1);
#pragma unroll
                for (int w = 0; w < VW; ++w) {
                    float o = acc[w];
#pragma unroll
                    for (int d = 1; d < NC; ++d)
                        o += (w + d < VW) ? acc[d * VW + (w + d) % VW] : nx[d * VW + (w + d) % VW];
                    out[w] = o;
                }
            } else {
#pragma unroll
                for (int w = 0; w < VW; ++w) {
                    out[w] = acc[w];
                    if constexpr (SLOTS == 4) out[w] += __shfl_xor_sync(0xffffffffu, out[w], 8);
                    if constexpr (SLOTS >= 2) out[w] += __shfl_xor_sync(0xffffffffu, out[w], 16);
                }
            }
            if (slot == 0) {
#pragma unroll
                for (int w = 0; w < VW; ++w) tile[(warp * QPW + t) * PITCH + VW * sub + w] = out[w];
            }
        };

        // The warp's buckets are contiguous in the list: stream it in batches that
        // never cross a bucket end (full batches of G groups, then the tail as
        // G/2, G/4, ..., 1 groups), prefetching the next 32 entries each time.
        uint32_t g = __shfl_sync(0xffffffffu, gbl, 0);
        uint32_t e_cur = load_entries(g);
        float w_cur = load_weights(g);
        auto step = [&](auto gg, auto padded, auto *acc) {
            constexpr int GG = decltype(gg)::value;
            const uint32_t e_nxt = load_entries(g + GG);
            const float w_nxt = load_weights(g + GG);
            batch(gg, padded, e_cur, w_cur, acc);
            g += GG;
            e_cur = e_nxt;
            w_cur = w_nxt;
        };
        for (int t = 0; t < nb; ++t) {
            const uint32_t gE = __shfl_sync(0xffffffffu, gbl, t + 1);
            constexpr std::true_type last{};
            constexpr int NA = kPacked ? NC * VW / 2 : NC * VW;
            typename std::conditional<kPacked, f32x2, float>::type acc[NA];
#pragma unroll
            for (int w = 0; w < NA; ++w) acc[w] = 0;
            if constexpr (kFewer) {
                while (gE - g > (uint32_t)G) step(std::integral_constant<int, G>(), std::false_type(), acc);
                if (gE - g == (uint32_t)G) step(std::integral_constant<int, G>(), last, acc);
            } else {
                while (gE - g >= (uint32_t)G) step(std::integral_constant<int, G>(), last, acc);
            }
            const uint32_t r = gE - g;   // < G
            if constexpr (G >= 8) if (r & 4u) step(std::integral_constant<int, 4>(), last, acc);
            if constexpr (G >= 4) if (r & 2u) step(std::integral_constant<int, 2>(), last, acc);
            if (r & 1u) step(std::integral_constant<int, 1>(), last, acc);
            if constexpr (kPacked) {
                float sums[NC * VW];
#pragma unroll
                for (int w = 0; w < NA; ++w) unpack2(acc[w], sums[2 * w], sums[2 * w + 1]);
                flush(t, sums);
            } else {
                flush(t, acc);
            }
        }
    }
    __syncthreads();

    if constexpr (sizeof(OutT) == 1) {
        // FP8: cluster rank r holds columns 32r .. 32r+31 of the slice.  Per row:
        // partial max over 32 columns here, the slice max from all four ranks.
        static_assert(QT == 32, "FP8 tiles are the quarters of a 128-column scale slice");
        namespace cg = cooperative_groups;
        __shared__ float amax_part[TF];
        cg::cluster_group cl = cg::this_cluster();
        for (int t = 0; t < TF / kWarps; ++t) {
            const int ff = warp * (TF / kWarps) + t;
            float a = fabsf(tile[lane * PITCH + ff]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
            if (lane == 0) amax_part[ff] = a;
        }
        cl.sync();
        const bool scale_writer = cl.block_rank() == 0 && lane == 0;
        for (int t = 0; t < TF / kWarps; ++t) {
            const int ff = warp * (TF / kWarps) + t;
            const int64_t frow = f0 + ff;
            float a = lane < 4 ? *cl.map_shared_rank(amax_part + ff, (unsigned)lane) : 0.f;
            a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 1));
            a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 2));
            a = __shfl_sync(0xffffffffu, a, 0);
            if (ff < TFO && frow < F) {
                const int e = fp8_scale_exponent(a);
                const float inv = ldexpf(1.f, -e);
                Yt[frow * ldy + q0 + lane] = __nv_fp8_e4m3(tile[lane * PITCH + ff] * inv);   // RNE, saturating
                if (scale_writer) scales[(q0 / 128) * lds + frow] = ldexpf(1.f, e);           // slice-major
            }
        }
        cl.sync();   // the partial maxima stay readable until every rank is done
    } else {
        // Transposed write-out: warp w writes rows f0 + 16w .. 16w+15 of Y^T.
        if constexpr (QT < 32) {
            // 32 / QT rows per warp pass, QT lanes per row
            constexpr int RPI = 32 / QT;
            const int qq = lane % QT, rr = lane / QT;
            for (int t = 0; t < TF / kWarps; t += RPI) {
                const int ff = warp * (TF / kWarps) + t + rr;
                const int64_t frow = f0 + ff;
                const int q = q0 + qq;
                if (ff < TFO && frow < F && q < qend) {
                    const float v = tile[qq * PITCH + ff];
                    OutT *dst = Yt + frow * ldy + q;
                    if constexpr (std::is_same<OutT, Tf32Pair>::value) {
                        float *d0 = reinterpret_cast<float *>(dst);
                        const float hi = __uint_as_float(__float_as_uint(v) & 0xffffe000u);
                        d0[0] = hi;
                        d0[plane_elems] = v - hi;
                    } else if constexpr (sizeof(OutT) == 4) {
                        *dst = v;
                    } else {
                        *dst = __float2bfloat16_rn(v);
                    }
                }
            }
            return;
        }
        constexpr int VPL = QT >= 32 ? QT / 32 : 1;   // values per lane per row
        for (int t = 0; t < TF / kWarps; ++t) {
            const int ff = warp * (TF / kWarps) + t;
            const int64_t frow = f0 + ff;
            if (ff >= TFO || frow >= F) break;
            float v[VPL];
#pragma unroll
            for (int k = 0; k < VPL; ++k) v[k] = tile[(lane + 32 * k) * PITCH + ff];
            OutT *dst = Yt + frow * ldy + q0;
            if constexpr (std::is_same<OutT, Tf32Pair>::value) {
                // FP32 as hi + lo: hi keeps 10 mantissa bits (exact in TF32), lo = x - hi (exact)
                float *d0 = reinterpret_cast<float *>(dst);
#pragma unroll
                for (int k = 0; k < VPL; ++k) {
                    const int q = q0 + lane + 32 * k;
                    if (q < qend) {
                        const float hi = __uint_as_float(__float_as_uint(v[k]) & 0xffffe000u);
                        d0[lane + 32 * k] = hi;
                        d0[plane_elems + lane + 32 * k] = v[k] - hi;
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < VPL; ++k) {
                    const int q = q0 + lane + 32 * k;
                    if (q < qend) {
                        if constexpr (sizeof(OutT) == 4)
                            dst[lane + 32 * k] = v[k];
                        else
                            dst[lane + 32 * k] = __float2bfloat16_rn(v[k]);
                    }
                }
            }
        }
    }
}

// Strip-major packing of the right operand: Xs[s][i][t] = X[i, 128s + t]
// (zero past the free extent F).  One thread moves 16 bytes; consecutive
// threads read consecutive pieces of a row and write consecutive pieces of a
// strip row.
template <typename T, bool kVec>
__global__ void __launch_bounds__(256) pack_rows_kernel(const T *__restrict__ X, int64_t ldx, int64_t n,
                                                        int64_t F, int64_t nstrips, T *__restrict__ Xs) {
    constexpr int V = 16 / sizeof(T);                // elements per 16-byte piece
    constexpr int SW = strip_of<T>();                // strip width
    constexpr int PPS = SW / V;                      // pieces per strip row
    const int64_t pieces_per_row = nstrips * PPS;
    const int64_t total = n * pieces_per_row;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / pieces_per_row;
        const int64_t pr = t - i * pieces_per_row;
        const int64_t s = pr / PPS, pc = pr - s * PPS;
        const int64_t c0 = s * SW + pc * V;
        uint4 u = make_uint4(0u, 0u, 0u, 0u);
        if (kVec && c0 + V <= F) {
            u = __ldg(reinterpret_cast<const uint4 *>(X + i * ldx + c0));
        } else {
            T *e = reinterpret_cast<T *>(&u);
#pragma unroll
            for (int k = 0; k < V; ++k) e[k] = c0 + k < F ? X[i * ldx + c0 + k] : T(0.f);
        }
        *reinterpret_cast<uint4 *>(Xs + (s * n + i) * SW + pc * V) = u;
    }
}

// Strip-major packing of the left operand (a transpose): Xs[s][i][t] =
// A[128s + t, i] (zero for rows past m).  A CTA moves a 32-row x 256-column
// tile of A (a quarter of a strip's width) through shared memory with 16-byte
// loads and stores; every strip row receives one contiguous 32-element piece.
template <typename T, bool kVec>
__global__ void __launch_bounds__(256) pack_cols_kernel(const T *__restrict__ A, int64_t lda, int64_t m,
                                                        int64_t n, T *__restrict__ Xs) {
    constexpr int W = 256;                          // columns of A per tile
    constexpr int V = 16 / sizeof(T);               // elements per 16-byte vector
    __shared__ T tile[32][W + 1];
    const int64_t rb = blockIdx.y;                  // 32-row block of A
    constexpr int SW = strip_of<T>();               // strip width: SW / 32 row blocks per strip
    const int64_t s = rb / (SW / 32), quarter = rb % (SW / 32);
    const int64_t i0 = (int64_t)blockIdx.x * W;
    const int tid = threadIdx.x;
    const bool whole = kVec && rb * 32 + 32 <= m && i0 + W <= n;
    if (whole) {
        for (int idx = tid; idx < 32 * W / V; idx += 256) {
            const int r = idx / (W / V), cv = idx - r * (W / V);
            const uint4 u = __ldg(reinterpret_cast<const uint4 *>(A + (rb * 32 + r) * lda + i0 + cv * V));
            const T *e = reinterpret_cast<const T *>(&u);
#pragma unroll
            for (int k = 0; k < V; ++k) tile[r][cv * V + k] = e[k];
        }
    } else {
        for (int idx = tid; idx < 32 * W; idx += 256) {
            const int r = idx / W, c = idx - r * W;
            const int64_t row = rb * 32 + r, col = i0 + c;
            tile[r][c] = (row < m && col < n) ? A[row * lda + col] : T(0.f);
        }
    }
    __syncthreads();
    // output: W strip rows, each receiving 32 elements (elements 32*quarter ..)
    for (int idx = tid; idx < W * 32 / V; idx += 256) {
        const int c = idx / (32 / V), rq = idx - c * (32 / V);
        const int64_t col = i0 + c;
        if (col >= n) continue;
        uint4 u;
        T *e = reinterpret_cast<T *>(&u);
#pragma unroll
        for (int k = 0; k < V; ++k) e[k] = tile[rq * V + k][c];
        *reinterpret_cast<uint4 *>(Xs + (s * n + col) * SW + quarter * 32 + rq * V) = u;
    }
}

// The same for BF16: tiles of 64 rows x 128 columns, so that a strip row receives a
// whole 128-byte line, with two rows per 32-bit word in shared memory (a quarter of
// the shared accesses of 2-byte elements: 219 -> 172 us for 4096 x 65536 on GB300, 158
// at the copy rate).  Column c of word row rp is at rp * 129 + c with the low five
// bits of c rotated by c / 32: conflict-free for the writes (lanes: 16 pieces of 8
// columns, word rows rp and rp + 4) and the reads (8 groups of 4 word rows, 4 columns).
// For rows that start on 16-byte boundaries; others take pack_cols_kernel, whose
// element loads are no slower than word-building ones (18940 x 2617: 127 against 180 us
// for the whole left sketch).
__global__ void __launch_bounds__(256) pack_cols_bf16_kernel(const __nv_bfloat16 *__restrict__ A, int64_t lda,
                                                             int64_t m, int64_t n, __nv_bfloat16 *__restrict__ Xs) {
    constexpr int W = 128, PITCH = 129, SW = strip_of<__nv_bfloat16>();
    __shared__ uint32_t tile[32 * PITCH];
    auto at = [](int rp, int c) { return rp * PITCH + (c & ~31) + ((c + (c >> 5)) & 31); };
    const int64_t rb = blockIdx.y, row0 = rb * 64, i0 = (int64_t)blockIdx.x * W;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (i0 + W <= n) {
        const int cv = lane & 15;
        const uint4 none = make_uint4(0u, 0u, 0u, 0u);   // rows past m
        uint4 x[2], y[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int item = 2 * warp + u, rp = 8 * (item >> 2) + (item & 3) + 4 * (lane >> 4);
            const __nv_bfloat16 *src = A + (row0 + 2 * rp) * lda + i0 + 8 * cv;
            x[u] = row0 + 2 * rp < m ? __ldg(reinterpret_cast<const uint4 *>(src)) : none;
            y[u] = row0 + 2 * rp + 1 < m ? __ldg(reinterpret_cast<const uint4 *>(src + lda)) : none;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int item = 2 * warp + u, rp = 8 * (item >> 2) + (item & 3) + 4 * (lane >> 4);
            const uint32_t xs[4] = {x[u].x, x[u].y, x[u].z, x[u].w}, ys[4] = {y[u].x, y[u].y, y[u].z, y[u].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tile[at(rp, 8 * cv + 2 * k)] = __byte_perm(xs[k], ys[k], 0x5410);
                tile[at(rp, 8 * cv + 2 * k + 1)] = __byte_perm(xs[k], ys[k], 0x7632);
            }
        }
    } else {
        const unsigned short *src = reinterpret_cast<const unsigned short *>(A);
#pragma unroll 8
        for (int idx = tid; idx < 32 * W; idx += 256) {
            const int rp = idx / W, c = idx % W;
            const int64_t r = row0 + 2 * rp, col = i0 + c;
            const uint32_t lo = r < m && col < n ? src[r * lda + col] : 0u;
            const uint32_t hi = r + 1 < m && col < n ? src[(r + 1) * lda + col] : 0u;
            tile[at(rp, c)] = lo | hi << 16;
        }
    }
    __syncthreads();
    const int64_t s = rb / (SW / 64), quarter = rb % (SW / 64);
    const int rq = lane & 7;                      // 8 rows (4 word rows) per lane
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int c = 4 * (8 * u + warp) + (lane >> 3);
        if (i0 + c >= n) continue;
        const uint4 o = make_uint4(tile[at(4 * rq, c)], tile[at(4 * rq + 1, c)], tile[at(4 * rq + 2, c)],
                                   tile[at(4 * rq + 3, c)]);
        *reinterpret_cast<uint4 *>(Xs + (s * n + i0 + c) * SW + quarter * 64 + rq * 8) = o;
    }
}

// dX[r, i] = scale * sum_{t < k} sigma_j(i) T[r, t*b + h_j(i)], j = kept[t]  (T holds the kept blocks only)
template <typename OutT>
__global__ void __launch_bounds__(256) unsketch_cols_kernel(
    const float *__restrict__ T, int64_t m, int64_t ldt, const uint32_t *__restrict__ hs, int64_t n,
    int32_t b, BlockList kept, float scale, OutT *__restrict__ dX, int64_t ldx) {
    const int64_t r = blockIdx.y;
    const float *trow = T + r * ldt;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float acc = 0.f;
        for (int t = 0; t < kept.count; ++t) {
            const int j = kept.idx[t];
            const uint32_t v = __ldg(hs + (int64_t)j * n + i);
            const float x = __ldg(trow + (int64_t)t * b + (v & kIndexMask));   // kept blocks compacted
            acc += (v & kSignBit) ? -x : x;
        }
        acc *= scale;
        if constexpr (sizeof(OutT) == 4)
            dX[r * ldx + i] = acc;
        else
            dX[r * ldx + i] = __float2bfloat16_rn(acc);
    }
}

// The same sums with the CTA's R rows of T staged in shared memory: a CTA owns
// rows r0 .. r0+R-1 of dX and sweeps all n columns, so each table entry h_j(i)
// is read once for R rows and the k random reads per output hit shared memory
// instead of a 32-byte L2 sector each.  The R rows are interleaved (column c of
// the R rows at ts[c*R .. c*R+R-1]): one 4R-byte shared load serves all R
// rows.  Same order of operations as above, so the results are bitwise equal.
template <int R> struct RowVec;
template <> struct RowVec<1> { using T = float; };
template <> struct RowVec<2> { using T = float2; };
template <> struct RowVec<4> { using T = float4; };
template <int R>
__device__ __forceinline__ float row_of(const typename RowVec<R>::T &v, int r) {
    if constexpr (R == 1) return v;
    else if constexpr (R == 2) return r == 0 ? v.x : v.y;
    else return r == 0 ? v.x : r == 1 ? v.y : r == 2 ? v.z : v.w;
}

template <typename OutT, int R>
__global__ void __launch_bounds__(1024) unsketch_cols_smem_kernel(
    const float *__restrict__ T, int64_t m, int64_t ldt, int64_t kb, const uint32_t *__restrict__ hs, int64_t n,
    int32_t b, BlockList kept, float scale, OutT *__restrict__ dX, int64_t ldx) {
    using V = typename RowVec<R>::T;
    extern __shared__ float4 ts4[];
    V *ts = reinterpret_cast<V *>(ts4);     // [kb] columns of R interleaved rows
    const int64_t r0 = (int64_t)blockIdx.x * R;
    const int rows = (int)(m - r0 < R ? m - r0 : R);
    for (int64_t c = threadIdx.x; c < kb; c += blockDim.x) {
        float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r < rows) x[r] = __ldg(T + (r0 + r) * ldt + c);
        if constexpr (R == 1) ts[c] = x[0];
        else if constexpr (R == 2) ts[c] = make_float2(x[0], x[1]);
        else ts[c] = make_float4(x[0], x[1], x[2], x[3]);
    }
    __syncthreads();
    // four columns per thread and pass, so that four table loads per kept block
    // are in flight at once
    constexpr int NI = 4;
    for (int64_t i0 = threadIdx.x; i0 < n; i0 += NI * (int64_t)blockDim.x) {
        float acc[NI][R];
#pragma unroll
        for (int u = 0; u < NI; ++u)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[u][r] = 0.f;
        // the table entries of four kept blocks at a time: 16 loads in flight
        constexpr int TB = 4;
        for (int t0 = 0; t0 < kept.count; t0 += TB) {
            uint32_t v[TB][NI];
#pragma unroll
            for (int tt = 0; tt < TB; ++tt) {
                const uint32_t *hrow = hs + (int64_t)kept.idx[t0 + tt < kept.count ? t0 + tt : t0] * n;
#pragma unroll
                for (int u = 0; u < NI; ++u) {
                    const int64_t i = i0 + (int64_t)u * blockDim.x;
                    v[tt][u] = i < n && t0 + tt < kept.count ? __ldg(hrow + i) : 0u;
                }
            }
#pragma unroll
            for (int tt = 0; tt < TB; ++tt) {
                if (t0 + tt >= kept.count) break;
#pragma unroll
                for (int u = 0; u < NI; ++u) {
                    const int64_t c = (int64_t)(t0 + tt) * b + (v[tt][u] & kIndexMask);   // kept blocks compacted
                    const bool neg = (v[tt][u] & kSignBit) != 0u;
                    const V xv = ts[c];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float x = row_of<R>(xv, r);
                        acc[u][r] += neg ? -x : x;
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            const int64_t i = i0 + (int64_t)u * blockDim.x;
            if (i >= n) continue;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r < rows) {
                    const float y = acc[u][r] * scale;
                    if constexpr (sizeof(OutT) == 4)
                        dX[(r0 + r) * ldx + i] = y;
                    else
                        dX[(r0 + r) * ldx + i] = __float2bfloat16_rn(y);
                }
            }
        }
    }
}

template <typename OutT>
__global__ void __launch_bounds__(256) unsketch_rows_kernel(
    const float *__restrict__ U, int64_t l, int64_t ldu, const uint32_t *__restrict__ hs, int64_t n,
    int32_t b, BlockList kept, float scale, OutT *__restrict__ dG, int64_t ldg) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + warp;
    if (i >= n) return;
    const int64_t c0 = (int64_t)blockIdx.y * 1024 + lane;
    float acc[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) acc[q] = 0.f;
    // the k table entries of row i, loaded at once: lane t holds kept blocks t and t + 32
    const uint32_t v_lo = lane < kept.count ? __ldg(hs + (int64_t)kept.idx[lane] * n + i) : 0u;
    const uint32_t v_hi = lane + 32 < kept.count ? __ldg(hs + (int64_t)kept.idx[lane + 32] * n + i) : 0u;
    for (int t = 0; t < kept.count; ++t) {
        const uint32_t v = __shfl_sync(0xffffffffu, t < 32 ? v_lo : v_hi, t & 31);
        const float sg = (v & kSignBit) ? -scale : scale;
        const float *urow = U + ((int64_t)t * b + (v & kIndexMask)) * ldu;   // kept blocks compacted
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            const int64_t c = c0 + 32 * q;
            if (c < l) acc[q] = fmaf(sg, __ldg(urow + c), acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 32; ++q) {
        const int64_t c = c0 + 32 * q;
        if (c < l) {
            if constexpr (sizeof(OutT) == 4)
                dG[i * ldg + c] = acc[q];
            else
                dG[i * ldg + c] = __float2bfloat16_rn(acc[q]);
        }
    }
}

// The same sums with 16-byte accesses (l, ldu and ldg multiples of 4, U and dG
// 16-byte aligned): lane t covers columns 4t .. 4t+3 of every 128-column group,
// a quarter of the load instructions for the same bytes.  Same order of
// operations, so the results are bitwise equal.
template <typename OutT>
__global__ void __launch_bounds__(256) unsketch_rows_vec_kernel(
    const float *__restrict__ U, int64_t l, int64_t ldu, const uint32_t *__restrict__ hs, int64_t n,
    int32_t b, BlockList kept, float scale, OutT *__restrict__ dG, int64_t ldg) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + warp;
    if (i >= n) return;
    const int64_t c0 = (int64_t)blockIdx.y * 1024 + 4 * lane;
    float4 acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t v_lo = lane < kept.count ? __ldg(hs + (int64_t)kept.idx[lane] * n + i) : 0u;
    const uint32_t v_hi = lane + 32 < kept.count ? __ldg(hs + (int64_t)kept.idx[lane + 32] * n + i) : 0u;
    for (int t = 0; t < kept.count; ++t) {
        const uint32_t v = __shfl_sync(0xffffffffu, t < 32 ? v_lo : v_hi, t & 31);
        const float sg = (v & kSignBit) ? -scale : scale;
        const float *urow = U + ((int64_t)t * b + (v & kIndexMask)) * ldu;   // kept blocks compacted
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int64_t c = c0 + 128 * q;
            if (c < l) {
                const float4 u = __ldg(reinterpret_cast<const float4 *>(urow + c));
                acc[q].x = fmaf(sg, u.x, acc[q].x);
                acc[q].y = fmaf(sg, u.y, acc[q].y);
                acc[q].z = fmaf(sg, u.z, acc[q].z);
                acc[q].w = fmaf(sg, u.w, acc[q].w);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int64_t c = c0 + 128 * q;
        if (c < l) {
            if constexpr (sizeof(OutT) == 4) {
                *reinterpret_cast<float4 *>(dG + i * ldg + c) = acc[q];
            } else {
                __nv_bfloat162 h[2] = {__floats2bfloat162_rn(acc[q].x, acc[q].y),
                                       __floats2bfloat162_rn(acc[q].z, acc[q].w)};
                *reinterpret_cast<uint2 *>(dG + i * ldg + c) = *reinterpret_cast<uint2 *>(h);
            }
        }
    }
}

// dX[r, i] = sum_t sigma_j(i) Tt[t*b + h_j(i), r], j = kept[t], from the transpose
// Tt (kb x m) of the kept blocks' T: the gather of unsketch_rows (whole 512-byte row
// pieces out of L2: Tt is taken in strips of 128 of m, k b 512 bytes each) with its
// 64 x 128 tile transposed through shared memory on the way out.  Gathering single
// columns of T from shared memory instead (unsketch_cols_smem_kernel) is held by
// bank conflicts: 4096 x 65536 BF16 from 4 blocks of 2048 took 421 us on GB300, this
// 316 (the L1 is the busiest unit).  The same additions in the same order.
// Shared tile: row i holds 32 chunks of 4 r's, chunk c at position c ^ ((i ^ i / 8) % 8),
// so that both the row writes (16 bytes per lane) and the column reads (8 i's of 4
// r's per warp, i = 8 (lane / 4) + s) touch every bank once.  Rows of dX without
// 16-byte alignment are stored 32 elements per instruction instead (reads four to a
// bank), not 8 per lane.
constexpr int kUtRows = 64;
template <typename OutT, bool kVec>
__global__ void __launch_bounds__(256, 4) unsketch_cols_t_kernel(
    const float *__restrict__ Tt, int64_t m, int64_t ldt, const uint32_t *__restrict__ hs, int64_t n, int32_t b,
    const __grid_constant__ BlockList kept, OutT *__restrict__ dX, int64_t ldx) {
    __shared__ float4 tile[kUtRows][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i0 = (int64_t)blockIdx.x * kUtRows, r0 = (int64_t)blockIdx.y * 128;
    const bool live = r0 + 4 * lane < m;                 // the pitch is a multiple of 4 that holds m
    const uint64_t base = reinterpret_cast<uint64_t>(Tt + (live ? r0 + 4 * lane : r0));
    const uint32_t row_bytes = (uint32_t)(4 * ldt);      // the launch keeps 4 ldt below 2^32
    const uint64_t block_bytes = (uint64_t)b * row_bytes;
    // Warp w: rows 8w .. 8w + 7 of the tile, four at a time.  Lane 4q + u holds the table
    // entry of kept block t0 + q and row u of the four: one load per four blocks, issued
    // ahead, so that no row piece waits for its own entry.
    auto entries = [&](int h, int t0) -> uint32_t {
        const int t = t0 + (lane >> 2);
        const int64_t i = i0 + 8 * warp + 4 * h + (lane & 3);
        return lane < 16 && t < kept.count && i < n ? __ldg(hs + (int64_t)kept.idx[t] * n + i) : 0u;
    };
    uint32_t first[2] = {entries(0, 0), entries(1, 0)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        f32x2 acc[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u][0] = acc[u][1] = 0;
        uint32_t e = first[h];
        uint64_t bt = base;                               // row 0 of kept block t
        // kept blocks t0 + q .. + Q - 1: 4 Q loads per lane in flight
        auto blocks = [&](auto qq, int q) {
            constexpr int Q = decltype(qq)::value;
            uint32_t v[4 * Q];
            uint4 x[4 * Q];
#pragma unroll
            for (int k = 0; k < 4 * Q; ++k) {
                v[k] = __shfl_sync(0xffffffffu, e, 4 * q + k);
                const uint64_t row = (k >> 2) ? bt + block_bytes : bt;
                x[k] = __ldg(reinterpret_cast<const uint4 *>((uint64_t)(v[k] & kIndexMask) * row_bytes + row));
            }
#pragma unroll
            for (int k = 0; k < 4 * Q; ++k) {
                const float sg = __uint_as_float(0x3f800000u | (v[k] & kSignBit));
                const f32x2 w2 = pack2(sg, sg);
                fma2(acc[k & 3][0], w2, Pairs<float>::get(x[k], 0));
                fma2(acc[k & 3][1], w2, Pairs<float>::get(x[k], 1));
            }
            bt += Q * block_bytes;
        };
        for (int t0 = 0; t0 < kept.count; t0 += 4) {
            const uint32_t next = t0 + 4 < kept.count ? entries(h, t0 + 4) : 0u;
            const int left = kept.count - t0;
            if (left >= 2) blocks(std::integral_constant<int, 2>(), 0);
            if (left >= 4) blocks(std::integral_constant<int, 2>(), 2);
            else if (left == 3) blocks(std::integral_constant<int, 1>(), 2);
            else if (left == 1) blocks(std::integral_constant<int, 1>(), 0);
            e = next;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float4 o;
            unpack2(acc[u][0], o.x, o.y);
            unpack2(acc[u][1], o.z, o.w);
            tile[8 * warp + 4 * h + u][lane ^ ((4 * h + u) ^ warp)] = o;   // i = 8 warp + 4 h + u
        }
    }
    __syncthreads();
    // chunk c of r's: 4 per warp
    const float *flat = reinterpret_cast<const float *>(tile);
    if constexpr (!kVec) {
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            const int c = 4 * warp + (k >> 2), w = k & 3;
            const int64_t r = r0 + 4 * c + w;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int i = 32 * half + lane;
                const float y = flat[i * 128 + 4 * (c ^ ((i ^ (i >> 3)) & 7)) + w];
                if (r < m && i0 + i < n) {
                    if constexpr (sizeof(OutT) == 4) dX[r * ldx + i0 + i] = y;
                    else dX[r * ldx + i0 + i] = __float2bfloat16_rn(y);
                }
            }
        }
        return;
    }
    // lane: r = 4c + lane % 4, i = 8 (lane / 4) .. + 7
    const int w = lane & 3, ig = lane >> 2;
    const int64_t i = i0 + 8 * ig;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = 4 * warp + k;
        const int64_t r = r0 + 4 * c + w;
        float y[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) y[s] = flat[(8 * ig + s) * 128 + 4 * (c ^ (s ^ ig)) + w];
        if (r >= m) continue;
        OutT *dst = dX + r * ldx + i;
        if (i + 8 <= n) {
            if constexpr (sizeof(OutT) == 4) {
                reinterpret_cast<float4 *>(dst)[0] = make_float4(y[0], y[1], y[2], y[3]);
                reinterpret_cast<float4 *>(dst)[1] = make_float4(y[4], y[5], y[6], y[7]);
            } else {
                const __nv_bfloat162 q[4] = {__floats2bfloat162_rn(y[0], y[1]), __floats2bfloat162_rn(y[2], y[3]),
                                             __floats2bfloat162_rn(y[4], y[5]), __floats2bfloat162_rn(y[6], y[7])};
                *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(q);
            }
        } else {
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                if (i + s >= n) break;
                if constexpr (sizeof(OutT) == 4) dst[s] = y[s];
                else dst[s] = __float2bfloat16_rn(y[s]);
            }
        }
    }
}

// The signed scale of every entry of the listed blocks' padded bucket lists,
// in list order: w[j][pos] = sigma_j(i) * s_i for the entry (i, sigma) at pos
// (0 for padding), so the gather loads the weights of 32 entries with one
// coalesced load instead of 32 scattered loads of s.
__global__ void __launch_bounds__(256) entry_weights_kernel(const uint32_t *__restrict__ pperm,
                                                            const uint32_t *__restrict__ poffs, int64_t pstride,
                                                            int32_t b, const float *__restrict__ s,
                                                            BlockList blocks, float *__restrict__ w) {
    const int j = blocks.idx[blockIdx.y];
    const int64_t len = __ldg(poffs + (int64_t)j * (b + 1) + b);     // padded list length
    const uint32_t *pl = pperm + (int64_t)j * pstride;
    float *wl = w + (int64_t)j * pstride;
    for (int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; pos < len;
         pos += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t ent = __ldg(pl + pos);
        wl[pos] = ent == kPadEntry ? 0.f
                                   : __uint_as_float(__float_as_uint(__ldg(s + (ent & kIndexMask))) ^ (ent & kSignBit));
    }
}

os_status launch_entry_weights(const Plan *p, const float *s, uint64_t block_mask, float *w, cudaStream_t st) {
    const BlockList blocks = mask_to_list(block_mask ? block_mask : ~0ull, p->P);
    const int64_t per = (p->pstride + 255) / 256;
    dim3 grid((unsigned)(per < 1024 ? per : 1024), (unsigned)blocks.count);
    entry_weights_kernel<<<grid, 256, 0, st>>>(p->pperm, p->poffs, p->pstride, p->b, s, blocks, w);
    return check_launch();
}

// FP8 codes and UE8M0 scales from FP32 sums staged in global memory; the same rule
// as the gather's fused FP8 epilogue (smallest e with amax <= 448 * 2^e, codes =
// RNE(x / 2^e)), so the codes and scales are the same bits.  A warp quantises Q
// consecutive 128-column slices of a row at once, the warps of the grid one after the
// other over the slices of all rows.  Memory-bound: one slice per warp (16 bytes per lane
// in flight) ran at 3.2 TB/s on GB300, and the two quantisations of an 8192 x 32768 x 8192
// product took about 50 us longer together.  Q = 1 while all slices have a warp on the
// GPU at once (left sketch of 8 x 20001, 8 blocks of 640: 14.4 us, with Q = 4 16.4).  Turns
// are dealt over all rows: a CTA per row left most warps idle where a row has few slices
// (700 x 8192 x 700 FP8 product with 3: 61.6 us against 58.5).
constexpr int kQuant = 4;

template <int Q_>
__global__ void __launch_bounds__(256) quantize_fp8_kernel(const float *__restrict__ Y, int64_t ldy, int64_t rows,
                                                           int32_t b, BlockList blocks,
                                                           __nv_fp8_e4m3 *__restrict__ Q, int64_t ldq,
                                                           float *__restrict__ scales, int64_t lds) {
    const int lane = threadIdx.x & 31;
    const int spb = b / 128;                       // slices per block
    const int per_row = blocks.count * spb;
    const uint32_t per = (uint32_t)((per_row + Q_ - 1) / Q_);   // warps' turns per row
    const int64_t total = rows * per, step = (int64_t)gridDim.x * 8;
    for (int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); w < total; w += step) {
        const int64_t r = total < (int64_t(1) << 32) ? (int64_t)((uint32_t)w / per) : w / per;
        const int s0 = (int)(w - r * per) * Q_;
        float4 v[Q_];
        int64_t q0[Q_];
#pragma unroll
        for (int u = 0; u < Q_; ++u) {
            const int s = min(s0 + u, per_row - 1);
            const int bt = s / spb;
            q0[u] = (int64_t)blocks.idx[bt] * b + (int64_t)(s - bt * spb) * 128;
            v[u] = __ldcs(reinterpret_cast<const float4 *>(Y + r * ldy + q0[u]) + lane);
        }
#pragma unroll
        for (int u = 0; u < Q_; ++u) {
            if (s0 + u >= per_row) break;
            float a = fmaxf(fmaxf(fabsf(v[u].x), fabsf(v[u].y)), fmaxf(fabsf(v[u].z), fabsf(v[u].w)));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
            const int e = fp8_scale_exponent(a);
            const float inv = ldexpf(1.f, -e);
            __nv_fp8_e4m3 c[4] = {__nv_fp8_e4m3(v[u].x * inv), __nv_fp8_e4m3(v[u].y * inv),
                                  __nv_fp8_e4m3(v[u].z * inv), __nv_fp8_e4m3(v[u].w * inv)};
            *reinterpret_cast<uint32_t *>(Q + r * ldq + q0[u] + 4 * lane) = *reinterpret_cast<const uint32_t *>(c);
            if (lane == 0) scales[(q0[u] / 128) * lds + r] = ldexpf(1.f, e);   // slice-major
        }
    }
}

os_status launch_quantize_fp8(const Plan *p, const float *Y, int64_t ldy, int64_t rows, uint64_t block_mask,
                              void *Q, int64_t ldq, float *scales, int64_t lds, cudaStream_t st) {
    const BlockList blocks = mask_to_list(block_mask ? block_mask : ~0ull, p->P);
    const int64_t per_row = (int64_t)blocks.count * (p->b / 128);
    const bool one = rows * per_row <= 152 * 64;
    const int64_t ctas = (rows * (one ? per_row : (per_row + kQuant - 1) / kQuant) + 7) / 8;
    auto k = one ? quantize_fp8_kernel<1> : quantize_fp8_kernel<kQuant>;
    k<<<(unsigned)(ctas < 152 * 64 ? ctas : 152 * 64), 256, 0, st>>>(Y, ldy, rows, p->b, blocks, (__nv_fp8_e4m3 *)Q, ldq,
                                                                   scales, lds);
    return check_launch();
}

// A strip is first read from DRAM and then, by its other blocks' CTAs, from L2, and its
// CTAs sweep their lists in step.  Dealing the next strip's first block out between
// them overlaps the two, as long as two strips fit in L2 with room to spare.  GB300,
// FP32 rows with scales, 20 blocks of 1024: 965 -> 918 us for 40960 x 5120 (strips of
// 21 MB), 30 blocks of 512: 983 -> 956 for 30720 x 5120; strips of 33 MB gain nothing
// and larger ones lose (without scales, 64 MB: 429 -> 507 us).
constexpr int64_t kMixBytes = int64_t(24) << 20;

template <typename InT, typename OutT, int QT, int SLOTS, bool kMis = false>
os_status launch_gather_t(const Plan *p, const InT *X, int64_t strip_stride, int64_t ldx, int64_t F,
                          const float *wts, void *Yt, int64_t ldy, float *scales, int64_t scale_ld,
                          const BlockList &blocks, cudaStream_t st, int64_t plane_elems = 0,
                          const uint64_t *dmask = nullptr) {
    const int z = p->P * p->b;
    const int tpb = (p->b + QT - 1) / QT;
    constexpr int TF = strip_of<InT>() / SLOTS;
    constexpr int TFO = kMis ? TF - 4 : TF;   // free indices written per CTA
    dim3 grid((unsigned)(tpb * blocks.count), (unsigned)((F + TFO - 1) / TFO));
    if (grid.y > 65535u) return OS_ERR_UNSUPPORTED;
    const size_t smem = sizeof(float) * QT * (TF + 1);
    const bool mix = wts && !kMis && sizeof(InT) == 4 && sizeof(OutT) != 1 && blocks.count > 1 && grid.y > 1 &&
                     p->n * (int64_t)(TF * sizeof(InT)) <= kMixBytes;
    auto k = wts ? sketch_gather_kernel<InT, OutT, QT, true, SLOTS, kMis>
                       : sketch_gather_kernel<InT, OutT, QT, false, SLOTS, kMis>;
    if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if constexpr (sizeof(OutT) == 1) {
        // clusters of the 4 CTAs of a 128-column scale slice (b % 128 == 0, so
        // grid.x is a multiple of 4 and no cluster straddles two blocks)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(kWarps * 32);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 4;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        OSK_CUDA_TRY(cudaLaunchKernelEx(&cfg, k, X, strip_stride, ldx, F, (const uint32_t *)p->pperm,
                                        (const uint32_t *)p->poffs, p->pstride, p->b, z, wts, (OutT *)Yt, ldy,
                                        scales, scale_ld, blocks, tpb, plane_elems, dmask));
    } else {
        k<<<grid, kWarps * 32, smem, st>>>(X, strip_stride, ldx, F, p->pperm, p->poffs, p->pstride, p->b, z,
                                          wts, (OutT *)Yt, ldy, scales, scale_ld, blocks, mix ? -tpb : tpb, plane_elems, dmask);
    }
    return check_launch();
}

// Gather from an operand packed in 128-wide strips (n rows each) in tiles of
// 32 sketched columns, which keeps the CTAs that run together on few strips.
// Sketched columns per gather CTA (FP8 outputs: 32, the quarter of a scale slice).
// 16 puts 512 CTAs on each strip of the square workload (b = 1024, 8 kept
// blocks), so fewer strips are in flight at once than with 32 and more of the
// gathered rows hit L2 (right sketch 1.89 -> 1.74 ms on GB300).
constexpr int kGatherQT = 16;

// ss, W: the distance between strips and between rows of a strip (elements);
// the defaults are the packed workspace layout.
template <typename InT>
os_status launch_gather(const Plan *p, const InT *Xs, int64_t F, const float *wts, void *Yt,
                        os_dtype out_t, int64_t ldy, float *scales, int64_t scale_ld, uint64_t block_mask,
                        cudaStream_t st, int64_t plane_rows = 0, const uint64_t *dmask = nullptr,
                        int64_t ss = -1, int64_t W = strip_of<InT>()) {
    const BlockList blocks = mask_to_list(block_mask ? block_mask : ~0ull, p->P);
    if (ss < 0) ss = p->n * W;
    switch (out_t) {
        case OS_F32:
            return launch_gather_t<InT, float, kGatherQT, 1>(p, Xs, ss, W, F, wts, Yt, ldy, scales, scale_ld, blocks, st, 0, dmask);
        case OS_BF16:
            return launch_gather_t<InT, __nv_bfloat16, kGatherQT, 1>(p, Xs, ss, W, F, wts, Yt, ldy, scales, scale_ld,
                                                              blocks, st, 0, dmask);
        case OS_FP8E4M3:
            return launch_gather_t<InT, __nv_fp8_e4m3, 32, 1>(p, Xs, ss, W, F, wts, Yt, ldy, scales, scale_ld,
                                                               blocks, st, 0, dmask);
        case OS_TF32X2:
            return launch_gather_t<InT, Tf32Pair, kGatherQT, 1>(p, Xs, ss, W, F, wts, Yt, ldy, scales, scale_ld, blocks,
                                                         st, plane_rows * ldy, dmask);
    }
    return OS_ERR_DTYPE;
}

// Gather straight from a row-major FP32 operand in 128-wide strips (512-byte row
// pieces: one address translation per 512 bytes is cheap enough that no
// packing pass is needed).  F must be a multiple of 128.  With kMis the rows
// need only 4-byte alignment: strips are 124 wide, each lane loads the 16-byte
// granule holding its first element, and the sums are kept per misalignment
// class and realigned once per bucket (F a multiple of 124).
template <bool kMis>
os_status launch_gather_direct(const Plan *p, const float *X, int64_t ldx, int64_t F, const float *wts,
                               void *Yt, os_dtype out_t, int64_t ldy, float *scales, int64_t scale_ld,
                               uint64_t block_mask, cudaStream_t st, int64_t plane_rows = 0,
                               const uint64_t *dmask = nullptr) {
    const BlockList blocks = mask_to_list(block_mask ? block_mask : ~0ull, p->P);
    constexpr int64_t ss = kMis ? kStrip - 4 : kStrip;
    switch (out_t) {
        case OS_F32:
            return launch_gather_t<float, float, kGatherQT, 1, kMis>(p, X, ss, ldx, F, wts, Yt, ldy, nullptr,
                                                                    scale_ld, blocks, st, 0, dmask);
        case OS_BF16:
            return launch_gather_t<float, __nv_bfloat16, kGatherQT, 1, kMis>(p, X, ss, ldx, F, wts, Yt, ldy, nullptr,
                                                                            scale_ld, blocks, st, 0, dmask);
        case OS_FP8E4M3:
            return launch_gather_t<float, __nv_fp8_e4m3, 32, 1, kMis>(p, X, ss, ldx, F, wts, Yt, ldy, scales,
                                                                     scale_ld, blocks, st, 0, dmask);
        case OS_TF32X2:
            return launch_gather_t<float, Tf32Pair, kGatherQT, 1, kMis>(p, X, ss, ldx, F, wts, Yt, ldy, nullptr,
                                                                       scale_ld, blocks, st, plane_rows * ldy, dmask);
    }
    return OS_ERR_DTYPE;
}

template <typename T>
os_status launch_pack_rows(const T *X, int64_t ldx, int64_t n, int64_t F, T *Xs, cudaStream_t st) {
    constexpr int64_t SW = strip_of<T>();
    const int64_t nstrips = (F + SW - 1) / SW;
    const int64_t total = n * nstrips * (SW / (16 / (int64_t)sizeof(T)));
    const int64_t blocks = (total + 255) / 256 < 152 * 64 ? (total + 255) / 256 : 152 * 64;
    const bool vec = aligned16(X) && (ldx * (int64_t)sizeof(T)) % 16 == 0;
    if (vec)
        pack_rows_kernel<T, true><<<(unsigned)blocks, 256, 0, st>>>(X, ldx, n, F, nstrips, Xs);
    else
        pack_rows_kernel<T, false><<<(unsigned)blocks, 256, 0, st>>>(X, ldx, n, F, nstrips, Xs);
    return check_launch();
}

os_status launch_pack_cols(const float *A, int64_t lda, int64_t m, int64_t n, float *Xs, cudaStream_t st) {
    // 32-row blocks of the (zero-padded) strips
    constexpr int64_t SW = strip_of<float>();
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)((m + SW - 1) / SW * (SW / 32)));
    if (grid.y > 65535u) return OS_ERR_UNSUPPORTED;
    if (aligned16(A) && lda % 4 == 0)
        pack_cols_kernel<float, true><<<grid, 256, 0, st>>>(A, lda, m, n, Xs);
    else
        pack_cols_kernel<float, false><<<grid, 256, 0, st>>>(A, lda, m, n, Xs);
    return check_launch();
}

os_status launch_pack_cols(const __nv_bfloat16 *A, int64_t lda, int64_t m, int64_t n, __nv_bfloat16 *Xs,
                           cudaStream_t st) {
    constexpr int64_t SW = strip_of<__nv_bfloat16>();
    const bool rows16 = aligned16(A) && lda % 8 == 0;
    const int64_t w = rows16 ? 128 : 256, h = rows16 ? 64 : 32;   // the kernels' tiles
    dim3 grid((unsigned)((n + w - 1) / w), (unsigned)((m + SW - 1) / SW * (SW / h)));
    if (grid.y > 65535u) return OS_ERR_UNSUPPORTED;
    if (rows16)
        pack_cols_bf16_kernel<<<grid, 256, 0, st>>>(A, lda, m, n, Xs);
    else
        pack_cols_kernel<__nv_bfloat16, false><<<grid, 256, 0, st>>>(A, lda, m, n, Xs);
    return check_launch();
}

os_status check_out(const Plan *p, int64_t rows, void *Yt, os_dtype out_t, int64_t ldy,
                    float *scales) {
    const int64_t z = (int64_t)p->P * p->b;
    if (rows < 0) return OS_ERR_INVALID_ARG;
    if (out_t != OS_F32 && out_t != OS_BF16 && out_t != OS_FP8E4M3 && out_t != OS_TF32X2) return OS_ERR_DTYPE;
    if (ldy < z || (ldy * (int64_t)dtype_size(out_t)) % 16 != 0) return OS_ERR_INVALID_ARG;
    if (out_t == OS_FP8E4M3 && p->b % 128 != 0) return OS_ERR_UNSUPPORTED;
    if (rows == 0) return OS_OK;   // an empty output: nothing is written
    if (!Yt || !aligned16(Yt)) return OS_ERR_INVALID_ARG;
    if (out_t == OS_FP8E4M3 && !scales) return OS_ERR_INVALID_ARG;
    return OS_OK;
}

}  // namespace

namespace {
size_t ws_align(size_t x) { return (x + 255) / 256 * 256; }
// ceil(F/128) packed strips of n x 128 elements
size_t strip_bytes(const Plan *p, int64_t F, os_dtype in_t) {
    const int64_t sw = 32 * (16 / (int64_t)dtype_size(in_t));   // strip_of<> of the element type
    return (size_t)((F + sw - 1) / sw) * sw * (size_t)p->n * dtype_size(in_t);
}
}  // namespace

// Sketch workspace for F free indices: the packed strips, then the signed
// scale of every bucket-list entry (P x pstride FP32, used by scaled sketches).
size_t sketch_workspace_bytes(const Plan *p, int64_t F, os_dtype in_t) {
    return ws_align(strip_bytes(p, F, in_t)) + (size_t)p->P * p->pstride * sizeof(float) + 256;
}

// FP8 output staged in FP32: a workspace this much larger (F x z FP32 sums after the
// regular workspace) lets the sketch gather FP32 sums without clusters and quantise
// them in a second pass (same codes and scales as the fused FP8 epilogue).
size_t fp8_staging_bytes(const Plan *p, int64_t F) { return (size_t)F * (size_t)p->P * p->b * sizeof(float) + 256; }

namespace {
float *fp8_staging(const Plan *p, void *ws, size_t ws_bytes, int64_t F, os_dtype in_t) {
    const size_t off = ws_align(sketch_workspace_bytes(p, F, in_t));
    if (!ws || ws_bytes < off + fp8_staging_bytes(p, F)) return nullptr;
    const uintptr_t a = (reinterpret_cast<uintptr_t>(ws) + off + 255) & ~uintptr_t(255);
    return reinterpret_cast<float *>(a);
}
}  // namespace

namespace {
void *ws_base(void *ws) {
    return reinterpret_cast<void *>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255));
}
// the entry weights of a workspace whose strips hold F free indices
float *ws_weights(const Plan *p, void *ws, int64_t F, os_dtype in_t) {
    return reinterpret_cast<float *>(reinterpret_cast<char *>(ws_base(ws)) + ws_align(strip_bytes(p, F, in_t)));
}
// the entry weights for scale s (NULL without a scale)
os_status make_weights(const Plan *p, const float *s, uint64_t block_mask, float *w, const float **out,
                       cudaStream_t st) {
    *out = nullptr;
    if (!s) return OS_OK;
    OSK_TRY(launch_entry_weights(p, s, block_mask, w, st));
    *out = w;
    return OS_OK;
}
}  // namespace

// The argument checks of the left sketch that need no workspace (OS_OK for a
// valid call, including an empty output m == 0).
os_status sketch_left_check(const Plan *p, const void *A, os_dtype a_t, int64_t m, int64_t lda, void *At,
                            os_dtype out_t, int64_t ldat, float *scales, uint64_t block_mask) {
    if (!p || m < 0) return OS_ERR_INVALID_ARG;
    if (block_mask) OSK_TRY(check_mask(block_mask, p->P));
    if (a_t != OS_F32 && a_t != OS_BF16) return OS_ERR_DTYPE;
    if (lda < p->n) return OS_ERR_INVALID_ARG;
    OSK_TRY(check_out(p, m, At, out_t, ldat, scales));
    if (m == 0) return OS_OK;
    if (!A) return OS_ERR_INVALID_ARG;
    return OS_OK;
}

os_status sketch_left_impl(const Plan *p, const void *A, os_dtype a_t, int64_t m, int64_t lda,
                           void *At, os_dtype out_t, int64_t ldat, float *scales,
                           const float *col_scale, uint64_t block_mask, void *ws, size_t ws_bytes,
                           cudaStream_t st, const uint64_t *dmask = nullptr) {
    OSK_NVTX("sketch_left");
    OSK_TRY(sketch_left_check(p, A, a_t, m, lda, At, out_t, ldat, scales, block_mask));
    if (m == 0) return OS_OK;
    if (!ws || ws_bytes < sketch_workspace_bytes(p, m, a_t)) return OS_ERR_WORKSPACE;
    if (out_t == OS_FP8E4M3 && !dmask) {
        if (float *stg = fp8_staging(p, ws, ws_bytes, m, a_t)) {
            const int64_t z = (int64_t)p->P * p->b;
            OSK_TRY(sketch_left_impl(p, A, a_t, m, lda, stg, OS_F32, z, nullptr, col_scale, block_mask, ws, ws_bytes,
                                     st, dmask));
            return launch_quantize_fp8(p, stg, z, m, block_mask, At, ldat, scales, fp8_scale_ld(m), st);
        }
    }
    void *Xs = ws_base(ws);
    const float *wts = nullptr;
    OSK_TRY(make_weights(p, col_scale, block_mask, ws_weights(p, ws, m, a_t), &wts, st));
    if (a_t == OS_F32) {
        OSK_TRY(launch_pack_cols((const float *)A, lda, m, p->n, (float *)Xs, st));
        return launch_gather<float>(p, (const float *)Xs, m, wts, At, out_t, ldat, scales, fp8_scale_ld(m),
                                    block_mask, st, m, dmask);
    }
    OSK_TRY(launch_pack_cols((const __nv_bfloat16 *)A, lda, m, p->n, (__nv_bfloat16 *)Xs, st));
    return launch_gather<__nv_bfloat16>(p, (const __nv_bfloat16 *)Xs, m, wts, At, out_t, ldat, scales,
                                        fp8_scale_ld(m), block_mask, st, m, dmask);
}

os_status sketch_right_impl(const Plan *p, const void *B, os_dtype b_t, int64_t l, int64_t ldb,
                            void *BtT, os_dtype out_t, int64_t ldbt, float *scales, uint64_t block_mask,
                            void *ws, size_t ws_bytes, cudaStream_t st, const float *row_scale = nullptr,
                            const uint64_t *dmask = nullptr) {
    OSK_NVTX("sketch_right");
    if (!p || l < 0) return OS_ERR_INVALID_ARG;
    if (block_mask) OSK_TRY(check_mask(block_mask, p->P));
    if (b_t != OS_F32 && b_t != OS_BF16) return OS_ERR_DTYPE;
    if (ldb < l) return OS_ERR_INVALID_ARG;
    OSK_TRY(check_out(p, l, BtT, out_t, ldbt, scales));
    if (l == 0) return OS_OK;
    if (!B) return OS_ERR_INVALID_ARG;
    if (out_t == OS_FP8E4M3 && !dmask) {
        if (float *stg = fp8_staging(p, ws, ws_bytes, l, b_t)) {
            const int64_t z = (int64_t)p->P * p->b;
            OSK_TRY(sketch_right_impl(p, B, b_t, l, ldb, stg, OS_F32, z, nullptr, block_mask, ws, ws_bytes, st,
                                      row_scale, dmask));
            return launch_quantize_fp8(p, stg, z, l, block_mask, BtT, ldbt, scales, fp8_scale_ld(l), st);
        }
    }
    // FP32 input: gather whole strips in place, and pack only a ragged remainder
    // narrower than a strip.  Strips are 128 wide for 16-byte aligned rows; other
    // rows are gathered in 124-wide strips (about twice the instructions per row
    // piece: on GB300 that beats packing B first while at most 6 blocks are
    // gathered, 1.82 vs 2.35 ms for 4 blocks of 65536 x 16383, and loses above,
    // 3.28 vs 3.01 ms for 8 blocks).
    const bool aligned = aligned16(B) && ldb % 4 == 0;
    const uint64_t listed = (block_mask ? block_mask : ~0ull) & (p->P >= 64 ? ~0ull : (1ull << p->P) - 1);
    const bool mis_pays = __builtin_popcountll(listed) <= 6;
    const int64_t sw = aligned ? kStrip : kStrip - 4;
    // (a misaligned strip reads up to 4 elements past its end: keep them in the row)
    const int64_t lf = aligned ? l / sw * sw : (l >= 4 ? (l - 4) / sw * sw : 0);
    const bool direct = b_t == OS_F32 && (reinterpret_cast<uintptr_t>(B) & 3u) == 0 &&
                        ldb * 4 < (int64_t(1) << 32) && lf > 0 && (aligned || mis_pays);
    if (direct) {
        // the workspace holds the remainder's strips (if any) and the entry weights
        if ((lf < l || row_scale) && (!ws || ws_bytes < sketch_workspace_bytes(p, l - lf, b_t)))
            return OS_ERR_WORKSPACE;
        const float *wts = nullptr;
        if (row_scale) OSK_TRY(make_weights(p, row_scale, block_mask, ws_weights(p, ws, l - lf, b_t), &wts, st));
        if (aligned)
            OSK_TRY(launch_gather_direct<false>(p, (const float *)B, ldb, lf, wts, BtT, out_t, ldbt, scales,
                                                fp8_scale_ld(l), block_mask, st, l, dmask));
        else
            OSK_TRY(launch_gather_direct<true>(p, (const float *)B, ldb, lf, wts, BtT, out_t, ldbt, scales,
                                               fp8_scale_ld(l), block_mask, st, l, dmask));
        if (lf == l) return OS_OK;
        float *Xs = (float *)ws_base(ws);
        OSK_TRY(launch_pack_rows<float>((const float *)B + lf, ldb, p->n, l - lf, Xs, st));
        char *yt = (char *)BtT + (size_t)lf * ldbt * dtype_size(out_t);
        float *sc = scales ? scales + lf : nullptr;   // slice-major: the remainder's rows start at lf
        return launch_gather<float>(p, Xs, l - lf, wts, yt, out_t, ldbt, sc, fp8_scale_ld(l), block_mask, st, l, dmask);
    }
    // BF16 input with 16-byte aligned rows: 256-wide strips gathered in place (the
    // same 512-byte row pieces as a packed strip), a ragged remainder packed
    constexpr int64_t sw16 = strip_of<__nv_bfloat16>();
    const int64_t lf16 = l / sw16 * sw16;
    if (b_t == OS_BF16 && aligned16(B) && ldb % 8 == 0 && ldb * 2 < (int64_t(1) << 32) && lf16 > 0) {
        if ((lf16 < l || row_scale) && (!ws || ws_bytes < sketch_workspace_bytes(p, l - lf16, b_t)))
            return OS_ERR_WORKSPACE;
        const float *wts = nullptr;
        if (row_scale) OSK_TRY(make_weights(p, row_scale, block_mask, ws_weights(p, ws, l - lf16, b_t), &wts, st));
        const __nv_bfloat16 *Bh = (const __nv_bfloat16 *)B;
        OSK_TRY(launch_gather<__nv_bfloat16>(p, Bh, lf16, wts, BtT, out_t, ldbt, scales, fp8_scale_ld(l), block_mask,
                                             st, l, dmask, sw16, ldb));
        if (lf16 == l) return OS_OK;
        __nv_bfloat16 *Xs = (__nv_bfloat16 *)ws_base(ws);
        OSK_TRY(launch_pack_rows<__nv_bfloat16>(Bh + lf16, ldb, p->n, l - lf16, Xs, st));
        char *yt = (char *)BtT + (size_t)lf16 * ldbt * dtype_size(out_t);
        float *sc = scales ? scales + lf16 : nullptr;
        return launch_gather<__nv_bfloat16>(p, Xs, l - lf16, wts, yt, out_t, ldbt, sc, fp8_scale_ld(l), block_mask,
                                            st, l, dmask);
    }
    if (!ws || ws_bytes < sketch_workspace_bytes(p, l, b_t)) return OS_ERR_WORKSPACE;
    void *Xs = ws_base(ws);
    const float *wts = nullptr;
    OSK_TRY(make_weights(p, row_scale, block_mask, ws_weights(p, ws, l, b_t), &wts, st));
    if (b_t == OS_F32) {
        OSK_TRY(launch_pack_rows<float>((const float *)B, ldb, p->n, l, (float *)Xs, st));
        return launch_gather<float>(p, (const float *)Xs, l, wts, BtT, out_t, ldbt, scales, fp8_scale_ld(l),
                                    block_mask, st, l, dmask);
    }
    OSK_TRY(launch_pack_rows<__nv_bfloat16>((const __nv_bfloat16 *)B, ldb, p->n, l, (__nv_bfloat16 *)Xs, st));
    return launch_gather<__nv_bfloat16>(p, (const __nv_bfloat16 *)Xs, l, wts, BtT, out_t, ldbt, scales,
                                        fp8_scale_ld(l), block_mask, st, l, dmask);
}

os_status unsketch_cols_impl(const Plan *p, const float *T, int64_t m, int64_t ldt, uint64_t mask,
                             float scale, void *dX, os_dtype x_t, int64_t ldx, cudaStream_t st) {
    if (!p || m < 0) return OS_ERR_INVALID_ARG;
    OSK_TRY(check_mask(mask, p->P));
    const int kcnt = __builtin_popcountll(mask);
    if (ldt < (int64_t)kcnt * p->b || ldx < p->n) return OS_ERR_INVALID_ARG;
    if (x_t != OS_F32 && x_t != OS_BF16) return OS_ERR_DTYPE;
    if (m == 0) return OS_OK;   // an empty dX
    if (!T || !dX) return OS_ERR_INVALID_ARG;
    const BlockList kept = mask_to_list(mask, p->P);
    // rows of T staged per CTA (1024 threads): 4, 2 or 1, the most that fit in
    // 200 KB, else the unstaged kernel
    const int64_t kb = (int64_t)kcnt * p->b;
    const size_t row_bytes = (size_t)kb * sizeof(float);
    const int R = row_bytes * 4 <= 200 * 1024 ? 4 : row_bytes * 2 <= 200 * 1024 ? 2 : row_bytes <= 200 * 1024 ? 1 : 0;
    if (R > 0) {
        const size_t smem = row_bytes * R;
        const unsigned gxs = (unsigned)((m + R - 1) / R);
        auto launch = [&](auto kern, auto *out) -> os_status {
            if (smem > 48 * 1024)
                OSK_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            kern<<<gxs, 1024, smem, st>>>(T, m, ldt, kb, p->hs, p->n, p->b, kept, scale, out, ldx);
            return check_launch();
        };
        if (x_t == OS_F32) {
            float *o = (float *)dX;
            if (R == 4) return launch(unsketch_cols_smem_kernel<float, 4>, o);
            if (R == 2) return launch(unsketch_cols_smem_kernel<float, 2>, o);
            return launch(unsketch_cols_smem_kernel<float, 1>, o);
        }
        __nv_bfloat16 *o = (__nv_bfloat16 *)dX;
        if (R == 4) return launch(unsketch_cols_smem_kernel<__nv_bfloat16, 4>, o);
        if (R == 2) return launch(unsketch_cols_smem_kernel<__nv_bfloat16, 2>, o);
        return launch(unsketch_cols_smem_kernel<__nv_bfloat16, 1>, o);
    }
    if (m > 65535) return OS_ERR_UNSUPPORTED;
    const int64_t gx = (p->n + 255) / 256 < 1024 ? (p->n + 255) / 256 : 1024;
    dim3 grid((unsigned)gx, (unsigned)m);
    if (x_t == OS_F32)
        unsketch_cols_kernel<float><<<grid, 256, 0, st>>>(T, m, ldt, p->hs, p->n, p->b, kept, scale,
                                                          (float *)dX, ldx);
    else
        unsketch_cols_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(T, m, ldt, p->hs, p->n, p->b, kept,
                                                                  scale, (__nv_bfloat16 *)dX, ldx);
    return check_launch();
}

os_status unsketch_rows_impl(const Plan *p, const float *U, int64_t l, int64_t ldu, uint64_t mask,
                             float scale, void *dG, os_dtype g_t, int64_t ldg, cudaStream_t st) {
    if (!p || l < 0) return OS_ERR_INVALID_ARG;
    OSK_TRY(check_mask(mask, p->P));
    if (ldu < l || ldg < l) return OS_ERR_INVALID_ARG;
    if (g_t != OS_F32 && g_t != OS_BF16) return OS_ERR_DTYPE;
    if (l == 0) return OS_OK;   // an empty dG
    if (!U || !dG) return OS_ERR_INVALID_ARG;
    const BlockList kept = mask_to_list(mask, p->P);
    dim3 grid((unsigned)((p->n + 7) / 8), (unsigned)((l + 1023) / 1024));
    if (grid.y > 65535u) return OS_ERR_UNSUPPORTED;
    const bool vec = l % 4 == 0 && ldu % 4 == 0 && ldg % 4 == 0 && aligned16(U) && aligned16(dG);
    if (g_t == OS_F32) {
        if (vec)
            unsketch_rows_vec_kernel<float><<<grid, 256, 0, st>>>(U, l, ldu, p->hs, p->n, p->b, kept, scale,
                                                                  (float *)dG, ldg);
        else
            unsketch_rows_kernel<float><<<grid, 256, 0, st>>>(U, l, ldu, p->hs, p->n, p->b, kept, scale,
                                                              (float *)dG, ldg);
    } else {
        if (vec)
            unsketch_rows_vec_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(U, l, ldu, p->hs, p->n, p->b, kept,
                                                                          scale, (__nv_bfloat16 *)dG, ldg);
        else
            unsketch_rows_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(U, l, ldu, p->hs, p->n, p->b, kept,
                                                                      scale, (__nv_bfloat16 *)dG, ldg);
    }
    return check_launch();
}

// dX (m x n) from the transposed kept blocks Tt (kb x m, pitch ldt < 2^30, a multiple of 4).
os_status unsketch_cols_t_impl(const Plan *p, const float *Tt, int64_t m, int64_t ldt, uint64_t mask, void *dX,
                               os_dtype x_t, int64_t ldx, cudaStream_t st) {
    const BlockList kept = mask_to_list(mask, p->P);
    if (ldt % 4 != 0 || ldt >= (int64_t(1) << 30) || !aligned16(Tt)) return OS_ERR_UNSUPPORTED;
    auto launch = [&](auto *out) -> os_status {
        using O = typename std::remove_pointer<decltype(out)>::type;
        const bool vec = aligned16(dX) && (ldx * (int64_t)sizeof(O)) % 16 == 0;
        auto k = vec ? unsketch_cols_t_kernel<O, true> : unsketch_cols_t_kernel<O, false>;
        constexpr int64_t kRows = 65535 * int64_t(128);   // rows of dX per launch (grid.y)
        for (int64_t r = 0; r < m; r += kRows) {
            const int64_t rows = m - r < kRows ? m - r : kRows;
            const dim3 grid((unsigned)((p->n + kUtRows - 1) / kUtRows), (unsigned)((rows + 127) / 128));
            k<<<grid, 256, 0, st>>>(Tt + r, rows, ldt, p->hs, p->n, p->b, kept, out + r * ldx, ldx);
            OSK_TRY(check_launch());
        }
        return OS_OK;
    };
    return x_t == OS_F32 ? launch((float *)dX) : launch((__nv_bfloat16 *)dX);
}

}  // namespace osk

using namespace osk;

extern "C" os_status oversketch_sketch_workspace(oversketch_plan_t plan, int64_t free_extent,
                                                 os_dtype in_t, size_t *bytes) {
    const Plan *p = reinterpret_cast<const Plan *>(plan);
    if (!p || !bytes || free_extent < 0) return OS_ERR_INVALID_ARG;
    if (in_t != OS_F32 && in_t != OS_BF16) return OS_ERR_DTYPE;
    *bytes = sketch_workspace_bytes(p, free_extent, in_t);
    return OS_OK;
}

extern "C" os_status oversketch_sketch_left(oversketch_plan_t plan, const void *A, os_dtype a_t,
                                            int64_t m, int64_t lda, void *At, os_dtype out_t,
                                            int64_t ldat, float *scales, const float *col_scale,
                                            uint64_t block_mask, void *workspace, size_t ws_bytes,
                                            void *stream) {
    return sketch_left_impl(reinterpret_cast<const Plan *>(plan), A, a_t, m, lda, At, out_t, ldat,
                            scales, col_scale, block_mask, workspace, ws_bytes, as_stream(stream));
}

extern "C" os_status oversketch_sketch_right(oversketch_plan_t plan, const void *B, os_dtype b_t,
                                             int64_t l, int64_t ldb, void *BtT, os_dtype out_t,
                                             int64_t ldbt, float *scales, const float *row_scale,
                                             uint64_t block_mask, void *workspace, size_t ws_bytes,
                                             void *stream) {
    return sketch_right_impl(reinterpret_cast<const Plan *>(plan), B, b_t, l, ldb, BtT, out_t, ldbt,
                             scales, block_mask, workspace, ws_bytes, as_stream(stream), row_scale);
}

extern "C" os_status oversketch_unsketch_cols(oversketch_plan_t plan, const float *T, int64_t m,
                                              int64_t ldt, uint64_t mask, float scale, void *dX,
                                              os_dtype x_t, int64_t ldx, void *stream) {
    OSK_NVTX("unsketch_cols");
    return unsketch_cols_impl(reinterpret_cast<const Plan *>(plan), T, m, ldt, mask, scale, dX, x_t,
                              ldx, as_stream(stream));
}

extern "C" os_status oversketch_unsketch_rows(oversketch_plan_t plan, const float *U, int64_t l,
                                              int64_t ldu, uint64_t mask, float scale, void *dG,
                                              os_dtype g_t, int64_t ldg, void *stream) {
    OSK_NVTX("unsketch_rows");
    return unsketch_rows_impl(reinterpret_cast<const Plan *>(plan), U, l, ldu, mask, scale, dG, g_t,
                              ldg, as_stream(stream));
}
