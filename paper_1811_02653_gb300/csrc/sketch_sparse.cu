// Left sketch of a sparse operand stored dense (Alg. 4 step 3 / Alg. 5 over the
// nonzeros only: the paper prices sketching at O(nnz(A) (N+e)), Sec. 4).
//
//   At[r, j*b + c] = sum_{i : A[r,i] != 0, h_j(i) = c} sigma_j(i) * s_i * A[r, i]
//
// The dense gather path reads every element k times from L2 (once per kept
// block) and, when a 128-wide strip of the sketched dimension no longer fits in
// L2 (n = 2^20: 512 MB per strip), from DRAM.  Here one CTA per row reads the
// row once, coalesced, and routes only its nonzeros.  Two kernels, one after
// the other:
//
// One-pass kernel (b <= 4096): the whole row's nonzeros are held in shared memory,
// then routed one kept block at a time.  A group of warps (half of the CTA, or all
// of it) owns a row:
//   1. compaction (sp1_compact): each warp streams its share of the row, 16 bytes
//      per lane and load, and appends the nonzeros (index, value) to its own region
//      in ascending index order: ballots only, no block barrier;
//   2. per kept block (sp1_route): bucket codes h_j(i), sigma_j(i) of every entry
//      and the bucket counts (integer shared-memory atomics), a scan into bucket
//      starts, a scatter of entry numbers into their buckets, then each thread
//      sorts the entry numbers of its buckets and adds the members in that order
//      (= ascending index) and writes the sums out in the output dtype (BF16 RNE,
//      FP8 with the per-128-column UE8M0 scale, FP32, or TF32 hi/lo planes).  No
//      float atomics: bitwise reproducible.
//   Two groups of 512 threads share a CTA and take turns at the routing, so that one
//   row streams from HBM while the other is routed; the bucket tables exist once.  Rows
//   of many nonzeros are taken one at a time by all 1024 threads (sp1_groups).
//   A row with more nonzeros in some warp's share than a region holds is left to the
//   flushing kernel: its first kept output gets a marker value.
//   Bound by HBM and instruction issue together.  4096 x 2^20 FP32 at 1 % (17.2 GB,
//   2.54 ms at the copy rate), 6 kept blocks of 4096, with column scales, on GB300: 3.73
//   ms (3.97 before regions of a size known at compile time; 5.47 with an earlier kernel of
//   one row at a time; the compaction alone 2.71).
//   Routing both rows at once, with bucket tables for each group, took 4.28 ms.
//   What the routing's instructions cost decides: predicated accesses in place of
//   branches around them, and sums without branches, gave 4.80 -> 4.02; buckets
//   spread over all lanes (lane i of a warp has buckets i, i + 32, ..) the rest, and
//   at 1024 x 2^20 with blocks of 512 (20 entries a bucket) 3.97 -> 1.87 ms.
//
// Flushing kernel (any density; all rows when b > 4096, else the marked ones):
//   1. compaction: the row streams through registers in chunks of 16 elements
//      per thread (an L2 prefetch runs a few chunks ahead); a block-wide scan
//      appends the nonzeros in ascending index order to an entry buffer;
//   2. flush (buffer full or row done): values take their scale s_i; then for
//      every kept block the entries are counted per bucket, scanned into
//      bucket offsets, scattered into their buckets, and each thread adds the
//      members of its own buckets to their accumulators in ascending index
//      order (the same order as the one-pass kernel: the same bits);
//   3. the row's k*b accumulators are written out in the output dtype.
//   Shared memory holds the k*b accumulators and two b-entry bucket tables:
//   4*k*b + 8*b bytes plus an entry buffer of at least 1024 entries must fit
//   (k*b <= kSparseMaxBuckets).
#include <cstdint>
#include <type_traits>

#include "common.cuh"

namespace osk {

namespace {

constexpr int kSpThreads = 1024;
constexpr int kSpWarps = kSpThreads / 32;
constexpr int kSpElems = 16;                         // elements per thread per chunk
constexpr int kSpChunk = kSpThreads * kSpElems;      // elements per chunk
constexpr int kSpPrefetchChunks = 4;                 // L2 prefetch distance
constexpr int kSmemLimit = 232448;                   // usable shared memory per CTA (227 KB)
constexpr int kEntryBytes = 20;                      // index, value, code, sorted entry, sorted value
constexpr int kMinEntries = 1024;

}  // namespace

// Largest number of kept buckets (k*b) whose accumulators fit beside a useful entry buffer.
constexpr int kSparseMaxBuckets = 32768;

namespace {

// 16 consecutive elements of a row as FP32 (vector loads when aligned, bounds-checked otherwise).
template <typename InT, bool kVec>
__device__ __forceinline__ void load16(const InT *__restrict__ p, int64_t i0, int64_t n, float (&v)[16]) {
    if (kVec && i0 + 16 <= n) {
        if constexpr (std::is_same<InT, float>::value) {
            const float4 *q = reinterpret_cast<const float4 *>(p + i0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 t = __ldcs(q + u);   // streamed: no reuse
                v[4 * u] = t.x; v[4 * u + 1] = t.y; v[4 * u + 2] = t.z; v[4 * u + 3] = t.w;
            }
        } else {
            const uint4 *q = reinterpret_cast<const uint4 *>(p + i0);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint4 t = __ldcs(q + u);
                const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[h]));
                    v[8 * u + 2 * h] = f.x;
                    v[8 * u + 2 * h + 1] = f.y;
                }
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            if (i0 + q < n) {
                if constexpr (std::is_same<InT, float>::value) v[q] = p[i0 + q];
                else v[q] = __bfloat162float(p[i0 + q]);
            } else {
                v[q] = 0.f;
            }
        }
    }
}

// Exclusive block-wide scan of one int per thread (1024 threads); returns the
// thread's offset and writes the total to *total.  Two barriers.
__device__ __forceinline__ int block_scan(int x, int *warp_tot, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int t = warp_tot[lane];
        int ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        warp_tot[32 + lane] = ti - t;            // exclusive warp offsets
        if (lane == 31) warp_tot[64] = ti;
    }
    __syncthreads();
    *total = warp_tot[64];
    return warp_tot[32 + warp] + inc - x;
}

struct SpSmem {
    float *state;        // [k*b] the row's accumulators, block t at t*b
    uint32_t *ent_i;     // [emax] entry index i
    float *ent_v;        // [emax] entry value (scaled by s_i at flush time)
    uint32_t *codes;     // [emax] hs entry of the current block (bucket | sign)
    uint32_t *srt_c;     // [emax] entry numbers grouped by bucket
    float *srt_v;        // [emax] signed values grouped by bucket
    int *bcnt;           // [b] entries per bucket, then the scatter cursor
    int *bstart;         // [b+1] first entry of each bucket in srt_*
    int *warp_tot;       // [72] block-scan scratch
};

// shared memory beyond the accumulators and the entry arrays
__host__ __device__ constexpr size_t sp_fixed_bytes(int b) { return sizeof(int) * ((size_t)2 * b + 1 + 72 + 7); }

__device__ __forceinline__ SpSmem sp_layout(void *base, int kb, int b, int emax) {
    SpSmem s;
    s.state = reinterpret_cast<float *>(base);
    s.ent_i = reinterpret_cast<uint32_t *>(s.state + kb);
    s.ent_v = reinterpret_cast<float *>(s.ent_i + emax);
    s.codes = reinterpret_cast<uint32_t *>(s.ent_v + emax);
    s.srt_c = s.codes + emax;
    s.srt_v = reinterpret_cast<float *>(s.srt_c + emax);
    s.bcnt = reinterpret_cast<int *>(s.srt_v + emax);
    s.bstart = s.bcnt + b;
    s.warp_tot = s.bstart + b + 1;
    return s;
}

constexpr int kSpPerThread = 8;   // entries per thread in a flush (emax <= kSpThreads * kSpPerThread)

// Route the nent buffered entries into the accumulators of every kept block.
// Called by all threads; starts and ends with the buffer stable (barriers).
// Per block: count the entries of every bucket (integer shared-memory atomics),
// scan the counts into bucket offsets, scatter the entry numbers into their
// buckets (in whatever order the atomics give), then every thread adds the
// members of its own buckets in ascending entry order (= ascending index i),
// picking them from the short unordered lists: a fixed order, no float atomics.
template <bool kScale>
__device__ void sp_flush(const SpSmem &s, int nent, const uint32_t *__restrict__ hs, int64_t n, int32_t b,
                         const BlockList &blocks, const float *__restrict__ col_scale, uint64_t seed,
                         bool hashed) {
    const int tid = threadIdx.x;
    if constexpr (kScale) {
        // all of a thread's scale loads in flight at once
        float sc[kSpPerThread];
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u) {
            const int e = tid + u * kSpThreads;
            sc[u] = e < nent ? __ldg(col_scale + s.ent_i[e]) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u) {
            const int e = tid + u * kSpThreads;
            if (e < nent) s.ent_v[e] *= sc[u];
        }
    }
    // bucket codes of the next block, one block ahead: recomputed from the seed for
    // hashed plans (random reads of the table would miss L2 while the operand
    // streams through it), else loaded (the latency hides behind the current block)
    uint32_t nxt[kSpPerThread];
    auto load_codes = [&](int t) {
        if (hashed) {
            const uint64_t key = block_key(seed, blocks.idx[t]);
#pragma unroll
            for (int u = 0; u < kSpPerThread; ++u) {
                const int e = tid + u * kSpThreads;
                nxt[u] = e < nent ? hash_code(key, (int64_t)s.ent_i[e], b) : 0u;
            }
        } else {
            const uint32_t *hj = hs + (int64_t)blocks.idx[t] * n;
#pragma unroll
            for (int u = 0; u < kSpPerThread; ++u) {
                const int e = tid + u * kSpThreads;
                nxt[u] = e < nent ? __ldg(hj + s.ent_i[e]) : 0u;
            }
        }
    };
    load_codes(0);
    for (int t = 0; t < blocks.count; ++t) {
        for (int c = tid; c < b; c += kSpThreads) s.bcnt[c] = 0;
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u) {
            const int e = tid + u * kSpThreads;
            if (e < nent) s.codes[e] = nxt[u];
        }
        __syncthreads();
        if (t + 1 < blocks.count) load_codes(t + 1);
        // counts (the thread's codes stay in registers for the scatter)
        uint32_t code[kSpPerThread];
        float val[kSpPerThread];
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u) {
            const int e = tid + u * kSpThreads;
            code[u] = e < nent ? s.codes[e] : 0u;
            val[u] = e < nent ? s.ent_v[e] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u)
            if (tid + u * kSpThreads < nent) atomicAdd(&s.bcnt[code[u] & kIndexMask], 1);
        __syncthreads();
        // exclusive scan of the b counts: thread t owns a contiguous run of buckets
        const int per = (b + kSpThreads - 1) / kSpThreads;
        const int c0 = min(b, tid * per), c1 = min(b, c0 + per);
        int run = 0;
        for (int c = c0; c < c1; ++c) run += s.bcnt[c];
        int total = 0;
        int off = block_scan(run, s.warp_tot, &total);
        for (int c = c0; c < c1; ++c) {
            const int k = s.bcnt[c];
            s.bstart[c] = off;
            s.bcnt[c] = off;          // cursor for the scatter
            off += k;
        }
        if (tid == 0) s.bstart[b] = total;
        __syncthreads();
        // scatter entry numbers and signed values into their buckets
        int pos[kSpPerThread];
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u)
            pos[u] = tid + u * kSpThreads < nent ? atomicAdd(&s.bcnt[code[u] & kIndexMask], 1) : 0;
#pragma unroll
        for (int u = 0; u < kSpPerThread; ++u) {
            const int e = tid + u * kSpThreads;
            if (e < nent) {
                s.srt_c[pos[u]] = (uint32_t)e;
                s.srt_v[pos[u]] = (code[u] & kSignBit) ? -val[u] : val[u];
            }
        }
        __syncthreads();
        // each bucket's members in ascending entry order, one FP32 chain per bucket
        float *acc = s.state + t * b;
        for (int c = tid; c < b; c += kSpThreads) {
            const int p0 = s.bstart[c], p1 = s.bstart[c + 1];
            if (p0 == p1) continue;
            float a = acc[c];
            if (p1 - p0 == 1) {
                a += s.srt_v[p0];
            } else if (p1 - p0 == 2) {
                const bool swap = s.srt_c[p0] > s.srt_c[p0 + 1];
                const float x0 = s.srt_v[p0], x1 = s.srt_v[p0 + 1];
                a += swap ? x1 : x0;
                a += swap ? x0 : x1;
            } else {
                // longer lists: the members in ascending entry order by repeated minimum
                int last = -1;
                for (int k = p0; k < p1; ++k) {
                    int best = 0x7fffffff, bp = p0;
                    for (int q = p0; q < p1; ++q) {
                        const int eq = (int)s.srt_c[q];
                        if (eq > last && eq < best) best = eq, bp = q;
                    }
                    a += s.srt_v[bp];
                    last = best;
                }
            }
            acc[c] = a;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void l2_prefetch(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)), "r"(bytes)
                 : "memory");
}

template <typename OutT>
__device__ __forceinline__ void sp_store(OutT *dst, int64_t plane_elems, float v) {
    if constexpr (std::is_same<OutT, Tf32Pair>::value) {
        // FP32 as hi + lo: hi keeps 10 mantissa bits (exact in TF32), lo = x - hi (exact)
        float *d = reinterpret_cast<float *>(dst);
        const float hi = __uint_as_float(__float_as_uint(v) & 0xffffe000u);
        d[0] = hi;
        d[plane_elems] = v - hi;
    } else if constexpr (std::is_same<OutT, float>::value) {
        *dst = v;
    } else {
        *dst = __float2bfloat16_rn(v);
    }
}

// The row in flushes (any density): the nonzeros are appended to an entry buffer
// in ascending index order and routed into the k*b accumulators whenever it
// fills; see the file comment.  Starts and ends with all threads in step.
template <typename InT, typename OutT, bool kScale>
__device__ __forceinline__ void sp_row_flushing(const InT *__restrict__ row, int64_t r, int64_t n, bool vec,
                                const uint32_t *__restrict__ hs, uint64_t seed, bool hashed, int32_t b,
                                const BlockList &blocks, int emax, const float *__restrict__ col_scale,
                                OutT *__restrict__ At, int64_t ldat, float *__restrict__ scales, int64_t lds,
                                int64_t plane_elems, void *smem) {
    const int kb = blocks.count * b;
    const SpSmem s = sp_layout(smem, kb, b, emax);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t chunk_bytes = (int64_t)kSpChunk * sizeof(InT);
    for (int q = tid; q < kb; q += kSpThreads) s.state[q] = 0.f;
    int nent = 0;
    for (int64_t base = 0; base < n; base += kSpChunk) {
        if (vec && tid == 0) {
            const int64_t pf = base + (int64_t)kSpPrefetchChunks * kSpChunk;
            if (pf < n) {
                const int64_t bytes = ((n - pf) * (int64_t)sizeof(InT) < chunk_bytes
                                           ? (n - pf) * (int64_t)sizeof(InT) : chunk_bytes) & ~int64_t(15);
                if (bytes > 0) l2_prefetch(row + pf, (uint32_t)bytes);
            }
        }
        float v[kSpElems];
        const int64_t i0 = base + (int64_t)tid * kSpElems;
        if (vec) load16<InT, true>(row, i0, n, v);
        else load16<InT, false>(row, i0, n, v);
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < kSpElems; ++q) cnt += v[q] != 0.f;
        int total = 0;
        const int off = block_scan(cnt, s.warp_tot, &total);
        // append in index order; a chunk with more nonzeros than the buffer holds
        // is appended in pieces, flushing in between
        int done = 0;
        while (done < total) {
            if (nent == emax) {
                sp_flush<kScale>(s, nent, hs, n, b, blocks, col_scale, seed, hashed);
                nent = 0;
            }
            const int take = min(total - done, emax - nent);
            int rank = off;
#pragma unroll
            for (int q = 0; q < kSpElems; ++q) {
                if (v[q] != 0.f) {
                    if (rank >= done && rank < done + take) {
                        s.ent_i[nent + rank - done] = (uint32_t)(i0 + q);
                        s.ent_v[nent + rank - done] = v[q];
                    }
                    ++rank;
                }
            }
            nent += take;
            done += take;
            if (done < total) __syncthreads();   // the pieces so far are visible to the flush
        }
    }
    __syncthreads();
    if (nent > 0) sp_flush<kScale>(s, nent, hs, n, b, blocks, col_scale, seed, hashed);

    // write the row's sums of every listed block
    for (int t = 0; t < blocks.count; ++t) {
        const int64_t col0 = (int64_t)blocks.idx[t] * b;
        const float *acc = s.state + t * b;
        OutT *dst = At + r * ldat + col0;
        if constexpr (sizeof(OutT) == 1) {
            // FP8: warp per 128-column slice; lane holds 4 consecutive sums
            for (int sl = warp; sl < b / 128; sl += kSpWarps) {
                const float4 x = *reinterpret_cast<const float4 *>(acc + 128 * sl + 4 * lane);
                float a = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w)));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
                const int e = fp8_scale_exponent(a);
                const float inv = ldexpf(1.f, -e);
                __nv_fp8_e4m3 q[4] = {__nv_fp8_e4m3(x.x * inv), __nv_fp8_e4m3(x.y * inv),
                                      __nv_fp8_e4m3(x.z * inv), __nv_fp8_e4m3(x.w * inv)};
                *reinterpret_cast<uint32_t *>(dst + 128 * sl + 4 * lane) = *reinterpret_cast<uint32_t *>(q);
                if (lane == 0) scales[(col0 / 128 + sl) * lds + r] = ldexpf(1.f, e);
            }
        } else {
            for (int c = tid; c < b; c += kSpThreads) sp_store(dst + c, plane_elems, acc[c]);
        }
    }
    __syncthreads();   // the shared memory is free for the next row
}

// ---- one-pass rows ----
//
// NG groups of 1024 / NG threads per CTA.  Shared memory: the bucket counters (16
// bits each, two per word) and the sorted entry numbers, once; per group the values
// and column indices of its row's entries, a region of cw per warp.  Indices are
// relative to the warp's share of the row: 16 bits in two groups (n <= 2^20), 32 in one.
constexpr int kSp1MaxBuckets = 4096;
constexpr int kSp1Ahead = 3;     // L2 prefetch distance of a warp, in steps

template <int NG> struct Sp1 {
    static constexpr int GT = kSpThreads / NG;          // threads per group
    static constexpr int GW = GT / 32;                  // warps per group
    static constexpr int BPT = kSp1MaxBuckets / GT;     // buckets per thread
    using Idx = typename std::conditional<NG == 2, uint16_t, uint32_t>::type;
    static constexpr int64_t kMaxN = NG == 2 ? int64_t(1) << 20 : (int64_t(1) << 31) - 1;
    static constexpr int kEntryBytes = 2 + NG * (4 + (int)sizeof(Idx));
    static constexpr int kMaxPairs = 16;                // codes of a lane's entries, two per register
    static constexpr int kMaxRegion = 64 * kMaxPairs;   // entries per warp
    static constexpr size_t kFixed = sizeof(uint32_t) * (kSp1MaxBuckets / 2 + 40 * NG) + 16;
    static constexpr int kFits = (int)((kSmemLimit - kFixed - 64) / (GW * kEntryBytes) / 4 * 4);
    static constexpr int kRegion = kFits < kMaxRegion ? kFits : kMaxRegion;   // entries per warp that there is room for
    static constexpr size_t kSmem = kFixed + (size_t)kEntryBytes * GW * kRegion;
    static_assert(kMaxRegion * GW <= 32768, "entry numbers have 15 bits");
};

// Shared memory by 32-bit address: the one-pass kernel keeps its array bases in one
// register each (recomputing them, as the compiler does for pointers into extern
// shared memory here, took a tenth of the routing's instructions).
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint4 lds_v4(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
    uint32_t v;
    asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_v4(uint32_t a, uint4 v) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
// The same under a condition, as one predicated instruction (a branch around an
// access costs three more).
__device__ __forceinline__ void sts_u32_if(bool c, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u32 [%1], %2;\n\t}"
                 ::"r"((uint32_t)c), "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u16_if(bool c, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u16 [%1], %2;\n\t}"
                 ::"r"((uint32_t)c), "r"(a), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ void reds_add_if(bool c, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p red.shared.add.u32 [%1], %2;\n\t}"
                 ::"r"((uint32_t)c), "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atoms_add_if(bool c, uint32_t a, uint32_t v) {
    uint32_t o;
    asm volatile("{\n\t.reg .pred p;\n\tmov.u32 %0, 0;\n\tsetp.ne.u32 p, %1, 0;\n\t@p atom.shared.add.u32 %0, [%2], %3;\n\t}"
                 : "=&r"(o) : "r"((uint32_t)c), "r"(a), "r"(v) : "memory");
    return o;
}
// A row entry's column index (relative to its warp's share): 16 or 32 bits.
template <typename IdxT> __device__ __forceinline__ uint32_t lds_idx(uint32_t a, uint32_t k) {
    return sizeof(IdxT) == 2 ? lds_u16(a + 2 * k) : lds_u32(a + 4 * k);
}
template <typename IdxT> __device__ __forceinline__ void sts_idx_if(bool c, uint32_t a, uint32_t k, uint32_t v) {
    if (sizeof(IdxT) == 2) sts_u16_if(c, a + 2 * k, v);
    else sts_u32_if(c, a + 4 * k, v);
}

__device__ __forceinline__ void group_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void group_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// Barrier of the group that also ORs a predicate over its threads.
__device__ __forceinline__ bool group_or(int id, int threads, bool p) {
    uint32_t r;
    asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %1, 0;\n\tbar.red.or.pred b, %2, %3, a;\n\tselp.u32 %0, 1, 0, b;\n\t}"
                 : "=r"(r)
                 : "r"((uint32_t)p), "r"(id), "r"(threads)
                 : "memory");
    return r != 0;
}

// One lane's 16 bytes of a row: E elements, tested and picked by their bits.
template <typename InT> struct Piece;
template <> struct Piece<float> {
    static constexpr int E = 4;
    __device__ static bool any(const uint4 &u) { return ((u.x | u.y | u.z | u.w) & 0x7fffffffu) != 0u; }
    __device__ static uint32_t mask(const uint4 &u) {
        return ((u.x & 0x7fffffffu) ? 1u : 0u) | ((u.y & 0x7fffffffu) ? 2u : 0u) | ((u.z & 0x7fffffffu) ? 4u : 0u) |
               ((u.w & 0x7fffffffu) ? 8u : 0u);
    }
    __device__ static float pick(const uint4 &u, int j) {
        const uint32_t a = (j & 1) ? u.y : u.x, b = (j & 1) ? u.w : u.z;
        return __uint_as_float((j & 2) ? b : a);
    }
    // the first nonzero (j, v) of a piece that has one; whether any lane's piece has more
    __device__ static bool first(const uint4 &u, int &j, float &v) {
        uint32_t more;
        asm volatile(
            "{\n\t.reg .pred x, y, z, w, a, b;\n\t.reg .u32 t;\n\t.reg .f32 f;\n\t"
            "setp.neu.f32 x, %3, 0f00000000;\n\tsetp.neu.f32 y, %4, 0f00000000;\n\t"
            "setp.neu.f32 z, %5, 0f00000000;\n\tsetp.neu.f32 w, %6, 0f00000000;\n\t"
            "selp.u32 t, 2, 3, z;\n\tselp.u32 t, 1, t, y;\n\tselp.u32 %1, 0, t, x;\n\t"
            "selp.f32 f, %5, %6, z;\n\tselp.f32 f, %4, f, y;\n\tselp.f32 %2, %3, f, x;\n\t"
            "and.pred a, z, w;\n\tor.pred b, z, w;\n\tand.pred z, y, b;\n\tor.pred b, y, b;\n\t"
            "and.pred x, x, b;\n\tor.pred a, a, z;\n\tor.pred a, a, x;\n\t"
            "vote.sync.any.pred a, a, 0xffffffff;\n\tselp.u32 %0, 1, 0, a;\n\t}"
            : "=r"(more), "=r"(j), "=f"(v)
            : "f"(__uint_as_float(u.x)), "f"(__uint_as_float(u.y)), "f"(__uint_as_float(u.z)), "f"(__uint_as_float(u.w)));
        return more != 0u;
    }
};
template <> struct Piece<__nv_bfloat16> {
    static constexpr int E = 8;
    __device__ static bool any(const uint4 &u) { return ((u.x | u.y | u.z | u.w) & 0x7fff7fffu) != 0u; }
    __device__ static uint32_t two(uint32_t w) { return ((w & 0x7fffu) ? 1u : 0u) | ((w & 0x7fff0000u) ? 2u : 0u); }
    __device__ static uint32_t mask(const uint4 &u) {
        return two(u.x) | two(u.y) << 2 | two(u.z) << 4 | two(u.w) << 6;
    }
    __device__ static float pick(const uint4 &u, int j) {
        const uint32_t a = (j & 2) ? u.y : u.x, b = (j & 2) ? u.w : u.z, w = (j & 4) ? b : a;
        return __uint_as_float((j & 1) ? (w & 0xffff0000u) : (w << 16));
    }
    __device__ static bool first(const uint4 &u, int &j, float &v) {
        const uint32_t nz = mask(u);
        j = __ffs((int)nz) - 1;
        v = pick(u, j);
        return __any_sync(0xffffffffu, (nz & (nz - 1u)) != 0u);
    }
};

// Compaction of columns [s0, s1) of a row by one warp: its nonzeros, ascending, to
// val / idx (indices relative to s0).  Steps of four 16-byte loads per lane (the
// next step's issued before this one is processed); each load's 32 pieces take a
// ballot, and only the pieces with a nonzero (most have one at a percent) the rest.
// Returns the count, or -1 when the region of cw entries overflows.
template <typename InT, typename IdxT>
__device__ __forceinline__ int sp1_compact(const InT *__restrict__ row, int64_t s0, int64_t s1, bool vec,
                                           uint32_t val, uint32_t idx, int cw) {
    using P = Piece<InT>;
    constexpr int Q = 4, E = P::E;
    constexpr int kChunk = 32 * E, kStep = Q * kChunk;
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    int have = 0;
    auto process = [&](int at0, const uint4 (&u)[Q]) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const bool any = P::any(u[q]);
            const uint32_t bal = __ballot_sync(0xffffffffu, any);
            if (bal == 0u) continue;
            const int at = at0 + q * kChunk;
            int k;
            float v;
            if (P::first(u[q], k, v)) {
                // some lane holds two or more: a lane's first position by a ballot per element
                const uint32_t nz = P::mask(u[q]);
                int pos = have, total = 0;
#pragma unroll 1
                for (int j = 0; j < E; ++j) {
                    const uint32_t bj = __ballot_sync(0xffffffffu, (nz >> j) & 1u);
                    pos += __popc(bj & below);
                    total += __popc(bj);
                }
#pragma unroll 1
                for (int j = 0; j < E; ++j) {
                    if (((nz >> j) & 1u) && pos < cw) {
                        sts_u32(val + 4 * pos, __float_as_uint(P::pick(u[q], j)));
                        sts_idx_if<IdxT>(true, idx, pos, (uint32_t)(at + j));
                        ++pos;
                    }
                }
                have += total;
            } else {
                const int pos = have + __popc(bal & below);
                const bool put = any & (pos < cw);
                sts_u32_if(put, val + 4 * pos, __float_as_uint(v));
                sts_idx_if<IdxT>(put, idx, pos, (uint32_t)(at + k));
                have += __popc(bal);
            }
        }
    };
    const InT *p = row + s0 + E * lane;
    auto load = [&](const InT *from, uint4 (&u)[Q]) {
#pragma unroll
        for (int q = 0; q < Q; ++q) u[q] = __ldcs(reinterpret_cast<const uint4 *>(from + q * kChunk));   // streamed
    };
    const int steps = vec ? (int)((s1 - s0) / kStep) : 0;   // whole steps, 16-byte loads
    int at = E * lane;
    uint4 ua[Q], ub[Q];
    if (steps > 0) load(p, ua);
    for (int st = 0; st < steps; st += 2) {
        if (lane == 0 && st + kSp1Ahead + 2 <= steps)
            l2_prefetch(p + kSp1Ahead * kStep, 2 * kStep * (uint32_t)sizeof(InT));
        if (st + 1 < steps) load(p + kStep, ub);
        process(at, ua);
        if (st + 1 >= steps) break;
        if (st + 2 < steps) load(p + 2 * kStep, ua);
        process(at + kStep, ub);
        p += 2 * kStep;
        at += 2 * kStep;
        if (have > cw) return -1;   // warp-uniform
    }
    // the rest of the share (all of it for rows without 16-byte alignment)
    for (int64_t i0 = s0 + (int64_t)steps * kStep; i0 < s1; i0 += kStep) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t i = i0 + q * kChunk + E * lane;
            InT e[E];
#pragma unroll
            for (int j = 0; j < E; ++j) e[j] = i + j < s1 ? row[i + j] : InT(0.f);
            ua[q] = *reinterpret_cast<const uint4 *>(e);
        }
        process((int)(i0 - s0) + E * lane, ua);
        if (have > cw) return -1;
    }
    return have > cw ? -1 : have;
}

__device__ __forceinline__ void cex(uint32_t &a, uint32_t &b) {
    const uint32_t lo = min(a, b);
    b = max(a, b);
    a = lo;
}

// The routing of one row (`have` entries in this warp's region): see the file
// comment.
template <typename OutT, int NG>
__device__ __forceinline__ void sp1_route(uint32_t cnt, uint32_t warp_tot, uint32_t srt, uint32_t val, uint32_t idx,
                                          int have, uint32_t base, int cw, int64_t r,
                                          const uint32_t *__restrict__ hs, int64_t n, uint64_t seed, bool hashed,
                                          int32_t b, const BlockList &blocks, OutT *__restrict__ At, int64_t ldat,
                                          float *__restrict__ scales, int64_t lds, int64_t plane_elems, int bar) {
    using S = Sp1<NG>;
    using Idx = typename S::Idx;
    constexpr int GT = S::GT, GW = S::GW, BPT = S::BPT, WPT = BPT / 2;
    const int tid = threadIdx.x % GT, lane = tid & 31, warp = tid >> 5;
    const int e0 = warp * cw;                 // this warp's first entry number
    const uint32_t own = idx + (uint32_t)(sizeof(Idx) * e0);
    uint32_t code[S::kMaxPairs];              // bucket | sign << 15 of entries lane + 64 u (low) and + 32 (high)
    auto fill = [&](auto &&code_of) {
#pragma unroll
        for (int u = 0; u < S::kMaxPairs; ++u) {
            if (64 * u >= have) break;
            uint32_t cd[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                cd[h] = code_of(base + lds_idx<Idx>(own, min(64 * u + 32 * h + lane, have - 1)));   // repeats the last entry
                cd[h] = (cd[h] & 0x7fffu) | ((cd[h] >> 16) & 0x8000u);
            }
            code[u] = cd[0] | cd[1] << 16;
        }
    };
    auto load_codes = [&](int jb) {
        if (hashed) {
            const uint64_t key = block_key(seed, jb);
            fill([&](uint32_t i) { return hash_code(key, (int64_t)i, b); });
        } else {
            const uint32_t *hj = hs + (int64_t)jb * n;
            fill([&](uint32_t i) { return __ldg(hj + i); });
        }
    };
    // the thread's buckets: BPT*tid .. BPT*tid + BPT-1 (counter words WPT*tid ..)
    const uint32_t words = cnt + 4 * WPT * tid;
    auto read_words = [&](uint32_t (&w)[WPT]) {
        if constexpr (WPT == 4) {
            const uint4 q = lds_v4(words);
            w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
        } else {
            w[0] = lds_u32(words);
            w[1] = lds_u32(words + 4);
        }
    };
    auto write_words = [&](const uint32_t (&w)[WPT]) {
        if constexpr (WPT == 4) {
            sts_v4(words, make_uint4(w[0], w[1], w[2], w[3]));
        } else {
            sts_u32(words, w[0]);
            sts_u32(words + 4, w[1]);
        }
    };
#pragma unroll 1
    for (int t = 0; t < blocks.count; ++t) {
        const int jb = blocks.idx[t];
        load_codes(jb);
        if (t > 0) group_sync(bar, GT);   // the block before is done with the counters and entry lists
        {
            const uint32_t zero[WPT] = {};
            write_words(zero);
        }
        group_sync(bar, GT);
#pragma unroll
        for (int u = 0; u < S::kMaxPairs; ++u) {
            if (64 * u >= have) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t bk = (code[u] >> (16 * h)) & 0x7fffu;
                reds_add_if(64 * u + 32 * h + lane < have, cnt + 4 * (bk >> 1), (bk & 1u) ? 0x10000u : 1u);
            }
        }
        group_sync(bar, GT);
        // bucket starts: the thread's counts, a warp scan, the totals of the warps before
        uint32_t w[WPT];
        read_words(w);
        int mine = 0;
#pragma unroll
        for (int q = 0; q < WPT; ++q) mine += (int)(w[q] & 0xffffu) + (int)(w[q] >> 16);
        int inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) sts_u32(warp_tot + 4 * warp, (uint32_t)inc);
        group_sync(bar, GT);
        int before = lane < warp ? (int)lds_u32(warp_tot + 4 * lane) : 0;   // warp <= 31
        before = __reduce_add_sync(0xffffffffu, before);
        const int start = before + inc - mine;
        {
            int off = start;
#pragma unroll
            for (int q = 0; q < WPT; ++q) {
                const int k0 = (int)(w[q] & 0xffffu), k1 = (int)(w[q] >> 16);
                w[q] = (uint32_t)off | ((uint32_t)(off + k0) << 16);
                off += k0 + k1;
            }
        }
        write_words(w);
        group_sync(bar, GT);
        // entry numbers (and signs) into their buckets
#pragma unroll
        for (int u = 0; u < S::kMaxPairs; ++u) {
            if (64 * u >= have) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t cd = code[u] >> (16 * h), bk = cd & 0x7fffu;
                const int k = 64 * u + 32 * h + lane;
                const uint32_t old = atoms_add_if(k < have, cnt + 4 * (bk >> 1), (bk & 1u) ? 0x10000u : 1u);
                const uint32_t pos = (bk & 1u) ? old >> 16 : old & 0xffffu;
                sts_u16_if(k < have, srt + 2 * pos, ((uint32_t)(e0 + k) << 1) | ((cd >> 15) & 1u));
            }
        }
        group_sync(bar, GT);
        // The counters now hold the buckets' ends.  A warp owns `per` consecutive buckets,
        // lane i buckets i, i + 32, ..: every lane has one down to b = 32 GW, and its
        // sums are stored whole lines at a time.  A bucket's members are added in
        // ascending entry order (= ascending index) behind a sorting network over 4, 6
        // or 8 of them, straight-line and predicated; longer lists are sorted by
        // insertion in their slice of srt.
        auto bucket_end = [&](int c) -> int {   // 0 for c < 0
            const uint32_t w = lds_u32(cnt + 4 * (max(c, 0) >> 1));
            return c < 0 ? 0 : (int)((c & 1) ? w >> 16 : w & 0xffffu);
        };
        auto term = [&](uint32_t m) -> float {   // the sign is the entry number's lowest bit
            return __uint_as_float(lds_u32(val + 2 * (m & 0xfffeu)) ^ (m << 31));
        };
        auto bucket_sum = [&](int q) -> float {   // bucket q (zero past the last); all lanes of the warp together
            const int p0 = q < b ? bucket_end(q - 1) : 0;
            const int c = q < b ? bucket_end(q) - p0 : 0;
            const uint32_t from = srt + 2 * p0;
            auto sorted_sum = [&](auto nn) -> float {
                constexpr int N = decltype(nn)::value;
                uint32_t m[N];   // reads past the bucket (and past srt's end, into its padding) are dropped
#pragma unroll
                for (int k = 0; k < N; ++k) m[k] = lds_u16(from + 2 * k);
#pragma unroll
                for (int k = 0; k < N; ++k) m[k] = k < c ? m[k] : 0xffffu;
                // Batcher's odd-even merge sort
                cex(m[0], m[1]); cex(m[2], m[3]); cex(m[0], m[2]); cex(m[1], m[3]); cex(m[1], m[2]);
                if constexpr (N == 6) {
                    cex(m[4], m[5]);
                    cex(m[0], m[4]); cex(m[1], m[5]); cex(m[2], m[4]); cex(m[3], m[5]); cex(m[1], m[2]); cex(m[3], m[4]);
                } else if constexpr (N == 8) {
                    cex(m[4], m[5]); cex(m[6], m[7]); cex(m[4], m[6]); cex(m[5], m[7]); cex(m[5], m[6]);
                    cex(m[0], m[4]); cex(m[1], m[5]); cex(m[2], m[6]); cex(m[3], m[7]);
                    cex(m[2], m[4]); cex(m[3], m[5]);
                    cex(m[1], m[2]); cex(m[3], m[4]); cex(m[5], m[6]);
                }
                float x[N];
#pragma unroll
                for (int k = 0; k < N; ++k) x[k] = term(k < c ? m[k] : 0u);
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < N; ++k) s = k < c ? s + x[k] : s;
                return s;
            };
            const int most = __reduce_max_sync(0xffffffffu, c <= 8 ? c : 0);
            float s;
            if (most <= 4) s = sorted_sum(std::integral_constant<int, 4>());
            else if (most <= 6) s = sorted_sum(std::integral_constant<int, 6>());
            else s = sorted_sum(std::integral_constant<int, 8>());
            if (c > 8) {
#pragma unroll 1
                for (int k = 1; k < c; ++k) {
                    const uint32_t x = lds_u16(from + 2 * k);
                    int j = k - 1;
                    for (; j >= 0; --j) {
                        const uint32_t y = lds_u16(from + 2 * j);
                        if (y <= x) break;
                        sts_u16(from + 2 * j + 2, y);
                    }
                    sts_u16(from + 2 * j + 2, x);
                }
                s = 0.f;
#pragma unroll 1
                for (int k = 0; k < c; ++k) s += term(lds_u16(from + 2 * k));
            }
            return s;
        };
        const int64_t col0 = (int64_t)jb * b;
        OutT *dst = At + r * ldat + col0;
        if constexpr (sizeof(OutT) == 1) {
            // FP8 (b % 128 == 0): whole 128-column slices per warp
            const int per = ((b + GW - 1) / GW + 127) / 128 * 128;
#pragma unroll 1
            for (int q0 = warp * per; q0 < min(b, (warp + 1) * per); q0 += 128) {
                float a[4], am = 0.f;
#pragma unroll 1
                for (int i = 0; i < 4; ++i) {
                    const float x = bucket_sum(q0 + 32 * i + lane);
                    am = fmaxf(am, fabsf(x));
                    if (i == 0) a[0] = x;
                    else if (i == 1) a[1] = x;
                    else if (i == 2) a[2] = x;
                    else a[3] = x;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
                const int e = fp8_scale_exponent(am);
                const float inv = ldexpf(1.f, -e);
#pragma unroll
                for (int i = 0; i < 4; ++i) dst[q0 + 32 * i + lane] = __nv_fp8_e4m3(a[i] * inv);
                if (lane == 0) scales[((col0 + q0) / 128) * lds + r] = ldexpf(1.f, e);
            }
        } else {
            const int per = ((b + GW - 1) / GW + 31) / 32 * 32;
#pragma unroll 1
            for (int q0 = warp * per; q0 < min(b, (warp + 1) * per); q0 += 32) {
                const float x = bucket_sum(q0 + lane);
                if (q0 + lane < b) sp_store(dst + q0 + lane, plane_elems, x);
            }
        }
    }
}

// Bits that mark a row the one-pass kernel left to the flushing kernel, stored
// in the row's first kept output: a quiet NaN with a payload (FP32, BF16, and
// the hi plane of TF32 pairs) or the E4M3 NaN code.  A genuine output with the
// same bits only makes the flushing kernel recompute that row.
template <typename OutT>
struct RowMark;
template <> struct RowMark<float> { using U = uint32_t; static constexpr U bits = 0x7fd1c0deu; };
template <> struct RowMark<Tf32Pair> { using U = uint32_t; static constexpr U bits = 0x7fd1c0deu; };
template <> struct RowMark<__nv_bfloat16> { using U = uint16_t; static constexpr U bits = 0x7fd1u; };
template <> struct RowMark<__nv_fp8_e4m3> { using U = uint8_t; static constexpr U bits = 0x7fu; };

template <typename OutT>
__device__ __forceinline__ typename RowMark<OutT>::U *row_mark(OutT *At, int64_t r, int64_t ldat, int64_t col) {
    return reinterpret_cast<typename RowMark<OutT>::U *>(At + r * ldat + col);
}

// The CTA's rows.  Group g takes every NG-th of them; with two groups the routing (the
// shared counters and entry lists) goes from one to the other row by row, so each group
// compacts while the other routes.  A row whose nonzeros overflow a warp's region is
// marked for the flushing kernel.
template <typename InT, typename OutT, bool kScale, int NG>
__device__ __forceinline__ void sp1_rows(const InT *__restrict__ A, int64_t lda, int64_t rows, int64_t n, bool vec,
                                         const uint32_t *__restrict__ hs, uint64_t seed, bool hashed, int32_t b,
                                         const BlockList &blocks, const float *__restrict__ col_scale,
                                         OutT *__restrict__ At, int64_t ldat, float *__restrict__ scales, int64_t lds,
                                         int64_t plane_elems, float4 *sp_smem) {
    using S = Sp1<NG>;
    using Idx = typename S::Idx;
    constexpr int cw = S::kRegion;
    const int ge = S::GW * cw;                      // entries per group
    uint32_t cnt;                                   // kSp1MaxBuckets / 2 words, then 40 words per group for the scan
    asm volatile("mov.u32 %0, %1;" : "=r"(cnt) : "r"((uint32_t)__cvta_generic_to_shared(sp_smem)));
    const uint32_t warp_tot = cnt + 2 * kSp1MaxBuckets;
    const uint32_t vals = warp_tot + 160 * NG;      // [NG][ge] FP32
    const uint32_t idxs = vals + 4 * NG * ge;       // [NG][ge] Idx
    const uint32_t srt = idxs + (uint32_t)sizeof(Idx) * NG * ge;   // [ge] 16 bits
    const int g = threadIdx.x / S::GT, warp = (threadIdx.x % S::GT) >> 5, lane = threadIdx.x & 31;
    const int bar = 1 + g;
    const uint32_t val = vals + 4 * g * ge, idx = idxs + (uint32_t)sizeof(Idx) * g * ge;
    const uint32_t wval = val + 4 * warp * cw, widx = idx + (uint32_t)sizeof(Idx) * warp * cw;   // the warp's region
    const int64_t seg = ((n + S::GW - 1) / S::GW + 1023) / 1024 * 1024;   // columns per warp: whole steps
    const int64_t s0 = min(n, (int64_t)warp * seg), s1 = min(n, s0 + seg);
    for (int64_t q = g; q < rows; q += NG) {
        const int64_t r = blockIdx.x + q * gridDim.x;
        const int have = sp1_compact<InT, Idx>(A + r * lda, s0, s1, vec, wval, widx, cw);
        if constexpr (kScale) {
            __syncwarp();
#pragma unroll 8
            for (int k = lane; k < have; k += 32) {
                const float f = __ldg(col_scale + s0 + lds_idx<Idx>(widx, k));
                sts_u32(wval + 4 * k, __float_as_uint(__uint_as_float(lds_u32(wval + 4 * k)) * f));
            }
        }
        const bool over = group_or(bar, S::GT, have < 0);
        if (NG == 2 && q > 0) group_sync(3 + g, kSpThreads);   // this group's turn
        if (!over)
            sp1_route<OutT, NG>(cnt, warp_tot + 160 * g, srt, val, idx, have, (uint32_t)s0, cw, r, hs, n, seed, hashed, b, blocks,
                                At, ldat, scales, lds, plane_elems, bar);
        else if (threadIdx.x % S::GT == 0)
            *row_mark(At, r, ldat, (int64_t)blocks.idx[0] * b) = RowMark<OutT>::bits;
        if (NG == 2 && q + 1 < rows) group_arrive(3 + (g ^ 1), kSpThreads);
        group_sync(bar, S::GT);   // the group's entries are free for its next row
    }
}

// Nonzeros (x) among the elements (y) of 4 pieces of 16 bytes per thread, over the CTA:
// piece q of a thread is at place(q).x in row place(q).y of A.
template <typename InT, typename Place>
__device__ __forceinline__ int2 sp1_sample(const InT *__restrict__ A, int64_t lda, int64_t n, bool vec, Place place,
                                           float4 *sp_smem) {
    using P = Piece<InT>;
    constexpr int Q = 4, E = P::E;
    uint32_t *sums = reinterpret_cast<uint32_t *>(sp_smem);
    uint4 u[Q];
    uint32_t s = 0;   // both counts stay below 2^16 over the CTA
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const longlong2 at = place(q);
        u[q] = make_uint4(0u, 0u, 0u, 0u);
        if (at.x + E > n) continue;
        s += E << 16;
        const InT *from = A + at.y * lda + at.x;
        if (vec) {
            u[q] = __ldg(reinterpret_cast<const uint4 *>(from));
        } else {
            InT e[E];
#pragma unroll
            for (int j = 0; j < E; ++j) e[j] = from[j];
            u[q] = *reinterpret_cast<const uint4 *>(e);
        }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) s += __popc(P::mask(u[q]));
    s = __reduce_add_sync(0xffffffffu, s);
    if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = s;
    __syncthreads();
    s = __reduce_add_sync(0xffffffffu, sums[threadIdx.x & 31]);
    __syncthreads();   // the shared memory is free
    return make_int2((int)(s & 0xffffu), (int)(s >> 16));
}

// How the CTA takes its rows: two at a time, one, or none (0: all left to the flushing
// kernel), by the nonzeros a row has, estimated from 64 pieces of 512 bytes of each of its
// first two rows.  Two groups hide the streaming of one row behind the routing of
// another, but route with half the threads and hold fewer entries: 996 in each 16th of a
// row against 700 in each 32nd, so that uniform rows of 2^20 columns overflow from 1.44 %
// and from 1.85 % on, and a row that does is read twice.  us on GB300, two groups / one:
// 2048 rows of 2^20, b = 2048: 1 % 2655 / 2468, 1.35 % 3796 / 3091, 1.44 % 7534 / 3244,
// 1.6 % 6563 / 3523; 1216 rows, b = 4096: 0.6 % 920 / 1093, 1.2 % 1403 / 1484; 608 rows of
// 2^19, b = 2048: 1.2 % 455 / 459, 2 % 753 / 656; 456 rows of 65536, b = 2048: 2 % 106 /
// 106, 20 % 634 / 473; b = 512: 2 % 111 / 119.  Blocks below 1024 (long bucket lists) go
// straight to the flushing kernel then: 1216 rows of 2^20 at 1.44 %, b = 256: one group
// 7.3 ms, flushed 5.0.  Where rows may overflow every CTA takes the same larger sample of all
// of A: some leaving their rows and some not would wait for each other in both kernels.
// Not inlined: the row loops' registers are allocated 2 % better without it.
template <typename InT>
__device__ __noinline__ int sp1_groups(const InT *__restrict__ A, int64_t lda, int64_t m, int64_t rows, int64_t n,
                                          int32_t b, bool vec, float4 *sp_smem) {
    constexpr int E = Piece<InT>::E;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t seg = ((n + 15) / 16 + 1023) / 1024 * 1024, s0 = (warp & 15) * seg;
    const int64_t r = blockIdx.x + (rows > 1 ? (int64_t)(warp >> 4) * gridDim.x : 0);
    // the shares' first steps come into L2 meanwhile
    if (vec && lane == 0 && s0 + 3 * 128 * E <= n) l2_prefetch(A + r * lda + s0, 3 * 128 * E * (uint32_t)sizeof(InT));
    int2 s = sp1_sample<InT>(A, lda, n, vec,
                             [&](int q) { return make_longlong2(s0 + q * (seg / 4) + E * lane, r); }, sp_smem);
    auto more_than = [&](int64_t entries) { return s.x * n > entries * s.y; };   // a row
    if (more_than(11264)) {
        s = make_int2(0, 0);
#pragma unroll 1
        for (int k0 = 0; k0 < 2 * 4 * kSpThreads; k0 += 4 * kSpThreads) {
            // rows in order, columns scattered
            const int2 part = sp1_sample<InT>(A, lda, n, vec, [&](int q) {
                const uint32_t k = (uint32_t)k0 + threadIdx.x * 4 + q;
                return make_longlong2((int64_t)((uint64_t)(k * 0x9E3779B1u) * (uint64_t)n >> 32) & ~int64_t(E - 1),
                                      (int64_t)((uint64_t)k * (uint64_t)m / (8 * kSpThreads)));
            }, sp_smem);
            s.x += part.x;
            s.y += part.y;
        }
    }
    if (more_than(b < 1024 ? 14336 : 19456)) return 0;
    if (b >= 1024 && more_than(b <= 3072 ? 12288 : 13312)) return 1;
    return rows < 2 || (b >= 1024 && more_than(n / 64)) ? 1 : 2;
}

// The one-pass kernel (persistent over rows), with kTwo in two groups where that pays.
template <typename InT, typename OutT, bool kScale, bool kTwo>
__global__ void __launch_bounds__(kSpThreads, 1)
sketch_left_onepass_kernel(const InT *__restrict__ A, int64_t lda, int64_t m, int64_t n, bool vec,
                           const uint32_t *__restrict__ hs, uint64_t seed, bool hashed, int32_t b,
                           const __grid_constant__ BlockList blocks, const float *__restrict__ col_scale,
                           OutT *__restrict__ At, int64_t ldat, float *__restrict__ scales, int64_t lds,
                           int64_t plane_elems) {
    extern __shared__ float4 sp_smem[];
    const int64_t rows = (m - blockIdx.x + gridDim.x - 1) / gridDim.x;   // of this CTA
    const int groups = kTwo ? sp1_groups<InT>(A, lda, m, rows, n, b, vec, sp_smem) : 1;
    if (groups == 2)
        sp1_rows<InT, OutT, kScale, 2>(A, lda, rows, n, vec, hs, seed, hashed, b, blocks, col_scale, At, ldat, scales,
                                       lds, plane_elems, sp_smem);
    else if (groups == 1)
        sp1_rows<InT, OutT, kScale, 1>(A, lda, rows, n, vec, hs, seed, hashed, b, blocks, col_scale, At, ldat, scales,
                                       lds, plane_elems, sp_smem);
    else
        for (int64_t q = threadIdx.x; q < rows; q += kSpThreads)
            *row_mark(At, blockIdx.x + q * gridDim.x, ldat, (int64_t)blocks.idx[0] * b) = RowMark<OutT>::bits;
}

// The flushing kernel: one CTA per row (persistent over rows); with kMarked,
// only the rows the one-pass kernel marked.
template <typename InT, typename OutT, bool kScale, bool kMarked>
__global__ void __launch_bounds__(kSpThreads, 1)
sketch_left_sparse_kernel(const InT *__restrict__ A, int64_t lda, int64_t m, int64_t n, bool vec,
                          const uint32_t *__restrict__ hs, uint64_t seed, bool hashed, int32_t b,
                          BlockList blocks, int emax,
                          const float *__restrict__ col_scale, OutT *__restrict__ At, int64_t ldat,
                          float *__restrict__ scales, int64_t lds, int64_t plane_elems) {
    extern __shared__ float4 sp_smem[];
    if constexpr (kMarked) {
        // 32 of the CTA's rows at a time: every warp reads their marks (the same
        // ballot in every warp), then the CTA runs the marked ones.  One row of each
        // gridDim.x consecutive ones, at a place that moves on from one set to the next, so
        // that the rows one CTA of the one-pass kernel left are shared by many here, and so
        // are consecutive rows.
        const int lane = threadIdx.x & 31;
        auto row_of = [&](int64_t k) -> int64_t {
            return k * gridDim.x + (blockIdx.x + (uint64_t)k * 37u) % gridDim.x;
        };
        for (int64_t base = 0; base * gridDim.x < m; base += 32) {
            const int64_t rl = row_of(base + lane);
            const bool take = rl < m && *row_mark(At, rl, ldat, (int64_t)blocks.idx[0] * b) == RowMark<OutT>::bits;
            uint32_t todo = __ballot_sync(0xffffffffu, take);
            while (todo) {
                const int t = __ffs(todo) - 1;
                todo &= todo - 1;
                const int64_t r = row_of(base + t);
                sp_row_flushing<InT, OutT, kScale>(A + r * lda, r, n, vec, hs, seed, hashed, b, blocks, emax,
                                                   col_scale, At, ldat, scales, lds, plane_elems, sp_smem);
            }
        }
    } else {
        for (int64_t r = blockIdx.x; r < m; r += gridDim.x)
            sp_row_flushing<InT, OutT, kScale>(A + r * lda, r, n, vec, hs, seed, hashed, b, blocks, emax,
                                               col_scale, At, ldat, scales, lds, plane_elems, sp_smem);
    }
}

// Entries the buffer holds beside kb accumulators and the bucket tables (multiple of 32).
int sparse_entry_capacity(int64_t kb, int64_t b) {
    const int64_t avail = (int64_t)kSmemLimit - 4 * kb - (int64_t)sp_fixed_bytes((int)b) - 64;
    if (avail <= 0) return 0;
    const int64_t e = avail / kEntryBytes / 32 * 32;
    return (int)(e < kSpThreads * kSpPerThread ? e : kSpThreads * kSpPerThread);
}

int sp_num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

template <typename InT, typename OutT>
os_status launch_sparse_t(const InT *A, int64_t lda, int64_t m, int64_t n, const Plan *p, const BlockList &blocks,
                          const float *col_scale, void *At, int64_t ldat, float *scales, int64_t lds,
                          int64_t plane_elems, cudaStream_t st) {
    const int kb = blocks.count * p->b;
    const int emax = sparse_entry_capacity(kb, p->b);
    if (emax < kMinEntries) return OS_ERR_UNSUPPORTED;
    const size_t smem0 = sizeof(float) * (size_t)kb + (size_t)kEntryBytes * emax + sp_fixed_bytes(p->b);
    const bool vec = aligned16(A) && (lda * (int64_t)sizeof(InT)) % 16 == 0;
    const int64_t grid = m < sp_num_sms() ? m : sp_num_sms();
    // one-pass rows: two rows at a time per SM when there are enough rows (and their
    // indices fit 16 bits), else one row by the whole CTA
    const bool onepass = p->b <= kSp1MaxBuckets;
    if (onepass) {
        const bool two = m > sp_num_sms() && n <= Sp1<2>::kMaxN;
        auto k1 = two ? (col_scale ? sketch_left_onepass_kernel<InT, OutT, true, true>
                                   : sketch_left_onepass_kernel<InT, OutT, false, true>)
                      : (col_scale ? sketch_left_onepass_kernel<InT, OutT, true, false>
                                   : sketch_left_onepass_kernel<InT, OutT, false, false>);
        const size_t smem1 = Sp1<1>::kSmem > Sp1<2>::kSmem ? Sp1<1>::kSmem : Sp1<2>::kSmem;
        OSK_CUDA_TRY(cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1));
        k1<<<(unsigned)grid, kSpThreads, smem1, st>>>(A, lda, m, n, vec, p->hs, p->seed, p->hashed != 0, p->b, blocks,
                                                      col_scale, (OutT *)At, ldat, scales, lds, plane_elems);
        OSK_TRY(check_launch());
    }
    auto k = onepass ? (col_scale ? sketch_left_sparse_kernel<InT, OutT, true, true>
                                 : sketch_left_sparse_kernel<InT, OutT, false, true>)
                    : (col_scale ? sketch_left_sparse_kernel<InT, OutT, true, false>
                                 : sketch_left_sparse_kernel<InT, OutT, false, false>);
    OSK_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem0));
    k<<<(unsigned)grid, kSpThreads, smem0, st>>>(A, lda, m, n, vec, p->hs, p->seed, p->hashed != 0, p->b, blocks,
                                                 emax, col_scale, (OutT *)At, ldat, scales, lds, plane_elems);
    return check_launch();
}

template <typename InT>
os_status launch_sparse(const InT *A, int64_t lda, int64_t m, const Plan *p, const BlockList &blocks,
                        const float *col_scale, void *At, os_dtype out_t, int64_t ldat, float *scales,
                        cudaStream_t st) {
    const int64_t lds = fp8_scale_ld(m);
    switch (out_t) {
        case OS_F32:
            return launch_sparse_t<InT, float>(A, lda, m, p->n, p, blocks, col_scale, At, ldat, nullptr, lds, 0, st);
        case OS_BF16:
            return launch_sparse_t<InT, __nv_bfloat16>(A, lda, m, p->n, p, blocks, col_scale, At, ldat, nullptr, lds,
                                                       0, st);
        case OS_FP8E4M3:
            return launch_sparse_t<InT, __nv_fp8_e4m3>(A, lda, m, p->n, p, blocks, col_scale, At, ldat, scales, lds,
                                                       0, st);
        case OS_TF32X2:
            return launch_sparse_t<InT, Tf32Pair>(A, lda, m, p->n, p, blocks, col_scale, At, ldat, nullptr, lds,
                                                  m * ldat, st);
    }
    return OS_ERR_DTYPE;
}

}  // namespace

// Whether the sparse-row left sketch can hold the accumulators of these blocks.
bool sketch_left_sparse_fits(const Plan *p, uint64_t block_mask) {
    const BlockList blocks = mask_to_list(block_mask ? block_mask : ~0ull, p->P);
    const int64_t kb = (int64_t)blocks.count * p->b;
    return kb <= kSparseMaxBuckets && p->b <= kSparseMaxBuckets &&
           sparse_entry_capacity(kb, p->b) >= kMinEntries;
}

os_status sketch_left_sparse_impl(const Plan *p, const void *A, os_dtype a_t, int64_t m, int64_t lda, void *At,
                                  os_dtype out_t, int64_t ldat, float *scales, const float *col_scale,
                                  uint64_t block_mask, cudaStream_t st) {
    if (!p || m < 0) return OS_ERR_INVALID_ARG;
    if (block_mask) OSK_TRY(check_mask(block_mask, p->P));
    if (a_t != OS_F32 && a_t != OS_BF16) return OS_ERR_DTYPE;
    if (out_t != OS_F32 && out_t != OS_BF16 && out_t != OS_FP8E4M3 && out_t != OS_TF32X2) return OS_ERR_DTYPE;
    const int64_t z = (int64_t)p->P * p->b;
    if (lda < p->n || ldat < z || (ldat * (int64_t)dtype_size(out_t)) % 16 != 0) return OS_ERR_INVALID_ARG;
    if (out_t == OS_FP8E4M3 && p->b % 128 != 0) return OS_ERR_UNSUPPORTED;
    if (!sketch_left_sparse_fits(p, block_mask)) return OS_ERR_UNSUPPORTED;
    if (m == 0) return OS_OK;   // an empty output
    if (!A || !At || !aligned16(At)) return OS_ERR_INVALID_ARG;
    if (out_t == OS_FP8E4M3 && !scales) return OS_ERR_INVALID_ARG;
    const BlockList blocks = mask_to_list(block_mask ? block_mask : ~0ull, p->P);
    if (a_t == OS_F32)
        return launch_sparse<float>((const float *)A, lda, m, p, blocks, col_scale, At, out_t, ldat, scales, st);
    return launch_sparse<__nv_bfloat16>((const __nv_bfloat16 *)A, lda, m, p, blocks, col_scale, At, out_t, ldat,
                                        scales, st);
}

}  // namespace osk

using namespace osk;

extern "C" os_status oversketch_sketch_left_sparse(oversketch_plan_t plan, const void *A, os_dtype a_t, int64_t m,
                                                   int64_t lda, void *At, os_dtype out_t, int64_t ldat,
                                                   float *scales, const float *col_scale, uint64_t block_mask,
                                                   void *stream) {
    OSK_NVTX("sketch_left_sparse");
    return sketch_left_sparse_impl(reinterpret_cast<const Plan *>(plan), A, a_t, m, lda, At, out_t, ldat, scales,
                                   col_scale, block_mask, as_stream(stream));
}
