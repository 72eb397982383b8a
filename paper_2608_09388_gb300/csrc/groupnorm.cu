// Sparse group normalisation (Eqs. 7-9): for every frame b and channel group
// g, mean and variance over the frame's active rows [offsets[b], offsets[b+1])
// and the group's C/G channels only, then (x - mean) / sqrt(var + eps),
// optional per-channel affine, and the activation of Eq. 10 fused.
//
// Statistics. Values are read in chunks; per chunk its mean (shifted by the
// chunk's first value) and centred sum of squares, merged into a running
// (count, mean, M2) by the pairwise update of Chan, Golub and LeVeque, and
// partial results merged the same way. The variance is never formed as
// E[x^2] - mean^2, and a group of equal values gets exactly that mean and
// M2 = 0, so it normalises to exactly 0. All in fp32: GB300's fp64 rate is
// far too low for a bandwidth-bound kernel.
//
// Fast path (rows in 16-byte chunks, C/VEC a power of two <= 256, and either
// VEC | C/G or C/G | VEC): the compact rows [offsets[0], offsets[B]) are cut
// into gridDim.x equal contiguous ranges, one per CTA, independent of frame
// boundaries. That balances the load whatever the frame sizes, and whole
// rows are read with coalesced 16-byte loads; each thread owns one chunk
// column, hence a fixed set of groups and fixed gamma/beta values.
//   gn_stats_kernel: per frame segment of its range, a block merge per group
//     and one partial (n, mean, M2) per (frame b, CTA c), written to slot
//     b + c of the workspace. Frames are contiguous and in order, so the
//     slots of frame b, b + [first CTA, last CTA], end before those of frame
//     b + 1 begin: slots never collide and (B + gridDim.x) * G suffice.
//   gn_apply_kernel: same ranges; per frame segment, merge the partials of
//     the CTAs that hold the frame, normalise and store. Segments and rows
//     are walked in reverse, so the most recently read rows, still in L2,
//     are consumed first, and its loads and stores carry an L2 evict-first
//     policy (last use), which keeps the rest of the input in L2.
// Frames are located by a kThreads-ary block search of the frame table and
// read a window of kThreads frames at a time into shared memory; loads are
// issued a batch ahead of the arithmetic.
// Many frames take the cluster path further down, which reads x once.
// The general path (one CTA per (frame, group)) serves every other layout,
// and small frames (a group slice within its register cache), where one
// launch beats the two latency-bound row-range launches.
// Partials from the convolution: the tensor-core convolution can write the
// (n, mean, M2) partials of its stored output itself, one per (frame b,
// 32-row block c lying inside the frame) in slot b + c (the slot argument
// above with ranges of 32 rows), and one per row for the rows of blocks that
// straddle a frame boundary, so that gn_apply_kernel alone finishes the
// layer.
// The output may alias the input in both paths. Deterministic, no atomics.
#include <cuda_bf16.h>

#include <mutex>

#include "hc_internal.cuh"

namespace hc {
namespace {

constexpr int kThreads = 256;
constexpr int kBatch = 4;
constexpr int kMaxGroupsFast = 2048;
constexpr int kMergeBatch = 4;  // partials a lane loads before merging them

// VEC consecutive elements as one raw chunk (16 bytes when VEC > 1).
template <typename T, int VEC>
struct Chunk;
template <>
struct Chunk<float, 1> {
    using Raw = float;
    static __device__ __forceinline__ Raw load(const float* p) { return *p; }
    static __device__ __forceinline__ void unpack(Raw r, float* v) { v[0] = r; }
    static __device__ __forceinline__ void store(float* p, const float* v) { *p = v[0]; }
};
template <>
struct Chunk<float, 4> {
    using Raw = float4;
    static __device__ __forceinline__ Raw load(const float* p) {
        return *reinterpret_cast<const float4*>(p);
    }
    static __device__ __forceinline__ void unpack(Raw r, float* v) {
        v[0] = r.x, v[1] = r.y, v[2] = r.z, v[3] = r.w;
    }
    static __device__ __forceinline__ void store(float* p, const float* v) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <>
struct Chunk<__nv_bfloat16, 1> {
    using Raw = __nv_bfloat16;
    static __device__ __forceinline__ Raw load(const __nv_bfloat16* p) { return *p; }
    static __device__ __forceinline__ void unpack(Raw r, float* v) { v[0] = __bfloat162float(r); }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, const float* v) {
        *p = __float2bfloat16_rn(v[0]);
    }
};
template <>
struct Chunk<__nv_bfloat16, 8> {
    using Raw = uint4;
    static __device__ __forceinline__ Raw load(const __nv_bfloat16* p) {
        return *reinterpret_cast<const uint4*>(p);
    }
    static __device__ __forceinline__ void unpack(Raw r, float* v) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = __uint_as_float(w[k] << 16);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, const float* v) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
            w[k] = *reinterpret_cast<const uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};

template <typename Raw>
__device__ __forceinline__ Raw as_raw(uint4 v) {
    return *reinterpret_cast<const Raw*>(&v);
}
template <typename Raw>
__device__ __forceinline__ uint4 as_u4(const Raw& v) {
    return *reinterpret_cast<const uint4*>(&v);
}

// Running (count, mean, M2), fp32. Counts are exact integers below 2^24.
struct Stats {
    float n = 0.f, mean = 0.f, m2 = 0.f;
    template <int VEC>
    __device__ __forceinline__ void add_chunk(const float* v) {
        float s = 0.f;
#pragma unroll
        for (int k = 1; k < VEC; ++k) s += v[k] - v[0];
        const float cm = v[0] + s * (1.f / VEC);
        float q = 0.f;
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            const float d = v[k] - cm;
            q = fmaf(d, d, q);
        }
        const float nn = n + (float)VEC;
        const float d = cm - mean;
        const float r = (float)VEC * __frcp_rn(nn);
        mean = fmaf(d, r, mean);
        m2 += q + d * d * n * r;
        n = nn;
    }
};

// Pairwise merge of (nb, mb, qb) into (n, mean, m2).
__device__ __forceinline__ void merge(float& n, float& mean, float& m2, float nb, float mb,
                                      float qb) {
    if (nb == 0.f) return;
    const float nn = n + nb;
    const float d = mb - mean;
    const float r = nb * __frcp_rn(nn);
    mean = fmaf(d, r, mean);
    m2 += qb + d * d * n * r;
    n = nn;
}

__device__ __forceinline__ void merge_xor(float& n, float& mean, float& m2, int o) {
    const float nb = __shfl_xor_sync(0xffffffffu, n, o);
    const float mb = __shfl_xor_sync(0xffffffffu, mean, o);
    const float qb = __shfl_xor_sync(0xffffffffu, m2, o);
    merge(n, mean, m2, nb, mb, qb);
}

// Merge over the whole block; every thread gets the result.
__device__ __forceinline__ void block_merge(float& n, float& mean, float& m2, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) merge_xor(n, mean, m2, o);
    if ((threadIdx.x & 31) == 0) {
        red[3 * (threadIdx.x >> 5)] = n;
        red[3 * (threadIdx.x >> 5) + 1] = mean;
        red[3 * (threadIdx.x >> 5) + 2] = m2;
    }
    __syncthreads();
    n = mean = m2 = 0.f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w)
        merge(n, mean, m2, red[3 * w], red[3 * w + 1], red[3 * w + 2]);
}

// ---- fast path: contiguous row ranges ------------------------------------
struct GnPart {
    float n, mean, m2, pad;
};

// Row range of CTA c over [off0, end): R = ceil((end - off0) / grid).
struct RangeMap {
    long long off0, end, R;
    __device__ __forceinline__ long long cta_of(long long row) const { return (row - off0) / R; }
};

// First frame b in [0, B] with offsets[b + 1] > row (B if none): a
// kThreads-ary search, every thread of the block taking part, so one round
// trip to the table per factor of kThreads frames. A malformed (unsorted)
// table yields some b in [0, B].
__device__ __forceinline__ int find_frame(const int32_t* offsets, int B, long long row) {
    long long wlo = 0, whi = B;
    while (whi > wlo) {
        const long long step = (whi - wlo + kThreads - 1) / kThreads;
        const long long p = wlo + (long long)threadIdx.x * step;
        const int before = p < whi && (long long)__ldg(offsets + p + 1) <= row;
        const int k = __syncthreads_count(before);
        if (step == 1) return (int)(wlo + k);
        const long long nlo = k == 0 ? wlo : wlo + (long long)(k - 1) * step + 1;
        const long long nhi = wlo + (long long)k * step < whi ? wlo + (long long)k * step : whi;
        wlo = nlo;
        whi = nhi;
    }
    __syncthreads();  // every exit path passes the same number of barriers
    return (int)wlo;
}

// offsets[wb + j] for j in [0, n] into s_off (n <= kThreads).
__device__ __forceinline__ void load_window(const int32_t* offsets, int wb, int n, int* s_off) {
    __syncthreads();  // the previous window is no longer read
    for (int j = threadIdx.x; j <= n; j += kThreads) s_off[j] = __ldg(offsets + wb + j);
    __syncthreads();
}

// Thread layout: cpr chunks per row; thread t owns chunk column t % cpr and
// rows rg, rg + rpp, ... of a segment (rg = t / cpr, rpp = kThreads / cpr).
// GPC groups per chunk when a group is narrower than a chunk, else 1 (the
// chunk lies in group col / cpc, cpc = chunks per group).
struct Layout {
    int cpr, rpp, col, rg, cpc;
};

template <int VEC, int GPC>
__device__ __forceinline__ Layout make_layout(int C, int G) {
    Layout l;
    l.cpr = C / VEC;
    l.rpp = kThreads / l.cpr;
    l.col = threadIdx.x % l.cpr;
    l.rg = threadIdx.x / l.cpr;
    l.cpc = GPC == 1 ? (C / G) / VEC : 1;
    return l;
}

// This CTA's row range [lo, hi); false if there is nothing to do or the
// frame table's span is unusable (reported).
__device__ __forceinline__ bool range_from(long long o0, long long oB, long long capacity,
                                           unsigned* status, RangeMap& m, long long& lo,
                                           long long& hi) {
    if (o0 < 0 || oB < o0 || oB > capacity) {
        if (threadIdx.x == 0 && blockIdx.x == 0) report(status, kErrIndex);
        return false;
    }
    const long long total = oB - o0;
    if (total == 0) return false;
    m.off0 = o0;
    m.end = oB;
    m.R = (total + gridDim.x - 1) / gridDim.x;
    lo = o0 + (long long)blockIdx.x * m.R;
    hi = lo + m.R < oB ? lo + m.R : oB;
    return lo < hi;
}

__device__ __forceinline__ bool range_setup(const int32_t* offsets, int B, long long capacity,
                                            unsigned* status, RangeMap& m, long long& lo,
                                            long long& hi) {
    return range_from(__ldg(offsets), __ldg(offsets + B), capacity, status, m, lo, hi);
}

template <typename T, int VEC, int GPC>
__global__ void __launch_bounds__(kThreads, 2)
    gn_stats_kernel(const T* x, const int32_t* __restrict__ offsets, int B, int C, int G,
                    long long capacity, GnPart* __restrict__ part, unsigned* status) {
    using CK = Chunk<T, VEC>;
    using Raw = typename CK::Raw;
    constexpr int SUB = VEC / GPC;  // elements of one group inside a chunk (GPC > 1)
    __shared__ float red[kThreads * GPC * 3];
    __shared__ int s_off[kThreads + 1];
    pdl_wait();
    pdl_trigger();
    // frames must be in order (each CTA checks a share of the table)
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < B;
         i += (long long)gridDim.x * kThreads)
        if (__ldg(offsets + i + 1) < __ldg(offsets + i)) report(status, kErrIndex);
    RangeMap m;
    long long lo, hi;
    if (!range_setup(offsets, B, capacity, status, m, lo, hi)) return;
    const Layout l = make_layout<VEC, GPC>(C, G);
    // after the warp merge: row slots (warps, or thread rows) x cpr columns
    const int nrs = l.cpr < 32 ? kThreads / 32 : kThreads / l.cpr;
    const long long step = (long long)kBatch * l.rpp;

    auto segment = [&](int b, long long s0, long long s1) {
        Stats st[GPC];
        Raw cur[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const long long r = s0 + l.rg + (long long)i * l.rpp;
            if (r < s1) cur[i] = CK::load(x + r * C + l.col * VEC);
        }
        for (long long r0 = s0 + l.rg; r0 < s1; r0 += step) {
            Raw nxt[kBatch];  // next batch in flight while this one is reduced
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const long long r = r0 + step + (long long)i * l.rpp;
                if (r < s1) nxt[i] = CK::load(x + r * C + l.col * VEC);
            }
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                if (r0 + (long long)i * l.rpp < s1) {
                    float v[VEC];
                    CK::unpack(cur[i], v);
#pragma unroll
                    for (int q = 0; q < GPC; ++q) st[q].template add_chunk<SUB>(v + q * SUB);
                }
            }
#pragma unroll
            for (int i = 0; i < kBatch; ++i) cur[i] = nxt[i];
        }
        // lanes holding the same column: merge across the warp
#pragma unroll
        for (int q = 0; q < GPC; ++q)
            for (int o = l.cpr; o < 32; o <<= 1) merge_xor(st[q].n, st[q].mean, st[q].m2, o);
        const int lane = threadIdx.x & 31;
        __syncthreads();  // red[] of the previous segment has been read
        if (l.cpr >= 32 || lane < l.cpr) {
            const int slot = l.cpr < 32 ? (int)(threadIdx.x >> 5) : l.rg;
#pragma unroll
            for (int q = 0; q < GPC; ++q) {
                float* e = red + 3 * ((slot * l.cpr + l.col) * GPC + q);
                e[0] = st[q].n, e[1] = st[q].mean, e[2] = st[q].m2;
            }
        }
        __syncthreads();
        GnPart* out = part + (long long)(b + blockIdx.x) * G;
        for (int g = threadIdx.x; g < G; g += kThreads) {
            const int c0 = GPC == 1 ? g * l.cpc : g / GPC, nc = GPC == 1 ? l.cpc : 1;
            const int q = GPC == 1 ? 0 : g % GPC;
            float n = 0.f, mean = 0.f, m2 = 0.f;
            for (int rs = 0; rs < nrs; ++rs)
                for (int c = c0; c < c0 + nc; ++c) {
                    const float* e = red + 3 * ((rs * l.cpr + c) * GPC + q);
                    merge(n, mean, m2, e[0], e[1], e[2]);
                }
            out[g] = GnPart{n, mean, m2, 0.f};
        }
    };

    // frames overlapping [lo, hi), a window of kThreads frames at a time
    for (int wb = find_frame(offsets, B, lo); wb < B; wb += kThreads) {
        const int nw = B - wb < kThreads ? B - wb : kThreads;
        load_window(offsets, wb, nw, s_off);
        bool past = false;
        for (int j = 0; j < nw; ++j) {
            const long long f0 = s_off[j], f1 = s_off[j + 1];
            if (f0 >= hi) {
                past = true;
                break;
            }
            const long long s0 = f0 > lo ? f0 : lo, s1 = f1 < hi ? f1 : hi;
            if (s0 < s1) segment(wb + j, s0, s1);  // f1 < f0 is reported above
        }
        if (past || (long long)s_off[nw] >= hi) break;
    }
}

template <typename T, int VEC, int GPC>
__global__ void __launch_bounds__(kThreads, 2)
    gn_apply_kernel(const T* x, const int32_t* __restrict__ offsets, int B, int C, int G,
                    long long capacity, const GnPart* __restrict__ part, float eps,
                    const float* __restrict__ gamma, const float* __restrict__ beta, int act, T* y,
                    int part_rows, const float2* __restrict__ row_part,
                    const int32_t* __restrict__ count, unsigned* status) {
    using CK = Chunk<T, VEC>;
    using Raw = typename CK::Raw;
    static_assert(sizeof(Raw) == 16, "the row-range path moves 16-byte chunks");
    constexpr int SUB = VEC / GPC;
    __shared__ float s_mu[kMaxGroupsFast], s_inv[kMaxGroupsFast];
    __shared__ int s_off[kThreads + 1];
    // part_rows > 0: the partials come from the convolution (the kernel
    // before this one) over the rows [0, *count): one per (frame b, block c
    // of part_rows rows inside the frame) in slot b + c, one per row
    // (row_part, C/G values each) for the frame's other rows. The frame table
    // must cover exactly those rows, in order (checked here, as the
    // statistics kernel does otherwise). The table, count, gamma and
    // beta were written before that convolution started, so they are read
    // before waiting for it: the set-up overlaps its last blocks.
    __shared__ int s_count;
    const bool early = part_rows > 0;
    if (!early) pdl_wait();
    pdl_trigger();
    const Layout l = make_layout<VEC, GPC>(C, G);
    float ga[VEC], be[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        ga[k] = gamma ? __ldg(gamma + l.col * VEC + k) : 1.f;
        be[k] = beta ? __ldg(beta + l.col * VEC + k) : 0.f;
    }
    // B <= kThreads: the whole frame table (and the row count) in one round
    // trip; the checks and the row range then come from shared memory
    const bool small = B <= kThreads;
    if (small) {
        for (int j = threadIdx.x; j <= B; j += kThreads) s_off[j] = __ldg(offsets + j);
        if (threadIdx.x == 0) s_count = early ? __ldg(count) : 0;
        __syncthreads();
    }
    if (early) {
        if (small) {
            if (threadIdx.x < B && s_off[threadIdx.x + 1] < s_off[threadIdx.x])
                report(status, kErrIndex);
        } else {
            for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < B;
                 i += (long long)gridDim.x * kThreads)
                if (__ldg(offsets + i + 1) < __ldg(offsets + i)) report(status, kErrIndex);
        }
        const int o0 = small ? s_off[0] : __ldg(offsets), oB = small ? s_off[B] : __ldg(offsets + B);
        const int n = small ? s_count : __ldg(count);
        if (o0 != 0 || oB != n) {
            if (threadIdx.x == 0 && blockIdx.x == 0) report(status, kErrIndex);
            return;
        }
    }
    RangeMap m;
    long long lo, hi;
    if (small) {
        if (!range_from(s_off[0], s_off[B], capacity, status, m, lo, hi)) return;
    } else if (!range_setup(offsets, B, capacity, status, m, lo, hi)) {
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long step = (long long)kBatch * l.rpp;
    const uint64_t pol = l2_evict_first_policy();

    auto segment = [&](int b, long long f0, long long f1, long long s0, long long s1) {
        // partials of the CTAs that hold frame b: slots b + c, c in [c0, c1]
        // (clamped to the table's span, so a malformed table cannot index
        // outside the workspace)
        const long long p0 = f0 > m.off0 ? f0 : m.off0, p1 = (f1 < m.end ? f1 : m.end) - 1;
        const long long c0 = m.cta_of(p0), c1 = m.cta_of(p1);
        const GnPart* pb = part + (long long)b * G;
        // rows of the segment last to first (the statistics pass read them
        // first to last, so the most recent ones are still in L2); every
        // line is read and written here for the last time: evict first. The
        // first batch is issued before the partials are merged.
        auto row_at = [&](long long r) { return (s0 + r) * C + l.col * VEC; };
        const long long top = (s1 - s0) - 1 - l.rg;  // this thread's highest row offset
        Raw cur[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i)
            if (top - (long long)i * l.rpp >= 0)
                cur[i] = as_raw<Raw>(ld_hint(x + row_at(top - (long long)i * l.rpp), pol));
        __syncthreads();  // s_mu / s_inv of the previous segment have been read
        if (part_rows > 0) {
            // whole blocks [w0, w1) of the frame's rows [p0, p1], and its
            // other rows (at most 2 * part_rows - 2) [p0, h1) and [t0, p1]
            const long long P = part_rows, w0 = (p0 + P - 1) / P, w1 = (p1 + 1) / P;
            const bool any = w0 < w1;
            const long long nw = any ? w1 - w0 : 0;
            const long long h1 = any ? w0 * P : p1 + 1, t0 = any ? w1 * P : p1 + 1;
            const long long nh = h1 - p0, items = nw + nh + (p1 + 1 - t0);
            const float cpg = (float)(C / G);
            for (int g = warp; g < G; g += kThreads / 32) {
                float n = 0.f, mean = 0.f, m2 = 0.f;
                // kMergeBatch items per lane loaded together, then merged
                for (long long i0 = lane; i0 < items; i0 += 32 * kMergeBatch) {
                    float4 q[kMergeBatch];
#pragma unroll
                    for (int k = 0; k < kMergeBatch; ++k) {
                        const long long i = i0 + 32 * k;
                        q[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (i < nw) {
                            const GnPart p = pb[(w0 + i) * G + g];
                            q[k] = make_float4(p.n, p.mean, p.m2, 0.f);
                        } else if (i < items) {
                            const long long r = i - nw < nh ? p0 + (i - nw) : t0 + (i - nw - nh);
                            const float2 v = row_part[r * G + g];
                            q[k] = make_float4(cpg, v.x, v.y, 0.f);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < kMergeBatch; ++k) merge(n, mean, m2, q[k].x, q[k].y, q[k].z);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) merge_xor(n, mean, m2, o);
                if (lane == 0) {
                    s_mu[g] = mean;
                    s_inv[g] = 1.f / sqrtf(m2 / n + eps);
                }
            }
        } else if (c1 - c0 < 8) {
            for (int g = threadIdx.x; g < G; g += kThreads) {
                float n = 0.f, mean = 0.f, m2 = 0.f;
                for (long long c = c0; c <= c1; ++c) {
                    const GnPart q = pb[c * G + g];
                    merge(n, mean, m2, q.n, q.mean, q.m2);
                }
                s_mu[g] = mean;
                s_inv[g] = 1.f / sqrtf(m2 / n + eps);
            }
        } else {
            for (int g = warp; g < G; g += kThreads / 32) {
                float n = 0.f, mean = 0.f, m2 = 0.f;
                for (long long c = c0 + lane; c <= c1; c += 32) {
                    const GnPart q = pb[c * G + g];
                    merge(n, mean, m2, q.n, q.mean, q.m2);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) merge_xor(n, mean, m2, o);
                if (lane == 0) {
                    s_mu[g] = mean;
                    s_inv[g] = 1.f / sqrtf(m2 / n + eps);
                }
            }
        }
        __syncthreads();
        float mu[GPC], inv[GPC];
#pragma unroll
        for (int q = 0; q < GPC; ++q) {
            const int g = GPC == 1 ? l.col / l.cpc : l.col * GPC + q;
            mu[q] = s_mu[g];
            inv[q] = s_inv[g];
        }
        for (long long r0 = top; r0 >= 0; r0 -= step) {
            Raw nxt[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const long long r = r0 - step - (long long)i * l.rpp;
                if (r >= 0) nxt[i] = as_raw<Raw>(ld_hint(x + row_at(r), pol));
            }
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const long long r = r0 - (long long)i * l.rpp;
                if (r >= 0) {
                    float v[VEC];
                    CK::unpack(cur[i], v);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        const int q = k / SUB;
                        const float z = fmaf((v[k] - mu[q]) * inv[q], ga[k], be[k]);
                        v[k] = act_apply(z, act);
                    }
                    T* dst = y + row_at(r);
                    Raw packed;
                    CK::store(reinterpret_cast<T*>(&packed), v);
                    st_hint(dst, as_u4(packed), pol);
                }
            }
#pragma unroll
            for (int i = 0; i < kBatch; ++i) cur[i] = nxt[i];
        }
    };

    // frames overlapping [lo, hi) of a window (frames wb .. wb + nw - 1, so
    // holding offsets[wb + j]), last to first; true when hi is reached
    auto walk = [&](int wb, int nw, const int* so) {
        int nf = 0;  // frames of the window that start before hi
        while (nf < nw && (long long)so[nf] < hi) ++nf;
        if (early) pdl_wait();  // x and the partials come from the convolution
        for (int j = nf - 1; j >= 0; --j) {
            const long long f0 = so[j], f1 = so[j + 1];
            if (f1 < f0) continue;  // reported by the statistics kernel
            const long long s0 = f0 > lo ? f0 : lo, s1 = f1 < hi ? f1 : hi;
            if (s0 < s1) segment(wb + j, f0, f1, s0, s1);
        }
        return nf < nw || (long long)so[nw] >= hi;
    };
    if (small) {
        // the first frame of the range (the number of frames ending at or
        // before lo), found in the table in shared memory
        const int wb =
            __syncthreads_count(threadIdx.x < B && (long long)s_off[threadIdx.x + 1] <= lo);
        if (wb < B) walk(wb, B - wb, s_off + wb);
        return;
    }
    // windows of kThreads frames
    for (int wb = find_frame(offsets, B, lo); wb < B; wb += kThreads) {
        const int nw = B - wb < kThreads ? B - wb : kThreads;
        load_window(offsets, wb, nw, s_off);
        if (walk(wb, nw, s_off)) break;
    }
}

// ---- general path: one CTA per (frame, group) ----------------------------
// Any C, G and alignment. The group's part of a row is read in chunks of VEC
// elements (16 bytes, or single elements); chunk e of the slice is at row
// r0 + e / vpr, channel c0 + (e % vpr) * VEC. The first batch of every
// thread stays in registers; pass 2 walks the other batches in reverse.
struct SliceMap {
    long long r0;
    int C, c0, vpr, VEC;
    bool narrow;  // 32-bit division suffices
    __device__ __forceinline__ long long at(long long e, int& c) const {
        long long q;
        int rem;
        if (narrow) {
            const unsigned qe = (unsigned)e / (unsigned)vpr;
            q = qe;
            rem = (int)((unsigned)e - qe * (unsigned)vpr);
        } else {
            q = e / vpr;
            rem = (int)(e - q * vpr);
        }
        c = c0 + rem * VEC;
        return (r0 + q) * C + c;
    }
};

template <typename T, int VEC>
__global__ void __launch_bounds__(kThreads, 4)
    group_norm_slice_kernel(const T* x, const int32_t* __restrict__ offsets, int C, int G,
                            long long capacity, float eps, const float* __restrict__ gamma,
                            const float* __restrict__ beta, int act, T* y, unsigned* status) {
    using CK = Chunk<T, VEC>;
    using Raw = typename CK::Raw;
    constexpr long long kStride = (long long)kThreads * kBatch;
    __shared__ float red[3 * (kThreads / 32)];
    pdl_wait();
    pdl_trigger();
    const int b = blockIdx.x / G, g = blockIdx.x - b * G;
    const long long r0 = __ldg(offsets + b), r1 = __ldg(offsets + b + 1);
    if (r0 < 0 || r1 < r0 || r1 > capacity) {
        if (threadIdx.x == 0) report(status, kErrIndex);
        return;
    }
    const int cpg = C / G;
    const SliceMap map{r0, C, g * cpg, cpg / VEC, VEC, (r1 - r0) * (cpg / VEC) < (1ll << 31)};
    const long long nv = (r1 - r0) * map.vpr;
    if (nv == 0) return;

    // pass 1: statistics
    Raw keep[kBatch];
    Stats st;
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
        const long long e = threadIdx.x + (long long)i * kThreads;
        int c;
        if (e < nv) keep[i] = CK::load(x + map.at(e, c));
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
        if (threadIdx.x + (long long)i * kThreads < nv) {
            float v[VEC];
            CK::unpack(keep[i], v);
            st.add_chunk<VEC>(v);
        }
    }
    for (long long base = threadIdx.x + kStride; base < nv; base += kStride) {
        Raw t[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            int c;
            if (base + (long long)i * kThreads < nv)
                t[i] = CK::load(x + map.at(base + i * kThreads, c));
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (base + (long long)i * kThreads < nv) {
                float v[VEC];
                CK::unpack(t[i], v);
                st.add_chunk<VEC>(v);
            }
        }
    }
    float n = st.n, mean = st.mean, m2 = st.m2;
    block_merge(n, mean, m2, red);
    const float mu = mean;
    const float inv = 1.f / sqrtf(m2 / n + eps);

    // pass 2: normalise, affine, activation, store
    auto finish = [&](Raw r, long long off, int c) {
        float v[VEC];
        CK::unpack(r, v);
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            float z = (v[k] - mu) * inv;
            if (gamma) z *= __ldg(gamma + c + k);
            if (beta) z += __ldg(beta + c + k);
            v[k] = act_apply(z, act);
        }
        CK::store(y + off, v);
    };
    for (long long j = (nv - 1) / kStride; j >= 1; --j) {
        const long long base = threadIdx.x + j * kStride;
        Raw t[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            int c;
            if (base + (long long)i * kThreads < nv)
                t[i] = CK::load(x + map.at(base + i * kThreads, c));
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (base + (long long)i * kThreads < nv) {
                int c;
                const long long off = map.at(base + i * kThreads, c);
                finish(t[i], off, c);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
        const long long e = threadIdx.x + (long long)i * kThreads;
        if (e < nv) {
            int c;
            const long long off = map.at(e, c);
            finish(keep[i], off, c);
        }
    }
}

// ---- cluster path: one pass over memory ------------------------------------
// A unit is one frame's rows of one part of the channels (128 bytes of a row,
// or one whole group where that is wider). The g CTAs of a unit (part of a
// cluster of kClCtas) split its rows, each keeping its rows in shared memory
// from the statistics to the normalisation, so that x is read once: a slot of
// 16 bytes belongs to one thread, which copies it in (cp.async), sums it,
// normalises it and stores it, and then starts the copy of the next unit's
// chunk into it. Reads of the next unit thus overlap the writes of this one,
// and no barrier guards the slots; the block only meets to merge statistics,
// the CTAs of a unit through each other's shared memory and the cluster's
// barrier. Rows past kClSlots per thread are read a second time instead. g is
// the fewest CTAs that hold an average frame, or more where there would be
// idle ones, chosen on the device from the frame table (the same in every CTA).
// Frames of very different sizes are taken by size (gn_cluster_uneven): by the
// average alone one frame of 10475 rows among 63 empty ones fell to 4 CTAs (48
// us; 17-19 us as it is, 21 us by the row ranges; 8 such frames 70, 23 and 31 us;
// every other frame 78, 61 and 66 us; 512 channels, one frame: 92, 24 and 27 us).
// Telling them apart, behind the first copies, costs every call 0.5-1.5 us (64 x
// 10475 94.7 -> 96.4 us).
// Two CTAs share an SM, so that one's arithmetic overlaps the other's memory
// accesses.
// The issue slots bound it next to memory, hence the packed arithmetic and four
// chunks to a merge: 64 frames x 10475 x 128 bf16 (343 MB read and written) 112
// us by the row ranges (two passes over x), 137 us here with a merge per chunk
// and scalar arithmetic, 96 us as it is (3.6 TB/s; 36 clusters take the 256
// units in 8 rounds, the last of them nearly empty). At 25% / 5% density 39 /
// 24 -> 29 / 14 us. 512 threads a CTA: 120 us; three CTAs an SM: 97 us.
constexpr int kClCtas = 8;
constexpr int kClThreads = 256;
constexpr int kClSlots = 24;
constexpr int kClGroup = 8;  // slots per cp.async group
constexpr int kClList = 512;  // frames listed at most
constexpr size_t kClSlotBytes = (size_t)kClSlots * kClThreads * 16;

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ float ld_cluster(uint32_t addr, int rank) {
    uint32_t a;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(a) : "memory");
    return v;
}

// Two fp32 values in one 64-bit register pair: the packed instructions do
// both in one issue slot, which is what this kernel runs out of first.
__device__ __forceinline__ uint64_t pk(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpk(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// merge, and onto nothing exactly, whatever nb.
__device__ __forceinline__ void merge_into(float& n, float& mean, float& m2, float nb, float mb,
                                           float qb) {
    if (n == 0.f) n = nb, mean = mb, m2 = qb;
    else merge(n, mean, m2, nb, mb, qb);
}
__device__ __forceinline__ void merge_into_xor(float& n, float& mean, float& m2, int o) {
    const float nb = __shfl_xor_sync(0xffffffffu, n, o);
    const float mb = __shfl_xor_sync(0xffffffffu, mean, o);
    const float qb = __shfl_xor_sync(0xffffffffu, m2, o);
    merge_into(n, mean, m2, nb, mb, qb);
}

// Stats of 4 chunks at once: their mean about the first value, then the
// squares about that mean, one merge (a group of equal values keeps exactly
// that mean and M2 = 0, as with add_chunk).
template <int VEC, class Raw, class CK>
__device__ __forceinline__ void add_four(Stats& st, const Raw (&raw)[4]) {
    constexpr int N = 4 * VEC;
    uint64_t v[N / 2];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float f[VEC];
        CK::unpack(raw[c], f);
#pragma unroll
        for (int k = 0; k < VEC / 2; ++k) v[c * (VEC / 2) + k] = pk(f[2 * k], f[2 * k + 1]);
    }
    float first, other;
    unpk(v[0], first, other);
    const uint64_t shift = pk(-first, -first);
    uint64_t s0 = add2(v[0], shift), s1 = add2(v[1], shift);
#pragma unroll
    for (int k = 2; k < N / 2; k += 2) {
        s0 = add2(s0, add2(v[k], shift));
        s1 = add2(s1, add2(v[k + 1], shift));
    }
    float a, b;
    unpk(add2(s0, s1), a, b);
    const float cm = first + (a + b) * (1.f / N);
    const uint64_t off = pk(-cm, -cm);
    uint64_t q0 = 0, q1 = 0;  // +0, +0
#pragma unroll
    for (int k = 0; k < N / 2; k += 2) {
        const uint64_t d0 = add2(v[k], off), d1 = add2(v[k + 1], off);
        q0 = fma2(d0, d0, q0);
        q1 = fma2(d1, d1, q1);
    }
    unpk(add2(q0, q1), a, b);
    const float nn = st.n + (float)N;
    const float d = cm - st.mean;
    const float r = (float)N * __frcp_rn(nn);
    st.mean = fmaf(d, r, st.mean);
    st.m2 += (a + b) + d * d * st.n * r;
    st.n = nn;
}

struct ClShared {  // behind the slots
    float red[kClThreads / 32][32][3];
    float part[2][32][3];  // this CTA's sums of the unit, by round parity
    float mu[32], inv[32];
    int warp[kClThreads / 32];
    int order[kClList];  // frames in the order they are taken
};
constexpr size_t kClSmem = kClSlotBytes + sizeof(ClShared);

template <typename T>
struct ClArgs {
    const T* x;
    const int32_t* offsets;
    int B, C, pc_max, cpc;
    float eps;
    const float *gamma, *beta;
    T* y;
    long long o0, oB;  // the table's ends

    // half-width parts where the slots of a cluster do not hold a frame of
    // `rows` rows at full width
    __device__ int held() const { return kClCtas * kClSlots * (kClThreads / pc_max); }
    __device__ int part_chunks(long long rows) const {
        return rows > held() && pc_max / 2 >= cpc && pc_max / 2 >= 4 ? pc_max / 2 : pc_max;
    }
    // CTAs of a unit, frames of `rows` rows on average
    __device__ int ctas(long long frames, long long rows, int pc) const {
        const long long units = frames * (C / (16 / (int)sizeof(T)) / pc);
        int g = 1;
        while (g < kClCtas &&
               (rows > (long long)g * kClSlots * (kClThreads / pc) || units * g * 2 <= gridDim.x))
            g *= 2;
        return g;
    }
};

// The frames from..to - 1 of the table (kListed: of the listed order), without
// those above skip rows, in parts of pc chunks, g CTAs a unit, unit after unit
// over the clusters. par: parity of the rounds so far. go_on() is asked behind
// the first copies; without it nothing is done.
template <typename T, int ACT, bool kListed, class GoOn>
__device__ __forceinline__ void gn_cluster_run(const ClArgs<T>& a, int from, int to, int pc, int g,
                                               int skip, int& par, GoOn&& go_on) {
    constexpr int VEC = 16 / (int)sizeof(T);
    using CK = Chunk<T, VEC>;
    using Raw = typename CK::Raw;
    constexpr int kWarps = kClThreads / 32;
    extern __shared__ __align__(16) uint8_t slots[];
    ClShared& sh = *reinterpret_cast<ClShared*>(slots + kClSlotBytes);
    const T* const x = a.x;
    const int32_t* const __restrict__ offsets = a.offsets;
    const float *const __restrict__ gamma = a.gamma, *const __restrict__ beta = a.beta;
    T* const y = a.y;
    const int C = a.C, cpc = a.cpc;
    const float eps = a.eps;
    const long long o0 = a.o0, oB = a.oB;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rank = blockIdx.x % kClCtas, cluster = blockIdx.x / kClCtas;
    const int clusters = gridDim.x / kClCtas;
    const int parts = C / VEC / pc;
    const int rpp = kClThreads / pc;  // rows of a slot
    const long long units = (long long)(to - from) * parts;
    const int per = kClCtas / g;  // units of a cluster at a time
    const int sub = rank / g, r = rank - sub * g;
    const long long rounds = (units + (long long)clusters * per - 1) / ((long long)clusters * per);
    const int tc = t % pc, tr = t / pc;
    const int groups = pc / cpc;
    const uint32_t slot0 = smem_u32(slots) + (uint32_t)t * 16u;

    // a round's unit: this thread's first chunk, and how many rows of the CTA's
    // share lie at and after it (slot i holds the chunk i * rpp rows further)
    struct Share {
        long long at;  // element offset of the first chunk
        int rows, col;
    };
    auto locate = [&](long long round) {
        Share s{0, 0, tc * VEC};
        const long long u = (round * clusters + cluster) * per + sub;
        if (round >= rounds || u >= units) return s;
        const int f = (int)(u / parts), b = kListed ? sh.order[from + f] : from + f;
        s.col = ((int)(u - (long long)f * parts) * pc + tc) * VEC;
        const long long f0 = __ldg(offsets + b), f1 = __ldg(offsets + b + 1);
        if (f0 < o0 || f1 < f0 || f1 > oB) return s;  // reported above, or outside the span
        const long long n = f1 - f0, r0 = f0 + n * r / g, r1 = f0 + n * (r + 1) / g;
        if (!kListed && n > skip) return s;
        s.rows = (int)(r1 - r0) - tr;
        s.at = (r0 + tr) * C + s.col;
        return s;
    };
    const long long step = (long long)rpp * C;
    auto copies = [&](const Share& s, int i0, int i1) {
#pragma unroll 4
        for (int i = i0; i < i1; ++i)
            if (i * rpp < s.rows)
                cp_async_16(slot0 + (uint32_t)i * (kClThreads * 16u), x + s.at + i * step, true);
        cp_async_commit();
    };
    auto slot = [&](int i) {
        return *reinterpret_cast<const Raw*>(slots + (size_t)(i * kClThreads + t) * 16);
    };

    Share cur = locate(0);
    for (int i = 0; i < kClSlots; i += kClGroup) copies(cur, i, i + kClGroup);
    if (!go_on()) {
        cp_async_wait_all();
        return;
    }
    for (long long round = 0; round < rounds; ++round, par ^= 1) {
        // statistics
        Stats st;
        const int mine = cur.rows > 0 ? (cur.rows + rpp - 1) / rpp : 0;  // chunks of this thread
        auto add = [&](int i0) {
            int i = i0;
            for (; i + 4 <= i0 + kClGroup && i + 4 <= mine; i += 4) {
                const Raw raw[4] = {slot(i), slot(i + 1), slot(i + 2), slot(i + 3)};
                add_four<VEC, Raw, CK>(st, raw);
            }
            for (; i < i0 + kClGroup && i < mine; ++i) {
                float v[VEC];
                CK::unpack(slot(i), v);
                st.template add_chunk<VEC>(v);
            }
        };
        static_assert(kClSlots == 3 * kClGroup, "three copy groups a unit");
        cp_async_wait_group<2>();
        add(0);
        cp_async_wait_group<1>();
        add(kClGroup);
        cp_async_wait_group<0>();
        add(2 * kClGroup);
        // chunks without a slot
        int ex = kClSlots;
        for (; ex + 4 <= mine; ex += 4) {
            Raw raw[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) raw[k] = CK::load(x + cur.at + (ex + k) * step);
            add_four<VEC, Raw, CK>(st, raw);
        }
        for (; ex < mine; ++ex) {
            float v[VEC];
            CK::unpack(CK::load(x + cur.at + ex * step), v);
            st.template add_chunk<VEC>(v);
        }
        // lanes of a group (cpc chunk columns, every row of the warp)
        for (int o = 1; o < cpc; o <<= 1) merge_into_xor(st.n, st.mean, st.m2, o);
        for (int o = pc; o < 32; o <<= 1) merge_into_xor(st.n, st.mean, st.m2, o);
        if (lane < pc && lane % cpc == 0) {
            float* e = sh.red[warp][lane / cpc];
            e[0] = st.n, e[1] = st.mean, e[2] = st.m2;
        }
        __syncthreads();
        if (t < groups) {
            float n = 0.f, mean = 0.f, m2 = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w)
                merge_into(n, mean, m2, sh.red[w][t][0], sh.red[w][t][1], sh.red[w][t][2]);
            sh.part[par][t][0] = n, sh.part[par][t][1] = mean, sh.part[par][t][2] = m2;
        }
        if (g > 1) cluster_sync();
        else __syncthreads();
        for (int q = warp; q < groups; q += kWarps) {
            float n = 0.f, mean = 0.f, m2 = 0.f;
            if (lane < g) {
                const uint32_t e = smem_u32(&sh.part[par][q][0]);
                n = ld_cluster(e, sub * g + lane);
                mean = ld_cluster(e + 4u, sub * g + lane);
                m2 = ld_cluster(e + 8u, sub * g + lane);
            }
            for (int o = 1; o < g; o <<= 1) merge_into_xor(n, mean, m2, o);
            if (lane == 0) {
                sh.mu[q] = mean;
                sh.inv[q] = 1.f / sqrtf(m2 / n + eps);
            }
        }
        __syncthreads();
        const float mu = sh.mu[tc / cpc], inv = sh.inv[tc / cpc];
        const uint64_t off = pk(-mu, -mu);
        uint64_t sc[VEC / 2], be[VEC / 2];
#pragma unroll
        for (int k = 0; k < VEC / 2; ++k) {
            const int c = cur.col + 2 * k;
            sc[k] = gamma ? pk(inv * __ldg(gamma + c), inv * __ldg(gamma + c + 1)) : pk(inv, inv);
            be[k] = beta ? pk(__ldg(beta + c), __ldg(beta + c + 1)) : 0;
        }
        auto finish = [&](Raw raw, int i) {
            float v[VEC];
            CK::unpack(raw, v);
#pragma unroll
            for (int k = 0; k < VEC / 2; ++k) {
                const uint64_t z = fma2(add2(pk(v[2 * k], v[2 * k + 1]), off), sc[k], be[k]);
                float z0, z1;
                unpk(z, z0, z1);
                if (ACT == HC_ACT_ELU) {  // max(z, 0) + (exp(min(z, 0)) - 1)
                    const uint64_t e = pk(__expf(fminf(z0, 0.f)), __expf(fminf(z1, 0.f)));
                    unpk(add2(pk(fmaxf(z0, 0.f), fmaxf(z1, 0.f)), add2(e, pk(-1.f, -1.f))), v[2 * k],
                         v[2 * k + 1]);
                } else {
                    v[2 * k] = act_fixed<ACT>(z0);
                    v[2 * k + 1] = act_fixed<ACT>(z1);
                }
            }
            Raw packed;
            CK::store(reinterpret_cast<T*>(&packed), v);
            __stcs(reinterpret_cast<uint4*>(y + cur.at + i * step), as_u4(packed));
        };
        ex = kClSlots;
        for (; ex + 4 <= mine; ex += 4) {
            Raw raw[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) raw[k] = CK::load(x + cur.at + (ex + k) * step);
#pragma unroll
            for (int k = 0; k < 4; ++k) finish(raw[k], ex + k);
        }
        for (; ex < mine; ++ex) finish(CK::load(x + cur.at + ex * step), ex);
        // every slot: this unit's chunk out, then the next unit's on its way in
        const Share next = locate(round + 1);
        for (int i0 = 0; i0 < kClSlots; i0 += kClGroup) {
#pragma unroll 4
            for (int i = i0; i < i0 + kClGroup; ++i)
                if (i < mine) finish(slot(i), i);
            copies(next, i0, i0 + kClGroup);
        }
        cur = next;
    }
    if (g > 1) cluster_sync();  // no CTA goes on or leaves while another reads its sums
}

// Uneven frames: those far above the average first (all, where whole clusters
// take an average frame too), by whole clusters, then the others; both by
// falling size, so that the clusters' shares are even, and without the empty
// ones. Of many frames only the large ones are listed (the bound keeps them
// few enough). Out of line: the even frames' code is what it is without this.
template <typename T, int ACT>
__device__ __noinline__ void gn_cluster_uneven(const ClArgs<T> a, int largest, int pc_avg, int g_avg) {
    constexpr int kWarps = kClThreads / 32;
    extern __shared__ __align__(16) uint8_t slots[];
    ClShared& sh = *reinterpret_cast<ClShared*>(slots + kClSlotBytes);
    int2* const frame = reinterpret_cast<int2*>(slots);  // (frame, rows); the slots are free yet
    static_assert(kClList * sizeof(int2) <= kClSlotBytes, "the list fits");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, B = a.B;
    const long long total = a.oB - a.o0, avg = (total + B - 1) / B;
    int large = 2 * avg < a.held() ? (int)(2 * avg) : a.held();
    if (large < total / kClList) large = (int)(total / kClList);
    const int fits = g_avg * kClSlots * (kClThreads / pc_avg);
    if (large < fits) large = fits;
    const bool all = B <= kClList;
    if (all && g_avg == kClCtas) large = 0;
    int listed = 0;
    for (int i0 = 0; i0 < B; i0 += kClThreads) {
        const int i = i0 + t;
        const int n = i < B ? __ldg(a.offsets + i + 1) - __ldg(a.offsets + i) : 0;
        const bool on = n > (all ? 0 : large);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        __syncthreads();  // sh.warp is free
        if (lane == 0) sh.warp[warp] = __popc(m);
        __syncthreads();
        int at = listed + __popc(m & ((1u << lane) - 1u));
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            at += w < warp ? sh.warp[w] : 0;
            listed += sh.warp[w];
        }
        if (on && at < kClList) frame[at] = make_int2(i, n);
    }
    if (listed > kClList) listed = kClList;  // a table out of order (reported)
    __syncthreads();
    int n_large = 0;
    unsigned rest = 0;  // rows of the listed frames that are not large
    for (int e = t; e < listed; e += kClThreads) {
        const int2 f = frame[e];
        int place = 0;
        for (int j = 0; j < listed; ++j) {
            const int n = frame[j].y;
            place += n > f.y || (n == f.y && j < e);
        }
        sh.order[place] = f.x;
        if (f.y > large) ++n_large;
        else rest += (unsigned)f.y;
    }
    n_large = __reduce_add_sync(0xffffffffu, n_large);
    rest = __reduce_add_sync(0xffffffffu, rest);
    __syncthreads();
    if (lane == 0) frame[warp] = make_int2(n_large, (int)rest);
    __syncthreads();
    n_large = 0, rest = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        n_large += frame[w].x;
        rest += (unsigned)frame[w].y;
    }
    __syncthreads();  // the slots are the frames' from here on
    int par = 0;
    for (int part = 0; part < (all ? 2 : 1); ++part) {
        const int from = part == 0 ? 0 : n_large, to = part == 0 ? n_large : listed;
        const int rows = part == 0 ? largest : (int)(rest / (unsigned)(to > from ? to - from : 1));
        const int pc = a.part_chunks(rows);
        gn_cluster_run<T, ACT, true>(a, from, to, pc,
                                     part == 0 ? kClCtas : a.ctas(to - from, rows, pc), 0, par,
                                     [] { return true; });
    }
    if (!all)
        gn_cluster_run<T, ACT, false>(a, 0, B, pc_avg, g_avg, large, par, [] { return true; });
}

template <typename T, int ACT>
__global__ void __launch_bounds__(kClThreads, 2)
    gn_cluster_kernel(const T* x, const int32_t* __restrict__ offsets, int B, int C, int pc_max, int cpc,
                      long long capacity, float eps, const float* __restrict__ gamma,
                      const float* __restrict__ beta, T* y, unsigned* status) {
    extern __shared__ __align__(16) uint8_t slots[];
    ClShared& sh = *reinterpret_cast<ClShared*>(slots + kClSlotBytes);
    const int t = threadIdx.x;
    pdl_wait();
    pdl_trigger();
    const long long o0 = __ldg(offsets), oB = __ldg(offsets + B);
    if (o0 < 0 || oB < o0 || oB > capacity) {
        if (t == 0 && blockIdx.x == 0) report(status, kErrIndex);
        return;  // every CTA alike
    }
    const ClArgs<T> a{x, offsets, B, C, pc_max, cpc, eps, gamma, beta, y, o0, oB};
    const long long avg = (oB - o0 + B - 1) / B;
    const int pc = a.part_chunks(avg), g = a.ctas(B, avg, pc);
    // Uneven: some frame is more than a CTA holds, and the frames' mean square
    // is well above their mean's (equal frames 1, sizes spread evenly from 0 on
    // 1.33, every other frame empty 2), unless each unit has a cluster anyway.
    // The same in every CTA.
    int largest = 0;
    bool uneven = false;
    auto even = [&] {
        float squares = 0.f;
        bool ordered = true;
#pragma unroll 4
        for (int i = t; i < B; i += kClThreads) {
            const int lo = __ldg(offsets + i), hi = __ldg(offsets + i + 1);
            if (hi < lo) ordered = false;
            const int n = hi < lo ? 0 : hi - lo;
            largest = n > largest ? n : largest;
            squares = fmaf((float)n, (float)n, squares);
        }
        if (!ordered) report(status, kErrIndex);  // frames must be in order
        largest = __reduce_max_sync(0xffffffffu, largest);
        for (int o = 16; o > 0; o >>= 1) squares += __shfl_xor_sync(0xffffffffu, squares, o);
        if ((t & 31) == 0) {
            sh.warp[t >> 5] = largest;
            sh.mu[t >> 5] = squares;
        }
        __syncthreads();
        squares = 0.f;
#pragma unroll
        for (int w = 0; w < kClThreads / 32; ++w) {
            largest = sh.warp[w] > largest ? sh.warp[w] : largest;
            squares += sh.mu[w];
        }
        const float mean = (float)(oB - o0) / (float)B;
        uneven = largest > kClSlots * (kClThreads / pc_max) && squares > 1.6f * mean * mean * (float)B &&
                 (g < kClCtas || (long long)B * (C / (16 / (int)sizeof(T)) / pc) * g > gridDim.x);
        return !uneven;
    };
    int par = 0;
    gn_cluster_run<T, ACT, false>(a, 0, B, pc, g, 0x7fffffff, par, even);
    if (uneven) gn_cluster_uneven<T, ACT>(a, largest, pc, g);
}

long long fast_grid(const DeviceCtx* ctx, long long capacity) {
    // ranges of at least ~64 rows; 2 CTAs per SM at most (the kernels' bound)
    long long grid = (capacity + 63) / 64;
    const long long cap = (long long)ctx->num_sms * 2;
    if (grid > cap) grid = cap;
    return grid < 1 ? 1 : grid;
}

template <typename T, int VEC, int GPC>
hc_status launch_fast(const DeviceCtx* ctx, const void* x, const int32_t* offsets, int B,
                      long long capacity, int C, int G, float eps, const float* gamma,
                      const float* beta, int act, void* y, cudaStream_t s) {
    const long long grid = fast_grid(ctx, capacity);
    GnPart* part = (GnPart*)stream_workspace(s, sizeof(GnPart) * (size_t)(B + grid) * G);
    if (!part) return HC_ERR_CUDA;
    hc_status st = launch_pdl(gn_stats_kernel<T, VEC, GPC>, dim3((unsigned)grid), dim3(kThreads),
                              0, s, "gn_stats_kernel", (const T*)x, offsets, B, C, G, capacity,
                              part, ctx->status);
    if (st != HC_OK) return st;
    return launch_pdl(gn_apply_kernel<T, VEC, GPC>, dim3((unsigned)grid), dim3(kThreads), 0, s,
                      "gn_apply_kernel", (const T*)x, offsets, B, C, G, capacity,
                      (const GnPart*)part, eps, gamma, beta, act, (T*)y, 0,
                      (const float2*)nullptr, (const int32_t*)nullptr, ctx->status);
}


// The part of a row that a unit of the cluster path covers, in 16-byte chunks
// (0: the path does not take this layout): 128 bytes, or one group where that
// is wider, and both whole powers of two of chunks, one thread of a warp each.
int cluster_part_chunks(int C, int cpg, int vec) {
    if (cpg % vec != 0) return 0;
    const int cpc = cpg / vec, cpr = C / vec;
    if ((cpc & (cpc - 1)) != 0 || cpc > 32) return 0;
    const int pc = cpc > 8 ? cpc : 8;
    return cpr % pc == 0 ? pc : 0;
}

template <typename T, int ACT>
hc_status launch_cluster(const DeviceCtx* ctx, const T* x, const int32_t* offsets, int B,
                         long long capacity, int C, int pc, int cpc, float eps, const float* gamma,
                         const float* beta, T* y, cudaStream_t s, bool& taken) {
    auto kernel = gn_cluster_kernel<T, ACT>;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kClCtas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = kClSmem;
    cfg.stream = s;
    cfg.attrs = attr;
    // clusters that fit the device at a time (0: none), looked up once
    static std::mutex mutex;
    static int resident[64] = {};
    static bool known[64] = {};
    int clusters = 0;
    {
        std::lock_guard<std::mutex> lock(mutex);
        if (!known[ctx->device]) {
            hc_status st = check_cuda(
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem),
                "cudaFuncSetAttribute(gn_cluster_kernel)");
            if (st == HC_OK)
                st = check_cuda(
                    cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1),
                    "cudaFuncSetAttribute(gn_cluster_kernel)");
            if (st != HC_OK) return st;
            cfg.gridDim = dim3(kClCtas);
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            resident[ctx->device] = n;
            known[ctx->device] = true;
        }
        clusters = resident[ctx->device];
    }
    taken = clusters > 0;
    if (!taken) return HC_OK;
    cfg.gridDim = dim3((unsigned)(clusters * kClCtas));
    cfg.numAttrs = 2;
    return check_cuda(cudaLaunchKernelEx(&cfg, kernel, x, offsets, B, C, pc, cpc, capacity, eps,
                                         gamma, beta, y, ctx->status),
                      "gn_cluster_kernel");
}

template <typename T>
hc_status launch_typed(const DeviceCtx* ctx, const void* x, const int32_t* offsets, int B,
                       long long capacity, int C, int G, float eps, const float* gamma,
                       const float* beta, int act, void* y, cudaStream_t s) {
    constexpr int kVec = 16 / (int)sizeof(T);
    const int cpg = C / G;
    const uintptr_t al = (uintptr_t)x | (uintptr_t)y;
    const bool aligned = C % kVec == 0 && al % 16 == 0;
    const int cpr = C / kVec;
    // Small frames: when the average frame's group slice is within twice
    // the per-thread register cache of the per-(frame, group) kernel (the
    // rest re-read from L2) and there are enough (frame, group) blocks to
    // fill the GPU, that single launch beats the two latency-bound row-range
    // launches.
    const long long avg_chunks = (capacity + B - 1) / B * (long long)(cpg / kVec);
    const bool small_frames = cpg % kVec == 0 && aligned &&
                              avg_chunks <= 2ll * kThreads * kBatch &&
                              (long long)B * G >= ctx->num_sms;
    // a test may force the per-(frame, group) kernel (1) or the row-range
    // kernels where the layout allows (2), to cover both on any shape
    const int forced = test_group_norm_path();
    const bool force_slice = forced == 1;
    const bool force_rows = forced == 2;
    const bool fast_rows = aligned && cpr >= 1 && cpr <= kThreads && (cpr & (cpr - 1)) == 0 &&
                           G <= kMaxGroupsFast && !force_slice && (force_rows || !small_frames);
    // The cluster path reads x once. It needs enough units (frames x parts) to
    // give every cluster work, else the row ranges spread few large frames over
    // the whole GPU (two 10475-row frames: the same 22.6 us either way). Small
    // frames stay with one CTA per (frame, group) while those are one wave, 4
    // an SM (64 frames x 8 groups: 6-8 us there, 10 us here); past it the
    // cluster path is ahead (256 frames x 8 groups, 655 rows: 26.8 us there,
    // 20.5 us here; 128 x 8: 16.8 and 13.6; 100 x 8: 14.4 either way).
    const int pc = aligned ? cluster_part_chunks(C, cpg, kVec) : 0;
    const bool one_wave = small_frames && (long long)B * G <= 4ll * ctx->num_sms;
    if (pc > 0 && forced == 0 && !one_wave && (long long)B * (cpr / pc) >= 16) {
        bool taken = false;
        const int cpc = cpg / kVec;
        const hc_status st =
            act == HC_ACT_ELU ? launch_cluster<T, HC_ACT_ELU>(ctx, (const T*)x, offsets, B, capacity, C, pc, cpc,
                                                              eps, gamma, beta, (T*)y, s, taken)
            : act == HC_ACT_RELU
                ? launch_cluster<T, HC_ACT_RELU>(ctx, (const T*)x, offsets, B, capacity, C, pc, cpc, eps,
                                                 gamma, beta, (T*)y, s, taken)
                : launch_cluster<T, HC_ACT_NONE>(ctx, (const T*)x, offsets, B, capacity, C, pc, cpc, eps,
                                                 gamma, beta, (T*)y, s, taken);
        if (st != HC_OK || taken) return st;
    }
    if (fast_rows && cpg % kVec == 0)
        return launch_fast<T, kVec, 1>(ctx, x, offsets, B, capacity, C, G, eps, gamma, beta, act,
                                       y, s);
    if (fast_rows && kVec % cpg == 0) {
        if (kVec / cpg == 2)
            return launch_fast<T, kVec, 2>(ctx, x, offsets, B, capacity, C, G, eps, gamma, beta,
                                           act, y, s);
        if (kVec / cpg == 4)
            return launch_fast<T, kVec, 4>(ctx, x, offsets, B, capacity, C, G, eps, gamma, beta,
                                           act, y, s);
        if constexpr (kVec == 8)
            return launch_fast<T, kVec, 8>(ctx, x, offsets, B, capacity, C, G, eps, gamma, beta,
                                           act, y, s);
    }
    const dim3 grid((unsigned)((long long)B * G));
    if (cpg % kVec == 0 && aligned)
        return launch_pdl(group_norm_slice_kernel<T, kVec>, grid, dim3(kThreads), 0, s,
                          "group_norm_slice_kernel", (const T*)x, offsets, C, G, capacity, eps,
                          gamma, beta, act, (T*)y, ctx->status);
    return launch_pdl(group_norm_slice_kernel<T, 1>, grid, dim3(kThreads), 0, s,
                      "group_norm_slice_kernel", (const T*)x, offsets, C, G, capacity, eps, gamma,
                      beta, act, (T*)y, ctx->status);
}

}  // namespace

bool group_norm_parts_supported(hc_dtype dt, int C, int G, const void* y) {
    const int cpr = C / 8;
    return dt == HC_BF16 && C % 8 == 0 && (C / G) % 8 == 0 && (uintptr_t)y % 16 == 0 &&
           cpr >= 1 && cpr <= kThreads && (cpr & (cpr - 1)) == 0 && G <= kMaxGroupsFast;
}

hc_status launch_group_norm_apply(const DeviceCtx* ctx, void* y, const int32_t* offsets, int B,
                                  long long capacity, int C, int G, const float* part,
                                  const float* rows, int part_rows, const int32_t* count,
                                  float eps, const float* gamma, const float* beta, int act,
                                  cudaStream_t s) {
    using T = __nv_bfloat16;
    return launch_pdl(gn_apply_kernel<T, 8, 1>, dim3((unsigned)fast_grid(ctx, capacity)),
                      dim3(kThreads), 0, s, "gn_apply_kernel", (const T*)y, offsets, B, C, G,
                      capacity, (const GnPart*)part, eps, gamma, beta, act, (T*)y, part_rows,
                      (const float2*)rows, count, ctx->status);
}

hc_status launch_group_norm(const DeviceCtx* ctx, const void* x, hc_dtype dt,
                            const int32_t* offsets, int B, long long capacity, int C, int G,
                            float eps, const float* gamma, const float* beta, int act, void* y,
                            cudaStream_t s) {
    if (dt == HC_F32)
        return launch_typed<float>(ctx, x, offsets, B, capacity, C, G, eps, gamma, beta, act, y, s);
    return launch_typed<__nv_bfloat16>(ctx, x, offsets, B, capacity, C, G, eps, gamma, beta, act,
                                       y, s);
}

}  // namespace hc
