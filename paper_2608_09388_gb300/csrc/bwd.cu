// Backward of the sparse spiral convolution (the chain rule on Eqs. 4-5, 6
// and 10; the paper gives the forward only). Through the Eq. 4 mapping
// rulebook[l][n] = input row j read by tap l of output row n (or -1):
//   dz[n][o]  = dy[n][o] * act'(y[n][o])           act' read off the output
//   dbias[o]  = sum_n dz[n][o]
//   dW[l*C_in + c][o] = sum_n x[j(n,l)][c] * dz[n][o]
//   dx[j][c]  = sum over taps (n, l) reading j of (dz[n] W_l^T)[c]
// Most taps of a sparse mask are absent, so every contraction runs over the
// present taps (n, l) only, gathered slot by slot. Kernels (every sum in a
// fixed order, no floating-point atomics):
//   act_bwd_kernel      dz (stored in the layer dtype) and per-block column
//                       sums of dz in fp32 (act_bwd_vec_kernel: 16-byte
//                       chunks); further blocks of the same launch list
//                       the present taps per (slot, row unit) for wgrad and
//                       count the taps of the transposed mapping per slot for dgrad.
//   wgrad               dW_l = sum over the slot's present taps: equal runs
//                       of the lists per CTA, x and dz rows gathered; tcgen05 (fp32
//                       accumulators in TMEM) or CUDA cores (fp32).
//                       bwd_collect adds a slot's runs and dbias's blocks.
//   dgrad               tap_slots: the taps of the transposed mapping listed
//                       per slot; tap GEMM: P[e] = dz[n] W_l^T for the e-th
//                       tap (n, l) of the mapping; seg_sum: every input row
//                       sums its own, consecutive rows of P, in (n, l) order.
//                       With few channels P is over all (row, slot) pairs.
// The transposed mapping itself: rb_* kernels (counts, exclusive scan, fill,
// per-row sort).
#include <cuda.h>
#include <cuda_bf16.h>

#include "hc_internal.cuh"

namespace hc {
namespace {

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) {
    return v;
}
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}
template <typename T>
__device__ __forceinline__ T from_f(float v);
template <>
__device__ __forceinline__ float from_f<float>(float v) {
    return v;
}
template <>
__device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}

__device__ __forceinline__ long long clamp_rows(const int32_t* count, long long capacity,
                                                unsigned* status) {
    long long n = *count;
    if (n < 0) {
        if (threadIdx.x == 0) report(status, kErrIndex);
        return 0;
    }
    if (n > capacity) {
        if (threadIdx.x == 0) report(status, kErrCapacity);
        return capacity;
    }
    return n;
}

// ---------------------------------------------------------------- tap counts
// Present taps, counted by the first blocks of the dz launch (they read other
// inputs than dz and hide behind it):
//   unit_cnt[l * kUnits + u]  taps of slot l in the row unit u (the rows cut
//                             into kUnits equal pieces), a warp each: where
//                             wgrad cuts the present taps into equal runs;
//   unit_list                 those taps as (j + 1, n + 1) in row order, unit
//                             u of slot l from entry l * capacity + (its
//                             first row) on (zeros mean an absent tap);
//   hist[b * L + l]           taps of slot l in the b-th of hist_blocks equal
//                             pieces of the transposed mapping: where
//                             tap_slots places them.
constexpr int kUnits = 128;

__host__ __device__ inline long long unit_rows(long long rows) {
    const long long r = (rows + kUnits - 1) / kUnits;
    return r < 64 ? 64 : r;
}

struct PrepArgs {
    int act_blocks, unit_blocks, hist_blocks, w_blocks;  // 0 = not wanted, but act_blocks
    const int32_t* rb;
    int L, x_rows;
    int32_t* unit_cnt;
    int2* unit_list;
    const int32_t* row_ptr;
    const int32_t* taps;
    int32_t* hist;
    const void* W;  // copy_w
    void* w_out;
    int C_in, Cp, Cz;
    unsigned* status;
};

// Taps of the transposed mapping (the table's end, inside its capacity).
__device__ __forceinline__ long long total_taps(const int32_t* row_ptr, int x_rows,
                                                long long capL) {
    const long long t = __ldg(row_ptr + x_rows);
    return t < 0 ? 0 : (t > capL ? capL : t);
}
// Keys outside [0, capL) count as slot 0 (their row of P is zeros).
__device__ __forceinline__ int slot_of(int key, int L, long long capL, int& n) {
    if (key < 0 || key >= capL) {
        n = -1;
        return 0;
    }
    n = key / L;
    return key - n * L;
}

__device__ void count_taps(const PrepArgs& p, const int32_t* count, long long capacity) {
    const int lane = threadIdx.x & 31;
    int b = (int)blockIdx.x;
    if (b < p.unit_blocks) {
        const int unit = b * 8 + (threadIdx.x >> 5);
        if (unit >= p.L * kUnits) return;
        long long rows = *count;
        rows = rows < 0 ? 0 : (rows > capacity ? capacity : rows);
        const long long ur = unit_rows(rows);
        const int l = unit / kUnits, u = unit - l * kUnits;
        const long long r0 = u * ur, r1 = r0 + ur < rows ? r0 + ur : rows;
        const int32_t* src = p.rb + l * capacity;
        int2* dst = p.unit_list + l * capacity + r0;
        int c = 0;
        unsigned err = 0;
        for (long long r = r0; r < r1; r += 256) {
            int j[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const long long n = r + 32 * q + lane;
                j[q] = n < r1 ? __ldg(src + n) : -1;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const bool on = j[q] >= 0 && j[q] < p.x_rows;
                if (!on && j[q] != -1) err |= kErrIndex;
                const unsigned m = __ballot_sync(0xffffffffu, on);
                if (on)
                    dst[c + __popc(m & ((1u << lane) - 1u))] =
                        make_int2(j[q] + 1, (int)(r + 32 * q + lane) + 1);
                c += __popc(m);
            }
        }
        if (lane == 0) p.unit_cnt[unit] = c;
        if (err) report(p.status, err);
        return;
    }
    b -= p.unit_blocks;
    __shared__ int s_hist[HC_MAX_SPIRAL];
    if (threadIdx.x < HC_MAX_SPIRAL) s_hist[threadIdx.x] = 0;
    __syncthreads();
    const long long capL = capacity * p.L;
    const long long T = total_taps(p.row_ptr, p.x_rows, capL);
    const long long E = (T + p.hist_blocks - 1) / p.hist_blocks;
    const long long e0 = b * E, e1 = e0 + E < T ? e0 + E : T;
    for (long long e = e0 + threadIdx.x; e - lane < e1; e += 256) {
        const bool in = e < e1;
        int n;
        const int l = in ? slot_of(__ldg(p.taps + e), p.L, capL, n) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, l);
        if (in && lane == __ffs(same) - 1) atomicAdd(&s_hist[l], __popc(same));
    }
    __syncthreads();
    if ((int)threadIdx.x < p.L) p.hist[b * p.L + threadIdx.x] = s_hist[threadIdx.x];
}

// W as the products of dgrad read it, by further blocks of the dz launch (a
// launch of its own cost 1.5 us): over all pairs (Cp > 0), W^T [Cz][L * Cp]
// with zeros where c >= C_in or o >= C_out, a 32 x 32 piece a block; else rows
// of Cz columns, 1024 entries a block.
template <typename T>
__device__ void copy_w(const PrepArgs& p, int b, int C_out) {
    __shared__ T tile[32][33];
    const T* __restrict__ W = static_cast<const T*>(p.W);
    T* __restrict__ out = static_cast<T*>(p.w_out);
    if (p.Cp == 0) {
        const long long n = (long long)p.L * p.C_in * p.Cz;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const long long i = b * 1024ll + q * 256 + threadIdx.x;
            if (i >= n) break;
            int o;
            const long long m = div32(i, p.Cz, o);
            out[i] = o < C_out ? W[m * C_out + o] : from_f<T>(0.f);
        }
        return;
    }
    const int K = p.L * p.Cp, kb = (K + 31) / 32;
    const int k0 = b % kb * 32, o0 = b / kb * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        const int k = k0 + i, l = k / p.Cp, c = k - l * p.Cp, o = o0 + tx;
        tile[i][tx] = k < K && c < p.C_in && o < C_out
                          ? W[((long long)l * p.C_in + c) * C_out + o]
                          : from_f<T>(0.f);
    }
    __syncthreads();
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        const int o = o0 + i, k = k0 + tx;
        if (k < K && o < p.Cz) out[(long long)o * K + k] = tile[tx][i];
    }
}

// ---------------------------------------------------------------- dz, dbias
// Rows of dz have `pitch` columns: C_out, or with zeros behind them up to a
// whole number of 16-byte chunks.
// Block (64, 4): thread (tx, ty) takes columns g*64 + tx of rows r0 + ty +
// 4 i of the block's row chunks (chunks blockIdx.x, + prep.act_blocks, ...); the
// four row lanes' sums meet in shared memory and the block writes one
// partial per column.
constexpr int kActRowsPerBlock = 16;

template <typename T>
__global__ void __launch_bounds__(256)
    act_bwd_kernel(const T* __restrict__ y, const T* __restrict__ dy, const int32_t* count,
                   long long capacity, int C_out, int act, T* __restrict__ dz, int pitch,
                   float* __restrict__ bpart, const PrepArgs prep, unsigned* status) {
    __shared__ float red[4][64];
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x < prep.unit_blocks + prep.hist_blocks) {
        count_taps(prep, count, capacity);
        return;
    }
    int block = (int)blockIdx.x - prep.unit_blocks - prep.hist_blocks;
    if (block < prep.w_blocks) {
        copy_w<T>(prep, block, C_out);
        return;
    }
    block -= prep.w_blocks;
    const long long rows = clamp_rows(count, capacity, status);
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    for (int g0 = 0; g0 < C_out; g0 += 64) {
        const int o = g0 + tx;
        float sum = 0.f;
        if (o < pitch)
            for (long long r0 = (long long)block * kActRowsPerBlock; r0 < rows;
                 r0 += (long long)prep.act_blocks * kActRowsPerBlock) {
                const long long r1 = r0 + kActRowsPerBlock < rows ? r0 + kActRowsPerBlock : rows;
                for (long long rb0 = r0 + ty; rb0 < r1; rb0 += 16) {
                    // four rows' loads in flight, then their arithmetic
                    float yv[4], gv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const long long r = rb0 + 4 * i;
                        const bool in = r < r1 && o < C_out;
                        yv[i] = in ? to_f(y[r * C_out + o]) : 0.f;
                        gv[i] = in ? to_f(dy[r * C_out + o]) : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const long long r = rb0 + 4 * i;
                        if (r >= r1) continue;
                        float d = 1.f;
                        if (act == HC_ACT_ELU) d = yv[i] > 0.f ? 1.f : yv[i] + 1.f;
                        else if (act == HC_ACT_RELU) d = yv[i] > 0.f ? 1.f : 0.f;
                        const float v = gv[i] * d;
                        dz[r * pitch + o] = from_f<T>(v);  // columns past C_out: zeros
                        sum += v;
                    }
                }
            }
        red[ty][tx] = sum;
        __syncthreads();
        if (ty == 0 && o < C_out)
            bpart[(long long)block * C_out + o] = ((red[0][tx] + red[1][tx]) + red[2][tx]) + red[3][tx];
        __syncthreads();
    }
}

// Vectorised dz for rows of 16-byte chunks (cpr = C_out / VEC of them,
// cpr dividing 256): a block takes kActVecItems / cpr consecutive rows
// (ranges block, + prep.act_blocks, ...); thread t always holds chunk
// t % cpr, so it sums its VEC columns over its rows in registers, and the
// 256 / cpr row lanes of a column meet in shared memory in a fixed order.
constexpr int kActVecItems = 1024;

template <typename T>
__global__ void __launch_bounds__(256)
    act_bwd_vec_kernel(const T* __restrict__ y, const T* __restrict__ dy, const int32_t* count,
                       long long capacity, int C_out, int act, T* __restrict__ dz, int,
                       float* __restrict__ bpart, const PrepArgs prep, unsigned* status) {
    constexpr int VEC = 16 / sizeof(T);
    constexpr int kPer = kActVecItems / 256;
    __shared__ float red[256 * VEC];
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x < prep.unit_blocks + prep.hist_blocks) {
        count_taps(prep, count, capacity);
        return;
    }
    int block = (int)blockIdx.x - prep.unit_blocks - prep.hist_blocks;
    if (block < prep.w_blocks) {
        copy_w<T>(prep, block, C_out);
        return;
    }
    block -= prep.w_blocks;
    const long long rows = clamp_rows(count, capacity, status);
    const int t = threadIdx.x;
    const int cpr = C_out / VEC, lanes = 256 / cpr;
    const int c = t % cpr, rl = t / cpr;
    const int R = kActVecItems / cpr;
    float sum[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) sum[k] = 0.f;
    for (long long r0 = (long long)block * R; r0 < rows; r0 += (long long)prep.act_blocks * R) {
        uint4 yv[kPer], gv[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long r = r0 + rl + (long long)q * lanes;
            if (r < rows) {
                yv[q] = *reinterpret_cast<const uint4*>(y + r * C_out + c * VEC);
                gv[q] = *reinterpret_cast<const uint4*>(dy + r * C_out + c * VEC);
            }
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const long long r = r0 + rl + (long long)q * lanes;
            if (r >= rows) continue;
            const T* yp = reinterpret_cast<const T*>(&yv[q]);
            const T* gp = reinterpret_cast<const T*>(&gv[q]);
            uint4 out;
            T* op = reinterpret_cast<T*>(&out);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                const float yk = to_f(yp[k]);
                float d = 1.f;
                if (act == HC_ACT_ELU) d = yk > 0.f ? 1.f : yk + 1.f;
                else if (act == HC_ACT_RELU) d = yk > 0.f ? 1.f : 0.f;
                const float v = to_f(gp[k]) * d;
                op[k] = from_f<T>(v);
                sum[k] += v;
            }
            *reinterpret_cast<uint4*>(dz + r * C_out + c * VEC) = out;
        }
    }
#pragma unroll
    for (int k = 0; k < VEC; ++k) red[rl * C_out + c * VEC + k] = sum[k];
    __syncthreads();
    for (int o = t; o < C_out; o += 256) {
        float s = 0.f;
        for (int j = 0; j < lanes; ++j) s += red[j * C_out + o];
        bpart[(long long)block * C_out + o] = s;
    }
}

// ---------------------------------------------------------------- transposed mapping
// taps of input row j: entries n*L + l with rulebook[l][n] == j, n < rows.
//   rb_zero    the counts
//   rb_count   counts per input row; the counter's old value is the entry's
//              place among its row's (in whatever order the blocks ran), kept
//              so that the fill needs no counters of its own
//   scan_tiles, scan_apply   ptr, the exclusive scan of the counts: sums of
//              tiles of kScanTile, then each tile behind the sums before it
//   rb_fill    every entry to its place
//   rb_sort    each row's entries in ascending order
// Each is a launch of a few microseconds bound by its one or two dependent
// round trips, so the entries of a thread go through them four at a time.
// Bench layer (16.4k rows x 12 slots into 335k input rows), whole training
// step 107.8 -> 102.2 us; 167k rows x 9 into 670k, 25% present: 572 -> 543 us
// (the fill's own counters, a third scan launch and a warp per row in the sort
// gone: scan_sums 2.9, fill 13.6 -> 7.5, sort 33 -> 8 us in the second case).
__global__ void __launch_bounds__(256) rb_zero_kernel(int32_t* __restrict__ cnt, int n) {
    pdl_wait();
    pdl_trigger();
    for (long long i = (blockIdx.x * 256ll + threadIdx.x) * 4; i < n; i += gridDim.x * 1024ll) {
        if (i + 4 <= n) {
            *reinterpret_cast<int4*>(cnt + i) = make_int4(0, 0, 0, 0);  // cnt: 16-byte aligned
        } else {
            for (long long k = i; k < n; ++k) cnt[k] = 0;
        }
    }
}

constexpr int kRbBatch = 4;  // entries of a thread in flight

// Block column blockIdx.y: slot l; rows n = thread, + the grid's threads, ...
__global__ void __launch_bounds__(256)
    rb_count_kernel(const int32_t* __restrict__ rb, const int32_t* count, long long capacity,
                    int x_rows, int32_t* __restrict__ cnt, int32_t* __restrict__ place,
                    unsigned* status) {
    pdl_wait();
    pdl_trigger();
    const long long rows = clamp_rows(count, capacity, status);
    const int32_t* src = rb + blockIdx.y * capacity;
    int32_t* dst = place + blockIdx.y * capacity;
    const long long step = gridDim.x * 256ll;
    unsigned err = 0;
    for (long long n0 = blockIdx.x * 256ll + threadIdx.x; n0 < rows; n0 += kRbBatch * step) {
        int j[kRbBatch], at[kRbBatch];
#pragma unroll
        for (int q = 0; q < kRbBatch; ++q)
            j[q] = n0 + q * step < rows ? __ldg(src + n0 + q * step) : -1;
#pragma unroll
        for (int q = 0; q < kRbBatch; ++q) {
            at[q] = -1;
            if (j[q] >= 0 && j[q] < x_rows) at[q] = atomicAdd(cnt + j[q], 1);
            else if (j[q] != -1) err |= kErrIndex;
        }
#pragma unroll
        for (int q = 0; q < kRbBatch; ++q)
            if (at[q] >= 0) dst[n0 + q * step] = at[q];
    }
    if (err) report(status, err);
}

constexpr int kScanThreads = 1024;
constexpr int kScanTile = 4 * kScanThreads;

__device__ __forceinline__ int block_excl_scan(int v, int* sh, int& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        sh[lane] = s;
    }
    __syncthreads();
    total = sh[(blockDim.x >> 5) - 1];
    const int before = w > 0 ? sh[w - 1] : 0;
    __syncthreads();
    return before + x - v;
}

// Four consecutive counts of a thread (cnt: 16-byte aligned).
__device__ __forceinline__ int4 load_counts(const int32_t* cnt, long long base, int n) {
    if (base + 4 <= n) return __ldg(reinterpret_cast<const int4*>(cnt + base));
    return make_int4(base < n ? __ldg(cnt + base) : 0, base + 1 < n ? __ldg(cnt + base + 1) : 0,
                     base + 2 < n ? __ldg(cnt + base + 2) : 0, 0);
}

__global__ void __launch_bounds__(kScanThreads)
    scan_tiles_kernel(const int32_t* __restrict__ cnt, int n, int32_t* __restrict__ tsum) {
    __shared__ int sh[32];
    pdl_wait();
    pdl_trigger();
    const int4 c = load_counts(cnt, (long long)blockIdx.x * kScanTile + threadIdx.x * 4, n);
    const int v = __reduce_add_sync(0xffffffffu, (c.x + c.y) + (c.z + c.w));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int t = __reduce_add_sync(0xffffffffu, sh[threadIdx.x]);
        if (threadIdx.x == 0) tsum[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kScanThreads)
    scan_apply_kernel(const int32_t* __restrict__ cnt, int n, const int32_t* __restrict__ tsum,
                      int32_t* __restrict__ ptr) {
    __shared__ int sh[32], s_before[32];
    pdl_wait();
    pdl_trigger();
    const long long base = (long long)blockIdx.x * kScanTile + threadIdx.x * 4;
    const int4 c = load_counts(cnt, base, n);
    // the tiles before this one
    int before = 0;
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kScanThreads) before += __ldg(tsum + i);
    before = __reduce_add_sync(0xffffffffu, before);
    if ((threadIdx.x & 31) == 0) s_before[threadIdx.x >> 5] = before;
    int total;
    int run = block_excl_scan((c.x + c.y) + (c.z + c.w), sh, total);  // synchronises
    for (int w = 0; w < kScanThreads / 32; ++w) run += s_before[w];
    const int v[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (base + i < n) {
            ptr[base + i] = run;
            run += v[i];
        }
    if (base <= n - 1 && n - 1 < base + 4) ptr[n] = run;  // the total, by the holder of n - 1
}

__global__ void __launch_bounds__(256)
    rb_fill_kernel(const int32_t* __restrict__ rb, const int32_t* count, long long capacity, int L,
                   int x_rows, const int32_t* __restrict__ ptr, const int32_t* __restrict__ place,
                   int32_t* __restrict__ taps) {
    pdl_wait();
    pdl_trigger();
    long long rows = *count;
    rows = rows < 0 ? 0 : (rows > capacity ? capacity : rows);
    const int l = blockIdx.y;
    const int32_t* src = rb + l * capacity;
    const int32_t* pl = place + l * capacity;
    const long long step = gridDim.x * 256ll;
    for (long long n0 = blockIdx.x * 256ll + threadIdx.x; n0 < rows; n0 += kRbBatch * step) {
        int j[kRbBatch], at[kRbBatch];
#pragma unroll
        for (int q = 0; q < kRbBatch; ++q) {
            const bool in = n0 + q * step < rows;
            j[q] = in ? __ldg(src + n0 + q * step) : -1;
            at[q] = in ? __ldg(pl + n0 + q * step) : 0;  // not written where j is out of range
        }
#pragma unroll
        for (int q = 0; q < kRbBatch; ++q) {
            if (j[q] >= x_rows) j[q] = -1;
            if (j[q] >= 0) at[q] += __ldg(ptr + j[q]);
        }
#pragma unroll
        for (int q = 0; q < kRbBatch; ++q)
            if (j[q] >= 0) taps[at[q]] = (int32_t)((n0 + q * step) * L + l);
    }
}

// A block takes `per` consecutive rows (at most kSortRows), whose entries are
// one slice of taps, staged in shared memory in one coalesced copy. A thread
// per entry counts the smaller entries of its row (about L of them; keys are
// unique) and writes it at that place, so the work is even however few of the
// rows have entries (5% of them in a dense input: a thread per row took twice
// as long). A slice has about L entries a row where every tap is present and
// is not even, hence sort_rows: it fits kSortKeys with a quarter to spare (with
// 256 rows at every L, the slices of 20 and more slots did not fit: 83.8k rows,
// 24 slots, all present: 719 us, 72 us as it is). A slice that does not fit all the same (a few
// rows with very many entries) is sorted row by row: up to 32 entries by a
// warp, more by one of its lanes.
constexpr int kSortRows = 256;
constexpr int kSortKeys = 5120;

constexpr int sort_rows(int L) {
    return L <= kSortKeys * 4 / 5 / kSortRows ? kSortRows : kSortRows / 2;
}
static_assert(sort_rows(HC_MAX_SPIRAL) * HC_MAX_SPIRAL <= kSortKeys * 4 / 5, "a slice fits");

__device__ __forceinline__ void insertion_sort(int32_t* taps, int a, int b) {
    for (int i = a + 1; i < b; ++i) {
        const int key = taps[i];
        int k = i - 1;
        while (k >= a && taps[k] > key) {
            taps[k + 1] = taps[k];
            --k;
        }
        taps[k + 1] = key;
    }
}

// The warp sorts taps[a, b).
__device__ __forceinline__ void sort_row(int32_t* taps, int a, int b) {
    const int lane = threadIdx.x & 31, len = b - a;
    if (len <= 1) return;
    if (len <= 32) {
        const int key = lane < len ? taps[a + lane] : 0x7fffffff;
        int rank = 0;
#pragma unroll
        for (int k = 0; k < 32; ++k) rank += __shfl_sync(0xffffffffu, key, k) < key;
        if (lane < len) taps[a + rank] = key;
    } else if (lane == 0) {
        insertion_sort(taps, a, b);
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kSortRows)
    rb_sort_kernel(const int32_t* __restrict__ ptr, int x_rows, int per, int32_t* __restrict__ taps) {
    __shared__ int32_t s_keys[kSortKeys];
    __shared__ uint8_t s_row[kSortKeys];  // row (in the block) of an entry
    __shared__ int s_ptr[kSortRows + 1];
    static_assert(kSortRows <= 256, "s_row holds a byte");
    pdl_wait();
    pdl_trigger();
    const int t = threadIdx.x;
    const long long r0 = (long long)blockIdx.x * per;
    const int n = x_rows - r0 < per ? (int)(x_rows - r0) : per;
    if (t < n) s_ptr[t] = __ldg(ptr + r0 + t);
    if (t == 0) s_ptr[n] = __ldg(ptr + r0 + n);
    __syncthreads();
    const int base = s_ptr[0], len = s_ptr[n] - base;
    if (len > kSortKeys) {
        for (int r = t >> 5; r < n; r += kSortRows / 32) sort_row(taps, s_ptr[r], s_ptr[r + 1]);
        return;
    }
    for (int i = t; i < len; i += kSortRows) s_keys[i] = taps[base + i];
    if (t < n)
        for (int i = s_ptr[t] - base; i < s_ptr[t + 1] - base; ++i) s_row[i] = (uint8_t)t;
    __syncthreads();
    for (int i = t; i < len; i += kSortRows) {
        const int key = s_keys[i], r = s_row[i];
        const int lo = s_ptr[r] - base, hi = s_ptr[r + 1] - base;
        int rank = 0;
        for (int k = lo; k < hi; ++k) rank += s_keys[k] < key;
        taps[base + lo + rank] = key;
    }
}

// ---------------------------------------------------------------- wgrad
// dW_l[c][o] = sum over the present taps (n, j) of slot l of x[j][c] dz[n][o].
// The present taps of all slots, slot by slot and in row order, are one list
// of T positions; CTA g of G takes positions [g Q, (g + 1) Q), Q = T / G
// rounded up to kBK, whatever slots and rows they fall into (its "segments":
// one per slot it touches). Cutting by taps and not by rows keeps the CTAs
// even although slot 0 (the vertex itself) is always present and the others
// are as dense as the mask. A segment's sum goes to partial g + l: within a
// CTA l rises, and a later CTA starts at the slot where the one before it
// ended, so no two segments share one, and G + L partials suffice.
constexpr int kTile = 128;
constexpr int kBK = 64;

struct WgradArgs {
    const void* x;
    const int32_t* count;
    const void* dz;
    long long capacity;
    int L, C_in, C_out;
    int z_pitch;                 // columns of a row of dz
    int c_tiles, o_tiles, G;     // grid: G x (c_tiles * o_tiles)
    const int32_t* unit_cnt;     // [L][kUnits]
    const int2* unit_list;       // [L][capacity]
    int32_t* slot_pos;           // [L + 2]: first position of each slot, T, Q (for the reduction)
    float* part;                 // [c_tiles * o_tiles][G + L][BC][kTile]
    unsigned* status;
};

// Positions of the units: s_pre[i] = present taps before unit i of the [L][kUnits]
// list, s_pre[L * kUnits] = T, by the first 256 threads of the block (the
// caller synchronises after it). red: 8 ints.
__device__ __forceinline__ void unit_positions(const int32_t* __restrict__ cnt, int n, int* s_pre,
                                               int* red) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (n + 255) / 256;
    int sum = 0;
    if (t < 256)
        for (int i = t; i < n; i += 256) s_pre[i] = __ldg(cnt + i);
    __syncthreads();
    int own[HC_MAX_SPIRAL * kUnits / 256];
    if (t < 256) {
#pragma unroll
        for (int q = 0; q < HC_MAX_SPIRAL * kUnits / 256; ++q) {
            const int i = t * per + q;
            own[q] = q < per && i < n ? s_pre[i] : 0;
            sum += own[q];
        }
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (t < 256 && lane == 31) red[warp] = x;
    __syncthreads();
    if (t < 256) {
        int run = x - sum;
        for (int w = 0; w < warp; ++w) run += red[w];
#pragma unroll
        for (int q = 0; q < HC_MAX_SPIRAL * kUnits / 256; ++q) {
            const int i = t * per + q;
            if (q < per && i < n) s_pre[i] = run;
            run += own[q];
        }
        if (t == 255) s_pre[n] = run;
    }
}

// The run of a CTA: positions [p0, p1), and its segments in order.
struct Run {
    const int* s_pre;
    int L;
    long long p0, p1;
    __device__ __forceinline__ Run(const int* pre, int L_, int G, int g) : s_pre(pre), L(L_) {
        const long long T = pre[L_ * kUnits];
        const long long Q = ((T + G - 1) / G + kBK - 1) / kBK * kBK;
        p0 = g * Q;
        p1 = p0 + Q < T ? p0 + Q : T;
    }
    // The segment at position pos < p1: its slot (l = the slot of an earlier
    // position, or 0) and its end.
    __device__ __forceinline__ long long segment(long long pos, int& l) const {
        while (s_pre[(l + 1) * kUnits] <= pos) ++l;
        const long long end = s_pre[(l + 1) * kUnits];
        return end < p1 ? end : p1;
    }
    // Entry of the unit lists (see count_taps) of position pos of slot l. u:
    // the unit of an earlier position of the slot (or the slot's first), moved
    // on to pos's: mostly the same one or the next, else searched for.
    __device__ __forceinline__ long long entry(int l, int pos, long long urows, long long capacity,
                                               int& u) const {
        if (s_pre[u + 1] <= pos && s_pre[++u + 1] <= pos) {
            int lo = u + 1, hi = (l + 1) * kUnits - 1;  // last unit with s_pre <= pos
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_pre[mid] <= pos) lo = mid;
                else hi = mid - 1;
            }
            u = lo;
        }
        return l * capacity + (u - l * kUnits) * urows + (pos - s_pre[u]);
    }
};
// tcgen05: D[o][c] (M = 128 output channels of dz, N = BC channels of x),
// both operands MN-major as gathered: per stage kBK taps, dz's rows as up to
// two and x's as BC / 64 atoms of 64 channels (kBK rows x 128 bytes each,
// 128-byte swizzle). What bounds it is the gather: a stage moves up to 32 KB
// for 2.1 MFLOP. Warp 9 (index) copies the taps' (j, n) from
// the unit lists into tables of kBK for the producers, up to kQueue ahead, by
// cp.async, so that no lookup's latency is on the gather's path. (Compacting
// the rulebook in this warp instead kept the gather waiting for 20 of 58 us
// at 25% density: the scan's shared-memory accesses queue behind the
// producers' copies.) Warps 0-3 gather
// with 16-byte cp.async, warp 8 issues the MMAs, warps 4-7 move a finished
// segment's sums from TMEM to its partial while the next one accumulates.
// 167k rows, 9 slots, 128 -> 128, 25% present: 146 -> 37 us (two thirds of the
// taps were multiplied as zeros, the lookups' latency was paid per stage);
// 16.4k rows, 12 slots, 64 -> 128, 84% present: 17.5 -> 18.9 us (the rows of
// dz are gathered per slot, 24 KB a stage). fp32, 25k rows, 9 slots, 64 -> 128,
// 24% present: 374 -> 31 us. All cold under ncu.
constexpr int kQueue = 8;
constexpr int kProducerWarps = 4, kEpilogueWarps = 4;
constexpr int kMmaWarp = kProducerWarps + kEpilogueWarps;
constexpr int kIndexWarp = kMmaWarp + 1;
constexpr int kThreadsTc = (kIndexWarp + 1) * 32;
constexpr int kAtomBytes = kBK * 128;  // 64 channels of kBK rows

template <int BC>
struct WgradCfg {
    static constexpr int kStageBytes = (2 + BC / 64) * kAtomBytes;
    static constexpr int kStages = BC == 64 ? 8 : 6;
    static constexpr uint32_t kTmemCols = 2 * BC;
    static constexpr int kBars = 2 * kStages + 2 * kQueue + 5;
    static constexpr int kMisc = kStages * kStageBytes;  // barriers, tmem address, abort flag, scan
    static constexpr int kTables = kMisc + (8 * kBars + 16 + 32 + 127) / 128 * 128;
    static constexpr int kPre = kTables + kQueue * kBK * 8;
    // kind::f16: D fp32, A and B bf16, both MN-major, N = BC, M = 128
    static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) |
                                       (1u << 16) | ((uint32_t)(BC >> 3) << 17) |
                                       ((uint32_t)(kTile >> 4) << 24);
    static size_t smem_bytes(int L) { return 1024 + kPre + sizeof(int) * ((size_t)L * kUnits + 1); }
};

template <int BC>
__global__ void __launch_bounds__(kThreadsTc, 1) wgrad_tc_kernel(const WgradArgs a) {
    using C = WgradCfg<BC>;
    constexpr int kStages = C::kStages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* const base_ptr = smem_raw + (base - raw);
    const uint32_t sBar = base + C::kMisc;
    auto full_bar = [&](int s) { return sBar + 8u * s; };
    auto empty_bar = [&](int s) { return sBar + 8u * (kStages + s); };
    auto qfull_bar = [&](int q) { return sBar + 8u * (2 * kStages + q); };
    auto qempty_bar = [&](int q) { return sBar + 8u * (2 * kStages + kQueue + q); };
    auto tfull_bar = [&](int i) { return sBar + 8u * (2 * kStages + 2 * kQueue + i); };
    auto tempty_bar = [&](int i) { return sBar + 8u * (2 * kStages + 2 * kQueue + 2 + i); };
    const uint32_t fin_bar = sBar + 8u * (2 * kStages + 2 * kQueue + 4);
    uint8_t* const misc = base_ptr + C::kMisc + 8 * C::kBars;
    volatile uint32_t* const tmem_holder = reinterpret_cast<volatile uint32_t*>(misc);
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(misc + 4);
    int* const red = reinterpret_cast<int*>(misc + 16);
    int* const s_pre = reinterpret_cast<int*>(base_ptr + C::kPre);
    const uint32_t tables = base + C::kTables;  // [kQueue][kBK] (j, n)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full_bar(s), kProducerWarps * 32);
            mbar_init(empty_bar(s), 1);
        }
        for (int q = 0; q < kQueue; ++q) {
            mbar_init(qfull_bar(q), 32);
            mbar_init(qempty_bar(q), kProducerWarps * 32);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(tfull_bar(i), 1);
            mbar_init(tempty_bar(i), kEpilogueWarps * 32);
        }
        mbar_init(fin_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32((const void*)tmem_holder), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();
    pdl_trigger();

    long long rows = *a.count;
    rows = rows < 0 ? 0 : (rows > a.capacity ? a.capacity : rows);
    unit_positions(a.unit_cnt, a.L * kUnits, s_pre, red);
    __syncthreads();
    const int g = blockIdx.x;
    const int ct = (int)blockIdx.y % a.c_tiles, ot = (int)blockIdx.y / a.c_tiles;
    const Run run(s_pre, a.L, a.G, g);
    if (g == 0 && blockIdx.y == 0 && (int)threadIdx.x <= a.L + 1) {
        const long long T = s_pre[a.L * kUnits];
        a.slot_pos[threadIdx.x] = (int)threadIdx.x <= a.L
                                      ? s_pre[threadIdx.x * kUnits]
                                      : (int)(((T + a.G - 1) / a.G + kBK - 1) / kBK * kBK);
    }

    if (warp < kProducerWarps) {
        const __nv_bfloat16* __restrict__ x = static_cast<const __nv_bfloat16*>(a.x);
        const __nv_bfloat16* __restrict__ dz = static_cast<const __nv_bfloat16*>(a.dz);
        const int t = threadIdx.x;
        // dz: 16-byte chunk t % 16 of rows t / 16 + 8 i; x: the same, or with
        // one atom chunk t % 8 of rows t / 8 + 16 i. Columns past the
        // channels are left as they are (their sums are never stored).
        constexpr int kXc = BC / 8, kXrows = kProducerWarps * 32 / kXc, kXper = kBK / kXrows;
        const int zc = t & 15, zr = t >> 4;
        const int xc = t % kXc, xrow = t / kXc;
        const int o = ot * kTile + zc * 8, c = ct * BC + xc * 8;
        const bool o_ok = o < a.C_out, c_ok = c < a.C_in;
        int st = 0;  // stage and table of the current iteration, and their phases
        uint32_t ph = 0;
        int qt = 0;
        uint32_t qph = 0;
        bool ok = true;
        int l = 0;
        for (long long pos = run.p0; pos < run.p1 && ok;) {
            const long long end = run.segment(pos, l);
            for (; pos < end; pos += kBK) {
                if (!mbar_wait(qfull_bar(qt), qph, abort_flag, a.status)) {
                    ok = false;
                    break;
                }
                const uint32_t tab = tables + (uint32_t)(qt * kBK * 8);
                int n[8], j[kXper];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    n[i] = lds_s32(tab + (uint32_t)(zr + 8 * i) * 8u + 4u) - 1;
#pragma unroll
                for (int i = 0; i < kXper; ++i)
                    j[i] = lds_s32(tab + (uint32_t)(xrow + kXrows * i) * 8u) - 1;
                mbar_arrive(qempty_bar(qt));
                if (++qt == kQueue) {
                    qt = 0;
                    qph ^= 1u;
                }
                if (!mbar_wait(empty_bar(st), ph ^ 1u, abort_flag, a.status)) {
                    ok = false;
                    break;
                }
                const uint32_t z_st = base + st * C::kStageBytes + (zc >> 3) * kAtomBytes;
                const uint32_t x_st =
                    base + st * C::kStageBytes + 2 * kAtomBytes + (xc >> 3) * kAtomBytes;
                if (o_ok)
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int r = zr + 8 * i;
                        const bool v = n[i] >= 0;
                        cp_async_16(z_st + r * 128 + (((zc & 7) ^ (r & 7)) << 4),
                                    dz + (v ? (long long)n[i] * a.C_out + o : 0), v);
                    }
                if (c_ok)
#pragma unroll
                    for (int i = 0; i < kXper; ++i) {
                        const int r = xrow + kXrows * i;
                        const bool v = j[i] >= 0;
                        cp_async_16(x_st + r * 128 + (((xc & 7) ^ (r & 7)) << 4),
                                    x + (v ? (long long)j[i] * a.C_in + c : 0), v);
                    }
                cp_async_arrive_noinc(full_bar(st));
                if (++st == kStages) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            if (pos > end) pos = end;
        }
        cp_async_wait_all();
    } else if (warp == kIndexWarp) {
        const long long urows = unit_rows(rows);
        int qt = 0;
        uint32_t qph = 0;
        bool ok = true;
        int l = 0;
        for (long long pos = run.p0; pos < run.p1 && ok;) {
            const long long end = run.segment(pos, l);
            int unit[2] = {l * kUnits, l * kUnits};
            for (; pos < end; pos += kBK) {
                // position pos + i -> entry i; zeros past the segment's end
                long long src[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const long long p = pos + lane + 32 * i;
                    src[i] = p < end ? run.entry(l, (int)p, urows, a.capacity, unit[i]) : -1;
                }
                if (!mbar_wait(qempty_bar(qt), qph ^ 1u, abort_flag, a.status)) {
                    ok = false;
                    break;
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    cp_async_8(tables + (uint32_t)((qt * kBK + lane + 32 * i) * 8),
                               a.unit_list + (src[i] >= 0 ? src[i] : 0), src[i] >= 0);
                cp_async_arrive_noinc(qfull_bar(qt));
                if (++qt == kQueue) {
                    qt = 0;
                    qph ^= 1u;
                }
            }
            pos = end;
        }
        cp_async_wait_all();
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            int st = 0;
            uint32_t ph = 0;
            int seg = 0, l = 0;
            bool ok = true;
            for (long long pos = run.p0; pos < run.p1 && ok; ++seg) {
                const long long end = run.segment(pos, l);
                const int acc = seg & 1;
                if (!mbar_wait(tempty_bar(acc), (uint32_t)(((seg >> 1) & 1) ^ 1), abort_flag,
                               a.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                bool first = true;
                for (; pos < end; pos += kBK) {
                    if (!mbar_wait(full_bar(st), ph, abort_flag, a.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    fence_proxy_async_smem();  // operands written by cp.async
                    const uint32_t z_st = base + st * C::kStageBytes, x_st = z_st + 2 * kAtomBytes;
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k) {
                        const uint64_t zd = smem_desc_sw128(z_st + k * 16 * 128, kAtomBytes, 1024);
                        const uint64_t xd = smem_desc_sw128(x_st + k * 16 * 128, kAtomBytes, 1024);
                        tc_mma_bf16(tmem_base + (uint32_t)(acc * BC), zd, xd, C::kIdesc,
                                    first ? 0u : 1u);
                        first = false;
                    }
                    tc_commit(empty_bar(st));
                    if (++st == kStages) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (!ok) break;
                tc_commit(tfull_bar(acc));
                pos = end;
            }
            tc_commit(fin_bar);
            mbar_wait_drain(fin_bar, 0, a.status);
        }
        __syncwarp();
    } else {
        const int ew = warp - kProducerWarps;  // TMEM lanes 32 ew ..: output channels
        int seg = 0, l = 0;
        for (long long pos = run.p0; pos < run.p1; ++seg) {
            const long long end = run.segment(pos, l);
            const int acc = seg & 1;
            if (!mbar_wait(tfull_bar(acc), (uint32_t)((seg >> 1) & 1), abort_flag, a.status)) break;
            tc_fence_after();
            float* dst = a.part + ((long long)blockIdx.y * (a.G + a.L) + g + l) * (BC * kTile) +
                         ew * 32 + lane;
#pragma unroll 1
            for (int cb = 0; cb < BC / 32; ++cb) {
                uint32_t r[32];
                tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(ew * 32) << 16) +
                                       (uint32_t)(acc * BC + cb * 32),
                                   r);
                tmem_ld_wait();
#pragma unroll
                for (int jj = 0; jj < 32; ++jj) dst[(cb * 32 + jj) * kTile] = __uint_as_float(r[jj]);
            }
            tc_fence_before();
            mbar_arrive(tempty_bar(acc));
            pos = end;
        }
    }
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

// CUDA cores (fp32, and bf16 shapes off the tensor cores' alignment): the
// same runs; a block reads kSimtBatch taps of the lists at a time and
// multiplies them kSimtBK at a time, the next rows in registers
// while the current ones are multiplied. 64 channels of x by 128 of dz per
// block, 4 x 8 per thread: 12 shared-memory words for 32 multiply-adds. With
// up to 16 channels of x (BC 16) a quarter of the threads covers them, and the
// four quarters take every fourth tap and add up at the end (with 64 the
// padding was multiplied: 41.9k rows, every tap present, fp32 3 -> 64 160 us
// and 80 us, 137 on tiles over all pairs; 12% of them 21 and 16 us, 45).
constexpr int kSimtBK = 16;
constexpr int kSimtBatch = 256;  // the block's threads: one entry each

template <typename T, int BC>
__global__ void __launch_bounds__(256, 2) wgrad_simt_kernel(const WgradArgs a) {
    constexpr int kParts = 64 / BC;                 // groups of threads, each with its taps
    constexpr int kXper = kSimtBK * BC / 256;       // x values a thread loads
    static_assert(BC == 64 || BC == 16, "4 x 8 outputs a thread");
    __shared__ __align__(16) float Xs[2][kSimtBK][BC];
    __shared__ __align__(16) float Zs[2][kSimtBK][kTile];
    __shared__ int s_j[kSimtBatch], s_n[kSimtBatch], red[8];
    extern __shared__ int s_pre[];  // [L * kUnits + 1]
    pdl_wait();
    pdl_trigger();
    const T* __restrict__ x = static_cast<const T*>(a.x);
    const T* __restrict__ dz = static_cast<const T*>(a.dz);
    long long rows = *a.count;
    rows = rows < 0 ? 0 : (rows > a.capacity ? a.capacity : rows);
    unit_positions(a.unit_cnt, a.L * kUnits, s_pre, red);
    __syncthreads();
    const int g = blockIdx.x;
    const int ct = (int)blockIdx.y % a.c_tiles, ot = (int)blockIdx.y / a.c_tiles;
    const Run run(s_pre, a.L, a.G, g);
    const int t = threadIdx.x;
    if (g == 0 && blockIdx.y == 0 && t <= a.L + 1) {
        const long long T_ = s_pre[a.L * kUnits];
        a.slot_pos[t] = t <= a.L ? s_pre[t * kUnits]
                                 : (int)(((T_ + a.G - 1) / a.G + kBK - 1) / kBK * kBK);
    }
    const long long urows = unit_rows(rows);
    // outputs: c = ty * 4 .., o = tx * 4 .. and 64 + tx * 4 .., of taps part, + kParts, ..
    const int tx = t & 15, ty = (t >> 4) % (BC / 4), part = (t >> 4) / (BC / 4);
    // loads: x channel t % BC of taps t / BC + (256 / BC) i; dz channel t % 128 of taps t / 128 + 2 i
    const int c = ct * BC + (t & (BC - 1)), o = ot * kTile + (t & 127);
    const bool c_ok = c < a.C_in, o_ok = o < a.C_out;
    int l = 0;
    for (long long pos = run.p0; pos < run.p1;) {
        const long long end = run.segment(pos, l);
        int unit = l * kUnits;
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) acc[i][jj] = 0.f;
        for (; pos < end; pos += kSimtBatch) {
            const int want = end - pos < kSimtBatch ? (int)(end - pos) : kSimtBatch;
            if (t < want) {
                const int2 e = __ldg(a.unit_list + run.entry(l, (int)pos + t, urows, a.capacity, unit));
                s_j[t] = e.x - 1;
                s_n[t] = e.y - 1;
            }
            __syncthreads();
            float xv[kXper], zv[8];
            auto fetch = [&](int k0) {
#pragma unroll
                for (int i = 0; i < kXper; ++i) {
                    const int k = k0 + t / BC + (256 / BC) * i;
                    const int j = k < want ? s_j[k] : -1;
                    xv[i] = j >= 0 && c_ok ? to_f(x[(long long)j * a.C_in + c]) : 0.f;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int k = k0 + (t >> 7) + 2 * i;
                    const int n = k < want ? s_n[k] : -1;
                    zv[i] = n >= 0 && o_ok ? to_f(dz[(long long)n * a.z_pitch + o]) : 0.f;
                }
            };
            fetch(0);
            int buf = 0;
            for (int k0 = 0; k0 < want; k0 += kSimtBK, buf ^= 1) {
#pragma unroll
                for (int i = 0; i < kXper; ++i)
                    Xs[buf][t / BC + (256 / BC) * i][t & (BC - 1)] = xv[i];
#pragma unroll
                for (int i = 0; i < 8; ++i) Zs[buf][(t >> 7) + 2 * i][t & 127] = zv[i];
                __syncthreads();
                if (k0 + kSimtBK < want) fetch(k0 + kSimtBK);
#pragma unroll
                for (int kk = 0; kk < kSimtBK / kParts; ++kk) {
                    const int k = kk * kParts + part;
                    const float4 xa = *reinterpret_cast<const float4*>(&Xs[buf][k][ty * 4]);
                    const float4 za = *reinterpret_cast<const float4*>(&Zs[buf][k][tx * 4]);
                    const float4 zb = *reinterpret_cast<const float4*>(&Zs[buf][k][64 + tx * 4]);
                    const float av[4] = {xa.x, xa.y, xa.z, xa.w};
                    const float bv[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int jj = 0; jj < 8; ++jj) acc[i][jj] = fmaf(av[i], bv[jj], acc[i][jj]);
                }
            }
            __syncthreads();  // the list and the buffers are free
        }
        if (kParts > 1) {  // the parts' sums onto the first's, in order
            float* const sum = &Zs[0][0][0];  // [BC][kTile]
            static_assert(kParts == 1 || BC * kTile <= 2 * kSimtBK * kTile, "a tile fits");
            for (int p = 1; p < kParts; ++p) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 8; ++jj) {
                        float& e = sum[(ty * 4 + i) * kTile + (jj / 4) * 64 + tx * 4 + jj % 4];
                        if (part == p) e = acc[i][jj];
                    }
                __syncthreads();
                if (part == 0)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int jj = 0; jj < 8; ++jj)
                            acc[i][jj] += sum[(ty * 4 + i) * kTile + (jj / 4) * 64 + tx * 4 + jj % 4];
                __syncthreads();
            }
        }
        if (part == 0) {
            float* dst = a.part + ((long long)blockIdx.y * (a.G + a.L) + g + l) * (BC * kTile);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float* d = dst + (ty * 4 + i) * kTile + tx * 4;
                *reinterpret_cast<float4*>(d) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
                *reinterpret_cast<float4*>(d + 64) =
                    make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
            }
        }
        pos = end;
    }
}

// Lists of the taps of each slot (e and its n) for dgrad.
struct SlotArgs {
    const int32_t* row_ptr;
    const int32_t* taps;
    int x_rows, L, blocks;
    long long capL;
    const int32_t* hist;   // [blocks][L]
    int32_t* slot_off;     // [L + 1]: where each slot's list starts
    int32_t* list_n;       // source row of dz, -1: zeros
    int32_t* list_e;       // row of P
    unsigned* status;
};

// Block b of a.blocks: the b-th piece of the mapping, each slot's taps behind
// those of the pieces before (their counts come with the dz launch).
__device__ void tap_slots(const SlotArgs& a, int b) {
    __shared__ int s_tot[HC_MAX_SPIRAL], s_bef[HC_MAX_SPIRAL], s_cur[HC_MAX_SPIRAL];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const long long T = total_taps(a.row_ptr, a.x_rows, a.capL);
    const long long E = (T + a.blocks - 1) / a.blocks;
    const long long e0 = b * E, e1 = e0 + E < T ? e0 + E : T;
    int key0 = e0 + t < e1 ? __ldg(a.taps + e0 + t) : 0;
    for (int l = warp; l < a.L; l += 8) {
        int tot = 0, bef = 0;
        for (int i0 = lane; i0 < a.blocks; i0 += 256) {
            int h[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                h[q] = i0 + 32 * q < a.blocks ? __ldg(a.hist + (i0 + 32 * q) * a.L + l) : 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                tot += h[q];
                bef += i0 + 32 * q < b ? h[q] : 0;
            }
        }
        tot = __reduce_add_sync(0xffffffffu, tot);
        bef = __reduce_add_sync(0xffffffffu, bef);
        if (lane == 0) {
            s_tot[l] = tot;
            s_bef[l] = bef;
        }
    }
    __syncthreads();
    if (t == 0) {
        int run = 0;
        for (int l = 0; l < a.L; ++l) {
            s_cur[l] = run + s_bef[l];
            if (b == 0) a.slot_off[l] = run;
            run += s_tot[l];
        }
        if (b == 0) a.slot_off[a.L] = run;
    }
    __syncthreads();
    unsigned err = 0;
    for (long long e = e0 + t; e - lane < e1; e += 256) {
        const bool in = e < e1;
        const int key = key0;
        if (e + 256 < e1) key0 = __ldg(a.taps + e + 256);
        int n = -1;
        const int l = in ? slot_of(key, a.L, a.capL, n) : -1;
        if (in && n < 0) err |= kErrIndex;
        const unsigned same = __match_any_sync(0xffffffffu, l);
        const int leader = __ffs(same) - 1;
        int at = 0;
        if (in && lane == leader) at = atomicAdd(&s_cur[l], __popc(same));
        at = __shfl_sync(0xffffffffu, at, leader) + __popc(same & ((1u << lane) - 1u));
        if (in) {
            a.list_n[at] = n;
            a.list_e[at] = (int)e;
        }
    }
    if (err) report(a.status, err);
}

// One launch for three short independent jobs (each on its own is a launch of
// 6 to 9 us that leaves the GPU idle):
//   blocks 0 ..          tap_slots, when dx is wanted;
//   the next dw_blocks   dW[m][o] = sum over the runs that hold taps of the
//                        slot of m, in a fixed order;
//   the rest             dbias[o] = sum of the dz blocks' column sums (8
//                        columns a block, 32 lanes of blocks each).
struct ReduceArgs {
    const float* part;
    const int32_t* slot_pos;
    int L, C_in, C_out, BC, c_tiles, G, dw_blocks;
    float* dW;
    const float* bpart;
    int act_blocks;
    float* dbias;
};

__global__ void __launch_bounds__(256)
    bwd_collect_kernel(const ReduceArgs a, const SlotArgs slots) {
    __shared__ float red[32][9], s_sum[4][64];
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x < slots.blocks) {
        tap_slots(slots, blockIdx.x);
        return;
    }
    const int block = (int)blockIdx.x - slots.blocks;
    if (block >= a.dw_blocks) {
        const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
        const int o = (block - a.dw_blocks) * 8 + tx;
        float s = 0.f;
        if (o < a.C_out)
            for (int b0 = ty; b0 < a.act_blocks; b0 += 32 * 8) {
                float v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    v[q] = b0 + 32 * q < a.act_blocks
                               ? __ldg(a.bpart + (long long)(b0 + 32 * q) * a.C_out + o)
                               : 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) s += v[q];
            }
        red[ty][tx] = s;
        __syncthreads();
        if (ty == 0 && o < a.C_out) {
            float tot = 0.f;
#pragma unroll
            for (int i = 0; i < 32; ++i) tot += red[i][tx];
            a.dbias[o] = tot;
        }
        return;
    }
    // 64 entries of dW per block and step, four threads each: thread k adds
    // the runs first + k, + 4, ... (slot 0 has the most, all rows' taps)
    const long long total = (long long)a.L * a.C_in * a.C_out;
    const int Q = a.slot_pos[a.L + 1];
    const int ei = threadIdx.x & 63, k = threadIdx.x >> 6;
    for (long long e0 = block * 64ll; e0 < total; e0 += a.dw_blocks * 64ll) {
        const long long e = e0 + ei;
        float s = 0.f;
        if (e < total) {
            int o, c;
            const int m = (int)div32(e, a.C_out, o);
            const int l = (int)div32(m, a.C_in, c);
            const int s0 = a.slot_pos[l], s1 = a.slot_pos[l + 1];
            if (s1 > s0) {
                const int tile = (o / kTile) * a.c_tiles + c / a.BC;
                const long long stride = (long long)a.BC * kTile;
                const float* src = a.part + (long long)tile * (a.G + a.L) * stride +
                                   (long long)(c % a.BC) * kTile + (o & (kTile - 1)) + l * stride;
                const int g1 = (s1 - 1) / Q;
                for (int g = s0 / Q + k; g <= g1; g += 32) {
                    float v[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) v[q] = g + 4 * q <= g1 ? src[(g + 4 * q) * stride] : 0.f;
#pragma unroll
                    for (int q = 0; q < 8; ++q) s += v[q];
                }
            }
        }
        s_sum[k][ei] = s;
        __syncthreads();
        if (k == 0 && e < total)
            a.dW[e] = ((s_sum[0][ei] + s_sum[1][ei]) + s_sum[2][ei]) + s_sum[3][ei];
        __syncthreads();
    }
}

// ---------------------------------------------------------------- dgrad
// dx[j] = sum over the taps (n, l) of row j, in (n, l) order, of dz[n] W_l^T.
// The transposed mapping lists them row by row, so with P[e] = dz[n] W_l^T
// for its e-th tap every row of dx sums consecutive rows of P. Only the
// present taps have a row in P (a [rows, L * C_in] product computes, writes
// and rounds all of them; at 25% density two thirds are absent).
// tap_slots (above) lists the taps of each slot, so that a tile of the product
// has one W_l.
struct TapGemmArgs {
    const void* dz;
    const void* W;
    const int32_t* slot_off;
    const int32_t* list_n;
    const int32_t* list_e;
    void* P;                      // [taps][Cp]
    int L, C_in, C_out, Cp, c_tiles;
    unsigned* status;
};

// Tiles of BM listed taps, slot by slot: s_tile[l] = tiles before slot l. By
// one warp; s_off[l] = the slot's first list entry.
template <int BM>
__device__ __forceinline__ void slot_tiles(const int32_t* slot_off, int L, int* s_off,
                                           int* s_tile) {
    const int lane = threadIdx.x & 31;
    const int off = lane < L ? __ldg(slot_off + lane) : 0;
    const int nxt = lane < L ? __ldg(slot_off + lane + 1) : 0;
    const int tiles = (int)(((long long)nxt - off + BM - 1) / BM);
    int x = tiles;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane < L) {
        s_off[lane] = off;
        s_tile[lane] = x - tiles;
    }
    if (lane == L - 1) {
        s_off[L] = nxt;
        s_tile[L] = x;
    }
}

// tcgen05: 128 listed taps x BN channels of W_l per item, contraction over
// C_out. A: the taps' rows of dz, gathered by cp.async as in the forward
// conv (K-major); B: rows l * C_in + c of W as they lie (K-major, C_out
// contiguous), by TMA, so no transposed copy of W is needed; both 128-byte
// swizzled. Each item is short (C_out / 64 stages), so what bounds it is the
// rows' gather and the scattered rows of P (whole 64-byte pieces). Warps 0-3
// gather (list entries two items ahead in registers), 9 loads W, 8 issues the
// MMAs, 4-7 and 10-13 round and store the item before (half of its columns
// each: with four warps the stores took longer than the gather), two
// accumulators in turn.
// With seg_sum, against the product over all (row, slot) pairs and a scattered
// sum: 114 + 107 -> 48 + 40 us at 167k rows, 9 slots, 128 -> 128, 25% present;
// 17 + 17 -> 17 + 18 us at 16.4k rows, 12 slots, 64 -> 128, 84% present; fp32,
// 25k rows, 24% present: 142 + 24 -> 38 + 13 us.
template <int BN>
struct TapCfg {
    static constexpr int kABytes = 128 * 128;
    static constexpr int kStageBytes = kABytes + BN * 128;
    static constexpr int kStages = BN == 64 ? 8 : 6;
    static constexpr uint32_t kTmemCols = 2 * BN;
    static constexpr int kBars = 3 * kStages + 5;
    static constexpr int kMisc = kStages * kStageBytes;
    static constexpr int kEpi = kMisc + (8 * kBars + 16 + 2 * 33 * 4 + 127) / 128 * 128;
    static constexpr size_t kSmem = 1024 + kEpi + 8 * 2048;
    // D fp32, A and B bf16, both K-major, N = BN, M = 128
    static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                       ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
};

// P is written once and read once soon after: its lines are kept in L2 where
// possible (evict last) and let go with their read (evict first), and dx, which
// nothing here reads again, streams past it (training step at 64 x 10475, 25%
// density, 128 MB of P: 268.8 -> 264 us).
constexpr int kTapEpilogueWarps = 8;  // 4-7 and 10-13: half of the columns each
constexpr int kTapThreads = (kIndexWarp + 1 + 4) * 32;

template <int BN>
__global__ void __launch_bounds__(kTapThreads, 1)
    tap_gemm_tc_kernel(const TapGemmArgs a, const __grid_constant__ CUtensorMap tmap_w) {
    using C = TapCfg<BN>;
    constexpr int kStages = C::kStages;
    constexpr int kWeightWarp = kIndexWarp;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* const base_ptr = smem_raw + (base - raw);
    const uint32_t sBar = base + C::kMisc;
    auto full_bar = [&](int s) { return sBar + 8u * s; };
    auto empty_bar = [&](int s) { return sBar + 8u * (kStages + s); };
    auto wfull_bar = [&](int s) { return sBar + 8u * (2 * kStages + s); };
    auto tfull_bar = [&](int i) { return sBar + 8u * (3 * kStages + i); };
    auto tempty_bar = [&](int i) { return sBar + 8u * (3 * kStages + 2 + i); };
    const uint32_t fin_bar = sBar + 8u * (3 * kStages + 4);
    uint8_t* const misc = base_ptr + C::kMisc + 8 * C::kBars;
    volatile uint32_t* const tmem_holder = reinterpret_cast<volatile uint32_t*>(misc);
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(misc + 4);
    int* const s_off = reinterpret_cast<int*>(misc + 16);
    int* const s_tile = s_off + 33;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full_bar(s), kProducerWarps * 32);
            mbar_init(wfull_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(tfull_bar(i), 1);
            mbar_init(tempty_bar(i), kTapEpilogueWarps * 32);
        }
        mbar_init(fin_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == kWeightWarp && lane == 0) prefetch_tensormap(&tmap_w);
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32((const void*)tmem_holder), C::kTmemCols);
        tmem_relinquish();
    }
    pdl_wait();
    pdl_trigger();
    if (warp == 0) slot_tiles<128>(a.slot_off, a.L, s_off, s_tile);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    const long long items = (long long)s_tile[a.L] * a.c_tiles;
    const int nkb = (a.C_out + 63) / 64;
    // item w: tile w / c_tiles (slot l, list entries [first, first + 128) of
    // the slot's), channels c0 ..
    auto locate = [&](long long w, int& l, int& first, int& c0) {
        const int tile = (int)(w / a.c_tiles);
        c0 = (int)(w - (long long)tile * a.c_tiles) * BN;
        while (s_tile[l + 1] <= tile) ++l;
        first = s_off[l] + (tile - s_tile[l]) * 128;
    };

    if (warp < kProducerWarps) {
        const __nv_bfloat16* __restrict__ dz = static_cast<const __nv_bfloat16*>(a.dz);
        const int t = threadIdx.x, q = t & 7;
        int n1[8], n2[8];  // list entries of the next item and the one after it
        int l = 0;
        auto entries = [&](long long w, int (&n)[8]) {
            int first, c0;
            if (w < items) {
                locate(w, l, first, c0);
                const int end = s_off[l + 1];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = (t >> 3) + 16 * i;
                    n[i] = r < end - first ? __ldg(a.list_n + first + r) : -1;
                }
            }
        };
        entries(blockIdx.x, n1);
        entries(blockIdx.x + (long long)gridDim.x, n2);
        int st = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (long long w = blockIdx.x; w < items && ok; w += gridDim.x) {
            int n[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                n[i] = n1[i];
                n1[i] = n2[i];
            }
            entries(w + 2ll * gridDim.x, n2);
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(empty_bar(st), ph ^ 1u, abort_flag, a.status)) {
                    ok = false;
                    break;
                }
                const int k = kb * 64 + q * 8;
                const uint32_t a_st = base + st * C::kStageBytes;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = (t >> 3) + 16 * i;
                    const bool v = n[i] >= 0 && k < a.C_out;
                    cp_async_16(a_st + r * 128 + ((q ^ (r & 7)) << 4),
                                dz + (v ? (long long)n[i] * a.C_out + k : 0), v);
                }
                cp_async_arrive_noinc(full_bar(st));
                if (++st == kStages) {
                    st = 0;
                    ph ^= 1u;
                }
            }
        }
        cp_async_wait_all();
    } else if (warp == kWeightWarp) {
        if (lane == 0) {
            long long it = 0;
            int st = 0, l = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (long long w = blockIdx.x; w < items && ok; w += gridDim.x) {
                int first, c0;
                locate(w, l, first, c0);
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait(empty_bar(st), ph ^ 1u, abort_flag, a.status)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(wfull_bar(st), BN * 128);
                    tma_load_2d(base + st * C::kStageBytes + C::kABytes, &tmap_w, kb * 64,
                                l * a.C_in + c0, wfull_bar(st));
                    ++it;
                    if (++st == kStages) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
            }
            // copies already issued land before the CTA exits; their barriers
            // count nothing else (with the gather's arrivals, which an unwinding
            // producer does not make, each would be waited for to the limit)
            if (!ok)
                for (long long j = it > kStages ? it - kStages : 0; j < it; ++j)
                    mbar_wait_drain(wfull_bar((int)(j % kStages)), (uint32_t)((j / kStages) & 1),
                                    a.status);
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            int st = 0, lt = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (long long w = blockIdx.x; w < items && ok; w += gridDim.x, ++lt) {
                const int acc = lt & 1;
                if (!mbar_wait(tempty_bar(acc), (uint32_t)(((lt >> 1) & 1) ^ 1), abort_flag,
                               a.status))
                    break;
                tc_fence_after();
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait(full_bar(st), ph, abort_flag, a.status) ||
                        !mbar_wait(wfull_bar(st), ph, abort_flag, a.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    fence_proxy_async_smem();
                    const uint32_t a_st = base + st * C::kStageBytes, b_st = a_st + C::kABytes;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        tc_mma_bf16(tmem_base + (uint32_t)(acc * BN),
                                    smem_desc_sw128(a_st + k * 32, 16, 1024),
                                    smem_desc_sw128(b_st + k * 32, 16, 1024), C::kIdesc,
                                    (kb | k) != 0 ? 1u : 0u);
                    tc_commit(empty_bar(st));
                    if (++st == kStages) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (!ok) break;
                tc_commit(tfull_bar(acc));
            }
            tc_commit(fin_bar);
            mbar_wait_drain(fin_bar, 0, a.status);
        }
        __syncwarp();
    } else {
        // lane = listed tap; its 32-column pieces leave through a 2 KB buffer
        // as in the forward conv: a store writes eight taps x 64 bytes
        const int ew = warp & 3;                       // TMEM lanes 32 ew ..
        const int half = warp < kMmaWarp ? 0 : 1;      // columns half * BN / 2 ..
        const uint32_t stage = base + C::kEpi + (half * 4 + (warp < kMmaWarp ? ew : warp - 10)) * 2048;
        __nv_bfloat16* P = static_cast<__nv_bfloat16*>(a.P);
        const uint64_t keep = l2_evict_last_policy();
        int lt = 0, l = 0, c0 = 0, c0_next = 0;
        long long e_next = -1;  // the next item's, read one item ahead
        auto entry = [&](long long w) {
            if (w >= items) return;
            int first;
            locate(w, l, first, c0_next);
            const int r = ew * 32 + lane;
            e_next = r < s_off[l + 1] - first ? __ldg(a.list_e + first + r) : -1;
        };
        entry(blockIdx.x);
        for (long long w = blockIdx.x; w < items; w += gridDim.x, ++lt) {
            const long long e = e_next;
            c0 = c0_next;
            entry(w + gridDim.x);
            const int acc = lt & 1;
            long long ek[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) ek[k] = __shfl_sync(0xffffffffu, e, 8 * k + (lane >> 2));
            if (!mbar_wait(tfull_bar(acc), (uint32_t)((lt >> 1) & 1), abort_flag, a.status)) break;
            tc_fence_after();
#pragma unroll 1
            for (int cb = half * (BN / 64); cb < (half + 1) * (BN / 64); ++cb) {
                uint32_t r[32];
                tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(ew * 32) << 16) +
                                       (uint32_t)(acc * BN + cb * 32),
                                   r);
                tmem_ld_wait();
#pragma unroll
                for (int j8 = 0; j8 < 4; ++j8) {
                    uint32_t p[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const __nv_bfloat162 v =
                            __floats2bfloat162_rn(__uint_as_float(r[8 * j8 + 2 * h]),
                                                  __uint_as_float(r[8 * j8 + 2 * h + 1]));
                        p[h] = *reinterpret_cast<const uint32_t*>(&v);
                    }
                    sts_v4(stage + (uint32_t)(lane * 64 + ((j8 ^ ((lane >> 1) & 3)) << 4)),
                           make_uint4(p[0], p[1], p[2], p[3]));
                }
                __syncwarp();
                const int col = c0 + cb * 32 + (lane & 3) * 8;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int R = 8 * k + (lane >> 2);
                    const uint4 v =
                        lds_u4(stage + (uint32_t)(R * 64 + (((lane & 3) ^ ((R >> 1) & 3)) << 4)));
                    if (col < a.Cp && ek[k] >= 0) st_hint(P + ek[k] * a.Cp + col, v, keep);
                }
                __syncwarp();
            }
            tc_fence_before();
            mbar_arrive(tempty_bar(acc));
        }
    }
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

// CUDA cores (fp32): 128 listed taps x 64 channels per item, 8 x 4 per thread over
// chunks of 32 of C_out, the next chunk in registers while one is multiplied.
// Both operands' rows are contiguous along C_out and are turned round on their
// way into shared memory: a warp loads 8 values of 4 rows at a time, which are
// 32-byte pieces in global memory and 32 different banks in shared memory.
// Shared memory returns one word per lane and clock: 8 x 4 reads 12 for 32
// multiply-adds (4 x 4 reads 8 for 16: 38 us instead of 35, 25k rows, 64 ->
// 128, 24% of the taps present).
constexpr int kTgBM = 128, kTgBN = 64, kTgBK = 32;

__global__ void __launch_bounds__(256, 2) tap_gemm_simt_kernel(const TapGemmArgs a) {
    __shared__ __align__(16) float As[kTgBK][kTgBM + 4];
    __shared__ __align__(16) float Bs[kTgBK][kTgBN + 4];
    __shared__ int s_off[33], s_tile[33], s_e[kTgBM];
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x < 32) slot_tiles<kTgBM>(a.slot_off, a.L, s_off, s_tile);
    __syncthreads();
    const float* __restrict__ dz = static_cast<const float*>(a.dz);
    const float* __restrict__ W = static_cast<const float*>(a.W);
    float* __restrict__ P = static_cast<float*>(a.P);
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    // loads: k = kl + 8 j; taps ra + 4 i, channels rb + 4 i
    const int kl = t & 7, ra = (t >> 5) * 16 + ((t >> 3) & 3), rb = (t >> 5) * 8 + ((t >> 3) & 3);
    const long long items = (long long)s_tile[a.L] * a.c_tiles;
    int l = 0;
    for (long long w = blockIdx.x; w < items; w += gridDim.x) {
        const int tile = (int)(w / a.c_tiles);
        const int c0 = (int)(w - (long long)tile * a.c_tiles) * kTgBN;
        while (s_tile[l + 1] <= tile) ++l;
        const int first = s_off[l] + (tile - s_tile[l]) * kTgBM, end = s_off[l + 1];
        if (t < kTgBM) s_e[t] = t < end - first ? __ldg(a.list_e + first + t) : -1;
        long long za[4], wb[2];  // first element of this thread's rows, -1: none
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = ra + 4 * i;
            const int n = r < end - first ? __ldg(a.list_n + first + r) : -1;
            za[i] = n >= 0 ? (long long)n * a.C_out : -1;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c = c0 + rb + 4 * i;
            wb[i] = c < a.C_in ? ((long long)l * a.C_in + c) * a.C_out : -1;
        }
        float acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
        float av[4][4], bv[2][4];
        auto fetch = [&](int k0) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = k0 + kl + 8 * j;
                const bool in = k < a.C_out;
#pragma unroll
                for (int i = 0; i < 4; ++i) av[i][j] = in && za[i] >= 0 ? dz[za[i] + k] : 0.f;
#pragma unroll
                for (int i = 0; i < 2; ++i) bv[i][j] = in && wb[i] >= 0 ? W[wb[i] + k] : 0.f;
            }
        };
        fetch(0);
        for (int k0 = 0; k0 < a.C_out; k0 += kTgBK) {
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
                for (int i = 0; i < 4; ++i) As[kl + 8 * j][ra + 4 * i] = av[i][j];
#pragma unroll
                for (int i = 0; i < 2; ++i) Bs[kl + 8 * j][rb + 4 * i] = bv[i][j];
            }
            __syncthreads();
            if (k0 + kTgBK < a.C_out) fetch(k0 + kTgBK);
#pragma unroll 8
            for (int k = 0; k < kTgBK; ++k) {
                const float4 xa = *reinterpret_cast<const float4*>(&As[k][ty * 8]);
                const float4 xb = *reinterpret_cast<const float4*>(&As[k][ty * 8 + 4]);
                const float4 w4 = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
                const float xr[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
                const float wr[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xr[i], wr[j], acc[i][j]);
            }
        }
        // P's rows are whole 16-byte chunks (Cp)
        const int c = c0 + tx * 4;
        if (c < a.Cp)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const long long e = s_e[ty * 8 + i];
                if (e >= 0) *reinterpret_cast<float4*>(P + e * a.Cp + c) =
                    make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            }
        __syncthreads();  // s_e is free
    }
}

// dx[j] = sum of P[ptr[j]] .. P[ptr[j + 1] - 1]. A block takes R consecutive
// rows, their table in shared memory. Most rows of a dense input have no tap:
// those with taps are listed first, so that every thread of the block then has
// a (row, 16-byte chunk) item to sum, four taps in flight, and the others are
// zeroed by stores in order. (With the items dealt out row by row, empty rows
// included, the few long rows of a warp ran one after the other: 79 us at 335k
// rows, 5% of them with taps.) Short ranges, one block each: a compact input's
// active rows are its first ones, so with longer ranges (R = 1024) a quarter
// of the blocks had all the work at 25% density (103 us instead of 40). A
// row whose range leaves the table is reported and becomes zeros.
constexpr int kSegRows = 128;

// kKeys: P has a row per key n*L + l (the product over all pairs), and e's row
// is that of taps[e]; keys that no row has are reported and skipped.
template <typename T, bool kKeys>
__global__ void __launch_bounds__(256, 6)
    seg_sum_kernel(const T* __restrict__ P, const int32_t* __restrict__ ptr,
                   const int32_t* __restrict__ taps, int x_rows, int C_in, int Cp, long long capL,
                   T* __restrict__ dx, int vec_ok, unsigned* status) {
    constexpr int VEC = 16 / (int)sizeof(T);
    __shared__ int32_t s_ptr[kSegRows + 1];
    __shared__ uint16_t s_busy[kSegRows];
    __shared__ uint8_t s_on[kSegRows];
    __shared__ int s_nb;
    pdl_wait();
    pdl_trigger();
    const int t = threadIdx.x, lane = t & 31;
    const int cpr = Cp / VEC;
    const long long r0 = (long long)blockIdx.x * kSegRows;
    const int n = x_rows - r0 < kSegRows ? (int)(x_rows - r0) : kSegRows;
    if (t <= n) s_ptr[t] = __ldg(ptr + r0 + t);
    const long long total = total_taps(ptr, x_rows, capL);
    if (t == 0) s_nb = 0;
    __syncthreads();
    bool on = false;
    if (t < n) {
        const int a0 = s_ptr[t], b0 = s_ptr[t + 1];
        const bool ok = a0 >= 0 && b0 >= a0 && b0 <= total;
        if (!ok) report(status, kErrIndex);
        on = ok && b0 > a0;
        s_on[t] = on ? 1 : 0;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    int at = 0;
    if (lane == 0 && bal) at = atomicAdd(&s_nb, __popc(bal));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (on) s_busy[at + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)t;
    __syncthreads();
    auto store = [&](long long row, int col, const float* v) {
        T* dst = dx + row * C_in + col;
        if (vec_ok) {
            uint4 out;
            T* ov = reinterpret_cast<T*>(&out);
#pragma unroll
            for (int k = 0; k < VEC; ++k) ov[k] = from_f<T>(v[k]);
            __stcs(reinterpret_cast<uint4*>(dst), out);
        } else {
#pragma unroll
            for (int k = 0; k < VEC; ++k)
                if (col + k < C_in) dst[k] = from_f<T>(v[k]);
        }
    };
    const uint64_t let_go = l2_evict_first_policy();
    const int nb = s_nb;
    if (nb < n) {
        const float zero[VEC] = {};
        for (int f = t; f < n * cpr; f += 256) {
            const int i = (unsigned)f / (unsigned)cpr;
            if (!s_on[i]) store(r0 + i, (f - i * cpr) * VEC, zero);
        }
    }
    for (int f = t; f < nb * cpr; f += 256) {
        const int bi = (unsigned)f / (unsigned)cpr;
        const int i = s_busy[bi], col = (f - bi * cpr) * VEC;
        const int e1 = s_ptr[i + 1];
        float acc[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) acc[k] = 0.f;
        for (int e = s_ptr[i]; e < e1; e = e1 - e > 4 ? e + 4 : e1) {
            uint4 v[4];
            bool use[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                use[q] = q < e1 - e;
                if (!kKeys) {
                    if (use[q]) v[q] = ld_hint(P + (long long)(e + q) * Cp + col, let_go);
                } else if (use[q]) {
                    const int key = __ldg(taps + e + q);
                    use[q] = key >= 0 && key < capL;
                    if (use[q]) v[q] = ld_hint(P + (long long)key * Cp + col, let_go);
                    else report(status, kErrIndex);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (kKeys ? use[q] : q < e1 - e) {
                    const T* p = reinterpret_cast<const T*>(&v[q]);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) acc[k] += to_f(p[k]);
                }
        }
        store(r0 + i, col, acc);
    }
}

template <typename Kernel>
hc_status allow_smem(const DeviceCtx* ctx, Kernel k, size_t bytes, bool (&done)[64],
                     const char* what) {
    if (done[ctx->device]) return HC_OK;
    hc_status st = check_cuda(
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), what);
    if (st == HC_OK) done[ctx->device] = true;
    return st;
}

template <int BC>
hc_status launch_wgrad_tc(const DeviceCtx* ctx, const WgradArgs& w, cudaStream_t s) {
    static bool done[64] = {};
    hc_status st = allow_smem(ctx, wgrad_tc_kernel<BC>, WgradCfg<BC>::smem_bytes(HC_MAX_SPIRAL),
                              done, "cudaFuncSetAttribute(wgrad_tc_kernel)");
    if (st != HC_OK) return st;
    return launch_pdl(wgrad_tc_kernel<BC>, dim3((unsigned)w.G, (unsigned)(w.c_tiles * w.o_tiles)),
                      dim3(kThreadsTc), WgradCfg<BC>::smem_bytes(w.L), s, "wgrad_tc_kernel", w);
}

template <int BN>
hc_status launch_tap_gemm_tc(const DeviceCtx* ctx, const TapGemmArgs& g, cudaStream_t s) {
    static bool done[64] = {};
    hc_status st = allow_smem(ctx, tap_gemm_tc_kernel<BN>, TapCfg<BN>::kSmem, done,
                              "cudaFuncSetAttribute(tap_gemm_tc_kernel)");
    if (st != HC_OK) return st;
    CUtensorMap tw;
    st = encode_map_2d(&tw, g.W, (long long)g.L * g.C_in, g.C_out, 64, BN);
    if (st != HC_OK) return st;
    return launch_pdl(tap_gemm_tc_kernel<BN>, dim3((unsigned)ctx->num_sms), dim3(kTapThreads),
                      TapCfg<BN>::kSmem, s, "tap_gemm_tc_kernel", g, tw);
}

// dx with few input channels: the product over all (row, slot) pairs, absent ones
// too, as one linear layer dz W^T (rows of dz and slots of W padded to whole
// chunks), whose rows seg_sum reads by key. A tile of the tap product has 64
// channels of one slot, mostly padding here, and reads a row of dz for every tap
// of it. 41.9k rows (mask full) or 4.9k (12%), 9 slots, dx alone, tap product and
// this: bf16 16 -> 64 46 and 32 us, 14.6 and 12.4; 32 -> 64 46.7 and 35, 15.0 and
// 13.0 (64 -> 64: 53 and 58); fp32 3 -> 64 97 and 35, 16.9 and 13.8; 8 -> 64 98
// and 47, 17.7 and 16.2 (16 -> 64: 100 and 75, but 17.7 and 22.4).
bool dx_by_pairs(const BwdArgs& b) {
    return b.C_in <= (b.dt == HC_BF16 ? 32 : 8);
}

template <typename T>
hc_status launch_act(const BwdArgs& b, const PrepArgs& prep, bool wide, T* dz, int pitch,
                     float* bpart, unsigned* status, cudaStream_t s) {
    const dim3 grid((unsigned)(prep.act_blocks + prep.unit_blocks + prep.hist_blocks + prep.w_blocks));
    return launch_pdl(wide ? act_bwd_vec_kernel<T> : act_bwd_kernel<T>, grid, dim3(256), 0, s,
                      "act_bwd_kernel", (const T*)b.y, (const T*)b.dy, b.count,
                      (long long)b.capacity, b.C_out, b.act, dz, pitch, bpart, prep, status);
}

}  // namespace

hc_status launch_rulebook_transpose(const DeviceCtx* ctx, const int32_t* rb, const int32_t* count,
                                    int capacity, int L, int x_rows, int32_t* ptr, int32_t* taps,
                                    cudaStream_t s) {
    const int ntiles = (x_rows + kScanTile - 1) / kScanTile;
    // workspace: per-row counts, tile sums, each entry's place in its row
    const size_t cnt_n = ((size_t)x_rows + 63) / 64 * 64, sum_n = ((size_t)ntiles + 63) / 64 * 64;
    int32_t* cnt = (int32_t*)stream_workspace(
        s, sizeof(int32_t) * (cnt_n + sum_n + (size_t)capacity * L));
    if (!cnt) return HC_ERR_CUDA;
    int32_t* tsum = cnt + cnt_n;
    int32_t* place = tsum + sum_n;
    long long zblocks = ((long long)x_rows + 1023) / 1024;
    if (zblocks > 8ll * ctx->num_sms) zblocks = 8ll * ctx->num_sms;
    hc_status st = launch_pdl(rb_zero_kernel, dim3((unsigned)zblocks), dim3(256), 0, s,
                              "rb_zero_kernel", cnt, x_rows);
    if (st != HC_OK) return st;
    // about eight blocks per SM over all slots
    long long blocks = ((long long)capacity + 255) / 256;
    const long long cap = (8ll * ctx->num_sms + L - 1) / L;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const dim3 grid((unsigned)blocks, (unsigned)L);
    st = launch_pdl(rb_count_kernel, grid, dim3(256), 0, s, "rb_count_kernel", rb, count,
                    (long long)capacity, x_rows, cnt, place, ctx->status);
    if (st != HC_OK) return st;
    st = launch_pdl(scan_tiles_kernel, dim3((unsigned)ntiles), dim3(kScanThreads), 0, s,
                    "scan_tiles_kernel", (const int32_t*)cnt, x_rows, tsum);
    if (st != HC_OK) return st;
    st = launch_pdl(scan_apply_kernel, dim3((unsigned)ntiles), dim3(kScanThreads), 0, s,
                    "scan_apply_kernel", (const int32_t*)cnt, x_rows, (const int32_t*)tsum, ptr);
    if (st != HC_OK) return st;
    st = launch_pdl(rb_fill_kernel, grid, dim3(256), 0, s, "rb_fill_kernel", rb, count,
                    (long long)capacity, L, x_rows, (const int32_t*)ptr, (const int32_t*)place, taps);
    if (st != HC_OK) return st;
    const int per = sort_rows(L);
    return launch_pdl(rb_sort_kernel, dim3((unsigned)(((long long)x_rows + per - 1) / per)),
                      dim3(kSortRows), 0, s, "rb_sort_kernel", (const int32_t*)ptr, x_rows, per, taps);
}

hc_status launch_conv_bwd(const DeviceCtx* ctx, const BwdArgs& b, cudaStream_t s) {
    const bool bf = b.dt == HC_BF16;
    const int eb = bf ? 2 : 4, vec = 16 / eb;
    const long long capL = (long long)b.capacity * b.L;
    // dz: 16-byte chunks when a row is a whole number of them dividing 256
    const int act_cpr = b.C_out / vec;
    const bool act_wide = b.C_out % vec == 0 && 256 % act_cpr == 0 &&
                          ((uintptr_t)b.y | (uintptr_t)b.dy) % 16 == 0;
    const long long act_rows = act_wide ? kActVecItems / act_cpr : kActRowsPerBlock;
    long long act_blocks = ((long long)b.capacity + act_rows - 1) / act_rows;
    const long long act_cap = (act_wide ? 4ll : 8ll) * ctx->num_sms;
    if (act_blocks > act_cap) act_blocks = act_cap;
    if (act_blocks < 1) act_blocks = 1;

    // wgrad: tensor cores for bf16 rows of whole 16-byte chunks; one CTA per
    // SM over all tiles (two on CUDA cores)
    const bool w_tc = bf && b.C_in % 8 == 0 && b.C_out % 8 == 0 && (uintptr_t)b.x % 16 == 0;
    const int BC = w_tc ? (b.C_in > 64 ? 128 : 64) : (b.C_in > 16 ? 64 : 16);
    const int c_tiles = (b.C_in + BC - 1) / BC, o_tiles = (b.C_out + kTile - 1) / kTile;
    int G = (w_tc ? 1 : 2) * ctx->num_sms / (c_tiles * o_tiles);
    if (G < 1) G = 1;
    // dgrad: P's rows padded to whole 16-byte chunks, and dz's and W's where
    // the product needs it (bf16 off the tensor cores' alignment ran on CUDA cores
    // otherwise: 64 -> 42, 41.9k rows, dx 130 us against 61)
    const int Cp = (b.C_in + vec - 1) / vec * vec;
    const bool pairs = b.dx && dx_by_pairs(b);
    const bool by_taps = b.dx && !pairs;
    const bool pad = by_taps && bf && (b.C_out % 8 != 0 || (uintptr_t)b.W % 16 != 0);
    const int Cz = pairs || pad ? (b.C_out + vec - 1) / vec * vec : b.C_out;  // columns of dz
    const size_t w_elems = pairs ? (size_t)b.L * Cp * Cz : pad ? (size_t)b.L * b.C_in * Cz : 0;

    const int slot_blocks = 2 * ctx->num_sms;

    // workspace
    size_t total = 0;
    auto take = [&](bool wanted, size_t bytes) {
        const size_t at = total;
        if (wanted) total += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t dz_at = take(true, (size_t)b.capacity * Cz * eb);
    const size_t bp_at = take(true, sizeof(float) * (size_t)act_blocks * b.C_out);
    const size_t part_at = take(b.dW, sizeof(float) * (size_t)c_tiles * o_tiles * (G + b.L) * BC * kTile);
    const size_t unit_at = take(b.dW, sizeof(int32_t) * (size_t)b.L * kUnits);
    const size_t pos_at = take(b.dW, sizeof(int32_t) * (size_t)(b.L + 2));
    const size_t p_at = take(b.dx, (size_t)capL * Cp * eb);
    // wgrad is done with its lists before P (at least 16 bytes an entry) is written
    const size_t ul_at = b.dx ? p_at : take(b.dW, sizeof(int2) * (size_t)capL);
    const size_t w_at = take(w_elems > 0, w_elems * eb);
    const size_t ln_at = take(by_taps, sizeof(int32_t) * (size_t)capL);
    const size_t le_at = take(by_taps, sizeof(int32_t) * (size_t)capL);
    const size_t hist_at = take(by_taps, sizeof(int32_t) * (size_t)slot_blocks * b.L);
    const size_t off_at = take(by_taps, sizeof(int32_t) * (size_t)(b.L + 1));
    uint8_t* ws = (uint8_t*)stream_workspace(s, total);
    if (!ws) return HC_ERR_CUDA;
    void* dz = ws + dz_at;
    float* bpart = (float*)(ws + bp_at);

    PrepArgs prep{};
    prep.act_blocks = (int)act_blocks;
    prep.unit_blocks = b.dW ? (b.L * kUnits + 7) / 8 : 0;
    prep.hist_blocks = by_taps ? slot_blocks : 0;
    prep.rb = b.rulebook;
    prep.L = b.L;
    prep.x_rows = b.x_rows;
    prep.unit_cnt = (int32_t*)(ws + unit_at);
    prep.unit_list = (int2*)(ws + ul_at);
    prep.status = ctx->status;
    prep.row_ptr = b.row_ptr;
    prep.taps = b.taps;
    prep.hist = (int32_t*)(ws + hist_at);
    prep.w_blocks = pairs ? ((b.L * Cp + 31) / 32) * ((Cz + 31) / 32) : (int)((w_elems + 1023) / 1024);
    prep.W = b.W;
    prep.w_out = ws + w_at;
    prep.C_in = b.C_in;
    prep.Cp = pairs ? Cp : 0;
    prep.Cz = Cz;
    hc_status st = bf ? launch_act<__nv_bfloat16>(b, prep, act_wide, (__nv_bfloat16*)dz, Cz, bpart,
                                                  ctx->status, s)
                      : launch_act<float>(b, prep, act_wide, (float*)dz, Cz, bpart, ctx->status, s);
    if (st != HC_OK) return st;

    if (b.dW) {
        WgradArgs w{};
        w.x = b.x;
        w.count = b.count;
        w.dz = dz;
        w.capacity = b.capacity;
        w.L = b.L;
        w.C_in = b.C_in;
        w.C_out = b.C_out;
        w.z_pitch = Cz;
        w.c_tiles = c_tiles;
        w.o_tiles = o_tiles;
        w.G = G;
        w.unit_cnt = prep.unit_cnt;
        w.unit_list = prep.unit_list;
        w.slot_pos = (int32_t*)(ws + pos_at);
        w.part = (float*)(ws + part_at);
        w.status = ctx->status;
        const dim3 grid((unsigned)G, (unsigned)(c_tiles * o_tiles));
        const size_t pre = sizeof(int) * ((size_t)b.L * kUnits + 1);
        if (w_tc)
            st = BC == 64 ? launch_wgrad_tc<64>(ctx, w, s) : launch_wgrad_tc<128>(ctx, w, s);
        else
            st = launch_pdl(bf ? (BC == 16 ? wgrad_simt_kernel<__nv_bfloat16, 16>
                                           : wgrad_simt_kernel<__nv_bfloat16, 64>)
                               : (BC == 16 ? wgrad_simt_kernel<float, 16> : wgrad_simt_kernel<float, 64>),
                            grid, dim3(256), pre, s, "wgrad_simt_kernel", w);
        if (st != HC_OK) return st;
    }
    SlotArgs sl{};
    if (by_taps) {
        sl.row_ptr = b.row_ptr;
        sl.taps = b.taps;
        sl.x_rows = b.x_rows;
        sl.L = b.L;
        sl.blocks = slot_blocks;
        sl.capL = capL;
        sl.hist = prep.hist;
        sl.slot_off = (int32_t*)(ws + off_at);
        sl.list_n = (int32_t*)(ws + ln_at);
        sl.list_e = (int32_t*)(ws + le_at);
        sl.status = ctx->status;
    }
    ReduceArgs r{};
    r.L = b.L;
    r.C_in = b.C_in;
    r.C_out = b.C_out;
    r.BC = BC;
    r.c_tiles = c_tiles;
    r.G = G;
    if (b.dW) {
        long long blocks = ((long long)b.L * b.C_in * b.C_out + 63) / 64;
        if (blocks > 8ll * ctx->num_sms) blocks = 8ll * ctx->num_sms;
        r.dw_blocks = (int)blocks;
    }
    r.part = (const float*)(ws + part_at);
    r.slot_pos = (const int32_t*)(ws + pos_at);
    r.dW = b.dW;
    r.bpart = bpart;
    r.act_blocks = (int)act_blocks;
    r.dbias = b.dbias;
    const int collect = sl.blocks + r.dw_blocks + (b.dbias ? (b.C_out + 7) / 8 : 0);
    if (collect > 0) {
        st = launch_pdl(bwd_collect_kernel, dim3((unsigned)collect), dim3(256), 0, s,
                        "bwd_collect_kernel", r, sl);
        if (st != HC_OK) return st;
    }

    if (!b.dx) return st;
    void* const P = ws + p_at;
    if (pairs) {
        ConvArgs c{};  // P [rows][L * Cp] = dz W^T
        c.x = dz;
        c.count = b.count;
        c.W = prep.w_out;
        c.y = P;
        c.capacity = c.x_rows = b.capacity;
        c.B = 1;
        c.V = b.capacity;
        c.L = 1;
        c.C_in = c.K = Cz;
        c.C_out = b.L * Cp;
        c.mode = kLinear;
        c.act = HC_ACT_NONE;
        st = dispatch_conv(ctx, c, b.dt, s);  // Cz whole chunks: needs no workspace
    } else {
        TapGemmArgs g{};
        g.dz = dz;
        g.W = pad ? prep.w_out : b.W;
        g.slot_off = sl.slot_off;
        g.list_n = sl.list_n;
        g.list_e = sl.list_e;
        g.P = P;
        g.L = b.L;
        g.C_in = b.C_in;
        g.C_out = Cz;
        g.Cp = Cp;
        g.status = ctx->status;
        if (bf) {
            g.c_tiles = (b.C_in + (b.C_in <= 64 ? 63 : 127)) / (b.C_in <= 64 ? 64 : 128);
            st = b.C_in <= 64 ? launch_tap_gemm_tc<64>(ctx, g, s) : launch_tap_gemm_tc<128>(ctx, g, s);
        } else {
            g.c_tiles = (b.C_in + kTgBN - 1) / kTgBN;
            st = launch_pdl(tap_gemm_simt_kernel, dim3((unsigned)(2 * ctx->num_sms)), dim3(256),
                            0, s, "tap_gemm_simt_kernel", g);
        }
    }
    if (st != HC_OK) return st;
    const int vec_ok = b.C_in % vec == 0 && (uintptr_t)b.dx % 16 == 0;
    const dim3 blocks((unsigned)(((long long)b.x_rows + kSegRows - 1) / kSegRows));
    if (bf)
        return launch_pdl(pairs ? seg_sum_kernel<__nv_bfloat16, true> : seg_sum_kernel<__nv_bfloat16, false>,
                          blocks, dim3(256), 0, s, "seg_sum_kernel", (const __nv_bfloat16*)P, b.row_ptr,
                          b.taps, b.x_rows, b.C_in, Cp, capL, (__nv_bfloat16*)b.dx, vec_ok, ctx->status);
    return launch_pdl(pairs ? seg_sum_kernel<float, true> : seg_sum_kernel<float, false>, blocks, dim3(256),
                      0, s, "seg_sum_kernel", (const float*)P, b.row_ptr, b.taps, b.x_rows, b.C_in, Cp,
                      capL, (float*)b.dx, vec_ok, ctx->status);
}

}  // namespace hc
