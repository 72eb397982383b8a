// Spiral convolution / linear layer on CUDA cores (FFMA, fp32 accumulate) for
// bf16 shapes the tensor-core kernel does not take (output channel counts that
// are not a multiple of 8, misaligned rows), and for fp32 layers of few input
// channels and the fp32 dense layer at some widths; other fp32 layers have a
// kernel of their own (conv_f32.cu). And the narrow linear heads of both types.
//
// Each CTA owns a 64-row x 64-column output tile and walks K = L*C_in in
// chunks of KC (128 when K <= 256, else 64): the A chunk is gathered through the per-tile table of source
// rows (idx() of Eq. 4: -1 when the tap is absent) and the W chunk read
// directly, every load of a chunk issued before any is used (one dependent
// round trip per KC of K rather than per 16: the small layers this kernel
// serves are latency-bound; deeper layers take the smaller chunk, whose
// registers and shared memory let more CTAs share an SM); each thread then
// accumulates a 4x4 block. The
// grid is persistent over row tiles because the row count N' is only known on
// the device.
#include <cuda_bf16.h>

#include "hc_internal.cuh"
#include "tap_table.cuh"

namespace hc {
namespace {

constexpr int kBM = 64;
constexpr int kBN = 64;
constexpr int kThreads = 256;
constexpr int kAPitch = kBM + 4;  // floats per As row (16-byte aligned rows)

// Shared memory of a chunk depth: As [KC][kAPitch] and Bs [KC][kBN] floats.
template <int KC>
constexpr size_t chunk_smem_bytes() {
    return sizeof(float) * (size_t)(KC * kAPitch + KC * kBN);
}

template <typename T>
__device__ __forceinline__ float to_float(T v);
template <>
__device__ __forceinline__ float to_float<float>(float v) {
    return v;
}
template <>
__device__ __forceinline__ float to_float<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}
template <typename T>
__device__ __forceinline__ T from_float(float v);
template <>
__device__ __forceinline__ float from_float<float>(float v) {
    return v;
}
template <>
__device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}

template <typename T, int kKC>
__global__ void __launch_bounds__(kThreads) conv_simt_kernel(const ConvArgs a) {
    constexpr int kAsFloats = kKC * kAPitch;
    constexpr int kBsFloats = kKC * kBN;
    // per thread per chunk: A rows tid/kKC + (256/kKC) i, B k-rows tid/64 + 4i
    constexpr int kAPer = kBM * kKC / kThreads;
    constexpr int kBPer = kKC * kBN / kThreads;
    constexpr int kAStep = kThreads / kKC;
    // dynamic: As [kKC][kAPitch] float, Bs [kKC][kBN] float, src_tab [kBM][L] int
    extern __shared__ __align__(16) float smem_f[];
    float* const As = smem_f;
    float* const Bs = smem_f + kAsFloats;
    int* const src_tab = reinterpret_cast<int*>(smem_f + kAsFloats + kBsFloats);

    const T* __restrict__ x = static_cast<const T*>(a.x);
    const T* __restrict__ W = static_cast<const T*>(a.W);
    T* __restrict__ y = static_cast<T*>(a.y);
    pdl_wait();
    pdl_trigger();
    const long long rows = active_rows(a);
    const long long m_tiles = (rows + kBM - 1) / kBM;
    const int n0 = blockIdx.y * kBN;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int L = a.L, C_in = a.C_in, C_out = a.C_out, K = a.K;

    for (long long mt = blockIdx.x; mt < m_tiles; mt += gridDim.x) {
        const long long m0 = mt * kBM;
        __syncthreads();  // the previous tile is done with src_tab
        fill_tap_table<kBM, kThreads>(a, rows, m0, rows, src_tab, L, 1);
        __syncthreads();

        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

        // this thread's A column of every chunk (k = k0 + ka) and B column o
        const int ka = tid & (kKC - 1), ra = tid / kKC;
        const int ob = tid & (kBN - 1), kbr = tid >> 6;
        for (int k0 = 0; k0 < K; k0 += kKC) {
            const int k = k0 + ka;
            const bool kin = k < K;
            const int l = kin ? k / C_in : 0, c = kin ? k - l * C_in : 0;
            float av_[kAPer], bv_[kBPer];
            // every load of the chunk first ...
#pragma unroll
            for (int i = 0; i < kAPer; ++i) {
                const int r = ra + kAStep * i;
                const int s = kin ? src_tab[r * L + l] : -1;
                av_[i] = s >= 0 ? to_float(x[(long long)s * C_in + c]) : 0.f;
            }
#pragma unroll
            for (int i = 0; i < kBPer; ++i) {
                const int kk = kbr + 4 * i, col = n0 + ob;
                bv_[i] = (k0 + kk < K && col < C_out)
                             ? to_float(W[(long long)(k0 + kk) * C_out + col])
                             : 0.f;
            }
            // ... then the stores to shared memory
#pragma unroll
            for (int i = 0; i < kAPer; ++i) As[ka * kAPitch + ra + kAStep * i] = av_[i];
#pragma unroll
            for (int i = 0; i < kBPer; ++i) Bs[(kbr + 4 * i) * kBN + ob] = bv_[i];
            __syncthreads();
            const int kn = K - k0 < kKC ? K - k0 : kKC;
#pragma unroll 16
            for (int kk = 0; kk < kn; ++kk) {
                const float4 av = *reinterpret_cast<const float4*>(&As[kk * kAPitch + ty * 4]);
                const float4 bv = *reinterpret_cast<const float4*>(&Bs[kk * kBN + tx * 4]);
                const float ar[4] = {av.x, av.y, av.z, av.w};
                const float br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
            }
            __syncthreads();
        }

#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const long long n = m0 + ty * 4 + i;
            if (n >= rows) continue;
            T* dp = nullptr;  // fused scatter destination row, if any
            if (a.out_dense) {
                const int b = __ldg(a.out_coords + 2 * n), v = __ldg(a.out_coords + 2 * n + 1);
                if (b >= 0 && b < a.out_B && v >= 0 && v < a.out_V)
                    dp = static_cast<T*>(a.out_dense) + ((long long)b * a.out_V + v) * C_out;
                else
                    report(a.status, kErrIndex);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int col = n0 + tx * 4 + j;
                if (col >= C_out) continue;
                const float z = acc[i][j] + (a.bias ? __ldg(a.bias + col) : 0.f);
                const T val = from_float<T>(act_apply(z, a.act));
                if (y) y[n * C_out + col] = val;
                if (dp) dp[col] = val;
            }
        }
    }
}

// ---------------------------------------------------------------- narrow linear heads
// y[n] = act(x[n] W + bias) on compact rows for at most kHeadMaxOut output
// channels (the 42- and 1-channel heads, which the tensor-core kernel does not
// take). The 64 x 64 tiles above leave most of their columns idle there, and
// a warp's loads of a K chunk of one row at a time make them latency-bound.
// Here a block stages kHeadRows rows of x and the whole of W (as fp32) in
// shared memory with one round trip of wide loads; thread t then owns row
// t % kHeadRows and every second group of kHeadGroup output channels: its
// row's channels come 16 bytes at a time (the padded pitch keeps eight lanes'
// pieces on distinct banks), W's are the same word for the whole warp. The
// finished rows are one contiguous piece of y and leave through the same
// shared memory in order. Sums run over c = 0, 1, ... in one fp32 chain, then
// the bias, as in the kernel above: the same bits. What bounds it: reading
// x once (25k rows x 64 bf16 channels is 3.2 MB) and the launch.
// Measured on the 64 -> 1 bf16 head over 25k active rows of 168k (cold, ncu):
// 46.4 us on the 64 x 64 tiles, 9.4 us here; the motion encoder (256 frames)
// 124 -> 103 us on the device.
constexpr int kHeadThreads = 256;
constexpr int kHeadRows = 128;
constexpr int kHeadGroup = 4;
constexpr int kHeadMaxOut = 64;
constexpr int kHeadMaxRowBytes = 512;  // of x
constexpr int kHeadMaxWFloats = 64 * 64;

__host__ __device__ constexpr int head_pitch(int row_bytes) {
    return (row_bytes + 15) / 16 * 16 + 16;
}
__host__ __device__ constexpr int head_wpitch(int C_out) {
    return (C_out + kHeadGroup - 1) / kHeadGroup * kHeadGroup;
}
inline size_t head_smem_bytes(int C_in, int C_out, int eb) {
    const size_t xb = (size_t)kHeadRows * head_pitch(C_in * eb);
    const size_t yb = (size_t)kHeadRows * C_out * eb;
    return (xb > yb ? xb : yb) + sizeof(float) * (size_t)C_in * head_wpitch(C_out);
}

// kMaxG: groups a thread owns at most (1 for up to 8 outputs, else 8).
template <typename T, int kMaxG>
__global__ void __launch_bounds__(kHeadThreads) linear_head_kernel(const ConvArgs a, int vec_ok) {
    constexpr int VEC = 16 / (int)sizeof(T);
    extern __shared__ __align__(16) uint8_t head_smem[];
    const int C_in = a.C_in, C_out = a.C_out;
    const int row_bytes = C_in * (int)sizeof(T);
    const int pitch = head_pitch(row_bytes), wp = head_wpitch(C_out);
    float* const sW = reinterpret_cast<float*>(head_smem);  // [C_in][wp], zero-padded
    uint8_t* const sX = head_smem + sizeof(float) * (size_t)C_in * wp;
    T* const sY = reinterpret_cast<T*>(sX);
    const T* __restrict__ x = static_cast<const T*>(a.x);
    const T* __restrict__ W = static_cast<const T*>(a.W);
    T* __restrict__ y = static_cast<T*>(a.y);
    const int t = threadIdx.x, row = t & (kHeadRows - 1), half = t / kHeadRows;
    pdl_wait();
    pdl_trigger();
    // the weights' loads go out with the row count's
#pragma unroll 4
    for (int i = t; i < C_in * wp; i += kHeadThreads) {
        const int c = i / wp, o = i - c * wp;
        sW[i] = o < C_out ? to_float(W[c * C_out + o]) : 0.f;
    }
    const long long rows = active_rows(a);
    for (long long m0 = (long long)blockIdx.x * kHeadRows; m0 < rows;
         m0 += (long long)gridDim.x * kHeadRows) {
        const int nr = rows - m0 < kHeadRows ? (int)(rows - m0) : kHeadRows;
        __syncthreads();  // the previous rows have left through sY
        if (vec_ok) {
            const int cpr = row_bytes / 16;
            const uint4* src = reinterpret_cast<const uint4*>(x + m0 * C_in);
#pragma unroll 4
            for (int i = t; i < nr * cpr; i += kHeadThreads) {
                const int r = i / cpr, q = i - r * cpr;
                *reinterpret_cast<uint4*>(sX + r * pitch + q * 16) = src[i];
            }
        } else {
            const T* src = x + m0 * C_in;
#pragma unroll 4
            for (int i = t; i < nr * C_in; i += kHeadThreads) {
                const int r = i / C_in, c = i - r * C_in;
                *reinterpret_cast<T*>(sX + r * pitch + c * (int)sizeof(T)) = src[i];
            }
        }
        __syncthreads();
        // groups half, half + 2, ... of kHeadGroup outputs; the results are
        // kept until every thread has read its row (sY shares the memory)
        float acc[kMaxG][kHeadGroup];
        const int groups = wp / kHeadGroup;
#pragma unroll
        for (int g = 0; g < kMaxG; ++g)
#pragma unroll
            for (int j = 0; j < kHeadGroup; ++j) acc[g][j] = 0.f;
        const uint8_t* xr = sX + row * pitch;
        if (row < nr)
            for (int c0 = 0; c0 < C_in; c0 += VEC) {
                const uint4 raw = *reinterpret_cast<const uint4*>(xr + c0 * (int)sizeof(T));
                const T* v = reinterpret_cast<const T*>(&raw);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    if (c0 + k >= C_in) break;
                    const float xv = to_float(v[k]);
                    const float* wr = sW + (c0 + k) * wp + half * kHeadGroup;
#pragma unroll
                    for (int g = 0; g < kMaxG; ++g) {
                        if (half + 2 * g >= groups) break;
                        const float4 w = *reinterpret_cast<const float4*>(wr + 2 * g * kHeadGroup);
                        acc[g][0] = fmaf(xv, w.x, acc[g][0]);
                        acc[g][1] = fmaf(xv, w.y, acc[g][1]);
                        acc[g][2] = fmaf(xv, w.z, acc[g][2]);
                        acc[g][3] = fmaf(xv, w.w, acc[g][3]);
                    }
                }
            }
        __syncthreads();
        if (row < nr)
#pragma unroll
            for (int g = 0; g < kMaxG; ++g)
#pragma unroll
                for (int j = 0; j < kHeadGroup; ++j) {
                    const int o = (half + 2 * g) * kHeadGroup + j;
                    if (o < C_out) {
                        const float z = acc[g][j] + (a.bias ? __ldg(a.bias + o) : 0.f);
                        sY[row * C_out + o] = from_float<T>(act_apply(z, a.act));
                    }
                }
        __syncthreads();
        T* dst = y + m0 * C_out;
        for (int i = t; i < nr * C_out; i += kHeadThreads) dst[i] = sY[i];
    }
}

template <typename T>
hc_status launch_head_typed(const DeviceCtx* ctx, const ConvArgs& a, cudaStream_t s) {
    const int row_bytes = a.C_in * (int)sizeof(T);
    const int vec_ok = row_bytes % 16 == 0 && (uintptr_t)a.x % 16 == 0;
    static bool attr_set[64] = {};
    if (!attr_set[ctx->device]) {
        const size_t most = (size_t)kHeadRows * head_pitch(kHeadMaxRowBytes) +
                            sizeof(float) * (size_t)kHeadMaxWFloats;
        for (auto kernel : {linear_head_kernel<T, 1>, linear_head_kernel<T, 8>}) {
            hc_status st = check_cuda(
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most),
                "cudaFuncSetAttribute(linear_head_kernel)");
            if (st != HC_OK) return st;
        }
        attr_set[ctx->device] = true;
    }
    long long grid = (a.capacity + kHeadRows - 1) / kHeadRows;
    const long long cap = 4ll * ctx->num_sms;
    if (grid > cap) grid = cap;
    return launch_pdl(a.C_out <= 2 * kHeadGroup ? linear_head_kernel<T, 1> : linear_head_kernel<T, 8>,
                      dim3((unsigned)grid), dim3(kHeadThreads),
                      head_smem_bytes(a.C_in, a.C_out, (int)sizeof(T)), s, "linear_head_kernel", a,
                      vec_ok);
}

}  // namespace

// Linear layers on compact rows with few outputs, whose row of x and weights
// fit in shared memory.
bool linear_head_supported(const ConvArgs& a, hc_dtype dt) {
    // fp32 with more than 16 outputs is faster on the fp32 conv's taller tiles
    // (64 -> 64 over 4k rows: 12.3 us there, 24.7 us here)
    const int eb = dt == HC_F32 ? 4 : 2, most = dt == HC_F32 ? 16 : kHeadMaxOut;
    return a.mode == kLinear && a.out_dense == nullptr && a.C_out <= most &&
           (long long)a.C_in * eb <= kHeadMaxRowBytes &&
           a.C_in * head_wpitch(a.C_out) <= kHeadMaxWFloats;
}

// Of those, the ones the 64 x 64 tiles serve better. A thread has a row's half
// of the outputs, C_in channels of some groups of four one after the other; as
// long as every SM has at most one 64-row tile, those tiles' 256 threads a tile
// share that chain out further (655 rows, bf16 64 -> 60: 13.7 us there, 19.7
// here; 128 -> 20: 15.4 and 19.5; 64 -> 28: 13.5 and 13.3; fp32 128 -> 16: 10.5
// and 16.5; 64 -> 16: 8.7 and 9.8; 16 -> 16: 7.8 and 5.0), bf16 heads of more
// than 48 outputs up to two tiles an SM (19k rows, 64 -> 60: 16.4 and 20.1; 64
// -> 42: 16.4 and 17.0; 21k rows 27.7 and 21.9).
bool linear_head_on_tiles(const DeviceCtx* ctx, const ConvArgs& a, hc_dtype dt) {
    const int groups = (head_wpitch(a.C_out) / kHeadGroup + 1) / 2;  // of a thread
    const int chain = a.C_in * groups;
    const bool f32 = dt == HC_F32;
    const long long tiles = !f32 && a.C_out > 48 ? 2 : 1;
    return (f32 ? chain >= 128 : chain > 256) && a.capacity <= 64 * tiles * ctx->num_sms;
}

hc_status launch_linear_head(const DeviceCtx* ctx, const ConvArgs& a, hc_dtype dt, cudaStream_t s) {
    return dt == HC_F32 ? launch_head_typed<float>(ctx, a, s)
                        : launch_head_typed<__nv_bfloat16>(ctx, a, s);
}

template <typename T>
static hc_status launch_simt_typed(const DeviceCtx* ctx, const ConvArgs& a, cudaStream_t s) {
    long long cap_tiles = (a.capacity + kBM - 1) / kBM;
    long long gx = cap_tiles < (long long)ctx->num_sms * 8 ? cap_tiles : (long long)ctx->num_sms * 8;
    if (gx < 1) gx = 1;
    dim3 grid((unsigned)gx, (unsigned)((a.C_out + kBN - 1) / kBN));
    const size_t tab = sizeof(int) * (size_t)kBM * a.L;
    static bool attr_set[64] = {};
    if (!attr_set[ctx->device]) {
        hc_status st = HC_OK;
        auto allow = [&](auto kernel, size_t bytes) {
            if (st == HC_OK)
                st = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)bytes),
                                "cudaFuncSetAttribute(conv_simt_kernel)");
        };
        const size_t tab_max = sizeof(int) * (size_t)kBM * HC_MAX_SPIRAL;
        allow(conv_simt_kernel<T, 128>, chunk_smem_bytes<128>() + tab_max);
        allow(conv_simt_kernel<T, 64>, chunk_smem_bytes<64>() + tab_max);
        if (st != HC_OK) return st;
        attr_set[ctx->device] = true;
    }
    if (a.K <= 256)
        return launch_pdl(conv_simt_kernel<T, 128>, grid, dim3(kThreads),
                          chunk_smem_bytes<128>() + tab, s, "conv_simt_kernel", a);
    return launch_pdl(conv_simt_kernel<T, 64>, grid, dim3(kThreads), chunk_smem_bytes<64>() + tab, s,
                      "conv_simt_kernel", a);
}

hc_status launch_conv_simt(const DeviceCtx* ctx, const ConvArgs& a, hc_dtype dt, cudaStream_t s) {
    return dt == HC_F32 ? launch_simt_typed<float>(ctx, a, s)
                        : launch_simt_typed<__nv_bfloat16>(ctx, a, s);
}

}  // namespace hc
