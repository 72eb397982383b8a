// Spiral convolution / linear layer in fp32 on CUDA cores: genuine IEEE fp32
// multiply-adds (no TF32), one chain per output over the present taps in slot
// and channel order, then bias and activation (Eqs. 4-6, 10).
//
// Most taps of a sparse mask are absent (three quarters at 15% density), so a
// block multiplies the present ones only: per slot it lists the rows of its
// tile whose tap is present, and multiplies those rows by the slot's weights,
// adding onto the tile's sums, which stay in shared memory (the chain of an
// output passes through it unrounded). A step is KC channels of one slot: the
// listed rows' channels, gathered, and the [KC][BN] weights, through a ring of
// S stages filled by cp.async (16 bytes where channel counts and pointers
// allow, else 4), one block barrier a step. A step's units of 4 UR listed rows
// x 8 UC outputs are dealt to the warps; a lane has UR rows x UC outputs and
// reads UR + UC words a channel for UR UC multiply-adds. What bounds it is
// those reads: shared memory returns 128 bytes a clock, one word to each lane
// of a warp, against four warps' multiply-adds, so 2 x 4 a lane runs at a third
// of the multiply-add rate, 4 x 4 at half, 8 x 4 at two thirds; the
// shape with the fewest clocks for the slot's row count is taken (unit_cost),
// and sixteen warps hide the reads' latency (8 x 8 a lane with eight warps, in
// balance on paper, was slower at every density). Hence tiles as tall as shared memory allows
// (up to 192 rows), so that slots list enough rows for tall units (at 15%
// density 64-row tiles took 77 us, 192-row ones 56); the row count is
// known on the device only, and a tile takes as many rows as make the blocks'
// shares even.
//
// 25k rows, 9 slots, 64 -> 128, 24% of the taps present: 133 us on the 64 x 64
// tiles of conv_simt.cu, 56 us here (cold); all taps present (41.9k rows, 64 ->
// 64): 121 us there, 114 us here; 74 rows, 16 -> 64: 18.7 us there, 11 us here.
#include "hc_internal.cuh"
#include "tap_table.cuh"

namespace hc {
namespace {

constexpr int kMinRows = 16;  // fewest rows of a tile

// BM: most rows of a tile; BN: outputs of a tile.
template <int WARPS_, int BM_, int BN_, int KC_, int S_>
struct Cfg32 {
    static constexpr int WARPS = WARPS_, THREADS = 32 * WARPS;
    static constexpr int BM = BM_, BN = BN_, KC = KC_, S = S_;
    static constexpr int kXPitch = KC + 4;  // rows of a unit on distinct banks
    static constexpr int kStageFloats = KC * BN + BM * kXPitch;
    // ring | sums [BM][BN] | sources [L][BM] int | rows [L][BM] byte
    static size_t smem_bytes(int L) {
        return sizeof(float) * ((size_t)S * kStageFloats + (size_t)BM * BN) + 5 * (size_t)L * BM;
    }
};

// Unit (rg, cg): listed rows rg * 4 UR .. of the m of the slot (their tile
// rows in row_id, their channels at sx), outputs cg * 8 UC .. of the weights
// sw; a lane has rows (lane / 8) + 4 q and outputs (lane % 8) * 4 + 32 p ..
template <int UR, int UC, class C>
__device__ __forceinline__ void unit(int rg, int cg, int m, int kn, const uint8_t* row_id,
                                     const float* sx, const float* sw, float* sums) {
    constexpr int P = UC / 4;
    const int lane = threadIdx.x & 31;
    const int r0 = rg * 4 * UR + (lane >> 3), col = cg * 8 * UC + (lane & 7) * 4;
    float acc[UR][UC];
    int at[UR];  // the rows' sums, -1: no row
#pragma unroll
    for (int q = 0; q < UR; ++q) {
        const int i = r0 + 4 * q;
        at[q] = i < m ? row_id[i] * C::BN + col : -1;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float4 v = i < m ? *reinterpret_cast<const float4*>(sums + at[q] + 32 * p)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
            acc[q][4 * p] = v.x, acc[q][4 * p + 1] = v.y, acc[q][4 * p + 2] = v.z,
                     acc[q][4 * p + 3] = v.w;
        }
    }
    const float* xr = sx + r0 * C::kXPitch;
    const float* wr = sw + col;
#pragma unroll 2
    for (int k = 0; k < kn; k += 4) {
        float4 xv[UR];
#pragma unroll
        for (int q = 0; q < UR; ++q) xv[q] = *reinterpret_cast<const float4*>(xr + q * 4 * C::kXPitch + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float4 wv[P];
#pragma unroll
            for (int p = 0; p < P; ++p)
                wv[p] = *reinterpret_cast<const float4*>(wr + (k + j) * C::BN + 32 * p);
#pragma unroll
            for (int q = 0; q < UR; ++q) {
                const float xq = j == 0 ? xv[q].x : j == 1 ? xv[q].y : j == 2 ? xv[q].z : xv[q].w;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    acc[q][4 * p] = fmaf(xq, wv[p].x, acc[q][4 * p]);
                    acc[q][4 * p + 1] = fmaf(xq, wv[p].y, acc[q][4 * p + 1]);
                    acc[q][4 * p + 2] = fmaf(xq, wv[p].z, acc[q][4 * p + 2]);
                    acc[q][4 * p + 3] = fmaf(xq, wv[p].w, acc[q][4 * p + 3]);
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < UR; ++q)
        if (at[q] >= 0)
#pragma unroll
            for (int p = 0; p < P; ++p)
                *reinterpret_cast<float4*>(sums + at[q] + 32 * p) = make_float4(
                    acc[q][4 * p], acc[q][4 * p + 1], acc[q][4 * p + 2], acc[q][4 * p + 3]);
}

// Clocks a channel of m listed rows takes in units of UR x UC a lane: the
// larger of the words read (one clock each and unit) and the busiest of the
// four schedulers' multiply-adds.
template <int UR, int UC, int BN>
__device__ __forceinline__ int unit_cost(int m) {
    const int units = (m + 4 * UR - 1) / (4 * UR) * (BN / (8 * UC));
    const int words = units * (UR + UC);
    const int fma = (units + 3) / 4 * (UR * UC);
    return words > fma ? words : fma;
}

template <int UR, int UC, class C>
__device__ __forceinline__ void units(int m, int kn, const uint8_t* row_id, const float* sx,
                                      const float* sw, float* sums) {
    constexpr int CG = C::BN / (8 * UC);
    const int n = (m + 4 * UR - 1) / (4 * UR) * CG;
    for (int u = threadIdx.x >> 5; u < n; u += C::WARPS)
        unit<UR, UC, C>(u / CG, u % CG, m, kn, row_id, sx, sw, sums);
}

template <class C>
__global__ void __launch_bounds__(C::THREADS, 1)
    conv_f32_kernel(const ConvArgs a, const int x_vec, const int w_vec) {
    constexpr int kThreads = C::THREADS, kWarps = C::WARPS;
    constexpr int KC = C::KC, S = C::S, kBM = C::BM, BN = C::BN, XP = C::kXPitch;
    extern __shared__ __align__(16) float ring[];
    __shared__ int s_cnt[HC_MAX_SPIRAL];
    float* const sums = ring + S * C::kStageFloats;
    int* const s_src = reinterpret_cast<int*>(sums + kBM * BN);             // [L][kBM]
    uint8_t* const s_row = reinterpret_cast<uint8_t*>(s_src + a.L * kBM);  // [L][kBM]
    const float* __restrict__ x = static_cast<const float*>(a.x);
    const float* __restrict__ W = static_cast<const float*>(a.W);
    float* __restrict__ y = static_cast<float*>(a.y);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int C_in = a.C_in, C_out = a.C_out;
    pdl_wait();
    pdl_trigger();
    const long long rows = active_rows(a);
    const int n_tiles = (C_out + BN - 1) / BN;
    const bool out_vec = C_out % 4 == 0 && ((uintptr_t)y | (uintptr_t)a.out_dense) % 16 == 0;
    const int per_slot = (C_in + KC - 1) / KC, steps = a.L * per_slot;
    // rows of a tile: the fewest rounds over the blocks, shared evenly
    const long long rounds = ((rows + kBM - 1) / kBM * n_tiles + gridDim.x - 1) / gridDim.x;
    long long tr = rounds > 0 ? (rows * n_tiles + rounds * gridDim.x - 1) / (rounds * gridDim.x) : kBM;
    tr = tr < kMinRows ? kMinRows : (tr + 7) / 8 * 8;
    if (tr > kBM) tr = kBM;
    const long long items = (rows + tr - 1) / tr * n_tiles;

    for (long long w = blockIdx.x; w < items; w += gridDim.x) {
        const long long mt = w / n_tiles;
        const int n0 = (int)(w - mt * n_tiles) * BN;
        const long long m0 = mt * tr;
        const long long end = m0 + tr < rows ? m0 + tr : rows;
        __syncthreads();  // the previous item is done with the tables, sums and ring
        fill_tap_table<kBM, kThreads>(a, rows, m0, end, s_src, 1, kBM);
        for (int i = t; i < kBM * BN / 4; i += kThreads)
            reinterpret_cast<float4*>(sums)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        // each slot's present rows to the front, in order
        for (int l = warp; l < a.L; l += kWarps) {
            int src[kBM / 32], at = 0;
#pragma unroll
            for (int q = 0; q < kBM / 32; ++q) src[q] = s_src[l * kBM + 32 * q + lane];
            __syncwarp();
#pragma unroll
            for (int q = 0; q < kBM / 32; ++q) {
                const unsigned m = __ballot_sync(0xffffffffu, src[q] >= 0);
                if (src[q] >= 0) {
                    const int p = l * kBM + at + __popc(m & ((1u << lane) - 1u));
                    s_src[p] = src[q];
                    s_row[p] = (uint8_t)(32 * q + lane);
                }
                at += __popc(m);
            }
            if (lane == 0) s_cnt[l] = at;
        }
        __syncthreads();

        int ls = 0, lc = 0;  // slot and first channel of the step loaded next
        auto load = [&](int buf) {
            float* const sw = ring + buf * C::kStageFloats;
            float* const sx = sw + KC * BN;
            const float* wsrc = W + (long long)(ls * C_in + lc) * C_out + n0;
            const int* src = s_src + ls * kBM;
            const int m = s_cnt[ls];
            // channels past C_in are zeros up to the next multiple of four;
            // outputs past C_out are left as they are (never stored)
            const int kn = C_in - lc < KC ? (C_in - lc + 3) / 4 * 4 : KC;
            if (m > 0) {
                if (w_vec) {
#pragma unroll
                    for (int i = t; i < KC * BN / 4; i += kThreads) {
                        const int k = i / (BN / 4), c = (i % (BN / 4)) * 4;
                        const bool in = lc + k < C_in;
                        if (k < kn && n0 + c < C_out)
                            cp_async_16(smem_u32(sw + k * BN + c),
                                        in ? wsrc + (long long)k * C_out + c : W, in);
                    }
                } else {
                    for (int i = t; i < KC * BN; i += kThreads) {
                        const int k = i / BN, c = i % BN;
                        const bool in = lc + k < C_in;
                        if (k < kn && n0 + c < C_out)
                            cp_async_4(smem_u32(sw + k * BN + c),
                                       in ? wsrc + (long long)k * C_out + c : W, in);
                    }
                }
                if (x_vec) {
                    for (int i = t; i < m * (KC / 4); i += kThreads) {
                        const int r = i / (KC / 4), c = (i % (KC / 4)) * 4;
                        if (c < kn)
                            cp_async_16(smem_u32(sx + r * XP + c), x + (long long)src[r] * C_in + lc + c,
                                        true);
                    }
                } else {
                    for (int i = t; i < m * KC; i += kThreads) {
                        const int r = i / KC, c = i % KC;
                        const bool in = lc + c < C_in;
                        if (c < kn)
                            cp_async_4(smem_u32(sx + r * XP + c),
                                       x + (in ? (long long)src[r] * C_in + lc + c : 0), in);
                    }
                }
            }
            lc += KC;
            if (lc >= C_in) {
                lc = 0;
                ++ls;
            }
        };

#pragma unroll
        for (int s = 0; s < S - 1; ++s) {
            if (s < steps) load(s);
            cp_async_commit();
        }
        int slot = 0, c0 = 0, buf = 0, shape = 0;
        for (int s = 0; s < steps; ++s) {
            cp_async_wait_group<S - 2>();
            __syncthreads();  // stage s is complete; step s - 1 is done
            if (s + S - 1 < steps) load(buf == 0 ? S - 1 : buf - 1);
            cp_async_commit();
            const int m = s_cnt[slot];
            const int kn = C_in - c0 < KC ? C_in - c0 : KC;
            const float* sw = ring + buf * C::kStageFloats;
            const float* sx = sw + KC * BN;
            const uint8_t* row_id = s_row + slot * kBM;
            if (c0 == 0) {  // the slot's unit shape
                int best = unit_cost<2, 4, BN>(m);
                shape = 0;
                const int c1 = unit_cost<4, 4, BN>(m), c2 = unit_cost<8, 4, BN>(m);
                if (c1 <= best) best = c1, shape = 1;
                if (c2 <= best) best = c2, shape = 2;
            }
            if (shape == 2) units<8, 4, C>(m, kn, row_id, sx, sw, sums);
            else if (shape == 1) units<4, 4, C>(m, kn, row_id, sx, sw, sums);
            else units<2, 4, C>(m, kn, row_id, sx, sw, sums);
            c0 += KC;
            if (c0 >= C_in) {
                c0 = 0;
                ++slot;
            }
            if (++buf == S) buf = 0;
        }
        __syncthreads();

        // bias, activation and stores: BN / 4 threads per row
        const int col = (t % (BN / 4)) * 4;
        float bias[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            bias[c] = a.bias && n0 + col + c < C_out ? __ldg(a.bias + n0 + col + c) : 0.f;
#pragma unroll 4
        for (long long n = m0 + t / (BN / 4); n < end; n += kThreads / (BN / 4)) {
            float* dp = nullptr;  // fused scatter destination row, if any
            if (a.out_dense) {
                const int b = __ldg(a.out_coords + 2 * n), v = __ldg(a.out_coords + 2 * n + 1);
                if (b >= 0 && b < a.out_B && v >= 0 && v < a.out_V)
                    dp = static_cast<float*>(a.out_dense) + ((long long)b * a.out_V + v) * C_out;
                else if (col == 0)
                    report(a.status, kErrIndex);
            }
            const float4 z = *reinterpret_cast<const float4*>(sums + (n - m0) * BN + col);
            const float o[4] = {act_apply(z.x + bias[0], a.act), act_apply(z.y + bias[1], a.act),
                                act_apply(z.z + bias[2], a.act), act_apply(z.w + bias[3], a.act)};
            auto store = [&](float* dst) {
                if (out_vec) {
                    if (n0 + col < C_out)
                        *reinterpret_cast<float4*>(dst + n0 + col) = make_float4(o[0], o[1], o[2], o[3]);
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (n0 + col + c < C_out) dst[n0 + col + c] = o[c];
                }
            };
            if (y) store(y + n * C_out);
            if (dp) store(dp);
        }
    }
}

// Calls that 64-row tiles cannot share out twice over the SMs.
bool small_call(const DeviceCtx* ctx, const ConvArgs& a) {
    return a.capacity <= 64ll * ctx->num_sms;
}

template <class C>
hc_status launch_cfg(const DeviceCtx* ctx, const ConvArgs& a, cudaStream_t s) {
    static bool attr_set[64] = {};
    if (!attr_set[ctx->device]) {
        hc_status st = check_cuda(
            cudaFuncSetAttribute(conv_f32_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)C::smem_bytes(HC_MAX_SPIRAL)),
            "cudaFuncSetAttribute(conv_f32_kernel)");
        if (st != HC_OK) return st;
        attr_set[ctx->device] = true;
    }
    const int x_vec = a.C_in % 4 == 0 && (uintptr_t)a.x % 16 == 0;
    const int w_vec = a.C_out % 4 == 0 && (uintptr_t)a.W % 16 == 0;
    const long long items = (a.capacity + kMinRows - 1) / kMinRows * ((a.C_out + C::BN - 1) / C::BN);
    long long grid = ctx->num_sms;
    if (grid > items) grid = items;
    if (grid < 1) grid = 1;
    return launch_pdl(conv_f32_kernel<C>, dim3((unsigned)grid), dim3(C::THREADS), C::smem_bytes(a.L), s,
                      "conv_f32_kernel", a, x_vec, w_vec);
}

}  // namespace

// Where the 64 x 64 tiles of conv_simt.cu, eight blocks an SM, stay ahead. A
// step is one slot, so with few input channels its barrier, gather and round
// trip of the sums are for next to no multiply-adds, while those tiles take
// several slots a step (41.9k rows, 9 slots, 3 -> 64: 44 us here, 22 there at
// every tap present, 12.4 and 10.3 at 15%; 32 slots 129 and 30 us): below 16
// channels, or 8 with the 128-output tiles (8 -> 128: 23 us here, 27 there at
// half of the taps present). A sparse layer above that is taken whatever
// its mask, which only the device knows: with every tap present the tiles would
// be ahead up to 48 channels (16 -> 64: 49 us here, 44 there; 45 -> 64: 112 and
// 88), at half of the taps (21 and 26; 43 and 66) and below it is not close.
// The dense layer has no absent tap to skip besides, so it is not taken where
// channels come element by element (45 -> 42 over 42k rows: 90 us there, 123
// here), where an odd number of 64-wide tiles above one splits the outputs
// (192 -> 192 over 5k rows: 199 and 223), and, with enough rows for the tall
// tiles, where steps are mostly padding: 64-output tiles with steps of 64
// channels (16 -> 64: 44 us there, 49 here; 36: 74 and 78; 56: 105 and 102; 72:
// 134 and 141; 96: 173 and 171), 128-output ones with steps of 32 beyond the
// first (32 -> 128: 110 and 107; 40: 134 and 148; 56: 180 and 181; 128: 390 and
// 380; from 256 outputs on all are ahead here: 40: 260 and 252).
bool conv_f32_preferred(const DeviceCtx* ctx, const ConvArgs& a) {
    const int tiles64 = (a.C_out + 63) / 64;
    const bool wide = tiles64 % 2 == 0;
    if (a.C_in < 8 || (a.C_in < 16 && !wide)) return false;
    if (a.mode != kDense) return true;
    if (a.C_in % 4 != 0 || a.C_in < 16 || (tiles64 > 1 && !wide)) return false;
    if (small_call(ctx, a) || tiles64 >= 4) return true;
    if (wide) return a.C_in <= 32 || 5 * a.C_in >= 4 * ((a.C_in + 31) / 32 * 32);
    return a.C_in > 64 ? a.C_in % 64 == 0 || a.C_in % 64 >= 32 : a.C_in >= 48;
}

hc_status launch_conv_f32(const DeviceCtx* ctx, const ConvArgs& a, cudaStream_t s) {
    // Small calls are bound by round trips: the smaller table is resolved with
    // fewer of them, and more steps are in flight. 16 input channels (a network's first layer) fit
    // half a step.
    const bool small = small_call(ctx, a);
    const bool narrow = a.C_in <= 16;
    // 64-output tiles where 128-output ones would be half empty
    if ((a.C_out + 63) / 64 % 2 == 1) {
        if (small) return narrow ? launch_cfg<Cfg32<8, 64, 64, 16, 8>>(ctx, a, s)
                                 : launch_cfg<Cfg32<8, 64, 64, 32, 6>>(ctx, a, s);
        return a.C_in <= 32 ? launch_cfg<Cfg32<16, 192, 64, 32, 4>>(ctx, a, s)
                            : launch_cfg<Cfg32<16, 192, 64, 64, 2>>(ctx, a, s);
    }
    if (small) return narrow ? launch_cfg<Cfg32<8, 64, 128, 16, 8>>(ctx, a, s)
                             : launch_cfg<Cfg32<8, 64, 128, 32, 6>>(ctx, a, s);
    return launch_cfg<Cfg32<16, 192, 128, 32, 2>>(ctx, a, s);
}

}  // namespace hc
