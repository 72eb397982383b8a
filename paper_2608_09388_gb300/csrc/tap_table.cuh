// Tap table of a tile of output rows for the CUDA-core kernels: the input row
// feeding every (row, slot), idx() of Eq. 4, or -1 where the tap is absent.
#pragma once

#include "hc_internal.cuh"

namespace hc {

// Rows m0 .. end - 1 of the call (at most BM; the call has `rows` active ones,
// entries of the others are -1) by a block of NT threads, NT / BM (a divisor of
// HC_MAX_SPIRAL) threads per row: entry (r, l) goes to tab[r * row_pitch + l * slot_pitch]. The coordinate, the spiral entries and
// the row_of lookups are each issued together (three dependent round trips),
// from clamped, always-valid addresses, and checked afterwards. The caller
// synchronises before and after.
template <int BM, int NT>
__device__ __forceinline__ void fill_tap_table(const ConvArgs& a, long long rows, long long m0,
                                               long long end, int* tab, int row_pitch, int slot_pitch) {
    constexpr int kPer = NT / BM;                 // threads per row
    static_assert(HC_MAX_SPIRAL % kPer == 0, "whole slots per thread");
    constexpr int kSlots = HC_MAX_SPIRAL / kPer;  // slots l = part + kPer * j of a thread
    const int r = threadIdx.x / kPer, part = threadIdx.x % kPer, L = a.L;
    if (r >= BM) return;
    const long long n = m0 + r;
    const bool in = n < end;
    const long long nn = in ? n : 0;
    unsigned err = 0;
    int b = 0, v = 0;
    if (a.mode == kSparseDenseX || a.mode == kSparseCompactX) {
        b = __ldg(a.coords + 2 * nn);
        v = __ldg(a.coords + 2 * nn + 1);
    } else if (a.mode == kDense) {
        b = (int)(nn / a.V);
        v = (int)(nn - (long long)b * a.V);
    }
    const bool in_range = b >= 0 && b < a.B && v >= 0 && v < a.V;
    if (in && !in_range) err |= kErrIndex;
    const bool ok = in && in_range;
    if (!ok) b = v = 0;
    const bool linear = a.mode == kLinear;
    const bool rb = a.mode == kRulebook;
    int u[kSlots];
#pragma unroll
    for (int j = 0; j < kSlots; ++j) {
        const int l = part + kPer * j < L ? part + kPer * j : L - 1;
        u[j] = linear ? 0
               : rb   ? __ldg(a.rulebook + (long long)l * a.capacity + nn)
                      : __ldg(a.spiral + (long long)v * L + l);
    }
#pragma unroll
    for (int j = 0; j < kSlots; ++j) {
        const int l = part + kPer * j;
        if (l >= L) continue;
        int src = -1;
        if (ok && linear) {
            src = (int)n;
        } else if (ok && rb) {
            if (u[j] < -1 || u[j] >= a.x_rows) err |= kErrIndex;
            else src = u[j];
        } else if (ok) {
            const int uu = u[j];
            if (uu < -1 || uu >= a.V) err |= kErrIndex;
            if (uu >= 0 && uu < a.V) {
                const long long dr = (long long)b * a.V + uu;
                if (a.mode == kDense) {
                    src = (int)dr;
                } else {
                    const int jj = __ldg(a.row_of + dr);
                    if (jj < -1 || jj >= rows) err |= kErrIndex;
                    if (jj >= 0 && jj < rows) src = a.mode == kSparseDenseX ? (int)dr : jj;
                }
            }
        }
        tab[r * row_pitch + l * slot_pitch] = src;
    }
    if (err) report(a.status, err);
}

}  // namespace hc
