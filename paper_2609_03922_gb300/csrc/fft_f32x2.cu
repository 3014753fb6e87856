// Selection of the complex64 kernels with two pencils per thread.
#include <algorithm>

#include "fft_f32x2.cuh"
#include "internal.h"
#include "kernel_table.h"

namespace spdba {

// The choices below are the fastest of the shapes measured per length (pencils
// per tile, threads, CTAs per SM) against the one-pencil kernels, which keep the
// lengths that are left out.
template <int L, int P, int NT, int OCC> static bool strided(int sign, KernelInfo* ki) {
    ki->P = P;
    ki->NT = NT;
    ki->pipe = true;
    ki->smem = 2 * L * P * (int)sizeof(float2);
    ki->func = sign < 0 ? (const void*)fft_pipe2_kernel<L, P, NT, -1, OCC> : (const void*)fft_pipe2_kernel<L, P, NT, +1, OCC>;
    return true;
}
template <int L, int P, int NT, int OCC> static bool rows(int sign, int mode, KernelInfo* ki) {
    ki->P = P;
    ki->NT = NT;
    ki->pipe = false;
    ki->smem = RowLayout<L, P / 2>::SIZE * (int)sizeof(cf32x2);
    ki->func = mode == PASS_CH_NL ? (const void*)fft_rows2_kernel<L, P, NT, -1, PASS_CH_NL, OCC>
               : mode == PASS_R2C ? (const void*)fft_rows2_kernel<L, P, NT, -1, PASS_R2C, OCC>
               : mode == PASS_C2R ? (const void*)fft_rows2_kernel<L, P, NT, +1, PASS_C2R, OCC>
               : sign < 0         ? (const void*)fft_rows2_kernel<L, P, NT, -1, PASS_PLAIN, OCC>
                                  : (const void*)fft_rows2_kernel<L, P, NT, +1, PASS_PLAIN, OCC>;
    return true;
}

bool get_pass2_kernel(int64_t L, int sign, int mode, bool strided_axis, bool narrow, KernelInfo* ki) {
    if (strided_axis) {
        if (mode != PASS_PLAIN || narrow) return false;
        if (L == 128) return strided<128, 16, 64, 6>(sign, ki);
        if (L == 256) return strided<256, 16, 128, 3>(sign, ki);
        if (L == 384) return strided<384, 16, 192, 2>(sign, ki);
        return false;
    }
    if (mode != PASS_PLAIN && mode != PASS_CH_NL && mode != PASS_R2C && mode != PASS_C2R) return false;
    if (narrow) {
        // four rows a tile
        switch (L) {
            case 64: return rows<64, 4, 32, 16>(sign, mode, ki);
            case 128: return rows<128, 4, 32, 16>(sign, mode, ki);
            case 192: return rows<192, 4, 64, 8>(sign, mode, ki);
            case 256: return rows<256, 4, 32, 16>(sign, mode, ki);
            case 384: return rows<384, 4, 96, 6>(sign, mode, ki);
            case 512: return rows<512, 4, 128, 4>(sign, mode, ki);
            default: return false;
        }
    }
    switch (L) {
        case 64: return rows<64, 16, 64, 8>(sign, mode, ki);
        case 128: return rows<128, 16, 64, 7>(sign, mode, ki);
        case 192: return rows<192, 16, 192, 3>(sign, mode, ki);
        case 256: return rows<256, 16, 128, 4>(sign, mode, ki);
        case 384: return rows<384, 8, 64, 6>(sign, mode, ki);
        case 512: return rows<512, 8, 128, 4>(sign, mode, ki);
        default: return false;
    }
}

bool get_transpose2_kernel(int64_t L, int sign, KernelInfo* ki) {
    if (L != 512) return false;   // the row length of every four-step transform
    constexpr int P = 16, NT = 256, OCC = 2;
    ki->P = P;
    ki->NT = NT;
    ki->pipe = false;
    ki->smem = LayoutA<512, P / 2, true>::SIZE * (int)sizeof(cf32x2);
    ki->func = sign < 0 ? (const void*)fft_rows_transpose2_kernel<512, P, NT, -1, OCC>
                        : (const void*)fft_rows_transpose2_kernel<512, P, NT, +1, OCC>;
    return true;
}

template <int L, int P, int NT, int OCC> static bool chain(KernelInfo* ki) {
    ki->P = P;
    ki->NT = NT;
    ki->pipe = false;
    ki->smem = 2 * L * P * (int)sizeof(float2);
    ki->func = (const void*)fft_chain2_kernel<L, P, NT, OCC>;
    return true;
}
bool get_chain2_kernel(int64_t L, bool narrow, KernelInfo* ki) {
    if (narrow) return false;
    switch (L) {
        case 64: return chain<64, 16, 64, 8>(ki);
        case 128: return chain<128, 16, 128, 5>(ki);
        case 192: return chain<192, 16, 192, 3>(ki);
        case 256: return chain<256, 16, 128, 3>(ki);
        case 384: return chain<384, 16, 384, 2>(ki);
        default: return false;
    }
}

int chain2_step(int64_t L) {
    switch (L) {
        case 64: return 64 / Radices_last<f32x2, 64>::value;
        case 128: return 128 / Radices_last<f32x2, 128>::value;
        case 192: return 192 / Radices_last<f32x2, 192>::value;
        case 256: return 256 / Radices_last<f32x2, 256>::value;
        case 384: return 384 / Radices_last<f32x2, 384>::value;
        default: return 1;
    }
}

template <int L, int P, int NT, int OCC, bool ST> static bool nl_half(int mode, int nhp, KernelInfo* ki) {
    ki->P = P;
    ki->NT = NT;
    ki->pipe = false;
    const int tile = RowLayout<L, P / 4>::SIZE * (int)sizeof(cf32x2);
    ki->smem = ST && mode != PASS_R2C_HALF ? std::max(tile, P * nhp * (int)sizeof(float2)) : tile;
    ki->func = mode == PASS_NL_HALF    ? (const void*)fft_nl_half2_kernel<L, P, NT, OCC, ST, PASS_NL_HALF>
               : mode == PASS_R2C_HALF ? (const void*)fft_nl_half2_kernel<L, P, NT, OCC, ST, PASS_R2C_HALF>
                                       : (const void*)fft_nl_half2_kernel<L, P, NT, OCC, ST, PASS_C2R_HALF>;
    return true;
}
bool get_nl_half2_kernel(int64_t L, int mode, int nhp, KernelInfo* ki) {
    switch (L) {
        case 64: return nl_half<64, 32, 64, 8, false>(mode, nhp, ki);
        case 128: return nl_half<128, 32, 64, 8, true>(mode, nhp, ki);
        case 256: return nl_half<256, 32, 128, 5, true>(mode, nhp, ki);
        case 384: return nl_half<384, 16, 64, 6, true>(mode, nhp, ki);
        case 512: return mode != PASS_NL_HALF && nl_half<512, 16, 128, 4, true>(mode, nhp, ki);
        default: return false;
    }
}

}  // namespace spdba
