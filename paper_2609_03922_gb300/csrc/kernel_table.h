// Lookup of compiled pass kernels by (length, direction, mode, orientation).
#pragma once
#include <stdint.h>

namespace spdba {
struct KernelInfo {
    const void* func = nullptr;
    int P = 0, NT = 0, smem = 0;
    bool pipe = false;  // persistent, double-buffered kernel: grid = resident CTAs
    double cost = 1;    // of a narrow tile: time of a pencil against the wide tile's, the SMs full
};
// Tile sizes of a pass: TILE_WIDE fills 128-byte rows and a CTA; TILE_NARROW is for
// passes of fewer wide tiles than the GPU has SMs; TILE_GENERIC takes any
// pencil count (simple kernel).
enum TileKind { TILE_WIDE = 0, TILE_NARROW = 1, TILE_GENERIC = 2 };
template <typename T>
bool get_pass_kernel(int64_t L, int sign, int mode, bool loadp, bool storep, TileKind kind, bool fourstep,
                     KernelInfo* ki);
// complex64 kernels with two pencils per thread (fft_f32x2.cuh), where they are the faster ones
bool get_pass2_kernel(int64_t L, int sign, int mode, bool strided, bool narrow, KernelInfo* ki);
// rows in, transposed out (unit-stride pencils on the output)
bool get_transpose2_kernel(int64_t L, int sign, KernelInfo* ki);
bool get_chain2_kernel(int64_t L, bool narrow, KernelInfo* ki);
bool get_nl_half2_kernel(int64_t L, int mode, int nhp, KernelInfo* ki);
// the step chain (PASS_CH_CHAIN) along the first axis
template <typename T> bool get_chain_kernel(int64_t L, bool narrow, KernelInfo* ki);
// complex64 half-spectrum passes (PASS_HERM_INV, PASS_NL_HALF, PASS_MIRROR,
// PASS_UPD_HALF); nhp = half row length (PASS_NL_HALF shared memory)
bool get_half_kernel(int64_t L, int mode, int nhp, KernelInfo* ki);
}  // namespace spdba
