// Reaction-cross-diffusion (RCD) kernels: M coupled components per mode
// (Supplementary S4.1-S4.3).
#pragma once
#include "internal.h"

namespace spdba {

// Largest component count the RCD kernels take.
constexpr int kRcdMaxComponents = 64;

template <typename T> struct RcdArgs {
    cx_t<T>* u_hat;          // M * n transformed components (component-major)
    const cx_t<T>* g_hat;    // M * n: FFT of the reaction term
    const T* V;              // M x M eigenvectors of D, row-major V[i * M + j] (D = V diag(lam) V^T)
    const T* lam;            // M eigenvalues of D
    const T* k2ax[3];        // |k_a|^2 per axis (padded to 3 axes)
    const T* taper[3];       // transition taper per axis
    const uint8_t* states;
    const uint8_t* chi;
    const int32_t* list;
    const int32_t* count;
    T dt;
    int M;
    // packed (complex64): g_hat holds (M + 1) / 2 fields, components 2c and 2c + 1 of
    // the reaction's transform separated as they are read
    int packed = 0;
    long long n;             // modes per component
    DevStats* stats;         // one (the plan's single run)
};

// R_i(u) = u_i (r - a u_i - sum_{j != i} alpha_ij u_j) at every grid point,
// in place on the inverse transform's output (real parts read, (R, 0) written).
template <typename T>
spdba_status launch_rcd_reaction(cx_t<T>* work, long long n, int M, T r, T a, T alpha, T beta, cudaStream_t st);

// Packed transforms of a complex64 run (rcd_pack.cu): the first inverse pass, which
// forms the packed fields; ok: kernels exist for the shape.
struct RcdPack {
    bool ok = false;
    const void* func = nullptr;
    int H = 0, nt = 0, smem = 0;   // row pairs and threads per CTA
    int M = 0, Mh = 0, N0 = 1, N1 = 1, npairs = 0, tiles = 0;
    long long n = 0;
    FastDiv fd_tiles;
    const float2* tw = nullptr;
};
spdba_status rcd_pack_prepare(RcdPack* o, int ndim, const int64_t* d, int M, TwiddleCache<float>& tw, cudaStream_t st);
spdba_status launch_rcd_pack(const RcdPack& o, const float2* u, float2* z, cudaStream_t st);
// The reaction on the packed fields, in place (z unscaled on entry).
spdba_status launch_rcd_reaction_packed(const RcdPack& o, float2* z, float r, float a, float alpha, float beta,
                                        cudaStream_t st);
// Live rows (n0 * n1) and planes (n0) of the packed forward passes under the states.
spdba_status launch_rcd_live(const Geom& g, const uint8_t* states, uint8_t* row_live, uint8_t* plane_live,
                             cudaStream_t st);

// Per block: maxsq[b] = max_{k in B} A(k)^2 with A(k)^2 = (1/M) sum_m |u_m(k)|^2
// (FP64-accurate: a double-float sum of exact squares for complex64, FP64 for
// complex128); gmax[0] = max over all k, gmax[1] = max over k != 0 (max-reduced:
// zero before).
template <typename T>
spdba_status launch_rcd_activity(const Geom& g, const cx_t<T>* u_hat, int M, double* maxsq, double* gmax,
                                 cudaStream_t st);

// The update (I + dt k^2 D)^{-1} [u_hat + dt g_hat] = V (I + dt k^2 Lambda)^{-1} V^T [...]
// on the listed blocks (dense = 0) or on every block (dense = 1); transition
// blocks blend with the taper.  Adds the step's non-frozen share to the stats.
template <typename T> spdba_status launch_rcd_update(const Geom& g, const RcdArgs<T>& a, int dense, cudaStream_t st);
// Sets the update kernel's shared-memory limit and records its launch shape
// for M components (once per process; call at plan creation).
template <typename T> spdba_status rcd_prepare(int M);

}  // namespace spdba
