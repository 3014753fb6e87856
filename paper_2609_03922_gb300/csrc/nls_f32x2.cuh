// complex64 NLS passes of long signals with two pencils per thread (see
// fft_f32x2.cuh): rows k1, k1 + 1 of a signal, or columns n2, n2 + 1.  The same
// arithmetic as the one-pencil kernels.
#pragma once
#include "fft_f32x2.cuh"
#include "nls.h"

namespace spdba {

// Blockwise half-step of element m of rows k1, k1 + 1 (one block, neighbouring
// places i, i + 1 in it).
struct NlsHalfPair {
    const NLSArgs<float>& a;
    const uint8_t* s_sc;
    const HPair<float>* h0;   // H of row k1 (row k1 + 1 follows 512 entries on)
    int k1;
    __device__ __forceinline__ static cf32x2 half(cf32x2 v, cf32x2 hi, cf32x2 lo, int st, f32x2 sg) {
        const cf32x2 x = cmul(v, hi), y = cmul(v, lo);
        const cf32x2 nw = cadd(x, y);
        if (st == SPDBA_ACTIVE) return nw;
        return mk<cf32x2>(fma_rn(sg, nw.x - v.x, v.x), fma_rn(sg, nw.y - v.y, v.y));
    }
    __device__ __forceinline__ cf32x2 apply(int m, cf32x2 x, bool close, bool open) const {
        const unsigned e = s_sc[m >> a.mb_shift];
        const int st = (int)(e & 3u);
        if (st == SPDBA_FROZEN) return x;
        const float4 p = __ldg(reinterpret_cast<const float4*>(h0 + m));
        const float4 q = __ldg(reinterpret_cast<const float4*>(h0 + 512 + m));
        const cf32x2 hi = mk<cf32x2>(f32x2(p.x, q.x), f32x2(p.y, q.y));
        const cf32x2 lo = mk<cf32x2>(f32x2(p.z, q.z), f32x2(p.w, q.w));
        f32x2 sg(1.f);
        if (st == SPDBA_TRANSITION) {
            const int i = k1 + (int)a.n1 * (m & ((1 << a.mb_shift) - 1));
            const unsigned chi = e >> 2;
            if (chi & 1u) sg = mul_rn(sg, f32x2(a.taper[i], a.taper[i + 1]));
            if (chi & 2u) sg = mul_rn(sg, f32x2(a.taper[a.B - 1 - i], a.taper[a.B - 2 - i]));
        }
        if (close) x = half(x, hi, lo, st, sg);
        if (open) x = half(x, hi, lo, st, sg);
        return x;
    }
};
static_assert(sizeof(HPair<float>) == 16, "H loads move as 16 bytes");

// The tile's half-steps; pencil pair p is rows k1p + 2p, k1p + 2p + 1.
struct NlsRowHalves2 {
    const NLSArgs<float>& a;
    const uint8_t* s_sc;
    int k1p;
    bool close, open;
    __device__ __forceinline__ cf32x2 at(int p, int m, cf32x2 x) const {
        const int k1 = k1p + 2 * p;
        return NlsHalfPair{a, s_sc, a.H + (long long)k1 * 512, k1}.apply(m, x, close, open);
    }
};
struct NlsRowMid2 {
    NlsRowHalves2 h;
    __device__ __forceinline__ void begin(int, int) {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m, cf32x2 x) { return h.at(p, m, x); }
};
struct NlsRowIn2 {
    static constexpr bool EXT = true;
    RowPairIn in;
    NlsRowHalves2 h;
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const {
        const cf32x2 x = in(p, m);
        return h.close || h.open ? h.at(p, m, x) : x;
    }
};
struct NlsRowOut2 {
    static constexpr bool SYNC = false;
    float2* base;   // row 0 of the tile
    NlsRowHalves2 h;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float2* pa = base + (2 * p * 512 + j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int m = j + r * (512 / R);
            const float4 q = quad_of(h.close || h.open ? h.at(p, m, v[r]) : v[r]);
            pa[r * (512 / R)] = make_float2(q.x, q.y);
            pa[r * (512 / R) + 512] = make_float2(q.z, q.w);
        }
    }
};
// Inverse outputs times W_n^{-k1 n2}.
struct NlsRowTwOut2 {
    static constexpr bool SYNC = false;
    float2* base;
    const float2* tw2;   // row k1p of the table
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float2* pa = base + (2 * p * 512 + j);
        const float2* ta = tw2 + (2 * p * 512 + j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 w0 = __ldg(ta + r * (512 / R)), w1 = __ldg(ta + r * (512 / R) + 512);
            const float4 q = quad_of(cmul(v[r], mk<cf32x2>(f32x2(w0.x, w1.x), f32x2(-w0.y, -w1.y))));
            pa[r * (512 / R)] = make_float2(q.x, q.y);
            pa[r * (512 / R) + 512] = make_float2(q.z, q.w);
        }
    }
};

// Row pass, P rows of one signal per CTA: the forward transform (FWD), the closing
// and / or opening half-steps, the inverse transform with its twiddles (INV).
template <int P, int NT, int OCC, bool FWD, bool INV>
__global__ void __launch_bounds__(NT, OCC) nls_row2_kernel(NLSArgs<float> a, FastDiv fd_n1) {
    pdl_wait();
    constexpr int L = 512, H = P / 2;
    using LY = RowLayout<L, H>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    __shared__ uint8_t s_sc[512];
    const uint32_t q0 = blockIdx.x * (uint32_t)P;
    const uint32_t sig = fd_n1.div(q0);   // a tile lies within one signal (P divides n1)
    const int k1p = (int)(q0 - sig * (uint32_t)a.n1);
    stage_twiddles<L, NT>(s_tw, a.tw);
    const bool halves = a.do_close || a.do_open;
    if (halves) {
        for (int b = threadIdx.x; b < a.nblk; b += NT) {
            const long long id = (long long)sig * a.nblk + b;
            s_sc[b] = a.dense ? (uint8_t)SPDBA_ACTIVE : (uint8_t)(a.states[id] | (a.chi[id] << 2));
        }
        if constexpr (!FWD) __syncthreads();   // else the first stage's barrier makes them visible
    }
    const float2* src = a.in + (long long)q0 * L;
    float2* dst = a.S + (long long)q0 * L;
    const NlsRowHalves2 h{a, s_sc, k1p, a.do_close != 0, a.do_open != 0};
    if constexpr (FWD && INV) {
        RowPairIn in{src, L};
        NlsRowMid2 mid{h};
        NlsRowTwOut2 out{dst, a.tw4 + (long long)k1p * 512};
        transform_pair_in<f32x2, L, H, NT, -1, +1, LY>(sm, s_tw, in, mid, out);
    } else if constexpr (FWD) {
        RowPairIn in{src, L};
        NlsRowOut2 out{dst, h};
        run_stages_in_out<f32x2, L, H, NT, -1, LY>(sm, s_tw, in, out);
    } else {
        // the half-steps read the block states: staged before the first stage reads
        NlsRowIn2 in{{src, L}, h};
        NlsRowTwOut2 out{dst, a.tw4 + (long long)k1p * 512};
        __syncthreads();
        run_stages_in_out<f32x2, L, H, NT, +1, LY>(sm, s_tw, in, out);
    }
}

// E = x / n and the Kerr phase of both columns.
struct NlsKerrMid2 {
    float inv_n, gamma_h;
    bool kerr;
    float pw;
    __device__ __forceinline__ void begin(int, int) {}
    __device__ __forceinline__ cf32x2 operator()(int, int, cf32x2 x) {
        x = cscale(x, f32x2(inv_n));
        if (!kerr) return x;
        const float2 e0 = nls_kerr(make_float2(x.x.lo(), x.y.lo()), gamma_h, pw);
        const float2 e1 = nls_kerr(make_float2(x.x.hi(), x.y.hi()), gamma_h, pw);
        return mk<cf32x2>(f32x2(e0.x, e1.x), f32x2(e0.y, e1.y));
    }
};
// Forward outputs times W_n^{n2 k1}; inverse outputs alone: E = x / n (INV).
template <int L> struct NlsColTwOut2 {
    static constexpr bool SYNC = false;
    float2* base;
    const float2* tw2;   // column n2 of row 0
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float2* po = base + (2 * p + j * 512);
        const float2* t = tw2 + (2 * p + j * 512);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 w = __ldg(reinterpret_cast<const float4*>(t + r * (L / R) * 512));
            *reinterpret_cast<float4*>(po + r * (L / R) * 512) = quad_of(cmul(v[r], pair_of(w)));
        }
    }
};

// Column pass, P columns of one signal per CTA: inverse transform, Kerr, forward
// transform (INV && FWD), or one of them (get_field, set_field).
template <int L, int P, int NT, int OCC, bool INV, bool FWD>
__global__ void __launch_bounds__(NT, OCC) nls_col2_kernel(NLSArgs<float> a) {
    pdl_wait();
    constexpr int H = P / 2;
    using LY = LayoutB<L, H>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    constexpr int TPS = 512 / P;   // tiles per signal
    const long long sig = blockIdx.x / TPS;
    const int n20 = (int)(blockIdx.x % TPS) * P;
    if constexpr (INV && FWD) nls_step_stats<float>(a);
    stage_twiddles<L, NT>(s_tw, a.tw);
    GlobalPairIn in{a.in + (sig * a.n + n20), 512};
    float2* dst = a.S + (sig * a.n + n20);
    if constexpr (INV && FWD) {
        NlsKerrMid2 mid{a.inv_n, a.gamma_h, a.do_kerr != 0, 0.f};
        NlsColTwOut2<L> out{dst, a.tw4 + n20};
        transform_pair_in<f32x2, L, H, NT, +1, -1, LY>(sm, s_tw, in, mid, out);
        if (a.power) {
            const double w = warp_sum((double)mid.pw);
            if ((threadIdx.x & 31) == 0) atomicAdd(a.power + sig * a.power_stride, w);
        }
    } else if constexpr (FWD) {
        NlsColTwOut2<L> out{dst, a.tw4 + n20};
        run_stages_in_out<f32x2, L, H, NT, -1, LY>(sm, s_tw, in, out);
    } else {
        GlobalPairOut<L> out{dst, 512, f32x2(a.inv_n)};
        run_stages_in_out<f32x2, L, H, NT, +1, LY>(sm, s_tw, in, out);
    }
}

struct NlsRow2 {
    static constexpr int P = 4, NT = 128, OCC = 6;
    static int smem() { return RowLayout<512, P / 2>::SIZE * (int)sizeof(cf32x2); }
    template <bool F, bool I> static const void* func() { return (const void*)nls_row2_kernel<P, NT, OCC, F, I>; }
};
// threads and CTAs per SM per column length (16 columns a tile)
template <int L> struct NlsCol2Cfg;
template <> struct NlsCol2Cfg<32> { static constexpr int NT = 64, OCC = 8; };
template <> struct NlsCol2Cfg<64> { static constexpr int NT = 64, OCC = 8; };
template <> struct NlsCol2Cfg<128> { static constexpr int NT = 128, OCC = 5; };
template <> struct NlsCol2Cfg<256> { static constexpr int NT = 128, OCC = 4; };
template <> struct NlsCol2Cfg<512> { static constexpr int NT = 512, OCC = 1; };
template <int L> struct NlsCol2 {
    static constexpr int P = 16, NT = NlsCol2Cfg<L>::NT, OCC = NlsCol2Cfg<L>::OCC;
    static int smem() { return LayoutB<L, P / 2>::SIZE * (int)sizeof(cf32x2); }
    template <bool I, bool F> static const void* func() { return (const void*)nls_col2_kernel<L, P, NT, OCC, I, F>; }
    static spdba_status prepare() {
        const void* f[3] = {func<true, true>(), func<true, false>(), func<false, true>()};
        for (const void* k : f) {
            if (smem() > 48 * 1024)
                SPDBA_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem()));
            SPDBA_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        }
        return SPDBA_OK;
    }
    static spdba_status launch(const NLSArgs<float>& a, cudaStream_t st) {
        const void* k = a.do_inv ? (a.do_fwd ? func<true, true>() : func<true, false>()) : func<false, true>();
        NLSArgs<float> v = a;
        void* args[] = {&v};
        SPDBA_CUDA(pdl_launch_ptr(k, dim3((unsigned)(a.batch * (512 / P))), dim3(NT), args, (size_t)smem(), st));
        return SPDBA_OK;
    }
};

}  // namespace spdba
