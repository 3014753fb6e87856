// complex64 passes with two pencils per thread.
//
// A thread's butterfly carries the same element of two neighbouring pencils as
// packed FP32 pairs (Cx<f32x2>), so that every transform operation is one
// packed instruction for both: half the issue slots of the arithmetic, the same
// bits as the scalar kernels.  First-stage inputs come straight from global
// memory into registers (16-byte loads of the two pencils) and last-stage
// outputs go straight back, so shared memory holds one tile, its traffic is
// halved, and CTAs of one tile each overlap one another instead of a second
// buffer.
#pragma once
#include "fft_core.cuh"

namespace spdba {

// (re0, im0, re1, im1) in memory <-> packed pair
__device__ __forceinline__ cf32x2 pair_of(float4 q) { return mk<cf32x2>(f32x2(q.x, q.z), f32x2(q.y, q.w)); }
__device__ __forceinline__ float4 quad_of(cf32x2 c) { return make_float4(c.x.lo(), c.y.lo(), c.x.hi(), c.y.hi()); }

// The shared twiddle table of tw_at, stage after stage (L minus the first radix entries).
// A table in index order with each factor stored twice (16 bytes) made half of the row
// kernels' shared wavefronts: strides of the last stages put up to eight lanes on one
// bank.  As it is now, with fields in and out: 256^3 half 2739 -> 2646 us (20 steps),
// 384^3 6372 -> 6100 us (10), the 64-run ensemble 6258 -> 5865 us, 64 NLS signals 4709 ->
// 4181 us, 32 transforms of 2^18 forward and back 140 -> 130 us.
template <int L, int NT, int I = 1>
__device__ __forceinline__ void stage_twiddles(float2* s_tw, const float2* __restrict__ tw) {
    constexpr int NS = ns_at<f32x2, L>(I), R = radix_at<f32x2, L>(I);
    float2* dst = s_tw + (NS - radix_at<f32x2, L>(0));
#pragma unroll
    for (int e = threadIdx.x; e < (R - 1) * NS; e += NT) {
        const int r = e / NS + 1, jm = e % NS;
        dst[e] = __ldg(tw + r * jm * (L / (NS * R)));
    }
    if constexpr (I + 1 < NSTAGES<f32x2, L>::value) stage_twiddles<L, NT, I + 1>(s_tw, tw);
}

// L2 priority of c_hat's lines in the chain.  stream: they are dropped first, so
// that the workspace the passes share stays in the L2.
__device__ __forceinline__ unsigned long long chat_policy(int stream) {
    unsigned long long first, normal;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(first));
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(normal));
    return stream ? first : normal;
}
__device__ __forceinline__ void cp_async16_hint(void* smem, const void* gmem, unsigned long long pol) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;\n" ::"r"(d), "l"(gmem), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_hint(float4* p, float4 v, unsigned long long pol) {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;\n" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z),
                 "f"(v.w), "l"(pol) : "memory");
}

// Input element m of pencil pair p, row-major global tile (pencils adjacent).
struct GlobalPairIn {
    static constexpr bool EXT = true;
    const float2* base;   // (pencil 0 of the tile, element 0)
    int sJ;
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const {
        return pair_of(*reinterpret_cast<const float4*>(base + (2 * p + m * sJ)));
    }
};
// Raw (interleaved) tile in shared memory, pairs of row m at m * H + p.
template <int H, bool X = false> struct RawPairIn {
    static constexpr bool EXT = X;   // X: the raw tile is not the buffer the transform works in
    const float4* cs;
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const { return pair_of(cs[m * H + p]); }
};
template <int L> struct GlobalPairOut {
    static constexpr bool SYNC = false;
    float2* base;
    int sJ;
    f32x2 scale;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float2* po = base + (2 * p + j * sJ);
#pragma unroll
        for (int r = 0; r < R; ++r)
            *reinterpret_cast<float4*>(po + r * (L / R) * sJ) = quad_of(cscale(v[r], scale));
    }
};

// ---------------------------------------------------------------- plain strided pass
// Pipelined: persistent CTAs walk the tiles; the next tile streams into the
// second buffer with cp.async while the current one is transformed in place.
// HBM and the L2 bound it.  256 points over a 256 x 256 x 144 array in place:
// 20.9 us with one pencil per thread, 19.2 us with two (7.9 TB/s read + written);
// 384 points over 384 x 384 x 208: 143 us (8-pencil tiles) and 87 us.  With 128 points so
// too: RCD 128^3 x 48 with fields in and out 12373 -> 12129 us, 192 x 128 x 256 1999 -> 1946 us.
template <int L, int P, int NT, int SIGN, int OCC>
__global__ void __launch_bounds__(NT, OCC) fft_pipe2_kernel(PassParams<float> a) {
    pdl_wait();
    constexpr int H = P / 2;
    using LY = LayoutB<L, H>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const b0 = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    stage_twiddles<L, NT>(s_tw, a.tw);   // visible after the loop's first barrier
    const int ntiles = (int)((a.O * a.I) / P), G = (int)gridDim.x, sJ = (int)a.isJ;
    const int p = (int)(threadIdx.x % H), j0 = (int)(threadIdx.x / H);
    static_assert(NT % H == 0, "each thread copies one pencil pair");
    auto next_live = [&](int t) {
        if (a.col_live == nullptr && a.seg_live == nullptr) return t;
        while (t < ntiles && !tile_live<float, P, PASS_PLAIN>(a, (long long)t * P)) t += G;
        return t;
    };
    auto issue = [&](cf32x2* b, int t) {
        const long long q0 = (long long)t * P, o = a.fd_I.div((uint32_t)q0);
        const float2* base = a.in + (o * a.isO + (q0 - o * a.I)) + 2 * p;
#pragma unroll 8
        for (int j = j0; j < L; j += NT / H) cp_async16(b + j * H + p, base + j * sJ);
    };
    int t = next_live(blockIdx.x);
    if (t < ntiles) issue(b0, t);
    cp_async_commit();
    int buf = 0;
    while (t < ntiles) {
        const int tn = next_live(t + G);
        if (tn < ntiles) issue(b0 + (buf ^ 1) * LY::SIZE, tn);
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();
        cf32x2* const sm = b0 + buf * LY::SIZE;
        const long long q0 = (long long)t * P, o = a.fd_I.div((uint32_t)q0);
        GlobalPairOut<L> out{a.out + (o * a.osO + (q0 - o * a.I)), (int)a.osJ, f32x2(a.scale)};
        RawPairIn<H> in{reinterpret_cast<const float4*>(sm)};
        run_stages_in_out<f32x2, L, H, NT, SIGN, LY>(sm, s_tw, in, out);
        __syncthreads();
        buf ^= 1;
        t = tn;
    }
    cp_async_wait<0>();
}

// ---------------------------------------------------------------- step chain
// fft_chain_kernel with two pencils per thread.  Blocks have an even edge along
// the fast axis, so that both pencils of a pair lie in one block, and an edge
// along the pass axis that divides the butterfly's element step Q = L / R, so
// that a thread's elements j + r Q all sit at one place in blocks that follow
// one another at a fixed step: no division, and no index arithmetic but adds,
// per element (the update, not the transforms, was two thirds of the kernel's
// instructions).  Measured (all blocks updated, g and c_hat in place): 256 points
// over 256 x 256 x 144 79.9 us with one pencil per thread, 63.2 us here with c_hat
// streamed past the L2 (73 us without); 192 x 256 x 144 73.8 -> 44.7 us; 384 x 384 x
// 208 330 -> 232 us; 64 x 64 x 144 7.0 -> 4.7 us.
template <int L, int H, int Q> struct ChainMid2 {
    const CHFuse<float>& f;
    const uint8_t* tab;
    const float* kp;
    const float4* cs;
    float2* cb;           // c_hat of (the pair's first pencil, j = 0)
    int nbx, bstep, lx, l_out, osJ;
    bool d3;
    f32x2 kx, ndt, dtk;
    float kc;
    // of the current butterfly: its first element, that element's table entry,
    // place in the block and c_hat
    int j0, lj;
    const uint8_t* te;
    float2* ce;
    unsigned long long pol;
    // edge: pair p is at columns x0 + 2 (p & 1) of row cy + p / 2, else x0 + 2 p of row cy
    __device__ __forceinline__ ChainMid2(const PassParams<float>& a, const UpdTile& u, bool edge, long long at,
                                         const uint8_t* tab_, const float* kp_, const float4* cs_,
                                         unsigned long long pol_)
        : f(a.fu), tab(tab_), kp(kp_), cs(cs_) {
        d3 = f.g.ndim == 3;
        nbx = u.nbx;
        const int p = (int)(threadIdx.x % H);
        const int x = u.x0 + 2 * (edge ? p & 1 : p), bx = (int)f.fd_b2.div((uint32_t)x);
        int cy = u.cy;
        l_out = u.l_out;
        if (edge) {
            cy += p >> 1;
            const int by = (int)f.fd_b1.div((uint32_t)cy);
            l_out = cy - by * f.g.b[1];
            tab += by - (int)f.fd_b1.div((uint32_t)u.cy);
        } else {
            tab += bx - u.bx0;
        }
        bstep = (int)f.fd_bp.div((uint32_t)Q) * nbx;
        lx = x - bx * f.g.b[2];
        kx = f32x2(f.k2ax[2][x], f.k2ax[2][x + 1]);
        kc = d3 ? f.k2ax[1][cy] : f.k2ax[0][cy];
        cb = f.c_hat + at;
        osJ = (int)a.osJ;
        ndt = f32x2(-f.dt);
        dtk = f32x2(f.dtkappa);
        pol = pol_;
    }
    __device__ __forceinline__ void begin(int, int j) {
        j0 = j;
        const int bp = (int)f.fd_bp.div((uint32_t)j);
        lj = j - bp * (int)f.fd_bp.d;
        te = tab + bp * nbx;
        ce = cb + (long long)j * osJ;
    }
    __device__ __forceinline__ cf32x2 operator()(int p, int m, cf32x2 gv) {
        const int r = (m - j0) / Q;   // a constant once unrolled
        const cf32x2 c = pair_of(cs[m * H + p]);
        const unsigned e = te[r * bstep];
        const int st = (int)(e & 3u);
        if (st == SPDBA_FROZEN) return c;
        // ch_new for both modes, operation by operation
        const f32x2 k2 = f32x2(kp[m] + kc) + kx;
        const f32x2 den = fma_rn(dtk, mul_rn(k2, k2), f32x2(1.f));
        const f32x2 inv(rcp_approx(den.lo()), rcp_approx(den.hi()));
        const f32x2 na = mul_rn(ndt, k2);
        cf32x2 nv = mk<cf32x2>(mul_rn(fma_rn(na, gv.x, c.x), inv), mul_rn(fma_rn(na, gv.y, c.y), inv));
        if (st == SPDBA_TRANSITION) {
            const int l0 = d3 ? lj : 0, l1 = d3 ? l_out : lj;
            const float2 b0 = ch_blend<float>(make_float2(c.x.lo(), c.y.lo()), make_float2(nv.x.lo(), nv.y.lo()),
                                              f.taper, f.g, e >> 2, l0, l1, lx);
            const float2 b1 = ch_blend<float>(make_float2(c.x.hi(), c.y.hi()), make_float2(nv.x.hi(), nv.y.hi()),
                                              f.taper, f.g, e >> 2, l0, l1, lx + 1);
            nv = mk<cf32x2>(f32x2(b0.x, b1.x), f32x2(b0.y, b1.y));
        }
        st_hint(reinterpret_cast<float4*>(ce + (long long)r * (Q * osJ)), quad_of(nv), pol);
        return nv;
    }
};

// A thread's one pencil pair (base: its element 0) in the pass's arrays, read while the
// thread's cp.async copies land: complete, and visible to every thread after the
// stage's barrier.
struct ThreadPairIn {
    static constexpr bool EXT = true;
    const float2* base;
    int sJ;
    __device__ __forceinline__ void before_write() const { cp_async_wait<0>(); }
    __device__ __forceinline__ cf32x2 operator()(int, int m) const {
        return pair_of(*reinterpret_cast<const float4*>(base + m * sJ));
    }
};
template <int L> struct ThreadPairOut {
    static constexpr bool SYNC = false;
    float2* base;
    int sJ;
    f32x2 scale;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int, int j, cf32x2 (&v)[R]) {
        float2* po = base + j * sJ;
#pragma unroll
        for (int r = 0; r < R; ++r)
            *reinterpret_cast<float4*>(po + r * (L / R) * sJ) = quad_of(cscale(v[r], scale));
    }
};

// Pencil pair p of a tile of the chain: columns q0 + 2 p and the next of one row, or in an
// edge tile the columns q0 .. q0 + 3 of P / 4 rows, two pairs a row.  A stored half has
// one used column right of its whole tiles (129 of 144 at 256 points, 33 of 48 at 64);
// a tile per row would transform and move 15 columns of padding beside it.  Four columns
// are a sector of 32 bytes: with two, half sectors were written, and 256^3 took 3 us a
// step more, not less.
struct PairTile {
    int q0, row;   // row: 0, or the row width of an edge tile
    __device__ __forceinline__ int pencil(int p) const {
        return row == 0 ? q0 + 2 * p : q0 + (p >> 1) * row + 2 * (p & 1);
    }
};
template <int P> __device__ __forceinline__ PairTile pair_tile(const PassParams<float>& a, int t) {
    if (!a.edge) return PairTile{t * P, 0};
    const int w = (int)a.fu.g.n[2], per_row = (int)a.fd_seg.d, t0 = (int)a.fu.g.n[1] * per_row;
    if (t >= t0) return PairTile{(t - t0) * (P / 4) * w + per_row * P, w};
    const int row = (int)a.fd_seg.div((uint32_t)t);
    return PairTile{row * w + (t - row * per_row) * P, 0};
}

template <int L, int P, int NT, int OCC>
__global__ void __launch_bounds__(NT, OCC) fft_chain2_kernel(PassParams<float> a) {
    pdl_wait();
    constexpr int H = P / 2;
    using LY = LayoutB<L, H>;
    static_assert(NT % H == 0, "each thread keeps one pencil pair");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    float4* const cs = reinterpret_cast<float4*>(sm + LY::SIZE);
    __shared__ uint8_t s_tab[kUpdTable];
    __shared__ float s_kp[L];
    __shared__ float2 s_tw[L];
    const CHFuse<float>& f = a.fu;
    const PairTile pt = pair_tile<P>(a, (int)blockIdx.x);
    const bool edge = pt.row != 0;
    UpdTile u = upd_tile<float, P>(a, pt.q0);
    if (edge) {
        // one table column per row of blocks that the tile's rows meet
        u.nbx = (int)f.fd_b1.div((uint32_t)(u.cy + P / 4 - 1)) - (int)f.fd_b1.div((uint32_t)u.cy) + 1;
        u.bxstep = (int)f.g.nb[2];
    }
    const unsigned long long pol = chat_policy(a.stream_chat);
    const int p = (int)(threadIdx.x % H);
    const int q = pt.pencil(p), o = (int)a.fd_I.div((uint32_t)q);
    const long long at = o * a.osO + (q - o * a.I);   // in place: input strides are the output's
    {
        const int j0 = (int)(threadIdx.x / H), sJ = (int)a.osJ;
        const float2* cbase = f.c_hat + at;
#pragma unroll 8
        for (int j = j0; j < L; j += NT / H) cp_async16_hint(cs + j * H + p, cbase + j * sJ, pol);
        cp_async_commit();
    }
    ch_update_table<float, L, P, NT>(s_tab, a, u);
    const float* kpg = f.g.ndim == 3 ? f.k2ax[0] : f.k2ax[1];
    for (int j = threadIdx.x; j < L; j += NT) s_kp[j] = kpg[j];
    stage_twiddles<L, NT>(s_tw, a.tw);
    ch_update_stats<float, NT>(f, f.dense);
    bool live = true;
    if (!f.dense) {
        const int nent = (int)(f.g.ndim == 3 ? f.g.nb[0] : f.g.nb[1]) * u.nbx;
        __syncthreads();
        int any = 0;
        for (int k = threadIdx.x; k < nent; k += NT) any |= (s_tab[k] & 3) != SPDBA_FROZEN;
        live = __syncthreads_or(any) != 0;
    }
    ThreadPairOut<L> out{a.out + at, (int)a.osJ, f32x2(1.f)};
    if (live) {
        ThreadPairIn in{a.in + at, (int)a.isJ};
        ChainMid2<L, H, L / Radices_last<f32x2, L>::value> mid(a, u, edge, at, s_tab, s_kp, cs, pol);
        transform_pair_in<f32x2, L, H, NT, -1, +1, LY>(sm, s_tw, in, mid, out, a.last != 0);
    } else {
        cp_async_wait<0>();
        if (a.last) return;
        __syncthreads();
        RawPairIn<H, true> in{cs};
        run_stages_in_out<f32x2, L, H, NT, +1, LY>(sm, s_tw, in, out);
    }
}

// ---------------------------------------------------------------- rows (contiguous pencils)
// Pencils p and p + 1 of a pair are neighbouring rows; lanes run along a row.
template <int L, int H> using RowLayout = LayoutA<L, H, false>;

struct RowPairIn {
    static constexpr bool EXT = true;
    const float2* base;   // row 0 of the tile
    int sI;               // row stride
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const {
        const float2 a = base[2 * p * sI + m], b = base[(2 * p + 1) * sI + m];
        return mk<cf32x2>(f32x2(a.x, b.x), f32x2(a.y, b.y));
    }
};
template <int L> struct RowPairOut {
    static constexpr bool SYNC = false;
    float2* base;
    int sI;
    f32x2 scale;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float2* pa = base + (2 * p * sI + j);
        float2* pb = pa + sI;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 q = quad_of(cscale(v[r], scale));
            pa[r * (L / R)] = make_float2(q.x, q.y);
            pb[r * (L / R)] = make_float2(q.z, q.w);
        }
    }
};

// Real rows in or out (base: the float field).
struct RealRowPairIn {
    static constexpr bool EXT = true;
    const float* base;
    int sI;
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const {
        return mk<cf32x2>(f32x2(base[2 * p * sI + m], base[(2 * p + 1) * sI + m]), f32x2(0.f));
    }
};
template <int L> struct RealRowPairOut {
    static constexpr bool SYNC = false;
    float* base;
    int sI;
    f32x2 scale;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float* pa = base + (2 * p * sI + j);
        float* pb = pa + sI;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const f32x2 x = mul_rn(v[r].x, scale);
            pa[r * (L / R)] = x.lo();
            pb[r * (L / R)] = x.hi();
        }
    }
};

// MODE: PASS_PLAIN, PASS_R2C / PASS_C2R (real rows in / real parts out), or PASS_CH_NL
// (inverse, c = Re / N and g = c^3 - c, forward).
// Measured (rows x length, in place; pipelined one-pencil kernel before): plain
// 65536 x 256 56.8 -> 51.9 us, 147456 x 384 323 -> 194 us, 32768 x 64 7.6 -> 5.6 us;
// nonlinear 70.2 -> 60.1, 455 -> 285, 10.0 -> 7.5 us.
template <int L, int P, int NT, int SIGN, int MODE, int OCC>
__global__ void __launch_bounds__(NT, OCC) fft_rows2_kernel(PassParams<float> a) {
    pdl_wait();
    constexpr int H = P / 2;
    using LY = RowLayout<L, H>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    const long long q0 = (long long)blockIdx.x * P;
    const long long o = a.fd_I.div((uint32_t)q0), i0 = q0 - o * a.I;
    if (MODE == PASS_PLAIN && a.seg_live != nullptr) {
        // P rows of one field (its rows are a whole number of tiles)
        const uint32_t r0 = (uint32_t)q0 - a.fd_seg.div((uint32_t)q0) * a.fd_seg.d;
        bool live = false;
#pragma unroll
        for (int p = 0; p < P; ++p) live |= a.seg_live[r0 + p] != 0;
        if (!live) return;
    }
    stage_twiddles<L, NT>(s_tw, a.tw);
    RowPairIn in{a.in + (o * a.isO + i0 * a.isI), (int)a.isI};
    RowPairOut<L> out{a.out + (o * a.osO + i0 * a.osI), (int)a.osI, f32x2(a.scale)};
    if constexpr (MODE == PASS_CH_NL) {
        ChNlMid<f32x2> mid{f32x2(a.nl_scale), f32x2(0.f)};
        transform_pair_in<f32x2, L, H, NT, +1, -1, LY>(sm, s_tw, in, mid, out);
        if (a.mass != nullptr) {
            const double ms = warp_sum((double)mid.msum.lo() + (double)mid.msum.hi());
            if ((threadIdx.x & 31) == 0) atomicAdd(a.mass + (q0 / a.mass_ppr) * a.mass_stride, ms);
        }
    } else if constexpr (MODE == PASS_R2C) {
        RealRowPairIn rin{reinterpret_cast<const float*>(a.in) + i0 * a.isI, (int)a.isI};
        run_stages_in_out<f32x2, L, H, NT, SIGN, LY>(sm, s_tw, rin, out);
    } else if constexpr (MODE == PASS_C2R) {
        RealRowPairOut<L> rout{reinterpret_cast<float*>(a.out) + i0 * a.osI, (int)a.osI, f32x2(a.scale)};
        run_stages_in_out<f32x2, L, H, NT, SIGN, LY>(sm, s_tw, in, rout);
    } else {
        run_stages_in_out<f32x2, L, H, NT, SIGN, LY>(sm, s_tw, in, out);
    }
}

// Natural-order outputs to shared memory.
template <int L, class LY> struct SmemOut2 {
    static constexpr bool SYNC = true;
    cf32x2* sm;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
#pragma unroll
        for (int r = 0; r < R; ++r) sm[LY::idx(p, j + r * (L / R))] = v[r];
    }
};

// Rows in, columns out: the second pass of a four-step transform, whose pencils
// are rows of the input and adjacent in the output.  The last stage leaves the
// tile in shared memory (odd row stride: lanes then read across the rows without
// conflicts) and pairs of pencils leave as 16-byte columns, 128 bytes a tile row.
// The one-pencil kernel (76 us for 32 x 512 rows of 512) loaded, transformed and
// stored a tile with nothing in flight; with this pass and the twiddles in the
// first one, 32 transforms of 2^18 forward and back take 140 us, 416 before.
template <int L, int P, int NT, int SIGN, int OCC>
__global__ void __launch_bounds__(NT, OCC) fft_rows_transpose2_kernel(PassParams<float> a) {
    pdl_wait();
    constexpr int H = P / 2;
    using LY = LayoutA<L, H, true>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    const long long q0 = (long long)blockIdx.x * P;
    const long long o = a.fd_I.div((uint32_t)q0), i0 = q0 - o * a.I;
    stage_twiddles<L, NT>(s_tw, a.tw);
    RowPairIn in{a.in + (o * a.isO + i0 * a.isI), (int)a.isI};
    SmemOut2<L, LY> so{sm};
    run_stages_in_out<f32x2, L, H, NT, SIGN, LY>(sm, s_tw, in, so);
    __syncthreads();
    float2* out = a.out + (o * a.osO + i0);
    const f32x2 scale(a.scale);
    const int sJ = (int)a.osJ, h = (int)(threadIdx.x % H);
    static_assert(NT % H == 0, "each thread keeps one pencil pair");
#pragma unroll 4
    for (int j = (int)(threadIdx.x / H); j < L; j += NT / H)
        *reinterpret_cast<float4*>(out + (2 * h + j * sJ)) = quad_of(cscale(sm[LY::idx(h, j)], scale));
}

// ---------------------------------------------------------------- x rows of the half-spectrum forms
// fft_nl_half_kernel's transform of two real rows as one complex pencil, with
// two such pencils (four rows) per thread.
template <int L, bool X> struct QuadPackIn {
    static constexpr bool EXT = X;
    const float2* base;   // row 0 of the tile
    int nhp;
    bool r2c;
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int k) const {
        const bool up = k > L / 2;
        const float2* q = base + (4 * p * nhp + (up ? L - k : k));
        float2 a1 = q[0], a2 = q[nhp], b1 = q[2 * nhp], b2 = q[3 * nhp];
        if (r2c && (k == 0 || k == L / 2)) a1.y = a2.y = b1.y = b2.y = 0.f;
        const f32x2 x1(a1.x, b1.x), y1(a1.y, b1.y), x2(a2.x, b2.x), y2(a2.y, b2.y);
        // X1[k] + i X2[k], past N/2 conj(X1[N-k]) + i conj(X2[N-k])
        return up ? mk<cf32x2>(x1 + y2, x2 - y1) : mk<cf32x2>(x1 - y2, y1 + x2);
    }
};
struct ChNlQuadMid {
    f32x2 scale, msum;
    __device__ __forceinline__ void begin(int, int) {}
    __device__ __forceinline__ cf32x2 operator()(int, int, cf32x2 x) {
        const f32x2 c0 = mul_rn(x.x, scale), c1 = mul_rn(x.y, scale);
        msum = msum + (c0 + c1);
        return mk<cf32x2>(fma_rn(mul_rn(c0, c0), c0, -c0), fma_rn(mul_rn(c1, c1), c1, -c1));
    }
};
// Four real rows in: rows 4p .. 4p + 3 as pencils (row, row + 1) of pair p.
struct QuadRealIn {
    static constexpr bool EXT = true;
    const float* base;   // row 0 of the tile, rows of n
    int n;
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const {
        const float* q = base + (4 * p * n + m);
        return mk<cf32x2>(f32x2(q[0], q[2 * n]), f32x2(q[n], q[3 * n]));
    }
};
template <int L> struct QuadRealOut {
    static constexpr bool SYNC = false;
    float* base;
    f32x2 scale;
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        float* q = base + (4 * p * L + j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 w = quad_of(cscale(v[r], scale));
            q[r * (L / R)] = w.x;
            q[r * (L / R) + L] = w.y;
            q[r * (L / R) + 2 * L] = w.z;
            q[r * (L / R) + 3 * L] = w.w;
        }
    }
};

// MODE: PASS_NL_HALF (half rows -> real -> g = c^3 - c -> half rows), PASS_R2C_HALF (real
// rows -> half rows) or PASS_C2R_HALF (half rows -> real rows).
// P real rows per tile, P / 4 pencils of the packed transform.  Measured (rows x
// N2, in place, one thread one pencil before): 65536 x 256 35.3 -> 32.2 us,
// 147456 x 384 233 -> 161 us, 65536 x 128 22.0 -> 18.7 us, 4096 x 64 3.7 -> 2.8 us;
// at 512 points two pencils' registers leave too few threads (95 against 102 us)
// and fft_nl_half_kernel stays.
// ST: the tile's rows are staged in shared memory (the transform then works over
// them); else the packed elements are read from global memory, each row twice.
template <int L, int P, int NT, int OCC, bool ST, int MODE = PASS_NL_HALF>
__global__ void __launch_bounds__(NT, OCC) fft_nl_half2_kernel(PassParams<float> a) {
    pdl_wait();
    constexpr int H = P / 4, M = L / 2;
    using LY = RowLayout<L, H>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    const int NHP = a.hg.NHP;
    const long long q0 = (long long)blockIdx.x * P;
    stage_twiddles<L, NT>(s_tw, a.tw);
    const float2* src = a.in + q0 * NHP;
    float2* rows = reinterpret_cast<float2*>(smem_raw);
    if constexpr (ST && MODE != PASS_R2C_HALF) {
        for (int u = threadIdx.x; u < P * NHP / 2; u += NT) cp_async16(rows + 2 * u, src + 2 * u);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        src = rows;
    }
    QuadPackIn<L, !ST> in{src, NHP, a.hg.r2c != 0};
    ChNlQuadMid mid{f32x2(a.nl_scale), f32x2(0.f)};
    SmemOut2<L, LY> so{sm};
    if constexpr (MODE == PASS_C2R_HALF) {
        QuadRealOut<L> out{reinterpret_cast<float*>(a.out) + q0 * L, f32x2(a.nl_scale)};
        run_stages_in_out<f32x2, L, H, NT, +1, LY>(sm, s_tw, in, out);
        return;
    } else if constexpr (MODE == PASS_R2C_HALF) {
        QuadRealIn rin{reinterpret_cast<const float*>(a.in) + q0 * L, L};
        run_stages_in_out<f32x2, L, H, NT, -1, LY>(sm, s_tw, rin, so);
    } else {
        transform_pair_in<f32x2, L, H, NT, +1, -1, LY>(sm, s_tw, in, mid, so);
    }
    __syncthreads();
    // the two rows' half spectra of each transform: G1[k] = (W[k] + conj W[-k]) / 2,
    // G2[k] = (W[k] - conj W[-k]) / (2i), an entry of four rows an item (padding
    // entries zero).  Two neighbouring entries an item (16-byte stores) would read the
    // tile at every other element, two wavefronts for one.
    float2* dst = a.out + q0 * NHP;
    const f32x2 half(0.5f), nhalf(-0.5f);
    for (int it = threadIdx.x; it < H * NHP; it += NT) {
        const int p = (int)a.hg.fd_NHP.div((uint32_t)it), k = it - p * NHP;
        float2* d = dst + (4 * p * NHP + k);
        if (k > M) {
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i * NHP] = make_float2(0.f, 0.f);
            continue;
        }
        const cf32x2 w = sm[LY::idx(p, k)], v = sm[LY::idx(p, k == 0 ? 0 : L - k)];
        const f32x2 g1x = mul_rn(half, w.x + v.x), g1y = mul_rn(half, w.y - v.y);
        const f32x2 g2x = mul_rn(half, w.y + v.y), g2y = mul_rn(nhalf, w.x - v.x);
        d[0] = make_float2(g1x.lo(), g1y.lo());
        d[NHP] = make_float2(g2x.lo(), g2y.lo());
        d[2 * NHP] = make_float2(g1x.hi(), g1y.hi());
        d[3 * NHP] = make_float2(g2x.hi(), g2y.hi());
    }
    if (a.mass != nullptr) {
        const double ms = warp_sum((double)mid.msum.lo() + (double)mid.msum.hi());
        if ((threadIdx.x & 31) == 0) atomicAdd(a.mass + (q0 / a.mass_ppr) * a.mass_stride, ms);
    }
}

}  // namespace spdba
