// Packed transforms of the reaction-cross-diffusion step (complex64).
//
// The M component fields are real, so two share one complex field: with h_m the
// Hermitian part of u_m, (u_m(k) + conj u_m(-k)) / 2, the inverse transform of
// Z = h_a + i h_b is Re(IFFT(u_a)) + i Re(IFFT(u_b)), and the transform W of
// R_a + i R_b separates into R_a(k) = (W(k) + conj W(-k)) / 2 and R_b(k) = (W(k) -
// conj W(-k)) / (2 i), which the update does as it reads W.  Every pass between the
// two moves half the data, the reaction too.  The two components of a field share the rounding
// of its transforms, relative to the larger one; so do all M in the update, whose product with
// the eigenvectors of D mixes them.  Measured against complex128 over 1, 20 and 100 steps, with every
// other component 1, 1e-3, 1e-6 or 0 of its neighbour (M = 2, 3, 8, 64 x 64 and 32 x 32 x 64, with and
// without cross diffusion), each component's error is that of the M separate transforms; alone
// two components without cross diffusion, one exactly zero, differ: it stays within 3e-12 of the other
// one, 5e-17 before.  The inverse starts with the rows, where
// Z is formed (this file); rows r and -r are needed together, and share a thread.
#include <algorithm>

#include "fft_f32x2.cuh"
#include "rcd.h"

namespace spdba {

// Field rows (kz, ky) with their mirrors (-kz, -ky): representative q of the row
// pairs, q < rcd_row_pairs(N0, N1).  Planes kz = 0 and N0 / 2 mirror onto
// themselves, with rows ky = 0 .. N1 / 2 as representatives.
struct RowPair {
    int d, m;   // row kz * N1 + ky and its mirror
};
__host__ __device__ inline long long rcd_row_pairs(int N0, int N1) {
    const long long self = N0 > 1 ? 2 : 1;
    return self * (N1 / 2 + 1) + (N0 > 1 ? (long long)(N0 / 2 - 1) * N1 : 0);
}
__device__ __forceinline__ RowPair rcd_row_pair(int q, int N0, int N1) {
    const int h = N1 / 2 + 1, self = N0 > 1 ? 2 : 1;
    int kz, ky;
    if (q < self * h) {
        kz = q < h ? 0 : N0 / 2;
        ky = q < h ? q : q - h;
    } else {
        q -= self * h;
        kz = 1 + q / N1;
        ky = q - (kz - 1) * N1;
    }
    const int mz = kz == 0 ? 0 : N0 - kz, my = ky == 0 ? 0 : N1 - ky;
    return RowPair{kz * N1 + ky, mz * N1 + my};
}

// Packed element m of row pair p: Z at (row d, m) and (row m, m) from the staged
// rows a_d, b_d, a_m, b_m (the transform works over them once its inputs are in
// registers).
template <int L> struct RcdPackIn {
    static constexpr bool EXT = false;
    const float2* rows;   // pair p: four rows of L
    __device__ __forceinline__ void before_write() const {}
    __device__ __forceinline__ cf32x2 operator()(int p, int m) const {
        const float2* q = rows + 4 * p * L;
        const int mm = m == 0 ? 0 : L - m;
        const float2 ad = q[m], bd = q[L + m], am = q[2 * L + m], bm = q[3 * L + m];
        const float2 adr = q[mm], bdr = q[L + mm], amr = q[2 * L + mm], bmr = q[3 * L + mm];
        // a + i b at k, conj a + i conj b at -k
        const f32x2 x = (f32x2(ad.x, am.x) - f32x2(bd.y, bm.y)) + (f32x2(amr.x, adr.x) + f32x2(bmr.y, bdr.y));
        const f32x2 y = (f32x2(ad.y, am.y) + f32x2(bd.x, bm.x)) + (f32x2(bmr.x, bdr.x) - f32x2(amr.y, adr.y));
        const f32x2 half(0.5f);
        return mk<cf32x2>(mul_rn(half, x), mul_rn(half, y));
    }
};
template <int L, int H> struct RcdPackOut {
    static constexpr bool SYNC = false;
    float2* field;        // the packed field
    const RowPair* pr;    // shared: the tile's row pairs (d < 0: none)
    __device__ __forceinline__ void pre() {}
    __device__ __forceinline__ void begin(int, int, int) {}
    template <int R> __device__ __forceinline__ void emit(int, int p, int j, cf32x2 (&v)[R]) {
        const RowPair q = pr[p];
        if (q.d < 0) return;
        float2* d = field + (long long)q.d * L + j;
        float2* m = field + (long long)q.m * L + j;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 w = quad_of(v[r]);
            d[r * (L / R)] = make_float2(w.x, w.y);
            if (q.m != q.d) m[r * (L / R)] = make_float2(w.z, w.w);
        }
    }
};

// First inverse pass (along the rows) of every packed field: H row pairs of one
// field per CTA.  HBM bounds it: M fields read, M / 2 written.
template <int L, int H, int NT, int OCC>
__global__ void __launch_bounds__(NT, OCC)
    rcd_pack_rows_kernel(const float2* __restrict__ u, float2* __restrict__ z, int M, int N0, int N1, int npairs,
                         int tiles, FastDiv fd_tiles, const float2* __restrict__ tw) {
    pdl_wait();
    using LY = RowLayout<L, H>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* const rows = reinterpret_cast<float2*>(smem_raw);           // 4 H rows
    cf32x2* const sm = reinterpret_cast<cf32x2*>(smem_raw);
    __shared__ float2 s_tw[L];
    __shared__ RowPair s_pr[H];
    const int c = (int)fd_tiles.div(blockIdx.x), q0 = ((int)blockIdx.x - c * tiles) * H;
    const long long n = (long long)N0 * N1 * L;
    const float2* a = u + (long long)(2 * c) * n;
    const bool pair = 2 * c + 1 < M;   // an odd last component stands alone
    if (threadIdx.x < H)
        s_pr[threadIdx.x] = q0 + (int)threadIdx.x < npairs ? rcd_row_pair(q0 + threadIdx.x, N0, N1) : RowPair{-1, -1};
    stage_twiddles<L, NT>(s_tw, tw);
    __syncthreads();
    constexpr int U = L / 2;   // 16-byte units per row
    for (int w = threadIdx.x; w < 4 * H * U; w += NT) {
        const int r = w / U, e = (w % U) * 2;
        const RowPair q = s_pr[r >> 2];
        float2* dst = rows + r * L + e;
        if (q.d < 0 || ((r & 1) && !pair)) {
            *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            cp_async16(dst, a + ((r & 1) ? n : 0) + (long long)((r & 2) ? q.m : q.d) * L + e);
        }
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    RcdPackIn<L> in{rows};
    RcdPackOut<L, H> out{z + (long long)c * n, s_pr};
    run_stages_in_out<f32x2, L, H, NT, +1, LY>(sm, s_tw, in, out);
}

// Reaction on packed fields: u_{2c} = Re, u_{2c+1} = Im in, (R_{2c}, R_{2c+1}) out.
// scale: 1 / N of the inverse transform.
constexpr int RCD_PRX_NT = 256;
__global__ void __launch_bounds__(RCD_PRX_NT) rcd_reaction_packed_kernel(float2* __restrict__ w, long long n, int M,
                                                                         float scale, float r, float a, float alpha,
                                                                         float beta) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* su = reinterpret_cast<float*>(smem_raw);
    const int tid = threadIdx.x, Mh = (M + 1) / 2;
    for (long long x = (long long)blockIdx.x * blockDim.x + tid; x < n; x += (long long)gridDim.x * blockDim.x) {
        float S = 0.f;
#pragma unroll 4
        for (int c = 0; c < Mh; ++c) {
            const float2 v = w[(long long)c * n + x];
            const float v0 = mul_rn(v.x, scale), v1 = 2 * c + 1 < M ? mul_rn(v.y, scale) : 0.f;
            su[2 * c * RCD_PRX_NT + tid] = v0;
            su[(2 * c + 1) * RCD_PRX_NT + tid] = v1;
            S += v0;
            S += v1;
        }
        auto react = [&](int m) {
            const float um = su[m * RCD_PRX_NT + tid];
            float inter;
            if (M >= 3) {
                const float prev = su[(m == 0 ? M - 1 : m - 1) * RCD_PRX_NT + tid];
                const float next = su[(m + 1 == M ? 0 : m + 1) * RCD_PRX_NT + tid];
                inter = beta * (S - um) + alpha * (prev + next);
            } else {
                inter = (beta + alpha) * (S - um);
            }
            return um * (r - a * um - inter);
        };
#pragma unroll 4
        for (int c = 0; c < Mh; ++c)
            w[(long long)c * n + x] = make_float2(react(2 * c), 2 * c + 1 < M ? react(2 * c + 1) : 0.f);
    }
}

// Rows (kz, ky) whose packed transform the update of non-frozen blocks reads (their
// own blocks or those of the mirrored row), and planes kz with such rows.  One CTA
// per plane.
__global__ void __launch_bounds__(256) rcd_live_kernel(Geom g, const uint8_t* __restrict__ states,
                                                       uint8_t* __restrict__ row_live,
                                                       uint8_t* __restrict__ plane_live) {
    pdl_wait();
    const int N0 = (int)g.n[0], N1 = (int)g.n[1], nb1 = (int)g.nb[1], nb2 = (int)g.nb[2];
    const int kz = blockIdx.x, mz = kz == 0 ? 0 : N0 - kz;
    const uint8_t* sd = states + (long long)(kz / g.b[0]) * nb1 * nb2;
    const uint8_t* sm = states + (long long)(mz / g.b[0]) * nb1 * nb2;
    int any = 0;
    for (int ky = threadIdx.x; ky < N1; ky += blockDim.x) {
        const int my = ky == 0 ? 0 : N1 - ky;
        unsigned live = 0;
        for (int bx = 0; bx < nb2; ++bx) live |= sd[(ky / g.b[1]) * nb2 + bx] | sm[(my / g.b[1]) * nb2 + bx];
        row_live[(long long)kz * N1 + ky] = live != 0;
        any |= live != 0;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) plane_live[kz] = any != 0;
}

// ------------------------------------------------------------------ host
namespace {
template <int L, int H, int NT, int OCC> void pack_info(RcdPack* o) {
    o->H = H;
    o->nt = NT;
    o->smem = std::max(4 * H * L * (int)sizeof(float2), RowLayout<L, H>::SIZE * (int)sizeof(cf32x2));
    o->func = (const void*)rcd_pack_rows_kernel<L, H, NT, OCC>;
}
}  // namespace

spdba_status rcd_pack_prepare(RcdPack* o, int ndim, const int64_t* d, int M, TwiddleCache<float>& tw, cudaStream_t st) {
    o->ok = false;
    const int64_t L = d[ndim - 1];
    const int N0 = ndim == 3 ? (int)d[0] : 1, N1 = (int)d[ndim - 2];
    // one component has nothing to share a field with
    if (M < 2 || N1 % 2 != 0 || (N0 > 1 && N0 % 2 != 0)) return SPDBA_OK;
    switch (L) {
        case 32: pack_info<32, 16, 64, 8>(o); break;
        case 64: pack_info<64, 8, 64, 8>(o); break;
        case 128: pack_info<128, 8, 64, 6>(o); break;
        case 256: pack_info<256, 4, 64, 6>(o); break;
        default: return SPDBA_OK;   // no packing kernel is built for other rows: they keep the M transforms
    }
    // at most 34 KB; the whole carveout, so that as many CTAs fit as the registers allow
    SPDBA_CUDA(cudaFuncSetAttribute(o->func, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    const int smem = 2 * ((M + 1) / 2) * RCD_PRX_NT * (int)sizeof(float);
    if (smem > 48 * 1024)
        SPDBA_CUDA(cudaFuncSetAttribute((const void*)rcd_reaction_packed_kernel,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        kRcdMaxComponents * RCD_PRX_NT * (int)sizeof(float)));
    spdba_status s = SPDBA_OK;
    if (!(o->tw = tw.get(L, st, &s))) return s;
    o->M = M;
    o->Mh = (M + 1) / 2;
    o->N0 = N0;
    o->N1 = N1;
    o->n = (long long)N0 * N1 * L;
    o->npairs = (int)rcd_row_pairs(N0, N1);
    o->tiles = (o->npairs + o->H - 1) / o->H;
    o->fd_tiles.init((uint32_t)o->tiles);
    o->ok = true;
    return SPDBA_OK;
}

spdba_status launch_rcd_pack(const RcdPack& o, const float2* u, float2* z, cudaStream_t st) {
    int M = o.M, N0 = o.N0, N1 = o.N1, np = o.npairs, tiles = o.tiles;
    FastDiv fd = o.fd_tiles;
    const float2* tw = o.tw;
    void* args[] = {&u, &z, &M, &N0, &N1, &np, &tiles, &fd, &tw};
    SPDBA_CUDA(pdl_launch_ptr(o.func, dim3((unsigned)(tiles * o.Mh)), dim3(o.nt), args, (size_t)o.smem, st));
    return SPDBA_OK;
}

spdba_status launch_rcd_reaction_packed(const RcdPack& o, float2* z, float r, float a, float alpha, float beta,
                                        cudaStream_t st) {
    const int smem = 2 * o.Mh * RCD_PRX_NT * (int)sizeof(float);
    long long grid = (o.n + RCD_PRX_NT - 1) / RCD_PRX_NT;
    if (grid > 152 * 8) grid = 152 * 8;
    pdl_launch(rcd_reaction_packed_kernel, (unsigned)grid, RCD_PRX_NT, smem, st, z, o.n, o.M,
               (float)(1.0 / (double)o.n), r, a, alpha, beta);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

spdba_status launch_rcd_live(const Geom& g, const uint8_t* states, uint8_t* row_live, uint8_t* plane_live,
                             cudaStream_t st) {
    pdl_launch(rcd_live_kernel, (unsigned)g.n[0], 256, 0, st, g, states, row_live, plane_live);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

}  // namespace spdba
