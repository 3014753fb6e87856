// Learned block-activity predictor (no counterpart in the paper): a small 3-D
// convolutional network over the block map that predicts which blocks will be
// non-frozen over the next K steps, so that most exact activity scans can be
// skipped (the exact scan stays as a periodic judge).
//
//   a1 = conv(x, W1) + b1, h1 = relu(a1)    2 -> 8 channels, 3x3x3, periodic
//   a2 = conv(h1, W2) + b2, h2 = relu(a2)   8 -> 16
//   a3 = conv(h2, W3) + b3, h3 = relu(a3)   16 -> 8
//   z = h3 . wh + bh, p = sigmoid(z);  loss = mean BCE(p, y)
//
// Convolutions are implicit GEMMs on the BF16 tensor cores (mma.sync m16n8k16,
// FP32 accumulate): forward and input-gradient use M = voxels, N = output
// channels, K = 27 x input channels; the weight gradient uses M = output
// channels, N = 27 x input channels, K = voxels.  Activations are channels-
// last, stored as BF16 between layers; master weights and Adam state are FP32.
// The GEMM shapes are tiny (N = 8 or 16), so these kernels are latency-bound; a
// CTA works on a voxel tile staged with its halo in shared memory.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "blocks.h"

namespace spdba {

typedef __nv_bfloat16 bf16;

constexpr int NPARAM = 8 * 27 * 2 + 8 + 16 * 27 * 8 + 16 + 8 * 27 * 16 + 8 + 8 + 1;
// offsets of the flat parameter vector: W1, b1, W2, b2, W3, b3, wh, bh
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + 8 * 27 * 2, OFF_W2 = OFF_B1 + 8, OFF_B2 = OFF_W2 + 16 * 27 * 8,
              OFF_W3 = OFF_B2 + 16, OFF_B3 = OFF_W3 + 8 * 27 * 16, OFF_WH = OFF_B3 + 8, OFF_BH = OFF_WH + 8;
static_assert(OFF_BH + 1 == NPARAM, "parameter layout");

__host__ __device__ constexpr int kpad(int k) { return (k + 15) / 16 * 16; }

struct MapDims {
    int D, H, W;
    long long V;  // voxels per map
};

__device__ __forceinline__ uint32_t ld_pair(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ------------------------------------------------------------------ voxel tiles
// A CTA works on a tile of kTZ x kTY x kTX voxels of one map; the tile and its
// periodic halo are staged in shared memory once (648 voxels for 256), so that
// the 27 taps of a voxel are shared-memory reads at compile-time offsets.  One
// MMA row block is the 16 voxels of a tile row along x.  Gathering each tap
// from global memory instead cost three 64-bit divisions per lane and tap, which
// bound every kernel here: one inference and one gradient over two 48^3 maps
// took 4.49 ms, and 0.255 ms with the tiles.
constexpr int kTX = 16, kTY = 4, kTZ = 4;
constexpr int kHX = kTX + 2, kHY = kTY + 2, kHZ = kTZ + 2;
constexpr int kHalo = kHX * kHY * kHZ;
constexpr int kRows = kTY * kTZ;   // 16-voxel rows of a tile

// Channels a voxel takes in shared memory: 16 channels are padded to 48 bytes,
// so that the eight 16-byte rows of an 8x8 ldmatrix start in distinct banks
// (16-byte voxels of 8 channels do so unpadded).
template <int C> struct VoxStride { static constexpr int value = C == 16 ? 24 : C; };

__host__ __device__ constexpr int tap_off(int tap) {
    return ((tap / 9 - 1) * kHY + (tap / 3 % 3 - 1)) * kHX + (tap % 3 - 1);
}
__host__ __device__ constexpr int row_base(int r) { return ((r / kTY + 1) * kHY + (r % kTY + 1)) * kHX + 1; }

struct TilePos {
    int z0, y0, x0;
    long long base;   // first voxel of the tile's map
};
struct TileGrid {
    int tx, ty, tz;
    long long tiles;  // over all maps
};
static TileGrid tile_grid(const MapDims& m, int nmaps) {
    TileGrid t{(m.W + kTX - 1) / kTX, (m.H + kTY - 1) / kTY, (m.D + kTZ - 1) / kTZ, 0};
    t.tiles = (long long)t.tx * t.ty * t.tz * nmaps;
    return t;
}
__device__ __forceinline__ TilePos tile_pos(const MapDims& m, const TileGrid& t, long long tile) {
    TilePos p;
    long long q = tile / t.tx;
    p.x0 = (int)(tile - q * t.tx) * kTX;
    long long q2 = q / t.ty;
    p.y0 = (int)(q - q2 * t.ty) * kTY;
    const long long mp = q2 / t.tz;
    p.z0 = (int)(q2 - mp * t.tz) * kTZ;
    p.base = mp * m.V;
    return p;
}
__device__ __forceinline__ int wrap(int c, int n) {
    c %= n;
    return c < 0 ? c + n : c;
}

// Tile and halo of X into shared memory (periodic; positions past the map in a
// ragged tile hold wrapped voxels, which no stored result depends on).
template <int C> __device__ __forceinline__ void stage_halo(bf16* sX, const bf16* __restrict__ X, const MapDims& m,
                                                            const TilePos& p) {
    for (int i = threadIdx.x; i < kHalo; i += blockDim.x) {
        const int hx = i % kHX, q = i / kHX, hy = q % kHY, hz = q / kHY;
        const int z = wrap(p.z0 + hz - 1, m.D), y = wrap(p.y0 + hy - 1, m.H), x = wrap(p.x0 + hx - 1, m.W);
        const bf16* src = X + (p.base + ((long long)z * m.H + y) * m.W + x) * C;
        bf16* dst = sX + i * VoxStride<C>::value;
        if constexpr (C == 2) {
            *reinterpret_cast<uint32_t*>(dst) = ld_pair(src);
        } else {
#pragma unroll
            for (int c = 0; c < C; c += 8)
                *reinterpret_cast<uint4*>(dst + c) = *reinterpret_cast<const uint4*>(src + c);
        }
    }
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t& r0, uint32_t& r1, const bf16* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(r0), "=r"(r1) : "r"(a) : "memory");
}

// ------------------------------------------------------------------ conv (forward / input gradient)
enum ConvMode { CONV_FWD = 0, CONV_DGRAD = 1 };

// One tile per CTA, four rows of 16 voxels per warp.  Wt: [COUT][kpad(27 CIN)]
// bf16 (zero padded); a warp keeps all its weight fragments in registers (54 to
// 56 of them at most) for its four rows.
// FWD: out_pre = acc + bias (FP32; left out when null), out = bf16(relu(.)).
// DGRAD: out = bf16(acc * (mask_pre > 0)).
template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(128) conv_kernel(MapDims m, TileGrid tg, const bf16* __restrict__ X,
                                                   const bf16* __restrict__ Wt, const float* __restrict__ bias,
                                                   float* __restrict__ out_pre, const float* __restrict__ mask_pre,
                                                   bf16* __restrict__ out) {
    pdl_wait();
    constexpr int K = 27 * CIN, KP = kpad(K), NT = COUT / 8, KC = KP / 16, VS = VoxStride<CIN>::value;
    __shared__ __align__(16) bf16 sX[kHalo * VS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const TilePos p = tile_pos(m, tg, blockIdx.x);
    stage_halo<CIN>(sX, X, m, p);
    uint32_t b[KC][NT][2];
#pragma unroll
    for (int kc = 0; kc < KC; ++kc)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const bf16* wr = Wt + (n * 8 + g) * KP + kc * 16 + 2 * t;
            b[kc][n][0] = ld_pair(wr);
            b[kc][n][1] = ld_pair(wr + 8);
        }
    // CIN = 2: this lane's taps of each chunk (columns 2t and 2t + 8)
    int off2[CIN == 2 ? KC : 1][2];
    if constexpr (CIN == 2) {
#pragma unroll
        for (int kc = 0; kc < KC; ++kc)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int tap = kc * 8 + 4 * h + t;
                off2[kc][h] = tap < 27 ? tap_off(tap) : -(1 << 20);
            }
    }
    __syncthreads();
    const int lrow = (lane & 7) + ((lane >> 3) & 1) * 8;   // ldmatrix: this lane's row address
#pragma unroll 1
    for (int rr = 0; rr < kRows / 4; ++rr) {
        const int r = warp * (kRows / 4) + rr;
        const int vb = row_base(r);
        float acc[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
        for (int kc = 0; kc < KC; ++kc) {
            uint32_t a[4];
            if constexpr (CIN == 16) {
                ldsm4(a, sX + (vb + lrow + tap_off(kc)) * VS + (lane >> 4) * 8);
            } else if constexpr (CIN == 8) {
                // two taps per chunk; the chunk past the last tap multiplies zero weights
                const int o0 = tap_off(2 * kc), o1 = 2 * kc + 1 < 27 ? tap_off(2 * kc + 1) : o0;
                ldsm4(a, sX + (vb + lrow + (lane < 16 ? o0 : o1)) * VS);
                if (2 * kc + 1 >= 27) a[2] = a[3] = 0u;
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int o = off2[kc][h];
                    const bool ok = o > -(1 << 20);
                    a[2 * h] = ok ? ld_pair(sX + (vb + g + o) * VS) : 0u;
                    a[2 * h + 1] = ok ? ld_pair(sX + (vb + g + 8 + o) * VS) : 0u;
                }
            }
#pragma unroll
            for (int n = 0; n < NT; ++n) mma16816(acc[n], a[0], a[1], a[2], a[3], b[kc][n][0], b[kc][n][1]);
        }
        // D: voxels x0 + g and x0 + g + 8 of the row, columns co = n*8 + 2t, +1
        const int z = p.z0 + r / kTY, y = p.y0 + r % kTY;
        if (z >= m.D || y >= m.H) continue;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int co = n * 8 + 2 * t;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int x = p.x0 + g + 8 * h;
                if (x >= m.W) continue;
                const long long v = p.base + ((long long)z * m.H + y) * m.W + x;
                float x0 = acc[n][2 * h], x1 = acc[n][2 * h + 1];
                if (MODE == CONV_FWD) {
                    x0 += bias[co];
                    x1 += bias[co + 1];
                    if (out_pre) *reinterpret_cast<float2*>(out_pre + v * COUT + co) = make_float2(x0, x1);
                    x0 = fmaxf(x0, 0.f);
                    x1 = fmaxf(x1, 0.f);
                } else {
                    const float2 mp = *reinterpret_cast<const float2*>(mask_pre + v * COUT + co);
                    if (!(mp.x > 0.f)) x0 = 0.f;
                    if (!(mp.y > 0.f)) x1 = 0.f;
                }
                *reinterpret_cast<uint32_t*>(out + v * COUT + co) =
                    pack2(__float2bfloat16_rn(x0), __float2bfloat16_rn(x1));
            }
        }
    }
}

// ------------------------------------------------------------------ weight gradient
// dW[co][k] += sum_v dA[v][co] X[neighbour(v, tap(k))][ci(k)], k < 27 CIN, on
// the tensor cores: A = dA^T (rows co, padded to 16), B = im2col(X) (rows =
// voxels, columns = 8 k), reduction over the 16 voxels of a row per mma.  CTAs
// walk the tiles in a fixed stride; warp w owns taps 3w .. 3w + 2 (CIN = 2: the
// column tile w of the seven) and keeps their sums in registers over all its
// CTA's tiles, then adds them into dW.  Both fragments come transposed out of
// voxel-major shared memory (ldmatrix.trans).
constexpr int kWgNT = 288;
template <int CIN, int COUT>
__global__ void __launch_bounds__(kWgNT) wgrad_kernel(MapDims m, TileGrid tg, const bf16* __restrict__ dA,
                                                      const bf16* __restrict__ X, float* __restrict__ dW,
                                                      float* __restrict__ dbias) {
    pdl_wait();
    constexpr int K = 27 * CIN, VS = VoxStride<CIN>::value, DS = VoxStride<COUT>::value;
    constexpr int NACC = CIN == 2 ? 1 : 3 * CIN / 8;
    __shared__ __align__(16) bf16 sX[kHalo * VS];
    __shared__ __align__(16) bf16 sD[kRows * kTX * DS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    float acc[NACC][4];
#pragma unroll
    for (int n = 0; n < NACC; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
    float bsum0 = 0.f, bsum1 = 0.f;   // bias gradient of channel g (and g + 8), warp 0
    int off = 0;                       // CIN = 2: this lane's column's tap
    if constexpr (CIN == 2) {
        const int tap = (warp * 8 + g) / 2;
        off = tap < 27 ? tap_off(tap) : 0;
    }
    for (long long tile = blockIdx.x; tile < tg.tiles; tile += gridDim.x) {
        const TilePos p = tile_pos(m, tg, tile);
        __syncthreads();   // the previous tile's reads are done
        stage_halo<CIN>(sX, X, m, p);
        for (int i = threadIdx.x; i < kRows * kTX; i += kWgNT) {
            const int x = p.x0 + i % kTX, r = i / kTX, y = p.y0 + r % kTY, z = p.z0 + r / kTY;
            const bool ok = x < m.W && y < m.H && z < m.D;   // voxels past the map add nothing
            const bf16* src = dA + (p.base + ((long long)z * m.H + y) * m.W + x) * COUT;
#pragma unroll
            for (int c = 0; c < COUT; c += 8)
                *reinterpret_cast<uint4*>(sD + i * DS + c) =
                    ok ? *reinterpret_cast<const uint4*>(src + c) : make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
        if (CIN == 2 && warp >= 7) continue;
#pragma unroll 2
        for (int r = 0; r < kRows; ++r) {
            if (p.z0 + r / kTY >= m.D || p.y0 + r % kTY >= m.H) continue;   // warp-uniform
            const bf16* drow = sD + r * kTX * DS;
            uint32_t a[4] = {0u, 0u, 0u, 0u};
            if constexpr (COUT == 16)
                ldsm4t(a, drow + ((lane & 7) + (lane >> 4) * 8) * DS + ((lane >> 3) & 1) * 8);
            else
                ldsm2t(a[0], a[2], drow + (lane & 15) * DS);
            if (warp == 0) {
                auto two = [](uint32_t u) {
                    return __uint_as_float(u << 16) + __uint_as_float(u & 0xffff0000u);
                };
                bsum0 += two(a[0]) + two(a[2]);
                bsum1 += two(a[1]) + two(a[3]);
            }
            const int vb = row_base(r);
            if constexpr (CIN == 2) {
                const bf16* c = sX + (vb + off + 2 * t) * 2 + (g & 1);
                mma16816(acc[0], a[0], a[1], a[2], a[3], pack2(c[0], c[2]), pack2(c[16], c[18]));
            } else {
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    // taps 3 warp + j: dx = j - 1, (dz, dy) from the warp
                    const int o = ((warp / 3 - 1) * kHY + (warp % 3 - 1)) * kHX + (j - 1);
                    if constexpr (CIN == 16) {
                        uint32_t bb[4];
                        ldsm4t(bb, sX + (vb + o + (lane & 15)) * VS + (lane >> 4) * 8);
                        mma16816(acc[2 * j], a[0], a[1], a[2], a[3], bb[0], bb[1]);
                        mma16816(acc[2 * j + 1], a[0], a[1], a[2], a[3], bb[2], bb[3]);
                    } else {
                        uint32_t b0, b1;
                        ldsm2t(b0, b1, sX + (vb + o + (lane & 15)) * VS);
                        mma16816(acc[j], a[0], a[1], a[2], a[3], b0, b1);
                    }
                }
            }
        }
    }
    if (CIN == 2 && warp >= 7) return;
#pragma unroll
    for (int n = 0; n < NACC; ++n) {
        const int kc = (CIN == 2 ? warp * 8 : warp * 3 * CIN + n * 8) + 2 * t;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int co = g + 8 * h;
            if (co >= COUT) continue;
            if (kc < K) atomicAdd(&dW[co * K + kc], acc[n][2 * h]);
            if (kc + 1 < K) atomicAdd(&dW[co * K + kc + 1], acc[n][2 * h + 1]);
        }
    }
    if (warp == 0) {
        // lanes with equal g hold partial sums of the same channel
        bsum0 += __shfl_xor_sync(0xffffffffu, bsum0, 1);
        bsum0 += __shfl_xor_sync(0xffffffffu, bsum0, 2);
        bsum1 += __shfl_xor_sync(0xffffffffu, bsum1, 1);
        bsum1 += __shfl_xor_sync(0xffffffffu, bsum1, 2);
        if (t == 0) {
            atomicAdd(&dbias[g], bsum0);
            if (g + 8 < COUT) atomicAdd(&dbias[g + 8], bsum1);
        }
    }
}

// ------------------------------------------------------------------ head, loss and its gradient
// z = h3 . wh + bh, p = sigmoid(z).  With labels: loss += BCE / n, dz = (p - y) / n,
// dwh += dz h3, dbh += dz, da3 = bf16(dz wh * (a3 > 0)).
// The sums of a CTA are combined in shared memory first, so that each of the ten
// addresses sees one atomic per CTA (one per warp queued on them: 46 us for two
// 48^3 maps).
constexpr int kHeadNT = 256;
__global__ void __launch_bounds__(kHeadNT) head_kernel(long long nvox, const bf16* __restrict__ h3,
                                                       const float* __restrict__ a3,
                                                       const float* __restrict__ params, float* __restrict__ prob,
                                                       const float* __restrict__ labels, double inv_n,
                                                       bf16* __restrict__ da3, float* __restrict__ grads,
                                                       double* __restrict__ loss) {
    pdl_wait();
    const float* wh = params + OFF_WH;
    const float bh = params[OFF_BH];
    float gw[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    float gb = 0.f;
    double ls = 0.0;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < nvox;
         v += (long long)gridDim.x * blockDim.x) {
        const uint4 hq = *reinterpret_cast<const uint4*>(h3 + v * 8);
        const uint32_t hw[4] = {hq.x, hq.y, hq.z, hq.w};
        float hv[8];
        float z = bh;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            hv[c] = __uint_as_float(c & 1 ? hw[c / 2] & 0xffff0000u : hw[c / 2] << 16);
            z = fmaf(hv[c], wh[c], z);
        }
        const float p = 1.f / (1.f + expf(-z));
        if (prob) prob[v] = p;
        if (labels) {
            const float y = labels[v];
            const float eps = 1e-12f;
            ls -= (double)(y * logf(p + eps) + (1.f - y) * logf(1.f - p + eps));
            const float dz = (float)((double)(p - y) * inv_n);
            gb += dz;
            float av[8];
            *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(a3 + v * 8);
            *reinterpret_cast<float4*>(av + 4) = *reinterpret_cast<const float4*>(a3 + v * 8 + 4);
            uint32_t dw[4];
#pragma unroll
            for (int c = 0; c < 8; c += 2) {
                gw[c] = fmaf(dz, hv[c], gw[c]);
                gw[c + 1] = fmaf(dz, hv[c + 1], gw[c + 1]);
                const float d0 = av[c] > 0.f ? dz * wh[c] : 0.f, d1 = av[c + 1] > 0.f ? dz * wh[c + 1] : 0.f;
                dw[c / 2] = pack2(__float2bfloat16_rn(d0), __float2bfloat16_rn(d1));
            }
            *reinterpret_cast<uint4*>(da3 + v * 8) = make_uint4(dw[0], dw[1], dw[2], dw[3]);
        }
    }
    if (!labels) return;
    __shared__ float s_g[9][kHeadNT / 32];
    __shared__ double s_l[kHeadNT / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < 8; ++c) gw[c] = warp_sumf(gw[c]);
    gb = warp_sumf(gb);
    ls = warp_sum(ls);
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < 8; ++c) s_g[c][warp] = gw[c];
        s_g[8][warp] = gb;
        s_l[warp] = ls;
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        float t = 0.f;
        for (int w = 0; w < kHeadNT / 32; ++w) t += s_g[threadIdx.x][w];
        atomicAdd(&grads[OFF_WH + threadIdx.x], t);   // the bias follows the eight weights
    } else if (threadIdx.x == 9) {
        double t = 0.0;
        for (int w = 0; w < kHeadNT / 32; ++w) t += s_l[w];
        atomicAdd(loss, t * inv_n);
    }
}

// ------------------------------------------------------------------ weights, features, Adam
// FP32 master -> BF16 forward layout Wt[co][k] (k = tap*CIN + ci, zero padded) and
// input-gradient layout Wd[ci][k'] (k' = tap'*COUT + co, tap' = 26 - tap).
__global__ void convert_weights_kernel(const float* __restrict__ P, int off, int cin, int cout, bf16* __restrict__ Wt,
                                       bf16* __restrict__ Wd) {
    pdl_wait();
    const int K = 27 * cin, KP = kpad(K), Kd = 27 * cout, KPd = kpad(Kd);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cout * KP; i += gridDim.x * blockDim.x) {
        int co = i / KP, k = i % KP;
        Wt[i] = __float2bfloat16_rn(k < K ? P[off + co * K + k] : 0.f);
    }
    if (!Wd) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cin * KPd; i += gridDim.x * blockDim.x) {
        int ci = i / KPd, k = i % KPd;
        float w = 0.f;
        if (k < Kd) {
            int tapd = k / cout, co = k % cout;
            int tap = 26 - tapd;
            w = P[off + co * K + tap * cin + ci];
        }
        Wd[i] = __float2bfloat16_rn(w);
    }
}

// x[v][0] = clamp(log10(A_B / tau) / 8, -1, 1), x[v][1] = 1 if the block is not FROZEN.
__global__ void features_kernel(long long V, int nmaps, const double* __restrict__ maxsq, const double* __restrict__ tau,
                                const uint8_t* __restrict__ states, bf16* __restrict__ x) {
    pdl_wait();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < V * nmaps;
         i += (long long)gridDim.x * blockDim.x) {
        const long long mp = i / V;
        const double a = sqrt(maxsq[i]);
        const double tv = tau[mp];
        double f = (a > 0 && tv > 0) ? log10(a / tv) / 8.0 : (a > 0 ? 1.0 : -1.0);
        f = f < -1.0 ? -1.0 : (f > 1.0 ? 1.0 : f);
        x[2 * i] = __float2bfloat16_rn((float)f);
        x[2 * i + 1] = __float2bfloat16_rn(states[i] != 0 ? 1.f : 0.f);
    }
}

__global__ void adam_kernel(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ M,
                            float* __restrict__ Vv, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    pdl_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float g = G[i];
        float m = b1 * M[i] + (1.f - b1) * g;
        float v = b2 * Vv[i] + (1.f - b2) * g * g;
        M[i] = m;
        Vv[i] = v;
        P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    }
}

__global__ void prob_to_measure_kernel(const float* __restrict__ p, double* __restrict__ out, long long n) {
    pdl_wait();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = (double)p[i];
}

}  // namespace spdba

using namespace spdba;

struct spdba_predictor {
    MapDims m;
    int max_batch;
    float *P, *G, *M, *Vv, *prob, *a1, *a2, *a3, *labels;
    bf16 *W1t, *W2t, *W3t, *W2d, *W3d, *h1, *h2, *h3, *da1, *da2, *da3;
    double* loss;
    long long adam_t;
    std::vector<void*> allocs;
    template <typename Q> spdba_status alloc(Q** p, size_t bytes) {
        void* q = nullptr;
        cudaError_t e = spdba::dev_alloc(&q, bytes);
        if (e != cudaSuccess) return cuda_fail(e, "device allocation (predictor buffer)");
        allocs.push_back(q);
        *p = (Q*)q;
        return SPDBA_OK;
    }
};

namespace spdba {

static unsigned grid_of(long long n, int nt) {
    long long g = (n + nt - 1) / nt;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)(g < 1 ? 1 : g);
}

static spdba_status refresh_weights(spdba_predictor* pr, cudaStream_t st) {
    pdl_launch(convert_weights_kernel, 32, 256, 0, st, pr->P, OFF_W1, 2, 8, pr->W1t, nullptr);
    pdl_launch(convert_weights_kernel, 32, 256, 0, st, pr->P, OFF_W2, 8, 16, pr->W2t, pr->W2d);
    pdl_launch(convert_weights_kernel, 32, 256, 0, st, pr->P, OFF_W3, 16, 8, pr->W3t, pr->W3d);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

// keep_pre: the pre-activations are stored too (the backward pass reads their signs).
static spdba_status forward(spdba_predictor* pr, const bf16* x, int nmaps, bool keep_pre, cudaStream_t st) {
    const TileGrid tg = tile_grid(pr->m, nmaps);
    const unsigned g = (unsigned)tg.tiles;
    pdl_launch(conv_kernel<2, 8, CONV_FWD>, g, 128, 0, st, pr->m, tg, x, pr->W1t, pr->P + OFF_B1,
                                                   keep_pre ? pr->a1 : nullptr, nullptr, pr->h1);
    pdl_launch(conv_kernel<8, 16, CONV_FWD>, g, 128, 0, st, pr->m, tg, pr->h1, pr->W2t, pr->P + OFF_B2,
                                                    keep_pre ? pr->a2 : nullptr, nullptr, pr->h2);
    pdl_launch(conv_kernel<16, 8, CONV_FWD>, g, 128, 0, st, pr->m, tg, pr->h2, pr->W3t, pr->P + OFF_B3,
                                                    keep_pre ? pr->a3 : nullptr, nullptr, pr->h3);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

static unsigned head_grid(long long nvox) { return std::min(grid_of(nvox, kHeadNT), 152u * 4u); }

template <int CIN, int COUT>
static void wgrad(spdba_predictor* pr, const TileGrid& tg, const bf16* dA, const bf16* X, int offW, int offB,
                  cudaStream_t st) {
    const unsigned g = (unsigned)std::min<long long>(tg.tiles, 152 * 3);
    pdl_launch(wgrad_kernel<CIN, COUT>, g, kWgNT, 0, st, pr->m, tg, dA, X, pr->G + offW, pr->G + offB);
}

static spdba_status backward(spdba_predictor* pr, const bf16* x, const float* labels, int nmaps, cudaStream_t st) {
    const long long nvox = pr->m.V * nmaps;
    const TileGrid tg = tile_grid(pr->m, nmaps);
    const unsigned g = (unsigned)tg.tiles;
    SPDBA_CUDA(cudaMemsetAsync(pr->G, 0, sizeof(float) * NPARAM, st));
    SPDBA_CUDA(cudaMemsetAsync(pr->loss, 0, sizeof(double), st));
    pdl_launch(head_kernel, head_grid(nvox), kHeadNT, 0, st, nvox, pr->h3, pr->a3, pr->P, pr->prob, labels,
               1.0 / (double)nvox, pr->da3, pr->G, pr->loss);
    wgrad<16, 8>(pr, tg, pr->da3, pr->h2, OFF_W3, OFF_B3, st);
    pdl_launch(conv_kernel<8, 16, CONV_DGRAD>, g, 128, 0, st, pr->m, tg, pr->da3, pr->W3d, nullptr, nullptr, pr->a2, pr->da2);
    wgrad<8, 16>(pr, tg, pr->da2, pr->h1, OFF_W2, OFF_B2, st);
    pdl_launch(conv_kernel<16, 8, CONV_DGRAD>, g, 128, 0, st, pr->m, tg, pr->da2, pr->W2d, nullptr, nullptr, pr->a1, pr->da1);
    wgrad<2, 8>(pr, tg, pr->da1, x, OFF_W1, OFF_B1, st);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

}  // namespace spdba

// ------------------------------------------------------------------ C ABI
extern "C" int64_t spdba_predictor_num_params(void) { return NPARAM; }

extern "C" void spdba_predictor_destroy(spdba_predictor* pr) {
    if (!pr) return;
    cudaDeviceSynchronize();
    for (void* p : pr->allocs) spdba::dev_free(p);
    delete pr;
}

extern "C" spdba_status spdba_predictor_create(spdba_predictor** out, int32_t nd, int32_t nh, int32_t nw,
                                               int32_t max_batch, const float* init_params) {
    if (!out || nd < 3 || nh < 3 || nw < 3 || max_batch < 1 || !init_params)
        return fail(SPDBA_ERR_ARG, "spdba_predictor_create: bad arguments");
    spdba_predictor* pr = new spdba_predictor();
    pr->m = MapDims{nd, nh, nw, (long long)nd * nh * nw};
    pr->max_batch = max_batch;
    pr->adam_t = 0;
    const long long nv = pr->m.V * max_batch;
    spdba_status s = SPDBA_OK;
#define A(ptr, bytes) \
    if (s == SPDBA_OK) s = pr->alloc(&pr->ptr, bytes)
    A(P, sizeof(float) * NPARAM);
    A(G, sizeof(float) * NPARAM);
    A(M, sizeof(float) * NPARAM);
    A(Vv, sizeof(float) * NPARAM);
    A(prob, sizeof(float) * nv);
    A(labels, sizeof(float) * nv);
    A(a1, sizeof(float) * nv * 8);
    A(a2, sizeof(float) * nv * 16);
    A(a3, sizeof(float) * nv * 8);
    A(W1t, sizeof(bf16) * 8 * kpad(54));
    A(W2t, sizeof(bf16) * 16 * kpad(216));
    A(W3t, sizeof(bf16) * 8 * kpad(432));
    A(W2d, sizeof(bf16) * 8 * kpad(27 * 16));
    A(W3d, sizeof(bf16) * 16 * kpad(27 * 8));
    A(h1, sizeof(bf16) * nv * 8);
    A(h2, sizeof(bf16) * nv * 16);
    A(h3, sizeof(bf16) * nv * 8);
    A(da1, sizeof(bf16) * nv * 8);
    A(da2, sizeof(bf16) * nv * 16);
    A(da3, sizeof(bf16) * nv * 8);
    A(loss, sizeof(double));
#undef A
    if (s == SPDBA_OK) {
        cudaError_t e = cudaMemcpy(pr->P, init_params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemset(pr->M, 0, sizeof(float) * NPARAM);
        if (e == cudaSuccess) e = cudaMemset(pr->Vv, 0, sizeof(float) * NPARAM);
        if (e != cudaSuccess) s = cuda_fail(e, "predictor init");
    }
    if (s == SPDBA_OK) s = refresh_weights(pr, 0);
    if (s == SPDBA_OK) {
        cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) s = cuda_fail(e, "predictor init");
    }
    if (s != SPDBA_OK) {
        spdba_predictor_destroy(pr);
        return s;
    }
    *out = pr;
    return SPDBA_OK;
}

extern "C" spdba_status spdba_predictor_get_params(spdba_predictor* pr, float* host_out) {
    if (!pr || !host_out) return fail(SPDBA_ERR_ARG, "spdba_predictor_get_params: NULL");
    SPDBA_CUDA(cudaMemcpy(host_out, pr->P, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
    return SPDBA_OK;
}

extern "C" spdba_status spdba_predictor_set_params(spdba_predictor* pr, const float* host_in) {
    if (!pr || !host_in) return fail(SPDBA_ERR_ARG, "spdba_predictor_set_params: NULL");
    SPDBA_CUDA(cudaMemcpy(pr->P, host_in, sizeof(float) * NPARAM, cudaMemcpyHostToDevice));
    spdba_status s = refresh_weights(pr, 0);
    if (s != SPDBA_OK) return s;
    SPDBA_CUDA(cudaDeviceSynchronize());
    return SPDBA_OK;
}

extern "C" spdba_status spdba_predictor_features(spdba_predictor* pr, const double* maxsq, const double* tau,
                                                 const uint8_t* states, int32_t nmaps, void* x_bf16, void* stream) {
    if (!pr || !maxsq || !tau || !states || !x_bf16 || nmaps < 1 || nmaps > pr->max_batch)
        return fail(SPDBA_ERR_ARG, "spdba_predictor_features: bad arguments");
    pdl_launch(features_kernel, grid_of(pr->m.V * nmaps, 256), 256, 0, (cudaStream_t)stream, pr->m.V, nmaps, maxsq, tau,
               states, (bf16*)x_bf16);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

extern "C" spdba_status spdba_predictor_forward(spdba_predictor* pr, const void* x_bf16, int32_t nmaps, float* prob,
                                                void* stream) {
    if (!pr || !x_bf16 || !prob || nmaps < 1 || nmaps > pr->max_batch)
        return fail(SPDBA_ERR_ARG, "spdba_predictor_forward: bad arguments");
    cudaStream_t st = (cudaStream_t)stream;
    const long long nvox = pr->m.V * nmaps;
    spdba_status s = forward(pr, (const bf16*)x_bf16, nmaps, false, st);
    if (s != SPDBA_OK) return s;
    pdl_launch(head_kernel, head_grid(nvox), kHeadNT, 0, st, nvox, pr->h3, pr->a3, pr->P, prob, nullptr, 0.0, nullptr,
               nullptr, nullptr);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

extern "C" spdba_status spdba_predictor_gradients(spdba_predictor* pr, const void* x_bf16, const float* labels,
                                                  int32_t nmaps, double* loss_out, float* grads_host) {
    if (!pr || !x_bf16 || !labels || nmaps < 1 || nmaps > pr->max_batch)
        return fail(SPDBA_ERR_ARG, "spdba_predictor_gradients: bad arguments");
    spdba_status s = forward(pr, (const bf16*)x_bf16, nmaps, true, 0);
    if (s == SPDBA_OK) s = backward(pr, (const bf16*)x_bf16, labels, nmaps, 0);
    if (s != SPDBA_OK) return s;
    SPDBA_CUDA(cudaDeviceSynchronize());
    if (loss_out) SPDBA_CUDA(cudaMemcpy(loss_out, pr->loss, sizeof(double), cudaMemcpyDeviceToHost));
    if (grads_host) SPDBA_CUDA(cudaMemcpy(grads_host, pr->G, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
    return SPDBA_OK;
}

extern "C" spdba_status spdba_predictor_train_step(spdba_predictor* pr, const void* x_bf16, const float* labels,
                                                   int32_t nmaps, float lr, double* loss_out, void* stream) {
    if (!pr || !x_bf16 || !labels || nmaps < 1 || nmaps > pr->max_batch || !(lr > 0))
        return fail(SPDBA_ERR_ARG, "spdba_predictor_train_step: bad arguments");
    cudaStream_t st = (cudaStream_t)stream;
    spdba_status s = forward(pr, (const bf16*)x_bf16, nmaps, true, st);
    if (s == SPDBA_OK) s = backward(pr, (const bf16*)x_bf16, labels, nmaps, st);
    if (s != SPDBA_OK) return s;
    pr->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)pr->adam_t), c2 = 1.f - powf(b2, (float)pr->adam_t);
    pdl_launch(adam_kernel, grid_of(NPARAM, 256), 256, 0, st, pr->P, pr->G, pr->M, pr->Vv, NPARAM, lr, b1, b2, 1e-8f, c1, c2);
    SPDBA_CUDA(cudaGetLastError());
    if ((s = refresh_weights(pr, st)) != SPDBA_OK) return s;
    if (loss_out) {
        SPDBA_CUDA(cudaMemcpyAsync(loss_out, pr->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
        SPDBA_CUDA(cudaStreamSynchronize(st));
    }
    return SPDBA_OK;
}

// Predicted states: measure = p (as FP64) for the classifier, tau = prob_threshold.
spdba_status spdba_predictor_states_internal(spdba_predictor* pr, const double* maxsq, const double* tau,
                                             uint8_t* states, int32_t nmaps, void* x_scratch, double* measure_out,
                                             cudaStream_t st) {
    spdba_status s = spdba_predictor_features(pr, maxsq, tau, states, nmaps, x_scratch, st);
    if (s != SPDBA_OK) return s;
    if ((s = spdba_predictor_forward(pr, x_scratch, nmaps, pr->prob, st)) != SPDBA_OK) return s;
    const long long n = pr->m.V * nmaps;
    pdl_launch(prob_to_measure_kernel, grid_of(n, 256), 256, 0, st, pr->prob, measure_out, n);
    SPDBA_CUDA(cudaGetLastError());
    return SPDBA_OK;
}

bool spdba_predictor_map_matches(const spdba_predictor* pr, long long nd, long long nh, long long nw) {
    return pr && pr->m.D == nd && pr->m.H == nh && pr->m.W == nw;
}
