// Tensor-core convolutions of the learned preconditioner's U-Net (implicit
// GEMM on mma.sync m16n8k16 / m16n8k8, BF16 operands, FP32 accumulation).
//
// Layout: activations are channel-last BF16 with the channel count padded to
// a multiple of 8 (cp(c)), so that every voxel's channels start on a 16-byte
// boundary and 8 channels form one ldmatrix row.  A CTA of 256 threads
// (8 warps) owns tiles of 256 output voxels (3D 8 x 8 x 4, 2D 16 x 16) and
// stages their input halo in shared memory.  The voxel stride there is an odd
// multiple of 16 bytes (cps()), as is the row stride of the packed weights
// (kws()), so that the eight rows of an ldmatrix, and the eight weight rows of
// a B fragment, fall on different banks (cp + 8 halves for every cp, as
// before, gave 2-way conflicts at 8 channels and 4-way ones at 24).
//
// All kernels are persistent over the tiles and copy the next tile's halo with
// cp.async while the current one is multiplied (two buffers where they fit):
// a CTA that stages, waits and multiplies one tile spent most of its life
// waiting.  Measured on 128^3 voxels, before and after: 24 -> 8 channels 379
// and 126 us, 16 -> 8 100 and 89 us, 8 -> 8 92 and 47 us; weight gradients on
// 4 x 64^3 voxels: 24 -> 8 320 and 76 us, 8 -> 8 119 and 31 us.  The 8-channel
// layers are now bound by issue and the tensor pipe together (67 % and 40 %
// busy), the 16-channel ones by shared-memory reads (one A fragment feeds a
// single 8-column product).
// The input may come from two tensors (CU > 0): channels [0, CU) are those of
// the coarse voxel that contains the voxel (nearest 2x upsampling), the others
// the skip connection's, so the concatenated tensor is never written.
//
// * Forward / data gradient (k_conv_tc): out[v][co] = sum over taps and input
//   channels of in[v + tap][ci] W[co][tap][ci].  GEMM M = voxels (each warp
//   two 16-voxel m-tiles), N = output channels (n-tiles of 8), K = taps x
//   channels in chunks of 16 (one ldmatrix.x4 per m-tile: matrices 0 and 1
//   are rows 0-7 / 8-15 at channels 0-7 of the chunk, 2 and 3 at channels
//   8-15), with one k8 step for a channel count of 8 mod 16.  The packed
//   weights Wp[co][tap * cp + ci] sit in shared memory; B fragments are
//   32-bit loads.  The epilogue adds the bias, applies ReLU (or, for a data
//   gradient, the ReLU mask of the layer below) and stores BF16 and/or FP32.
//   The data gradient is the same kernel on the output gradient with the
//   flipped, transposed weights.
// * Weight gradient (k_wgrad_tc): dW[tap][ci][co] = sum over voxels
//   in[v + tap][ci] dY[v][co].  GEMM M = (tap, 8 input channels) groups, two
//   per 16-row tile (so no row is padding where a layer has 8 or 24 input
//   channels), N = output channels, K = voxels (16 per step), both operands by
//   ldmatrix.trans from the staged halo and output-gradient tile.  A warp
//   holds the accumulators of all its tiles at once: one B fragment load
//   serves them all, and their chains are independent.  After each voxel tile
//   they are added to the CTA's FP32 partial in shared memory (every entry
//   has one owner, so the sum order is fixed).  Every CTA writes its partial
//   and k_wgrad_reduce sums the partials in a fixed order: deterministic, no
//   atomics.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>

namespace unet_tc {

__host__ __device__ constexpr int cp8(int c) { return (c + 7) / 8 * 8; }

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm4(uint32_t (&a)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm2(uint32_t (&a)[2], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(a[0]), "=r"(a[1]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&a)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm2t(uint32_t (&a)[2], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(a[0]), "=r"(a[1]) : "r"(addr));
}
__device__ __forceinline__ void mma16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma8(float (&d)[4], const uint32_t (&a)[2], uint32_t b0) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(b0));
}

// Grid of one level, and the tile counts per axis with floor(2^32 / count)
// (a tile index is split into coordinates with one multiplication and one
// correction per axis).
struct TShape {
    int B, D, H, W;
    uint32_t ntx, nty, ntz, mx, my, mz;
};
__device__ __forceinline__ uint32_t div_by(uint32_t t, uint32_t d, uint32_t m, uint32_t& rem) {
    uint32_t q = __umulhi(t, m);                          // floor(t / d) or one less
    rem = t - q * d;
    if (rem >= d) { rem -= d; ++q; }
    return q;
}

// tile geometry: 3D 8 x 8 x 4 (KZ = 3), 2D 16 x 16 (KZ = 1); R = halo radius
template <int KZ, int KS>
struct Geo {
    static constexpr int TX = KZ == 3 ? 8 : 16, TY = KZ == 3 ? 8 : 16, TZ = KZ == 3 ? 4 : 1;
    static constexpr int R = KS / 2;
    static constexpr int RZ = KZ == 3 ? R : 0;
    static constexpr int HX = TX + 2 * R, HY = TY + 2 * R, HZ = TZ + 2 * RZ;
    static constexpr int NH = HX * HY * HZ;
    static constexpr int TAPS = (KZ == 3 ? KS : 1) * KS * KS;
    __host__ static TShape shape(int B, int D, int H, int W) {
        TShape s{B, D, H, W, (uint32_t)((W + TX - 1) / TX), (uint32_t)((H + TY - 1) / TY), (uint32_t)((D + TZ - 1) / TZ), 0, 0, 0};
        auto m = [](uint32_t d) { return d == 1 ? 0xffffffffu : (uint32_t)((1ull << 32) / d); };
        s.mx = m(s.ntx); s.my = m(s.nty); s.mz = m(s.ntz);
        return s;
    }
    __host__ __device__ static int tiles(const TShape& s) { return s.B * (int)(s.ntx * s.nty * s.ntz); }
    // tile t -> batch and origin
    __device__ static void origin(const TShape& s, int t, int& b, int& x0, int& y0, int& z0) {
        uint32_t r, q = div_by((uint32_t)t, s.ntx, s.mx, r);
        x0 = (int)r * TX;
        q = div_by(q, s.nty, s.my, r);
        y0 = (int)r * TY;
        b = (int)div_by(q, s.ntz, s.mz, r);
        z0 = (int)r * TZ;
    }
    // tap k -> offset in halo voxels
    __device__ static int tap_off(int k) {
        const int dx = k % KS, dy = (k / KS) % KS, dz = k / (KS * KS);
        return ((dz - RZ) * HY + (dy - R)) * HX + (dx - R);
    }
    // output voxel v of the tile -> its halo index (tap offset 0)
    __device__ static int halo_of(int v) {
        const int x = v % TX, y = (v / TX) % TY, z = v / (TX * TY);
        return ((z + RZ) * HY + (y + R)) * HX + (x + R);
    }
};

// Shared-memory strides in halves: odd multiples of 8 (16 bytes).
__host__ __device__ constexpr int cps(int cp) { return cp % 16 == 8 ? cp : cp + 8; }
__host__ __device__ constexpr int kws(int k) { return k % 16 == 8 ? k : k + 8; }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Copy of the input halo of one tile: CP channels (multiple of 8) per voxel,
// zero outside the grid, to shared memory with voxel stride cps(CP).  Channels
// [0, CU) come from Xc, the tensor of the next coarser level (CU channels),
// the others from X (CP - CU channels).  A thread copies the same 16-byte
// pieces of every tile: their offsets from the tile's first voxel (tile
// origins are even, so the coarse ones are constant too) and places are
// computed once, and a tile inside the grid needs no tests.  (Recomputed for
// every tile, this arithmetic was most of the kernel: 709 warp instructions
// per 32 voxels of an 8 -> 8 layer, 135 of them the products.)
template <int KZ, int KS, int CP, int CU>
struct Halo {
    using G = Geo<KZ, KS>;
    static constexpr int NG = CP / 8, N = (G::NH * NG + 255) / 256;
    static constexpr int UZ = KZ == 3 ? 1 : 0;             // the coarse level halves z in 3D only
    static constexpr uint32_t NONE = 0xffffffffu, UP = 1u << 31;
    using Rel = typename std::conditional<KZ == 3, int, int64_t>::type;
    Rel rel[N];                                            // from the tile's first voxel, in pieces of 8 channels
    uint32_t pos[N];                                       // shared offset / 16 (13 bits), hx, hy (5 bits), hz (4 bits), UP
    __device__ __forceinline__ void init(const TShape& s) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = threadIdx.x + 256 * i;
            const int gq = e % NG, v = e / NG;
            const int hx = v % G::HX, hy = (v / G::HX) % G::HY, hz = v / (G::HX * G::HY);
            const bool up = CU > 0 && gq < CU / 8;
            rel[i] = up ? (((Rel)((hz - G::RZ) >> UZ) * (s.H >> 1) + ((hy - G::R) >> 1)) * (s.W >> 1) + ((hx - G::R) >> 1)) *
                                  (CU / 8) + gq
                        : (((Rel)(hz - G::RZ) * s.H + (hy - G::R)) * s.W + (hx - G::R)) * ((CP - CU) / 8) + gq - CU / 8;
            pos[i] = (uint32_t)(v * (cps(CP) / 8) + gq) | (uint32_t)hx << 13 | (uint32_t)hy << 18 | (uint32_t)hz << 23 |
                     (up ? UP : 0u);
            if (e >= G::NH * NG) pos[i] = NONE;
        }
    }
    __device__ __forceinline__ void copy(const __nv_bfloat16* __restrict__ X, const __nv_bfloat16* __restrict__ Xc,
                                         const TShape& s, int b, int x0, int y0, int z0, uint32_t sx) const {
        const __nv_bfloat16* xb = X + ((((int64_t)b * s.D + z0) * s.H + y0) * s.W + x0) * (CP - CU);
        const __nv_bfloat16* cb = Xc;
        if (CU > 0)
            cb += ((((int64_t)b * (s.D >> UZ) + (z0 >> UZ)) * (s.H >> 1) + (y0 >> 1)) * (s.W >> 1) + (x0 >> 1)) * CU;
        const bool inside = x0 >= G::R && y0 >= G::R && z0 >= G::RZ && x0 + G::TX + G::R <= s.W &&
                            y0 + G::TY + G::R <= s.H && z0 + G::TZ + G::RZ <= s.D;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (pos[i] == NONE) continue;
            bool ok = true;
            if (!inside) {
                const int gx = x0 - G::R + (int)((pos[i] >> 13) & 31), gy = y0 - G::R + (int)((pos[i] >> 18) & 31),
                          gz = z0 - G::RZ + (int)((pos[i] >> 23) & 15);
                ok = (unsigned)gx < (unsigned)s.W && (unsigned)gy < (unsigned)s.H && (unsigned)gz < (unsigned)s.D;
            }
            const __nv_bfloat16* src = (CU > 0 && (pos[i] & UP) ? cb : xb) + 8 * (int64_t)rel[i];
            cp_async16(sx + 16u * (pos[i] & 0x1fffu), ok ? src : X, ok);
        }
    }
};

// ---- forward / data gradient ------------------------------------------------
// Wp: packed BF16 weights [COUTP][K] (K = TAPS * CP).  bias: FP32 [cout] or
// null.  Outputs: Yb (BF16, COUTP channels, the padded channels written as
// zero) and/or Yf (FP32, cout channels).  mask (or null): the layer-below
// activations with COUTP channels; outputs where they are not positive are
// written as zero (the adjoint of their ReLU).
template <int KZ, int KS, int CP, int COUTP>
struct ConvCfg {
    using G = Geo<KZ, KS>;
    static constexpr int CPS = cps(CP);
    static constexpr int K = G::TAPS * CP;
    static constexpr int KW = kws(K);
    static constexpr int NT = COUTP / 8;
    static constexpr size_t HALO = (size_t)G::NH * CPS * 2, WTS = (size_t)COUTP * KW * 2;
    // two halo buffers, unless that leaves fewer than two CTAs on an SM
    static constexpr int NBUF = 2 * (2 * HALO + WTS) <= 220 * 1024 ? 2 : 1;
    static constexpr size_t SMEM = NBUF * HALO + WTS;
};

template <int KZ, int KS, int CP, int COUTP, int CU>
__global__ void __launch_bounds__(256) k_conv_tc(const __nv_bfloat16* __restrict__ X,
                                                 const __nv_bfloat16* __restrict__ Xc, TShape s,
                                                 const __nv_bfloat16* __restrict__ Wp, const float* __restrict__ bias,
                                                 int cout, int relu, const __nv_bfloat16* __restrict__ mask,
                                                 __nv_bfloat16* __restrict__ Yb, float* __restrict__ Yf) {
    using C = ConvCfg<KZ, KS, CP, COUTP>;
    using G = typename C::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    const uint32_t sx0 = smem_addr(smraw);
    __nv_bfloat16* sw = reinterpret_cast<__nv_bfloat16*>(smraw + C::NBUF * C::HALO);
    const int ntiles = G::tiles(s);
    int tile = blockIdx.x;
    int b, x0, y0, z0;
    G::origin(s, tile, b, x0, y0, z0);
    Halo<KZ, KS, CP, CU> halo;
    halo.init(s);
    halo.copy(X, Xc, s, b, x0, y0, z0, sx0);
    cp_commit();
    // weights: [COUTP][K] -> stride KW, 16-byte pieces, once per CTA
    for (int e = threadIdx.x; e < COUTP * (C::K / 8); e += 256) {
        const int n = e / (C::K / 8), q = e % (C::K / 8);
        *reinterpret_cast<uint4*>(sw + n * C::KW + 8 * q) =
            *reinterpret_cast<const uint4*>(Wp + (int64_t)n * C::K + 8 * q);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int li = lane >> 3, lj = lane & 7;
    float bs[C::NT][2];
#pragma unroll
    for (int nt = 0; nt < C::NT; ++nt)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int c = 8 * nt + 2 * t + q;
            bs[nt][q] = bias && c < cout ? bias[c] : 0.f;
        }
    // ldmatrix rows: voxel (li & 1) * 8 + lj of each m-tile, channel half li >> 1
    uint32_t hrow[2];
#pragma unroll
    for (int m = 0; m < 2; ++m)
        hrow[m] = 2u * (uint32_t)(G::halo_of(32 * warp + 16 * m + (li & 1) * 8 + lj) * C::CPS);
    const uint32_t swa = smem_addr(sw) + 2u * (uint32_t)(g * C::KW + 2 * t);
    int buf = 0;
    for (; tile < ntiles; tile += gridDim.x) {
        const uint32_t sxa = sx0 + (uint32_t)(buf * C::HALO);
        const int next = tile + gridDim.x;
        int nb = 0, nx = 0, ny = 0, nz = 0;
        if (next < ntiles) G::origin(s, next, nb, nx, ny, nz);
        if constexpr (C::NBUF == 2) {
            if (next < ntiles) halo.copy(X, Xc, s, nb, nx, ny, nz, sx0 + (uint32_t)((buf ^ 1) * C::HALO));
            cp_commit();
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        float acc[2][C::NT][4];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int nt = 0; nt < C::NT; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[m][nt][q] = 0.f;
#pragma unroll
        for (int tap = 0; tap < G::TAPS; ++tap) {
            const int toff = 2 * G::tap_off(tap) * C::CPS;
            const int kbase = tap * CP;
#pragma unroll
            for (int c16 = 0; c16 < CP / 16; ++c16) {
                uint32_t a[2][4];
#pragma unroll
                for (int m = 0; m < 2; ++m) ldsm4(a[m], sxa + hrow[m] + (uint32_t)(toff + 32 * c16) + (li >> 1) * 16);
#pragma unroll
                for (int nt = 0; nt < C::NT; ++nt) {
                    const uint32_t wa = swa + 2u * (uint32_t)(8 * nt * C::KW + kbase + 16 * c16);
                    uint32_t b0, b1;
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(b0) : "r"(wa));
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(b1) : "r"(wa + 16u));
#pragma unroll
                    for (int m = 0; m < 2; ++m) mma16(acc[m][nt], a[m], b0, b1);
                }
            }
            if constexpr (CP % 16 == 8) {
                uint32_t a[2][2];
#pragma unroll
                for (int m = 0; m < 2; ++m) ldsm2(a[m], sxa + hrow[m] + (uint32_t)(toff + 2 * (CP - 8)));
#pragma unroll
                for (int nt = 0; nt < C::NT; ++nt) {
                    const uint32_t wa = swa + 2u * (uint32_t)(8 * nt * C::KW + kbase + CP - 8);
                    uint32_t b0;
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(b0) : "r"(wa));
#pragma unroll
                    for (int m = 0; m < 2; ++m) mma8(acc[m][nt], a[m], b0);
                }
            }
        }
        // epilogue: D[row][col] = acc[..][q]: rows g (q 0, 1) and g + 8 (q 2, 3), columns 2t, 2t + 1
        // (3D: x = g, y = 4 (warp % 2) + 2 m + h, z = warp / 2; 2D: x = g + 8 h, y = 2 warp + m)
        constexpr bool V3 = KZ == 3;
        const int xe = x0 + g, ye = y0 + (V3 ? 4 * (warp & 1) : 2 * warp), ze = z0 + (V3 ? warp >> 1 : 0);
        const int64_t oe = (((int64_t)b * s.D + ze) * s.H + ye) * s.W + xe;
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int dx = V3 ? 0 : 8 * h, dy = V3 ? 2 * m + h : m;
                if (xe + dx >= s.W || ye + dy >= s.H || ze >= s.D) continue;
                const int64_t o = oe + dy * s.W + dx;
#pragma unroll
                for (int nt = 0; nt < C::NT; ++nt) {
                    const int c = 8 * nt + 2 * t;
                    float v0 = acc[m][nt][2 * h], v1 = acc[m][nt][2 * h + 1];
                    if (bias) { v0 += bs[nt][0]; v1 += bs[nt][1]; }
                    if (relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
                    if (mask) {
                        const __nv_bfloat162 k = *reinterpret_cast<const __nv_bfloat162*>(mask + o * COUTP + c);
                        if (!(__low2float(k) > 0.f)) v0 = 0.f;
                        if (!(__high2float(k) > 0.f)) v1 = 0.f;
                    }
                    if (c >= cout) v0 = 0.f;
                    if (c + 1 >= cout) v1 = 0.f;
                    if (Yb) *reinterpret_cast<__nv_bfloat162*>(Yb + o * COUTP + c) = __floats2bfloat162_rn(v0, v1);
                    if (Yf) {
                        if (c < cout) Yf[o * cout + c] = v0;
                        if (c + 1 < cout) Yf[o * cout + c + 1] = v1;
                    }
                }
            }
        if constexpr (C::NBUF == 2) {
            buf ^= 1;
            __syncthreads();                              // the next step's copy overwrites the tile just read
        } else {
            __syncthreads();
            if (next < ntiles) halo.copy(X, Xc, s, nb, nx, ny, nz, sx0);
            cp_commit();
        }
        b = nb; x0 = nx; y0 = ny; z0 = nz;
    }
}

// ---- weight gradient ----------------------------------------------------------
// X (and Xc, CU): layer input as for k_conv_tc, dY: output gradient (BF16,
// COUTP channels).  part: FP32 [gridDim.x][TAPS * CP * COUTP + COUTP] partials
// (weights as [tap][ci][co], then the bias gradient).
template <int KZ, int KS, int CP, int COUTP>
struct WgCfg {
    using G = Geo<KZ, KS>;
    static constexpr int CPS = cps(CP);
    static constexpr int COS = cps(COUTP);
    static constexpr int NT = COUTP / 8;
    static constexpr int E = G::TAPS * CP * COUTP;
    static constexpr int GRP = G::TAPS * (CP / 8);            // groups of 8 rows (tap, 8 channels)
    static constexpr int UNITS = (GRP + 1) / 2;               // 16-row tiles
    static constexpr int UPW = (UNITS + 7) / 8;               // per warp
    static constexpr size_t HALO = (size_t)G::NH * CPS * 2, GRAD = (size_t)256 * COS * 2;
    static constexpr size_t DW = (size_t)(E + COUTP) * 4;
    static constexpr int NBUF = 2 * (2 * (HALO + GRAD) + DW) <= 220 * 1024 ? 2 : 1;
    static constexpr size_t SMEM = NBUF * (HALO + GRAD) + DW;
};

template <int KZ, int KS, int CP, int COUTP, int CU>
__global__ void __launch_bounds__(256) k_wgrad_tc(const __nv_bfloat16* __restrict__ X,
                                                  const __nv_bfloat16* __restrict__ Xc, TShape s,
                                                  const __nv_bfloat16* __restrict__ dY, float* __restrict__ part) {
    using C = WgCfg<KZ, KS, CP, COUTP>;
    using G = typename C::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    const uint32_t s0 = smem_addr(smraw);
    float* dw = reinterpret_cast<float*>(smraw + C::NBUF * (C::HALO + C::GRAD));     // [E] then [COUTP]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int li = lane >> 3, lj = lane & 7;
    const int ntiles = G::tiles(s);
    Halo<KZ, KS, CP, CU> halo;
    halo.init(s);
    // one tile's halo and output gradient into buffer q
    auto stage = [&](int tile, int q) {
        int b, x0, y0, z0;
        G::origin(s, tile, b, x0, y0, z0);
        const uint32_t sx = s0 + (uint32_t)(q * (C::HALO + C::GRAD)), sy = sx + (uint32_t)C::HALO;
        halo.copy(X, Xc, s, b, x0, y0, z0, sx);
        for (int e = threadIdx.x; e < 256 * C::NT; e += 256) {
            const int k = e % C::NT, v = e / C::NT;
            const int x = x0 + v % G::TX, y = y0 + (v / G::TX) % G::TY, z = z0 + v / (G::TX * G::TY);
            const bool ok = x < s.W && y < s.H && z < s.D;
            const __nv_bfloat16* src = dY + (ok ? ((((int64_t)b * s.D + z) * s.H + y) * s.W + x) * COUTP + 8 * k : 0);
            cp_async16(sy + 2u * (uint32_t)(v * C::COS + 8 * k), src, ok);
        }
    };
    int tile = blockIdx.x;
    stage(tile, 0);
    cp_commit();
    for (int e = threadIdx.x; e < C::E + COUTP; e += 256) dw[e] = 0.f;
    // the lane's ldmatrix offset of every unit u = warp + 8 i of the warp: rows
    // 0-7 are group 2u, rows 8-15 group 2u + 1 (a group past the end repeats
    // group 0, its fragment is zeroed)
    uint32_t uoff[C::UPW];
#pragma unroll
    for (int i = 0; i < C::UPW; ++i) {
        int grp = 2 * (warp + 8 * i) + (li & 1);
        if (grp >= C::GRP) grp = 0;
        uoff[i] = 2u * (uint32_t)(G::tap_off(grp / (CP / 8)) * C::CPS + 8 * (grp % (CP / 8)));
    }
    float bsum = 0.f;                                     // bias gradient: channel tid % COUTP, voxels tid / COUTP + k SEG
    constexpr int SEG = 256 / COUTP;
    int buf = 0;
    for (; tile < ntiles; tile += gridDim.x) {
        const uint32_t sxa = s0 + (uint32_t)(buf * (C::HALO + C::GRAD)), sya = sxa + (uint32_t)C::HALO;
        const int next = tile + gridDim.x;
        if constexpr (C::NBUF == 2) {
            if (next < ntiles) stage(next, buf ^ 1);
            cp_commit();
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        {
            const __nv_bfloat16* sy = reinterpret_cast<const __nv_bfloat16*>(smraw + buf * (C::HALO + C::GRAD) + C::HALO);
            float a = 0.f;
            for (int v = threadIdx.x / COUTP; v < SEG * COUTP; v += SEG)
                a += __bfloat162float(sy[v * C::COS + threadIdx.x % COUTP]);
            bsum += a;
        }
        float acc[C::UPW][C::NT][4];
#pragma unroll
        for (int i = 0; i < C::UPW; ++i)
#pragma unroll
            for (int nt = 0; nt < C::NT; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[i][nt][q] = 0.f;
        for (int c = 0; c < 16; ++c) {
            // B = dY: voxels 16 c .. 16 c + 15, all output channels
            const int vb = 16 * c + (li & 1) * 8 + lj;
            uint32_t bb[C::NT][2];
#pragma unroll
            for (int nt = 0; nt + 1 < C::NT; nt += 2) {
                uint32_t w4[4];
                ldsm4t(w4, sya + 2u * (uint32_t)(vb * C::COS + 8 * (nt + (li >> 1))));
                bb[nt][0] = w4[0]; bb[nt][1] = w4[1]; bb[nt + 1][0] = w4[2]; bb[nt + 1][1] = w4[3];
            }
            if constexpr (C::NT % 2 == 1) ldsm2t(bb[C::NT - 1], sya + 2u * (uint32_t)(vb * C::COS + 8 * (C::NT - 1)));
            // A = X^T: matrix li holds group (li & 1), voxels (li >> 1) * 8 + 0..7
            const uint32_t va = sxa + 2u * (uint32_t)(G::halo_of(16 * c + (li >> 1) * 8 + lj) * C::CPS);
#pragma unroll
            for (int i = 0; i < C::UPW; ++i) {
                const int u = warp + 8 * i;
                if (u < C::UNITS) {
                    uint32_t a[4];
                    ldsm4t(a, va + uoff[i]);
                    if (C::GRP % 2 == 1 && u == C::UNITS - 1) { a[1] = 0u; a[3] = 0u; }
#pragma unroll
                    for (int nt = 0; nt < C::NT; ++nt) mma16(acc[i][nt], a, bb[nt][0], bb[nt][1]);
                }
            }
        }
        // D[m = row][n = out channel]: rows g, g + 8; columns 2t, 2t + 1
#pragma unroll
        for (int i = 0; i < C::UPW; ++i)
#pragma unroll
            for (int nt = 0; nt < C::NT; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int grp = 2 * (warp + 8 * i) + h;
                    if (grp >= C::GRP) continue;
                    float* d = dw + (8 * grp + g) * COUTP + 8 * nt + 2 * t;
                    d[0] += acc[i][nt][2 * h];
                    d[1] += acc[i][nt][2 * h + 1];
                }
        __syncthreads();                                  // the buffer is free for the next copy
        if constexpr (C::NBUF == 2) {
            buf ^= 1;
        } else {
            if (next < ntiles) stage(next, 0);
            cp_commit();
        }
    }
    // bias gradient: the segments of each channel in order
    float* red = reinterpret_cast<float*>(smraw);
    cp_wait<0>();
    __syncthreads();
    red[threadIdx.x] = bsum;
    __syncthreads();
    if (threadIdx.x < COUTP) {
        float a = 0.f;
        for (int q = 0; q < SEG; ++q) a += red[q * COUTP + threadIdx.x];
        dw[C::E + threadIdx.x] = a;
    }
    __syncthreads();
    float* o = part + (int64_t)blockIdx.x * (C::E + COUTP);
    for (int e = threadIdx.x; e < C::E + COUTP; e += 256) o[e] = dw[e];
}

// dW[tap][ci][co] (ci < cin, co < cout) and db[co] from the partials of
// nparts CTAs: 32 entries per block, warp w sums partials w, w + 8, ... in
// order, then the eight sums are added in order (one thread summing all 304
// partials of an entry took 23 us a layer, all of it load latency).
__global__ void __launch_bounds__(256) k_wgrad_reduce(const float* __restrict__ part, int nparts, int taps, int cp,
                                                      int coutp, int cin, int cout, float* __restrict__ dW,
                                                      float* __restrict__ db) {
    __shared__ float red[8][32];
    const int E = taps * cp * coutp;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    float acc = 0.f;
    if (e < E + coutp) {
#pragma unroll 8
        for (int q = w; q < nparts; q += 8) acc += part[(int64_t)q * (E + coutp) + e];
    }
    red[w][lane] = acc;
    __syncthreads();
    if (w != 0 || e >= E + coutp) return;
    acc = red[0][lane];
    for (int q = 1; q < 8; ++q) acc += red[q][lane];
    if (e >= E) {
        const int co = e - E;
        if (co < cout) db[co] = acc;
        return;
    }
    const int co = e % coutp, ci = (e / coutp) % cp, tap = e / (coutp * cp);
    if (ci < cin && co < cout) dW[((int64_t)tap * cin + ci) * cout + co] = acc;
}

// Packed BF16 weights for k_conv_tc from the FP32 master W[tap][cin][cout]:
// forward  Wp[co][tap * cp + ci] = W[tap][ci][co];
// gradient Wp[ci][tap * cpo + co] = W[taps - 1 - tap][ci][co] (the data
//          gradient as a convolution of the output gradient).
// Padded rows and columns are zero.
struct PackLayer {
    const float* W;
    __nv_bfloat16* Wp;
    int taps, cin, cout, rows, cpk, grad;
};
struct PackList { PackLayer l[22]; };
// one launch packs every layer (blockIdx.y: the layer and direction)
__global__ void k_pack_weights(PackList list) {
    const PackLayer p = list.l[blockIdx.y];
    const int K = p.taps * p.cpk;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < p.rows * K; e += gridDim.x * blockDim.x) {
        const int n = e / K, k = e % K, tap = k / p.cpk, c = k % p.cpk;
        float v = 0.f;
        if (!p.grad) {
            if (n < p.cout && c < p.cin) v = p.W[((int64_t)tap * p.cin + c) * p.cout + n];
        } else {
            if (n < p.cin && c < p.cout) v = p.W[((int64_t)(p.taps - 1 - tap) * p.cin + n) * p.cout + c];
        }
        p.Wp[e] = __float2bfloat16(v);
    }
}

// FP32 channel-last (c channels, a multiple of 4) -> BF16 with cp channels
// (zero padded), one thread per four channels (32-bit index arithmetic; one
// thread per channel with 64-bit divisions took 99 us for 2 M voxels of 12
// channels, 27 us is the traffic).  vec: x lies on a 16-byte boundary.
__global__ void k_to_bf16_pad(const float* __restrict__ x, int64_t nvox, int c, int cp, int vec,
                              __nv_bfloat16* __restrict__ y) {
    const int nq = cp >> 2, per = blockDim.x / nq;        // voxels per block
    const int q = threadIdx.x % nq;
    const int64_t v = (int64_t)blockIdx.x * per + threadIdx.x / nq;
    if (threadIdx.x >= per * nq || v >= nvox) return;
    float f[4] = {0.f, 0.f, 0.f, 0.f};
    if (4 * q < c) {
        const float* p = x + v * c + 4 * q;
        if (vec) {
            const float4 w = *reinterpret_cast<const float4*>(p);
            f[0] = w.x; f[1] = w.y; f[2] = w.z; f[3] = w.w;
        } else {
            for (int k = 0; k < 4; ++k) f[k] = p[k];
        }
    }
    __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
    *reinterpret_cast<uint2*>(y + v * cp + 4 * q) =
        make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}

}  // namespace unet_tc
