// Learned preconditioner network: a three-level U-Net on the slot lattice.
//
// Tensors are channel-last, (B, D, H, W, C); activations are stored in BF16,
// every sum is accumulated in FP32, master weights and gradients are FP32.
// Weight layout per convolution: W[tap][cin][cout] (tap = (dz*KY + dy)*KX + dx
// with dz in 0..KZ-1), then bias[cout].  Layer order and widths:
//   enc0a cin->8, enc0b 8->8, enc1a 8->16, enc1b 16->16, enc2a 16->32,
//   enc2b 32->32, dec1a (32+16)->16, dec1b 16->16, dec0a (16+8)->8,
//   dec0b 8->8, out 8->cout (1x1)
// 3x3(x3) convolutions with zero padding 1 and ReLU; 2x average-pool down,
// nearest-neighbour up, concatenation [upsampled, skip].  In 2D, KZ = 1 and
// D = 1.
//
// Convolutions run on the tensor cores (unet_tc.cuh: implicit GEMM with
// mma.sync, BF16 operands, FP32 accumulation; activations and output
// gradients are staged channel-last with the channel count padded to a
// multiple of 8).  The upsampling and concatenation of the decoder are part
// of the staging of its convolutions (and of their weight gradients), the
// ReLU masks of the backward pass part of the epilogues that write the BF16
// gradients.  As kernels of their own these passes took longer than the
// convolutions: one thread per element with 64-bit divisions, 407 us to write
// the 24-channel concatenation of 128^3 voxels.  The data gradient is the
// forward kernel on the output gradient (rounded to BF16) with flipped,
// transposed weights; the weight gradient reduces per-CTA partials in a fixed
// order (no atomics), so a gradient is bit-reproducible.  Pooling, the
// adjoints that join two paths, the normalised squared-error loss and Adam
// are elementwise kernels, eight channels (16 bytes) per thread.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>
#include "internal.cuh"
#include "ctx.cuh"
#include "unet_tc.cuh"

using stk::warp_sum;

namespace {

struct Shape { int B, D, H, W; };
__host__ __device__ inline int64_t vox(const Shape& s) { return (int64_t)s.B * s.D * s.H * s.W; }


__device__ __forceinline__ void unpack8(const uint4& w, float (&f)[8]) {
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        f[2 * k] = __uint_as_float(u[k] << 16);
        f[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
    uint32_t u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
        u[k] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(u[0], u[1], u[2], u[3]);
}
__device__ __forceinline__ void load8(const float* p, float (&f)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
    f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
// item e of (voxel, group of 8 channels) -> coordinates
struct Item { int b, z, y, x, k; };
__device__ __forceinline__ Item item_of(int64_t e, const Shape& s, int ng) {
    Item i;
    const uint32_t v = (uint32_t)(e / ng);                // fewer than 2^31 voxels per level in any buffer that fits
    i.k = (int)(e - (int64_t)v * ng);
    uint32_t r = v / (uint32_t)s.W;
    i.x = (int)(v - r * (uint32_t)s.W);
    uint32_t q = r / (uint32_t)s.H;
    i.y = (int)(r - q * (uint32_t)s.H);
    i.b = (int)(q / (uint32_t)s.D);
    i.z = (int)(q - (uint32_t)i.b * (uint32_t)s.D);
    return i;
}
__device__ __forceinline__ int64_t vox_at(const Shape& s, int b, int z, int y, int x) {
    return (((int64_t)b * s.D + z) * s.H + y) * s.W + x;
}

// 2x average pooling: X fine (shape s), Y coarse (shape o); c a multiple of 8
__global__ void __launch_bounds__(256) k_pool(const __nv_bfloat16* __restrict__ X, Shape s, Shape o, int c, int pz,
                                              __nv_bfloat16* __restrict__ Y) {
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= vox(o) * (c / 8)) return;
    const Item i = item_of(e, o, c / 8);
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int dz = 0; dz < 1 + pz; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                float f[8];
                unpack8(*reinterpret_cast<const uint4*>(
                            X + vox_at(s, i.b, pz ? 2 * i.z + dz : i.z, 2 * i.y + dy, 2 * i.x + dx) * c + 8 * i.k), f);
#pragma unroll
                for (int k = 0; k < 8; ++k) sum[k] += f[k];
            }
    const float inv = pz ? 0.125f : 0.25f;                // exact
#pragma unroll
    for (int k = 0; k < 8; ++k) sum[k] *= inv;
    *reinterpret_cast<uint4*>(Y + e * 8) = pack8(sum);
}

// Gradient at a decoder input's coarse part: the adjoint of the upsampling
// (sum over the 2^d children of channels [0, c) of dY, fine, cy channels),
// through the ReLU of the coarse activations act, rounded to BF16.
__global__ void __launch_bounds__(256) k_up_adj(const float* __restrict__ dY, Shape s, Shape o, int c, int cy, int pz,
                                                const __nv_bfloat16* __restrict__ act, __nv_bfloat16* __restrict__ g) {
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= vox(o) * (c / 8)) return;
    const Item i = item_of(e, o, c / 8);
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int dz = 0; dz < 1 + pz; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                float f[8];
                load8(dY + vox_at(s, i.b, pz ? 2 * i.z + dz : i.z, 2 * i.y + dy, 2 * i.x + dx) * cy + 8 * i.k, f);
#pragma unroll
                for (int k = 0; k < 8; ++k) sum[k] += f[k];
            }
    float a[8];
    unpack8(*reinterpret_cast<const uint4*>(act + e * 8), a);
#pragma unroll
    for (int k = 0; k < 8; ++k) sum[k] = a[k] > 0.f ? sum[k] : 0.f;
    *reinterpret_cast<uint4*>(g + e * 8) = pack8(sum);
}

// Gradient at an encoder level's output, which feeds the skip connection
// (channels [c0, c0 + c) of dY, cy channels) and the pooling (its gradient dP,
// coarse): their sum through the ReLU of act, rounded to BF16.
__global__ void __launch_bounds__(256) k_skip_pool_adj(const float* __restrict__ dY, const float* __restrict__ dP,
                                                       Shape s, Shape o, int c, int c0, int cy, int pz,
                                                       const __nv_bfloat16* __restrict__ act,
                                                       __nv_bfloat16* __restrict__ g) {
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int ng = c / 8;
    if (e >= vox(s) * ng) return;
    const Item i = item_of(e, s, ng);
    float f[8], p[8], a[8];
    load8(dY + (e / ng) * cy + c0 + 8 * i.k, f);
    load8(dP + vox_at(o, i.b, pz ? i.z / 2 : i.z, i.y / 2, i.x / 2) * c + 8 * i.k, p);
    unpack8(*reinterpret_cast<const uint4*>(act + e * 8), a);
    const float inv = pz ? 0.125f : 0.25f;                // exact
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = a[k] > 0.f ? f[k] + p[k] * inv : 0.f;
    *reinterpret_cast<uint4*>(g + e * 8) = pack8(f);
}

// loss = mean_b ||out_b - y_b||^2 / ||y_b||^2; g = d loss / d out.  The two
// sums per sample are reduced deterministically: per-block partials (warp
// shuffles, then warps in order), then the blocks in order.  FP64 arithmetic
// and conversions are slow on this part (two per clock and SM; FP64 sums and an
// FP64 division per element took 319 us for 8.4 M elements), so the squares are
// summed, and the gradient's factor is applied, in three FP32 parts where FP32
// holds every part exactly: 1000 squares to 8e-20 relative (FP64 sums 3e-15, sums
// in two FP32 parts 6e-13), the gradient rounded once to FP32.  Values outside
// that range (below 2^-50 or above 2^50, not finite) are squared and summed in
// FP64.
constexpr int LOSS_BLOCKS = 256;      // most blocks per sample
struct Squares {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    double far = 0.0;
    // + (a + b + c)
    __device__ __forceinline__ void plus(float a, float b, float c) {
        float s, t, u, v;
        stk::two_sum(hi, a, s, t);
        hi = s;
        stk::two_sum(mid, b, s, u);
        stk::two_sum(s, t, mid, v);
        lo += c + u + v;
    }
    // a^2; false where a^2 and its error are not FP32 numbers: nothing is added
    __device__ __forceinline__ bool add(float a) {
        const float m = fabsf(a);
        const bool near = (m >= 0x1p-50f && m <= 0x1p50f) || m == 0.f;
        const float x = near ? a : 0.f, p = __fmul_rn(x, x);    // (rounded: the sums must not take it in unrounded)
        plus(p, fmaf(x, x, -p), 0.f);
        return near;
    }
    __device__ __forceinline__ void add_far(float a) {
        const float m = fabsf(a);
        if (!((m >= 0x1p-50f && m <= 0x1p50f) || m == 0.f)) far = fma((double)a, (double)a, far);
    }
    // sum over the warp (lane 0)
    __device__ __forceinline__ double warp() {
        for (int o = 16; o > 0; o >>= 1) {
            const float a = __shfl_xor_sync(0xffffffffu, hi, o), b = __shfl_xor_sync(0xffffffffu, mid, o),
                        c = __shfl_xor_sync(0xffffffffu, lo, o);
            plus(a, b, c);
        }
        double s = 0.0;
        if ((threadIdx.x & 31) == 0) s = (double)hi + ((double)mid + (double)lo);
        if (__any_sync(0xffffffffu, far != 0.0)) s += warp_sum(far);
        return s;
    }
};
__global__ void __launch_bounds__(256) k_loss_partials(const float* __restrict__ out, const float* __restrict__ y,
                                                       int64_t per, double* part) {
    __shared__ double red[2][8];
    const int b = blockIdx.y;
    Squares num, den;
    const float* ob = out + b * per;
    const float* yb = y + b * per;
    const int64_t step = (int64_t)gridDim.x * 256;
    int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    bool near = true;
    for (; e + 3 * step < per; e += 4 * step) {
        float o[4], t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { o[k] = ob[e + k * step]; t[k] = yb[e + k * step]; }
#pragma unroll
        for (int k = 0; k < 4; ++k) near = num.add(o[k] - t[k]) & den.add(t[k]) & near;
    }
    for (; e < per; e += step) { const float t = yb[e]; near = num.add(ob[e] - t) & den.add(t) & near; }
    // (a loop of its own: as predicated instructions the FP64 squares would cost
    // every element their 64 clocks: 75 us for 8.4 M elements instead of 26)
    if (!near)
        for (e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < per; e += step) {
            const float t = yb[e];
            num.add_far(ob[e] - t);
            den.add_far(t);
        }
    const double dn = num.warp(), dd = den.warp();
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { red[0][w] = dn; red[1][w] = dd; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, c = 0.0;
        for (int q = 0; q < 8; ++q) { a += red[0][q]; c += red[1][q]; }
        part[2 * (b * gridDim.x + blockIdx.x)] = a;
        part[2 * (b * gridDim.x + blockIdx.x) + 1] = c;
    }
}

// The gradient's factor 2 / (||y||^2 B) of a sample and ||y||^2.  The factor is
// (f0 + f1 + f2) scale, exactly the FP64 value, scale a power of two; zeros if it
// is far outside the FP32 range.
struct LossFactor {
    double den;
    float f0, f1, f2, scale;
};
// One warp per sample: the blocks' partials, a fixed tree; then the factor.
__global__ void k_loss_finish(const double* part, int nblocks, int B, double* sums, LossFactor* fac) {
    const int b = blockIdx.x, lane = threadIdx.x;
    double a = 0.0, c = 0.0;
    for (int q = lane; q < nblocks; q += 32) { a += part[2 * (b * nblocks + q)]; c += part[2 * (b * nblocks + q) + 1]; }
    a = warp_sum(a);
    c = warp_sum(c);
    if (lane != 0) return;
    sums[2 * b] = a;
    sums[2 * b + 1] = c;
    LossFactor f{c, 0.f, 0.f, 0.f, 0.f};
    int ex = 0;
    double m = c > 0.0 ? frexp(2.0 / c / B, &ex) : 0.0;
    if (abs(ex) <= 120) {
        f.f0 = (float)m;
        m -= (double)f.f0;
        f.f1 = (float)m;
        f.f2 = (float)(m - (double)f.f1);
        f.scale = ldexpf(1.f, ex);
    }
    fac[b] = f;
}

// Gradient entry 2 d / (||y||^2 B), rounded once to FP32: d f as the exact d f0
// and d f1 and a rounded d f2.  ok is cleared where the parts of the product or
// the result are not clear of FP32's ends (then it is loss_grad_far's).
__device__ __forceinline__ float loss_grad(float d, const LossFactor& f, bool& ok) {
    const float p = __fmul_rn(d, f.f0), e = fmaf(d, f.f0, -p), q = __fmul_rn(d, f.f1), g = fmaf(d, f.f1, -q);
    float s, t, u, v;
    stk::two_sum(e, q, s, t);
    stk::two_sum(p, s, u, v);
    const float r = (u + (v + (t + fmaf(d, f.f2, g)))) * f.scale;
    const float m = fabsf(d), a = fabsf(r);
    ok = ok && (d == 0.f || (m >= 0x1p-60f && m <= 0x1p100f && a >= 0x1p-100f && a <= 0x1p100f));
    return r;
}
__device__ __noinline__ float loss_grad_far(float d, double den, int B) { return (float)(2.0 * (double)d / den / B); }

// gradient of the loss at the output, in BF16 with cp channels (zero padded),
// as the output convolution's backward kernels read it: four channels a thread
__global__ void __launch_bounds__(256) k_loss_grad(const float* __restrict__ out, const float* __restrict__ y,
                                                   int64_t nvox, int c, int cp, const LossFactor* __restrict__ fac,
                                                   __nv_bfloat16* __restrict__ g) {
    const int nq = cp >> 2, per = 256 / nq;               // nq = 2 or 4
    const int q = threadIdx.x & (nq - 1);
    const int64_t vs = (int64_t)blockIdx.x * per + threadIdx.x / nq;
    if (vs >= nvox) return;
    const int64_t v = (int64_t)blockIdx.y * nvox + vs;
    const LossFactor f = fac[blockIdx.y];
    float r[4] = {0.f, 0.f, 0.f, 0.f};
    // (a sample whose target is zero contributes nothing)
    if (4 * q < c && f.den > 0.0) {
        const float* po = out + v * c + 4 * q;
        const float* py = y + v * c + 4 * q;
        float d[4];
        bool ok = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            d[k] = po[k] - py[k];
            r[k] = loss_grad(d[k], f, ok);
        }
        if (!ok)
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] = loss_grad_far(d[k], f.den, gridDim.y);
    }
    const __nv_bfloat162 lo = __floats2bfloat162_rn(r[0], r[1]), hi = __floats2bfloat162_rn(r[2], r[3]);
    *reinterpret_cast<uint2*>(g + v * cp + 4 * q) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

__global__ void k_adam(float* th, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    float gg = g[e];
    float mm = b1 * m[e] + (1.f - b1) * gg;
    float vv = b2 * v[e] + (1.f - b2) * gg * gg;
    m[e] = mm; v[e] = vv;
    th[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

inline unsigned nblk(int64_t n) { return (unsigned)((n + 255) / 256); }

}  // namespace

// ---------------------------------------------------------------------------
struct Conv {
    int cin, cout, ks;
    int64_t w_off, b_off, nw;
};

struct stokes_net_s {
    int dim = 3, cin = 0, cout = 0;
    int KZ = 3;
    int64_t max_vox = 0;
    std::vector<Conv> L;
    int64_t np = 0;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    // packed BF16 weights per layer: forward [cp(cout)][taps cp(cin)], data
    // gradient [cp(cin)][taps cp(cout)]; the forward ones are repacked after
    // every change of the parameters
    std::vector<__nv_bfloat16*> wf, wg;
    bool wf_valid = false;
    __nv_bfloat16 *gA = nullptr, *gB = nullptr;   // output gradients of two consecutive layers in BF16
    float* part = nullptr;          // weight-gradient partials, part_ctas x part_stride floats
    int part_ctas = 0, sms = 0, device = 0;
    int adam_t = 0;
    // activations (BF16) and gradients (FP32)
    __nv_bfloat16 *xin = nullptr, *e0a = nullptr, *e0 = nullptr, *p0 = nullptr, *e1a = nullptr, *e1 = nullptr,
                  *p1 = nullptr, *e2a = nullptr, *e2 = nullptr, *d1a = nullptr, *d1 = nullptr, *d0a = nullptr,
                  *d0 = nullptr;
    float* out = nullptr;
    // FP32 data gradients at the decoder inputs (24 and 48 channels) and at
    // the pooled tensors (8 and 16 channels)
    float *g_c0 = nullptr, *g_c1 = nullptr, *g_p0 = nullptr, *g_p1 = nullptr;
    double* sums = nullptr;
    LossFactor* fac = nullptr;      // per sample: the loss gradient's factor
    std::vector<void*> allocs;
    cudaStream_t s = nullptr;
    std::string err;
};

namespace {

using unet_tc::cp8;
// (cin, cout) the network supports: the tensor-core kernels are instantiated
// for input channels padded to 8 or 16 and output channels padded to 8 or 16
bool io_channels_ok(int c) { return c == 4 || c == 8 || c == 12 || c == 16; }
constexpr int MAX_DEVICES = 64;
constexpr int PART_STRIDE = 27 * 32 * 32 + 32;     // largest taps x cp(cin) x cp(cout) + cp(cout)

int taps_of(const stokes_net_s* n, const Conv& c) { return (n->KZ == 3 && c.ks == 3 ? 3 : 1) * c.ks * c.ks; }

// CTAs of a persistent kernel: the tiles, at most what fits on the device
// (and `cap`); resident: the kernel's cached answer for this process.
template <class K>
int persistent_ctas(const stokes_net_s* n, K k, size_t smem, int tiles, int cap, std::atomic<int>& resident) {
    int per = resident.load(std::memory_order_relaxed);
    if (per <= 0) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 256, smem);
        per = std::max(per, 1);
        resident.store(per, std::memory_order_relaxed);
    }
    return std::max(1, std::min({tiles, std::max(n->sms, 1) * per, cap}));
}

// Operands of one convolution: input (X, and Xc for the upsampled channels),
// packed weights, epilogue.
struct ConvArgs {
    const __nv_bfloat16 *X = nullptr, *Xc = nullptr, *Wp = nullptr, *mask = nullptr;
    const float* bias = nullptr;
    int cout = 0, relu = 0;
    __nv_bfloat16* Yb = nullptr;
    float* Yf = nullptr;
};

template <int KZ, int KS, int CP, int COUTP, int CU>
cudaError_t launch_conv_tc(stokes_net_s* n, Shape s, const ConvArgs& a) {
    using C = unet_tc::ConvCfg<KZ, KS, CP, COUTP>;
    auto k = unet_tc::k_conv_tc<KZ, KS, CP, COUTP, CU>;
    static std::atomic<int> resident[MAX_DEVICES];
    const unet_tc::TShape ts = C::G::shape(s.B, s.D, s.H, s.W);
    const int G = persistent_ctas(n, k, C::SMEM, C::G::tiles(ts), 1 << 30, resident[n->device]);
    k<<<G, 256, C::SMEM, n->s>>>(a.X, a.Xc, ts, a.Wp, a.bias, a.cout, a.relu, a.mask, a.Yb, a.Yf);
    return cudaGetLastError();
}

// one convolution on the tensor cores: cp input channels (cu of them from the
// coarse tensor), packed weights with coutp rows
cudaError_t conv_tc(stokes_net_s* n, int ks, int cp, int coutp, int cu, Shape s, const ConvArgs& a) {
#define CONV_CASE(KZ_, KS_, CP_, CO_, CU_)                                     \
    if (n->KZ == KZ_ && ks == KS_ && cp == CP_ && coutp == CO_ && cu == CU_)   \
        return launch_conv_tc<KZ_, KS_, CP_, CO_, CU_>(n, s, a);
#define CONV_CASES(KZ_)                                                                                    \
    CONV_CASE(KZ_, 3, 8, 8, 0) CONV_CASE(KZ_, 3, 16, 8, 0) CONV_CASE(KZ_, 3, 8, 16, 0)                     \
    CONV_CASE(KZ_, 3, 16, 16, 0) CONV_CASE(KZ_, 3, 16, 32, 0) CONV_CASE(KZ_, 3, 32, 32, 0)                 \
    CONV_CASE(KZ_, 3, 48, 16, 32) CONV_CASE(KZ_, 3, 24, 8, 16) CONV_CASE(KZ_, 3, 8, 24, 0)                 \
    CONV_CASE(KZ_, 3, 16, 48, 0) CONV_CASE(KZ_, 3, 32, 16, 0)                                              \
    CONV_CASE(KZ_, 1, 8, 8, 0) CONV_CASE(KZ_, 1, 8, 16, 0) CONV_CASE(KZ_, 1, 16, 8, 0)
    CONV_CASES(3)
    CONV_CASES(1)
#undef CONV_CASES
#undef CONV_CASE
    return cudaErrorInvalidValue;
}

template <int KZ, int KS, int CP, int COUTP, int CU>
cudaError_t launch_wgrad_tc(stokes_net_s* n, const __nv_bfloat16* X, const __nv_bfloat16* Xc, Shape s,
                            const __nv_bfloat16* g16, int cin, int cout, float* dW, float* db) {
    using C = unet_tc::WgCfg<KZ, KS, CP, COUTP>;
    static_assert(C::E + COUTP <= PART_STRIDE, "partial buffer too small");
    static_assert(256 % COUTP == 0, "the bias sums deal whole channels to the threads");
    auto k = unet_tc::k_wgrad_tc<KZ, KS, CP, COUTP, CU>;
    static std::atomic<int> resident[MAX_DEVICES];
    const unet_tc::TShape ts = C::G::shape(s.B, s.D, s.H, s.W);
    const int G = persistent_ctas(n, k, C::SMEM, C::G::tiles(ts), n->part_ctas, resident[n->device]);
    k<<<G, 256, C::SMEM, n->s>>>(X, Xc, ts, g16, n->part);
    const int tot = C::E + COUTP;
    unet_tc::k_wgrad_reduce<<<(tot + 31) / 32, 256, 0, n->s>>>(n->part, G, C::G::TAPS, CP, COUTP, cin, cout, dW, db);
    return cudaGetLastError();
}

cudaError_t wgrad_tc(stokes_net_s* n, int ks, int cp, int coutp, int cu, const __nv_bfloat16* X,
                     const __nv_bfloat16* Xc, Shape s, const __nv_bfloat16* g16, int cin, int cout, float* dW,
                     float* db) {
#define WG_CASE(KZ_, KS_, CP_, CO_, CU_)                                       \
    if (n->KZ == KZ_ && ks == KS_ && cp == CP_ && coutp == CO_ && cu == CU_)   \
        return launch_wgrad_tc<KZ_, KS_, CP_, CO_, CU_>(n, X, Xc, s, g16, cin, cout, dW, db);
#define WG_CASES(KZ_)                                                                                      \
    WG_CASE(KZ_, 3, 8, 8, 0) WG_CASE(KZ_, 3, 16, 8, 0) WG_CASE(KZ_, 3, 8, 16, 0) WG_CASE(KZ_, 3, 16, 16, 0) \
    WG_CASE(KZ_, 3, 16, 32, 0) WG_CASE(KZ_, 3, 32, 32, 0) WG_CASE(KZ_, 3, 48, 16, 32)                      \
    WG_CASE(KZ_, 3, 24, 8, 16) WG_CASE(KZ_, 1, 8, 8, 0) WG_CASE(KZ_, 1, 8, 16, 0)
    WG_CASES(3)
    WG_CASES(1)
#undef WG_CASES
#undef WG_CASE
    return cudaErrorInvalidValue;
}

// pack the forward (and, for training, data-gradient) weights of every layer
cudaError_t pack_weights(stokes_net_s* n, bool grad) {
    unet_tc::PackList list{};
    int m = 0, most = 0;
    for (size_t li = 0; li < n->L.size(); ++li) {
        const Conv& c = n->L[li];
        const int taps = taps_of(n, c), ci = cp8(c.cin), co = cp8(c.cout);
        if (!n->wf_valid) list.l[m++] = {n->theta + c.w_off, n->wf[li], taps, c.cin, c.cout, co, ci, 0};
        if (grad) list.l[m++] = {n->theta + c.w_off, n->wg[li], taps, c.cin, c.cout, ci, co, 1};
        most = std::max(most, taps * ci * co);
    }
    if (m) unet_tc::k_pack_weights<<<dim3(std::min(nblk(most), 32u), m), 256, 0, n->s>>>(list);
    n->wf_valid = true;
    return cudaGetLastError();
}

// the decoder's first convolutions read their upsampled channels from the
// coarse tensor
int up_channels(int li) { return li == 6 ? 32 : li == 8 ? 16 : 0; }

cudaError_t conv(stokes_net_s* n, int li, const __nv_bfloat16* X, Shape s, int relu, __nv_bfloat16* Yb, float* Yf,
                 const __nv_bfloat16* Xc = nullptr) {
    const Conv& c = n->L[li];
    ConvArgs a;
    a.X = X; a.Xc = Xc; a.Wp = n->wf[li]; a.bias = n->theta + c.b_off;
    a.cout = c.cout; a.relu = relu; a.Yb = Yb; a.Yf = Yf;
    return conv_tc(n, c.ks, cp8(c.cin), cp8(c.cout), up_channels(li), s, a);
}

// gradient step of layer li from its output gradient dY (BF16, cp(cout)
// channels, the ReLU mask applied): weight and bias gradient from the layer
// input X (and Xc); data gradient either through the ReLU of the layer input
// as BF16 (dXb) or as FP32 (dXf), or neither
cudaError_t conv_backward(stokes_net_s* n, int li, const __nv_bfloat16* X, Shape s, const __nv_bfloat16* dY,
                          __nv_bfloat16* dXb, float* dXf, const __nv_bfloat16* Xc = nullptr) {
    const Conv& c = n->L[li];
    cudaError_t e = wgrad_tc(n, c.ks, cp8(c.cin), cp8(c.cout), up_channels(li), X, Xc, s, dY, c.cin, c.cout,
                             n->grad + c.w_off, n->grad + c.b_off);
    if (e != cudaSuccess || (!dXb && !dXf)) return e;
    ConvArgs a;
    a.X = dY; a.Wp = n->wg[li]; a.cout = c.cin;
    a.mask = dXb ? X : nullptr; a.Yb = dXb; a.Yf = dXf;
    return conv_tc(n, c.ks, cp8(c.cout), cp8(c.cin), 0, s, a);
}

Shape half(const Shape& s, int pz) { return Shape{s.B, pz ? s.D / 2 : s.D, s.H / 2, s.W / 2}; }

void to_bf16(stokes_net_s* n, const float* x, Shape s) {
    const int cp = cp8(n->cin), per = 256 / (cp / 4);
    unet_tc::k_to_bf16_pad<<<(unsigned)((vox(s) + per - 1) / per), 256, 0, n->s>>>(
        x, vox(s), n->cin, cp, ((uintptr_t)x & 15u) == 0, n->xin);
}

// forward pass from xin; the output goes to `out` (FP32, cout channels)
cudaError_t forward(stokes_net_s* n, Shape s, float* out) {
    const int pz = n->KZ == 3;
    if (!n->wf_valid && pack_weights(n, false) != cudaSuccess) return cudaGetLastError();
    Shape s1 = half(s, pz), s2 = half(s1, pz);
    cudaError_t e;
    if ((e = conv(n, 0, n->xin, s, 1, n->e0a, nullptr))) return e;
    if ((e = conv(n, 1, n->e0a, s, 1, n->e0, nullptr))) return e;
    k_pool<<<nblk(vox(s1)), 256, 0, n->s>>>(n->e0, s, s1, 8, pz, n->p0);
    if ((e = conv(n, 2, n->p0, s1, 1, n->e1a, nullptr))) return e;
    if ((e = conv(n, 3, n->e1a, s1, 1, n->e1, nullptr))) return e;
    k_pool<<<nblk(vox(s2) * 2), 256, 0, n->s>>>(n->e1, s1, s2, 16, pz, n->p1);
    if ((e = conv(n, 4, n->p1, s2, 1, n->e2a, nullptr))) return e;
    if ((e = conv(n, 5, n->e2a, s2, 1, n->e2, nullptr))) return e;
    if ((e = conv(n, 6, n->e1, s1, 1, n->d1a, nullptr, n->e2))) return e;
    if ((e = conv(n, 7, n->d1a, s1, 1, n->d1, nullptr))) return e;
    if ((e = conv(n, 8, n->e0, s, 1, n->d0a, nullptr, n->d1))) return e;
    if ((e = conv(n, 9, n->d0a, s, 1, n->d0, nullptr))) return e;
    return conv(n, 10, n->d0, s, 0, nullptr, out);
}

// backward from dL/dout (BF16 in gA), parameter gradients in grad
cudaError_t backward(stokes_net_s* n, Shape s) {
    const int pz = n->KZ == 3;
    if (pack_weights(n, true) != cudaSuccess) return cudaGetLastError();
    Shape s1 = half(s, pz), s2 = half(s1, pz);
    cudaError_t e;
    __nv_bfloat16 *gA = n->gA, *gB = n->gB;
    if ((e = conv_backward(n, 10, n->d0, s, gA, gB, nullptr))) return e;              // gB = d d0
    if ((e = conv_backward(n, 9, n->d0a, s, gB, gA, nullptr))) return e;              // gA = d d0a
    if ((e = conv_backward(n, 8, n->e0, s, gA, nullptr, n->g_c0, n->d1))) return e;   // g_c0 = d [up d1, e0]
    k_up_adj<<<nblk(vox(s1) * 2), 256, 0, n->s>>>(n->g_c0, s, s1, 16, 24, pz, n->d1, gB);         // gB = d d1
    if ((e = conv_backward(n, 7, n->d1a, s1, gB, gA, nullptr))) return e;             // gA = d d1a
    if ((e = conv_backward(n, 6, n->e1, s1, gA, nullptr, n->g_c1, n->e2))) return e;  // g_c1 = d [up e2, e1]
    k_up_adj<<<nblk(vox(s2) * 4), 256, 0, n->s>>>(n->g_c1, s1, s2, 32, 48, pz, n->e2, gB);        // gB = d e2
    if ((e = conv_backward(n, 5, n->e2a, s2, gB, gA, nullptr))) return e;             // gA = d e2a
    if ((e = conv_backward(n, 4, n->p1, s2, gA, nullptr, n->g_p1))) return e;         // g_p1 = d p1
    k_skip_pool_adj<<<nblk(vox(s1) * 2), 256, 0, n->s>>>(n->g_c1, n->g_p1, s1, s2, 16, 32, 48, pz, n->e1, gB);  // d e1
    if ((e = conv_backward(n, 3, n->e1a, s1, gB, gA, nullptr))) return e;             // gA = d e1a
    if ((e = conv_backward(n, 2, n->p0, s1, gA, nullptr, n->g_p0))) return e;         // g_p0 = d p0
    k_skip_pool_adj<<<nblk(vox(s)), 256, 0, n->s>>>(n->g_c0, n->g_p0, s, s1, 8, 16, 24, pz, n->e0, gB);         // d e0
    if ((e = conv_backward(n, 1, n->e0a, s, gB, gA, nullptr))) return e;              // gA = d e0a
    return conv_backward(n, 0, n->xin, s, gA, nullptr, nullptr);
}

}  // namespace

extern "C" {

stokes_status stokes_net_destroy(stokes_net n) {
    if (!n) return STOKES_OK;
    for (void* p : n->allocs) cudaFree(p);
    if (n->s) cudaStreamDestroy(n->s);
    delete n;
    return STOKES_OK;
}

stokes_status stokes_net_create(stokes_net* out, int dim, int cin, int cout, int64_t max_voxels) {
    if (!out || (dim != 2 && dim != 3) || !io_channels_ok(cin) || !io_channels_ok(cout) || max_voxels < 1)
        return STOKES_ERR_ARG;
    auto* n = new stokes_net_s();
    n->dim = dim; n->cin = cin; n->cout = cout; n->KZ = dim == 3 ? 3 : 1;
    n->max_vox = max_voxels;
    int sizes[11][3] = {{cin, 8, 3}, {8, 8, 3}, {8, 16, 3}, {16, 16, 3}, {16, 32, 3}, {32, 32, 3},
                        {48, 16, 3}, {16, 16, 3}, {24, 8, 3}, {8, 8, 3}, {8, cout, 1}};
    int64_t off = 0;
    for (auto& q : sizes) {
        Conv c;
        c.cin = q[0]; c.cout = q[1]; c.ks = q[2];
        int taps = (dim == 3 && c.ks == 3 ? 3 : 1) * c.ks * c.ks;
        c.nw = (int64_t)taps * c.cin * c.cout;
        c.w_off = off; off += c.nw;
        c.b_off = off; off += c.cout;
        off = (off + 3) & ~3LL;       // float4-aligned weight blocks
        n->L.push_back(c);
    }
    n->np = off;
    cudaError_t e = cudaStreamCreate(&n->s);
    auto A = [&](void** p, size_t bytes) {
        if (e != cudaSuccess) return;
        e = cudaMalloc(p, bytes);
        if (e == cudaSuccess) { n->allocs.push_back(*p); e = cudaMemset(*p, 0, bytes); }
    };
    int64_t V = max_voxels;
    A((void**)&n->theta, 4 * off); A((void**)&n->grad, 4 * off); A((void**)&n->m, 4 * off); A((void**)&n->v, 4 * off);
    for (const Conv& c : n->L) {
        const int64_t taps = (dim == 3 && c.ks == 3 ? 3 : 1) * c.ks * c.ks;
        n->wf.push_back(nullptr);
        n->wg.push_back(nullptr);
        A((void**)&n->wf.back(), 2 * taps * cp8(c.cin) * cp8(c.cout));
        A((void**)&n->wg.back(), 2 * taps * cp8(c.cin) * cp8(c.cout));
    }
    int dev = 0;
    cudaGetDevice(&dev);
    n->device = dev >= 0 && dev < MAX_DEVICES ? dev : 0;
    cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev);
    n->part_ctas = 2 * std::max(n->sms, 1);
    A((void**)&n->part, 4 * (size_t)n->part_ctas * PART_STRIDE);
    // the levels hold at most V, V / 4 and V / 16 voxels (2D; fewer in 3D)
    A((void**)&n->gA, 2 * V * 16);
    A((void**)&n->gB, 2 * V * 16);
    A((void**)&n->xin, 2 * V * cp8(cin));
    __nv_bfloat16** full8[] = {&n->e0a, &n->e0, &n->d0a, &n->d0};
    for (auto p : full8) A((void**)p, 2 * V * 8);
    __nv_bfloat16** half16[] = {&n->p0, &n->e1a, &n->e1, &n->p1, &n->d1a, &n->d1};
    for (auto p : half16) A((void**)p, 2 * (V / 4 + 1) * 16);
    A((void**)&n->e2a, 2 * (V / 16 + 1) * 32); A((void**)&n->e2, 2 * (V / 16 + 1) * 32);
    A((void**)&n->out, 4 * V * cout);
    A((void**)&n->g_c0, 4 * V * 24); A((void**)&n->g_c1, 4 * (V / 4 + 1) * 48);
    A((void**)&n->g_p0, 4 * (V / 4 + 1) * 8); A((void**)&n->g_p1, 4 * (V / 16 + 1) * 16);
    A((void**)&n->fac, sizeof(LossFactor) * 1024);
    A((void**)&n->sums, 16 * 1024 + 16 * 1024 * LOSS_BLOCKS);   // sums, then the per-block partials
    if (e != cudaSuccess) { stokes_net_destroy(n); return STOKES_ERR_CUDA; }
    *out = n;
    return STOKES_OK;
}

int64_t stokes_net_param_count(stokes_net n) { return n ? n->np : -1; }

stokes_status stokes_net_set_params(stokes_net n, const float* host) {
    if (!n || !host) return STOKES_ERR_ARG;
    if (cudaMemcpy(n->theta, host, 4 * n->np, cudaMemcpyHostToDevice) != cudaSuccess) return STOKES_ERR_CUDA;
    n->wf_valid = false;
    cudaMemset(n->m, 0, 4 * n->np);
    cudaMemset(n->v, 0, 4 * n->np);
    n->adam_t = 0;
    return STOKES_OK;
}

stokes_status stokes_net_get_params(stokes_net n, float* host) {
    if (!n || !host) return STOKES_ERR_ARG;
    return cudaMemcpy(host, n->theta, 4 * n->np, cudaMemcpyDeviceToHost) == cudaSuccess ? STOKES_OK : STOKES_ERR_CUDA;
}

static bool shape_ok(stokes_net n, int B, int D, int H, int W) {
    int m = n->dim == 3 ? 4 : 1;
    return B >= 1 && D >= 1 && H >= 4 && W >= 4 && H % 4 == 0 && W % 4 == 0 && D % m == 0 &&
           (n->dim == 3 || D == 1) && (int64_t)B * D * H * W <= n->max_vox;
}

// x: FP32 device (B, D, H, W, cin) channel-last; y: FP32 device (.., cout)
stokes_status stokes_net_forward(stokes_net n, int B, int D, int H, int W, const float* x, float* y) {
    if (!n || !x || !y || !shape_ok(n, B, D, H, W)) return STOKES_ERR_ARG;
    Shape s{B, D, H, W};
    to_bf16(n, x, s);
    if (forward(n, s, y) != cudaSuccess) return STOKES_ERR_CUDA;
    return cudaStreamSynchronize(n->s) == cudaSuccess ? STOKES_OK : STOKES_ERR_CUDA;
}

// Loss (mean over samples of ||N(x) - y||^2 / ||y||^2) and its parameter
// gradient (left in the network; copied to grad_host if not NULL).
stokes_status stokes_net_gradient(stokes_net n, int B, int D, int H, int W, const float* x, const float* y,
                                  double* loss, float* grad_host) {
    if (!n || !x || !y || !shape_ok(n, B, D, H, W) || B > 1024) return STOKES_ERR_ARG;
    Shape s{B, D, H, W};
    to_bf16(n, x, s);
    if (forward(n, s, n->out) != cudaSuccess) return STOKES_ERR_CUDA;
    const int64_t nv = (int64_t)D * H * W, per = nv * n->cout;
    const int cp = cp8(n->cout);
    // eight elements per thread or more
    const int lb = (int)std::min<int64_t>(LOSS_BLOCKS, (per + 2047) / 2048);
    k_loss_partials<<<dim3(lb, B), 256, 0, n->s>>>(n->out, y, per, n->sums + 2 * 1024);
    k_loss_finish<<<B, 32, 0, n->s>>>(n->sums + 2 * 1024, lb, B, n->sums, n->fac);
    const int vpb = 256 / (cp / 4);
    k_loss_grad<<<dim3((unsigned)((nv + vpb - 1) / vpb), B), 256, 0, n->s>>>(n->out, y, nv, n->cout, cp, n->fac, n->gA);
    cudaMemsetAsync(n->grad, 0, 4 * n->np, n->s);
    if (backward(n, s) != cudaSuccess) return STOKES_ERR_CUDA;
    std::vector<double> sums(2 * B);
    cudaMemcpyAsync(sums.data(), n->sums, 16 * B, cudaMemcpyDeviceToHost, n->s);
    if (cudaStreamSynchronize(n->s) != cudaSuccess) return STOKES_ERR_CUDA;
    if (loss) {
        double L = 0;
        for (int b = 0; b < B; ++b) L += sums[2 * b + 1] > 0.0 ? sums[2 * b] / sums[2 * b + 1] : 0.0;
        *loss = L / B;
    }
    if (grad_host && cudaMemcpy(grad_host, n->grad, 4 * n->np, cudaMemcpyDeviceToHost) != cudaSuccess)
        return STOKES_ERR_CUDA;
    return STOKES_OK;
}

stokes_status stokes_net_train_step(stokes_net n, int B, int D, int H, int W, const float* x, const float* y, float lr,
                                    double* loss) {
    stokes_status st = stokes_net_gradient(n, B, D, H, W, x, y, loss, nullptr);
    if (st != STOKES_OK) return st;
    n->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.f - std::pow(b1, (float)n->adam_t), c2 = 1.f - std::pow(b2, (float)n->adam_t);
    k_adam<<<nblk(n->np), 256, 0, n->s>>>(n->theta, n->grad, n->m, n->v, n->np, lr, b1, b2, 1e-8f, c1, c2);
    n->wf_valid = false;
    return cudaStreamSynchronize(n->s) == cudaSuccess ? STOKES_OK : STOKES_ERR_CUDA;
}

// Per layer (cin, cout, kernel size, weight offset, bias offset) in the flat
// parameter vector, for host-side conversion between layouts.
stokes_status stokes_net_layer(stokes_net n, int i, int* cin, int* cout, int* ks, int64_t* w_off, int64_t* b_off) {
    if (!n || i < 0 || i >= (int)n->L.size()) return STOKES_ERR_ARG;
    const Conv& c = n->L[i];
    *cin = c.cin; *cout = c.cout; *ks = c.ks; *w_off = c.w_off; *b_off = c.b_off;
    return STOKES_OK;
}

}  // extern "C"
