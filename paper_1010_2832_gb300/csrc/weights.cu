// Weight build (stokes_build_weights): volume fractions of every sample's
// control volume (Section 5), face status and the null-space elimination of
// Section 8, operator coefficients, the Jacobi diagonal and the list of
// tiles that hold an active unknown.  One thread per slot of the padded
// vertex lattice; everything in FP64.
#include <algorithm>
#include "internal.cuh"
#include "ctx.cuh"

namespace stk {

// ---------------------------------------------------------------------------
// Fractions of {phi < 0} of the piecewise-linear interpolant on a simplex.
// Closed forms by the count k of negative vertices (sorted values s):
//   triangle  k=1: s0^2/((s0-s1)(s0-s2))       k=2: 1 - s2^2/((s2-s0)(s2-s1))
//   tetra     k=1: s0^3/((s0-s1)(s0-s2)(s0-s3)) k=3: 1 - s3^3/(...)
//             k=2: [x^2y^2 - (p+q)xy(x+y) + pq(x^2+xy+y^2)] / [(x-p)(x-q)(y-p)(y-q)]
// (the two-negative tetrahedron written without cancellation).
// ---------------------------------------------------------------------------
// Sign tests and ordering on the IEEE bit patterns (integer ALU; FP64
// compares and min/max run on the FP64 pipe, which is slow on this part).
// For finite values they decide exactly as v < 0, v > 0 and <= do
// (-0 is neither negative nor positive and orders with +0).
__device__ __forceinline__ bool dneg(double v) {
    const long long b = __double_as_longlong(v);
    return b < 0 && b != (long long)0x8000000000000000ULL;
}
__device__ __forceinline__ bool dpos(double v) { return __double_as_longlong(v) > 0; }
__device__ __forceinline__ long long dkey(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ void cswap(double& a, double& b) {
    if (dkey(b) < dkey(a)) {
        const double t = a;
        a = b;
        b = t;
    }
}

__device__ double tri_frac(double a, double b, double c) {
    cswap(a, b); cswap(b, c); cswap(a, b);
    int k = dneg(a) + dneg(b) + dneg(c);
    if (k == 0) return 0.0;
    if (k == 3) return 1.0;
    if (k == 1) return __dmul_rn(a, a) / __dmul_rn(__dsub_rn(a, b), __dsub_rn(a, c));
    return 1.0 - __dmul_rn(c, c) / __dmul_rn(__dsub_rn(c, a), __dsub_rn(c, b));
}

__device__ double tet_frac(double a, double b, double c, double d) {
    cswap(a, b); cswap(c, d); cswap(a, c); cswap(b, d); cswap(b, c);
    int k = dneg(a) + dneg(b) + dneg(c) + dneg(d);
    if (k == 0) return 0.0;
    if (k == 4) return 1.0;
    if (k == 1) {
        double num = __dmul_rn(__dmul_rn(a, a), a);
        double den = __dmul_rn(__dmul_rn(__dsub_rn(a, b), __dsub_rn(a, c)), __dsub_rn(a, d));
        return num / den;
    }
    if (k == 3) {
        double num = __dmul_rn(__dmul_rn(d, d), d);
        double den = __dmul_rn(__dmul_rn(__dsub_rn(d, a), __dsub_rn(d, b)), __dsub_rn(d, c));
        return 1.0 - num / den;
    }
    // evaluation order (left to right, no fused multiply-add):
    //   ((x x) y) y - (((p + q) x) y)(x + y) + (p q)((x x + x y) + y y)
    //   over (((x - p)(x - q))(y - p))(y - q)
    double x = a, y = b, p = c, q = d;
    double xx = __dmul_rn(x, x), yy = __dmul_rn(y, y), xy = __dmul_rn(x, y);
    double t1 = __dmul_rn(__dmul_rn(xx, y), y);
    double t2 = __dmul_rn(__dmul_rn(__dmul_rn(__dadd_rn(p, q), x), y), __dadd_rn(x, y));
    double t3 = __dmul_rn(__dmul_rn(p, q), __dadd_rn(__dadd_rn(xx, xy), yy));
    double num = __dadd_rn(__dsub_rn(t1, t2), t3);
    double den = __dmul_rn(__dmul_rn(__dmul_rn(__dsub_rn(x, p), __dsub_rn(x, q)), __dsub_rn(y, p)), __dsub_rn(y, q));
    return num / den;
}

// A CV without a negative lattice value is exactly 0, one without a positive
// value exactly 1.  Every operation
// above is rounded separately and in the same order as in the FP64 reference,
// so the values, and every W > 0 test on them, are reproducible bit for bit.
//
// The control volumes cut by an interface are few and cost hundreds of FP64
// operations each, on a pipe of two operations per clock and SM.  A CTA (256
// slots) therefore collects its cut CVs in a list, and all its threads work on
// the list in batches of 32 CVs: first every simplex is classified on the
// integer pipe (no negative vertex: 0; no other: 1; the non-negative vertices
// all zero: 1, the formulas' value), then the remaining ones are evaluated
// class by class (k = 1, 2, 3 negative vertices: one branch per warp), then
// one lane per CV adds its simplices in their fixed order.  (One CV at a time
// per warp, every lane adding all 24 values, the 3D weights of a 256^3 grid
// took 11.0 ms;
// now 1.4 ms, and 0.4 ms for the sign bits.)
template <int DIM> struct Cv;
template <> struct Cv<2> {
    static constexpr int NK = 4, NS = 8;                  // sample kinds, triangles (centre, edge midpoint, corner)
    static constexpr int BLK = 16;                        // lattice points of a slot's block
};
template <> struct Cv<3> {
    // 24 tetrahedra (centre, face centre, two consecutive corners of that
    // face), faces in the order -x, +x, -y, +y, -z, +z and corners cycling
    // (-,-), (+,-), (+,+), (-,+) over the two other axes in increasing order
    static constexpr int NK = 7, NS = 24;
    static constexpr int BLK = 64;
};

// |v| within [2^-200, 2^200): products of four such values neither overflow
// nor underflow
__device__ __forceinline__ bool moderate(double v) {
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e >= 823 && e < 1223;
}
// v > 0 (false for NaN)
__device__ __forceinline__ bool wpos(double v) {
    return (unsigned long long)(__double_as_longlong(v) - 1) < 0x7ff0000000000000ULL;
}
__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }

// vertices of simplex t of the CV whose centre is phi[0]
__device__ __forceinline__ void simplex2(const double* phi, int Lx, int t, double (&v)[3]) {
    // ring order E, NE, N, NW, W, SW, S, SE
    auto at = [&](int r) {
        return phi[(r >= 1 && r <= 3 ? Lx : r >= 5 ? -Lx : 0) + (r <= 1 || r == 7 ? 1 : r >= 3 && r <= 5 ? -1 : 0)];
    };
    v[0] = phi[0];
    v[1] = at(t);
    v[2] = at((t + 1) & 7);
}
__device__ __forceinline__ void simplex3(const double* phi, int64_t Lx, int64_t Lxy, int t, double (&v)[4]) {
    const int face = t >> 2, c0 = t & 3, c1 = (c0 + 1) & 3, axis = face >> 1;
    const int64_t sa = axis == 0 ? 1 : axis == 1 ? Lx : Lxy;     // strides along the face's axis and the other two
    const int64_t su = axis == 0 ? Lx : 1, sv = axis == 2 ? Lx : Lxy;
    const double* f = phi + ((face & 1) ? sa : -sa);
    v[0] = phi[0];
    v[1] = f[0];
    v[2] = f[((c0 == 1 || c0 == 2) ? su : -su) + (c0 >= 2 ? sv : -sv)];
    v[3] = f[((c1 == 1 || c1 == 2) ? su : -su) + (c1 >= 2 ? sv : -sv)];
}

// Shared scratch of the evaluation of a CTA's cut CVs.
template <int DIM> struct CutSmem {
    static constexpr int NS = Cv<DIM>::NS;
    unsigned short list[2 * Cv<DIM>::NK * 256];           // cut CVs: (slot of the CTA) | kind << 8 | level set << 11
    unsigned short cls[3][32 * NS];                       // simplices of a batch with k = 1, 2, 3 negative vertices
    double val[32][NS + 1];
    int pos[32];                                          // the CV has a simplex with a positive vertex
    int ncut, ncls[3];
};

// Evaluate the CTA's list (256 threads, every one must call it).  addr(entry)
// is the lattice address of a CV's centre, store(entry, fraction) keeps it.
template <int DIM, class Addr, class Store>
__device__ __forceinline__ void cut_fractions(CutSmem<DIM>& sm, int64_t Lx, int64_t Lxy, Addr addr, Store store) {
    constexpr int NS = Cv<DIM>::NS, NV = DIM + 1;
    const int t = threadIdx.x + 32 * threadIdx.y;
    auto vertices = [&](int item, double (&v)[NV], int base) {
        const double* c = addr(sm.list[base + item / NS]);
        if constexpr (DIM == 2) simplex2(c, (int)Lx, item % NS, v);
        else simplex3(c, Lx, Lxy, item % NS, v);
    };
    const int ncut = sm.ncut;
    for (int base = 0; base < ncut; base += 32) {
        const int m = min(32, ncut - base);
        if (t < 3) sm.ncls[t] = 0;
        if (t < 32) sm.pos[t] = 0;
        __syncthreads();
        for (int item = t; item < m * NS; item += 256) {
            double v[NV];
            vertices(item, v, base);
            int k = 0;
            bool pos = false, zeros = true, mod = true;   // every non-negative vertex is zero; every negative one moderate
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                if (dneg(v[q])) { ++k; mod = mod && moderate(v[q]); }
                else zeros = zeros && is_zero(v[q]);
                pos = pos || dpos(v[q]);
            }
            if (k == 0) sm.val[item / NS][item % NS] = 0.0;
            else if (k == NV || (zeros && mod)) sm.val[item / NS][item % NS] = 1.0;
            else sm.cls[k - 1][atomicAdd(&sm.ncls[k - 1], 1)] = (unsigned short)item;
            if (pos) sm.pos[item / NS] = 1;
        }
        __syncthreads();
        // (the order within a class list varies, the values do not)
#pragma unroll
        for (int k = 0; k < NV - 1; ++k)
            for (int e = t; e < sm.ncls[k]; e += 256) {
                const int item = sm.cls[k][e];
                double v[NV];
                vertices(item, v, base);
                if constexpr (DIM == 2) sm.val[item / NS][item % NS] = tri_frac(v[0], v[1], v[2]);
                else sm.val[item / NS][item % NS] = tet_frac(v[0], v[1], v[2], v[3]);
            }
        __syncthreads();
        if (t < m) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < NS; ++q) s += sm.val[t][q];
            s /= (double)NS;
            if (!sm.pos[t]) {
                // no positive value at all: exactly 1 (in 3D the edge midpoints
                // are in no simplex, so the whole CV is looked at)
                const double* c = addr(sm.list[base + t]);
                bool pos = false;
                for (int dz = DIM == 3 ? -1 : 0; dz <= (DIM == 3 ? 1 : 0); ++dz)
                    for (int dy = -1; dy <= 1; ++dy)
                        for (int dx = -1; dx <= 1; ++dx) pos |= dpos(c[dz * Lxy + dy * Lx + dx]);
                if (!pos) s = 1.0;
            }
            store(sm.list[base + t], s);
        }
        // the next batch's classification starts after a barrier and writes
        // other entries of val only after this one's lanes have passed it
    }
}

// Sample kinds.  2D: 0 cell, 1 node, 2 u, 3 v.  3D: 0 cell, 1 u, 2 v, 3 w,
// 4 exy, 5 exz, 6 eyz.  Lattice offset per axis (a = 2 i + off).
__constant__ int c_off2[4][2] = {{2, 2}, {1, 1}, {1, 2}, {2, 1}};
__constant__ int c_off3[7][3] = {{2, 2, 2}, {1, 2, 2}, {2, 1, 2}, {2, 2, 1}, {1, 1, 2}, {1, 2, 1}, {2, 1, 1}};

__host__ __device__ __forceinline__ bool exists2(int kind, int i, int j, int nx, int ny) {
    if (i < 0 || j < 0 || i > nx || j > ny) return false;
    switch (kind) {
        case 0: return i < nx && j < ny;
        case 1: return true;
        case 2: return j < ny;
        default: return i < nx;
    }
}

__host__ __device__ __forceinline__ bool exists3(int kind, int i, int j, int k, int nx, int ny, int nz) {
    if (i < 0 || j < 0 || k < 0 || i > nx || j > ny || k > nz) return false;
    switch (kind) {
        case 0: return i < nx && j < ny && k < nz;
        case 1: return j < ny && k < nz;
        case 2: return i < nx && k < nz;
        case 3: return i < nx && j < ny;
        case 4: return k < nz;
        case 5: return j < ny;
        default: return i < nx;
    }
}

// ---- kernel 1: fractions ----------------------------------------------------
// The CVs of all kinds of slot (i, j[, k]) lie in the block of lattice points
// [2i, 2i+3] per axis (clipped to the lattice, whose last index per axis is
// 2n+2; at i = n only kinds centred at 2i+1 exist, whose points end at 2n+2).
// A mask holds one bit per point of the block (1 = negative; bit x + 4 y + 16 z);
// this is the part of it that the CV centred at offsets (ox, oy, oz) covers.
__host__ __device__ constexpr uint64_t cv_mask(int ox, int oy, int oz) {
    uint64_t m = 0;
    for (int z = oz - 1; z <= oz + 1; ++z)
        for (int y = oy - 1; y <= oy + 1; ++y)
            for (int x = ox - 1; x <= ox + 1; ++x)
                if (z >= 0) m |= 1ull << (x + 4 * y + 16 * z);
    return m;
}
__host__ __device__ constexpr uint64_t kind_mask3(int kd) {
    return kd == 0 ? cv_mask(2, 2, 2) : kd == 1 ? cv_mask(1, 2, 2) : kd == 2 ? cv_mask(2, 1, 2) : kd == 3 ? cv_mask(2, 2, 1)
         : kd == 4 ? cv_mask(1, 1, 2) : kd == 5 ? cv_mask(1, 2, 1) : cv_mask(2, 1, 1);
}
__host__ __device__ constexpr uint32_t kind_mask2(int kd) {    // one plane of the 3D mask
    return (uint32_t)((kd == 0 ? cv_mask(2, 2, 1) : kd == 1 ? cv_mask(1, 1, 1) : kd == 2 ? cv_mask(1, 2, 1) : cv_mask(2, 1, 1)) & 0xffffu);
}

__global__ void __launch_bounds__(256) k_fractions2d(Layout L, const double* __restrict__ phiL,
                                                     const double* __restrict__ phiS, DevArrays D) {
    __shared__ CutSmem<2> sm;
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 8;
    const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
    const int Lx = 2 * L.nx + 3, Ly = 2 * L.ny + 3;
    if (threadIdx.x == 0 && threadIdx.y == 0) sm.ncut = 0;
    __syncthreads();
    if (i <= L.nx && j <= L.ny) {
        const int64_t o = L.off(i + 1, j + 1, 0);
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const double* phi = w ? phiS : phiL;
            uint32_t m = 0;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int a = min(2 * i + (e & 3), Lx - 1), b = min(2 * j + (e >> 2), Ly - 1);   // clipped: no kind reads it
                m |= (uint32_t)dneg(phi[(int64_t)b * Lx + a]) << e;
            }
#pragma unroll
            for (int kd = 0; kd < 4; ++kd) {
                if (!exists2(kd, i, j, L.nx, L.ny)) continue;
                const uint32_t part = m & kind_mask2(kd);
                if (part != 0 && part != kind_mask2(kd)) {
                    sm.list[atomicAdd(&sm.ncut, 1)] = (unsigned short)((threadIdx.x + 32 * threadIdx.y) | kd << 8 | w << 11);
                } else if (w == 0) {
                    D.WL[kd][o] = part ? 1.0 : 0.0;
                } else {
                    D.WF[kd][o] = part ? 0.0 : 1.0;
                }
            }
        }
    }
    __syncthreads();
    cut_fractions<2>(
        sm, Lx, 0,
        [&](int e) {
            const int kd = (e >> 8) & 7, si = i0 + (e & 31), sj = j0 + ((e >> 5) & 7);
            return ((e >> 11) ? phiS : phiL) + (int64_t)(2 * sj + c_off2[kd][1]) * Lx + (2 * si + c_off2[kd][0]);
        },
        [&](int e, double f) {
            const int kd = (e >> 8) & 7;
            const int64_t o = L.off(i0 + (e & 31) + 1, j0 + ((e >> 5) & 7) + 1, 0);
            if (e >> 11) D.WF[kd][o] = 1.0 - f;
            else D.WL[kd][o] = f;
        });
}

// Sign bits of the 3D lattices: bit a % 32 of word a / 32 of lattice row
// (b, c) is 1 where phi is negative (0 past the row's end); nw words per row.
// One coalesced pass over both level sets; the slots' block tests then read
// bits.  (Each slot reading its 64 values of both, overlapping eightfold, was
// bound by the load pipe.)
__host__ __device__ inline int sign_words(int nx) { return 2 * (nx / 32) + 3; }
__global__ void __launch_bounds__(256) k_sign_bits(const double* __restrict__ phiL, const double* __restrict__ phiS,
                                                   int Lx, int64_t rows, int nw, uint32_t* __restrict__ bits) {
    const double* phi = blockIdx.y ? phiS : phiL;
    uint32_t* out = bits + (int64_t)blockIdx.y * rows * nw;
    const int lane = threadIdx.x & 31;
    const int64_t n = rows * nw, w0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 8;
    if (w0 >= n) return;
    int64_t row = w0 / nw;
    int w = (int)(w0 - row * nw);
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int a = 32 * w + lane;
        v[q] = w0 + q < n && a < Lx ? phi[row * Lx + a] : 0.0;
        if (++w == nw) { w = 0; ++row; }
    }
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint32_t m = __ballot_sync(0xffffffffu, dneg(v[q]));
        if (lane == q) mine = m;
    }
    if (lane < 8 && w0 + lane < n) out[w0 + lane] = mine;
}

// One warp per 32 slots of a row: the 16 lattice rows of their blocks are
// combined (OR and AND of three words), which settles the slots whose block
// has one sign; the others build their mask and list their cut CVs.
__global__ void __launch_bounds__(256) k_fractions3d(Layout L, const double* __restrict__ phiL,
                                                     const double* __restrict__ phiS,
                                                     const uint32_t* __restrict__ bits, int nw, DevArrays D) {
    __shared__ CutSmem<3> sm;
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 8;
    const int i = i0 + threadIdx.x, j = j0 + threadIdx.y, k = blockIdx.z;
    const int lane = threadIdx.x;
    const int Lx = 2 * L.nx + 3, Ly = 2 * L.ny + 3, Lz = 2 * L.nz + 3;
    if (threadIdx.x == 0 && threadIdx.y == 0) sm.ncut = 0;
    __syncthreads();
    if (j <= L.ny) {                                      // whole warps
        const bool inside = i <= L.nx;
        const int64_t o = inside ? L.off(i + 1, j + 1, k + 1) : 0;
        const int db = (lane & 15) >> 2, dc = (lane & 15) & 3;
        const bool row_ok = lane < 16 && 2 * j + db < Ly && 2 * k + dc < Lz;
        const int wx = 2 * i0 / 32;
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const uint32_t* bw = bits + (int64_t)w * Ly * Lz * nw;
            uint32_t any[3], all[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const uint32_t v = row_ok ? bw[((int64_t)(2 * k + dc) * Ly + (2 * j + db)) * nw + wx + q] : 0u;
                // bits past the row's end count as negative in the AND
                const int past = 32 * (wx + q + 1) - Lx;
                const uint32_t pad = past <= 0 ? 0u : past >= 32 ? 0xffffffffu : ~(0xffffffffu >> past);
                any[q] = __reduce_or_sync(0xffffffffu, v);
                all[q] = __reduce_and_sync(0xffffffffu, row_ok ? v | pad : 0xffffffffu);
            }
            if (!inside) continue;
            const int sh = 2 * lane;                      // the slot's four bits start here
            const uint32_t a4 = (sh < 32 ? __funnelshift_r(any[0], any[1], sh) : __funnelshift_r(any[1], any[2], sh - 32)) & 15u;
            const uint32_t n4 = (sh < 32 ? __funnelshift_r(all[0], all[1], sh) : __funnelshift_r(all[1], all[2], sh - 32)) & 15u;
            uint64_t m = 0;
            const bool uniform = a4 == 0 || n4 == 15u;
            if (a4 != 0) {
                if (n4 == 15u) {
                    m = ~0ull;
                } else {
                    const int ws = 2 * i / 32;
#pragma unroll 4
                    for (int e = 0; e < 16; ++e) {
                        const int b = min(2 * j + (e & 3), Ly - 1), c = min(2 * k + (e >> 2), Lz - 1);   // clipped: no kind reads it
                        const uint32_t* r = bw + ((int64_t)c * Ly + b) * nw + ws;
                        m |= (uint64_t)(__funnelshift_r(r[0], r[1], (2 * i) & 31) & 15u) << (4 * e);
                    }
                }
            }
#pragma unroll
            for (int kd = 0; kd < 7; ++kd) {
                if (!exists3(kd, i, j, k, L.nx, L.ny, L.nz)) continue;
                constexpr uint64_t masks[7] = {kind_mask3(0), kind_mask3(1), kind_mask3(2), kind_mask3(3),
                                               kind_mask3(4), kind_mask3(5), kind_mask3(6)};
                const uint64_t part = m & masks[kd];
                if (!uniform && part != 0 && part != masks[kd]) {
                    sm.list[atomicAdd(&sm.ncut, 1)] = (unsigned short)((lane + 32 * threadIdx.y) | kd << 8 | w << 11);
                } else if (w == 0) {
                    D.WL[kd][o] = part ? 1.0 : 0.0;
                } else {
                    D.WF[kd][o] = part ? 0.0 : 1.0;
                }
            }
        }
    }
    __syncthreads();
    cut_fractions<3>(
        sm, Lx, (int64_t)Lx * Ly,
        [&](int e) {
            const int kd = (e >> 8) & 7, si = i0 + (e & 31), sj = j0 + ((e >> 5) & 7);
            return ((e >> 11) ? phiS : phiL) +
                   ((int64_t)(2 * k + c_off3[kd][2]) * Ly + (2 * sj + c_off3[kd][1])) * Lx + (2 * si + c_off3[kd][0]);
        },
        [&](int e, double f) {
            const int kd = (e >> 8) & 7;
            const int64_t o = L.off(i0 + (e & 31) + 1, j0 + ((e >> 5) & 7) + 1, k + 1);
            if (e >> 11) D.WF[kd][o] = 1.0 - f;
            else D.WL[kd][o] = f;
        });
}

// zero-fluid-weight multiplier: W_L > 0 and W_F == 0 (Section 8, solid side).
// (These kernels test signs on the integer pipe: the FP64 compares of every
// slot's neighbours were most of their time.)
__device__ __forceinline__ bool zwm(const DevArrays& D, int kind, int64_t o) {
    return wpos(D.WL[kind][o]) && is_zero(D.WF[kind][o]);
}

// ---- kernel 2: faces ----------------------------------------------------------
// Adjacent multiplier samples of each face (through D and G^T):
//   2D u(i,j): cells (i-1,j),(i,j); nodes (i,j),(i,j+1)
//   2D v(i,j): cells (i,j-1),(i,j); nodes (i,j),(i+1,j)
//   3D u: cells (i-1),(i); exy (i,j),(i,j+1); exz (i,j,k),(i,j,k+1)
//   3D v: cells (j-1),(j); exy (i,j),(i+1,j); eyz (i,j,k),(i,j,k+1)
//   3D w: cells (k-1),(k); exz (i,j,k),(i+1,j,k); eyz (i,j,k),(i,j+1,k)
// wl_min floors the liquid fraction of live faces where it is their mass
// (K and the recovery coefficient); 0 keeps the fractions as computed.
__global__ void k_faces2d(Layout L, double dt, double wl_min, const double* rho_u, const double* rho_v,
                          const double* ubc_u, const double* ubc_v, DevArrays D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i > L.nx || j > L.ny) return;
    for (int d = 0; d < 2; ++d) {
        int kind = 2 + d;
        if (!exists2(kind, i, j, L.nx, L.ny)) continue;
        int64_t o = L.off(i + 1, j + 1, 0);
        uint8_t fl = F_EXISTS;
        double wf = D.WF[kind][o], wl = D.WL[kind][o];
        bool wall = d == 0 ? (i == 0 || i == L.nx) : (j == 0 || j == L.ny);
        if (wall) { fl |= F_WALL; wf = 0.0; }
        if (wpos(wf)) {
            bool inval;
            if (d == 0)
                inval = (i > 0 && zwm(D, 0, L.off(i, j + 1, 0))) || (i < L.nx && zwm(D, 0, o)) ||
                        zwm(D, 1, o) || zwm(D, 1, L.off(i + 1, j + 2, 0));
            else
                inval = (j > 0 && zwm(D, 0, L.off(i + 1, j, 0))) || (j < L.ny && zwm(D, 0, o)) ||
                        zwm(D, 1, o) || zwm(D, 1, L.off(i + 2, j + 1, 0));
            if (inval) { fl |= F_INVALID; wf = 0.0; }
        }
        double K = 0.0, rec = 0.0;
        if (wpos(wf) && wpos(wl)) {
            fl |= F_LIVE;
            double rho = (d == 0 ? rho_u : rho_v)[fidx2(kind, i, j, L.nx, L.ny)];
            double wm = fmax(wl, wl_min);
            K = (dt * wf) / (rho * wm);
            rec = dt / (rho * wm);
        } else if (wpos(wf)) {
            fl |= F_BAD;
        }
        D.fflag[d][o] = fl;
        D.effWF[d][o] = wf;
        D.K64[d][o] = K;
        D.rec[d][o] = rec;
        D.ubc[d][o] = (d == 0 ? ubc_u : ubc_v)[fidx2(kind, i, j, L.nx, L.ny)];
    }
}

__global__ void k_faces3d(Layout L, double dt, double wl_min, Ptr3 rho, Ptr3 ubc, DevArrays D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    int k = blockIdx.z;
    if (i > L.nx || j > L.ny || k > L.nz) return;
    int64_t o = L.off(i + 1, j + 1, k + 1);
    for (int d = 0; d < 3; ++d) {
        int kind = 1 + d;
        if (!exists3(kind, i, j, k, L.nx, L.ny, L.nz)) continue;
        uint8_t fl = F_EXISTS;
        double wf = D.WF[kind][o], wl = D.WL[kind][o];
        bool wall = d == 0 ? (i == 0 || i == L.nx) : d == 1 ? (j == 0 || j == L.ny) : (k == 0 || k == L.nz);
        if (wall) { fl |= F_WALL; wf = 0.0; }
        if (wpos(wf)) {
            bool inval = false;
            // cells on both sides along d (interior faces: both exist)
            int64_t om = d == 0 ? L.off(i, j + 1, k + 1) : d == 1 ? L.off(i + 1, j, k + 1) : L.off(i + 1, j + 1, k);
            inval |= zwm(D, 0, om) || zwm(D, 0, o);
            if (d == 0) {
                inval |= zwm(D, 4, o) || zwm(D, 4, L.off(i + 1, j + 2, k + 1));
                inval |= zwm(D, 5, o) || zwm(D, 5, L.off(i + 1, j + 1, k + 2));
            } else if (d == 1) {
                inval |= zwm(D, 4, o) || zwm(D, 4, L.off(i + 2, j + 1, k + 1));
                inval |= zwm(D, 6, o) || zwm(D, 6, L.off(i + 1, j + 1, k + 2));
            } else {
                inval |= zwm(D, 5, o) || zwm(D, 5, L.off(i + 2, j + 1, k + 1));
                inval |= zwm(D, 6, o) || zwm(D, 6, L.off(i + 1, j + 2, k + 1));
            }
            if (inval) { fl |= F_INVALID; wf = 0.0; }
        }
        double K = 0.0, rec = 0.0;
        int64_t fi = fidx3(kind, i, j, k, L.nx, L.ny, L.nz);
        if (wpos(wf) && wpos(wl)) {
            fl |= F_LIVE;
            double r = rho.p[d][fi];
            double wm = fmax(wl, wl_min);
            K = (dt * wf) / (r * wm);
            rec = dt / (r * wm);
        } else if (wpos(wf)) {
            fl |= F_BAD;
        }
        D.fflag[d][o] = fl;
        D.effWF[d][o] = wf;
        D.K64[d][o] = K;
        D.rec[d][o] = rec;
        D.ubc[d][o] = ubc.p[d][fi];
    }
}

// ---- kernel 3: unknown validity and coefficients -------------------------------
__device__ __forceinline__ void face_state(const DevArrays& D, int d, int64_t o, bool& bad, bool& live) {
    uint8_t f = D.fflag[d][o];
    bad |= (f & F_BAD) != 0;
    live |= (f & F_LIVE) != 0;
}

__global__ void k_unknowns2d(Layout L, double inv_h, const double* mu_c, const double* mu_n, DevArrays D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i > L.nx || j > L.ny) return;
    int64_t o = L.off(i + 1, j + 1, 0);
    double* a_c = D.coef64 + 0 * L.stride;
    double* a_n = D.coef64 + 1 * L.stride;
    double* d_c = D.coef64 + 2 * L.stride;
    double* d_n = D.coef64 + 3 * L.stride;
    // cell: faces u(i), u(i+1), v(j), v(j+1)
    if (i < L.nx && j < L.ny) {
        bool bad = false, live = false;
        face_state(D, 0, o, bad, live);
        face_state(D, 0, L.off(i + 2, j + 1, 0), bad, live);
        face_state(D, 1, o, bad, live);
        face_state(D, 1, L.off(i + 1, j + 2, 0), bad, live);
        double wl = D.WL[0][o], wf = D.WF[0][o];
        bool act = wpos(wl) && !bad && live;
        a_c[o] = act ? wl * inv_h : 0.0;
        d_c[o] = act ? (wl * wf) / mu_c[fidx2(0, i, j, L.nx, L.ny)] : 1.0;
        D.act[0][o] = act;
    }
    // node: faces u(i, j-1), u(i, j), v(i-1, j), v(i, j)
    {
        bool bad = false, live = false;
        if (j > 0) face_state(D, 0, L.off(i + 1, j, 0), bad, live);
        if (j < L.ny) face_state(D, 0, o, bad, live);
        if (i > 0) face_state(D, 1, L.off(i, j + 1, 0), bad, live);
        if (i < L.nx) face_state(D, 1, o, bad, live);
        double wl = D.WL[1][o], wf = D.WF[1][o];
        bool act = wpos(wl) && !bad && (wpos(wf) || live);
        a_n[o] = act ? wl * inv_h : 0.0;
        d_n[o] = act ? (wl * wf) / mu_n[fidx2(1, i, j, L.nx, L.ny)] : 1.0;
        D.act[1][o] = act;
    }
}

__global__ void k_unknowns3d(Layout L, double inv_h, Ptr4 mu, DevArrays D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    int k = blockIdx.z;
    if (i > L.nx || j > L.ny || k > L.nz) return;
    int64_t o = L.off(i + 1, j + 1, k + 1);
    // coefficient fields: 0 a_c, 1 a_xy, 2 a_xz, 3 a_yz, 4 d_c, 5 d_xy, 6 d_xz, 7 d_yz
    auto A = [&](int f) { return D.coef64 + (int64_t)f * L.stride; };
    int64_t ox = L.off(i + 2, j + 1, k + 1), oy = L.off(i + 1, j + 2, k + 1), oz = L.off(i + 1, j + 1, k + 2);
    int64_t mx = L.off(i, j + 1, k + 1), my = L.off(i + 1, j, k + 1), mz = L.off(i + 1, j + 1, k);
    if (i < L.nx && j < L.ny && k < L.nz) {
        bool bad = false, live = false;
        face_state(D, 0, o, bad, live); face_state(D, 0, ox, bad, live);
        face_state(D, 1, o, bad, live); face_state(D, 1, oy, bad, live);
        face_state(D, 2, o, bad, live); face_state(D, 2, oz, bad, live);
        double wl = D.WL[0][o], wf = D.WF[0][o];
        bool act = wpos(wl) && !bad && live;
        A(0)[o] = act ? wl * inv_h : 0.0;
        A(4)[o] = act ? (wl * wf) / mu.p[0][fidx3(0, i, j, k, L.nx, L.ny, L.nz)] : 1.0;
        D.act[0][o] = act;
    }
    // exy (z-edge): u(i,j-1,k), u(i,j,k), v(i-1,j,k), v(i,j,k)
    if (k < L.nz) {
        bool bad = false, live = false;
        if (j > 0) face_state(D, 0, my, bad, live);
        if (j < L.ny) face_state(D, 0, o, bad, live);
        if (i > 0) face_state(D, 1, mx, bad, live);
        if (i < L.nx) face_state(D, 1, o, bad, live);
        double wl = D.WL[4][o], wf = D.WF[4][o];
        bool act = wpos(wl) && !bad && (wpos(wf) || live);
        A(1)[o] = act ? wl * inv_h : 0.0;
        A(5)[o] = act ? (wl * wf) / mu.p[1][fidx3(4, i, j, k, L.nx, L.ny, L.nz)] : 1.0;
        D.act[1][o] = act;
    }
    // exz (y-edge): u(i,j,k-1), u(i,j,k), w(i-1,j,k), w(i,j,k)
    if (j < L.ny) {
        bool bad = false, live = false;
        if (k > 0) face_state(D, 0, mz, bad, live);
        if (k < L.nz) face_state(D, 0, o, bad, live);
        if (i > 0) face_state(D, 2, mx, bad, live);
        if (i < L.nx) face_state(D, 2, o, bad, live);
        double wl = D.WL[5][o], wf = D.WF[5][o];
        bool act = wpos(wl) && !bad && (wpos(wf) || live);
        A(2)[o] = act ? wl * inv_h : 0.0;
        A(6)[o] = act ? (wl * wf) / mu.p[2][fidx3(5, i, j, k, L.nx, L.ny, L.nz)] : 1.0;
        D.act[2][o] = act;
    }
    // eyz (x-edge): v(i,j,k-1), v(i,j,k), w(i,j-1,k), w(i,j,k)
    if (i < L.nx) {
        bool bad = false, live = false;
        if (k > 0) face_state(D, 1, mz, bad, live);
        if (k < L.nz) face_state(D, 1, o, bad, live);
        if (j > 0) face_state(D, 2, my, bad, live);
        if (j < L.ny) face_state(D, 2, o, bad, live);
        double wl = D.WL[6][o], wf = D.WF[6][o];
        bool act = wpos(wl) && !bad && (wpos(wf) || live);
        A(3)[o] = act ? wl * inv_h : 0.0;
        A(7)[o] = act ? (wl * wf) / mu.p[3][fidx3(6, i, j, k, L.nx, L.ny, L.nz)] : 1.0;
        D.act[3][o] = act;
    }
}

// ---- kernel 4: Jacobi inverse diagonal, reduced-precision copies, tile flags
// Conversions run on the FP64 pipe; away from the liquid every value is 0 or
// 1, which the integer pipe recognises (256^3 column: 1.39 -> 1.04 ms).
__device__ __forceinline__ bool is_one(double v) { return __double_as_longlong(v) == 0x3ff0000000000000LL; }
__device__ __forceinline__ float narrow(double v) {
    if (__double_as_longlong(v) == 0) return 0.f;
    return is_one(v) ? 1.f : (float)v;
}
__device__ __forceinline__ __nv_bfloat16 narrow16(double v) {
    if (__double_as_longlong(v) == 0) return __ushort_as_bfloat16(0);
    return is_one(v) ? __ushort_as_bfloat16(0x3f80) : __double2bfloat16(v);
}
// (All of a slot's loads are issued before its first store, which might
// alias them as far as the compiler can tell.)  The K fields are fields 4, 5
// (3D: 8, 9, 10) of coef64.
__global__ void __launch_bounds__(256) k_finish2d(Layout L, DevArrays D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i > L.nx || j > L.ny) return;
    const int64_t o = L.off(i + 1, j + 1, 0), S = L.stride;
    double v[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) v[f] = D.coef64[f * S + o];
    const bool cell = i < L.nx && j < L.ny;
    const bool act_c = cell && D.act[0][o], act_n = D.act[1][o];
    const double *Ku = D.K64[0], *Kv = D.K64[1];
    const double ac = v[0], an = v[1], dc = v[2], dn = v[3];
    double m[3] = {cell ? 1.0 : 0.0, 1.0, cell ? 1.0 : 0.0};
    if (act_c) {
        const double sK = Ku[o] + Ku[L.off(i + 2, j + 1, 0)] + Kv[o] + Kv[L.off(i + 1, j + 2, 0)];
        m[0] = 1.0 / (dc + ac * ac * sK);
        m[2] = 1.0 / (ac * ac * sK);
    }
    if (act_n) {
        const double sK = Ku[o] + Ku[L.off(i + 1, j, 0)] + Kv[o] + Kv[L.off(i, j + 1, 0)];
        m[1] = 1.0 / (dn + an * an * sK);
    }
    uint32_t h[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        D.coef32[f * S + o] = narrow(v[f]);
        const __nv_bfloat16 b = narrow16(v[f]);
        D.coef16[f * S + o] = b;
        h[f] = __bfloat16_as_ushort(b);
    }
    // the same BF16 values in pairs (a_c, a_n), (d_c, d_n), (K_u, K_v)
#pragma unroll
    for (int k = 0; k < 3; ++k) D.pair16[k * S + o] = h[2 * k] | (h[2 * k + 1] << 16);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        D.minv64[f * S + o] = m[f];
        D.minv32[f * S + o] = narrow(m[f]);
    }
    if (act_c || act_n) {
        int c = i + 1, r = j + 1;
        D.tile_flag[(r / TY2) * L.ntx + c / TX] = 1;
        D.tile_flag4[(r / 4) * L.ntx + c / TX] = 1;
    }
}

__global__ void __launch_bounds__(256) k_finish3d(Layout L, DevArrays D) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    int k = blockIdx.z;
    if (i > L.nx || j > L.ny || k > L.nz) return;
    const int64_t o = L.off(i + 1, j + 1, k + 1), S = L.stride;
    double v[11];
#pragma unroll
    for (int f = 0; f < 11; ++f) v[f] = D.coef64[f * S + o];
    const bool ex[4] = {i < L.nx && j < L.ny && k < L.nz, k < L.nz, j < L.ny, i < L.nx};
    bool act[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) act[q] = D.act[q][o];      // zero where the site does not exist
    // unknown fields: 0 txx, 1 tyy, 2 txy, 3 txz, 4 tyz, 5 p
    double m[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) m[f] = ex[f < 2 || f == 5 ? 0 : f - 1] ? 1.0 : 0.0;
    if (act[0] || act[1] || act[2] || act[3]) {
        const double *Ku = D.K64[0], *Kv = D.K64[1], *Kw = D.K64[2];
        const int64_t ox = L.off(i + 2, j + 1, k + 1), oy = L.off(i + 1, j + 2, k + 1), oz = L.off(i + 1, j + 1, k + 2);
        const int64_t mx = L.off(i, j + 1, k + 1), my = L.off(i + 1, j, k + 1), mz = L.off(i + 1, j + 1, k);
        const double ku = v[8], kv = v[9], kw = v[10];
        if (act[0]) {
            const double ac = v[0], dc = v[4], a2 = ac * ac;
            const double su = ku + Ku[ox], sv = kv + Kv[oy], sw = kw + Kw[oz];
            m[0] = 1.0 / (dc + a2 * (su + sw));
            m[1] = 1.0 / (dc + a2 * (sv + sw));
            m[5] = 1.0 / (a2 * (su + sv + sw));
        }
        if (act[1]) m[2] = 1.0 / (v[5] + v[1] * v[1] * (Ku[my] + ku + Kv[mx] + kv));
        if (act[2]) m[3] = 1.0 / (v[6] + v[2] * v[2] * (Ku[mz] + ku + Kw[mx] + kw));
        if (act[3]) m[4] = 1.0 / (v[7] + v[3] * v[3] * (Kv[mz] + kv + Kw[my] + kw));
        int c = i + 1, r = j + 1, q = k + 1;
        D.tile_flag[((int64_t)(q / TZ3) * L.nty + r / TY3) * L.ntx + c / TX] = 1;
    }
    uint32_t h[8];
#pragma unroll
    for (int f = 0; f < 11; ++f) {
        D.coef32[f * S + o] = narrow(v[f]);
        const __nv_bfloat16 b = narrow16(v[f]);
        D.coef16[f * S + o] = b;
        if (f < 8) h[f] = __bfloat16_as_ushort(b);
    }
    // the same BF16 values in fours: (a_c, a_xy, a_xz, a_yz), (d_c, d_xy, d_xz, d_yz)
#pragma unroll
    for (int w = 0; w < 2; ++w)
        D.quad16[w * S + o] = make_uint2(h[4 * w] | (h[4 * w + 1] << 16), h[4 * w + 2] | (h[4 * w + 3] << 16));
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        D.minv64[f * S + o] = m[f];
        D.minv32[f * S + o] = narrow(m[f]);
    }
}

// Tile mask of every 3D apply unit (32 x 8 slots x zt tile layers; bit
// dy + 2 dz), tiles past the tile grid counted inactive.
__global__ void k_unit_masks(Layout L, int zt, const uint8_t* __restrict__ tflag, uint8_t* __restrict__ umask,
                             int nunits) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nunits) return;
    const int nuy = units_y(L.nty);
    const int ux = u % L.ntx, rest = u / L.ntx, uy = rest % nuy, uz = rest / nuy;
    unsigned m = 0;
    for (int dz = 0; dz < zt; ++dz)
        for (int dy = 0; dy < 2; ++dy) {
            const int ty = 2 * uy + dy, tz = zt * uz + dz;
            if (ty < L.nty && tz < L.ntz && tflag[((int64_t)tz * L.nty + ty) * L.ntx + ux]) m |= 1u << (dy + 2 * dz);
        }
    umask[u] = (uint8_t)m;
}

// Ordered compaction of the tile flags (one block; tile counts are small).
__global__ void k_compact_tiles(const uint8_t* flag, int n, int* list, int* count) {
    __shared__ int warp_tot[32];
    __shared__ int base;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int start = 0; start < n; start += blockDim.x) {
        int t = start + threadIdx.x;
        int f = (t < n && flag[t]) ? 1 : 0;
        unsigned m = __ballot_sync(0xffffffffu, f);
        int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        int before = __popc(m & ((1u << lane) - 1u));
        if (lane == 0) warp_tot[w] = __popc(m);
        __syncthreads();
        int off = 0;
        for (int q = 0; q < w; ++q) off += warp_tot[q];
        if (f) list[base + off + before] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot += warp_tot[q];
            base += tot;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = base;
}

size_t sign_bits_bytes(const Layout& L) {
    return L.dim == 3 ? sizeof(uint32_t) * 2 * (size_t)(2 * L.ny + 3) * (2 * L.nz + 3) * sign_words(L.nx) : 4;
}

cudaError_t launch_build_weights(Ctx* c, const double* phiL, const double* phiS, const double* const* rho,
                                 const double* const* mu, const double* const* ubc) {
    const Layout& L = c->L;
    cudaStream_t s = c->stream;
    DevArrays D = c->dev_arrays();
    cudaError_t e;
    cudaGetLastError();   // a stale, non-sticky error from earlier work is not this call's
    // Pads, guards and samples that do not exist were zeroed when the block was
    // allocated and no kernel writes them; every build writes all the others.
    // Only the tile flags are set without being cleared.  (Zeroing the whole
    // block again was 7.9 GB on a 256^3 grid.)
    if ((e = c->zero_tile_flags()) != cudaSuccess) return e;
    dim3 blk(32, 8);
    if (L.dim == 2) {
        dim3 grd((L.nx + 1 + 31) / 32, (L.ny + 1 + 7) / 8);
        k_fractions2d<<<grd, blk, 0, s>>>(L, phiL, phiS, D);
        k_faces2d<<<grd, blk, 0, s>>>(L, c->g.dt, c->min_face_liquid, rho[0], rho[1], ubc[0], ubc[1], D);
        k_unknowns2d<<<grd, blk, 0, s>>>(L, 1.0 / c->g.h, mu[0], mu[1], D);
        k_finish2d<<<grd, blk, 0, s>>>(L, D);
    } else {
        dim3 grd((L.nx + 1 + 31) / 32, (L.ny + 1 + 7) / 8, L.nz + 1);
        Ptr3 r3{{rho[0], rho[1], rho[2]}}, u3{{ubc[0], ubc[1], ubc[2]}};
        Ptr4 m4{{mu[0], mu[1], mu[2], mu[3]}};
        const int nw = sign_words(L.nx);
        const int64_t rows = (int64_t)(2 * L.ny + 3) * (2 * L.nz + 3);
        k_sign_bits<<<dim3((unsigned)((rows * nw + 63) / 64), 2), 256, 0, s>>>(phiL, phiS, 2 * L.nx + 3, rows, nw, c->sign_bits);
        k_fractions3d<<<grd, blk, 0, s>>>(L, phiL, phiS, c->sign_bits, nw, D);
        k_faces3d<<<grd, blk, 0, s>>>(L, c->g.dt, c->min_face_liquid, r3, u3, D);
        k_unknowns3d<<<grd, blk, 0, s>>>(L, 1.0 / c->g.h, m4, D);
        k_finish3d<<<grd, blk, 0, s>>>(L, D);
    }
    k_compact_tiles<<<1, 1024, 0, s>>>(D.tile_flag, c->ntiles_all, c->tiles, c->d_ntiles);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(&c->ntiles_active, c->d_ntiles, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return e;
    if (L.dim == 3) {
        // units of 4 tile layers (16 planes) when there are enough of them to
        // fill the device a few times over, else of one layer: a thin liquid
        // region has too few deep units to keep every SM busy.  CG-mode apply of
        // boxes, us at depth 1 and 4, FP64 and FP32: 64^3 (867 active tiles) 106 and
        // 148, 27.0 and 26.9; 96^3 (2,500) 280 and 321, 62.0 and 62.5; 128^3 (5,445)
        // 565 and 583, 112 and 103; 160^3 (10,086) 1013 and 924, 191 and 163; 192^3
        // (16,807) 1660 and 1458, 301 and 245; the thin column of a 256^3 grid (462)
        // is 1.35 times faster at depth 1.  The line lies at 96 tiles per SM (14,592),
        // above the crossing, where it was set with six CTAs of an earlier FP32 kernel
        // per SM; depth 2 is the faster one from 5,000 to 10,000 tiles (128^3 FP32 99
        // us).  Moving it reorders the dots' partial sums and so changes iterates.
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        // (12 deep units of 2 ZT_MAX tiles per SM)
        c->unit_zt = c->ntiles_active >= 2 * (2 * ZT_MAX) * 6 * std::max(sms, 1) ? ZT_MAX : 1;
        const int nu = L.ntx * units_y(L.nty) * units_z(L.ntz, c->unit_zt);
        k_unit_masks<<<(nu + 255) / 256, 256, 0, s>>>(L, c->unit_zt, D.tile_flag, D.unit_mask, nu);
        k_compact_tiles<<<1, 1024, 0, s>>>(D.unit_mask, nu, c->units, c->d_nunits);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(&c->nunits_active, c->d_nunits, sizeof(int), cudaMemcpyDeviceToHost, s)) !=
            cudaSuccess)
            return e;
    }
    return cudaStreamSynchronize(s);
}

}  // namespace stk
