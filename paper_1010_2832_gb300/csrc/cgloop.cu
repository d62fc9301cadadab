// Jacobi-PCG inner solves of small 2D systems in one cooperative kernel.
//
// A CG iteration of a small system is a chain of short dependent steps: with a
// kernel for each, most of its time is launches, block scheduling and the
// two-stage reductions (32^2 liquid disk, FP64: 18 us an iteration for 8 tiles
// of work).  Here one CTA owns one tile for the whole solve and an iteration
// has two grid-wide exchanges (grid_gather.cuh), p.q and then r.z with r.r.
//
// A CTA (k_cgloop2d) owns 32 x TY slots, one per thread.  The slot's x, r,
// p, Jacobi weight and coefficients, the face coefficients and the p of the
// halo stay in registers; the halo's p follows the same recurrence
// p = z + beta p, so only z of the tile's boundary goes through memory.  TY is
// 8 for FP32; FP64 (two operations per clock and SM on this part) takes the
// smaller of 2 and 4 rows whose CTAs fit (about 300), spreading the arithmetic
// over more SMs, and three more warps per CTA for the halo, since a warp's FP64
// instruction takes 64 clocks.  Rows of 32 slots without an active unknown or a
// residual do no arithmetic.
//
// The arithmetic of a slot is that of k_apply2d(_v4) and
// k_cg_update, and the dots are summed in those kernels' order, so the iterates
// are theirs bit for bit (CG on these systems is sensitive: another order of
// summation moved one test's iteration count from 11,880 to 18,951).
#include <algorithm>
#include <atomic>
#include "internal.cuh"
#include "ctx.cuh"
#include "apply2d_tile.cuh"
#include "grid_gather.cuh"
#include "loop_common.cuh"

namespace stk {


// ------------------------------- 2D -----------------------------------------
// Threads of a CTA: the slots, and in FP64 three warps for the halo.
template <class T, int TY> constexpr int loop2_threads() { return 32 * TY + (sizeof(T) == 8 ? 96 : 0); }
template <class T, int TY> struct Loop2Smem {
    static constexpr int NT = loop2_threads<T, TY>();
    T U[TY + 2][TX + 2], V[TY + 2][TX + 2], N[TY + 2][TX + 2];
    T Zu[TY + 1][TX + 1], Zv[TY + 1][TX + 1];
    T P[TY == 8 ? 3 : 1][TY == 8 ? TY : 1][TX], Y[TY == 8 ? 3 : 1][TY == 8 ? TY : 1][TX];   // FP32: p and A p for the dot
    WarpSums<T, TY> sums;
    typename GridGather<NT>::Smem g;
    double vals[GATHER_DIRECT * (TY == 8 ? 2 : 2 * TY)];       // a larger grid's reducer: dynamic shared memory
};

// WAIT_TEST: the options' hook; no CTA posts its z.
template <class T, class C, int TY, bool WAIT_TEST>
__global__ void __launch_bounds__(loop2_threads<T, TY>(), TY == 2 ? 3 : 2) k_cgloop2d(Layout L, const int* __restrict__ tiles, int ntiles,
                                                      Coef<C> cf, const double* __restrict__ r64,
                                                      const T* __restrict__ minv, T* __restrict__ xout,
                                                      unsigned long long* zw, CgScalars* sc, unsigned long long* slots) {
    static_assert(sizeof(T) == 8 ? TY < 8 : TY == 8, "FP32: a tile per CTA; FP64: a part of one");
    using Z = ZWords<T>;
    constexpr int NT = loop2_threads<T, TY>(), NS = 32 * TY;      // threads; slots
    constexpr int SUB = TY2 / TY;                          // CTAs per tile
    constexpr int HALO = 2 * (TX + 2) + 2 * TY;
    static_assert(HALO <= (NT > NS ? NT - NS : NT), "one halo position per thread");
    constexpr int NF = (TY + 1) * (TX + 1), FPT = (NF + NT - 1) / NT;
    constexpr int DZ = TY == 8 ? 2 : 2 * TY, DP = TY == 8 ? 2 : TY;     // doubles published: r.z and r.r; p.q
    __shared__ Loop2Smem<T, TY> sm;
    extern __shared__ __align__(16) unsigned char dyn[];
    const int t = threadIdx.x, tx = t & 31, ty = t >> 5;
    const int workers = ntiles * SUB;
    constexpr int POLLS = WAIT_TEST ? GATHER_TEST_POLLS : GATHER_POLLS;
    using Gather = GridGather<NT, POLLS>;
    Gather gather{slots, &sm.g, nullptr, workers};
    gather.vals = gather.direct() ? sm.vals : reinterpret_cast<double*>(dyn);
    const double* vals = gather.vals;
    const double tol_rel = sc->tol_rel;
    const int max_iter = sc->max_iter;
    // Block sums of the separate kernels.  k_cg_init, k_cg_update and k_apply2d:
    // a block per tile, its eight rows one after another (FP32: the CTA has
    // added them for r.z and r.r); k_apply2d_v4: four tiles, two warps each.
    auto part_z = [&](int b, int q) -> double {
        if constexpr (TY == 8) {
            return vals[2 * b + q];
        } else {
            double v = vals[b * SUB * DZ + q * TY];
#pragma unroll
            for (int k = 1; k < TY2; ++k) v += vals[(b * SUB + k / TY) * DZ + q * TY + k % TY];
            return v;
        }
    };
    auto part_p = [&](int b, int) -> double {
        double v = vals[8 * b];                            // FP32: two warps of four tiles; FP64: the tile's rows
        for (int q = 8 * b + 1; q < min(8 * b + 8, TY == 8 ? 2 * ntiles : 8 * ntiles); ++q) v += vals[q];
        return v;
    };
    auto none = [] {};
    const int nb_p = TY == 8 ? (ntiles + 3) / 4 : ntiles;
    double scalar;
    bool done;
    if (gather.reducer()) {
        bool ok = gather.template exchange<DZ, 2>(CG_START, nullptr, ntiles, tol_rel, max_iter, part_z, none, scalar, done);
        while (ok && !done) {
            ok = gather.template exchange<DP, 1>(CG_DIRECTION, nullptr, nb_p, tol_rel, max_iter, part_p, none, scalar, done);
            if (ok && !done)
                ok = gather.template exchange<DZ, 2>(CG_STEP, nullptr, ntiles, tol_rel, max_iter, part_z, none, scalar, done);
        }
        gather.finish(sc);
        return;
    }
    const int tile = tiles[blockIdx.x / SUB];
    const int c0 = (tile % L.ntx) * TX, r0 = (tile / L.ntx) * TY2 + (blockIdx.x % SUB) * TY;
    const int64_t S = L.stride;
    // own slot (threads below NS)
    const bool own = NT == NS || t < NS;
    const int64_t o = own ? L.off(c0 + tx, r0 + ty, 0) : 0;
    T ac = T(0), an = T(0), dc = T(0), dn = T(0);
    T x[3], r[3], p[3], m[3];
    const T scale = (T)sc->scale;
    bool busy = false;
    if (own) {
        ac = ld<T, C>(cf.f[0], o); an = ld<T, C>(cf.f[1], o); dc = ld<T, C>(cf.f[2], o); dn = ld<T, C>(cf.f[3], o);
        busy = ac != T(0) || an != T(0);
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        m[f] = own ? minv[f * S + o] : T(0);
        r[f] = own ? (T)(r64[f * S + o] * (double)scale) : T(0);
        x[f] = T(0);
        p[f] = T(0);
        busy = busy || !(r[f] == T(0));
    }
    // a row without an active unknown or a residual stays at zero
    const bool row = __any_sync(0xffffffffu, busy);
    const bool edge = (tx == 0 || tx == TX - 1 || ty == 0 || ty == TY - 1) && !WAIT_TEST;
    unsigned long long* const zown = zw + ((size_t)blockIdx.x * 3 * NS + (own ? t : 0)) * Z::N;      // field f: + f NS N
    // halo position of this thread, and where its owner posts z
    T hp[3] = {T(0), T(0), T(0)}, hac = T(0), han = T(0);
    const unsigned long long* hz = zw;
    int hs = -1;
    {
        const int h = NT > NS ? t - NS : t;
        if (h >= 0 && h < HALO) {
            int jj, ii;
            if (h < TX + 2) { jj = 0; ii = h; }
            else if (h < 2 * (TX + 2)) { jj = TY + 1; ii = h - (TX + 2); }
            else { jj = 1 + (h - 2 * (TX + 2)) / 2; ii = (h & 1) ? TX + 1 : 0; }
            const int c = c0 - 1 + ii, rr = r0 - 1 + jj;
            const int64_t oh = L.off(c, rr, 0);
            hac = ld<T, C>(cf.f[0], oh);
            han = ld<T, C>(cf.f[1], oh);
            if (hac != T(0) || han != T(0)) {              // an active unknown: its tile is in the list
                const int k = tile_place(tiles, ntiles, (rr / TY2) * L.ntx + c / TX);
                if (k >= 0) {
                    hs = jj * (TX + 2) + ii;
                    hz = zw + ((size_t)(k * SUB + (rr % TY2) / TY) * 3 * NS + (rr % TY) * TX + c % TX) * Z::N;
                }
            }
        }
    }
    T ku[FPT], kv[FPT];
#pragma unroll
    for (int q = 0; q < FPT; ++q) {
        const int e = t + q * NT;
        ku[q] = kv[q] = T(0);
        if (e < NF) {
            const int jj = e / (TX + 1), ii = e - jj * (TX + 1);
            ku[q] = ld<T, C>(cf.f[4], L.off(c0 + ii, r0 - 1 + jj, 0));
            kv[q] = ld<T, C>(cf.f[5], L.off(c0 - 1 + ii, r0 + jj, 0));
        }
    }
    // staged values and faces that stay zero are written once
    for (int e = t; e < (TY + 2) * (TX + 2); e += NT) (&sm.U[0][0])[e] = (&sm.V[0][0])[e] = (&sm.N[0][0])[e] = T(0);
    for (int e = t; e < NF; e += NT) (&sm.Zu[0][0])[e] = (&sm.Zv[0][0])[e] = T(0);
    T z[3] = {T(0), T(0), T(0)};
    unsigned tag = 1;                                      // of the z that the next direction uses
    // z = M^-1 r to the neighbours, r.z and r.r to the exchange; x += alpha p
    // while it is under way
    auto residual_dots = [&](int what, T alpha) -> bool {
        Acc<T> rz, rr;
        if (row) {
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                z[f] = m[f] * r[f];
                if (edge) Z::put(zown + (size_t)f * NS * Z::N, tag, z[f]);
                rz.add(r[f], z[f]);
                rr.add(r[f], r[f]);
            }
        }
        if (own) sm.sums.put2(ty, rz, TY + ty, rr, row);
        if constexpr (TY == 8) sm.sums.block2();
        return gather.template exchange<DZ, 2>(
            what, sm.sums.rows, ntiles, tol_rel, max_iter, part_z,
            [&] {
                if (row && what == CG_STEP)
#pragma unroll
                    for (int f = 0; f < 3; ++f) x[f] = x[f] + alpha * p[f];
            },
            scalar, done);
    };
    bool ok = residual_dots(CG_START, T(0));
    while (ok && !done) {
        const T beta = (T)scalar;
        // 1. p = z + beta p on the tile and its halo; stage
        if (row) {
#pragma unroll
            for (int f = 0; f < 3; ++f) p[f] = z[f] + beta * p[f];
            sm.U[ty + 1][tx + 1] = ac * (p[2] - p[0]);
            sm.V[ty + 1][tx + 1] = ac * (p[2] + p[0]);
            sm.N[ty + 1][tx + 1] = an * p[1];
        }
        if (hs >= 0) {
            unsigned long long v[3][Z::N];
            bool here = false;
#pragma unroll 1
            for (int poll = 0; !here && poll < POLLS; ++poll) {
                here = true;
#pragma unroll
                for (int f = 0; f < 3; ++f)
#pragma unroll
                    for (int k = 0; k < Z::N; ++k) v[f][k] = peek_word(hz + (size_t)f * NS * Z::N + k);
#pragma unroll
                for (int f = 0; f < 3; ++f)
#pragma unroll
                    for (int k = 0; k < Z::N; ++k) here = here && (unsigned)(v[f][k] >> 32) == tag;
            }
            ok = ok && here;
#pragma unroll
            for (int f = 0; f < 3; ++f) hp[f] = Z::get(v[f]) + beta * hp[f];
            (&sm.U[0][0])[hs] = hac * (hp[2] - hp[0]);
            (&sm.V[0][0])[hs] = hac * (hp[2] + hp[0]);
            (&sm.N[0][0])[hs] = han * hp[1];
        }
        ok = __syncthreads_and(ok);
        if (!ok) { gather.alive = false; break; }
        ++tag;
        // 2. faces
#pragma unroll
        for (int q = 0; q < FPT; ++q) {
            const int e = t + q * NT;
            const int jj = e / (TX + 1), ii = e - jj * (TX + 1);
            if (ku[q] != T(0))
                sm.Zu[jj][ii] = ku[q] * ((sm.U[jj][ii + 1] - sm.U[jj][ii]) + (sm.N[jj][ii + 1] - sm.N[jj + 1][ii + 1]));
            if (kv[q] != T(0))
                sm.Zv[jj][ii] = kv[q] * ((sm.V[jj + 1][ii] - sm.V[jj][ii]) + (sm.N[jj + 1][ii] - sm.N[jj + 1][ii + 1]));
        }
        __syncthreads();
        // 3. q = A p on the own slot, p.q
        T y[3] = {T(0), T(0), T(0)};
        if (row) {
            const T zu = sm.Zu[ty + 1][tx], zur = sm.Zu[ty + 1][tx + 1], zud = sm.Zu[ty][tx];
            const T zv = sm.Zv[ty][tx + 1], zvu = sm.Zv[ty + 1][tx + 1], zvl = sm.Zv[ty][tx];
            if (ac != T(0)) {
                y[2] = ac * ((zu - zur) + (zv - zvu));
                y[0] = fma_first(dc, p[0], ac, (zur - zu) + (zv - zvu));
            } else {
                y[2] = p[2];
                y[0] = p[0];
            }
            y[1] = fma_first(dn, p[1], an, (zu - zud) + (zv - zvl));
        }
        if constexpr (TY == 8) {
            // (k_apply2d_v4: 64 threads of four slots each)
#pragma unroll
            for (int f = 0; f < 3; ++f) { sm.P[f][ty][tx] = p[f]; sm.Y[f][ty][tx] = y[f]; }
            __syncthreads();
            if (t < 64) {
                Acc<T> acc;
                const int qr = t >> 3, qc = 4 * (t & 7);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int f = 0; f < 3; ++f) acc.add(sm.P[f][qr][qc + i], sm.Y[f][qr][qc + i]);
                sm.sums.put(ty, acc);
            }
            __syncthreads();
            if (t < 32) sm.sums.convert(2);
        } else {
            Acc<T> acc;
#pragma unroll
            for (int f = 0; f < 3; ++f) acc.add(p[f], y[f]);
            if (own) sm.sums.put(ty, acc, row);
        }
        ok = gather.template exchange<DP, 1>(CG_DIRECTION, sm.sums.rows, nb_p, tol_rel, max_iter, part_p, none, scalar, done);
        if (!ok || done) break;
        // 4. r -= alpha q, z = M^-1 r, x += alpha p
        const T alpha = (T)scalar;
        if (row) {
#pragma unroll
            for (int f = 0; f < 3; ++f) r[f] = r[f] - alpha * y[f];
        }
        ok = residual_dots(CG_STEP, alpha);
    }
    if (own)
#pragma unroll
        for (int f = 0; f < 3; ++f) xout[f * S + o] = x[f];
    gather.finish(sc);
}

// ---- launch ------------------------------------------------------------------
constexpr int LOOP2_WORKERS = 303;    // with the reducer, two CTAs on each of 152 SMs
constexpr size_t LOOP2_ZBYTES = sizeof(unsigned long long) * 3 * 256 * LOOP2_WORKERS;    // FP64: 128 threads, two words

// Workers and, past GATHER_DIRECT of them, the reducer.
static int with_reducer(int workers) { return workers <= GATHER_DIRECT ? workers : workers + 1; }

template <class T, class C, int TY, bool WAIT_TEST>
static cudaError_t launch2(Ctx* c, CgWork<T>& w, const T* minv, const Coef<C>& cf, bool* taken) {
    static std::atomic<int> cache[16];
    constexpr int NT = loop2_threads<T, TY>(), D = TY == 8 ? 2 : 2 * TY;
    const int workers = c->ntiles_active * (TY2 / TY);
    const size_t dyn = sizeof(double) * D * LOOP2_WORKERS;
    if (with_reducer(workers) > fit(k_cgloop2d<T, C, TY, WAIT_TEST>, NT, dyn, cache)) return cudaSuccess;
    cudaError_t e;
    if (!loop_words(c, c->zwords, LOOP2_ZBYTES)) return cudaSuccess;
    if ((e = cudaMemsetAsync(c->gather, 0, GATHER_BYTES, c->stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(c->zwords, 0, (size_t)workers * 3 * 32 * TY * sizeof(unsigned long long) * ZWords<T>::N, c->stream)) !=
        cudaSuccess)
        return e;
    Layout L = c->L;
    const int* tiles = c->tiles;
    int nt = c->ntiles_active;
    Coef<C> coef = cf;
    const double* r64 = c->w64.r;      // (FP64: the solve's own residual vector, which the kernel does not write)
    void* args[] = {&L, &tiles, &nt, &coef, &r64, &minv, &w.x, &c->zwords, &c->sc, &c->gather};
    *taken = loop_launched(cudaLaunchCooperativeKernel((const void*)k_cgloop2d<T, C, TY, WAIT_TEST>, with_reducer(workers), NT,
                                                       args, workers <= GATHER_DIRECT ? 0 : dyn, c->stream));
    return cudaSuccess;
}

// Run the inner solve in one cooperative kernel if the system is small enough
// (*taken); the graph of separate kernels takes the others (they are bound by
// what their kernels move, not by launches), and those that the device refuses.  update_ctas: CTAs of k_cg_update
// that fit on the device (up to that many tiles it gives each CTA one, the order
// that the sums here repeat).  The lines: one CTA per tile in FP32 and two per
// tile at most in FP64 while two CTAs per SM hold them all (303 workers; 124 and
// 128 registers); the separate FP64 apply also has one tile per CTA up to there.
// Measured, us per iteration, separate kernels and this: 32^2 disk (4 tiles) FP64
// 17.3 and 6.2, FP32 14.7 and 4.0; 96^2 bumps (22) 19.2 and 7.9, 17.3 and 5.9;
// 256^2 bumps (101) 19.0 and 12.3, 16.1 and 7.7; 256^2 box (297) FP32 17.7 and 9.9.
template <class T, class C>
cudaError_t launch_cg_loop(Ctx* c, CgWork<T>& w, const T* minv, const Coef<C>& cf, int update_ctas, bool* taken) {
    *taken = false;
    const int nt = c->ntiles_active;
    if (c->L.dim != 2 || nt > update_ctas) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        if (4 * nt <= LOOP2_WORKERS)
            return c->wait_test ? launch2<T, C, 2, true>(c, w, minv, cf, taken) : launch2<T, C, 2, false>(c, w, minv, cf, taken);
        if (2 * nt <= LOOP2_WORKERS)
            return c->wait_test ? launch2<T, C, 4, true>(c, w, minv, cf, taken) : launch2<T, C, 4, false>(c, w, minv, cf, taken);
    } else {
        if (nt <= LOOP2_WORKERS)
            return c->wait_test ? launch2<T, C, 8, true>(c, w, minv, cf, taken) : launch2<T, C, 8, false>(c, w, minv, cf, taken);
    }
    return cudaSuccess;
}

template cudaError_t launch_cg_loop<double, double>(Ctx*, CgWork<double>&, const double*, const Coef<double>&, int, bool*);
template cudaError_t launch_cg_loop<float, float>(Ctx*, CgWork<float>&, const float*, const Coef<float>&, int, bool*);
template cudaError_t launch_cg_loop<float, __nv_bfloat16>(Ctx*, CgWork<float>&, const float*, const Coef<__nv_bfloat16>&, int,
                                                          bool*);

}  // namespace stk
