// Schwarz-preconditioned CG of small 2D systems (FP32 vectors) in one
// cooperative kernel: the loop of schwarz_body (apply, local solves, gather) with
// one CTA per SM in two roles.
//
//   tile CTAs   own two tiles each (list places b and b + G, the pairs of
//               k_sw_finish), a slot per thread: x, r, p, coefficients, face
//               coefficients and the halo's p stay in registers;
//   patch CTAs  hold the stored factors of up to 16 patches in shared memory for
//               the whole solve, four patches at a time, 128 threads each.
//
// Per iteration: apply, p.q (grid_gather.cuh), r -= alpha q; the tiles post r, the
// patches answer with their local results, the tiles gather z, then r.z and r.r.
// Everything that crosses CTAs is a word tagged with the iteration, so a reader
// polls its data and no barrier or fence separates the phases.  A word is
// overwritten only after an exchange that all tiles enter after their results,
// and so the patches' reads, of the previous iteration are in.  Patches leave
// when the stop word is set.  Every wait is bounded.
//
// The arithmetic and the order of every sum are those of k_apply2d_v4,
// k_schwarz_gemv and k_sw_finish: iterates agree with the separate kernels' bit
// for bit.
#include "ctx.cuh"
#include "apply2d_tile.cuh"
#include "schwarz_plan.cuh"
#include "loop_common.cuh"

namespace stk {

constexpr int SWL_THREADS = 512, SWL_GROUPS = 4, SWL_PPG = 4;     // groups of a patch CTA, patches per group at most
constexpr int SWL_MAX_TILES = 303, SWL_MAX_PATCHES = 152 * SWL_GROUPS * SWL_PPG;
constexpr size_t SWL_TILE_WORDS = 3 * 256;                        // z or r of one tile
constexpr size_t SWL_PATCH_WORDS = PMAX;

struct SwLoopTile {
    float U[TY2 + 2][TX + 2], V[TY2 + 2][TX + 2], N[TY2 + 2][TX + 2];
    float Zu[TY2 + 1][TX + 1], Zv[TY2 + 1][TX + 1];
    float P[3][TY2][TX], Y[3][TY2][TX];                           // p and A p; then r and z (second tile) for the dots
};
struct SwLoopTileSmem {
    SwLoopTile tile[2];
    WarpSums<float, 8> sums;
    GridGather<SWL_THREADS>::Smem g;
    double vals[GATHER_DIRECT * 4];
};
struct SwLoopPatchScratch {
    alignas(16) float s[PMAX8];
    alignas(16) __half hb[SW_HB_HALVES];
};

struct SwLoopWords {
    unsigned long long *z, *r, *y, *stop;
};

// Poll one word until it carries the tag (true), the stop word is set or the
// polls run out (false).
template <int POLLS>
__device__ __forceinline__ bool poll_word(const unsigned long long* p, unsigned tag, const unsigned long long* stop, float& v) {
#pragma unroll 1
    for (int poll = 0; poll < POLLS; ++poll) {
        const unsigned long long w = peek_word(p), over = peek_word(stop);
        if ((unsigned)(w >> 32) == tag) {
            v = __uint_as_float((unsigned)w);
            return true;
        }
        if (over != 0) return false;
    }
    return false;
}

template <int POLLS>
__device__ __forceinline__ void patch_role(const Layout& L, const int* __restrict__ tiles, int ntiles, const SchwarzPlan& P,
                                           const SwLoopWords& W, unsigned char* smem, int ppg, int cta, int nctas, int max_iter) {
    const int gid = threadIdx.x >> 7, t = threadIdx.x & 127;
    const BarGroup grp{t, 1 + gid};
    uint8_t* const fac = smem + (size_t)gid * ppg * SW_FAC_BYTES;
    SwLoopPatchScratch& sm =
        *reinterpret_cast<SwLoopPatchScratch*>(smem + (size_t)SWL_GROUPS * ppg * SW_FAC_BYTES + gid * sizeof(SwLoopPatchScratch));
    constexpr int RR = PR * PR;
    // this thread's position (a cell's tau_xx and p, or a node's tau_xy) of each
    // patch of the group, as in k_schwarz_gemv
    int np = 0, n[SWL_PPG], kk[SWL_PPG], kp[SWL_PPG];
    float sa[SWL_PPG], sb[SWL_PPG];
    const unsigned long long* rw[SWL_PPG];
#pragma unroll
    for (int k = 0; k < SWL_PPG; ++k) {
        const int p = (k * nctas + cta) * SWL_GROUPS + gid;
        n[k] = 0; kk[k] = kp[k] = -1; sa[k] = sb[k] = 0.f; rw[k] = W.r;
        if (k >= ppg || p >= P.np) continue;
        np = k + 1;
        n[k] = P.nloc[p];
        const int cw = P.corner[p], a0 = PB * (cw & 0xffff) - 1, b0 = PB * (cw >> 16) - 1;
        const uint4* src = reinterpret_cast<const uint4*>(P.fac + (int64_t)p * SW_FAC_BYTES);
        uint4* dst = reinterpret_cast<uint4*>(fac + k * SW_FAC_BYTES);
        for (uint32_t e = t; e < sw_patch_bytes(n[k]) / 16; e += 128) dst[e] = src[e];
        if (t < 2 * RR) {
            const int rem = t % RR, c = a0 + rem % PR + 1, rr = b0 + rem / PR + 1;
            kk[k] = P.lmap[(int64_t)p * PMAX + t];
            sa[k] = P.scale[(int64_t)p * PMAX + t];
            if (t < RR) {
                kp[k] = P.lmap[(int64_t)p * PMAX + 2 * RR + t];
                sb[k] = P.scale[(int64_t)p * PMAX + 2 * RR + t];
            }
            if (kk[k] >= 0 || kp[k] >= 0) {               // an active unknown: its tile is in the list
                const int place = max(tile_place(tiles, ntiles, (rr / TY2) * L.ntx + c / TX), 0);
                rw[k] = W.r + (size_t)place * SWL_TILE_WORDS + (rr % TY2) * TX + c % TX + (t < RR ? 0 : 256);
            }
        }
    }
    if (np == 0) return;                                  // a group without a patch
    if (POLLS == GATHER_TEST_POLLS && cta == 0 && gid == 0) return;      // the wait test hook: no answers
    grp.sync();
    constexpr float H = 0.70710678118654752f;
    // (one answer per iteration and one for the start: a solve ends by max_iter)
    for (unsigned tag = 1; tag <= (unsigned)max_iter + 1u; ++tag) {
#pragma unroll
        for (int k = 0; k < SWL_PPG; ++k) {
            if (k >= np) continue;
            bool here = true;
            float* s = sm.s;
            if (t >= RR) {
                if (kk[k] >= 0) {
                    float rv = 0.f;
                    here = poll_word<POLLS>(rw[k], tag, W.stop, rv);
                    s[kk[k]] = rv * sa[k];
                }
            } else {
                float rt = 0.f, rp = 0.f;
                // (the two words are posted together: the second is seldom waited for)
                if (kk[k] >= 0) here = poll_word<POLLS>(rw[k], tag, W.stop, rt);
                if (kp[k] >= 0 && here) here = poll_word<POLLS>(rw[k] + 2 * 256, tag, W.stop, rp);
                if (kk[k] >= 0 && kp[k] >= 0) {
                    s[kk[k]] = (rt + rp) * H * sa[k];
                    s[kp[k]] = (rt - rp) * H * sb[k];
                } else if (kk[k] >= 0) {
                    s[kk[k]] = rt * sa[k];
                } else if (kp[k] >= 0) {
                    s[kp[k]] = rp * sb[k];
                }
            }
            if (t >= n[k] && t < (n[k] + 7) / 8 * 8) s[t] = 0.f;
            if (grp.any(!here)) return;                   // the solve is over (or a wait ran out: the tiles' run out too)
            sw_factor_products(grp, fac + k * SW_FAC_BYTES, n[k], s, s, sm.hb);
            unsigned long long* out = W.y + (size_t)((k * nctas + cta) * SWL_GROUPS + gid) * SWL_PATCH_WORDS;
            if (t < 2 * RR) {
                if (t >= RR) {
                    if (kk[k] >= 0) post_word(out + t, tag, __float_as_uint(s[kk[k]] * sa[k]));
                } else if (kk[k] >= 0 && kp[k] >= 0) {
                    const float2 z = sw_unrotate(s[kk[k]], sa[k], s[kp[k]], sb[k]);
                    post_word(out + t, tag, __float_as_uint(z.x));
                    post_word(out + 2 * RR + t, tag, __float_as_uint(z.y));
                } else if (kk[k] >= 0) {
                    post_word(out + t, tag, __float_as_uint(s[kk[k]] * sa[k]));
                } else if (kp[k] >= 0) {
                    post_word(out + 2 * RR + t, tag, __float_as_uint(s[kp[k]] * sb[k]));
                }
            }
            grp.sync();                                   // s is free for the next patch
        }
    }
}

// WAIT_TEST: the options' hook; one group of patches does not answer.
template <bool WAIT_TEST>
__global__ void __launch_bounds__(SWL_THREADS, 1) k_swloop(Layout L, const int* __restrict__ tiles, int ntiles,
                                                           Coef<float> cf, DevArrays D, SchwarzPlan P,
                                                           const double* __restrict__ r64, float* __restrict__ xout,
                                                           SwLoopWords W, int ppg, CgScalars* sc, unsigned long long* slots) {
    constexpr int POLLS = WAIT_TEST ? GATHER_TEST_POLLS : GATHER_POLLS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = (ntiles + 1) / 2;                       // tile CTAs
    const int first_patch = G <= GATHER_DIRECT ? G : G + 1;
    if ((int)blockIdx.x >= first_patch) {
        patch_role<POLLS>(L, tiles, ntiles, P, W, smem_raw, ppg, blockIdx.x - first_patch, gridDim.x - first_patch, sc->max_iter);
        return;
    }
    SwLoopTileSmem& sm = *reinterpret_cast<SwLoopTileSmem*>(smem_raw);
    const int t = threadIdx.x, half = t >> 8, lt = t & 255, tx = t & 31, ty = lt >> 5;
    using Gather = GridGather<SWL_THREADS, POLLS>;
    // (the reducer holds no tile: its partial sums may lie over them)
    Gather gather{slots, &sm.g, sm.vals, G};
    if (!gather.direct()) gather.vals = reinterpret_cast<double*>(&sm.tile[0]);
    const double* vals = gather.vals;
    const double tol_rel = sc->tol_rel;
    const int max_iter = sc->max_iter;
    // block sums of k_sw_finish (a CTA's pair of tiles) and of k_apply2d_v4 (four
    // tiles of the list, two warps each)
    auto part_z = [&](int b, int q) -> double { return vals[2 * b + q]; };
    auto part_p = [&](int b, int) -> double {
        double v = 0.0;
        for (int q = 4 * b; q < min(4 * b + 4, ntiles); ++q) {
            const double* u = vals + 4 * (q < G ? q : q - G) + (q < G ? 0 : 2);
            v += u[0];
            v += u[1];
        }
        return v;
    };
    auto none = [] {};
    const int nb_p = (ntiles + 3) / 4;
    double scalar;
    bool done;
    if ((int)blockIdx.x == G) {                           // the reducer (more than GATHER_DIRECT tile CTAs)
        bool ok = gather.template exchange<2, 2>(CG_START, nullptr, G, tol_rel, max_iter, part_z, none, scalar, done);
        while (ok && !done) {
            ok = gather.template exchange<4, 1>(CG_DIRECTION, nullptr, nb_p, tol_rel, max_iter, part_p, none, scalar, done);
            if (ok && !done)
                ok = gather.template exchange<2, 2>(CG_STEP, nullptr, G, tol_rel, max_iter, part_z, none, scalar, done);
        }
        gather.finish(sc);
        return;
    }
    SwLoopTile& T = sm.tile[half];
    const int place = blockIdx.x + half * G;
    const bool have = place < ntiles;
    const int tile = have ? tiles[place] : tiles[0];
    const int c0 = (tile % L.ntx) * TX, r0 = (tile / L.ntx) * TY2;
    const int64_t S = L.stride, o = L.off(c0 + tx, r0 + ty, 0);
    const int i = c0 + tx - 1, j = r0 + ty - 1;
    const bool real = i >= 0 && j >= 0 && i <= L.nx && j <= L.ny;
    float ac = 0.f, an = 0.f, dc = 0.f, dn = 0.f, x[3], r[3], p[3], z[3], y[3];
    bool act[3] = {false, false, false};
    if (have) { ac = cf.f[0][o]; an = cf.f[1][o]; dc = cf.f[2][o]; dn = cf.f[3][o]; }
    const double scale = sc->scale;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        r[f] = have ? (float)(r64[f * S + o] * scale) : 0.f;
        x[f] = p[f] = z[f] = y[f] = 0.f;
        act[f] = have && unknown_active(D, L, f, i, j);
    }
    const bool edge = tx == 0 || tx == TX - 1 || ty == 0 || ty == TY2 - 1;
    unsigned long long* const zown = W.z + (size_t)place * SWL_TILE_WORDS + lt;
    unsigned long long* const rown = W.r + (size_t)place * SWL_TILE_WORDS + lt;
    // the patches over the slot (the fixed 2 x 2 window of sw_gather_load) and
    // the slot's position in each; -1 where there is none
    int py[4];
    {
        const int ilo = max((i + PB - 1) / PB - 1, 0), ihi = min((i + 1) / PB, P.npx - 1);
        const int jlo = max((j + PB - 1) / PB - 1, 0), jhi = min((j + 1) / PB, P.npy - 1);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int I = ilo + (q & 1), J = jlo + (q >> 1);
            py[q] = -1;
            if (have && real && I <= ihi && J <= jhi) {
                const int id = P.pid[J * P.npx + I];
                const int ii = i - (PB * I - 1), jj = j - (PB * J - 1);
                if (id >= 0) py[q] = id * (int)SWL_PATCH_WORDS + jj * PR + ii;
            }
        }
    }
    // halo position of this thread, and where its owner posts z
    constexpr int HALO = 2 * (TX + 2) + 2 * TY2;
    float hp[3] = {0.f, 0.f, 0.f}, hac = 0.f, han = 0.f;
    const unsigned long long* hz = W.z;
    int hs = -1;
    if (have && lt < HALO) {
        int jj, ii;
        if (lt < TX + 2) { jj = 0; ii = lt; }
        else if (lt < 2 * (TX + 2)) { jj = TY2 + 1; ii = lt - (TX + 2); }
        else { jj = 1 + (lt - 2 * (TX + 2)) / 2; ii = (lt & 1) ? TX + 1 : 0; }
        const int c = c0 - 1 + ii, rr = r0 - 1 + jj;
        const int64_t oh = L.off(c, rr, 0);
        hac = cf.f[0][oh];
        han = cf.f[1][oh];
        if (hac != 0.f || han != 0.f) {
            const int k = tile_place(tiles, ntiles, (rr / TY2) * L.ntx + c / TX);
            if (k >= 0) {
                hs = jj * (TX + 2) + ii;
                hz = W.z + (size_t)k * SWL_TILE_WORDS + (rr % TY2) * TX + c % TX;
            }
        }
    }
    constexpr int NF = (TY2 + 1) * (TX + 1);
    float ku[2], kv[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = lt + q * 256;
        ku[q] = kv[q] = 0.f;
        if (have && e < NF) {
            const int jj = e / (TX + 1), ii = e - jj * (TX + 1);
            ku[q] = cf.f[4][L.off(c0 + ii, r0 - 1 + jj, 0)];
            kv[q] = cf.f[5][L.off(c0 - 1 + ii, r0 + jj, 0)];
        }
    }
    for (int e = lt; e < (TY2 + 2) * (TX + 2); e += 256) (&T.U[0][0])[e] = (&T.V[0][0])[e] = (&T.N[0][0])[e] = 0.f;
    for (int e = lt; e < NF; e += 256) (&T.Zu[0][0])[e] = (&T.Zv[0][0])[e] = 0.f;
    unsigned tag = 1;
    // r to the patches, z from them, r.z and r.r; x += alpha p under way
    auto precondition = [&](int what, float alpha) -> bool {
#pragma unroll
        for (int f = 0; f < 3; ++f)
            if (act[f]) post_word(rown + f * 256, tag, __float_as_uint(r[f]));
        if (what == CG_STEP)
#pragma unroll
            for (int f = 0; f < 3; ++f) x[f] = x[f] + alpha * p[f];
        bool here = false;
        unsigned long long v[3][4];
#pragma unroll 1
        for (int poll = 0; !here && poll < POLLS; ++poll) {
            here = true;
#pragma unroll
            for (int f = 0; f < 3; ++f)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (act[f] && py[q] >= 0) v[f][q] = peek_word(W.y + py[q] + f * PR * PR);
#pragma unroll
            for (int f = 0; f < 3; ++f)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (act[f] && py[q] >= 0) here = here && (unsigned)(v[f][q] >> 32) == tag;
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            float s = 0.f;
            if (act[f])
#pragma unroll
                for (int q = 0; q < 4; ++q) s += py[q] >= 0 ? __uint_as_float((unsigned)v[f][q]) : 0.f;
            z[f] = act[f] ? s : (real ? r[f] : 0.f);
            if (edge && act[f]) post_word(zown + f * 256, tag, __float_as_uint(z[f]));
        }
        if (!__syncthreads_and(here)) { gather.alive = false; return false; }
        // the dots of k_sw_finish: thread lt adds its slot of the first tile, then
        // of the second
        if (half) {
#pragma unroll
            for (int f = 0; f < 3; ++f) { T.P[f][ty][tx] = r[f]; T.Y[f][ty][tx] = z[f]; }
        }
        __syncthreads();
        if (!half) {
            Acc<float> rz, r2;
#pragma unroll
            for (int f = 0; f < 3; ++f) { rz.add(r[f], z[f]); r2.add(r[f], r[f]); }
            if ((int)blockIdx.x + G < ntiles) {
                const SwLoopTile& B = sm.tile[1];
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    const float rv = B.P[f][ty][tx], zv = B.Y[f][ty][tx];
                    rz.add(rv, zv);
                    r2.add(rv, rv);
                }
            }
            sm.sums.put(ty, rz);
            sm.sums.put(8 + ty, r2);
        }
        sm.sums.block2();
        return gather.template exchange<2, 2>(what, sm.sums.rows, G, tol_rel, max_iter, part_z, none, scalar, done);
    };
    bool ok = precondition(CG_START, 0.f);
    while (ok && !done) {
        const float beta = (float)scalar;
        // p = z + beta p on the tile and its halo; stage
#pragma unroll
        for (int f = 0; f < 3; ++f) p[f] = z[f] + beta * p[f];
        T.U[ty + 1][tx + 1] = ac * (p[2] - p[0]);
        T.V[ty + 1][tx + 1] = ac * (p[2] + p[0]);
        T.N[ty + 1][tx + 1] = an * p[1];
        if (hs >= 0) {
            // an unknown's z is posted where it is active, that is where its weight is not zero
            float v[3] = {0.f, 0.f, 0.f};
            bool got = false;
#pragma unroll 1
            for (int poll = 0; !got && poll < POLLS; ++poll) {
                unsigned long long w[3] = {0, 0, 0};
                if (hac != 0.f) { w[0] = peek_word(hz); w[2] = peek_word(hz + 512); }
                if (han != 0.f) w[1] = peek_word(hz + 256);
                got = (hac == 0.f || ((unsigned)(w[0] >> 32) == tag && (unsigned)(w[2] >> 32) == tag)) &&
                      (han == 0.f || (unsigned)(w[1] >> 32) == tag);
#pragma unroll
                for (int f = 0; f < 3; ++f) v[f] = __uint_as_float((unsigned)w[f]);
            }
            ok = ok && got;
#pragma unroll
            for (int f = 0; f < 3; ++f) hp[f] = v[f] + beta * hp[f];
            (&T.U[0][0])[hs] = hac * (hp[2] - hp[0]);
            (&T.V[0][0])[hs] = hac * (hp[2] + hp[0]);
            (&T.N[0][0])[hs] = han * hp[1];
        }
        ok = __syncthreads_and(ok);
        if (!ok) { gather.alive = false; break; }
        ++tag;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = lt + q * 256;
            const int jj = e / (TX + 1), ii = e - jj * (TX + 1);
            if (ku[q] != 0.f)
                T.Zu[jj][ii] = ku[q] * ((T.U[jj][ii + 1] - T.U[jj][ii]) + (T.N[jj][ii + 1] - T.N[jj + 1][ii + 1]));
            if (kv[q] != 0.f)
                T.Zv[jj][ii] = kv[q] * ((T.V[jj + 1][ii] - T.V[jj][ii]) + (T.N[jj + 1][ii] - T.N[jj + 1][ii + 1]));
        }
        __syncthreads();
        // q = A p on the own slot, p.q (k_apply2d_v4: 64 threads of four slots each)
        {
            const float zu = T.Zu[ty + 1][tx], zur = T.Zu[ty + 1][tx + 1], zud = T.Zu[ty][tx];
            const float zv = T.Zv[ty][tx + 1], zvu = T.Zv[ty + 1][tx + 1], zvl = T.Zv[ty][tx];
            if (ac != 0.f) {
                y[2] = ac * ((zu - zur) + (zv - zvu));
                y[0] = fma_first(dc, p[0], ac, (zur - zu) + (zv - zvu));
            } else {
                y[2] = p[2];
                y[0] = p[0];
            }
            y[1] = fma_first(dn, p[1], an, (zu - zud) + (zv - zvl));
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) { T.P[f][ty][tx] = p[f]; T.Y[f][ty][tx] = y[f]; }
        __syncthreads();
        if (lt < 64) {
            Acc<float> acc;
            const int qr = lt >> 3, qc = 4 * (lt & 7);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int f = 0; f < 3; ++f) acc.add(T.P[f][qr][qc + k], T.Y[f][qr][qc + k]);
            sm.sums.put(2 * half + (lt >> 5), acc, have);
        }
        __syncthreads();
        if (t < 32) sm.sums.convert(4);
        ok = gather.template exchange<4, 1>(CG_DIRECTION, sm.sums.rows, nb_p, tol_rel, max_iter, part_p, none, scalar, done);
        if (!ok || done) break;
        const float alpha = (float)scalar;
#pragma unroll
        for (int f = 0; f < 3; ++f) r[f] = r[f] - alpha * y[f];
        ok = precondition(CG_STEP, alpha);
    }
    if (t == 0) asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(W.stop), "l"(1ull) : "memory");
    if (have)
#pragma unroll
        for (int f = 0; f < 3; ++f) xout[f * S + o] = x[f];
    gather.finish(sc);
}

// Run the inner Schwarz-CG solve in one cooperative kernel if it fits (*taken).
// finish_ctas: CTAs of k_sw_finish that fit on the device (up to that many it
// gives each a pair of tiles, the order repeated here).  Measured, us per
// iteration, separate kernels and this: 96^2 bumps (22 tiles, one patch per group
// of threads) 20.6 and 11.2; 160^2 (56 tiles, two) 22.2 and 16.1; 224^2 (85 tiles,
// two) 22.5 and 20.6; 150^2 box (95 tiles, three) 24.9 and 24.2.  Past four
// patches per group, or factors that do not fit in the SMs' shared memory, or where
// the device refuses the launch, the separate kernels take over.
template <bool WAIT_TEST>
static cudaError_t launch(Ctx* c, const SchwarzPlan& P, int finish_ctas, bool* taken) {
    *taken = false;
    const int nt = c->ntiles_active, G = (nt + 1) / 2, first = G <= GATHER_DIRECT ? G : G + 1;
    if (c->L.dim != 2 || nt < 1 || P.np < 1 || nt > SWL_MAX_TILES || P.np > SWL_MAX_PATCHES || G > finish_ctas) return cudaSuccess;
    static std::atomic<int> cache[SWL_PPG + 1][16];
    int ppg = 0, grid = 0;
    size_t smem = 0;
    for (int k = 1; k <= SWL_PPG && !ppg; ++k) {
        const int pc = (P.np + SWL_GROUPS * k - 1) / (SWL_GROUPS * k);
        smem = std::max(sizeof(SwLoopTileSmem), (size_t)SWL_GROUPS * (k * SW_FAC_BYTES + sizeof(SwLoopPatchScratch)));
        if (first + pc > 152 * 4) continue;
        // (the attribute that admits the largest size is set before the first query)
        if (first + pc <= fit(k_swloop<WAIT_TEST>, SWL_THREADS, smem, cache[k])) { ppg = k; grid = first + pc; }
    }
    if (!ppg) return cudaSuccess;
    cudaError_t e;
    const size_t wt = sizeof(unsigned long long) * SWL_TILE_WORDS, wp = sizeof(unsigned long long) * SWL_PATCH_WORDS;
    if (!loop_words(c, c->swwords, 2 * wt * SWL_MAX_TILES + wp * SWL_MAX_PATCHES + 256)) return cudaSuccess;
    SwLoopWords W;
    W.stop = c->swwords;
    W.z = c->swwords + 32;
    W.r = W.z + SWL_TILE_WORDS * nt;
    W.y = W.r + SWL_TILE_WORDS * nt;
    if ((e = cudaMemsetAsync(c->gather, 0, GATHER_BYTES, c->stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(c->swwords, 0, 256 + 2 * wt * nt + wp * P.np, c->stream)) != cudaSuccess) return e;
    Layout L = c->L;
    const int* tiles = c->tiles;
    int n = nt;
    Coef<float> cf = c->coef<float>();
    DevArrays D = c->A;
    SchwarzPlan plan = P;
    const double* r64 = c->w64.r;
    float* x = c->w32.x;
    void* args[] = {&L, &tiles, &n, &cf, &D, &plan, &r64, &x, &W, &ppg, &c->sc, &c->gather};
    *taken = loop_launched(cudaLaunchCooperativeKernel((const void*)k_swloop<WAIT_TEST>, grid, SWL_THREADS, args, smem, c->stream));
    return cudaSuccess;
}

cudaError_t launch_schwarz_loop(Ctx* c, const SchwarzPlan& P, int finish_ctas, bool* taken) {
    return c->wait_test ? launch<true>(c, P, finish_ctas, taken) : launch<false>(c, P, finish_ctas, taken);
}

}  // namespace stk
