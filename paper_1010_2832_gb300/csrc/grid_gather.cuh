// Grid-wide sums inside a cooperative CG kernel.
//
// Every word that crosses CTAs is 64 bits: 32 bits of data and the epoch it
// belongs to, so a word is valid by itself and a reader polls the data, not a
// flag beside it.  Slots alternate between two sets: a CTA writes exchange
// e + 2 only after it has passed e + 1, that is, after every reader is done
// with exchange e.  Every wait is bounded: a reader gives up after GATHER_POLLS
// rounds (GATHER_TEST_POLLS under the options' wait test hook, where words are
// held back) and says so.
//
// Up to GATHER_DIRECT workers, each CTA reads everybody's partial sums and forms
// the total itself: one trip through L2 per exchange.  With more, that would be
// a quadratic number of reads (462 workers: 100 us per CG iteration); one more
// CTA, the reducer, reads the partial sums, does the scalar work of the CG step
// and posts the one number that the workers need.
//
// FP64 is slow on this part (two lanes per clock and SM, so 16 clocks for a
// warp's instruction however many lanes take part): totals and scalars are
// formed by one warp, FP32 kernels publish their float-float sums through one
// conversion for the whole CTA.
//
// The order of the additions is that of the two-stage reductions of the
// separate CG kernels (a block's warps one after another; thread t of a
// 256-thread block the partials t, t + 256, ...; a shuffle tree; the warps one
// after another), so a solve in one kernel and one launched kernel by kernel
// agree bit for bit.
#pragma once
#include "internal.cuh"

namespace stk {

constexpr int GATHER_MAX = 608;                    // workers at most
constexpr int GATHER_DIRECT = 64;
constexpr int GATHER_DOUBLES = 8;                  // per worker and exchange at most
constexpr int GATHER_PITCH = GATHER_MAX + 8;       // one row per word of a worker's: a warp reads 32 workers' words as one run
constexpr size_t GATHER_BYTES = sizeof(unsigned long long) * 2 * GATHER_PITCH * 2 * GATHER_DOUBLES;
constexpr int GATHER_POLLS = 1 << 21;              // each round is a load from L2 (half a microsecond or more)
constexpr int GATHER_TEST_POLLS = 1024;            // of a solve with the wait test hook

__device__ __forceinline__ void post_word(unsigned long long* p, unsigned epoch, unsigned data) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)epoch << 32) | data) : "memory");
}
__device__ __forceinline__ unsigned long long peek_word(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double from_words(unsigned long long lo, unsigned long long hi) {
    return __longlong_as_double((long long)((lo & 0xffffffffu) | (hi << 32)));
}

// x is finite; x > 0 and finite (integer tests)
__device__ __forceinline__ bool finite64(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }
__device__ __forceinline__ bool positive64(double x) { return __double_as_longlong(x) > 0 && finite64(x); }

// CG scalars and the tests of k_cg_init / k_cg_update, held by one warp.
struct CgState {
    double rz, rr, rr0, tol2, pq, alpha, beta;
    int iter, done, status;
    __device__ void start(double tol_rel, double trz, double trr) {
        rz = trz; rr = rr0 = trr;
        tol2 = tol_rel * tol_rel * trr;
        alpha = beta = pq = 0.0;
        iter = 0; status = 0;
        done = (trr <= tol2 || trr == 0.0) ? 1 : 0;
        if (!finite64(trr)) { done = 1; status = STOKES_ERR_NONFINITE; }
    }
    __device__ void direction(double tot) {
        pq = tot;
        if (!positive64(tot)) { done = 1; status = finite64(tot) ? STOKES_ERR_BREAKDOWN : STOKES_ERR_NONFINITE; }
        else alpha = rz / tot;
    }
    __device__ void step(int max_iter, double trz, double trr) {
        rr = trr;
        iter += 1;
        if (!finite64(trr) || !finite64(trz)) { done = 1; status = STOKES_ERR_NONFINITE; }
        else if (trr <= tol2) { done = 1; }
        else if (!positive64(trz)) { done = 1; status = STOKES_ERR_BREAKDOWN; }
        else if (iter >= max_iter) { done = 1; status = STOKES_ERR_NOT_CONVERGED; }
        beta = trz / rz;
        rz = trz;
    }
    // (the status of a CTA whose wait ran out stands, whichever comes first)
    __device__ void store(CgScalars* sc) const {
        sc->rz = rz; sc->rr = rr; sc->rr0 = rr0; sc->tol2 = tol2; sc->pq = pq; sc->alpha = alpha; sc->beta = beta;
        sc->iter = iter; sc->done = 1;
        atomicCAS(&sc->status, STOKES_OK, status);
    }
};

enum { CG_START = 0, CG_DIRECTION = 1, CG_STEP = 2 };

struct GatherSmem {
    double red[8][2];
    double scalar;               // alpha or beta
    int done, ok;
};

// NT threads per CTA; POLLS limits every wait (a constant: as an argument it cost
// the kernels registers that they then spilled).  An exchange orders nothing but
// its own words: other data crosses CTAs in tagged words too.
template <int NT, int POLLS = GATHER_POLLS> struct GridGather {
    static constexpr int NW = NT / 32;
    using Smem = GatherSmem;
    unsigned long long* slots;   // [2][2 * GATHER_DOUBLES][GATHER_PITCH], zero before the kernel starts; column GATHER_MAX is the result
    Smem* sm;
    double* vals;                // shared memory for the partial sums: workers * 8 doubles (reducer, or direct)
    int workers;
    unsigned epoch = 0;
    CgState cg;                  // warp 0 of a CTA that forms totals
    bool alive = true;

    __device__ bool direct() const { return workers <= GATHER_DIRECT; }
    __device__ bool reducer() const { return (int)blockIdx.x == workers; }
    __device__ unsigned long long* slot(int cta, int word) const {
        return slots + ((epoch & 1) * 2 * GATHER_DOUBLES + word) * GATHER_PITCH + cta;
    }
    // the result's words are neighbours: one line for its readers
    __device__ unsigned long long* result(int word) const { return slot(GATHER_MAX, 0) + word; }

    // One exchange.  Workers give D doubles in src (shared memory, complete in
    // program order of the calling thread or of others before a barrier);
    // part(b, q) is sum q of Q of block b of the separate kernels, formed from
    // vals (D doubles per worker), nb the number of those blocks; meanwhile()
    // runs while the words travel.  Afterwards every thread has the new scalar
    // (alpha after CG_DIRECTION, beta after CG_STEP) and whether the solve is
    // over; false on a time-out.
    template <int D, int Q, class Part, class Mean>
    __device__ bool exchange(int what, const double* src, int nb, double tol_rel, int max_iter, Part part, Mean meanwhile,
                             double& scalar, bool& done) {
        const int t = threadIdx.x, lane = t & 31, w = t >> 5;
        ++epoch;
        __syncthreads();
        const bool totals = direct() || reducer();
        if (!reducer() && t < 2 * D) {
            const unsigned long long u = __double_as_longlong(src[t >> 1]);
            post_word(slot(blockIdx.x, t), epoch, (unsigned)((t & 1) ? u >> 32 : u));
        }
        meanwhile();
        if (totals) {
            int ok = 1;
#pragma unroll 1
            for (int c = t; c < workers; c += NT) {
                unsigned long long v[2 * D];
                bool here = false;
#pragma unroll 1
                for (int poll = 0; !here && poll < POLLS; ++poll) {
                    here = true;
#pragma unroll
                    for (int k = 0; k < 2 * D; ++k) v[k] = peek_word(slot(c, k));
#pragma unroll
                    for (int k = 0; k < 2 * D; ++k) here = here && (unsigned)(v[k] >> 32) == epoch;
                }
                if (!here) ok = 0;
#pragma unroll
                for (int k = 0; k < D; ++k) vals[c * D + k] = from_words(v[2 * k], v[2 * k + 1]);
            }
            ok = __syncthreads_and(ok);
            // (in the trees below, steps that could only add zeros are left out)
            double tot[Q];
            if (nb * Q <= 32) {
                // one warp, each sum on its own 32 / Q lanes
                if (w == 0) {
                    constexpr int HALF = 32 / Q;
                    const int b = lane % HALF, q = lane / HALF;
                    double s = b < nb ? part(b, q) : 0.0;
                    for (int o = HALF / 2; o > 0; o >>= 1)
                        if (o < nb) s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
                    for (int k = 0; k < Q; ++k) tot[k] = __shfl_sync(0xffffffffu, s, k * HALF);
                }
            } else {
                const int ne = min((nb + 31) / 32, 8);
#pragma unroll 1
                for (int k = w; k < ne * Q; k += NW) {
                    const int e = k / Q, q = k % Q;
                    double s = 32 * e + lane < nb ? part(32 * e + lane, q) : 0.0;
                    for (int b = 32 * e + lane + 256; b < nb; b += 256) s += part(b, q);
                    __syncwarp();
                    s = warp_sum(s);
                    if (lane == 0) sm->red[e][q] = s;
                }
                __syncthreads();
                if (w == 0) {
                    double s = 0.0;
                    if (lane < Q) {
                        s = sm->red[0][lane];
                        for (int e = 1; e < ne; ++e) s += sm->red[e][lane];
                    }
#pragma unroll
                    for (int k = 0; k < Q; ++k) tot[k] = __shfl_sync(0xffffffffu, s, k);
                }
            }
            if (w == 0) {
                if (what == CG_START) cg.start(tol_rel, tot[0], tot[Q - 1]);
                else if (what == CG_DIRECTION) cg.direction(tot[0]);
                else cg.step(max_iter, tot[0], tot[Q - 1]);
                const double x = what == CG_DIRECTION ? cg.alpha : cg.beta;
                if (reducer() && lane < 3) {
                    const unsigned long long u = __double_as_longlong(x);
                    const unsigned flag = ok ? (unsigned)cg.done : 2u;
                    post_word(result(lane), epoch, lane == 0 ? (unsigned)u : lane == 1 ? (unsigned)(u >> 32) : flag);
                }
                if (lane == 0) { sm->scalar = x; sm->done = cg.done; sm->ok = ok; }
            }
        } else if (w == 0) {
            unsigned long long v = 0;
            bool here = lane >= 3;
#pragma unroll 1
            for (int poll = 0; !here && poll < POLLS; ++poll) {
                v = peek_word(result(lane));
                here = (unsigned)(v >> 32) == epoch;
            }
            const bool ok = __all_sync(0xffffffffu, here);
            const unsigned lo = __shfl_sync(0xffffffffu, (unsigned)v, 0), hi = __shfl_sync(0xffffffffu, (unsigned)v, 1),
                           flag = __shfl_sync(0xffffffffu, (unsigned)v, 2);
            if (lane == 0) {
                sm->scalar = from_words(lo, hi);
                sm->done = flag != 0;
                sm->ok = ok && flag != 2;
            }
        }
        __syncthreads();
        scalar = sm->scalar;
        done = sm->done != 0;
        alive = sm->ok != 0;
        return alive;
        // (sm and vals are written again only past the next exchange's first barrier)
    }
    // The end: the CTA that holds the scalars stores them; a time-out is marked.
    __device__ void finish(CgScalars* sc) const {
        if (!alive) {
            if (threadIdx.x == 0) { atomicExch(&sc->status, (int)STOKES_ERR_TIMEOUT); sc->done = 1; }
        } else if ((int)blockIdx.x == (direct() ? 0 : workers) && threadIdx.x == 0) {
            cg.store(sc);
        }
    }
};

}  // namespace stk
