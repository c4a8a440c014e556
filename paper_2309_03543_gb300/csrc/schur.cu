// Two-cyclic solves: on a two-coloured cell graph (red rows R, black rows B;
// no two neighbours share a colour) the scaled matrix is Ahat =
// [[I, E], [E^T, I]], and the black cells' Schur complement S = I - E^T E is
// formed explicitly, one row per black cell: a diagonal and at most six
// neighbours (two behind each of its three red cells).
//
//   - CPS_PC_REDUCED: CG on S.
//   - FP64 Jacobi: started with a zero red residual (y_R = bhat_R - E y_B),
//     every second Jacobi-PCG iteration of the full system leaves the red
//     residual zero again, and two of them are one CG iteration on S (J. K.
//     Reid, SIAM J. Numer. Anal. 9, 1972: systems with Property A).  So the
//     Jacobi solve runs on S too, counting two iterations per step.
//   - IC(0) in the two-colour order: from a zero red residual, PCG with M =
//     (D + L) D^-1 (D + L^T), D = diag(I, diag S), keeps it zero, and is CG on
//     S with the preconditioner diag(S): on D_B^-1/2 S D_B^-1/2 (unit
//     diagonal), the rows scaled here when that preconditioner is selected.
//
// Why explicit rows.  Applied as t = E r, w = r - E^T t, the product needs
// two neighbour waits an iteration, 36 B of matrix per red and per black row
// and a round trip of t: 88 B and 6 FP64 FMAs per black row.  A row of S is 80
// B and 7 FMAs and needs one wait.  The vectors halve against the full
// system's.
#include "cps_internal.cuh"
#include "exact_sum.cuh"
#include "grid_sync.cuh"

#include <cmath>
#include <cstddef>
#include <type_traits>

namespace cps {
namespace {

constexpr int kSlots = 6;

// Row k of S (black cell perm[nR + k]) from the red rows' entries only, so
// that S is symmetric to the last bit: red row c with entries v_i at black
// cells i gives S_ij -= v_i v_j.
__global__ void k_schur_rows(const double* __restrict__ a, const int32_t* __restrict__ col,
                             const double* __restrict__ s, const int32_t* __restrict__ perm,
                             const int32_t* __restrict__ iperm, int64_t nt, int64_t nR, int nB,
                             int64_t ld, double* __restrict__ v, int32_t* __restrict__ c6,
                             double* __restrict__ d, double* __restrict__ wt) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nB;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = perm[nR + k];
        double diag = 1.0, val[kSlots];
        int32_t idx[kSlots];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t c = col[j * nt + e];
            double own = 0.0, o[3];
            int32_t oc[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                oc[m] = col[m * nt + c];
                o[m] = a[m * nt + c];
            }
            bool seen = c == e;                   // unused slot: nothing behind it
#pragma unroll
            for (int m = 0; m < 3; ++m)
                if (!seen && oc[m] == e) {
                    own = o[m];
                    oc[m] = -1;
                    seen = true;
                }
            if (c == e) own = 0.0;
            diag = fma(-own, own, diag);
            int f = 2 * j;
            val[f] = val[f + 1] = 0.0;
            idx[f] = idx[f + 1] = (int32_t)k;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                if (c == e || oc[m] < 0 || oc[m] == c) continue;
                if (f < 2 * j + 2) {
                    // both slots are static registers: select by value
                    if (f == 2 * j) {
                        val[2 * j] = -(own * o[m]);
                        idx[2 * j] = (int32_t)(iperm[oc[m]] - nR);
                    } else {
                        val[2 * j + 1] = -(own * o[m]);
                        idx[2 * j + 1] = (int32_t)(iperm[oc[m]] - nR);
                    }
                    ++f;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
            v[j * ld + k] = val[j];
            c6[j * ld + k] = idx[j];
        }
        d[k] = diag;
        wt[k] = s[e];
    }
}

// Rows of D^-1/2 S D^-1/2 (D = diag S) in place; dsc = D^-1/2, and the weight
// of the stop test becomes s D^1/2 (the true residual of a black row).
__global__ void k_schur_scale(double* __restrict__ v, const int32_t* __restrict__ c6,
                              const double* __restrict__ d, int nB, int64_t ld,
                              double* __restrict__ dsc, double* __restrict__ wt) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nB;
         k += (int64_t)gridDim.x * blockDim.x) {
        const double sq = sqrt(d[k]);
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
            const double w = v[j * ld + k];
            if (w != 0.0) v[j * ld + k] = w / (sq * sqrt(d[c6[j * ld + k]]));
        }
        dsc[k] = 1.0 / sq;
        wt[k] *= sq;
    }
}

// Red cells (mesh order): y_R = b / s - E (S x)_B.
__global__ void __launch_bounds__(kBlock) k_tc_red(const double* __restrict__ b,
                                                   const double* __restrict__ x,
                                                   const double* __restrict__ s,
                                                   const double* __restrict__ a,
                                                   const int32_t* __restrict__ col,
                                                   const int32_t* __restrict__ perm, int64_t nt,
                                                   int64_t nR, double* __restrict__ y) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nR;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = perm[i];
        double acc = b[e] / s[e];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t c = col[j * nt + e];
            if (c != e) acc = fma(-a[j * nt + e], s[c] * x[c], acc);
        }
        y[e] = acc;
    }
}

// Black rows: y_B = S x, r = bhat - y_B - E^T y_R (scaled by dsc where the
// rows are), and the run's state: rho = r.r, ||b||^2 over all cells, ||S r||^2.
__global__ void __launch_bounds__(kBlock) k_tc_init(
    const double* __restrict__ b, const double* __restrict__ x, const double* __restrict__ s,
    const double* __restrict__ a, const int32_t* __restrict__ col,
    const int32_t* __restrict__ perm, const double* __restrict__ dsc,
    const double* __restrict__ y, int64_t nt, int64_t nR, double* __restrict__ yb,
    double* __restrict__ r, double rtol, long long budget, double* partials, CgState* st) {
    double rr = 0.0, bb = 0.0, nn = 0.0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nt;
         e += (int64_t)gridDim.x * blockDim.x) {
        const double be = b[e];
        bb = fma(be, be, bb);
    }
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nt - nR;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = perm[nR + k];
        const double se = s[e];
        const double ye = se * x[e];
        double ay = ye;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t c = col[j * nt + e];
            if (c != e) ay = fma(a[j * nt + e], y[c], ay);
        }
        double re = b[e] / se - ay;
        const double t = se * re;
        nn = fma(t, t, nn);
        if (dsc) {
            const double q = dsc[k];
            yb[k] = ye / q;
            re *= q;
        } else {
            yb[k] = ye;
        }
        r[k] = re;
        rr = fma(re, re, rr);
    }
    double t[3] = {rr, bb, nn};
    if (grid_sum<3>(t, partials, &st->arrive[2]) && threadIdx.x == 0) {
        st->rho = t[0];
        st->bnorm2 = t[1];
        st->thresh2 = rtol * rtol * t[1];
        st->rnorm2 = t[2];
        st->alpha = 0.0;
        st->beta = 0.0;
        st->gamma = 0.0;
        st->iter = 0;
        st->max_iter = budget;
        st->status = CPS_OK;
        st->done = (t[1] == 0.0 || t[2] <= st->thresh2 || budget <= 0) ? 2 : 0;
    }
}

// y of the whole system (mesh order) from the black solution:
// y_R = b / s - E y_B.
__global__ void __launch_bounds__(kBlock) k_tc_back(const double* __restrict__ b,
                                                    const double* __restrict__ yb,
                                                    const double* __restrict__ dsc,
                                                    const double* __restrict__ s,
                                                    const double* __restrict__ a,
                                                    const int32_t* __restrict__ col,
                                                    const int32_t* __restrict__ iperm, int64_t nt,
                                                    int64_t nR, double* __restrict__ y) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nt;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = (int64_t)iperm[e] - nR;
        if (k >= 0) {
            y[e] = dsc ? yb[k] * dsc[k] : yb[k];
            continue;
        }
        double acc = b[e] / s[e];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t c = col[j * nt + e];
            if (c == (int32_t)e) continue;
            const int64_t kc = (int64_t)iperm[c] - nR;
            acc = fma(-a[j * nt + e], dsc ? yb[kc] * dsc[kc] : yb[kc], acc);
        }
        y[e] = acc;
    }
}

// ------------------------------------------------------ the persistent loop

constexpr int kGridMax = 160;        // blocks (one per SM): five warps poll their totals
constexpr int kPollPer = kGridMax / 32;
constexpr int kQuant = 2;             // quantities of one reduction at most
constexpr int kSlotStride = 16;       // words of a slot: a 128-byte line per block, 16 bytes a quantity
constexpr size_t kSlotWords = 4 * (size_t)kGridMax * kSlotStride;   // [quantities][buffer][block]

struct SchurArgs {
    const double* v;
    const int32_t* c;
    const double* d;
    const double* wt;
    double* r;
    double* w;
    double* p;
    double* s;
    double* y;
    int n;
    int64_t ld;
    unsigned long long* pb;     // kSlotWords words of block totals, zero at launch
    GridSync* gs;
    CgState* st;
    int stall;                  // test hook: every reduction waits for a value that never comes
    double dmin;                // smallest diagonal of A (stop-test gate), 0 for none
};

// A block's total and the number of its use, one 16-byte access (single-copy
// atomic: 128-bit scoped loads and stores).
__device__ __forceinline__ void ld_total(const unsigned long long* p, double& v,
                                         unsigned long long& use) {
    unsigned long long bits;
    asm volatile(
        "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
        : "=l"(bits), "=l"(use)
        : "l"(p)
        : "memory");
    v = __longlong_as_double((long long)bits);
}

__device__ __forceinline__ void st_total(unsigned long long* p, double v, unsigned long long use) {
    asm volatile(
        "{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}"
        ::"l"(p), "l"((unsigned long long)__double_as_longlong(v)), "l"(use)
        : "memory");
}

// T 2^(E - 1075 + h) as a double, |T| <= 2^62, rounded half up, in integer
// arithmetic (NaN if the set held an infinity or NaN, infinity on overflow,
// a subnormal below the normal range): the FP64 pipe takes one warp instruction
// in 17 cycles.
__device__ __forceinline__ double fixed_bits(long long T, int E, int h) {
    unsigned long long m = T < 0 ? 0ull - (unsigned long long)T : (unsigned long long)T;
    const int e = E + h;                            // exponent field of a 53-bit m
    // m to 53 bits (right by sh, left if < 0), to fewer below the normal range
    const int sh = max(11 - __clzll((long long)m), 1 - e);
    m = sh > 0 ? (m + (1ull << (sh - 1))) >> sh : m << (-sh & 63);
    // bit 52 of m, and a carry into bit 53, count up the field
    unsigned long long bits = ((unsigned long long)(e + sh - 1) << 52) + m;
    if (bits > 0x7FF0000000000000ull) bits = 0x7FF0000000000000ull;
    if (T == 0) bits = 0;
    if (T < 0) bits |= 1ull << 63;
    if (E >= 2047) bits = 0x7FF8000000000000ull;
    return __longlong_as_double((long long)bits);
}

// v / 2^(E - 1075) for |v| < 2^(E - 1022), rounded half up: at most 2^53 in magnitude,
// every bit of the values in the largest one's binade.
__device__ __forceinline__ long long align_whole(double v, int E) {
    const long long bits = __double_as_longlong(v);
    const int e = (int)((bits >> 52) & 0x7FF);
    long long m = bits & 0xFFFFFFFFFFFFFLL;
    if (e) m |= 1LL << 52;
    const int sh = E - (e > 0 ? e : 1);
    if (sh > 0) m = sh > 62 ? 0 : (m + (1LL << (sh - 1))) >> sh;
    return bits < 0 ? -m : m;
}

// v > 0 and finite, on the bits (a compare on the FP64 pipe takes its latency).
__device__ __forceinline__ bool positive_finite(double v) {
    const long long b = __double_as_longlong(v);
    return b > 0 && b < 0x7FF0000000000000LL;
}

// Grid-wide sum of v[0..NV) over blocks of T threads: exact integer sums per
// warp and per block, rounded to a double once, and over the grid (trees of FP64
// adds, 116 cycles a step and one warp instruction in 17 cycles, measured 0.8
// to 1.3 us slower an iteration).  Each block stores its NV totals into its slot of
// one of two buffers, with the buffer's use count beside each.  A warp of every
// block polls 32 of the G slots of a quantity until all of them carry this use,
// and adds them; the first of a quantity's warps adds the warps' sums: a total and its arrival travel in one access, so the reduction
// costs one store and one load across the chip instead of a store, a counter
// and a load.  A slot is a 128-byte line of its own: with 152 blocks polling,
// an all-to-all of dense words takes 10000 cycles, of 32-byte sectors 5000, of
// lines 2100 (a counter and a read of the totals 2850; one block summing and
// writing the result back 2800; through clusters of 8 3400).  The two buffers
// alternate, so a slot is rewritten only after every block has passed the
// reduction in between, and every slot is written and polled at every use of
// its buffer: reductions of one and of two quantities have buffers and counts
// (ep) of their own.  Every block gets bit-identical totals.  Thread 0 then
// runs post(totals), the others go on at the barrier that follows the call.
// False (in s_fail, for all) if a wait ran out (about one second).
template <int T, int NV, typename Post>
__device__ __forceinline__ void tagged_allreduce(const double (&v)[NV], unsigned int& ep,
                                                 const SchurArgs& P, int& s_fail, Post post) {
    static_assert(NV >= 1 && NV <= kQuant, "quantities");
    __shared__ long long s_w[NV][32];          // sums of the warps, each in units of its own
    __shared__ int s_e[NV][32];
    __shared__ long long s_g[NV][kPollPer];    // sums of 32 blocks' totals, likewise
    __shared__ int s_ge[NV][kPollPer];
    __shared__ double s_tot[NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int G = (int)gridDim.x;
    const int nq = (G + 31) >> 5;              // warps that poll for a quantity
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int E = __reduce_max_sync(0xffffffffu, align_exp(v[k]));
        const long long t = warp_sum_fixed<52>(align_fixed(v[k], E, 1));
        if (lane == 0) {
            s_w[k][warp] = t;
            s_e[k][warp] = E;
        }
    }
    __syncthreads();
    if (warp < NV * nq) {
        const int k = NV > 1 && warp >= nq ? 1 : 0;
        const int q = warp - k * nq;
        const unsigned long long use = (unsigned long long)(ep >> 1) + 1;
        unsigned long long* slots =
            P.pb + ((NV - 1) * 2 + (size_t)(ep & 1u)) * kGridMax * kSlotStride + 2 * k;
        if (q == 0) {
            const int Ew = lane < T / 32 ? s_e[k][lane] : 1;
            const int E = __reduce_max_sync(0xffffffffu, Ew);
            // at most 2^57 a warp, in the largest unit
            const int sh = E - Ew;
            long long x = lane < T / 32 ? s_w[k][lane] : 0;
            if (sh > 0) x = sh > 60 ? 0 : (x + (1LL << (sh - 1))) >> sh;
            const long long t = warp_sum_fixed<57>(x);
            if (lane == 0) st_total(slots + blockIdx.x * kSlotStride, fixed_bits(t, E, 1), use);
        }
        slots += (lane + 32 * q) * kSlotStride;
        double got = 0.0;
        bool miss = lane + 32 * q < G;
        const bool never = P.stall != 0 && lane == 0;
        unsigned long long t0 = 0;
        for (long long spins = 0;; ++spins) {
            if (miss) {
                unsigned long long seen;
                ld_total(slots, got, seen);
                miss = seen != use || never;
            }
            if (__all_sync(0xffffffffu, !miss)) break;
            if ((spins & 255) == 255) {
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                const bool out = now - t0 > kWaitNs || spins > kSpinCap ||
                                 *(volatile int*)&P.gs->timeout != 0;
                if (__any_sync(0xffffffffu, out)) {
                    if (lane == 0) {
                        atomicExch(&P.gs->timeout, 1);
                        s_fail = 1;
                    }
                    break;
                }
            }
        }
        int E = __reduce_max_sync(0xffffffffu, align_exp(got));
        long long t = warp_sum_fixed<53>(align_whole(got, E));     // at most 2^58
        if (nq > 1) {
            if (lane == 0) {
                s_g[k][q] = t;
                s_ge[k][q] = E;
            }
            asm volatile("bar.sync 1, %0;" ::"r"(NV * nq * 32) : "memory");
            if (q == 0) {
                const int Eq = lane < nq ? s_ge[k][lane] : 1;
                E = __reduce_max_sync(0xffffffffu, Eq);
                const int sh = E - Eq;
                t = lane < nq ? s_g[k][lane] : 0;
                if (sh > 0) t = sh > 61 ? 0 : (t + (1LL << (sh - 1))) >> sh;
                // at most 2^58 a lane: biased into three limbs of 20 bits (as in
                // warp_sum_fixed; a tree of 64-bit shuffles takes twice as long)
                const unsigned long long u = (unsigned long long)t + (1ULL << 59);
                const unsigned int mask = (1u << 20) - 1u;
                const unsigned long long s0 = __reduce_add_sync(0xffffffffu, (unsigned)u & mask);
                const unsigned long long s1 =
                    __reduce_add_sync(0xffffffffu, (unsigned)(u >> 20) & mask);
                const unsigned long long s2 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 40));
                t = (long long)(s0 + (s1 << 20) + (s2 << 40) - (32ULL << 59));
            }
        }
        if (q == 0) {
            if (lane == 0) s_tot[k] = fixed_bits(t, E, 0);
            if (NV > 1) asm volatile("bar.sync 2, %0;" ::"n"(NV * 32) : "memory");
            if (threadIdx.x == 0 && !s_fail) post(s_tot);
        }
    }
    ++ep;
}

// Waits until every block in the bit set dep has posted `it` (a lane per block
// and word); a timeout recorded elsewhere shows at the next reduction.
__device__ __forceinline__ void dep_wait(GridSync* gs, const unsigned int* dep,
                                         unsigned long long it, int& s_fail) {
    if (threadIdx.x < 32) {
#pragma unroll
        for (int q = 0; q < kPollPer; ++q) {
            if (!((dep[q] >> threadIdx.x) & 1u)) continue;
            const unsigned long long* f = &gs->flag[(32 * q + threadIdx.x) * kFlagStride];
            unsigned long long t0 = 0;
            for (long long spins = 1; ld_acquire(f) < it; ++spins) {
                if ((spins & 255) != 0) continue;
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                if (now - t0 > kWaitNs || spins > kSpinCap) {
                    atomicExch(&gs->timeout, 1);
                    s_fail = 1;
                    break;
                }
            }
        }
    }
    __syncthreads();
}

// CG on rows with a unit or a given diagonal and K neighbours (K = 6: rows of
// S; K = 3: the scaled matrix itself, FP64 Jacobi on all cells) with the
// single-reduction (Chronopoulos-Gear) recurrences, from y, r and the state an
// init kernel left (rho, ||b||^2, thresholds):
//   [wait for the neighbours' r] w = A r, gamma = r.r, delta = w.r (every 8th:
//   ||wt r||^2) | one grid reduction: stop test, beta = gamma / gamma_old,
//   alpha = gamma / (delta - beta gamma / alpha_old) |
//   p = r + beta p; s = w + beta s; y += alpha p; r -= alpha s | post
// K + 7 FP64 FMAs a row (K + 6 with the unit diagonal).  A thread owns the same
// rows in both phases, so what only the owner reads stays in its block's shared
// memory across the iterations: RES vectors of p, s, y, w, r (a copy; the
// neighbours gather r from global memory), and with MAT the rows themselves.
// A block waits for the blocks that own its neighbours, whatever the numbering.
// 1/gamma and 1/(gamma alpha) are carried (one thread divides beside the wait
// for the neighbours), so one divide stays on the path the blocks wait on.
template <int T, int K, int RES, bool MAT, bool UNIT>
__global__ void __launch_bounds__(T, 1) k_resident_cg(SchurArgs P) {
    extern __shared__ double dyn[];
    // alpha, beta, 1/gamma, 1/(gamma alpha), ||S r||^2, stop threshold, gamma
    __shared__ double sc[7];
    __shared__ int s_stop;          // 0 run, 1 stop, 2 breakdown
    __shared__ int s_fail;          // a wait ran out
    __shared__ long long s_max_iter;
    __shared__ unsigned int s_dep[kPollPer];    // the blocks that own this one's neighbours
    CgState* st = P.st;
    if (st->done) return;                      // uniform: set before the launch
    constexpr int U = K <= 3 ? 2 : 1;          // rows a trip of the product (loads in flight)
    const int n = P.n;
    const int64_t ld = P.ld;
    const int R = (((n + (int)gridDim.x - 1) / (int)gridDim.x) + 31) & ~31;
    const int lo = (int)min((int64_t)blockIdx.x * R, (int64_t)n);
    const int cnt = (int)min((int64_t)lo + R, (int64_t)n) - lo;
    const int tid = (int)threadIdx.x;
    const double* const rall = P.r;
    double* const rg = P.r + lo;
    double* const p = RES >= 1 ? dyn : P.p + lo;
    double* const sv = RES >= 2 ? dyn + R : P.s + lo;
    double* const y = RES >= 3 ? dyn + 2 * R : P.y + lo;
    double* const w = RES >= 4 ? dyn + 3 * R : P.w + lo;
    double* const rl = RES >= 5 ? dyn + 4 * R : rg;
    // resident rows: values [K][R], diagonal [R] unless unit, columns [K][R]
    double* const vm = dyn + RES * R;
    double* const dm = vm + K * R;
    int32_t* const cm = reinterpret_cast<int32_t*>(dm + (UNIT ? 0 : R));
    const double* const vg = P.v + lo;
    const double* const dg = P.d + lo;
    const int32_t* const cg = P.c + lo;
    GridSync* gs = P.gs;

    if (tid < kPollPer) s_dep[tid] = 0u;
    if (tid == 0) {
        sc[2] = sc[3] = 0.0;
        sc[4] = st->rnorm2;
        sc[5] = st->thresh2;
        sc[6] = st->rho;
        s_stop = 0;
        s_fail = 0;
        s_max_iter = st->max_iter;
    }
    __syncthreads();
    for (int i = tid; i < cnt; i += T) {
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const int c = cg[j * ld + i];
            const int q = c / R;
            if (q != (int)blockIdx.x && !((s_dep[q >> 5] >> (q & 31)) & 1u))
                atomicOr(&s_dep[q >> 5], 1u << (q & 31));
            if (MAT) {
                cm[j * R + i] = c;
                vm[j * R + i] = vg[j * ld + i];
            }
        }
        if (MAT && !UNIT) dm[i] = dg[i];
        p[i] = 0.0;
        sv[i] = 0.0;
        if (RES >= 3) y[i] = P.y[lo + i];
        if (RES >= 5) rl[i] = rg[i];
    }
    __syncthreads();
    unsigned int ep1 = 0, ep2 = 0;  // reductions of one and of two quantities so far
    bool ok = true;
    long long it = 0;
    for (;;) {
        double v[U][K], dd[U];
        int c[U][K];
        auto load = [&](int u, int i) {
#pragma unroll
            for (int j = 0; j < K; ++j) {
                c[u][j] = MAT ? cm[j * R + i] : cg[j * ld + i];
                v[u][j] = MAT ? vm[j * R + i] : vg[j * ld + i];
            }
            dd[u] = UNIT ? 1.0 : (MAT ? dm[i] : dg[i]);
        };
        // the first trip's rows are on their way while the neighbours finish
        if (!MAT) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (tid + u * T < cnt) load(u, tid + u * T);
        }
        if (it > 0) {
            dep_wait(gs, s_dep, (unsigned long long)it, s_fail);
            ok = s_fail == 0;
            if (!ok) break;
        }
        // the stop test every 8th iteration, and only once it can hold:
        // ||S r||^2 >= min(diag A) r.r (gamma of the iteration before stands
        // in for this one's, with a margin of 64)
        const bool check = (it & 7) == 7 && P.dmin * sc[6] <= 64.0 * sc[5];
        double sums[2] = {0.0, 0.0}, nn = 0.0;
        // A loop of its own for the passes that test, and one for the rows of a
        // last, short trip: branches in the rows would be predicated, and FP64
        // instructions that are off take their turns on the pipe all the same (33.9
        // against 30.1 us a step at 1.05M rows).
        auto product = [&](auto test) {
            auto rows = [&](auto count, int i0) {
                constexpr int N = decltype(count)::value;
                double g[N][K], re[N];
                if (MAT || i0 != tid) {
#pragma unroll
                    for (int u = 0; u < N; ++u) load(u, i0 + u * T);
                }
#pragma unroll
                for (int u = 0; u < N; ++u) {
#pragma unroll
                    for (int j = 0; j < K; ++j) g[u][j] = rall[c[u][j]];
                    re[u] = rl[i0 + u * T];
                }
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    const int i = i0 + u * T;
                    double acc = UNIT ? re[u] : dd[u] * re[u];
#pragma unroll
                    for (int j = 0; j < K; ++j) acc = fma(v[u][j], g[u][j], acc);
                    w[i] = acc;
                    sums[0] = fma(re[u], re[u], sums[0]);
                    sums[1] = fma(acc, re[u], sums[1]);
                    if constexpr (decltype(test)::value) {
                        const double t = P.wt[lo + i] * re[u];
                        nn = fma(t, t, nn);
                    }
                }
            };
            int i0 = tid;
            if (U > 1)
                for (; i0 + (U - 1) * T < cnt; i0 += U * T)
                    rows(std::integral_constant<int, U>{}, i0);
            for (; i0 < cnt; i0 += T) rows(std::integral_constant<int, 1>{}, i0);
        };
        if (check) product(std::true_type{});
        else product(std::false_type{});
        const long long it0 = it;
        if (check) {
            const double one[1] = {nn};
            tagged_allreduce<T>(one, ep1, P, s_fail, [&](const double* t) { sc[4] = t[0]; });
            __syncthreads();
            ok = s_fail == 0;
            if (!ok) break;
        }
        tagged_allreduce<T>(sums, ep2, P, s_fail, [&](const double* t) {
            const double g = t[0], dl = t[1];
            // exact solution, budget; input that is not finite
            int f = (__double_as_longlong(g) <= 0 || it0 >= s_max_iter) ? 1 : 0;
            if (!f && !positive_finite(g)) f = 2;
            if (check && sc[4] <= sc[5]) f = 1;
            if (!f) {
                // from p = s = 0 on the run's first pass: den = delta, beta = 0
                const double den = it0 == 0 ? dl : fma(-(g * g), sc[3], dl);
                // on the first pass p.Ap <= 0: not SPD; later, the
                // recurrence's difference lost its digits at the FP64 floor:
                // stop, and let the true residual decide
                if (!positive_finite(den)) f = it0 > 0 ? 1 : 2;
                sc[0] = g / den;
                sc[1] = g * sc[2];
                sc[3] = den;
            }
            sc[6] = g;
            s_stop = f;
        });
        __syncthreads();
        ok = s_fail == 0;
        if (!ok || s_stop) break;
        {
            const double alpha = sc[0], beta = sc[1];
            auto rows = [&](auto count, int i0) {
                constexpr int N = decltype(count)::value;
                double re[N], pe[N], se[N], we[N], ye[N];
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    const int i = i0 + u * T;
                    re[u] = rl[i];
                    pe[u] = p[i];
                    se[u] = sv[i];
                    we[u] = w[i];
                    ye[u] = y[i];
                }
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    const int i = i0 + u * T;
                    const double pn = fma(beta, pe[u], re[u]);
                    const double sn = fma(beta, se[u], we[u]);
                    const double rn = fma(-alpha, sn, re[u]);
                    rg[i] = rn;
                    if (RES >= 5) rl[i] = rn;
                    p[i] = pn;
                    sv[i] = sn;
                    y[i] = fma(alpha, pn, ye[u]);
                }
            };
            int i0 = tid;
            for (; i0 + T < cnt; i0 += 2 * T) rows(std::integral_constant<int, 2>{}, i0);
            for (; i0 < cnt; i0 += T) rows(std::integral_constant<int, 1>{}, i0);
        }
        ++it;
        halo_post(gs, (unsigned long long)it);
        if (tid == 32) {
            // for the next iteration: off the path that the blocks wait on
            const double ig = 1.0 / sc[6];
            sc[2] = ig;
            sc[3] = sc[3] * ig * ig;
        }
    }
    if (RES >= 3)
        for (int i = tid; i < cnt; i += T) P.y[lo + i] = y[i];
    if (blockIdx.x == 0 && tid == 0) {
        st->iter = it;
        st->rho = sc[6];
        st->rnorm2 = sc[4];
        st->status = ok ? (s_stop == 2 ? CPS_ERR_NOT_SPD : CPS_OK) : CPS_ERR_TIMEOUT;
        st->done = 2;
    }
}

using SchurKernel = void (*)(SchurArgs);

// The kernel of rows with K neighbours whose resident part of R rows fits a
// block's shared memory, most first, the dynamic bytes it takes and its threads.
struct Form {
    int threads, res;
    bool mat;
    SchurKernel kern;
};

// Resident rows leave few rows a thread: 512 threads synchronise faster (7.9
// against 8.8 us a step at 90k rows).  Streamed rows want 1024 threads' loads in
// flight.
template <int K, bool UNIT>
const Form* forms(int* count) {
    // Jacobi on all cells (K = 3) not without resident vectors (jacobi_resident)
    static const Form f[] = {{512, 5, true, k_resident_cg<512, K, 5, true, UNIT>},
                             {1024, 5, false, k_resident_cg<1024, K, 5, false, UNIT>},
                             {1024, 4, false, k_resident_cg<1024, K, 4, false, UNIT>},
                             {1024, 3, false, k_resident_cg<1024, K, 3, false, UNIT>},
                             {1024, 0, false,
                              K == 3 ? nullptr : k_resident_cg<1024, 6, 0, false, UNIT>}};
    *count = K == 3 ? 4 : 5;
    return f;
}

const Form* pick_form(int K, bool unit, int64_t R, size_t limit, size_t* bytes) {
    int count = 0;
    const Form* f = K == 3 ? forms<3, true>(&count)
                           : (unit ? forms<6, true>(&count) : forms<6, false>(&count));
    for (int i = 0; i < count; ++i) {
        cudaFuncAttributes at;
        if (cudaFuncGetAttributes(&at, f[i].kern) != cudaSuccess) return nullptr;
        const size_t row = 8 * f[i].res + (f[i].mat ? K * 12 + (unit ? 0 : 8) : 0);
        if ((size_t)R * row + at.sharedSizeBytes <= limit) {
            // the same bound whatever the rows: solves on other host threads
            // may launch this kernel with other sizes meanwhile
            if (cudaFuncSetAttribute(f[i].kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(limit - at.sharedSizeBytes)) != cudaSuccess)
                return nullptr;
            *bytes = (size_t)R * row;
            return &f[i];
        }
    }
    return nullptr;
}

// One cooperative launch of the loop over G blocks on the rows in P (its gs,
// st, stall and pb set here), with a persisting L2 window if win_bytes > 0.
int launch_resident(cps_sys s, SchurArgs P, int K, bool unit, int G, const void* win,
                    size_t win_bytes, cudaStream_t stream) {
    const int rc = ensure_gsync(s);
    if (rc) return rc;
    const int64_t R = ((((int64_t)P.n + G - 1) / G) + 31) & ~(int64_t)31;
    size_t smem = 0;
    const Form* f = pick_form(K, unit, R, s->ctx->smem_optin, &smem);
    if (!f) {
        cudaGetLastError();
        cps::set_error(s->ctx, "persistent: no kernel for this device");
        return CPS_ERR_CUDA;
    }
    P.gs = reinterpret_cast<GridSync*>(s->gsync);
    P.pb = reinterpret_cast<unsigned long long*>(P.gs + 1);
    P.st = s->st;
    P.stall = s->inject == CPS_TEST_STALL_BARRIER ? 1 : 0;
    s->inject = 0;
    // counter, timeout, the G flags in use and the slots start at zero
    CPS_CUDA_TRY(s->ctx, cudaMemsetAsync(s->gsync, 0,
                                         offsetof(GridSync, flag) +
                                             sizeof(unsigned long long) * kFlagStride * G,
                                         stream));
    CPS_CUDA_TRY(s->ctx, cudaMemsetAsync(P.pb, 0, sizeof(unsigned long long) * kSlotWords, stream));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G, 1, 1);
    cfg.blockDim = dim3(f->threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeAccessPolicyWindow;
    at[1].val.accessPolicyWindow.base_ptr = const_cast<void*>(win);
    at[1].val.accessPolicyWindow.num_bytes = win_bytes;
    at[1].val.accessPolicyWindow.hitRatio = 1.0f;
    at[1].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    at[1].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    cfg.attrs = at;
    cfg.numAttrs = win_bytes > 0 ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, f->kern, P);
    if (e != cudaSuccess) {
        cudaGetLastError();
        cps::set_error(s->ctx, std::string("persistent launch: ") + cudaGetErrorString(e));
        return CPS_ERR_CUDA;
    }
    return CPS_OK;
}

// Blocks for n rows: one per SM, at least 256 rows each.
int resident_grid(cps_sys s, int64_t n) {
    int G = s->ctx->num_sms < kGridMax ? s->ctx->num_sms : kGridMax;
    const int64_t most = (n + 255) / 256;
    if (most < G) G = (int)(most < 1 ? 1 : most);
    return G;
}

}  // namespace

// Synchronisation state of a system's persistent launches: the flags, and the
// slots of the tagged reductions behind them.
int ensure_gsync(cps_sys s) {
    if (!s->gsync && cudaMalloc((void**)&s->gsync, sizeof(GridSync) + sizeof(unsigned long long) *
                                                       kSlotWords) != cudaSuccess) {
        cudaGetLastError();
        s->gsync = nullptr;
        cps::set_error(s->ctx, "persistent: cudaMalloc failed");
        return CPS_ERR_NOMEM;
    }
    return CPS_OK;
}

// Frees the Schur rows of a system.
void free_schur(cps_sys s) {
    if (s->sch.buf) cudaFree(s->sch.buf);
    s->sch = SchurData{};
}

// The rows of S for this system's colour order (two colours), or of
// D^-1/2 S D^-1/2 (scaled): built on first use and when the form changes.
int schur_setup(cps_sys s, bool scaled, cudaStream_t stream) {
    SchurData& h = s->sch;
    const int64_t nR = s->colour_start[1], nB = s->nt - nR;
    if (!h.buf) {
        h.ld = (nB + 31) & ~(int64_t)31;
        // r, w, p, s, y first: one contiguous range for an L2 window
        const size_t bytes = (size_t)h.ld * (8 * (5 + kSlots + 3) + 4 * kSlots);
        cudaError_t e = cudaMalloc(&h.buf, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            h.buf = nullptr;
            cps::set_error(s->ctx, "Schur rows: cudaMalloc failed");
            return CPS_ERR_NOMEM;
        }
        double* q = static_cast<double*>(h.buf);
        h.r = q;
        h.w = q + h.ld;
        h.p = q + 2 * h.ld;
        h.s = q + 3 * h.ld;
        h.y = q + 4 * h.ld;
        h.v = q + 5 * h.ld;
        h.d = q + (5 + kSlots) * h.ld;
        h.wt = h.d + h.ld;
        h.dsc = h.wt + h.ld;
        h.c = reinterpret_cast<int32_t*>(h.dsc + h.ld);
        h.nB = nB;
        h.form = 0;
    }
    const int want = scaled ? 2 : 1;
    if (h.form == want || nB == 0) return CPS_OK;
    const int g = grid_for(s->ctx, nB);
    k_schur_rows<<<g, kBlock, 0, stream>>>(s->a, s->col, s->s, s->perm, s->iperm, s->nt, nR,
                                           (int)nB, h.ld, h.v, h.c, h.d, h.wt);
    if (scaled) k_schur_scale<<<g, kBlock, 0, stream>>>(h.v, h.c, h.d, (int)nB, h.ld, h.dsc, h.wt);
    CPS_CUDA_TRY(s->ctx, cudaGetLastError());
    h.form = want;
    return CPS_OK;
}

// A run's start from x (mesh order): y_R, y_B, r and the state in s->st.
int schur_init(cps_sys s, const double* b, const double* x, double rtol, long long budget,
               cudaStream_t stream) {
    const SchurData& h = s->sch;
    const int64_t nR = s->colour_start[1];
    const double* dsc = h.form == 2 ? h.dsc : nullptr;
    k_tc_red<<<s->grid, kBlock, 0, stream>>>(b, x, s->s, s->a, s->col, s->perm, s->nt, nR, s->wy);
    k_tc_init<<<s->grid, kBlock, 0, stream>>>(b, x, s->s, s->a, s->col, s->perm, dsc, s->wy, s->nt,
                                              nR, h.y, h.r, rtol, budget, s->partials, s->st);
    CPS_CUDA_TRY(s->ctx, cudaGetLastError());
    return CPS_OK;
}

// y of the whole system from the black solution, into s->wy.
int schur_back(cps_sys s, const double* b, cudaStream_t stream) {
    const SchurData& h = s->sch;
    k_tc_back<<<s->grid, kBlock, 0, stream>>>(b, h.y, h.form == 2 ? h.dsc : nullptr, s->s, s->a,
                                              s->col, s->iperm, s->nt, s->colour_start[1], s->wy);
    CPS_CUDA_TRY(s->ctx, cudaGetLastError());
    return CPS_OK;
}

// Bytes of the five vectors (the L2 window of the loop).
size_t schur_window_bytes(cps_sys s) { return sizeof(double) * 5 * (size_t)s->sch.ld; }

// The CG run from schur_init's state as one cooperative launch, with the five
// vectors in persisting L2 if window (the caller holds the set-aside).  State in
// s->st.
int schur_run(cps_sys s, bool window, cudaStream_t stream) {
    SchurData& h = s->sch;
    const int G = resident_grid(s, h.nB);
    SchurArgs P{};
    P.v = h.v;
    P.c = h.c;
    P.d = h.d;
    P.wt = h.wt;
    P.r = h.r;
    P.w = h.w;
    P.p = h.p;
    P.s = h.s;
    P.y = h.y;
    P.n = (int)h.nB;
    P.ld = h.ld;
    P.dmin = h.form == 2 ? 0.0 : s->diag_min;
    return launch_resident(s, P, kSlots, h.form == 2, G, h.buf,
                           window ? schur_window_bytes(s) : 0, stream);
}

// Whether jacobi_run takes this system (the vectors then in shared memory, and in
// *rows whether the rows are too; else 0): p, s and y of a block's rows have to fit
// its shared memory (up to 1.44M cells on 152 SMs).  With fewer resident the L1
// that is left does not hold the gathers: at 2.09M cells p and s resident took
// 48.1 us an iteration, k_persistent_gear (nothing resident, the L1 whole) 42.5;
// at 0.98M 21.8 against 23.1, at 0.4M 11.6 against 13.8, at 33k 5.7 against 7.8.
int jacobi_resident(cps_sys s, bool* rows) {
    const int G = resident_grid(s, s->nt);
    size_t smem = 0;
    const Form* f = pick_form(3, true, ((((s->nt + G - 1) / G) + 31) & ~(int64_t)31),
                              s->ctx->smem_optin, &smem);
    if (rows) *rows = f && f->mat;
    return f ? f->res : 0;
}

// FP64 Jacobi on all cells from the state k_init64 left (y, r), the same loop on
// the scaled matrix's own rows (s = A p in q, w = A r in p1), with r, p, q, y, p1
// in persisting L2 over win_bytes from win.
int jacobi_run(cps_sys s, const void* win, size_t win_bytes, cudaStream_t stream) {
    const int G = resident_grid(s, s->nt);
    SchurArgs P{};
    P.v = s->a;
    P.c = s->col;
    P.d = s->diag;
    P.wt = s->s;
    P.r = s->wr;
    P.w = s->wp1;
    P.p = s->wp0;
    P.s = s->wq;
    P.y = s->wy;
    P.n = (int)s->nt;
    P.ld = s->nt;
    P.dmin = s->diag_min;
    return launch_resident(s, P, 3, true, G, win, win_bytes, stream);
}

}  // namespace cps
