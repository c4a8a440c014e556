// Incomplete Cholesky IC(0) set-up in a multicolour order (Sec. 3.2.2: the
// corrector systems are solved by PCG with an incomplete Cholesky
// factorisation, computed once before the time loop, Sec. 3.1).
//
//   1. colour the cell graph so that no two neighbours share a colour:
//      first try two colours (union-find with parity; the cell graph of the
//      triangular lattice is bipartite), else greedy Jones-Plassmann
//      colouring with hashed priorities (at most 4 colours: every cell has at
//      most 3 neighbours);
//   2. order the cells colour by colour (stable inside a colour) and permute
//      the scaled matrix;
//   3. factor Ahat ~ L D L^T with L unit lower triangular on the pattern of
//      Ahat (no fill), colour by colour:
//        l_ik = (a_ik - sum_{m<k, m~i, m~k} l_im d_m l_km) / d_k,
//        d_i  = 1 - sum_k l_ik^2 d_k,
//      storing l_ik in the lower slots of row i and l_ki in the upper slots.
// On a two-coloured graph no cell has two mutually adjacent neighbours, so
// l_ik = a_ik / d_k and the black pivots are d_i = 1 - sum_red a_ik^2.
#include "cps_internal.cuh"

#include <cstring>

namespace cps {
namespace {

constexpr int kMaxColours = 16;

__device__ __forceinline__ uint32_t hash32(uint32_t x) {
    // lowbias32 integer hash.
    x ^= x >> 16;
    x *= 0x7feb352dU;
    x ^= x >> 15;
    x *= 0x846ca68bU;
    x ^= x >> 16;
    return x;
}

// Two-colouring by union-find with parity.  Word w[u] = (parent << 1) | t,
// t = parity of u relative to its parent; a root is its own parent with
// t = 0.  Roots are only ever hooked under a root of smaller index, so
// parents strictly decrease and every walk ends.  For a side (u, v) the two
// roots are joined so that u and v get opposite absolute parities; a side
// whose ends already share a root and a parity proves an odd cycle.
__device__ __forceinline__ int32_t uf_find(long long* w, int32_t u, int* par, int64_t n) {
    int acc = 0;
    int32_t x = u;
    for (int64_t guard = 0; guard <= n; ++guard) {
        const long long wx = __ldcg(&w[x]);
        const int32_t px = (int32_t)(wx >> 1);
        if (px == x) break;
        const long long wp = __ldcg(&w[px]);
        const int32_t gp = (int32_t)(wp >> 1);
        if (gp != px) {
            // path halving: point x at its grandparent, parities composed
            const long long nw = ((long long)gp << 1) | ((wx ^ wp) & 1LL);
            atomicCAS(reinterpret_cast<unsigned long long*>(&w[x]), (unsigned long long)wx,
                      (unsigned long long)nw);
        }
        acc ^= (int)(wx & 1);
        x = px;
    }
    *par = acc;
    return x;
}

__global__ void k_uf_init(long long* w, int64_t n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        w[e] = (long long)e << 1;
}

__global__ void k_uf_union(const int32_t* __restrict__ col, int64_t n, long long* w, int* flags) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll 1
        for (int j = 0; j < 3; ++j) {
            const int32_t c = col[j * n + e];
            if (c <= (int32_t)e) continue;           // each side once
            bool ok = false;
            for (int attempt = 0; attempt < (1 << 20); ++attempt) {
                int pu, pv;
                const int32_t ru = uf_find(w, (int32_t)e, &pu, n);
                const int32_t rv = uf_find(w, c, &pv, n);
                if (ru == rv) {
                    if (pu == pv) flags[0] = 1;      // odd cycle
                    ok = true;
                    break;
                }
                const int32_t hi = ru > rv ? ru : rv, lo = ru > rv ? rv : ru;
                const long long t = (long long)(pu ^ pv ^ 1);
                const unsigned long long expect = (unsigned long long)((long long)hi << 1);
                const unsigned long long want = (unsigned long long)(((long long)lo << 1) | t);
                if (atomicCAS(reinterpret_cast<unsigned long long*>(&w[hi]), expect, want) == expect) {
                    ok = true;
                    break;
                }
            }
            if (!ok) flags[1] = 1;                   // gave up: use the general colouring
        }
    }
}

__global__ void k_uf_colour(int64_t n, long long* w, int32_t* __restrict__ colour) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        int par;
        uf_find(w, (int32_t)e, &par, n);
        colour[e] = par;
    }
}

// One Jones-Plassmann round: an uncoloured cell whose priority beats every
// uncoloured neighbour takes the smallest colour no coloured neighbour has.
__global__ void k_jp_round(const int32_t* __restrict__ col, int64_t n, int32_t* colour,
                           int* remaining) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (colour[e] >= 0) continue;
        const uint32_t pe = hash32((uint32_t)e);
        bool top = true;
        unsigned used = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t c = col[j * n + e];
            if (c == (int32_t)e) continue;
            const int32_t cc = __ldcg(&colour[c]);
            if (cc < 0) {
                const uint32_t pc = hash32((uint32_t)c);
                if (pc > pe || (pc == pe && c > (int32_t)e)) top = false;
            } else if (cc < 32) {
                used |= 1u << cc;
            }
        }
        if (top) {
            colour[e] = __ffs(~used) - 1;
        } else {
            *remaining = 1;
        }
    }
}

__global__ void k_colour_max(const int32_t* __restrict__ colour, int64_t n, int* cmax) {
    int m = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        m = max(m, colour[e]);
    atomicMax(cmax, m);
}

// Tile b = cells [b*kBlock, (b+1)*kBlock): counts[c * nblk + b].  With col also
// whether two neighbours share a colour.
__global__ void __launch_bounds__(kBlock) k_colour_count(const int32_t* __restrict__ colour,
                                                         int64_t n, int ncol, int64_t nblk,
                                                         int* __restrict__ counts,
                                                         const int32_t* __restrict__ col,
                                                         int* conflict) {
    const int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const int my = i < n ? colour[i] : -1;
    for (int c = 0; c < ncol; ++c) {
        const int cnt = __syncthreads_count(my == c);
        if (threadIdx.x == 0) counts[c * nblk + blockIdx.x] = cnt;
    }
    if (!col || i >= n) return;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int32_t c = col[j * n + i];
        if (c != (int32_t)i && colour[c] == my) *conflict = 1;
    }
}

// Exclusive scan of counts (length m) in one block; colour c starts at
// offsets[c * nblk].
__global__ void __launch_bounds__(1024) k_scan(const int* __restrict__ counts, int64_t m,
                                               long long* __restrict__ offsets) {
    __shared__ long long part[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t per = (m + blockDim.x - 1) / blockDim.x;
    const int64_t b0 = min(m, threadIdx.x * per);
    const int64_t b1 = min(m, b0 + per);
    long long s = 0;
    for (int64_t k = b0; k < b1; ++k) s += counts[k];
    auto warp_scan = [&](long long v) {              // inclusive
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += u;
        }
        return v;
    };
    const long long in = warp_scan(s);
    if (lane == 31) part[warp] = in;
    __syncthreads();
    if (warp == 0) {
        const long long v = part[lane];
        part[lane] = warp_scan(v) - v;
    }
    __syncthreads();
    long long run = part[warp] + in - s;
    for (int64_t k = b0; k < b1; ++k) {
        offsets[k] = run;
        run += counts[k];
    }
}

__global__ void __launch_bounds__(kBlock) k_colour_scatter(const int32_t* __restrict__ colour,
                                                           int64_t n, int ncol, int64_t nblk,
                                                           const long long* __restrict__ offsets,
                                                           int32_t* __restrict__ perm,
                                                           int32_t* __restrict__ iperm) {
    __shared__ int wcount[kMaxColours][kBlock / 32];
    const int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int my = i < n ? colour[i] : -1;
    unsigned mine = 0;
    for (int c = 0; c < ncol; ++c) {
        const unsigned m = __ballot_sync(0xffffffffu, my == c);
        if (my == c) mine = m;
        if (lane == 0) wcount[c][warp] = __popc(m);
    }
    __syncthreads();
    if (my >= 0) {
        int rank = __popc(mine & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) rank += wcount[my][w];
        const long long dst = offsets[(int64_t)my * nblk + blockIdx.x] + rank;
        perm[dst] = (int32_t)i;
        iperm[i] = (int32_t)dst;
    }
}

__global__ void k_permute_matrix(const double* __restrict__ a, const int32_t* __restrict__ col,
                                 const double* __restrict__ s, const int32_t* __restrict__ perm,
                                 const int32_t* __restrict__ iperm, int64_t n,
                                 double* __restrict__ pa, int32_t* __restrict__ pcol,
                                 double* __restrict__ ps, float* __restrict__ pa32,
                                 float* __restrict__ ps32) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = perm[i];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double v = a[j * n + o];
            pa[j * n + i] = v;
            pa32[j * n + i] = (float)v;
            pcol[j * n + i] = iperm[col[j * n + o]];
        }
        ps[i] = s[o];
        ps32[i] = (float)s[o];
    }
}

// IC(0) rows of one colour [cs, ce): lower slots have pcol < i.
__global__ void k_ic0_factor(const double* __restrict__ pa, const int32_t* __restrict__ pcol,
                             int64_t n, int64_t cs, int64_t ce, double* __restrict__ pl,
                             double* __restrict__ pdinv, double* __restrict__ pdiag, int* err) {
    for (int64_t i = cs + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ce;
         i += (int64_t)gridDim.x * blockDim.x) {
        int kk[3], sl[3], m = 0;
        double av[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t c = pcol[j * n + i];
            pl[j * n + i] = 0.0;
            if (c < i) {
                kk[m] = c;
                sl[m] = j;
                av[m] = pa[j * n + i];
                ++m;
            }
        }
        // ascending column order
        for (int u = 0; u < m; ++u)
            for (int v = u + 1; v < m; ++v)
                if (kk[v] < kk[u]) {
                    int t = kk[u]; kk[u] = kk[v]; kk[v] = t;
                    t = sl[u]; sl[u] = sl[v]; sl[v] = t;
                    double d = av[u]; av[u] = av[v]; av[v] = d;
                }
        double L[3] = {0.0, 0.0, 0.0};
        double dsum = 0.0;
        for (int u = 0; u < m; ++u) {
            const int32_t k = kk[u];
            double v = av[u];
            for (int w = 0; w < u; ++w) {
                const int32_t mm = kk[w];
                for (int t = 0; t < 3; ++t)
                    if (pcol[t * n + k] == mm) v -= L[w] * (1.0 / pdinv[mm]) * pl[t * n + k];
            }
            L[u] = v * pdinv[k];
            pl[sl[u] * n + i] = L[u];
            dsum += L[u] * v;
        }
        const double d = 1.0 - dsum;
        if (!(d > 0.0) || !isfinite(d)) {
            set_error(err, CPS_ERR_NOT_SPD);
            pdinv[i] = 1.0;
            pdiag[i] = 1.0;
        } else {
            pdinv[i] = 1.0 / d;
            pdiag[i] = d;
        }
    }
}

// Upper slots of row i (pcol > i) take l_ki from row k's slot pointing at i;
// also the binary32 copies.
__global__ void k_ic0_upper(const int32_t* __restrict__ pcol, int64_t n, double* __restrict__ pl,
                            const double* __restrict__ pdinv, float* __restrict__ pl32,
                            float* __restrict__ pdinv32) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int32_t k = pcol[j * n + i];
            if (k > i) {
                double v = 0.0;
                for (int t = 0; t < 3; ++t)
                    if (pcol[t * n + k] == (int32_t)i) v = pl[t * n + k];
                pl[j * n + i] = v;
            }
        }
        pdinv32[i] = (float)pdinv[i];
    }
}

__global__ void k_to_float(const double* __restrict__ v, int64_t m, float* __restrict__ o) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x)
        o[i] = (float)v[i];
}

}  // namespace

// perm and iperm, one allocation.
static int alloc_order(cps_sys s) {
    if (s->perm) return CPS_OK;
    const size_t half = ((size_t)s->nt + 63) & ~(size_t)63;
    cudaError_t e = cudaMalloc((void**)&s->perm, sizeof(int32_t) * 2 * half);
    if (e != cudaSuccess) {
        cudaGetLastError();
        s->perm = nullptr;
        cps::set_error(s->ctx, std::string("set_precond: cudaMalloc: ") + cudaGetErrorString(e));
        return CPS_ERR_NOMEM;
    }
    s->iperm = s->perm + half;
    return CPS_OK;
}

static int alloc_ic0(cps_sys s) {
    const int64_t n = s->nt;
    struct {
        void** p;
        size_t bytes;
    } req[] = {{(void**)&s->pa, 24 * (size_t)n},        {(void**)&s->pcol, 12 * (size_t)n},
               {(void**)&s->pl, 24 * (size_t)n},        {(void**)&s->pdinv, 8 * (size_t)n},
               {(void**)&s->pdiag, 8 * (size_t)n},
               {(void**)&s->ps, 8 * (size_t)n},         {(void**)&s->pa32, 12 * (size_t)n},
               {(void**)&s->pl32, 12 * (size_t)n},      {(void**)&s->pdinv32, 4 * (size_t)n},
               {(void**)&s->ps32, 4 * (size_t)n}};
    for (auto& r : req) {
        if (*r.p) continue;
        cudaError_t e = cudaMalloc(r.p, r.bytes);
        if (e != cudaSuccess) {
            cps::set_error(s->ctx, std::string("set_precond: cudaMalloc: ") + cudaGetErrorString(e));
            return CPS_ERR_NOMEM;
        }
    }
    return CPS_OK;
}

// The ordering's scratch, in vectors that only a solve uses.
struct ColourScratch {
    long long* w;         // [nt] union-find words
    int32_t* colour;      // [nt]
    int* counts;          // [colours][tiles]
    long long* offsets;   // likewise
    int* flags;           // [0] odd cycle, [1] union gave up, [2] parity conflict, [3] max
                          // colour, [4..4+kRounds) Jones-Plassmann rounds still colouring
};

constexpr int kRounds = 16;

static ColourScratch scratch_of(cps_sys s) {
    return {reinterpret_cast<long long*>(s->wr), reinterpret_cast<int32_t*>(s->wq),
            reinterpret_cast<int*>(s->wy), reinterpret_cast<long long*>(s->wp1),
            reinterpret_cast<int*>(s->partials)};
}

static int64_t tiles(cps_sys s) { return (s->nt + kBlock - 1) / kBlock; }

// What enqueue_two_colours reads back, in the system's pinned state.
struct TwoColours {
    int flags[4];
    long long reds;
};

// Two colours for the cells, and the tiles' counts and offsets in them; *hst what
// came of it once the stream is synchronised.
static int enqueue_two_colours(cps_sys s, cudaStream_t stream) {
    const ColourScratch c = scratch_of(s);
    const int64_t n = s->nt, nblk = tiles(s);
    const int g = grid_for(s->ctx, n);
    TwoColours* h = reinterpret_cast<TwoColours*>(s->hst);
    static_assert(sizeof(TwoColours) <= sizeof(CgState), "pinned state");
    CPS_CUDA_TRY(s->ctx, cudaMemsetAsync(c.flags, 0, sizeof(int) * 4, stream));
    k_uf_init<<<g, kBlock, 0, stream>>>(c.w, n);
    k_uf_union<<<g, kBlock, 0, stream>>>(s->col, n, c.w, c.flags);
    k_uf_colour<<<g, kBlock, 0, stream>>>(n, c.w, c.colour);
    k_colour_count<<<(unsigned)nblk, kBlock, 0, stream>>>(c.colour, n, 2, nblk, c.counts, s->col,
                                                        c.flags + 2);
    k_scan<<<1, 1024, 0, stream>>>(c.counts, 2 * nblk, c.offsets);
    CPS_CUDA_TRY(s->ctx, cudaGetLastError());
    CPS_CUDA_TRY(s->ctx, cudaMemcpyAsync(h->flags, c.flags, sizeof(int) * 3, cudaMemcpyDeviceToHost,
                                         stream));
    CPS_CUDA_TRY(s->ctx, cudaMemcpyAsync(&h->reds, c.offsets + nblk, sizeof(long long),
                                         cudaMemcpyDeviceToHost, stream));
    return CPS_OK;
}

// enqueue_two_colours' result (the stream synchronised since): ncolours -1 where the
// graph has not two colours.
static bool has_two_colours(cps_sys s) {
    const TwoColours h = *reinterpret_cast<const TwoColours*>(s->hst);
    if (!h.flags[0] && !h.flags[1] && !h.flags[2] && h.reds != s->nt) return true;
    s->ncolours = -1;
    return false;
}

// The order in two colours from the same results.
static int finish_two_colours(cps_sys s, cudaStream_t stream) {
    const TwoColours h = *reinterpret_cast<const TwoColours*>(s->hst);
    const int rc = alloc_order(s);
    if (rc) return rc;
    const ColourScratch c = scratch_of(s);
    k_colour_scatter<<<(unsigned)tiles(s), kBlock, 0, stream>>>(c.colour, s->nt, 2, tiles(s),
                                                              c.offsets, s->perm, s->iperm);
    CPS_CUDA_TRY(s->ctx, cudaGetLastError());
    s->colour_start[0] = 0;
    s->colour_start[1] = h.reds;
    s->colour_start[2] = s->nt;
    s->ncolours = 2;
    return CPS_OK;
}

// Jones-Plassmann colours (at most max degree + 1 = 4) and the order by them.
static int order_by_priorities(cps_sys s, cudaStream_t stream) {
    const int64_t n = s->nt, nblk = tiles(s);
    const int g = grid_for(s->ctx, n);
    const ColourScratch c = scratch_of(s);
    int h[4 + kRounds];
    int rc = alloc_order(s);
    if (rc) return rc;
    CPS_CUDA_TRY(s->ctx, cudaMemsetAsync(c.flags, 0, sizeof(int) * 4, stream));
    CPS_CUDA_TRY(s->ctx, cudaMemsetAsync(c.colour, 0xFF, sizeof(int32_t) * n, stream));
    for (int64_t round = 0; round <= n; round += kRounds) {
        CPS_CUDA_TRY(s->ctx, cudaMemsetAsync(c.flags + 4, 0, sizeof(int) * kRounds, stream));
        for (int r = 0; r < kRounds; ++r)
            k_jp_round<<<g, kBlock, 0, stream>>>(s->col, n, c.colour, c.flags + 4 + r);
        CPS_CUDA_TRY(s->ctx, cudaMemcpyAsync(h + 4, c.flags + 4, sizeof(int) * kRounds,
                                             cudaMemcpyDeviceToHost, stream));
        CPS_CUDA_TRY(s->ctx, cudaStreamSynchronize(stream));
        if (h[4 + kRounds - 1] == 0) break;
    }
    k_colour_max<<<g, kBlock, 0, stream>>>(c.colour, n, c.flags + 3);
    CPS_CUDA_TRY(s->ctx, cudaMemcpyAsync(h + 3, c.flags + 3, sizeof(int), cudaMemcpyDeviceToHost,
                                         stream));
    CPS_CUDA_TRY(s->ctx, cudaStreamSynchronize(stream));
    const int ncol = h[3] + 1;
    if (ncol > kMaxColours) {
        cps::set_error(s->ctx, "set_precond: too many colours");
        return CPS_ERR_ARG;
    }
    k_colour_count<<<(unsigned)nblk, kBlock, 0, stream>>>(c.colour, n, ncol, nblk, c.counts, nullptr,
                                                        nullptr);
    k_scan<<<1, 1024, 0, stream>>>(c.counts, ncol * nblk, c.offsets);
    k_colour_scatter<<<(unsigned)nblk, kBlock, 0, stream>>>(c.colour, n, ncol, nblk, c.offsets,
                                                          s->perm, s->iperm);
    long long starts[kMaxColours];
    for (int k = 0; k < ncol; ++k)
        CPS_CUDA_TRY(s->ctx, cudaMemcpyAsync(&starts[k], c.offsets + (int64_t)k * nblk,
                                             sizeof(long long), cudaMemcpyDeviceToHost, stream));
    CPS_CUDA_TRY(s->ctx, cudaStreamSynchronize(stream));
    CPS_CUDA_TRY(s->ctx, cudaGetLastError());
    for (int k = 0; k < ncol; ++k) s->colour_start[k] = starts[k];
    s->colour_start[ncol] = n;
    s->ncolours = ncol;
    return CPS_OK;
}

// Orders the cells colour by colour, in two colours where they suffice.
static int order_cells(cps_sys s, cudaStream_t stream) {
    if (s->ncolours > 0) return CPS_OK;
    if (s->ncolours == 0) {
        int rc = enqueue_two_colours(s, stream);
        if (rc) return rc;
        CPS_CUDA_TRY(s->ctx, cudaStreamSynchronize(stream));
        if (has_two_colours(s)) return finish_two_colours(s, stream);
    }
    return order_by_priorities(s, stream);
}

// The two-colour orders and the (unscaled) Schur rows of n systems for the
// two-cyclic solves; *ok false where one of their graphs has not two colours.
// One synchronisation for all of them, no scratch allocated: 0.3 ms a system
// before, which a short solve does not repay.
int two_cyclic_setup(const cps_sys* systems, int n, cudaStream_t stream, bool* ok) {
    *ok = true;
    bool pending = false;
    for (int i = 0; i < n; ++i) {
        if (systems[i]->ncolours != 0 && systems[i]->ncolours != 2) *ok = false;
        if (systems[i]->ncolours == 0) pending = true;
    }
    if (!*ok) return CPS_OK;
    if (pending) {
        for (int i = 0; i < n; ++i) {
            if (systems[i]->ncolours != 0) continue;
            const int rc = enqueue_two_colours(systems[i], stream);
            if (rc) return rc;
        }
        CPS_CUDA_TRY(systems[0]->ctx, cudaStreamSynchronize(stream));
        for (int i = 0; i < n; ++i)
            if (systems[i]->ncolours == 0 && !has_two_colours(systems[i])) *ok = false;
        if (!*ok) return CPS_OK;              // the others stay unordered: nothing is kept for them
        for (int i = 0; i < n; ++i) {
            if (systems[i]->ncolours != 0) continue;
            const int rc = finish_two_colours(systems[i], stream);
            if (rc) return rc;
        }
    }
    for (int i = 0; i < n; ++i) {
        const int rc = schur_setup(systems[i], false, stream);
        if (rc) return rc;
    }
    return CPS_OK;
}

__global__ void k_same_columns(const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                               int64_t m, int* differ) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m;
         k += (int64_t)gridDim.x * blockDim.x)
        if (u[k] != v[k]) *differ = 1;
}

// The same for two systems of one size, which share a cell graph as a rule (the x
// and y systems of a mesh): y takes x's order if their columns are the same.
int two_cyclic_setup_pair(cps_sys x, cps_sys y, cudaStream_t stream, bool* ok) {
    const cps_sys both[2] = {x, y};
    if (x->ncolours != 0 || y->ncolours != 0 || x->nt != y->nt)
        return two_cyclic_setup(both, 2, stream, ok);
    *ok = false;
    int rc = enqueue_two_colours(x, stream);
    if (rc) return rc;
    int* differ = scratch_of(y).flags;
    int* h = reinterpret_cast<int*>(y->hst);
    CPS_CUDA_TRY(x->ctx, cudaMemsetAsync(differ, 0, sizeof(int), stream));
    k_same_columns<<<grid_for(x->ctx, 3 * x->nt), kBlock, 0, stream>>>(x->col, y->col, 3 * x->nt,
                                                                       differ);
    CPS_CUDA_TRY(x->ctx, cudaGetLastError());
    CPS_CUDA_TRY(x->ctx, cudaMemcpyAsync(h, differ, sizeof(int), cudaMemcpyDeviceToHost, stream));
    CPS_CUDA_TRY(x->ctx, cudaStreamSynchronize(stream));
    const bool same = *h == 0;
    if (!has_two_colours(x)) {
        if (same) y->ncolours = -1;
        return CPS_OK;
    }
    rc = finish_two_colours(x, stream);
    if (rc) return rc;
    if (same) {
        rc = alloc_order(y);
        if (rc) return rc;
        const size_t bytes = (size_t)(reinterpret_cast<char*>(x->iperm + x->nt) -
                                      reinterpret_cast<char*>(x->perm));
        CPS_CUDA_TRY(x->ctx, cudaMemcpyAsync(y->perm, x->perm, bytes, cudaMemcpyDeviceToDevice,
                                             stream));
        for (int k = 0; k < 3; ++k) y->colour_start[k] = x->colour_start[k];
        y->ncolours = 2;
    }
    return two_cyclic_setup(both, 2, stream, ok);
}

// Permutes the matrix into the colour order and factors it.
static int factor_ic0(cps_sys s, cudaStream_t stream) {
    int rc = alloc_ic0(s);
    if (rc) return rc;
    const int64_t n = s->nt;
    const int g = grid_for(s->ctx, n);
    int* err = nullptr;
    CPS_CUDA_TRY(s->ctx, cudaMallocAsync((void**)&err, sizeof(int), stream));
    cudaMemsetAsync(err, 0, sizeof(int), stream);
    k_permute_matrix<<<g, kBlock, 0, stream>>>(s->a, s->col, s->s, s->perm, s->iperm, n, s->pa,
                                               s->pcol, s->ps, s->pa32, s->ps32);
    for (int c = 0; c < s->ncolours; ++c)
        k_ic0_factor<<<g, kBlock, 0, stream>>>(s->pa, s->pcol, n, s->colour_start[c],
                                               s->colour_start[c + 1], s->pl, s->pdinv, s->pdiag,
                                               err);
    k_ic0_upper<<<g, kBlock, 0, stream>>>(s->pcol, n, s->pl, s->pdinv, s->pl32, s->pdinv32);
    k_to_float<<<grid_for(s->ctx, 3 * n), kBlock, 0, stream>>>(s->pl, 3 * n, s->pl32);
    int herr = 0;
    cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, stream);
    cudaFreeAsync(err, stream);
    if (cudaStreamSynchronize(stream) != cudaSuccess || cudaGetLastError() != cudaSuccess)
        return CPS_ERR_CUDA;
    if (herr) {
        cps::set_error(s->ctx, "set_precond: IC(0) pivot <= 0");
        return herr;
    }
    s->factored = true;
    return CPS_OK;
}

int precond_impl(cps_sys s, int precond, cudaStream_t stream) {
    if (precond == CPS_PC_JACOBI) {
        s->precond = precond;
        return CPS_OK;
    }
    if (precond != CPS_PC_IC0 && precond != CPS_PC_REDUCED) {
        cps::set_error(s->ctx, "set_precond: unknown preconditioner");
        return CPS_ERR_ARG;
    }
    if (!s->factored) {          // the matrix is fixed: ordered and factored once
        int rc = order_cells(s, stream);
        if (rc == CPS_OK) rc = factor_ic0(s, stream);
        if (rc != CPS_OK) {
            if (s->ctx->last_error.empty()) cps::set_error(s->ctx, "set_precond: IC(0) set-up failed");
            return rc;
        }
        if (precond == CPS_PC_REDUCED && s->ncolours != 2) s->precond = CPS_PC_JACOBI;
    }
    if (precond == CPS_PC_REDUCED && s->ncolours != 2) {
        cps::set_error(s->ctx, "set_precond: the cell graph is not two-colourable");
        return CPS_ERR_ARG;
    }
    s->precond = precond;
    return CPS_OK;
}

}  // namespace cps
