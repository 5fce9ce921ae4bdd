// mr_field.cu -- whole-field kernels, spread over the GPU: the initial state
// (mr_set_initial) and the reconstruction of an instance on its finest level
// (mr_get_finest); mr_run_static uses both.
//
// The persistent kernel gives an instance one block, which suits a step over a
// few hundred cells and not a pass over 2^Jmax of them.  Here a block owns a
// run of finest cells and a lone instance fills as many SMs as it has runs.
#include <cuda_runtime.h>

#include "mr_kernels.cuh"

namespace mrg {

// Multiresolution reconstruction on the finest level (Definition V: tree values,
// and every other cell predicted from the level above it).  A block takes CH
// finest cells and rebuilds, in shared memory, the window that each level
// contributes to them: the parents of the window below and gamma cells on
// either side, (CH >> gap) + 4 gamma + 2 cells at most, so a level costs the
// block one short pass and nothing is written but the result.  All windows are
// loaded first (positions outside the tree too: their slots exist), so the
// latency of global memory is paid once and not per level; the internal cells
// hold projections (see Worker::project_by_flux_pass).
// What bounds it: the Jmax - Jmin dependent passes over shared memory, a few
// microseconds.  The one-block version (a projection sweep and one pass over
// each level through global memory) took 37 us at Jmax 9, 100 us at Jmax 14
// (FP64 Euler), 1.5 ms at Jmax 18.
// CH: 128 cells up to Jmax 16, so that an instance of Jmax 14 fills 128 SMs (its
// FP64 sums would take 24 us on 32), 512 beyond, where a block's margins would
// double its reads.  Windows: CH + 22 * 14 positions at most.

template <typename T, int NF, int CH>
__global__ void __launch_bounds__(CH == 128 ? 128 : 256) mr_finest(const InstDesc *desc, const Tables<T> *tabs, double *out) {
    constexpr bool DQ = NF >= 4;
    constexpr int q = DQ ? (NF == 4 ? 3 : 5) : 2 * NF, nf = DQ ? 2 : NF;
    constexpr int CAP = CH + 320, NT = CH == 128 ? 128 : 256, R = CH / NT;
    __shared__ T val[CAP * q];
    __shared__ unsigned char have[CAP];
    __shared__ int wa[MAXLEV + 1], woff[32];  // first position of a level's window, its place in val; woff[31]: all of them
    const InstDesc &d = *desc;
    const int Jmin = d.Jmin, Jmax = d.Jmax, bc = d.bc, g = d.gamma, tid = threadIdx.x;
    const int N = 1 << Jmax;
    const int ch = min(CH, N), c0 = blockIdx.x * ch;
    const T *V = (const T *)d.V - (1LL << Jmin) * q;
    const uint32_t *I = d.masks + (long long)d.st->cur * d.Wtot;
    // this thread's finest cells: their tree bits and values on their way while
    // the windows are built
    uint32_t word[R];
    T f[R][q];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = min(c0 + tid + NT * r, N - 1);
        word[r] = Jmax > Jmin ? __ldg(&I[(uint32_t)(N + k) >> 6]) : FULL;
#pragma unroll
        for (int j = 0; j < q; ++j) f[r][j] = __ldg(&V[(size_t)(N + k) * q + j]);
    }
    if (tid < 32) {
        // Parents of [a, b] and g cells on either side, from level to level: a + 2g
        // and b - 2g are halved.  Lane i holds level Jmax - 1 - i.
        const int l = Jmax - 1 - tid;
        int n = 0;
        if (l >= Jmin) {
            const int a = ((c0 + 2 * g) >> (tid + 1)) - 2 * g, b = ((c0 + ch - 1 - 2 * g) >> (tid + 1)) + 2 * g;
            wa[l] = a;
            n = b - a + 1;
        }
        int x = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (tid >= o) x += y;
        }
        if (l >= Jmin) woff[l] = x - n;
        if (tid == 31) woff[31] = x;
    }
    __syncthreads();
    const int total = woff[31];
    // position x of level l: wrapped, or the boundary cell beyond a copy boundary
    auto inside = [&](int x, int l) -> int { return bc == 0 ? (x & ((1 << l) - 1)) : min(max(x, 0), (1 << l) - 1); };
    for (int i = tid; i < total; i += NT) {
        // the coarsest level whose window starts at or before i (the finest is first)
        int l = Jmax - 1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (l - o >= Jmin && woff[l - o] <= i) l -= o;
        const uint32_t h = (1u << l) + (uint32_t)inside(wa[l] + i - woff[l], l);
        const uint32_t bits = __ldg(&I[h >> 6]);
        const T *p = V + (size_t)h * q;
#pragma unroll
        for (int j = 0; j < q; ++j) val[i * q + j] = __ldg(&p[j]);
        have[i] = (unsigned char)((bits >> ((h >> 1) & 31u)) & 1u);
    }
    __syncthreads();
    const T *c = tabs->pc[g];
    const T c1 = __ldg(&c[0]), c2 = __ldg(&c[1]), c3 = __ldg(&c[2]);
    // value j of position x (in the domain) of level l from the window of level l - 1
    auto predicted = [&](int x, int l, int j) -> T {
        const T *w = val + (woff[l - 1] + (x >> 1) - wa[l - 1]) * q + j;
        T t = c1 * (w[q] - w[-q]);
        if (g > 1) t = t + c2 * (w[2 * q] - w[-2 * q]);
        if (g > 2) t = t + c3 * (w[3 * q] - w[-3 * q]);
        return (x & 1) ? w[0] - t : w[0] + t;
    };
    // a thread takes one population of a cell: a level is one short chain
    const int ci = tid / q, j = tid - ci * q;
    constexpr int CPB = NT / q;
    for (int l = Jmin + 1; l < Jmax; ++l) {
        const int o = woff[l], n = woff[l - 1] - o;
        if (ci < CPB)
            for (int i = ci; i < n; i += CPB)
                if (!have[o + i]) {
                    const int x = bc == 0 ? wa[l] + i : inside(wa[l] + i, l);
                    val[(o + i) * q + j] = predicted(x, l, j);
                }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = c0 + tid + NT * r;
        if (k >= c0 + ch) break;
        if (!((word[r] >> (((uint32_t)(N + k) >> 1) & 31u)) & 1u)) {
#pragma unroll
            for (int i = 0; i < q; ++i) f[r][i] = predicted(k, Jmax, i);
        }
        if constexpr (DQ) {
            double m0 = 0.0, m1 = 0.0;
#pragma unroll
            for (int i = 0; i < q; ++i) {
                m0 += (double)f[r][i];
                m1 += (dq_w(i) * d.lam) * (double)f[r][i];
            }
            out[k] = m0;
            out[(long long)N + k] = m1;
        } else {
#pragma unroll
            for (int i = 0; i < nf; ++i) out[(long long)i * N + k] = (double)f[r][2 * i] + (double)f[r][2 * i + 1];
        }
    }
}

// ---------------------------------------------------------------------------
// Initial state: the full tree, populations at equilibrium, projections of every
// level, lists, and the details' decisions for the first adaptation.
//
// mr_init_cells: a block takes a run of INIT_CELLS finest cells, evaluates their
// populations and projects them in shared memory up to the one cell (or, below
// Jmin, to level Jmin) above the run; the block that finishes an instance last
// (a ticket, no waiting) projects the levels above the runs, folds the runs'
// totals in their order and writes the state.  mr_init_details: a warp takes a
// word of 32 internal cells and writes their KEEP and REF words.
// What bounds them: with data of constant stretches the passes over shared memory
// and their barriers (issue a third of the cycles, DRAM 24 % and 40 % busy); with
// others the FP64 operations of the equilibria and the 3 q of a detail (two lanes a
// cycle and SM).  One block per instance took 2.6 ms for the batch of 4096 (FP64)
// and 11 ms for a lone Euler instance of Jmax = 18 (FP32), and the first adaptation
// 0.9 ms more for the latter; now about 1.0 ms and 0.05 ms, first decisions included.
// (x + y) / 2; of two equal values below half the largest double the value
// itself, without FP64 operations
__device__ __forceinline__ double mean_of(double x, double y) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (__double_as_longlong(x) == __double_as_longlong(y) && (hi & 0x7FF00000u) < 0x7FE00000u) return x;
    return half_f64(x + y);
}
__device__ __forceinline__ float mean_of(float x, float y) { return half_of<float>(x + y); }

template <typename T, int NF>
__device__ __forceinline__ void init_cells(const InstDesc &d, int chunk, const double *mcons, unsigned char *smem) {
    constexpr bool DQ = NF >= 4;
    constexpr int q = DQ ? (NF == 4 ? 3 : 5) : 2 * NF, nf = DQ ? 2 : NF;
    const int Jmin = d.Jmin, Jmax = d.Jmax, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = 1 << Jmax, ch = min(INIT_CELLS, N), nch = init_chunks_of(Jmax), c0 = chunk * ch;
    T *a = (T *)smem, *b = a + INIT_CELLS * q;
    double(*red)[8] = (double(*)[8])(smem + sizeof(T) * q * (INIT_CELLS + INIT_CELLS / 2));
    __shared__ unsigned heads[INIT_CELLS / 32];
    __shared__ unsigned short hlist[INIT_CELLS];
    T *V = (T *)d.V - (1LL << Jmin) * q;
    uint32_t *leaves = d.lists + d.list_off[L_LEAF], *inner = d.lists + d.list_off[L_INT] - (1 << Jmin);
    const double dx = ldexp(d.b - d.a, -Jmax);
    // The cells whose moments differ from their left neighbour's (and the first
    // of every 32) head a stretch of equal cells; only heads are evaluated, side
    // by side, and the others copy: the data of a Riemann problem are constant
    // but for some jumps, and the evaluation is what costs (a warp's FP64
    // instruction takes 16 cycles of the SM).
    for (int t = tid; t < INIT_CELLS; t += 256) {
        bool head = false;
        if (t < ch) {
            head = (t & 31) == 0;
            for (int j = 0; j < nf && !head; ++j) {
                const long long *x = (const long long *)mcons + (long long)j * N + c0 + t;
                head = x[0] != x[-1];
            }
            leaves[c0 + t] = (uint32_t)(N + c0 + t);
        }
        const unsigned hb = __ballot_sync(FULL, head);
        if (lane == 0) heads[t >> 5] = hb;
    }
    __syncthreads();
    // the heads listed in order: every warp scans the words' counts
    const int own = lane < INIT_CELLS / 32 ? __popc(heads[lane]) : 0;
    int upto = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, upto, o);
        if (lane >= o) upto += y;
    }
    const int nh = __shfl_sync(FULL, upto, 31);
    for (int t = tid; t < INIT_CELLS; t += 256) {
        const unsigned hb = heads[t >> 5];
        const int r = __shfl_sync(FULL, upto - own, t >> 5);
        if ((hb >> lane) & 1u) hlist[r + __popc(hb & ((1u << lane) - 1u))] = (unsigned short)t;
    }
    __syncthreads();
    double m[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
    for (int r = tid; r < nh; r += 256) {
        const int t = hlist[r], at = t & 31;
        const unsigned rest = (heads[t >> 5] >> at) >> 1;
        const int len = min(rest ? __ffs(rest) : 32 - at, ch - t);
        double mc[3], f[q], m0 = 0.0, m1 = 0.0;
        for (int j = 0; j < nf; ++j) mc[j] = mcons[(long long)j * N + c0 + t];
        if constexpr (DQ)
            dq_equilibrium_populations<q>(d, mc, f);
        else
            equilibrium_populations<NF>(d, mc, f);
        const double wgt = dx * (double)len;
#pragma unroll
        for (int j = 0; j < q; ++j) {
            const T x = (T)f[j];
            f[j] = (double)x;
            a[t * q + j] = x;
            if constexpr (DQ) {
                m0 += (double)x;
                m1 += (dq_w(j) * d.lam) * (double)x;
            }
        }
        if constexpr (DQ) {
            m[0] += wgt * m0;
            m[1] += wgt * m1;
        } else {
#pragma unroll
            for (int j = 0; j < nf; ++j) m[j] += wgt * (f[2 * j] + f[2 * j + 1]);
        }
    }
    __syncthreads();
    for (int t = tid; t < ch; t += 256) {
        const unsigned le = heads[t >> 5] & (FULL >> (31 - (t & 31)));
        const int from = (t & ~31) + 31 - __clz(le);
        if (from != t)
#pragma unroll
            for (int j = 0; j < q; ++j) a[t * q + j] = a[from * q + j];
    }
    // the run's totals, into the interface array (free until the first step)
#pragma unroll
    for (int j = 0; j < nf; ++j) {
        if (32 * warp < nh)
            for (int o = 16; o > 0; o >>= 1) m[j] += __shfl_down_sync(FULL, m[j], o);
        if (lane == 0) red[j][warp] = m[j];
    }
    __syncthreads();
    // the values from the shared copy, whose layout is theirs, 16 bytes a thread
    // (a run starts at a multiple of four cells)
    {
        uint4 *to = reinterpret_cast<uint4 *>(V + (size_t)(N + c0) * q);
        const uint4 *from = reinterpret_cast<const uint4 *>(a);
        for (int i = tid; i < ch * q * (int)sizeof(T) / 16; i += 256) to[i] = from[i];
    }
    if (tid < nf) {
        double x = red[tid][0];
        for (int w = 1; w < 8 && 32 * w < nh; ++w) x += red[tid][w];
        ((double *)d.Phi)[3 * chunk + tid] = x;
    }
    int l = Jmax - 1;
    for (int n = ch / 2; n >= 1 && l >= Jmin; n >>= 1, --l) {
        const uint32_t h0 = (1u << l) + (uint32_t)(c0 >> (Jmax - l));
        for (int e = tid; e < n * q; e += 256) {
            const int t = e / q, i = t * q + e;  // population e - t q of cell t: its first child's at 2 t q + that
            const T x = mean_of(a[i], a[i + q]);
            b[e] = x;
            V[(size_t)h0 * q + e] = x;
        }
        for (int t = tid; t < n; t += 256) inner[h0 + t] = h0 + t;
        __syncthreads();
        T *x = a;
        a = b;
        b = x;
    }
    // the tree: every cell above Jmax is internal; the runs share the words
    const int W = d.Wtot, wpc = W / nch;
    for (int w = chunk * wpc + tid; w < (chunk + 1) * wpc; w += 256)
        d.masks[w] = w == 0 ? (Jmax >= 5 ? 0xFFFFFFFEu : (1u << (1 << Jmax)) - 2u) : FULL;
    // the run that finishes last completes the instance
    InstState &st = *d.st;
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&st.chunks, 1u) == (unsigned)(nch - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (l = Jmax - 10; l >= Jmin; --l) {  // the levels above the runs, from values in L2
        for (uint32_t h = (1u << l) + tid; h < (2u << l); h += 256) {
#pragma unroll
            for (int j = 0; j < q; ++j)
                V[(size_t)h * q + j] = mean_of(__ldcg(&V[(size_t)(2u * h) * q + j]), __ldcg(&V[(size_t)(2u * h + 1u) * q + j]));
            inner[h] = h;
        }
        __threadfence_block();
        __syncthreads();
    }
    for (int j = 0; j < nf; ++j) {
        double x = 0.0;
        for (int c = tid; c < nch; c += 256) x += __ldcg((const double *)d.Phi + 3 * c + j);
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(FULL, x, o);
        if (lane == 0) red[j][warp] = x;
    }
    for (int j = tid; j < d.OW; j += 256) {  // occupancy of the tree: no word is empty
        uint32_t *occ = d.masks + (long long)(NMASK + 1) * W;
        occ[j] = W >= 32 ? FULL : (1u << W) - 1u;
    }
    for (int k = tid; k < MAXLEV + 2; k += 256) {
        st.seg[L_INT][k] = max(0, (1 << min(k, Jmax)) - (1 << Jmin));
        st.seg[L_PRED][k] = st.seg[L_GH][k] = 0;
    }
    __syncthreads();
    if (tid == 0) {
        for (int j = 0; j < 3; ++j) {
            double x = 0.0;
            if (j < nf)
                for (int w = 0; w < 8; ++w) x += red[j][w];
            st.mass[j] = x;
        }
        st.cur = M_I0;
        st.nleaf = N;
        st.status = ST_DETAILS;
        st.near_ties = st.first_ties = 0;
        st.deplev[0] = st.deplev[1] = 0u;
        st.updates = st.steps = st.passes = 0ULL;
        st.audit = 0.0;
        st.chunks = 0u;
#ifdef MRG_PHASE_TIMERS
        for (int p = 0; p < NPHASE; ++p) st.ptime[p] = 0ULL;
#endif
    }
}

__device__ __forceinline__ int variant_of_desc(const InstDesc &d) { return d.eq == 4 ? 4 : d.eq == 5 ? 5 : d.nf; }

template <typename T>
__global__ void __launch_bounds__(256, 4) mr_init_cells(const InstDesc *descs, const int *chunk_inst, const double *mcons) {
    __shared__ __align__(16) unsigned char smem[sizeof(T) * 6 * (INIT_CELLS + INIT_CELLS / 2) + 3 * 8 * sizeof(double)];
    const int inst = chunk_inst ? chunk_inst[blockIdx.x] : 0;
    const InstDesc &d = descs[inst];
    const int chunk = (int)blockIdx.x - (chunk_inst ? d.chunk0 : 0);
    const double *m = mcons + d.m_off;
    switch (variant_of_desc(d)) {
    case 1: init_cells<T, 1>(d, chunk, m, smem); break;
    case 2: init_cells<T, 2>(d, chunk, m, smem); break;
    case 3: init_cells<T, 3>(d, chunk, m, smem); break;
    case 4: init_cells<T, 4>(d, chunk, m, smem); break;
    default: init_cells<T, 5>(d, chunk, m, smem); break;
    }
}

template <typename T, int q, bool WIDE>
__device__ __forceinline__ void init_details(const InstDesc &d, int chunk, const Tables<T> &tab, const Thresholds &th) {
    const int W = d.Wtot, wpc = W / init_chunks_of(d.Jmax), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T *V = (const T *)d.V - (1LL << d.Jmin) * q;
    for (int w = chunk * wpc + warp; w < (chunk + 1) * wpc; w += 8) {
        const uint32_t p = 32u * w + lane;
        bool keep = false, ref = false, tie = false;
        if (p >= (1u << d.Jmin) && p < (1u << d.Jmax)) {
            bool flat = false;
            if constexpr (sizeof(T) == 8) {
                // equal values all over the stencil: the detail is zero (FP64
                // operations only where some lane of the warp has another)
                flat = true;
                const uint32_t lo = level_first(p);
                const long long *x = (const long long *)V;
#pragma unroll
                for (int h = 0; h < q; ++h) {
                    const long long v = x[p * (uint32_t)q + h];
                    flat = flat && x[2u * p * (uint32_t)q + h] == v;
                    for (int a = 1; a <= (WIDE ? d.gamma : 1); ++a)
                        flat = flat && x[neighbour(p, a, lo, d.bc) * (uint32_t)q + h] == v && x[neighbour(p, -a, lo, d.bc) * (uint32_t)q + h] == v;
                }
            }
            if (flat)
                decide_bits(0ull, th.eps_l[level_of(p) + 1], th.big_l[level_of(p) + 1], level_of(p) + 1 < d.Jmax, keep, ref, tie);
            else
                pair_decision<T, q, WIDE>(V, p, d.Jmax, d.bc, d.gamma, tab, th, keep, ref, tie);
        }
        const unsigned kb = __ballot_sync(FULL, keep), rb = __ballot_sync(FULL, ref), tb = __ballot_sync(FULL, tie);
        if (lane == 0) {
            d.masks[(long long)M_KEEP * W + w] = kb;
            d.masks[(long long)M_REF * W + w] = rb;
            if (tb) atomicAdd(&d.st->first_ties, __popc(tb));
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(256) mr_init_details(const InstDesc *descs, const int *chunk_inst, const Tables<T> *tabs) {
    __shared__ Thresholds th;
    const int inst = chunk_inst ? chunk_inst[blockIdx.x] : 0;
    const InstDesc &d = descs[inst];
    const int chunk = (int)blockIdx.x - (chunk_inst ? d.chunk0 : 0);
    for (int l = threadIdx.x; l <= MAXLEV; l += 256) th.set(d, l);
    __syncthreads();
    const Tables<T> &tab = *tabs;
    switch (variant_of_desc(d) + (d.gamma > 1 ? 8 : 0)) {
    case 1: init_details<T, 2, false>(d, chunk, tab, th); break;
    case 2: init_details<T, 4, false>(d, chunk, tab, th); break;
    case 3: init_details<T, 6, false>(d, chunk, tab, th); break;
    case 4: init_details<T, 3, false>(d, chunk, tab, th); break;
    case 5: init_details<T, 5, false>(d, chunk, tab, th); break;
    case 9: init_details<T, 2, true>(d, chunk, tab, th); break;
    case 10: init_details<T, 4, true>(d, chunk, tab, th); break;
    default: init_details<T, 6, true>(d, chunk, tab, th); break;
    }
}

template <typename T>
static cudaError_t init_of(const InstDesc *descs, const int *chunk_inst, int nchunk, const Tables<T> *tabs, const double *mcons,
                           cudaStream_t s) {
    mr_init_cells<T><<<nchunk, 256, 0, s>>>(descs, chunk_inst, mcons);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    mr_init_details<T><<<nchunk, 256, 0, s>>>(descs, chunk_inst, tabs);
    return cudaGetLastError();
}

template <typename T, int CH>
static void finest_go(int var, int grid, const InstDesc *desc, const Tables<T> *tabs, double *out, cudaStream_t s) {
    constexpr int NT = CH == 128 ? 128 : 256;
    switch (var) {
    case 1: mr_finest<T, 1, CH><<<grid, NT, 0, s>>>(desc, tabs, out); break;
    case 2: mr_finest<T, 2, CH><<<grid, NT, 0, s>>>(desc, tabs, out); break;
    case 3: mr_finest<T, 3, CH><<<grid, NT, 0, s>>>(desc, tabs, out); break;
    case 4: mr_finest<T, 4, CH><<<grid, NT, 0, s>>>(desc, tabs, out); break;
    default: mr_finest<T, 5, CH><<<grid, NT, 0, s>>>(desc, tabs, out); break;
    }
}
template <typename T>
static cudaError_t finest_of(int var, int Jmax, const InstDesc *desc, const Tables<T> *tabs, double *out, cudaStream_t s) {
    if (Jmax <= 16)
        finest_go<T, 128>(var, Jmax > 7 ? 1 << (Jmax - 7) : 1, desc, tabs, out, s);
    else
        finest_go<T, 512>(var, 1 << (Jmax - 9), desc, tabs, out, s);
    return cudaGetLastError();
}

}  // namespace mrg

// tables: Tables<float> or Tables<double> in device memory, by precision
int mrg_finest(bool fp32, int var, int Jmax, const mrg::InstDesc *desc, const void *tables, double *out, void *stream) {
    if (fp32) return (int)mrg::finest_of<float>(var, Jmax, desc, (const mrg::Tables<float> *)tables, out, (cudaStream_t)stream);
    return (int)mrg::finest_of<double>(var, Jmax, desc, (const mrg::Tables<double> *)tables, out, (cudaStream_t)stream);
}

int mrg_init(bool fp32, const mrg::InstDesc *descs, const int *chunk_inst, int nchunk, const void *tables, const double *mcons,
             void *stream) {
    if (fp32)
        return (int)mrg::init_of<float>(descs, chunk_inst, nchunk, (const mrg::Tables<float> *)tables, mcons, (cudaStream_t)stream);
    return (int)mrg::init_of<double>(descs, chunk_inst, nchunk, (const mrg::Tables<double> *)tables, mcons, (cudaStream_t)stream);
}
