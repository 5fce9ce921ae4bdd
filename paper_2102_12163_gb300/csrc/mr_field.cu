// mr_field.cu -- whole-field kernels, spread over the GPU: the reconstruction
// of an instance on its finest level (mr_get_finest, mr_run_static).
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
constexpr int FIN_CH = 512, FIN_CAP = 896;  // finest cells of a block; positions of all its windows: 512 + 22 * 14 at most

template <typename T, int NF>
__global__ void __launch_bounds__(256) mr_finest(const InstDesc *desc, const Tables<T> *tabs, double *out) {
    constexpr bool DQ = NF >= 4;
    constexpr int q = DQ ? (NF == 4 ? 3 : 5) : 2 * NF, nf = DQ ? 2 : NF;
    __shared__ T val[FIN_CAP * q];
    __shared__ unsigned char have[FIN_CAP];
    __shared__ int wa[MAXLEV + 1], woff[MAXLEV + 2];  // first position of a level's window, its place in val
    const InstDesc &d = *desc;
    const int Jmin = d.Jmin, Jmax = d.Jmax, bc = d.bc, g = d.gamma, tid = threadIdx.x;
    const int N = 1 << Jmax;
    const int ch = min(FIN_CH, N), c0 = blockIdx.x * ch;
    const T *V = (const T *)d.V - (1LL << Jmin) * q;
    const uint32_t *I = d.masks + (long long)d.st->cur * d.Wtot;
    if (tid == 0) {
        int a = c0, b = c0 + ch - 1, o = 0;
        for (int l = Jmax - 1; l >= Jmin; --l) {
            a = (a >> 1) - g;
            b = (b >> 1) + g;
            wa[l] = a;
            woff[l] = o;
            o += b - a + 1;
        }
        woff[MAXLEV + 1] = o;
    }
    __syncthreads();
    const int total = Jmax > Jmin ? woff[MAXLEV + 1] : 0;
    // position x of level l: wrapped, or the boundary cell beyond a copy boundary
    auto inside = [&](int x, int l) -> int { return bc == 0 ? (x & ((1 << l) - 1)) : min(max(x, 0), (1 << l) - 1); };
    for (int i = tid; i < total; i += 256) {
        int l = Jmax - 1;
        while (l > Jmin && i >= woff[l - 1]) --l;
        const uint32_t h = (1u << l) + (uint32_t)inside(wa[l] + i - woff[l], l);
        const uint32_t word = __ldg(&I[h >> 6]);
        const T *p = V + (size_t)h * q;
#pragma unroll
        for (int j = 0; j < q; ++j) val[i * q + j] = __ldg(&p[j]);
        have[i] = (unsigned char)((word >> ((h >> 1) & 31u)) & 1u);
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
    for (int l = Jmin + 1; l < Jmax; ++l) {
        const int o = woff[l], n = woff[l - 1] - o;
        for (int i = tid; i < n; i += 256)
            if (!have[o + i]) {
                const int x = bc == 0 ? wa[l] + i : inside(wa[l] + i, l);
#pragma unroll
                for (int j = 0; j < q; ++j) val[(o + i) * q + j] = predicted(x, l, j);
            }
        __syncthreads();
    }
    for (int k = c0 + tid; k < c0 + ch; k += 256) {
        const uint32_t h = (uint32_t)(N + k);
        T f[q];
        if (Jmax == Jmin || bit_of(I, h >> 1)) {
            const T *p = V + (size_t)h * q;
#pragma unroll
            for (int j = 0; j < q; ++j) f[j] = p[j];
        } else {
#pragma unroll
            for (int j = 0; j < q; ++j) f[j] = predicted(k, Jmax, j);
        }
        if constexpr (DQ) {
            double m0 = 0.0, m1 = 0.0;
#pragma unroll
            for (int j = 0; j < q; ++j) {
                m0 += (double)f[j];
                m1 += (dq_w(j) * d.lam) * (double)f[j];
            }
            out[k] = m0;
            out[(long long)N + k] = m1;
        } else {
#pragma unroll
            for (int j = 0; j < nf; ++j) out[(long long)j * N + k] = (double)f[2 * j] + (double)f[2 * j + 1];
        }
    }
}

template <typename T>
static cudaError_t finest_of(int var, int Jmax, const InstDesc *desc, const Tables<T> *tabs, double *out, cudaStream_t s) {
    const int grid = Jmax > 9 ? 1 << (Jmax - 9) : 1;
    static_assert(FIN_CH == 1 << 9, "finest cells of a block");
    switch (var) {
    case 1: mr_finest<T, 1><<<grid, 256, 0, s>>>(desc, tabs, out); break;
    case 2: mr_finest<T, 2><<<grid, 256, 0, s>>>(desc, tabs, out); break;
    case 3: mr_finest<T, 3><<<grid, 256, 0, s>>>(desc, tabs, out); break;
    case 4: mr_finest<T, 4><<<grid, 256, 0, s>>>(desc, tabs, out); break;
    default: mr_finest<T, 5><<<grid, 256, 0, s>>>(desc, tabs, out); break;
    }
    return cudaGetLastError();
}

}  // namespace mrg

// tables: Tables<float> or Tables<double> in device memory, by precision
int mrg_finest(bool fp32, int var, int Jmax, const mrg::InstDesc *desc, const void *tables, double *out, void *stream) {
    if (fp32) return (int)mrg::finest_of<float>(var, Jmax, desc, (const mrg::Tables<float> *)tables, out, (cudaStream_t)stream);
    return (int)mrg::finest_of<double>(var, Jmax, desc, (const mrg::Tables<double> *)tables, out, (cudaStream_t)stream);
}
