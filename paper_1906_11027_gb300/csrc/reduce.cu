// reduce.cu -- deterministic double-precision reductions shared by all lattices.
// Every sum is formed in a fixed order (per-thread strided partials, then a
// fixed shared-memory tree), so results are bit-identical run to run.
#include <cuda_runtime.h>

#include "internal.h"

namespace lbm {

// One block: res[i] = sum over blocks of partials[b*width + i] for i < width-1,
// and the max for i = width-1.
__global__ void __launch_bounds__(256) k_sum_partials(const double* __restrict__ partials, int nblocks, int width,
                                                      double* __restrict__ res)
{
    __shared__ double sh[256];
    for (int i = 0; i < width; ++i) {
        const bool is_max = (i == width - 1) && (width == kObsWidth);
        double acc = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
            const double v = partials[static_cast<long long>(b) * width + i];
            acc = is_max ? fmax(acc, v) : acc + v;
        }
        sh[threadIdx.x] = acc;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) sh[threadIdx.x] = is_max ? fmax(sh[threadIdx.x], sh[threadIdx.x + s])
                                                          : sh[threadIdx.x] + sh[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) res[i] = sh[0];
        __syncthreads();
    }
}

cudaError_t launch_sum_partials(const double* partials, int nblocks, int width, double* res, cudaStream_t s)
{
    k_sum_partials<<<1, 256, 0, s>>>(partials, nblocks, width, res);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_block_sums(const double* __restrict__ x, long long n,
                                                    double* __restrict__ partials)
{
    __shared__ double sh[256];
    double acc = 0.0;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        acc += x[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

__global__ void k_divide(double* res, double n) { res[0] = res[0] / n; }

// res[0] = (sum of x) / n, deterministic.
cudaError_t launch_mean(const double* x, long long n, double* partials, int nblocks_max, double* res,
                        cudaStream_t s)
{
    long long nb = (n + 255) / 256;
    if (nb > nblocks_max) nb = nblocks_max;
    if (nb < 1) nb = 1;
    k_block_sums<<<static_cast<int>(nb), 256, 0, s>>>(x, n, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_sum_partials(partials, static_cast<int>(nb), 1, res, s);
    if (e != cudaSuccess) return e;
    k_divide<<<1, 1, 0, s>>>(res, static_cast<double>(n));
    return cudaGetLastError();
}

// Periodic distance of cell i to the centre node.  The offsets are whole numbers, so
// their squares are summed as integers and converted by the bits (a conversion
// instruction takes the FP64 pipe as long as an addition).
__device__ __forceinline__ int centre_offset(int i, int n)
{
    int d = i - n / 2;
    if (2 * d > n) d -= n;
    if (2 * d < -n) d += n;
    return d;
}
__device__ __forceinline__ double centre_distance(const DevParams64& p, int dim, long long i)
{
    const unsigned c = static_cast<unsigned>(i);
    const unsigned r = p.dnx.div(c);
    const int x = static_cast<int>(c - r * p.dnx.d);
    const int z = dim == 3 ? static_cast<int>(p.dny.div(r)) : 0;
    const int y = static_cast<int>(r) - z * p.ny;
    const long long dx = centre_offset(x, p.nx), dy = centre_offset(y, p.ny);
    const long long dz = dim == 3 ? centre_offset(z, p.nz) : 0;
    const unsigned long long q = static_cast<unsigned long long>(dx * dx + dy * dy + dz * dz);  // < 2^52
    return sqrt(__longlong_as_double(static_cast<long long>(q | 0x4330000000000000ull)) - 4503599627370496.0);
}

// Linear interpolation in a table of T densities over [-dmax, dmax], clamped.  scale =
// (T - 1) / (2 dmax).  The index comes from the bits of u - 1/2 + 1.5 2^52 (rounded to a
// whole number).
struct TableMap {
    double dmax, scale, shift;  // shift = dmax scale
    int T;
};
__device__ __forceinline__ double table_density(const double* table, const TableMap& m, double d)
{
    if ((__double2hiint(d) & 0x7fffffff) >= __double2hiint(m.dmax))  // |d| >= dmax, whose low word is zero
        return table[__double2hiint(d) < 0 ? 0 : m.T - 1];
    constexpr double magic = 6755399441055744.0;
    const double u = fma(d, m.scale, m.shift);
    const double t = fma(d, m.scale, m.shift - 0.5) + magic;
    int k = __double2loint(t);
    k = k < 0 ? 0 : k > m.T - 2 ? m.T - 2 : k;
    const double v = table[k];
    return fma(u - (t - magic), table[k + 1] - v, v);
}

__global__ void k_search_start(RadiusSearch* st, const double* res, double lo, double hi)
{
    RadiusSearch s{};
    s.cand[0] = lo;
    s.cand[1] = hi;
    s.cand[2] = hi;
    s.lo = lo;
    s.hi = hi;
    s.m0 = res[0];
    s.ok = 1;
    *st = s;
}

__device__ void search_update(RadiusSearch& s, const double (&m)[3])
{
    if (s.round == 0) {
        s.mlo = m[0];
        s.ok = isfinite(m[0]) && isfinite(m[1]) && (m[0] - s.m0) * (m[1] - s.m0) < 0.0;
    } else if (s.ok) {
        int k = 0;
        for (int it = 0; it < 2 && s.ok; ++it) {
            s.Re = s.cand[k];
            s.mm = m[k];
            s.last = k;
            if (!isfinite(s.mm)) {
                s.ok = 0;
            } else if ((s.mm - s.m0) * (s.mlo - s.m0) > 0.0) {
                s.lo = s.Re;
                s.mlo = s.mm;
                k = 2;
            } else {
                s.hi = s.Re;
                k = 1;
            }
        }
    }
    ++s.round;
    s.cand[0] = 0.5 * (s.lo + s.hi);
    s.cand[1] = 0.5 * (s.lo + s.cand[0]);
    s.cand[2] = 0.5 * (s.cand[0] + s.hi);
}

// Block sums of the candidates' fields, without storing them; the last block adds
// the blocks in their order and updates the search, so a round is two launches.
// Bounded by the FP64 pipe: a cell's distance is formed once for its 3 candidates,
// its offsets and table indices by integers, and the tables wait in shared memory as
// doubles.  Call with 256 x 256 cells: 0.82 ms -> 0.37 ms.
constexpr int kSearchT = 1024;
__global__ void __launch_bounds__(256) k_search_round(DevParams64 p, int dim, const float* __restrict__ tables,
                                                      TableMap map, RadiusSearch* st, double* partials)
{
    __shared__ double tab[3 * kSearchT];
    __shared__ double sh[256];
    __shared__ bool is_last;
    const double R[3] = {st->cand[0], st->cand[1], st->cand[2]};
    const int nc = st->round == 0 ? 2 : 3, T = map.T;
    for (int k = threadIdx.x; k < 3 * T; k += 256) tab[k] = static_cast<double>(tables[k]);
    __syncthreads();
    double acc[3] = {0.0, 0.0, 0.0};
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < p.N;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const double r = centre_distance(p, dim, i);
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] += table_density(tab + c * T, map, r - R[c]);
    }
    auto tree = [&](double v) {
        __syncthreads();
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
            __syncthreads();
        }
        return sh[0];
    };
    for (int c = 0; c < nc; ++c) {
        const double v = tree(acc[c]);
        if (threadIdx.x == 0) partials[static_cast<long long>(c) * gridDim.x + blockIdx.x] = v;
    }
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double m[3] = {0.0, 0.0, 0.0};
    for (int c = 0; c < nc; ++c) {
        double a = 0.0;
        for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += 256)
            a += __ldcg(partials + static_cast<long long>(c) * gridDim.x + b);
        m[c] = tree(a) / static_cast<double>(p.N);
    }
    if (threadIdx.x == 0) {
        RadiusSearch s = *st;
        search_update(s, m);
        s.done = 0;
        *st = s;
    }
}

__global__ void k_search_field(DevParams64 p, int dim, const float* __restrict__ tables, TableMap map,
                               const RadiusSearch* __restrict__ st, double* __restrict__ rho0)
{
    __shared__ double tab[kSearchT];
    const double R = st->Re, shift = st->m0 - st->mm;
    for (int k = threadIdx.x; k < map.T; k += blockDim.x) tab[k] = static_cast<double>(tables[st->last * map.T + k]);
    __syncthreads();
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < p.N;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        rho0[i] = table_density(tab, map, centre_distance(p, dim, i) - R) + shift;
}

static TableMap table_map(int T, double dmax)
{
    const double scale = (T - 1) / (2.0 * dmax);
    return {dmax, scale, dmax * scale, T};
}

cudaError_t launch_search_start(RadiusSearch* st, const double* res, double lo, double hi, cudaStream_t s)
{
    k_search_start<<<1, 1, 0, s>>>(st, res, lo, hi);
    return cudaGetLastError();
}

cudaError_t launch_search_round(const DevParams64& p, int dim, const float* tables, int T, double dmax,
                                RadiusSearch* st, double* partials, int nblocks_max, cudaStream_t s)
{
    long long nb = (p.N + 511) / 512;  // two cells a thread or more: every block loads the tables
    if (nb > nblocks_max) nb = nblocks_max;
    if (T != kSearchT) return cudaErrorInvalidValue;
    k_search_round<<<static_cast<int>(nb), 256, 0, s>>>(p, dim, tables, table_map(T, dmax), st, partials);
    return cudaGetLastError();
}

cudaError_t launch_search_field(const DevParams64& p, int dim, const float* tables, int T, double dmax,
                                const RadiusSearch* st, double* rho0, cudaStream_t s)
{
    const long long nb = (p.N + 255) / 256;
    if (T != kSearchT) return cudaErrorInvalidValue;
    k_search_field<<<static_cast<int>(nb < 2432 ? nb : 2432), 256, 0, s>>>(p, dim, tables, table_map(T, dmax), st, rho0);
    return cudaGetLastError();
}

}  // namespace lbm
