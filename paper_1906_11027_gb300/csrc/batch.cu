// batch.cu -- many independent 2-D D2Q9 domains (uneven sizes, each with its own
// G, tau, stencil order and initial droplet) advanced together by one persistent
// kernel per step, captured in a CUDA graph together with a per-domain steady
// check; converged domains retire and drop out of the work list.
//
// Work item = (domain, tile of TX cells along x, chunk of ZC rows along y); the
// tile width and chunk length are picked per batch by an autotuner that times
// each compiled shape on the batch's own domains (all shapes perform the same
// per-cell arithmetic, so the choice changes speed only).  Each
// item runs the one-pass march of the single-domain kernels: psi of the tile and
// its halo is formed one row ahead into a shared-memory ring, the populations
// wait in a shared-memory stash, then force (Eq. 1), Guo-forced BGK collision
// (Eqs. 3-4) and the pull-streamed store.  The item count lives in device
// memory, so a captured graph stays valid while the list shrinks.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "internal.h"
#include "trace.h"
#include "kernels.cuh"

namespace lbm {
namespace {

constexpr int kBMaxR = 3;  // largest stencil radius (10th order)
constexpr int kBNS = 2 * kBMaxR + 2;
constexpr int kQ9 = 9;

struct BatchDom {
    int nx, ny, order, ntx, nch, active;
    long long off;   // element offset of the domain in each population pool
    long long poff;  // element offset of the domain in the psi scratch field (two-pass shape)
    double G, omega, pref, rho_bar;
    float G_f, omega_f, pref_f, rho_bar_f;  // FP32 copies (set with the doubles on the host)
    Coll64 c64;                             // FP64 collision products
};

template <class Real>
__device__ __forceinline__ typename ParamsOf<Real>::T dom_params(const BatchDom& d)
{
    typename ParamsOf<Real>::T p{};
    p.nx = d.nx;
    p.ny = d.ny;
    p.nz = 1;
    p.N = static_cast<long long>(d.nx) * d.ny;
    p.G = d.G;
    p.omega = d.omega;
    p.pref = d.pref;
    p.rho_bar = d.rho_bar;
    p.G_f = d.G_f;
    p.omega_f = d.omega_f;
    p.pref_f = d.pref_f;
    p.rho_bar_f = d.rho_bar_f;
    if constexpr (std::is_same<Real, double>::value) p.c64 = d.c64;
    p.psi_kind = 0;
    return p;
}

// Operations with their rounding spelled out (the compiler may not contract them),
// on one cell or a packed pair of cells.
__device__ __forceinline__ float xadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float xmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float xfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float xrcp(float a) { return __frcp_rn(a); }  // = 1.f / a
__device__ __forceinline__ float2 xadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 xmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 xfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 xrcp(float2 a) { return make_float2(xrcp(a.x), xrcp(a.y)); }

// D2Q9 BGK collision on FP32 deviations: collide32's expressions with every rounding
// fixed, so that all FP32 shapes, one cell or two per thread, give the same bits.
// a: force sums of ForceSum, psi of the cell(s).
template <class V>
__device__ __forceinline__ void collide_batch(V (&f)[kQ9], V ax, V ay, V psi, const DevParams& p)
{
    auto c = [](float v) { return vsplat<V>(v); };
    auto sub = [&](V u, V v) { return xadd(u, vneg(v)); };
    const V gp = xmul(c(-p.G_f), psi);
    const V Fx = xmul(gp, ax), Fy = xmul(gp, ay);
    V s = f[0];
    const V d1 = sub(f[1], f[2]), d2 = sub(f[3], f[4]), d3 = sub(f[5], f[6]), d4 = sub(f[7], f[8]);
#pragma unroll
    for (int b = 1; b < kQ9; b += 2) s = xadd(s, xadd(f[b], f[b + 1]));
    const V jx = xadd(xadd(d1, d3), d4), jy = sub(xadd(d2, d3), d4);
    const V rho = xadd(c(p.rho_bar_f), s);
    const V inv = xrcp(rho);
    const V ux = xmul(xfma(c(0.5f), Fx, jx), inv), uy = xmul(xfma(c(0.5f), Fy, jy), inv);
    constexpr double cs2 = Lattice<kLatD2Q9>::cs2;
    const V ic2 = c(static_cast<float>(1.0 / cs2)), ic4 = c(static_cast<float>(1.0 / (cs2 * cs2)));
    const V om = c(p.omega_f), pref = c(p.pref_f), om1 = c(__fadd_rn(1.f, -p.omega_f));
    const V usq = xmul(xfma(ux, ux, xmul(uy, uy)), c(static_cast<float>(0.5 / cs2)));
    const V uF = xfma(ux, Fx, xmul(uy, Fy));
    const V orho = xmul(om, rho);
    const V nq = xmul(xmul(c(-1.f), orho), usq);
    const V A0 = xfma(xmul(xmul(c(-1.f), pref), uF), ic2, xfma(om, s, nq));
    const V Px = xmul(xfma(pref, Fx, xmul(orho, ux)), ic2), Py = xmul(xfma(pref, Fy, xmul(orho, uy)), ic2);
    const V h = xmul(c(0.5f), orho);
    const V Vx = xmul(xfma(pref, Fx, xmul(h, ux)), ic4), Vy = xmul(xfma(pref, Fy, xmul(h, uy)), ic4);
    const V w0 = c(static_cast<float>(4.0 / 9.0)), w1 = c(static_cast<float>(1.0 / 9.0)),
            w2 = c(static_cast<float>(1.0 / 36.0));
    f[0] = xfma(f[0], om1, xmul(w0, A0));
    auto pair = [&](int b, V cu, V cV, V cP, V w) {
        const V e = xfma(cu, cV, A0);
        f[b] = xfma(f[b], om1, xmul(w, xadd(e, cP)));
        f[b + 1] = xfma(f[b + 1], om1, xmul(w, sub(e, cP)));
    };
    pair(1, ux, Vx, Px, w1);
    pair(3, uy, Vy, Py, w1);
    pair(5, xadd(ux, uy), xadd(Vx, Vy), xadd(Px, Py), w2);
    pair(7, sub(ux, uy), sub(Vx, Vy), sub(Px, Py), w2);
}
template <class Real>
__device__ __forceinline__ void collide_any(Real (&f)[kQ9], const ForceSum<Real>& F, const typename ParamsOf<Real>::T& p)
{
    if constexpr (std::is_same<Real, float>::value) collide_batch<float>(f, F.a[0], F.a[1], F.psi, p);
    else collide<kLatD2Q9, 0>(f, F, p);
}

// One (tile, chunk) of one domain: the 2-D one-pass march with a shared-memory
// stash.  ring: [NS][EX] psi, stash: [R + 1][Q][TX] populations.
template <int ORD, class Real, int TX, int ZC>
__device__ void batch_item(const Real* __restrict__ A, Real* __restrict__ Bo, const typename ParamsOf<Real>::T& p, int x0, int m0,
                           Real* ring, Real* stash)
{
    using L = Lattice<kLatD2Q9>;
    using S = Stencil<2, ORD>;
    constexpr int R = S::radius;
    constexpr int RE = 1;
    constexpr int Q = kQ9;
    constexpr int EX = TX + 2 * R;
    constexpr int E = EX;
    constexpr int NS = 2 * R + 2;
    constexpr int NST = R + 1;
    Pops<Real, Q> P;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        P.in[b] = A + static_cast<long long>(b) * p.N;
        P.out[b] = Bo + static_cast<long long>(b) * p.N;
    }
    const int nm = p.ny;
    const int m1 = (m0 + ZC < nm) ? m0 + ZC : nm;
    const int tid = threadIdx.x;
    const int ix = x0 + tid;
    int ixo[2 * RE + 1];
    axis_offsets<RE>(wrap_any(ix, p.nx), p.nx, 1, ixo);
    const bool has_halo = tid < 2 * R;
    const int hex = (tid < R) ? tid : TX + tid;
    int hxo[2 * RE + 1];
    axis_offsets<RE>(wrap_any(x0 - R + hex, p.nx), p.nx, 1, hxo);
    const int zero[2 * RE + 1] = {};

    auto psi_slab = [&](int m) {
        int mo[2 * RE + 1];
        axis_offsets<RE>(wrap_near(m, nm), nm, p.nx, mo);
        Real* dst = ring + ring_slot(m, NS) * E;
        Real f[Q];
        gather_off<kLatD2Q9, Real, RE>(P, ixo, mo, zero, f);
        const Real s = sum_f<kLatD2Q9>(f);
        dst[tid + R] = psi_of<kLatD2Q9>(std::is_same<Real, float>::value ? Real(p.rho_bar) + s : s, p);
        Real* st = stash + static_cast<unsigned>(m + 4 * NST) % NST * (Q * TX) + tid;
        sfor<Q>([&](auto bI) {
            constexpr int b = decltype(bI)::value;
            st[b * TX] = f[b];
        });
        if (has_halo) {
            Real h[Q];
            gather_off<kLatD2Q9, Real, RE>(P, hxo, mo, zero, h);
            const Real sh = sum_f<kLatD2Q9>(h);
            dst[hex] = psi_of<kLatD2Q9>(std::is_same<Real, float>::value ? Real(p.rho_bar) + sh : sh, p);
        }
    };
    for (int m = m0 - R; m < m0 + R; ++m) psi_slab(m);
    const bool active = ix < p.nx;
    for (int m = m0; m < m1; ++m) {
        psi_slab(m + R);
        __syncthreads();
        if (active) {
            Real f[Q];
            const Real* st = stash + static_cast<unsigned>(m + 4 * NST) % NST * (Q * TX) + tid;
            sfor<Q>([&](auto bI) {
                constexpr int b = decltype(bI)::value;
                f[b] = st[b * TX];
            });
            ForceSum<Real> F;
            force_ring<kLatD2Q9, ORD, Real, EX, E, NS>(ring, m, tid + R, 0, F);
            collide_any(f, F, p);
            const int c = m * p.nx + ix;
            sfor<Q>([&](auto bI) {
                constexpr int b = decltype(bI)::value;
                P.out[b][c] = f[b];
            });
        }
    }
    (void)L::Q;
}

// Persistent step kernel: every CTA walks the work list with stride gridDim.x.
template <class Real, int TX, int ZC>
__global__ void __launch_bounds__(TX) k_batch_step(const BatchDom* __restrict__ doms, const int4* __restrict__ items,
                                                   const int* __restrict__ nitems, const Real* __restrict__ pool_in,
                                                   Real* __restrict__ pool_out)
{
    __shared__ Real ring[kBNS * (TX + 2 * kBMaxR)];
    __shared__ Real stash[(kBMaxR + 1) * kQ9 * TX];
    const int n = *nitems;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int4 w = items[it];
        const BatchDom d = doms[w.x];
        const auto p = dom_params<Real>(d);
        const Real* A = pool_in + d.off;
        Real* Bo = pool_out + d.off;
        const int x0 = w.y * TX, m0 = w.z * ZC;
        switch (d.order) {
        case 4: batch_item<4, Real, TX, ZC>(A, Bo, p, x0, m0, ring, stash); break;
        case 6: batch_item<6, Real, TX, ZC>(A, Bo, p, x0, m0, ring, stash); break;
        case 8: batch_item<8, Real, TX, ZC>(A, Bo, p, x0, m0, ring, stash); break;
        default: batch_item<10, Real, TX, ZC>(A, Bo, p, x0, m0, ring, stash); break;
        }
        __syncthreads();  // shared memory is reused by the next item
    }
}

// Segment-staged work item (FP32; nx a multiple of 4): the bulk-copy pipeline of
// the single-domain 2-D kernel.  A producer warp (threads TX .. TX + 31) copies,
// per row s and direction b, the contiguous segment of row s - c_by over
// x0 - 4 .. x0 + TX + 4 into a stage (two copies where it crosses the periodic x
// edge); the stage stays resident until the row collides.  mbarrier phases run
// on across the items a block processes.
template <int ORD, int TX, int ZC, int NSTG>
__device__ __forceinline__ void batch_item_seg(const float* __restrict__ A, float* __restrict__ Bo, const DevParams& p, int x0,
                               int m0, float* ring, float* stage, unsigned long long* bars, uint32_t& phase, bool& ok)
{
    using L = Lattice<kLatD2Q9>;
    constexpr int R = Stencil<2, ORD>::radius;
    constexpr int Q = kQ9;
    constexpr int XP = 4;
    constexpr int W = TX + 2 * XP;
    constexpr int EX = TX + 2 * R;
    constexpr int NS = 2 * R + 2;
    constexpr int STG = Q * W;
    static_assert(NSTG >= R + 2 && NSTG >= 2 * R && XP >= R + 1, "stages / pad");
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const bool producer = tid >= TX;
    const int nm = p.ny;
    const int m1 = (m0 + ZC < nm) ? m0 + ZC : nm;
    const long long N = static_cast<long long>(p.nx) * p.ny;
    int cby = 0;
    sfor<Q>([&](auto bI) {
        constexpr int b = decltype(bI)::value;
        constexpr int vy = L::T.v[b][1];
        if (lane == b) cby = vy;
    });
    const float* src_b = A + static_cast<long long>(lane < Q ? lane : 0) * N;
    const int base = m0 - R;
    auto issue = [&](int s) {
        const int slot = (s - base) % NSTG;
        const uint32_t bar = smem_u32(&bars[slot]);
        if (lane == 0) mbar_expect_tx(bar, static_cast<uint32_t>(STG * sizeof(float)));
        __syncwarp();
        if (lane < Q) {
            fence_proxy_async_smem();
            const float* row = src_b + static_cast<long long>(wrap_any(s - cby, nm)) * p.nx;
            uint32_t dst = smem_u32(stage + slot * STG + lane * W);
            int xs = x0 - XP, left = W;
            while (left > 0) {
                const int x = wrap_any(xs, p.nx);
                const int n = (p.nx - x < left) ? p.nx - x : left;
                bulk_g2s(dst, row + x, static_cast<uint32_t>(n * sizeof(float)), bar);
                dst += static_cast<uint32_t>(n * sizeof(float));
                xs += n;
                left -= n;
            }
        }
    };
    auto stage_of = [&](int s) { return stage + ((s - base) % NSTG) * STG; };
    auto wait_stage = [&](int s) {
        const int slot = (s - base) % NSTG;
        if (ok && !mbar_wait(smem_u32(&bars[slot]), (phase >> slot) & 1u)) ok = false;  // after a timeout, stop waiting
        phase ^= 1u << slot;
    };
    auto load_cell = [&](const float* st, int cx, float (&f)[Q]) {
        sfor<Q>([&](auto bI) {
            constexpr int b = decltype(bI)::value;
            constexpr int vx = L::T.v[b][0];
            f[b] = st[b * W + cx + XP - vx];
        });
    };
    auto rho_psi = [&](const float (&f)[Q]) {
        float sum = 0.f;
        sfor<Q>([&](auto bI) { sum += f[decltype(bI)::value]; });
        return psi_of<kLatD2Q9>(static_cast<float>(p.rho_bar) + sum, p);
    };
    auto psi_slab = [&](int s) {
        wait_stage(s);
        const float* st = stage_of(s);
        float* dst = ring + ring_slot(s, NS) * EX;
        float f[Q];
        load_cell(st, tid, f);
        dst[tid + R] = rho_psi(f);
        if (tid < 2 * R) {
            const int cx = (tid < R) ? tid - R : TX + tid - R;
            load_cell(st, cx, f);
            dst[cx + R] = rho_psi(f);
        }
    };
    int next = base;
    const int last = m1 - 1 + R;
    if (producer)
        for (; next <= last && next < base + NSTG; ++next) issue(next);
    if (!producer)
        for (int s = m0 - R; s < m0 + R; ++s) psi_slab(s);
    __syncthreads();
    if (producer)
        for (; next <= last && next < m0 + NSTG; ++next) issue(next);
    const bool active = !producer && (x0 + tid) < p.nx;
    for (int m = m0; m < m1; ++m) {
        if (!producer) psi_slab(m + R);
        __syncthreads();
        if (producer)
            for (; next <= last && next <= m - 1 + NSTG; ++next) issue(next);
        if (active) {
            float f[Q];
            load_cell(stage_of(m), tid, f);
            ForceSum<float> F;
            force_ring<kLatD2Q9, ORD, float, EX, EX, NS>(ring, m, tid + R, 0, F);
            collide_any(f, F, p);
            const long long c = static_cast<long long>(m) * p.nx + x0 + tid;
            sfor<Q>([&](auto bI) {
                constexpr int b = decltype(bI)::value;
                __stcs(Bo + b * N + c, f[b]);
            });
        }
    }
}

template <int TX, int ZC, int NSTG>
__global__ void __launch_bounds__(TX + 32) k_batch_step_seg(const BatchDom* __restrict__ doms,
                                                            const int4* __restrict__ items,
                                                            const int* __restrict__ nitems,
                                                            const float* __restrict__ pool_in,
                                                            float* __restrict__ pool_out, unsigned* __restrict__ err)
{
    __shared__ float ring[kBNS * (TX + 2 * kBMaxR)];
    __shared__ alignas(8) unsigned long long bars[NSTG];
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    float* stage = reinterpret_cast<float*>(dyn_smem);  // [NSTG][9][TX + 8]
    if (threadIdx.x == 0) {
        for (int k = 0; k < NSTG; ++k) mbar_init(smem_u32(&bars[k]), 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    bool ok = true;
    const int n = *nitems;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int4 w = items[it];
        const BatchDom d = doms[w.x];
        const auto p = dom_params<float>(d);
        const float* A = pool_in + d.off;
        float* Bo = pool_out + d.off;
        const int x0 = w.y * TX, m0 = w.z * ZC;
        switch (d.order) {
        case 4: batch_item_seg<4, TX, ZC, NSTG>(A, Bo, p, x0, m0, ring, stage, bars, phase, ok); break;
        case 6: batch_item_seg<6, TX, ZC, NSTG>(A, Bo, p, x0, m0, ring, stage, bars, phase, ok); break;
        case 8: batch_item_seg<8, TX, ZC, NSTG>(A, Bo, p, x0, m0, ring, stage, bars, phase, ok); break;
        default: batch_item_seg<10, TX, ZC, NSTG>(A, Bo, p, x0, m0, ring, stage, bars, phase, ok); break;
        }
        __syncthreads();  // stages and ring are reused by the next item
    }
    if (!ok && threadIdx.x == 0) atomicOr(err, kErrTimeout);
}

// Two-pass form of the batch step, for few active cells: the march of the other
// shapes runs its rows one after another, so a step cannot finish faster than
// one item's march however little work is left.  Here a step is two launches
// with one thread per cell and no sequential loop: k_batch_psi2 writes psi of
// every active cell to a scratch field, k_batch_fused2 gathers, takes the force
// from that field (the same pair order and arithmetic as the ring kernels, so the
// results are bitwise the same) and collides.  Work item = 256 consecutive cells
// of one domain.
template <int ORD, class Real>
__device__ __forceinline__ void force_global(const Real* __restrict__ psi, int nx, int ny, int x, int y,
                                             ForceSum<Real>& F)
{
    using S = Stencil<2, ORD>;
    F = ForceSum<Real>{};
    sfor<S::n / 2>([&](auto kI) {
        constexpr int a = 2 * decltype(kI)::value;
        constexpr int ex = S::T.v[a][0], ey = S::T.v[a][1];
        const Real d = psi[wrap_near(y + ey, ny) * nx + wrap_near(x + ex, nx)] -
                       psi[wrap_near(y - ey, ny) * nx + wrap_near(x - ex, nx)];
        force_add<kLatD2Q9, ORD, a>(F, d);
    });
    F.psi = psi[y * nx + x];
}

template <class Real>
__global__ void __launch_bounds__(256) k_batch_psi2(const BatchDom* __restrict__ doms, const int4* __restrict__ items,
                                                    const int* __restrict__ nitems, const Real* __restrict__ pool_in,
                                                    Real* __restrict__ psi_pool)
{
    const int n = *nitems;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int4 w = items[it];
        const BatchDom d = doms[w.x];
        const auto p = dom_params<Real>(d);
        const long long i = static_cast<long long>(w.y) * 256 + threadIdx.x;
        if (i >= p.N) continue;
        const int x = static_cast<int>(i % p.nx), y = static_cast<int>(i / p.nx);
        Real f[kQ9];
        gather<kLatD2Q9>(pool_in + d.off, p, x, y, 0, f);
        const Real s = sum_f<kLatD2Q9>(f);
        psi_pool[d.poff + i] = psi_of<kLatD2Q9>(std::is_same<Real, float>::value ? Real(p.rho_bar) + s : s, p);
    }
}

template <int ORD, class Real>
__device__ __forceinline__ void fused2_cell(const Real* __restrict__ A, const Real* __restrict__ psi,
                                            Real* __restrict__ Bo, const typename ParamsOf<Real>::T& p, long long i)
{
    const int x = static_cast<int>(i % p.nx), y = static_cast<int>(i / p.nx);
    Real f[kQ9];
    gather<kLatD2Q9>(A, p, x, y, 0, f);
    ForceSum<Real> F;
    force_global<ORD, Real>(psi, p.nx, p.ny, x, y, F);
    collide_any(f, F, p);
    sfor<kQ9>([&](auto bI) {
        constexpr int b = decltype(bI)::value;
        Bo[static_cast<long long>(b) * p.N + i] = f[b];
    });
}

template <class Real>
__global__ void __launch_bounds__(256) k_batch_fused2(const BatchDom* __restrict__ doms,
                                                      const int4* __restrict__ items, const int* __restrict__ nitems,
                                                      const Real* __restrict__ pool_in,
                                                      const Real* __restrict__ psi_pool, Real* __restrict__ pool_out)
{
    const int n = *nitems;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        const int4 w = items[it];
        const BatchDom d = doms[w.x];
        const auto p = dom_params<Real>(d);
        const long long i = static_cast<long long>(w.y) * 256 + threadIdx.x;
        if (i >= p.N) continue;
        const Real* A = pool_in + d.off;
        const Real* psi = psi_pool + d.poff;
        Real* Bo = pool_out + d.off;
        switch (d.order) {
        case 4: fused2_cell<4, Real>(A, psi, Bo, p, i); break;
        case 6: fused2_cell<6, Real>(A, psi, Bo, p, i); break;
        case 8: fused2_cell<8, Real>(A, psi, Bo, p, i); break;
        default: fused2_cell<10, Real>(A, psi, Bo, p, i); break;
        }
    }
}

// ---- resident shape (FP32, even nx): a domain lives in the shared memory of a cluster --
// Many steps per launch without touching HBM or L2 in between: a cluster of C blocks
// holds one domain, each block a band of rows with one halo row of populations and R
// halo rows of psi on each side, and wrapped columns left and right.  A step is two
// phases:
//   1. every thread pulls its cells' populations into registers and writes psi;
//   2. it forms the force from psi, collides and writes the populations back in place.
// What a neighbouring band needs (the psi rows, the three populations that leave
// through an edge row) goes straight into that block's halo through distributed shared
// memory, and one cluster barrier ends each phase, so a step costs no launch and no
// global traffic.  A thread takes the x-adjacent pair of cells of one column pair in up
// to kResRows rows: packed FP32 instructions, 8-byte shared accesses, addresses that
// differ by constants.  The per-cell arithmetic is that of the other shapes, bit for bit.
// Two warps per sub-partition with 255 registers each (8 rows of populations held across
// the barrier) beat four with spills or a branch per row.  Bound by the latency of
// shared-memory loads and packed instructions at that occupancy: 4096 cells of one SM
// take 4.6 us per step (order 4) to 5.6 us (order 10), 134 GLUPS with every SM busy;
// clusters of 16 leave part of a GPC idle (16 domains of 256^2: 69 GLUPS).  40 droplets of
// 64^2 to 256^2: 27 us per step with tile128_rows16, 15 us here; 5 of them 10.6 -> 5.4 us.
constexpr int kResThreads = 256;
constexpr int kResRows = 8;       // most rows per thread (144 registers of populations)
constexpr int kResMaxCluster = 16;
constexpr int kResTimed = 64;     // steps of the call that the tuner times

// (every thread arrives; the waits end because all blocks of a cluster run together and
// take the same number of steps)
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t addr, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

// Band of block `rank` of C: rows [y0, y0 + rows).
__host__ __device__ inline void band_of(int ny, int C, int rank, int& y0, int& rows)
{
    const int q = ny / C, rem = ny % C;
    rows = q + (rank < rem ? 1 : 0);
    y0 = rank * q + (rank < rem ? rank : rem);
}
// Columns on each side: of the populations (one wrapped, one for 8-byte pairs) and of
// psi (R rounded up to pairs).
constexpr int kResPad = 2;
__host__ __device__ constexpr int psi_pad(int R) { return (R + 1) / 2 * 2; }
// Shared memory of a block: populations [maxrows + 2][9][nx + 2 kResPad], psi
// [maxrows + 2R][nx + 2 psi_pad].
__host__ __device__ inline size_t resident_bytes(int nx, int maxrows, int R)
{
    return sizeof(float) * (static_cast<size_t>(maxrows + 2) * kQ9 * (nx + 2 * kResPad) +
                            static_cast<size_t>(maxrows + 2 * R) * (nx + 2 * psi_pad(R)));
}

// Rows that each thread takes: what a band needs, rounded up to 1, 2, 4 or 8 (more: the
// band does not fit).
__host__ __device__ inline int resident_rows_per_thread(int nx, int ny, int C)
{
    const int maxrows = (ny + C - 1) / C, per_col = kResThreads / (nx / 2);
    const int m = (maxrows + per_col - 1) / per_col;
    return m > 4 ? (m > kResRows ? m : 8) : m == 3 ? 4 : m;
}

// M: rows per thread.  A band's last strip of rows is moved up to end with the band, so
// every working thread has M rows and the compiler may interleave them; rows that two
// threads share get the same values from both.
template <int ORD, int M>
__device__ __forceinline__ void resident_domain(const BatchDom& d, const float* A0, float* B0,
                                                float* smem, int rank, int C, int nsteps)
{
    using L = Lattice<kLatD2Q9>;
    using S = Stencil<2, ORD>;
    constexpr int R = S::radius;
    constexpr int Q = kQ9;
    constexpr int XP = kResPad, PP = psi_pad(R);
    const auto p = dom_params<float>(d);
    const int nx = d.nx, ny = d.ny;
    int y0, rows;
    band_of(ny, C, rank, y0, rows);
    const int maxrows = (ny + C - 1) / C;
    const int SX = nx + 2 * XP, RS = Q * SX;  // population row: [9][SX]
    const int PS = nx + 2 * PP;
    float* A = smem;
    float* psi = smem + (maxrows + 2) * RS;
    const int N = nx * ny;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    constexpr int kWarps = kResThreads / 32;

    // the band with its halo rows and wrapped columns, a warp per row of one direction
    for (int k = warp; k < (rows + 2) * Q; k += kWarps) {
        const int r = k / Q, b = k - r * Q;
        const float* src = A0 + b * N + wrap_near(y0 + r - 1, ny) * nx;
        float* dst = A + r * RS + b * SX;
        for (int c = lane; c < SX; c += 32) dst[c] = src[wrap_near(c - XP, nx)];
    }
    // this thread's rows of its column pair
    const int half = nx / 2;
    const int per_col = kResThreads / half;  // threads per column pair (half <= kResThreads)
    const int strip = tid / half, x = 2 * (tid - strip * half);
    const bool active = strip < per_col && strip * M < rows;
    const int r0 = strip * M < rows - M ? strip * M : rows - M;
    const int up = rank == 0 ? C - 1 : rank - 1, dn = rank + 1 == C ? 0 : rank + 1;
    int yu, rows_up;
    band_of(ny, C, up, yu, rows_up);
    // this column pair in the halo rows of the neighbouring bands
    const uint32_t A_up = map_rank(smem_u32(A + (rows_up + 1) * RS + x + XP), up);
    const uint32_t A_dn = map_rank(smem_u32(A + x + XP), dn);
    const uint32_t psi_up = map_rank(smem_u32(psi + (rows_up + R) * PS + x + PP), up);
    const uint32_t psi_dn = map_rank(smem_u32(psi + x + PP), dn);
    const bool left = x == 0, right = x == nx - 2;
    const bool wrap_r = x < PP, wrap_l = x >= nx - PP;  // psi columns repeated past the right / left end
    const float rho_bar = static_cast<float>(p.rho_bar);
    float* const a = A + (r0 + 1) * RS + x + XP;
    float* const ps = psi + (r0 + R) * PS + x + PP;
    auto ld2 = [](const float* q) { return *reinterpret_cast<const float2*>(q); };
    auto st2 = [](float* q, float2 v) { *reinterpret_cast<float2*>(q) = v; };
    auto sync = [&]() {
        if (C == 1) __syncthreads();
        else cluster_sync();
    };
    __syncthreads();
    sync();  // every block of the cluster runs and holds its band

    for (int step = 0; step < nsteps; ++step) {
        float2 f[M][Q];
        if (active) {
            float2 v[M];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                float2 s = make_float2(0.f, 0.f);
                sfor<Q>([&](auto bI) {
                    constexpr int b = decltype(bI)::value;
                    constexpr int cx = L::T.v[b][0], cy = L::T.v[b][1];
                    const float* q = a + (i - cy) * RS + b * SX;
                    if constexpr (cx == 0) f[i][b] = ld2(q);
                    else f[i][b] = make_float2(q[-cx], q[1 - cx]);
                    s = xadd(s, f[i][b]);
                });
                v[i] = make_float2(psi_exp(__fadd_rn(rho_bar, s.x)), psi_exp(__fadd_rn(rho_bar, s.y)));
            }
#pragma unroll
            for (int i = 0; i < M; ++i) st2(ps + i * PS, v[i]);
            if (wrap_r || wrap_l) {
                const int o = wrap_r ? nx : -nx;
#pragma unroll
                for (int i = 0; i < M; ++i) st2(ps + i * PS + o, v[i]);
            }
            if (r0 < R) {
#pragma unroll
                for (int i = 0; i < M; ++i)
                    if (r0 + i < R) {
                        const uint32_t q = psi_up + 4u * ((r0 + i) * PS);
                        st_remote(q, v[i]);
                        if (wrap_r) st_remote(q + 4u * nx, v[i]);
                        if (wrap_l) st_remote(q - 4u * nx, v[i]);
                    }
            }
            if (r0 + M > rows - R) {
#pragma unroll
                for (int i = 0; i < M; ++i)
                    if (r0 + i >= rows - R) {
                        const uint32_t q = psi_dn + 4u * ((r0 + i - rows + R) * PS);
                        st_remote(q, v[i]);
                        if (wrap_r) st_remote(q + 4u * nx, v[i]);
                        if (wrap_l) st_remote(q - 4u * nx, v[i]);
                    }
            }
        }
        sync();
        if (active) {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                // psi of the pair shifted by (ex, ey), from aligned 8-byte loads
                auto tap = [&](auto exI, auto eyI) {
                    constexpr int ex = decltype(exI)::value, ey = decltype(eyI)::value;
                    const float* q = ps + (i + ey) * PS + ex;
                    if constexpr (ex % 2 == 0) return ld2(q);
                    else return make_float2(ld2(q - 1).y, ld2(q + 1).x);
                };
                float2 ax = make_float2(0.f, 0.f), ay = ax;
                sfor<S::n / 2>([&](auto kI) {
                    constexpr int k = 2 * decltype(kI)::value;
                    constexpr int ex = S::T.v[k][0], ey = S::T.v[k][1];
                    constexpr double wt = S::T.w[k] * L::cs2;
                    const float2 dp =
                        xadd(tap(std::integral_constant<int, ex>{}, std::integral_constant<int, ey>{}),
                             vneg(tap(std::integral_constant<int, -ex>{}, std::integral_constant<int, -ey>{})));
                    if constexpr (ex != 0) ax = xfma(vsplat<float2>(wt * ex), dp, ax);
                    if constexpr (ey != 0) ay = xfma(vsplat<float2>(wt * ey), dp, ay);
                });
                collide_batch<float2>(f[i], ax, ay, ld2(ps + i * PS), p);
            }
#pragma unroll
            for (int i = 0; i < M; ++i)
                sfor<Q>([&](auto bI) { st2(a + i * RS + decltype(bI)::value * SX, f[i][decltype(bI)::value]); });
            if (right) {
#pragma unroll
                for (int i = 0; i < M; ++i)
                    sfor<Q>([&](auto bI) {
                        constexpr int b = decltype(bI)::value, cx = L::T.v[b][0];
                        if constexpr (cx == 1) a[i * RS + b * SX + 1 - nx] = f[i][b].y;
                    });
            }
            if (left) {
#pragma unroll
                for (int i = 0; i < M; ++i)
                    sfor<Q>([&](auto bI) {
                        constexpr int b = decltype(bI)::value, cx = L::T.v[b][0];
                        if constexpr (cx == -1) a[i * RS + b * SX + nx] = f[i][b].x;
                    });
            }
            // what leaves the band, into the neighbours' halo rows
            auto leave = [&](uint32_t h, const float2 v, auto cxI) {
                constexpr int cx = decltype(cxI)::value;
                st_remote(h, v);
                if (cx == 1 && right) st_remote(h + 4u - 4u * nx, v.y);
                if (cx == -1 && left) st_remote(h + 4u * nx, v.x);
            };
            if (r0 == 0)
                sfor<Q>([&](auto bI) {
                    constexpr int b = decltype(bI)::value, cx = L::T.v[b][0], cy = L::T.v[b][1];
                    if constexpr (cy == -1) leave(A_up + 4u * (b * SX), f[0][b], std::integral_constant<int, cx>{});
                });
            if (r0 == rows - M)
                sfor<Q>([&](auto bI) {
                    constexpr int b = decltype(bI)::value, cx = L::T.v[b][0], cy = L::T.v[b][1];
                    if constexpr (cy == 1) leave(A_dn + 4u * (b * SX), f[M - 1][b], std::integral_constant<int, cx>{});
                });
        }
        sync();
    }
    // the band back to the pool
    for (int k = warp; k < rows * Q; k += kWarps) {
        const int r = k / Q, b = k - r * Q;
        const float* src = A + (r + 1) * RS + b * SX + XP;
        float* dst = B0 + b * N + (y0 + r) * nx;
        for (int c = lane; c < nx; c += 32) dst[c] = src[c];
    }
}

template <int ORD>
__device__ __forceinline__ void resident_rows(const BatchDom& d, const float* A0, float* B0, float* smem, int rank,
                                              int C, int nsteps)
{
    switch (resident_rows_per_thread(d.nx, d.ny, C)) {
    case 8: resident_domain<ORD, 8>(d, A0, B0, smem, rank, C, nsteps); break;
    case 4: resident_domain<ORD, 4>(d, A0, B0, smem, rank, C, nsteps); break;
    case 2: resident_domain<ORD, 2>(d, A0, B0, smem, rank, C, nsteps); break;
    default: resident_domain<ORD, 1>(d, A0, B0, smem, rank, C, nsteps); break;
    }
}

// One cluster per listed domain; every block of a cluster takes the same way through.
// After an even number of steps a domain goes back to where it came from, so the pools may
// be one buffer (all of it is read before the first cluster barrier, and written after the
// last).
__global__ void __launch_bounds__(kResThreads, 1) k_batch_resident(const BatchDom* __restrict__ doms,
                                                                   const int* __restrict__ list, int C,
                                                                   const float* pool_in, float* pool_out, int nsteps)
{
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    float* smem = reinterpret_cast<float*>(dyn_smem);
    const int rank = static_cast<int>(blockIdx.x) % C;
    const BatchDom d = doms[list[blockIdx.x / C]];
    if (!d.active) return;
    const float* A0 = pool_in + d.off;
    float* B0 = pool_out + d.off;
    switch (d.order) {
    case 4: resident_rows<4>(d, A0, B0, smem, rank, C, nsteps); break;
    case 6: resident_rows<6>(d, A0, B0, smem, rank, C, nsteps); break;
    case 8: resident_rows<8>(d, A0, B0, smem, rank, C, nsteps); break;
    default: resident_rows<10>(d, A0, B0, smem, rank, C, nsteps); break;
    }
}

// Per-cell macroscopic values of domain d at cell i (pulled populations, psi of
// the neighbourhood recomputed from the populations; used by the observables).
template <int ORD, class Real>
__device__ void batch_cell_obs(const Real* __restrict__ A, const typename ParamsOf<Real>::T& p, int x, int y, double& rho,
                               double (&mom)[3])
{
    using L = Lattice<kLatD2Q9>;
    using S = Stencil<2, ORD>;
    auto rho_at = [&](int xx, int yy) {
        Real f[kQ9];
        gather<kLatD2Q9>(A, p, wrap_any(xx, p.nx), wrap_any(yy, p.ny), 0, f);
        Real s = Real(0);
        sfor<kQ9>([&](auto bI) { s += f[decltype(bI)::value]; });
        return std::is_same<Real, float>::value ? Real(p.rho_bar) + s : s;
    };
    Real f[kQ9];
    gather<kLatD2Q9>(A, p, x, y, 0, f);
    double s = 0.0, j[2] = {0.0, 0.0};
    sfor<kQ9>([&](auto bI) {
        constexpr int b = decltype(bI)::value;
        constexpr int cx = L::T.v[b][0], cy = L::T.v[b][1];
        s += static_cast<double>(f[b]);
        j[0] += static_cast<double>(f[b]) * cx;
        j[1] += static_cast<double>(f[b]) * cy;
    });
    rho = std::is_same<Real, float>::value ? p.rho_bar + s : s;
    double acc[2] = {0.0, 0.0};
    sfor<S::n>([&](auto aI) {
        constexpr int a = decltype(aI)::value;
        constexpr int ex = S::T.v[a][0], ey = S::T.v[a][1];
        constexpr double wt = S::T.w[a] * L::cs2;
        const double ps = static_cast<double>(psi_of<kLatD2Q9>(rho_at(x + ex, y + ey), p));
        acc[0] += wt * ps * ex;
        acc[1] += wt * ps * ey;
    });
    const double gp = -p.G * static_cast<double>(psi_of<kLatD2Q9>(static_cast<Real>(rho), p));
    mom[0] = j[0] + 0.5 * (gp * acc[0]);
    mom[1] = j[1] + 0.5 * (gp * acc[1]);
    mom[2] = 0.0;
}

// Per-domain observables: one block per (domain, block slice); block partials
// are written per slice and summed per domain in a fixed order by k_batch_obs_final.
constexpr int kObsSlices = 8;
template <class Real>
__global__ void __launch_bounds__(256) k_batch_obs(const BatchDom* __restrict__ doms, const Real* __restrict__ pool,
                                                   const int* __restrict__ cur_of, const long long pool_stride,
                                                   double* __restrict__ partials, int ndom, int only_active)
{
    const int d = blockIdx.x / kObsSlices, slice = blockIdx.x % kObsSlices;
    if (d >= ndom) return;
    const BatchDom dm = doms[d];
    if (only_active && !dm.active) return;  // a retired domain keeps its last observables
    const auto p = dom_params<Real>(dm);
    const Real* A = pool + dm.off + (cur_of[d] ? pool_stride : 0);
    double v[kObsWidth] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    bool bad = false;
    for (long long i = static_cast<long long>(slice) * blockDim.x + threadIdx.x; i < p.N;
         i += static_cast<long long>(kObsSlices) * blockDim.x) {
        const int x = static_cast<int>(i % p.nx), y = static_cast<int>(i / p.nx);
        double rho, mom[3];
        switch (dm.order) {
        case 4: batch_cell_obs<4, Real>(A, p, x, y, rho, mom); break;
        case 6: batch_cell_obs<6, Real>(A, p, x, y, rho, mom); break;
        case 8: batch_cell_obs<8, Real>(A, p, x, y, rho, mom); break;
        default: batch_cell_obs<10, Real>(A, p, x, y, rho, mom); break;
        }
        const double ux = mom[0] / rho, uy = mom[1] / rho, uz = 0.0;
        const double um = sqrt(ux * ux + uy * uy + uz * uz);
        if (!isfinite(rho) || !isfinite(um)) bad = true;
        v[0] += rho;
        v[1] += mom[0];
        v[2] += mom[1];
        v[4] += um;
        v[5] = fmax(v[5], um);
    }
    if (bad) v[5] = INFINITY;  // a diverged domain reports max|u| = inf (fmax would skip NaN)
    block_reduce_obs(v, partials + static_cast<long long>(blockIdx.x) * kObsWidth);
}

// res[d*8 + 0..5] = sums (max) over the slices; 6: rho at the centre, 7: rho at node 0.
template <class Real>
__global__ void k_batch_obs_final(const BatchDom* __restrict__ doms, const Real* __restrict__ pool,
                                  const int* __restrict__ cur_of, const long long pool_stride,
                                  const double* __restrict__ partials, double* __restrict__ res, int ndom,
                                  int only_active)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= ndom) return;
    if (only_active && !doms[d].active) return;
    double acc[kObsWidth];
    for (int k = 0; k < kObsWidth; ++k) acc[k] = partials[static_cast<long long>(d) * kObsSlices * kObsWidth + k];
    for (int s = 1; s < kObsSlices; ++s)
        for (int k = 0; k < kObsWidth; ++k) {
            const double v = partials[(static_cast<long long>(d) * kObsSlices + s) * kObsWidth + k];
            acc[k] = (k == kObsWidth - 1) ? fmax(acc[k], v) : acc[k] + v;
        }
    for (int k = 0; k < kObsWidth; ++k) res[d * 8 + k] = acc[k];
    const BatchDom dm = doms[d];
    const auto p = dom_params<Real>(dm);
    const Real* A = pool + dm.off + (cur_of[d] ? pool_stride : 0);
    auto rho_at = [&](int x, int y) {
        Real f[kQ9];
        gather<kLatD2Q9>(A, p, x, y, 0, f);
        double s = 0.0;
        for (int b = 0; b < kQ9; ++b) s += static_cast<double>(f[b]);
        return std::is_same<Real, float>::value ? p.rho_bar + s : s;
    };
    res[d * 8 + 6] = rho_at(p.nx / 2, p.ny / 2);
    res[d * 8 + 7] = rho_at(0, 0);
}

template <class Real>
__global__ void k_batch_init(const BatchDom* __restrict__ doms, const double* __restrict__ init, int ndom,
                             Real* __restrict__ pool)
{
    using L = Lattice<kLatD2Q9>;
    const int d = blockIdx.y;
    if (d >= ndom) return;
    const BatchDom dm = doms[d];
    const auto p = dom_params<Real>(dm);
    const double rl = init[4 * d], rg = init[4 * d + 1], R = init[4 * d + 2], W = init[4 * d + 3];
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < p.N;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int x = static_cast<int>(i % p.nx), y = static_cast<int>(i / p.nx);
        sfor<kQ9>([&](auto bI) {
            constexpr int b = decltype(bI)::value;
            constexpr int cx = L::T.v[b][0], cy = L::T.v[b][1];
            constexpr double wb = L::T.w[b];
            // A_b(y) = w_b rho0(y + c_b): the pulled state is feq(rho0, 0)
            const int xs = shift_wrap_fwd<cx>(x, p.nx), ys = shift_wrap_fwd<cy>(y, p.ny);
            const double dx = min_image(xs, p.nx), dy = min_image(ys, p.ny);
            const double r = sqrt(dx * dx + dy * dy);
            const double rho0 = 0.5 * (rl + rg) - 0.5 * (rl - rg) * tanh(2.0 * (r - R) / W);
            const double v = std::is_same<Real, float>::value ? wb * (rho0 - p.rho_bar) : wb * rho0;
            pool[dm.off + static_cast<long long>(b) * p.N + i] = static_cast<Real>(v);
        });
    }
}

// State I/O of one domain, directions [q0, q0 + nq): f = pre-collision populations in double
// [nq][ny][nx], A the pool's storage of all nine (A_b(y) = f_b(y + c_b), FP32 less w_b rho_bar).  On the host the
// pull took 1.3 ms per 256 x 256 domain, here 10 us.
template <bool GET, class Real>
__global__ void __launch_bounds__(256) k_batch_io(int nx, int ny, double rho_bar, int q0, int nq,
                                                  Real* __restrict__ A, double* __restrict__ f)
{
    using L = Lattice<kLatD2Q9>;
    constexpr bool kDev = std::is_same<Real, float>::value;
    const long long N = static_cast<long long>(nx) * ny;
    const long long i = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
    if (i >= nq * N) return;
    const int k = static_cast<int>(i / N), b = q0 + k;
    const int y = static_cast<int>((i - k * N) / nx), x = static_cast<int>(i - k * N - static_cast<long long>(y) * nx);
    int cx = 0, cy = 0;
    double w = 0.0;
    sfor<kQ9>([&](auto bI) {
        constexpr int q = decltype(bI)::value;
        constexpr int vx = L::T.v[q][0], vy = L::T.v[q][1];
        constexpr double wq = L::T.w[q];
        if (b == q) {
            cx = vx;
            cy = vy;
            w = wq;
        }
    });
    if (GET) {
        const double v = static_cast<double>(A[b * N + static_cast<long long>(wrap_near(y - cy, ny)) * nx + wrap_near(x - cx, nx)]);
        f[i] = kDev ? v + w * rho_bar : v;
    } else {
        const double v = f[k * N + static_cast<long long>(wrap_near(y + cy, ny)) * nx + wrap_near(x + cx, nx)];
        A[b * N + i - k * N] = static_cast<Real>(kDev ? v - w * rho_bar : v);
    }
}

__global__ void k_batch_prev_init(const BatchDom* __restrict__ doms, const double* __restrict__ res,
                                  double* __restrict__ prev, int ndom)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d < ndom && doms[d].active) prev[d] = res[d * 8 + 5];
}

// Steady check after a block of K steps: retire domain d when
// |max|u|(t) - max|u|(t-K)| / K < max(tol, floor * max|u| / K).
__global__ void k_batch_check(BatchDom* __restrict__ doms, const double* __restrict__ res, double* __restrict__ prev,
                              int ndom, double tol, double floor_rel, int K, int* __restrict__ newly)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= ndom) return;
    if (!doms[d].active) return;
    const double u = res[d * 8 + 5];
    if (!isfinite(u)) {  // diverged: retire it, its observables stay non-finite
        doms[d].active = 0;
        atomicAdd(newly, 1);
        return;
    }
    const double thr = fmax(tol, floor_rel * u / K);
    if (prev[d] >= 0.0 && fabs(u - prev[d]) / K < thr) {
        doms[d].active = 0;
        atomicAdd(newly, 1);
    }
    prev[d] = u;
}

}  // namespace
}  // namespace lbm

using namespace lbm;

struct lbm_batch {
    int n;
    int fp32;
    int device;
    cudaStream_t stream;
    bool own_stream;
    lbm_params p0;
    std::vector<BatchDom> doms;
    std::vector<double> init;
    std::vector<int> cur_of;     // buffer holding each domain's state (0: pool A)
    std::vector<int64_t> steps;  // steps each domain has taken
    std::vector<int> retired_at_check;
    long long pool_elems;
    void* pool[2];
    void* psi_pool;  // psi of every cell, for the two-pass shape
    BatchDom* d_doms;
    int4* d_items;
    int* d_nitems;
    int* d_cur_of;
    double* d_init;
    double* d_partials;
    double* d_res;
    double* d_prev;
    int* d_newly;
    int* h_newly;  // pinned
    int nitems;
    int grid;
    int cur;  // global parity: pool[cur] holds the state of active domains
    int64_t global_step;
    cudaGraphExec_t graph[2];
    int graph_k;
    int graph_cur;  // parity the graph was captured from
    double graph_tol;  // tolerance of its check
    unsigned* d_err;  // device error word (a bounded wait that ran out)
    unsigned* h_err;  // pinned copy, read after every graph block
    int var;        // tile shape in use (index into the variant table)
    bool tuned;     // autotuner has run, or a shape was pinned
    bool pinned;    // a shape was pinned by lbm_batch_set_schedule (never re-tuned)
    long long tuned_cells;  // active cells when the shape was last tuned
    std::vector<double> tune_ms;  // ms per step of each shape (< 0: not timed; resident: of a call of kResTimed steps)
    bool res_tuned;               // the resident shape may take calls from `var`
    double res_fixed, res_step;   // ms of a resident call of n steps: res_fixed + n res_step
    // resident shape: domains by cluster size, largest first, each class on a stream
    // of its own so that the classes share the GPU
    struct ResClass {
        int C, first, count;  // list[first .. first + count)
        size_t bytes;         // shared memory of a block
    };
    std::vector<ResClass> res;
    int res_spread;      // how far the listed domains are spread (resident_sizes)
    int* d_list;
    cudaStream_t aux[kResMaxCluster];
    cudaEvent_t ev_fork, ev_join[kResMaxCluster];

    void* dalloc(size_t bytes)
    {
        if (p0.dev_alloc) return p0.dev_alloc(bytes, p0.alloc_ctx);
        void* p = nullptr;
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return p;
    }
    void dfree(void* p)
    {
        if (!p) return;
        if (p0.dev_free)
            p0.dev_free(p, p0.alloc_ctx);
        else
            cudaFree(p);
    }
};

namespace {

// Compiled tile shapes of the batch step kernel: TX cells per tile (= threads per
// CTA) by ZC rows per work item.
struct BatchVariant {
    const char* name;
    int tx, zc;
    cudaError_t (*launch)(lbm_batch* b, int parity);
    int (*occupancy)(int fp32);
    bool staged;   // bulk-copy staging: FP32 only, every nx a multiple of 4
    bool per_cell; // two-pass shape: items are 256 consecutive cells, not (tile, row chunk)
    bool resident; // steps a domain many times per launch inside a cluster: FP32 only, every domain must fit
};

template <int TX, int ZC>
cudaError_t launch_variant(lbm_batch* b, int parity)
{
    if (b->fp32)
        k_batch_step<float, TX, ZC><<<b->grid, TX, 0, b->stream>>>(
            b->d_doms, b->d_items, b->d_nitems, static_cast<const float*>(b->pool[parity]),
            static_cast<float*>(b->pool[parity ^ 1]));
    else
        k_batch_step<double, TX, ZC><<<b->grid, TX, 0, b->stream>>>(
            b->d_doms, b->d_items, b->d_nitems, static_cast<const double*>(b->pool[parity]),
            static_cast<double*>(b->pool[parity ^ 1]));
    return cudaGetLastError();
}

template <int TX, int ZC>
int occupancy_variant(int fp32)
{
    int occ = 0;
    if (fp32)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_step<float, TX, ZC>, TX, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_step<double, TX, ZC>, TX, 0);
    return occ;
}

template <int TX, int ZC, int NSTG>
constexpr size_t seg_dyn_bytes()
{
    return sizeof(float) * NSTG * kQ9 * (TX + 8);
}

template <int TX, int ZC, int NSTG>
cudaError_t launch_seg(lbm_batch* b, int parity)
{
    auto kern = &k_batch_step_seg<TX, ZC, NSTG>;
    kern<<<b->grid, TX + 32, seg_dyn_bytes<TX, ZC, NSTG>(), b->stream>>>(
        b->d_doms, b->d_items, b->d_nitems, static_cast<const float*>(b->pool[parity]),
        static_cast<float*>(b->pool[parity ^ 1]), b->d_err);
    return cudaGetLastError();
}

template <int TX, int ZC, int NSTG>
int occupancy_seg(int)
{
    auto kern = &k_batch_step_seg<TX, ZC, NSTG>;
    constexpr size_t dyn = seg_dyn_bytes<TX, ZC, NSTG>();
    // the 48 KB default covers static plus dynamic shared memory: set the limit for any request
    if (dyn > 0) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(dyn));
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, TX + 32, dyn);
    return occ;
}

cudaError_t launch_twopass(lbm_batch* b, int parity)
{
    if (b->fp32) {
        k_batch_psi2<float><<<b->grid, 256, 0, b->stream>>>(b->d_doms, b->d_items, b->d_nitems,
                                                             static_cast<const float*>(b->pool[parity]),
                                                             static_cast<float*>(b->psi_pool));
        k_batch_fused2<float><<<b->grid, 256, 0, b->stream>>>(
            b->d_doms, b->d_items, b->d_nitems, static_cast<const float*>(b->pool[parity]),
            static_cast<const float*>(b->psi_pool), static_cast<float*>(b->pool[parity ^ 1]));
    } else {
        k_batch_psi2<double><<<b->grid, 256, 0, b->stream>>>(b->d_doms, b->d_items, b->d_nitems,
                                                              static_cast<const double*>(b->pool[parity]),
                                                              static_cast<double*>(b->psi_pool));
        k_batch_fused2<double><<<b->grid, 256, 0, b->stream>>>(
            b->d_doms, b->d_items, b->d_nitems, static_cast<const double*>(b->pool[parity]),
            static_cast<const double*>(b->psi_pool), static_cast<double*>(b->pool[parity ^ 1]));
    }
    return cudaGetLastError();
}

int occupancy_twopass(int fp32)
{
    int a = 0, c = 0;
    if (fp32) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_batch_psi2<float>, 256, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, k_batch_fused2<float>, 256, 0);
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_batch_psi2<double>, 256, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, k_batch_fused2<double>, 256, 0);
    }
    return std::min(a, c);
}

// Whether bands of an nx x ny domain over C blocks fit the threads' rows and the shared
// memory; every band has the rows that its threads take at once.
bool resident_fits(int nx, int ny, int R, int C)
{
    const int M = resident_rows_per_thread(nx, ny, C);
    return M <= kResRows && ny / C >= std::max(R, M) && resident_bytes(nx, (ny + C - 1) / C, R) <= 227 * 1024;
}

// Blocks of the cluster that holds an nx x ny domain with a stencil of radius R: the
// fewest whose bands fit the threads' rows and the shared memory, times at most
// `spread` (to use SMs that would stand idle).  0: none does.
int resident_cluster(int nx, int ny, int R, int spread)
{
    if (nx % 2 != 0 || nx / 2 > kResThreads) return 0;
    for (int C = 1; C <= kResMaxCluster && ny / C >= R; ++C) {
        if (!resident_fits(nx, ny, R, C)) continue;
        for (int S = std::min({C * spread, kResMaxCluster, ny / R}); S > C; --S)
            if (resident_fits(nx, ny, R, S)) return S;
        return C;
    }
    return 0;
}

int radius_of(int order) { return order == 4 ? 1 : order == 10 ? 3 : 2; }

cudaLaunchConfig_t resident_config(int C, int count, size_t bytes, cudaStream_t s, cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(C * count));
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = static_cast<unsigned>(C);
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// FP32, and every domain fits a cluster of a size that the device can hold.
bool resident_applies(const lbm_batch* b)
{
    if (!b->fp32) return false;
    bool seen[kResMaxCluster + 1] = {};
    int most = 0;
    for (const auto& m : b->doms) {
        const int C = resident_cluster(m.nx, m.ny, radius_of(m.order), 1);
        if (C == 0) return false;
        seen[C] = true;
        most = std::max(most, resident_cluster(m.nx, m.ny, radius_of(m.order), kResMaxCluster));
    }
    seen[most] = true;  // domains spread at most this far
    if (cudaFuncSetAttribute(k_batch_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_batch_resident, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    for (int C = 1; C <= kResMaxCluster; ++C) {
        if (!seen[C]) continue;
        cudaLaunchAttribute attr{};
        const cudaLaunchConfig_t cfg = resident_config(C, 1, 227 * 1024, nullptr, &attr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_batch_resident, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            return false;
        }
    }
    return true;
}

cudaError_t resident_launch_class(lbm_batch* b, const lbm_batch::ResClass& k, int parity, int n, cudaStream_t s)
{
    cudaLaunchAttribute attr{};
    const cudaLaunchConfig_t cfg = resident_config(k.C, k.count, k.bytes, s, &attr);
    return cudaLaunchKernelEx(&cfg, k_batch_resident, static_cast<const BatchDom*>(b->d_doms),
                              static_cast<const int*>(b->d_list + k.first), k.C,
                              static_cast<const float*>(b->pool[parity]),
                              static_cast<float*>(b->pool[parity ^ (n & 1)]), n);
}

// n steps of every active domain: one launch per cluster size, forked from and joined
// to the batch's stream.
cudaError_t launch_resident(lbm_batch* b, int parity, int64_t n)
{
    constexpr int64_t kMost = 4096;  // steps per launch
    while (n > 0) {
        const int k = static_cast<int>(std::min(n, kMost));
        cudaError_t e = cudaSuccess;
        if (b->res.size() == 1) {
            e = resident_launch_class(b, b->res[0], parity, k, b->stream);
            if (e != cudaSuccess) return e;
        } else {
            if ((e = cudaEventRecord(b->ev_fork, b->stream)) != cudaSuccess) return e;
            for (size_t i = 0; i < b->res.size(); ++i) {
                if ((e = cudaStreamWaitEvent(b->aux[i], b->ev_fork, 0)) != cudaSuccess) return e;
                if ((e = resident_launch_class(b, b->res[i], parity, k, b->aux[i])) != cudaSuccess) return e;
                if ((e = cudaEventRecord(b->ev_join[i], b->aux[i])) != cudaSuccess) return e;
                if ((e = cudaStreamWaitEvent(b->stream, b->ev_join[i], 0)) != cudaSuccess) return e;
            }
        }
        parity ^= k & 1;
        n -= k;
    }
    return cudaSuccess;
}

const BatchVariant kBatchVariants[] = {
    {"tile64_rows16", 64, 16, &launch_variant<64, 16>, &occupancy_variant<64, 16>, false, false, false},
    {"tile32_rows16", 32, 16, &launch_variant<32, 16>, &occupancy_variant<32, 16>, false, false, false},
    {"tile32_rows32", 32, 32, &launch_variant<32, 32>, &occupancy_variant<32, 32>, false, false, false},
    {"tile64_rows8", 64, 8, &launch_variant<64, 8>, &occupancy_variant<64, 8>, false, false, false},
    {"tile64_rows32", 64, 32, &launch_variant<64, 32>, &occupancy_variant<64, 32>, false, false, false},
    {"tile128_rows16", 128, 16, &launch_variant<128, 16>, &occupancy_variant<128, 16>, false, false, false},
    {"tile128_rows32", 128, 32, &launch_variant<128, 32>, &occupancy_variant<128, 32>, false, false, false},
    {"staged64_rows32", 64, 32, &launch_seg<64, 32, 8>, &occupancy_seg<64, 32, 8>, true, false, false},
    {"staged128_rows32", 128, 32, &launch_seg<128, 32, 8>, &occupancy_seg<128, 32, 8>, true, false, false},
    {"staged128_rows64", 128, 64, &launch_seg<128, 64, 8>, &occupancy_seg<128, 64, 8>, true, false, false},
    {"staged256_rows64", 256, 64, &launch_seg<256, 64, 8>, &occupancy_seg<256, 64, 8>, true, false, false},
    {"staged64_rows1024", 64, 1024, &launch_seg<64, 1024, 8>, &occupancy_seg<64, 1024, 8>, true, false, false},
    {"staged128_rows1024", 128, 1024, &launch_seg<128, 1024, 8>, &occupancy_seg<128, 1024, 8>, true, false, false},
    {"tile32_rows8", 32, 8, &launch_variant<32, 8>, &occupancy_variant<32, 8>, false, false, false},
    {"twopass_cells256", 256, 1, &launch_twopass, &occupancy_twopass, false, true, false},
    {"resident_cluster", 0, 0, nullptr, nullptr, false, false, true},
};
constexpr int kNumBatchVariants = sizeof(kBatchVariants) / sizeof(kBatchVariants[0]);
constexpr int kMinTX = 32, kMinZC = 8;  // smallest tile and chunk of the table (item buffer size)

#define LBM_BCK(call)                                                                                  \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess) {                                                                       \
            char m_[256];                                                                              \
            std::snprintf(m_, sizeof(m_), "%s: %s", #call, cudaGetErrorString(e_));                    \
            return set_last_error(LBM_ECUDA, m_);                                                      \
        }                                                                                              \
    } while (0)

// Cluster sizes of the active domains (0: retired).  While the blocks would leave more
// than half of the SMs idle, domains spread over twice, four times, ... as many.  Returns
// the spread.
int resident_sizes(const lbm_batch* b, int nsm, std::vector<int>& C)
{
    C.assign(b->n, 0);
    int taken = 1;
    for (int spread = 1; spread <= kResMaxCluster; spread *= 2) {
        std::vector<int> Cs(b->n, 0);
        int blocks = 0;
        for (int d = 0; d < b->n; ++d) {
            const BatchDom& m = b->doms[d];
            if (!m.active) continue;
            Cs[d] = resident_cluster(m.nx, m.ny, radius_of(m.order), spread);
            blocks += Cs[d];
        }
        if (spread > 1 && blocks > nsm) break;
        C = Cs;
        taken = spread;
        if (2 * blocks > nsm) break;
    }
    return taken;
}

// Work of the resident shape: active domains grouped by cluster size, largest first.
// `only_if_better`: after domains have retired, only when the others would spread
// further or half of the listed clusters have nothing to do any more (a rebuilt list
// costs a new captured graph).  *rebuilt: whether the list was made anew.
int rebuild_resident(lbm_batch* b, bool only_if_better = false, bool* rebuilt = nullptr)
{
    int nsm = 0;
    LBM_BCK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, b->device));
    std::vector<int> C;
    const int spread = resident_sizes(b, nsm, C);
    int listed = 0, active = 0;
    for (const auto& k : b->res) listed += k.count;
    for (const auto& m : b->doms) active += m.active;
    if (rebuilt) *rebuilt = false;
    if (only_if_better && spread <= b->res_spread && 2 * active > listed) return LBM_OK;
    if (rebuilt) *rebuilt = true;
    b->res_spread = spread;
    std::vector<int> list;
    b->res.clear();
    for (int c = kResMaxCluster; c >= 1; --c) {
        lbm_batch::ResClass k{c, static_cast<int>(list.size()), 0, 0};
        for (int d = 0; d < b->n; ++d)
            if (C[d] == c) {
                const BatchDom& m = b->doms[d];
                list.push_back(d);
                ++k.count;
                k.bytes = std::max(k.bytes, resident_bytes(m.nx, (m.ny + c - 1) / c, radius_of(m.order)));
            }
        if (k.count) b->res.push_back(k);
    }
    if (!b->ev_fork) LBM_BCK(cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming));
    for (size_t i = 0; i < b->res.size(); ++i)
        if (!b->aux[i]) {
            LBM_BCK(cudaStreamCreateWithFlags(&b->aux[i], cudaStreamNonBlocking));
            LBM_BCK(cudaEventCreateWithFlags(&b->ev_join[i], cudaEventDisableTiming));
        }
    if (!list.empty())
        LBM_BCK(cudaMemcpyAsync(b->d_list, list.data(), sizeof(int) * list.size(), cudaMemcpyHostToDevice, b->stream));
    LBM_BCK(cudaStreamSynchronize(b->stream));
    return LBM_OK;
}

int rebuild_items(lbm_batch* b)
{
    const BatchVariant& v = kBatchVariants[b->var];
    if (v.resident) return LBM_OK;
    std::vector<int4> items;
    for (int d = 0; d < b->n; ++d) {
        BatchDom& m = b->doms[d];
        m.ntx = (m.nx + v.tx - 1) / v.tx;
        m.nch = (m.ny + v.zc - 1) / v.zc;
        if (!m.active) continue;
        if (v.per_cell) {
            const long long nb = (static_cast<long long>(m.nx) * m.ny + 255) / 256;
            for (long long k = 0; k < nb; ++k) items.push_back(make_int4(d, static_cast<int>(k), 0, 1));
            continue;
        }
        for (int c = 0; c < m.nch; ++c)
            for (int t = 0; t < m.ntx; ++t)
                items.push_back(make_int4(d, t, c, std::min(v.zc, m.ny - c * v.zc)));  // w: rows of the item
    }
    // longest items first: the persistent blocks take them in index order
    std::stable_sort(items.begin(), items.end(), [](const int4& a, const int4& c) { return a.w > c.w; });
    b->nitems = static_cast<int>(items.size());
    if (!items.empty())
        LBM_BCK(cudaMemcpyAsync(b->d_items, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice,
                                b->stream));
    LBM_BCK(cudaMemcpyAsync(b->d_nitems, &b->nitems, sizeof(int), cudaMemcpyHostToDevice, b->stream));
    LBM_BCK(cudaStreamSynchronize(b->stream));
    return LBM_OK;
}

// Whether a call of n steps goes to the resident shape.  It reads and writes the state
// once per call and forks and joins a stream per cluster size, which only many steps pay
// back: 40 domains of 64^2 to 256^2, us per step, in calls of 1, 4, 16 and 64 steps:
// resident 107, 38, 24, 20 and tile128_rows16 29, 27, 27, 27; one domain of 64^2: 10, 3.5,
// 1.6, 1.2 and 14, 13, 12, 12.
bool takes_resident(const lbm_batch* b, int64_t n)
{
    if (kBatchVariants[b->var].resident) return true;
    return b->res_tuned && b->res_fixed + n * b->res_step < n * b->tune_ms[b->var];
}

// n steps of every active domain from pool[parity]; the state ends in pool[parity ^ (n & 1)].
cudaError_t launch_steps(lbm_batch* b, int parity, int64_t n)
{
    if (takes_resident(b, n)) return launch_resident(b, parity, n);
    cudaError_t e = cudaSuccess;
    for (int64_t i = 0; i < n && e == cudaSuccess; ++i)
        e = kBatchVariants[b->var].launch(b, (parity + static_cast<int>(i & 1)) & 1);
    return e;
}

// Makes shape v current: persistent grid = SMs x resident CTAs, work list rebuilt,
// captured graphs dropped (they hold the previous kernel).
int select_variant(lbm_batch* b, int v)
{
    b->var = v;
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, b->device);
    for (int k = 0; k < 2; ++k)
        if (b->graph[k]) {
            cudaGraphExecDestroy(b->graph[k]);
            b->graph[k] = nullptr;
        }
    if (kBatchVariants[v].resident) return rebuild_resident(b);
    b->grid = std::max(1, nsm * std::max(1, kBatchVariants[v].occupancy(b->fp32)));
    if (int rc = rebuild_items(b)) return rc;
    // no more persistent blocks than items: the work list only shrinks until the
    // next selection, and the blocks loop over whatever it holds
    b->grid = std::max(1, std::min(b->grid, b->nitems));
    return LBM_OK;
}

// Times every shape on the batch's current state (a few steps each, from a saved
// copy that is put back afterwards, so the state does not advance) and keeps the
// fastest that steps launch by launch and, beside it, the resident shape with what a call
// and a step of it take.  Without room for the copy the default shape stays.
int autotune(lbm_batch* b, bool again = false)
{
    if (b->tuned && !(again && !b->pinned)) return LBM_OK;
    b->tuned = true;
    // the active domains' states are saved and put back (retired ones are not stepped)
    const size_t es = b->fp32 ? 4 : 8;
    size_t bytes = 0;
    long long cells = 0;
    for (const auto& m : b->doms)
        if (m.active) {
            bytes += es * kQ9 * static_cast<size_t>(m.nx) * m.ny;
            cells += static_cast<long long>(m.nx) * m.ny;
        }
    b->tuned_cells = cells;
    if (bytes == 0) return LBM_OK;
    char* save = static_cast<char*>(b->dalloc(bytes));
    if (!save) return LBM_OK;
    auto copy_states = [&](bool to_save) {
        size_t o = 0;
        for (const auto& m : b->doms) {
            if (!m.active) continue;
            const size_t n = es * kQ9 * static_cast<size_t>(m.nx) * m.ny;
            char* pool = static_cast<char*>(b->pool[b->cur]) + es * m.off;
            cudaError_t e = to_save ? cudaMemcpyAsync(save + o, pool, n, cudaMemcpyDeviceToDevice, b->stream)
                                    : cudaMemcpyAsync(pool, save + o, n, cudaMemcpyDeviceToDevice, b->stream);
            if (e != cudaSuccess) return e;
            o += n;
        }
        return cudaSuccess;
    };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = LBM_OK;
    auto ck = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == LBM_OK) rc = set_last_error(LBM_ECUDA, cudaGetErrorString(e));
    };
    ck(cudaEventCreate(&e0));
    ck(cudaEventCreate(&e1));
    ck(copy_states(true));
    constexpr int kWarm = 2, kTimed = 8;
    b->tune_ms.assign(kNumBatchVariants, -1.0);
    bool nx4 = true;
    for (const auto& m : b->doms) nx4 = nx4 && m.nx % 4 == 0;
    // calls of n steps, from an even number of steps after the saved state; ms of one
    auto timed = [&](int calls, int n) {
        float ms = 0.f;
        ck(cudaEventRecord(e0, b->stream));
        for (int i = 0; i < calls; ++i) ck(launch_steps(b, (b->cur + i * n) & 1, n));
        ck(cudaEventRecord(e1, b->stream));
        ck(cudaEventSynchronize(e1));
        ck(cudaEventElapsedTime(&ms, e0, e1));
        return static_cast<double>(ms) / calls;
    };
    int best = 0;
    bool resident = false;
    b->res_tuned = false;
    for (int v = 0; v < kNumBatchVariants && rc == LBM_OK; ++v) {
        if (kBatchVariants[v].staged && !(b->fp32 && nx4)) continue;
        if (kBatchVariants[v].resident && !resident_applies(b)) continue;
        if (int r = select_variant(b, v)) {
            rc = r;
            break;
        }
        ck(launch_steps(b, b->cur, kWarm));
        if (kBatchVariants[v].resident) {
            const double many = timed(1, kResTimed), one = timed(kTimed, 1);
            b->tune_ms[v] = many / kResTimed;
            b->res_step = std::max(0.0, many - one) / (kResTimed - 1);
            b->res_fixed = std::max(0.0, one - b->res_step);
            resident = true;
        } else {
            b->tune_ms[v] = timed(1, kTimed) / kTimed;
            if (b->tune_ms[v] < b->tune_ms[best]) best = v;
        }
        ck(copy_states(false));
    }
    ck(cudaStreamSynchronize(b->stream));
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    b->dfree(save);
    if (rc != LBM_OK) return rc;
    b->res_tuned = resident;
    return select_variant(b, best);
}

// Observables into d_res (the state pointed to by d_cur_of): of every domain, or
// (only_active, inside the steady-check graph) of the domains still stepping.
cudaError_t launch_obs(lbm_batch* b, int only_active = 0)
{
    const long long stride = static_cast<const char*>(b->pool[1]) - static_cast<const char*>(b->pool[0]);
    const long long es = b->fp32 ? 4 : 8;
    if (b->fp32) {
        k_batch_obs<float><<<b->n * kObsSlices, 256, 0, b->stream>>>(
            b->d_doms, static_cast<const float*>(b->pool[0]), b->d_cur_of, stride / es, b->d_partials, b->n,
            only_active);
        k_batch_obs_final<float><<<(b->n + 63) / 64, 64, 0, b->stream>>>(
            b->d_doms, static_cast<const float*>(b->pool[0]), b->d_cur_of, stride / es, b->d_partials, b->d_res,
            b->n, only_active);
    } else {
        k_batch_obs<double><<<b->n * kObsSlices, 256, 0, b->stream>>>(
            b->d_doms, static_cast<const double*>(b->pool[0]), b->d_cur_of, stride / es, b->d_partials, b->n,
            only_active);
        k_batch_obs_final<double><<<(b->n + 63) / 64, 64, 0, b->stream>>>(
            b->d_doms, static_cast<const double*>(b->pool[0]), b->d_cur_of, stride / es, b->d_partials,
            b->d_res, b->n, only_active);
    }
    return cudaGetLastError();
}

// Populations of domain d between its storage and a double host array [9][ny][nx].  They
// pass through the other pool, which nothing reads between steps where its domains' states
// lie in this one: all nine directions at once where neighbouring domains leave that much
// room, else as many as fit (four of an FP32 domain into its own part).  No memory is
// needed, and a copy costs some 70 us beside its bytes.
template <bool GET>
cudaError_t copy_populations(lbm_batch* b, int d, double* f_host)
{
    const BatchDom& m = b->doms[d];
    const long long N = static_cast<long long>(m.nx) * m.ny;
    const long long es = b->fp32 ? 4 : 8;
    const long long need = kQ9 * N * static_cast<long long>(sizeof(double));
    // the longest run of domains whose part of the other pool is free
    long long at = es * m.off, room = es * kQ9 * N;
    for (int k = 0, first = 0; k < b->n && room < need; ++k) {
        if (b->cur_of[k] != b->cur_of[d]) {
            first = k + 1;
            continue;
        }
        const BatchDom& z = b->doms[k];
        const long long start = es * b->doms[first].off;
        const long long bytes = es * (z.off + static_cast<long long>(kQ9) * z.nx * z.ny) - start;
        if (bytes > room) {
            room = bytes;
            at = start;
        }
    }
    const int most = static_cast<int>(std::min<long long>(kQ9, room / (N * static_cast<long long>(sizeof(double)))));
    void* state = static_cast<char*>(b->pool[b->cur_of[d]]) + es * m.off;
    double* via = reinterpret_cast<double*>(static_cast<char*>(b->pool[b->cur_of[d] ^ 1]) + at);
    for (int q0 = 0; q0 < kQ9; q0 += most) {
        const int nq = std::min(most, kQ9 - q0);
        const size_t bytes = sizeof(double) * nq * N;
        cudaError_t e = cudaSuccess;
        if (!GET) e = cudaMemcpyAsync(via, f_host + q0 * N, bytes, cudaMemcpyHostToDevice, b->stream);
        if (e != cudaSuccess) return e;
        const unsigned grid = static_cast<unsigned>((nq * N + 255) / 256);
        if (b->fp32)
            k_batch_io<GET, float><<<grid, 256, 0, b->stream>>>(m.nx, m.ny, m.rho_bar, q0, nq,
                                                                static_cast<float*>(state), via);
        else
            k_batch_io<GET, double><<<grid, 256, 0, b->stream>>>(m.nx, m.ny, m.rho_bar, q0, nq,
                                                                 static_cast<double*>(state), via);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (GET) e = cudaMemcpyAsync(f_host + q0 * N, via, bytes, cudaMemcpyDeviceToHost, b->stream);
        if (e != cudaSuccess) return e;
    }
    return cudaStreamSynchronize(b->stream);
}

double pressure_exp(double rho, double G)
{
    const double ps = -std::expm1(-rho);
    return rho / 3.0 + 0.5 * G / 3.0 * ps * ps;
}

}  // namespace

extern "C" {

int lbm_batch_create(const lbm_params* ps, const double* init, int n, lbm_batch** out)
{
    if (!ps || !init || !out || n < 1) return set_last_error(LBM_EINVAL, "lbm_batch_create: bad argument");
    const int fp32 = ps[0].precision == LBM_FP32_SHIFTED;
    for (int d = 0; d < n; ++d) {
        const lbm_params& p = ps[d];
        const int order = p.stencil == LBM_STENCIL_LATTICE ? 4 : p.stencil;
        if (p.lattice != LBM_D2Q9 || p.psi != LBM_PSI_EXP || p.collision != LBM_BGK || p.wall_rows != 0)
            return set_last_error(LBM_EUNSUPPORTED, "lbm_batch_create: batches are D2Q9, exp psi, BGK, no wall");
        if ((p.precision == LBM_FP32_SHIFTED) != (fp32 != 0))
            return set_last_error(LBM_EINVAL, "lbm_batch_create: one precision per batch");
        if (p.nx < 8 || p.ny < 8 || p.nz != 1 || !(p.tau > 0.5) ||
            !(order == 4 || order == 6 || order == 8 || order == 10))
            return set_last_error(LBM_EINVAL, "lbm_batch_create: bad domain parameters");
        if (!(init[4 * d + 3] > 0.0) || !(init[4 * d] > 0.0) || !(init[4 * d + 1] > 0.0))
            return set_last_error(LBM_EINVAL, "lbm_batch_create: bad initial droplet");
    }
    lbm_batch* b = new (std::nothrow) lbm_batch();
    if (!b) return set_last_error(LBM_ENOMEM, "host allocation failed");
    b->n = n;
    b->fp32 = fp32;
    b->p0 = ps[0];
    b->init.assign(init, init + 4 * n);
    b->cur_of.assign(n, 0);
    b->steps.assign(n, 0);
    cudaGetDevice(&b->device);
    if (ps[0].stream) {
        b->stream = static_cast<cudaStream_t>(ps[0].stream);
    } else {
        cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
        b->own_stream = true;
    }
    long long off = 0, poff = 0;
    b->doms.resize(n);
    for (int d = 0; d < n; ++d) {
        const lbm_params& p = ps[d];
        BatchDom& m = b->doms[d];
        m.nx = p.nx;
        m.ny = p.ny;
        m.order = p.stencil == LBM_STENCIL_LATTICE ? 4 : p.stencil;
        m.ntx = (p.nx + kMinTX - 1) / kMinTX;  // item buffer sized for the finest shape
        m.nch = (p.ny + kMinZC - 1) / kMinZC;
        m.active = 1;
        m.off = off;
        m.G = p.G;
        m.omega = 1.0 / p.tau;
        m.pref = 1.0 - 1.0 / (2.0 * p.tau);
        // FP32 deviations from the mean initial density (rectangle-rule mean of the
        // tanh droplet, computed on the host in double)
        double sum = 0.0;
        if (fp32) {
            for (int y = 0; y < p.ny; ++y)
                for (int x = 0; x < p.nx; ++x) {
                    auto mi = [](int i, int nn) {
                        double v = (double)i - (double)(nn / 2);
                        if (v > 0.5 * nn) v -= nn;
                        if (v < -0.5 * nn) v += nn;
                        return v;
                    };
                    const double dx = mi(x, p.nx), dy = mi(y, p.ny);
                    const double r = std::sqrt(dx * dx + dy * dy);
                    sum += 0.5 * (init[4 * d] + init[4 * d + 1]) -
                           0.5 * (init[4 * d] - init[4 * d + 1]) * std::tanh(2.0 * (r - init[4 * d + 2]) / init[4 * d + 3]);
                }
            m.rho_bar = sum / ((double)p.nx * p.ny);
        }
        m.G_f = static_cast<float>(m.G);
        m.omega_f = static_cast<float>(m.omega);
        m.pref_f = static_cast<float>(m.pref);
        m.rho_bar_f = static_cast<float>(m.rho_bar);
        DevParams dp{};
        dp.omega = m.omega;
        dp.pref = m.pref;
        dp.G = m.G;
        switch (m.order) {
        case 4: m.c64 = fill_c64<kLatD2Q9, 4, 0>(dp); break;
        case 6: m.c64 = fill_c64<kLatD2Q9, 6, 0>(dp); break;
        case 8: m.c64 = fill_c64<kLatD2Q9, 8, 0>(dp); break;
        default: m.c64 = fill_c64<kLatD2Q9, 10, 0>(dp); break;
        }
        off += (long long)kQ9 * p.nx * p.ny;
        off = (off + 63) / 64 * 64;  // 256-byte aligned domains
        m.poff = poff;
        poff += ((long long)p.nx * p.ny + 63) / 64 * 64;
    }
    b->pool_elems = off;
    const size_t es = fp32 ? 4 : 8;
    long long items = 0;
    for (auto& m : b->doms) items += (long long)m.ntx * m.nch;
    b->pool[0] = b->dalloc(es * off);
    b->pool[1] = b->dalloc(es * off);
    b->psi_pool = b->dalloc(es * poff);
    b->d_doms = static_cast<BatchDom*>(b->dalloc(sizeof(BatchDom) * n));
    b->d_items = static_cast<int4*>(b->dalloc(sizeof(int4) * items));
    b->d_list = static_cast<int*>(b->dalloc(sizeof(int) * n));
    b->d_nitems = static_cast<int*>(b->dalloc(256));
    b->d_cur_of = static_cast<int*>(b->dalloc(sizeof(int) * n));
    b->d_init = static_cast<double*>(b->dalloc(sizeof(double) * 4 * n));
    b->d_partials = static_cast<double*>(b->dalloc(sizeof(double) * n * kObsSlices * kObsWidth));
    b->d_res = static_cast<double*>(b->dalloc(sizeof(double) * n * 8));
    b->d_prev = static_cast<double*>(b->dalloc(sizeof(double) * n));
    b->d_newly = static_cast<int*>(b->dalloc(256));
    b->d_err = static_cast<unsigned*>(b->dalloc(256));
    if (!b->pool[0] || !b->pool[1] || !b->psi_pool || !b->d_doms || !b->d_items || !b->d_list || !b->d_nitems || !b->d_cur_of || !b->d_init ||
        !b->d_partials || !b->d_res || !b->d_prev || !b->d_newly || !b->d_err) {
        lbm_batch_destroy(b);
        return set_last_error(LBM_ENOMEM, "lbm_batch_create: device allocation failed");
    }
    if (cudaMallocHost(&b->h_newly, sizeof(int)) != cudaSuccess ||
        cudaMallocHost(&b->h_err, sizeof(unsigned)) != cudaSuccess) {
        lbm_batch_destroy(b);
        return set_last_error(LBM_ENOMEM, "pinned host allocation failed");
    }
    int rc = LBM_OK;
    auto ck = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == LBM_OK) rc = set_last_error(LBM_ECUDA, cudaGetErrorString(e));
    };
    ck(cudaMemcpyAsync(b->d_doms, b->doms.data(), sizeof(BatchDom) * n, cudaMemcpyHostToDevice, b->stream));
    ck(cudaMemcpyAsync(b->d_init, init, sizeof(double) * 4 * n, cudaMemcpyHostToDevice, b->stream));
    ck(cudaMemsetAsync(b->d_cur_of, 0, sizeof(int) * n, b->stream));
    ck(cudaMemsetAsync(b->d_err, 0, sizeof(unsigned), b->stream));
    std::vector<double> prev(n, -1.0);
    ck(cudaMemcpyAsync(b->d_prev, prev.data(), sizeof(double) * n, cudaMemcpyHostToDevice, b->stream));
    ck(cudaMemsetAsync(b->pool[1], 0, es * off, b->stream));
    int maxp = 1;
    for (auto& m : b->doms) maxp = std::max(maxp, m.nx * m.ny);
    const dim3 g((maxp + 255) / 256 < 1024 ? (maxp + 255) / 256 : 1024, n);
    if (fp32)
        k_batch_init<float><<<g, 256, 0, b->stream>>>(b->d_doms, b->d_init, n, static_cast<float*>(b->pool[0]));
    else
        k_batch_init<double><<<g, 256, 0, b->stream>>>(b->d_doms, b->d_init, n, static_cast<double*>(b->pool[0]));
    ck(cudaGetLastError());
    if (rc == LBM_OK) rc = select_variant(b, 0);
    if (rc != LBM_OK) {
        lbm_batch_destroy(b);
        return rc;
    }
    *out = b;
    return LBM_OK;
}

int lbm_batch_destroy(lbm_batch* b)
{
    if (!b) return LBM_OK;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    for (int k = 0; k < 2; ++k)
        if (b->graph[k]) cudaGraphExecDestroy(b->graph[k]);
    b->dfree(b->pool[0]);
    b->dfree(b->pool[1]);
    b->dfree(b->psi_pool);
    b->dfree(b->d_doms);
    b->dfree(b->d_items);
    b->dfree(b->d_list);
    for (int k = 0; k < kResMaxCluster; ++k) {
        if (b->aux[k]) cudaStreamDestroy(b->aux[k]);
        if (b->ev_join[k]) cudaEventDestroy(b->ev_join[k]);
    }
    if (b->ev_fork) cudaEventDestroy(b->ev_fork);
    b->dfree(b->d_nitems);
    b->dfree(b->d_cur_of);
    b->dfree(b->d_init);
    b->dfree(b->d_partials);
    b->dfree(b->d_res);
    b->dfree(b->d_prev);
    b->dfree(b->d_newly);
    b->dfree(b->d_err);
    if (b->h_newly) cudaFreeHost(b->h_newly);
    if (b->h_err) cudaFreeHost(b->h_err);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return LBM_OK;
}

// Advances every active domain by n steps (no steady check).
int lbm_batch_step(lbm_batch* b, int64_t n)
{
    lbm::TraceRange trace("lbm_batch_step");
    if (!b || n < 0) return set_last_error(LBM_EINVAL, "lbm_batch_step: bad argument");
    LBM_BCK(cudaSetDevice(b->device));
    if (n > 0)
        if (int rc = autotune(b)) return rc;
    LBM_BCK(launch_steps(b, b->cur, n));
    b->cur ^= static_cast<int>(n & 1);
    b->global_step += n;
    for (int d = 0; d < b->n; ++d)
        if (b->doms[d].active) {
            b->steps[d] += n;
            b->cur_of[d] = b->cur;
        }
    LBM_BCK(cudaMemcpyAsync(b->d_cur_of, b->cur_of.data(), sizeof(int) * b->n, cudaMemcpyHostToDevice, b->stream));
    return LBM_OK;
}

int lbm_batch_run_to_steady(lbm_batch* b, double tol, int64_t max_steps, int64_t check_every,
                            int64_t* steps_per_domain, lbm_obs* obs_per_domain)
{
    lbm::TraceRange trace("lbm_batch_run_to_steady");
    if (!b || !(tol > 0.0) || max_steps < 0 || check_every < 2 || check_every % 2)
        return set_last_error(LBM_EINVAL, "lbm_batch_run_to_steady: bad argument (check_every must be even)");
    LBM_BCK(cudaSetDevice(b->device));
    if (int rc = autotune(b)) return rc;
    const int K = static_cast<int>(check_every);
    const double floor_rel = b->fp32 ? 1e-6 : 0.0;
    // one graph per starting parity is not needed: K is even, so every block of K
    // steps starts from the same parity
    auto capture = [&]() -> int {
    if (!b->graph[0] || b->graph_k != K || b->graph_cur != b->cur || b->graph_tol != tol) {
        if (b->graph[0]) cudaGraphExecDestroy(b->graph[0]);
        b->graph[0] = nullptr;
        cudaGraph_t g = nullptr;
        LBM_BCK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = cudaSuccess;
        e = launch_steps(b, b->cur, K);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->d_newly, 0, sizeof(int), b->stream);
        if (e == cudaSuccess) e = launch_obs(b, 1);
        if (e == cudaSuccess) {
            k_batch_check<<<(b->n + 127) / 128, 128, 0, b->stream>>>(b->d_doms, b->d_res, b->d_prev, b->n, tol,
                                                                    floor_rel, K, b->d_newly);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(b->h_newly, b->d_newly, sizeof(int), cudaMemcpyDeviceToHost, b->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(b->h_err, b->d_err, sizeof(unsigned), cudaMemcpyDeviceToHost, b->stream);
        cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return set_last_error(LBM_ECUDA, cudaGetErrorString(e != cudaSuccess ? e : e2));
        }
        e = cudaGraphInstantiate(&b->graph[0], g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return set_last_error(LBM_ECUDA, cudaGetErrorString(e));
        b->graph_k = K;
        b->graph_tol = tol;
        b->graph_cur = b->cur;
    }
    return LBM_OK;
    };
    if (int rc = capture()) return rc;
    // the observables inside the graph read cur_of: active domains end each block
    // on the same parity as they started (K even)
    for (int d = 0; d < b->n; ++d)
        if (b->doms[d].active) b->cur_of[d] = b->cur;
    LBM_BCK(cudaMemcpyAsync(b->d_cur_of, b->cur_of.data(), sizeof(int) * b->n, cudaMemcpyHostToDevice, b->stream));
    // the first check compares against max|u| of the state the run starts from
    LBM_BCK(launch_obs(b));
    k_batch_prev_init<<<(b->n + 127) / 128, 128, 0, b->stream>>>(b->d_doms, b->d_res, b->d_prev, b->n);
    LBM_BCK(cudaGetLastError());
    int64_t taken = 0;
    int nactive = 0;
    for (auto& m : b->doms) nactive += m.active;
    while (nactive > 0 && taken + K <= max_steps) {
        LBM_BCK(cudaGraphLaunch(b->graph[0], b->stream));
        LBM_BCK(cudaStreamSynchronize(b->stream));
        if (*b->h_err & kErrTimeout) return set_last_error(LBM_ETIMEOUT, "a bounded device wait ran out");
        taken += K;
        b->global_step += K;
        for (int d = 0; d < b->n; ++d)
            if (b->doms[d].active) b->steps[d] += K;
        if (*b->h_newly > 0) {
            std::vector<BatchDom> dv(b->n);
            LBM_BCK(cudaMemcpy(dv.data(), b->d_doms, sizeof(BatchDom) * b->n, cudaMemcpyDeviceToHost));
            for (int d = 0; d < b->n; ++d) b->doms[d].active = dv[d].active;
            nactive = 0;
            for (auto& m : b->doms) nactive += m.active;
            if (int rc = rebuild_items(b)) return rc;
            // a captured graph holds the resident classes; retired domains are skipped by
            // their flag, and their clusters go once that is worth a new graph
            if (nactive > 0 && takes_resident(b, K)) {
                bool rebuilt = false;
                if (int rc = rebuild_resident(b, true, &rebuilt)) return rc;
                if (rebuilt) {
                    cudaGraphExecDestroy(b->graph[0]);
                    b->graph[0] = nullptr;
                    if (int rc = capture()) return rc;
                }
            }
            // when the active set has shrunk eightfold, finer items may fill the GPU
            // better: time the shapes again on what is left
            long long cells = 0;
            for (const auto& m : b->doms)
                if (m.active) cells += static_cast<long long>(m.nx) * m.ny;
            if (nactive > 0 && cells * 8 < b->tuned_cells) {
                if (int rc = autotune(b, true)) return rc;
                if (int rc = capture()) return rc;
            }
        }
    }
    LBM_BCK(launch_obs(b));
    std::vector<double> res(8 * (size_t)b->n);
    LBM_BCK(cudaMemcpyAsync(res.data(), b->d_res, sizeof(double) * 8 * b->n, cudaMemcpyDeviceToHost, b->stream));
    LBM_BCK(cudaStreamSynchronize(b->stream));
    for (int d = 0; d < b->n; ++d) {
        if (steps_per_domain) steps_per_domain[d] = b->steps[d];
        if (obs_per_domain) {
            lbm_obs o{};
            const double* r = &res[8 * (size_t)d];
            const double N = (double)b->doms[d].nx * b->doms[d].ny;
            o.mass = r[0];
            o.mom[0] = r[1];
            o.mom[1] = r[2];
            o.mean_u = r[4] / N;
            o.max_u = r[5];
            o.rho_l = r[6];
            o.rho_g = r[7];
            o.dp = pressure_exp(o.rho_l, b->doms[d].G) - pressure_exp(o.rho_g, b->doms[d].G);
            o.step = b->steps[d];
            obs_per_domain[d] = o;
        }
    }
    return nactive == 0 ? LBM_OK : set_last_error(LBM_ENOTCONVERGED, "some domains still changing at max_steps");
}

int lbm_batch_schedule_report(lbm_batch* b, char* buf, int len)
{
    if (!b || !buf || len < 1) return set_last_error(LBM_EINVAL, "lbm_batch_schedule_report: bad argument");
    LBM_BCK(cudaSetDevice(b->device));
    if (int rc = autotune(b)) return rc;
    int chosen = b->var;
    for (int v = 0; v < kNumBatchVariants; ++v)
        if (kBatchVariants[v].resident && takes_resident(b, kResTimed)) chosen = v;
    std::string s = std::string("chosen=") + kBatchVariants[chosen].name;
    for (int v = 0; v < kNumBatchVariants && v < (int)b->tune_ms.size(); ++v) {
        if (b->tune_ms[v] < 0) continue;
        char t[96];
        std::snprintf(t, sizeof(t), ";%s=%.5f", kBatchVariants[v].name, b->tune_ms[v]);
        s += t;
    }
    std::snprintf(buf, len, "%s", s.c_str());
    return LBM_OK;
}

int lbm_batch_set_schedule(lbm_batch* b, const char* name)
{
    if (!b || !name) return set_last_error(LBM_EINVAL, "lbm_batch_set_schedule: bad argument");
    LBM_BCK(cudaSetDevice(b->device));
    bool nx4 = true;
    for (const auto& m : b->doms) nx4 = nx4 && m.nx % 4 == 0;
    for (int v = 0; v < kNumBatchVariants; ++v)
        if (std::strcmp(kBatchVariants[v].name, name) == 0) {
            if (kBatchVariants[v].staged && !(b->fp32 && nx4))
                return set_last_error(LBM_EINVAL, "lbm_batch_set_schedule: staged shapes need FP32 and nx % 4 == 0");
            if (kBatchVariants[v].resident && !resident_applies(b))
                return set_last_error(LBM_EINVAL, "lbm_batch_set_schedule: the resident shape needs FP32 and domains that fit a cluster");
            b->tuned = true;
            b->pinned = true;
            b->res_tuned = false;
            return select_variant(b, v);
        }
    return set_last_error(LBM_EINVAL, "lbm_batch_set_schedule: unknown tile shape");
}

// Observables of every domain in its current state.
int lbm_batch_observables(lbm_batch* b, lbm_obs* obs_per_domain)
{
    if (!b || !obs_per_domain) return set_last_error(LBM_EINVAL, "lbm_batch_observables: bad argument");
    LBM_BCK(cudaSetDevice(b->device));
    LBM_BCK(cudaMemcpyAsync(b->d_cur_of, b->cur_of.data(), sizeof(int) * b->n, cudaMemcpyHostToDevice, b->stream));
    LBM_BCK(launch_obs(b));
    std::vector<double> res(8 * (size_t)b->n);
    LBM_BCK(cudaMemcpyAsync(res.data(), b->d_res, sizeof(double) * 8 * b->n, cudaMemcpyDeviceToHost, b->stream));
    LBM_BCK(cudaStreamSynchronize(b->stream));
    for (int d = 0; d < b->n; ++d) {
        lbm_obs o{};
        const double* r = &res[8 * (size_t)d];
        const double N = (double)b->doms[d].nx * b->doms[d].ny;
        o.mass = r[0];
        o.mom[0] = r[1];
        o.mom[1] = r[2];
        o.mean_u = r[4] / N;
        o.max_u = r[5];
        o.rho_l = r[6];
        o.rho_g = r[7];
        o.dp = pressure_exp(o.rho_l, b->doms[d].G) - pressure_exp(o.rho_g, b->doms[d].G);
        o.step = b->steps[d];
        obs_per_domain[d] = o;
    }
    return LBM_OK;
}

// Sets domain d's pre-collision populations from a double host array [9][ny][nx]
// (in the pool buffer that holds its state).
int lbm_batch_set_populations(lbm_batch* b, int d, const double* f_host)
{
    if (!b || !f_host || d < 0 || d >= b->n) return set_last_error(LBM_EINVAL, "lbm_batch_set_populations: bad argument");
    LBM_BCK(cudaSetDevice(b->device));
    LBM_BCK(copy_populations<false>(b, d, const_cast<double*>(f_host)));
    return LBM_OK;
}

// Pre-collision populations of domain d in double, [9][ny][nx].
int lbm_batch_get_populations(lbm_batch* b, int d, double* f_host)
{
    if (!b || !f_host || d < 0 || d >= b->n) return set_last_error(LBM_EINVAL, "lbm_batch_get_populations: bad argument");
    LBM_BCK(cudaSetDevice(b->device));
    LBM_BCK(copy_populations<true>(b, d, f_host));
    return LBM_OK;
}

}  // extern "C"
