// internal.h -- interface between the C-ABI layer (api.cu) and the kernel
// instantiations (one translation unit per lattice).  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace lbm {

// Error bits raised by kernels in the device error word.
enum : unsigned {
    kErrNonFinite = 1u,   // NaN/Inf density or velocity
    kErrNegativeSqrt = 2u,  // Peng-Robinson psi argument below zero
    kErrTimeout = 4u,     // a bounded wait (mbarrier) gave up
};

// psi buffer: periodic ghost layers, kGhostX cells on each side in x (so that
// every TMA box starts on a 16-byte boundary) and `g` = stencil radius in y, z.
constexpr int kGhostX = 4;

constexpr double kPrA = 2.0 / 49.0;  // Peng-Robinson a, b (R = 1), Sec. 3
constexpr double kPrB = 2.0 / 21.0;

// Division of 0 <= i < 2^31 by a fixed d > 0: q = (i * m) >> s with s = 31 + ceil(log2 d)
// and m = ceil(2^s / d) < 2^32, exact over that range.
struct FastDiv {
    unsigned d, m;
    int s;
    __host__ __device__ unsigned div(unsigned i) const
    {
        return static_cast<unsigned>((static_cast<unsigned long long>(i) * m) >> s);
    }
};
inline FastDiv make_fast_div(unsigned d)
{
    int l = 0;
    while ((1u << l) < d) ++l;
    const unsigned long long p = 1ull << (31 + l);
    return {d, static_cast<unsigned>((p + d - 1) / d), 31 + l};
}

// Parameter products of the FP64 collision (collide64), formed once per launch on
// the host.  w: weight of the lattice's largest shell, w1: first force weight
// times c_s^2 (the force sums come divided by it).
struct Coll64 {
    double gh, k0;      // -G w1 / 2, w omega / (2 c_s^2)
    double k1, k1l;     // -G w1 w pref / c_s^2, in two terms
    double omega, om1;  // omega, 1 - omega
    double g, gl;       // exact difference: -G w1, in two terms
    double kb, hT;      // exact difference: w / c_s^2, w / (2 c_s^2)
    double dmn[19];     // MRT: (omega - s_k) / |M_k|^2
};

// Runtime constants of one domain, passed by value to every kernel.
struct DevParams {
    int nx, ny, nz;
    long long N;         // cells
    int g;               // ghost width of psi in y (and z)
    int psx;             // psi row pitch in elements
    int psy;             // psi rows per z plane (ny + 2g)
    double G;
    double omega;        // 1 / tau
    double pref;         // 1 - 1/(2 tau)
    double rho_bar;      // reference density of FP32 deviation storage (0 in FP64)
    int psi_kind;        // 0 exp, 1 Peng-Robinson
    double pr_T;         // Peng-Robinson temperature T_over_Tc * T_c
    double pr_alpha;     // alpha(T)
    double rate[4];      // MRT rates by class: 1/tau, s_e, s_eps, s_q
    unsigned* err;       // device error word
    int wall_rows;       // rows y < wall_rows are solid (bounce-back); 0 = no wall
    double psi_w;        // psi of the wall's virtual density
    // Derived by finish_params(): the MRT correction factors omega - s per rate
    // class (class 0 relaxes at omega, so its factor is 0), and FP32 copies of
    // the scalars the FP32 kernels use, so they convert nothing per cell.
    double dmrt[4];
    float omega_f, pref_f, rho_bar_f, G_f;
    float dmrt_f[4];
};

// What the FP64 kernels take beside it (apart, because a kernel's parameters cost launch
// time: 270 bytes more slowed a 2.3 us FP32 step by 8%).
struct DevParams64 : DevParams {
    double pr_K;   // Peng-Robinson psi: 2 / (G c_s^2) and a alpha
    double pr_aa;
    Coll64 c64;        // collision products, set by the launchers (fill_c64)
    FastDiv dnx, dny;  // for x, y, z of a linear cell index
};
template <class Real> struct ParamsOf {
    using T = DevParams;
};
template <> struct ParamsOf<double> {
    using T = DevParams64;
};

// Fills the derived fields of p from the others; call after any change to
// omega, pref, rho_bar, G or rate.
__host__ __device__ inline void finish_params(DevParams& p)
{
    for (int c = 0; c < 4; ++c) {
        p.dmrt[c] = (c == 0) ? 0.0 : p.omega - p.rate[c];
        p.dmrt_f[c] = static_cast<float>(p.dmrt[c]);
    }
    p.omega_f = static_cast<float>(p.omega);
    p.pref_f = static_cast<float>(p.pref);
    p.rho_bar_f = static_cast<float>(p.rho_bar);
    p.G_f = static_cast<float>(p.G);
}

// Everything a launcher may need; unused fields are ignored.
struct LaunchArgs {
    DevParams64 p;
    const void* fin;       // populations read (current state)
    void* fout;            // populations written
    void* psi;             // ghosted psi buffer (base of the allocation)
    const CUtensorMap* tmap;  // TMA descriptor of the psi buffer
    double* partials;      // reduction scratch
    int nblocks_max;       // capacity of partials (blocks)
    double* res;           // reduction result (see api.cu for the slots)
    double* rho;           // density of every cell (FP64 two-pass schedule; part of fout)
    double* dbuf0;         // double work buffers (N or Q*N)
    double* dbuf1;
    int mode;              // init profile: 0 droplet, 1 flat
    int axis;
    double a0, a1, a2, a3; // init parameters (rho_l, rho_g, R, width)
    float* carry_in;       // carried density of the current state (schedules with carry_rows > 0)
    float* carry_out;      // carried density of the state written
};

// One compiled variant of the one-pass step kernel (tile shape, chunk length,
// minimum resident blocks); the autotuner picks among them.
struct StepVariant {
    const char* name;
    cudaError_t (*fn)(const LaunchArgs&, cudaStream_t);
    int nx_multiple;     // nx must be a multiple of this (two cells per thread, 16-byte rows)
    int nx_exact;        // nonzero: the variant is compiled for this nx only (whole rows in shared memory)
    int nx_max;          // nonzero: the variant takes rows of at most this many cells (shared-memory size)
    int carry_rows;      // nonzero: the step reads and writes a carried density for groups of this many rows
    long long min_cells; // the autotuner times the variant from this size on (< 0: never); it can always be pinned
};
constexpr int kMaxVariants = 48;

// One set of launchers per (lattice, stencil order, collision, precision).
struct KernelSet {
    int tile_x, tile_y, tile_z;  // fused-kernel tile (TMA box minus halo)
    cudaError_t (*psi)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*fused)(const LaunchArgs&, cudaStream_t);
    int n_onepass;                          // 0: no one-pass schedule
    StepVariant onepass[kMaxVariants];
    cudaError_t (*obs)(const LaunchArgs&, cudaStream_t, int* nblocks);
    cudaError_t (*probe)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*fields)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*init_profile)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*init_from_rho)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*get_f)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*set_f)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*rho_of_f)(const LaunchArgs&, cudaStream_t);
    cudaError_t (*carry_init)(const LaunchArgs&, int rows, cudaStream_t);  // null: no carried-density schedule
};

// Records msg as the calling thread's lbm_last_error() text and returns code.
int set_last_error(int code, const char* msg);

// Shared reduction helpers (reduce.cu).
cudaError_t launch_sum_partials(const double* partials, int nblocks, int width, double* res,
                                cudaStream_t s);
cudaError_t launch_mean(const double* x, long long n, double* partials, int nblocks_max,
                        double* res, cudaStream_t s);

// Failure-detection check (diag.cu): one block waits on an mbarrier that nothing
// completes, through the step kernels' bounded wait, and sets kErrTimeout in *err.
cudaError_t launch_wait_probe(unsigned* err, cudaStream_t s);

// Keeps the stream busy for about `ns` (at most 10 ms), so that the host can queue work
// ahead of it (diag.cu).
cudaError_t launch_delay(unsigned ns, cudaStream_t s);

// Warm-start network (mlp.cu): the network's density at T signed distances evenly
// spaced over [-dmax, dmax] for (G, tau, order, r_in * R_dev[c]), c < ncand, into
// tables_dev[c][T], on stream s.  The network's distance input spans |d| <= kMlpDmax.
constexpr double kMlpDmax = 24.0;
}  // namespace lbm
struct lbm_mlp;
namespace lbm {
int mlp_device(const lbm_mlp* n);  // that its parameters are on
cudaError_t mlp_profile_tables(const lbm_mlp* n, double G, double tau, double order, const double* R_dev, double r_in,
                               int ncand, int T, double dmax, float* tables_dev, cudaStream_t s);

// Mass-matching search of the learned start (reduce.cu), kept on the device: a
// radius bracket halved two times per round from three candidates, the midpoint
// and the midpoints of both halves, so the halvings follow the plain bisection.
struct RadiusSearch {
    double cand[3];   // radii the next tables are made for (first round: the bracket's ends)
    double lo, hi, mlo;
    double m0;        // mean density to match
    double Re, mm;    // last radius taken and its mean
    int last;         // its candidate index
    int ok;           // bracket valid and every mean finite
    int round;        // 0: the bracket itself
    unsigned done;    // blocks finished (last one updates)
};
// *st := start of a search over [lo, hi] for the mean res[0] (device).
cudaError_t launch_search_start(RadiusSearch* st, const double* res, double lo, double hi, cudaStream_t s);
// Means of the fields of the current candidates' tables, then one update of *st.
// partials: 3 * (number of blocks) doubles of the reduction scratch.
cudaError_t launch_search_round(const DevParams64& p, int dim, const float* tables, int T, double dmax,
                                RadiusSearch* st, double* partials, int nblocks_max, cudaStream_t s);
// rho0(cell) = table(r - R_e) + (m0 - mm) with r the periodic distance to the
// centre node, linear interpolation, clamped.
cudaError_t launch_search_field(const DevParams64& p, int dim, const float* tables, int T, double dmax,
                                const RadiusSearch* st, double* rho0, cudaStream_t s);

// Per-lattice lookup (defined in kernels_<lattice>.cu). Returns false if the
// combination is not instantiated.
bool kernels_d2q9(int order, int coll, int fp32, KernelSet* ks);
bool kernels_d3q19(int order, int coll, int fp32, KernelSet* ks);
bool kernels_d2q13(int order, int coll, int fp32, KernelSet* ks);
bool kernels_d2q25(int order, int coll, int fp32, KernelSet* ks);

// Slots of the reduction result array `res`.
enum ResSlot {
    kResMass = 0, kResMomX, kResMomY, kResMomZ, kResSumU, kResMaxU, kResCount,
    kResRhoCentre = 8, kResRhoOrigin = 9, kResLine = 16  // then nx values
};
constexpr int kObsWidth = 6;

}  // namespace lbm
