// kg_launch.h -- host-side launchers of the step passes (one definition per precision).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include <functional>
#include <string>

namespace kg {

// grid sizes of the grid-stride kernels (any count is correct; these fill a 152-SM GB300
// four or eight CTAs deep)
constexpr int kStrideCtas = 152 * 4;
constexpr int kStrideCtasDeep = 152 * 8;

struct KgDev;
struct EnsParams;
struct EnsInst;
struct EnsAxis;

// the composed scheme's per-substep data, passed by value to the update kernels
struct C4Args {
    const double2* kick;   // [3][stride]: (K_s, K_s omega^2) by integer m^2
    int stride;            // entries per substep table (3 (N/2)^2 + 1)
    double h[3];           // drift length of each substep
};

// the finaliser of a pass (kg_kernels.cuh): what it does, the pass's partials and the run state
enum { FIN_NONE = 0, FIN_X, FIN_X_AHEAD, FIN_AHEAD_DONE, FIN_PEEK, FIN_Z };
struct FinArgs {
    int kind = FIN_NONE;
    int count = 0;
    const double* part_sum = nullptr;
    const double* part_max = nullptr;
    KgDev* dev = nullptr;
    double norm = 0.0;
};

// precision ids match KG_FP64 / KG_DF64 / KG_MIXED of kg.h
struct PassLaunch {
    // x pass over W1 in the context's precision; mode 0 step, 1 peek.  Writes nparts partials
    // (of sum u^4 in a stepping pass when the step records or `record` is set).
    cudaError_t (*pass_x)(int N, int mode, void* W, KgDev* dev, double* part_sum, double* part_max, const void* tw,
                          double scale, double lam, int record, cudaStream_t st);
    // forward y columns W1 (x-lines) -> W2 (z-columns), inverse y columns W2 -> W1; z columns of
    // W2 in place (sign -1 forward, +1 inverse; FP64 only).  fin runs in one more CTA of the y pass.
    // lg: tiles of 2^lg columns in the z-columns (struct Lay): the context's, which the FP64 kernels
    // have to be told, being used by contexts of every precision; the others know theirs.
    cudaError_t (*yf)(int N, const void* W1, void* W2, const void* tw, int lg, const FinArgs& fin, cudaStream_t st);
    cudaError_t (*yi)(int N, const void* W2, void* W1, const void* tw, int lg, const FinArgs& fin, cudaStream_t st);
    cudaError_t (*zcol)(int N, int sign, void* W2, const void* tw, int lg, cudaStream_t st);
    // inverse z columns from an FP64 spectral source (chosen by dev->phase when dev != NULL) into W2
    cudaError_t (*z_from_f64)(int N, const double2* src0, const double2* src1, const KgDev* dev, void* W2,
                              const void* tw, int lg, cudaStream_t st);
    // streaming FP64 update between a forward and an inverse z column pass; writes
    // update_parts(N) Q partials when recording; c4: the composed scheme's tables (NULL:
    // Eq. (2))
    cudaError_t (*update)(int N, void* W, double2* S0, double2* S1, KgDev* dev, double* part_sum, const double2* coef,
                          const double* w2tab, double inv_dt, const C4Args* c4, cudaStream_t st);
    int (*update_parts)(int N);
    // `steps` steps of the ensemble, one persistent cooperative launch (kg_ensemble.cuh) in launch
    // schedule sched (0 .. kEnsSchedules-1) and unit order `order`, and the CTAs per SM that
    // schedule can hold
    cudaError_t (*ens_run)(const EnsParams& p, int grid, int sched, int order, int steps, cudaStream_t st);
    int (*ens_blocks_per_sm)(int sched);
    // fill the state (and the 16-byte work arrays) of Gaussian instances from their 1D transforms
    cudaError_t (*ens_fill)(const EnsInst* inst, int count, const EnsAxis* axis, const double* A, double lam,
                            const double2* coef64, const double2* coef128, cudaStream_t st);
    int (*x_parts)(int N);
    size_t store_bytes;  // bytes of one complex value of W
    int (*lg)(int N);    // layout of the state and of W2 in an N^3 context of this precision (struct Lay)
    // complex field (full N^3 spectrum, N columns per plane): x pass, column FFTs,
    // column FFT from an FP64 source, update, and their partial counts
    cudaError_t (*passc_x)(int N, int mode, void* W, KgDev* dev, double* part_sum, double* part_max, const void* tw,
                           double scale, double lam, cudaStream_t st);
    int (*xc_parts)(int N);
    cudaError_t (*yfc)(int N, const void* W1, void* W2, const void* tw, int lg, const FinArgs& fin, cudaStream_t st);
    cudaError_t (*yic)(int N, const void* W2, void* W1, const void* tw, int lg, const FinArgs& fin, cudaStream_t st);
    cudaError_t (*zcolc)(int N, int sign, void* W2, const void* tw, int lg, cudaStream_t st);
    cudaError_t (*zc_from_f64)(int N, const double2* src0, const double2* src1, const KgDev* dev, void* W2,
                               const void* tw, int lg, cudaStream_t st);
    cudaError_t (*updatec)(int N, void* W, double2* S0, double2* S1, KgDev* dev, double* part_sum,
                           const double2* coef, const double* w2tab, double inv_dt, cudaStream_t st);
    int (*updatec_parts)(int N);
    // the z pass in one kernel: forward z FFT, update (as update / updatec), inverse z
    // FFT, of a real (cplx = false) or complex field; zstep_parts(N, cplx) Q partials.
    // NULL where the step runs forward z, update and inverse z as three kernels.  tail: the two
    // finalisers that its last CTA runs (after plane; NULL: they ride in y passes).
    cudaError_t (*zstep)(int N, bool cplx, void* W, double2* S0, double2* S1, KgDev* dev, double* part_sum,
                         const void* tw, const double2* coef, const double* w2tab, double inv_dt, const C4Args* c4,
                         const FinArgs* tail, cudaStream_t st);
    int (*zstep_parts)(int N, bool cplx);
    // set-up and read-out transforms in the pass precision (NULL: the FP64 kernels serve):
    // x_setup: physical FP64 lines (lam u^3 when cube) -> half spectra along x in W format;
    // x_readout: W-format half spectra along x -> physical FP64 lines times scale;
    // z_to_f64: forward z columns of W2 into an FP64 spectral array
    cudaError_t (*x_setup)(int N, const double* u, void* spec, const void* tw, int cube, double lam, cudaStream_t st);
    cudaError_t (*x_readout)(int N, void* spec, double* u, const void* tw, double scale, cudaStream_t st);
    cudaError_t (*z_to_f64)(int N, const void* W2, double2* out, const void* tw, cudaStream_t st);
    // the same for a complex field (N-point lines, N columns per plane)
    cudaError_t (*xc_setup)(int N, const double2* u, void* spec, const void* tw, int cube, double lam,
                            cudaStream_t st);
    cudaError_t (*xc_readout)(int N, void* spec, double2* u, const void* tw, double scale, cudaStream_t st);
    cudaError_t (*zc_to_f64)(int N, const void* W2, double2* out, const void* tw, cudaStream_t st);
    // inverse y, x pass and forward y of every z-plane in one launch of thread-block
    // clusters (kg_xyfuse.cuh; NULL where not built): do_yi = 0 leaves out the inverse y
    // transforms (W1 holds the y-inverse; otherwise W2 is read); the result goes to W2; writes xy_parts(N) partials of the x
    // pass's statistics; cudaErrorNotSupported for grids it is not built for
    cudaError_t (*xy_fused)(int N, int do_yi, const void* W1, void* W2, KgDev* dev, double* part_sum, double* part_max,
                            const void* tw, double scale, double lam, cudaStream_t st);
    int (*xy_parts)(int N);
    // the same of a small grid, on z-columns in place (kg_plane.cuh; plane_parts(N) = 0, or NULL,
    // where not built): plane_parts(N) partials of sum u^4 when the step records, max |u| in the
    // run state; ahead (FIN_X_AHEAD, or FIN_NONE), before, after, phase_clk: see there
    cudaError_t (*plane)(int N, void* W, KgDev* dev, double* part_sum, const void* tw, double scale, double lam,
                         const FinArgs& ahead, KgDev* before, KgDev* after, long long* phase_clk, cudaStream_t st);
    int (*plane_parts)(int N);
};

extern const PassLaunch kLaunchF64;
extern const PassLaunch kLaunchDF;
extern const PassLaunch kLaunchF32;

// values a spectral array holds, padding included (struct Lay)
inline size_t spec_slots(int N, bool cplx) { return (size_t)N * N * (cplx ? N : (N / 2 + 8) / 8 * 8); }

// z-columns (the layout of the state) -> the packed order [kz][ky][kx], or back
cudaError_t launch_repack(int N, bool cplx, bool to_packed, const double2* in, double2* out, int lg, cudaStream_t st);

// FP64 set-up / read-out launchers
cudaError_t launch_x_forward(int N, const double* u, double2* out, const double2* tw, int cube, double lam,
                             cudaStream_t st);
cudaError_t launch_x_inverse(int N, const double2* in, double* u, const double2* tw, double scale, double* part_sum,
                             cudaStream_t st);
int x_inverse_parts(int N);   // partial sums launch_x_inverse writes
// cplx: full N^3 spectrum of a complex field instead of the half spectrum
cudaError_t launch_startup(int N, const double2* a, double2* b, const double2* f, const double2* coef, double dt,
                           bool cplx, int lg, cudaStream_t st);
// startup of the composed scheme (real field): b = vh^0 -> P^0 (k_startup_c4)
cudaError_t launch_startup_c4(int N, const double2* a, double2* b, const double2* f, const double2* kick0,
                              int lg, cudaStream_t st);
cudaError_t launch_energy_q(int N, const double2* x, const double2* y, const double* w2tab, double inv_dt,
                            double* part_sum, int nparts, bool cplx, int lg, cudaStream_t st);
// complex field, FP64: forward transform along x (u -> out; cube: of lam |u|^2 u) and
// inverse transform along x times scale (u may be NULL; part_sum: per-CTA sum |u|^4)
cudaError_t launch_xc_forward(int N, const double2* u, double2* out, const double2* tw, int cube, double lam,
                              cudaStream_t st);
cudaError_t launch_xc_inverse(int N, const double2* in, double2* u, const double2* tw, double scale,
                              double* part_sum, cudaStream_t st);
int xc_inverse_parts(int N);
// a finaliser as a kernel of its own; before / after (host memory the device can write, or
// NULL) receive the run state around it
cudaError_t launch_fin(const FinArgs& fin, KgDev* before, KgDev* after, cudaStream_t st);
cudaError_t launch_fin_sum(const double* ps, int count, double norm, double* out, cudaStream_t st);
// composed scheme: partials of the quadratic energy sum_k w_k (|p|^2 + omega^2 |a|^2) / 2 with
// the synchronised velocity p formed from the stored P, F = R2C(lam u^3) and the first kick table
cudaError_t launch_energy_c4(int N, const double2* a, const double2* P, const double2* f, const double2* kick0,
                             const double* w2tab, double* part_sum, int nparts, int lg, cudaStream_t st);
// FP64 forward 3D transform of a physical array (cube: of lam u^3 instead of u) into z-columns;
// lines: FP64 spectral scratch for the x-lines
int forward3d_f64(int N, const double* u, double2* lines, double2* out, const double2* tw64, int cube, double lam,
                  int lg, cudaStream_t st);

// ---------------------------------------------------------------------------
// shared host helpers (kg_host.cu)
// ---------------------------------------------------------------------------
const PassLaunch* launcher_for(int prec);

// device tables of one grid: twiddles exp(-2 pi i j/N) in the pass precision and in
// FP64, (2 c_k, 2 beta_k) and omega_k^2 by integer m^2 = mx^2 + my^2 + mz^2
struct Tables {
    void* tw;
    double2* tw64;
    double2* coef;
    double* w2;
};
typedef std::function<int(void**, size_t, const char*)> AllocFn;
int make_tables(int N, int prec, double L, double dt, const AllocFn& alloc, Tables* t);
// the composed scheme's merged-kick tables [3][3 (N/2)^2 + 1] of (K_s, K_s omega^2) and
// its substep lengths h[3] = (g1, g2, g1) dt
int make_kick_tables(int N, double L, double dt, const AllocFn& alloc, double2** kick, double h[3]);

// Set-up of one state from the physical field in phys (N^3 doubles, overwritten):
// S0 = uh^0, S1 = uh^{-1} (startup level of Eq. (2)) or, with kick0 (the composed
// scheme's first merged-kick table), S1 = P^0; W1 = yz-inverse of uh^0 in the pass
// precision.  W2 and fbuf are scratch of 16 bytes per slot (W2 is the step's second work
// array).  The transforms run in the pass precision where it has x_setup, through W1 and W2, and
// in FP64 elsewhere.
int init_state(int N, int prec, double dt, double lam, const Tables& tb, double* phys, const double* v0,
               bool v0_on_device, double2* S0, double2* S1, void* W1, void* W2, double2* fbuf, cudaStream_t st,
               const double2* kick0 = nullptr);

// the same for a complex field: phys and v0 hold N^3 complex values, the spectral arrays
// the full N^3 spectrum
int init_state_c(int N, int prec, double dt, double lam, const Tables& tb, double2* phys, const double2* v0,
                 bool v0_on_device, double2* S0, double2* S1, void* W1, void* W2, double2* fbuf, cudaStream_t st);

// record a failure for kg_last_error(); returns code
int set_last_error(int code, const std::string& msg);

}  // namespace kg
