// kg_launch_impl.cuh -- template launchers, instantiated once per precision.
#pragma once
#include <atomic>
#include <type_traits>
#include "kg_complex.cuh"
#include "kg_ensemble.cuh"
#include "kg_kernels.cuh"
#include "kg_launch.h"
#include "kg_plane.cuh"
#include "kg_xyfuse.cuh"

namespace kg {

// CTAs per cluster of the fused xy pass: a plane of FP32 W is 1.05 MB at N = 512, which
// eight CTAs hold in 136 KB of shared memory each
constexpr int kXyCluster = 8;

// dynamic shared memory limit of a kernel (static shared memory comes on top, so the
// attribute is set whatever the size)
template <class K>
static cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// The attribute is set once per kernel and device (a driver call of its own on every launch
// costs as much host time as the launch).
template <class K>
static cudaError_t set_smem_once(K kernel, size_t bytes, std::atomic<unsigned long long>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = set_smem(kernel, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// a launch that may start while the kernel before it drains (the kernel calls pdl_wait)
template <class... KA, class... A>
static cudaError_t launch_pdl(void (*kernel)(KA...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

#define KG_DISPATCH_N(N, ...)                               \
    switch (N) {                                            \
        case 16: { constexpr int NN = 16; __VA_ARGS__; }    \
        case 32: { constexpr int NN = 32; __VA_ARGS__; }    \
        case 64: { constexpr int NN = 64; __VA_ARGS__; }    \
        case 128: { constexpr int NN = 128; __VA_ARGS__; }  \
        case 256: { constexpr int NN = 256; __VA_ARGS__; }  \
        case 512: { constexpr int NN = 512; __VA_ARGS__; }  \
        default: return cudaErrorInvalidValue;              \
    }

template <class P>
struct Launchers {
    typedef typename P::S S;

    // persistent x pass: as many CTAs as fit on the device at once (both modes), at most
    // one per batch; cached per grid size
    template <int N>
    static size_t x_smem() {
        typedef XShape<N, XStep<N>::NT> X;
        return (size_t)(XPipelined<P>::value ? 2 : 1) * X::LPC * X::PADM * sizeof(S);
    }
    template <int N>
    static int x_grid_n() {
        static int grid = 0;
        if (!XPipelined<P>::value) return N * N / XShape<N, XStep<N>::NT>::LPC;
        if (grid == 0) {
            typedef XShape<N, XStep<N>::NT> X;
            int dev = 0, sms = 0, occ0 = 0, occ1 = 0;
            if (cudaGetDevice(&dev) != cudaSuccess ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
                return 0;
            if (set_smem(k_pass_x<P, N, MODE_STEP>, x_smem<N>()) != cudaSuccess ||
                set_smem(k_pass_x<P, N, MODE_PEEK>, x_smem<N>()) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ0, k_pass_x<P, N, MODE_STEP>, XStep<N>::NT,
                                                              x_smem<N>()) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ1, k_pass_x<P, N, MODE_PEEK>, XStep<N>::NT,
                                                              x_smem<N>()) != cudaSuccess)
                return 0;
            const int occ = occ0 < occ1 ? occ0 : occ1;
            const int nb = N * N / X::LPC;
            grid = occ * sms < nb ? occ * sms : nb;
            if (grid < 1) grid = 1;
        }
        return grid;
    }
    template <int N, int MODE>
    static cudaError_t pass_x_n(void* W, KgDev* dev, double* ps, double* pm, const void* tw, double scale, double lam,
                                int record, cudaStream_t st) {
        static std::atomic<unsigned long long> done{0};
        const int grid = x_grid_n<N>();
        if (grid == 0) return cudaErrorInvalidConfiguration;
        cudaError_t e = set_smem_once(k_pass_x<P, N, MODE>, x_smem<N>(), done);
        if (e != cudaSuccess) return e;
        return launch_pdl(k_pass_x<P, N, MODE>, grid, XStep<N>::NT, x_smem<N>(), st, (S*)W, dev, ps, pm, (const S*)tw,
                          scale, lam, record);
    }
    static cudaError_t pass_x(int N, int mode, void* W, KgDev* dev, double* ps, double* pm, const void* tw,
                              double scale, double lam, int record, cudaStream_t st) {
        if (mode == MODE_STEP) {
            KG_DISPATCH_N(N, return (pass_x_n<NN, MODE_STEP>(W, dev, ps, pm, tw, scale, lam, record, st)));
        }
        KG_DISPATCH_N(N, return (pass_x_n<NN, MODE_PEEK>(W, dev, ps, pm, tw, scale, lam, record, st)));
    }
    // partials the x pass writes (its grid); 0 when the device cannot be queried
    static int x_parts(int N) {
        KG_DISPATCH_N(N, return x_grid_n<NN>());
    }

    // column passes (k_col): Pin -> Pout in the layouts of direction DIR
    template <class Pin, class Pout, int N, int SIGN, int DIR, bool CPLX, int C>
    static cudaError_t col_n(const void* src, void* dst, const void* tw, int lg, const FinArgs& fin, cudaStream_t st) {
        static std::atomic<unsigned long long> done{0};
        constexpr size_t smem = (size_t)(N * C + N) * sizeof(S);
        static_assert(smem >= kFinSmem * sizeof(double), "a finaliser's shared memory");
        auto kern = k_col<Pin, P, Pout, N, SIGN, DIR, CPLX, C>;
        cudaError_t e = set_smem_once(kern, smem, done);
        if (e != cudaSuccess) return e;
        dim3 grid((Lay<N, CPLX>::NX + C - 1) / C, N + (fin.kind != FIN_NONE));
        return launch_pdl(kern, grid, C * N / 8, smem, st, (const typename Pin::S*)src, (typename Pout::S*)dst,
                          (const S*)tw, lg, fin);
    }
    template <bool CPLX>
    static cudaError_t yf_t(int N, const void* W1, void* W2, const void* tw, int lg, const FinArgs& fin, cudaStream_t st) {
        KG_DISPATCH_N(N, return (col_n<P, P, NN, -1, COL_YF, CPLX, ColStep<P, NN, true>::C>(W1, W2, tw, lg, fin, st)));
    }
    template <bool CPLX>
    static cudaError_t yi_t(int N, const void* W2, void* W1, const void* tw, int lg, const FinArgs& fin, cudaStream_t st) {
        KG_DISPATCH_N(N, return (col_n<P, P, NN, +1, COL_YI, CPLX, ColStep<P, NN, true>::C>(W2, W1, tw, lg, fin, st)));
    }
    // z columns in place: FP64 only (the other precisions have the fused z pass)
    template <bool CPLX>
    static cudaError_t zcol_t(int N, int sign, void* W2, const void* tw, int lg, cudaStream_t st) {
        if constexpr (!std::is_same<P, PrecF64>::value) {
            return cudaErrorNotSupported;
        } else {
            if (sign < 0) { KG_DISPATCH_N(N, return (col_n<P, P, NN, -1, COL_Z, CPLX, ColStep<P, NN, false>::C>(W2, W2, tw, lg, FinArgs{}, st))); }
            KG_DISPATCH_N(N, return (col_n<P, P, NN, +1, COL_Z, CPLX, ColStep<P, NN, false>::C>(W2, W2, tw, lg, FinArgs{}, st)));
        }
    }
    template <int N, bool CPLX>
    static cudaError_t z_from_f64_n(const double2* src0, const double2* src1, const KgDev* dev, void* W2,
                                    const void* tw, int lg, cudaStream_t st) {
        static std::atomic<unsigned long long> done{0};
        constexpr int C = ColShape<P>::C;
        const size_t smem = (size_t)(N * C + N) * sizeof(S);
        auto kern = k_col_sel<P, N, CPLX, C>;
        cudaError_t e = set_smem_once(kern, smem, done);
        if (e != cudaSuccess) return e;
        dim3 grid((Lay<N, CPLX>::NX + C - 1) / C, N);
        return launch_pdl(kern, grid, C * N / 8, smem, st, src0, src1, dev, (S*)W2, (const S*)tw, lg);
    }
    template <bool CPLX>
    static cudaError_t z_from_f64_t(int N, const double2* src0, const double2* src1, const KgDev* dev, void* W2,
                                    const void* tw, int lg, cudaStream_t st) {
        KG_DISPATCH_N(N, return (z_from_f64_n<NN, CPLX>(src0, src1, dev, W2, tw, lg, st)));
    }
    // forward z columns from W2 into an FP64 spectral array (pass-precision set-up)
    template <bool CPLX>
    static cudaError_t z_to_f64_t(int N, const void* W2, double2* out, const void* tw, cudaStream_t st) {
        if constexpr (!kPassIO) return cudaErrorNotSupported;
        else { KG_DISPATCH_N(N, return (col_n<P, PrecF64, NN, -1, COL_Z, CPLX, ColShape<P>::C>(W2, out, tw, 0, FinArgs{}, st))); }
    }

    // set-up and read-out transforms in the pass precision (double-float only: the FP32
    // passes would degrade the FP64 state, and the FP64 passes have their own kernels)
    static constexpr bool kPassIO = std::is_same<P, PrecDF>::value;
    template <int N, bool FWD>
    static cudaError_t x_io_n(const double* u_in, void* spec, double* u_out, const void* tw, int cube, double lam,
                              double scale, cudaStream_t st) {
        typedef XpShape<N> X;
        const size_t smem = (size_t)X::PPC * X::PADN * sizeof(S);
        auto kern = k_x_pair_io<P, N, FWD>;
        cudaError_t e = set_smem(kern, smem);
        if (e != cudaSuccess) return e;
        kern<<<N * N / 2 / X::PPC, kXThreads, smem, st>>>(u_in, (S*)spec, u_out, (const S*)tw, cube, lam, scale);
        return cudaGetLastError();
    }
    static cudaError_t x_setup(int N, const double* u, void* spec, const void* tw, int cube, double lam,
                               cudaStream_t st) {
        if constexpr (!kPassIO) return cudaErrorNotSupported;
        else { KG_DISPATCH_N(N, return (x_io_n<NN, true>(u, spec, nullptr, tw, cube, lam, 1.0, st))); }
    }
    static cudaError_t x_readout(int N, void* spec, double* u, const void* tw, double scale, cudaStream_t st) {
        if constexpr (!kPassIO) return cudaErrorNotSupported;
        else { KG_DISPATCH_N(N, return (x_io_n<NN, false>(nullptr, spec, u, tw, 0, 0.0, scale, st))); }
    }
    // the same for a complex field (one N-point transform per line, N columns per plane)
    template <int N, bool FWD>
    static cudaError_t xc_io_n(const double2* u_in, void* spec, double2* u_out, const void* tw, int cube,
                               double lam, double scale, cudaStream_t st) {
        typedef XcShape<N> X;
        const size_t smem = (size_t)X::LPC * X::PADN * sizeof(S);
        auto kern = k_xc_io<P, N, FWD>;
        cudaError_t e = set_smem(kern, smem);
        if (e != cudaSuccess) return e;
        kern<<<N * N / X::LPC, kXThreads, smem, st>>>(u_in, (S*)spec, u_out, (const S*)tw, cube, lam, scale);
        return cudaGetLastError();
    }
    static cudaError_t xc_setup(int N, const double2* u, void* spec, const void* tw, int cube, double lam,
                                cudaStream_t st) {
        if constexpr (!kPassIO) return cudaErrorNotSupported;
        else { KG_DISPATCH_N(N, return (xc_io_n<NN, true>(u, spec, nullptr, tw, cube, lam, 1.0, st))); }
    }
    static cudaError_t xc_readout(int N, void* spec, double2* u, const void* tw, double scale, cudaStream_t st) {
        if constexpr (!kPassIO) return cudaErrorNotSupported;
        else { KG_DISPATCH_N(N, return (xc_io_n<NN, false>(nullptr, spec, u, tw, 0, 0.0, scale, st))); }
    }
    static int update_parts(int N) {   // one partial per CTA over the slots
        KG_DISPATCH_N(N, return (int)((ModeIndex<NN, false>::slots(LayLg<P, NN>::value) + kUpdThreads - 1) / kUpdThreads));
    }
    template <int N>
    static cudaError_t update_n(void* W, double2* S0, double2* S1, KgDev* dev, double* ps, const double2* coef,
                                const double* w2, double inv_dt, const C4Args* c4, cudaStream_t st) {
        const double qr = 0.25 / (inv_dt * inv_dt), qc = 0.5 * inv_dt * inv_dt;
        if (c4)
            return launch_pdl(k_update<P, N, false, 1>, update_parts(N), kUpdThreads, 0, st, (S*)W, S0, S1, dev, ps,
                              coef, w2, qr, qc, *c4);
        return launch_pdl(k_update<P, N, false, 0>, update_parts(N), kUpdThreads, 0, st, (S*)W, S0, S1, dev, ps, coef,
                          w2, qr, qc, C4Args{});
    }
    static cudaError_t update(int N, void* W, double2* S0, double2* S1, KgDev* dev, double* ps, const double2* coef,
                              const double* w2, double inv_dt, const C4Args* c4, cudaStream_t st) {
        KG_DISPATCH_N(N, return update_n<NN>(W, S0, S1, dev, ps, coef, w2, inv_dt, c4, st));
    }
    // ---- complex field ----
    template <int N, int MODE>
    static cudaError_t passc_x_n(void* W, KgDev* dev, double* ps, double* pm, const void* tw, double scale, double lam,
                                 cudaStream_t st) {
        typedef XcShape<N, XcStep<N>::NT> X;
        static std::atomic<unsigned long long> done{0};
        const size_t smem = (size_t)X::LPC * X::PADN * sizeof(S);
        cudaError_t e = set_smem_once(k_pass_xc<P, N, MODE>, smem, done);
        if (e != cudaSuccess) return e;
        return launch_pdl(k_pass_xc<P, N, MODE>, N * N / X::LPC, XcStep<N>::NT, smem, st, (S*)W, dev, ps, pm,
                          (const S*)tw, scale, lam);
    }
    static cudaError_t passc_x(int N, int mode, void* W, KgDev* dev, double* ps, double* pm, const void* tw,
                               double scale, double lam, cudaStream_t st) {
        if (mode == MODE_STEP) {
            KG_DISPATCH_N(N, return (passc_x_n<NN, MODE_STEP>(W, dev, ps, pm, tw, scale, lam, st)));
        }
        KG_DISPATCH_N(N, return (passc_x_n<NN, MODE_PEEK>(W, dev, ps, pm, tw, scale, lam, st)));
    }
    static int xc_parts(int N) {
        KG_DISPATCH_N(N, return (NN * NN / XcShape<NN, XcStep<NN>::NT>::LPC));
    }
    static int updatec_parts(int N) { return (int)(((long long)N * N * N + kUpdThreads - 1) / kUpdThreads); }
    static cudaError_t updatec(int N, void* W, double2* S0, double2* S1, KgDev* dev, double* ps, const double2* coef,
                               const double* w2, double inv_dt, cudaStream_t st) {
        const double qr = 0.25 / (inv_dt * inv_dt), qc = 0.5 * inv_dt * inv_dt;
        KG_DISPATCH_N(N, {
            return launch_pdl(k_update<P, NN, true, 0>, updatec_parts(NN), kUpdThreads, 0, st, (S*)W, S0, S1, dev, ps,
                              coef, w2, qr, qc, C4Args{});
        });
    }

    // fused z pass (forward z FFT, update, inverse z FFT) of a real (cplx = false) or
    // complex field, Eq. (2) (SCHEME 0) or the composed scheme (SCHEME 1, real field);
    // zstep_parts: the Q partials it writes when recording
    template <int N, bool CPLX, int SCHEME, class TAIL = NoTail>
    static cudaError_t zstep_n(void* W, double2* S0, double2* S1, KgDev* dev, double* ps, const void* tw,
                               const double2* coef, const double* w2, double inv_dt, const C4Args& c4,
                               cudaStream_t st, const TAIL& tail = TAIL{}) {
        typedef ZStepShape<P, N> Z;
        static std::atomic<unsigned long long> done{0};
        constexpr int NX = Lay<N, CPLX>::NX;
        const size_t smem = (size_t)(N * Z::C + N) * sizeof(S);
        auto kern = k_zstep<P, N, CPLX, SCHEME, TAIL>;
        cudaError_t e = set_smem_once(kern, smem, done);
        if (e != cudaSuccess) return e;
        const double qr = 0.25 / (inv_dt * inv_dt), qc = 0.5 * inv_dt * inv_dt;
        dim3 grid((NX + Z::C - 1) / Z::C, N);
        return launch_pdl(kern, grid, Z::NT, smem, st, (S*)W, S0, S1, dev, ps, (const S*)tw, coef, w2, qr, qc, c4, tail);
    }
    static cudaError_t zstep(int N, bool cplx, void* W, double2* S0, double2* S1, KgDev* dev, double* ps,
                             const void* tw, const double2* coef, const double* w2, double inv_dt, const C4Args* c4,
                             const FinArgs* tail, cudaStream_t st) {
        if (tail) {
            if (cplx || plane_parts(N) == 0) return cudaErrorInvalidValue;
            const ZTail t{tail[0], tail[1]};
#define KG_TAIL_CASE(NN)                                                                                         \
    case NN:                                                                                                     \
        return c4 ? zstep_n<NN, false, 1, ZTail>(W, S0, S1, dev, ps, tw, coef, w2, inv_dt, *c4, st, t)            \
                  : zstep_n<NN, false, 0, ZTail>(W, S0, S1, dev, ps, tw, coef, w2, inv_dt, C4Args{}, st, t);
            if constexpr (kPlane) {
                switch (N) {
                    KG_TAIL_CASE(16)
                    KG_TAIL_CASE(32)
                    KG_TAIL_CASE(64)
                    default: break;
                }
            }
#undef KG_TAIL_CASE
            return cudaErrorInvalidValue;
        }
        if (cplx) {
            if (c4) return cudaErrorInvalidValue;   // the composed scheme is built for real fields
            KG_DISPATCH_N(N, return (zstep_n<NN, true, 0>(W, S0, S1, dev, ps, tw, coef, w2, inv_dt, C4Args{}, st)));
        }
        if (c4) { KG_DISPATCH_N(N, return (zstep_n<NN, false, 1>(W, S0, S1, dev, ps, tw, coef, w2, inv_dt, *c4, st))); }
        KG_DISPATCH_N(N, return (zstep_n<NN, false, 0>(W, S0, S1, dev, ps, tw, coef, w2, inv_dt, C4Args{}, st)));
    }
    static int zstep_parts(int N, bool cplx) {
        KG_DISPATCH_N(N, {
            constexpr int C = ZStepShape<P, NN>::C;
            return ((cplx ? NN : NN / 2 + 1) + C - 1) / C * NN;
        });
    }

    // ---- inverse y / x / forward y of a z-plane in one kernel (small grids, kg_plane.cuh) ----
    static constexpr bool kPlane = std::is_same<P, PrecDF>::value;
    template <int N>
    static cudaError_t plane_n(void* W, KgDev* dev, double* ps, const void* tw, double scale, double lam, const FinArgs& ahead,
                               KgDev* before, KgDev* after, long long* phase_clk, cudaStream_t st) {
        typedef PlaneShape<N> X;
        static std::atomic<unsigned long long> done{0};
        const size_t smem = (size_t)(X::SLAB + X::LINES + N) * sizeof(S);
        cudaError_t e = set_smem_once(k_plane<P, N>, smem, done);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(N * X::CL);
        cfg.blockDim = dim3(X::NT);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = X::CL;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = X::CL > 1 ? 2 : 1;
        return cudaLaunchKernelEx(&cfg, k_plane<P, N>, (S*)W, dev, ps, (const S*)tw, scale, lam, ahead, before, after, phase_clk);
    }
    static cudaError_t plane(int N, void* W, KgDev* dev, double* ps, const void* tw, double scale, double lam, const FinArgs& ahead,
                             KgDev* before, KgDev* after, long long* phase_clk, cudaStream_t st) {
        if constexpr (kPlane) {
            switch (N) {
                case 16: return plane_n<16>(W, dev, ps, tw, scale, lam, ahead, before, after, phase_clk, st);
                case 32: return plane_n<32>(W, dev, ps, tw, scale, lam, ahead, before, after, phase_clk, st);
                case 64: return plane_n<64>(W, dev, ps, tw, scale, lam, ahead, before, after, phase_clk, st);
                default: break;
            }
        }
        return cudaErrorNotSupported;
    }
    static int plane_parts(int N) {
        if (!kPlane) return 0;
        return N == 16 ? 16 * PlaneShape<16>::CL : N == 32 ? 32 * PlaneShape<32>::CL : N == 64 ? 64 * PlaneShape<64>::CL : 0;
    }

    // ---- fused inverse y / x / forward y pass (FP32 work array, real field) ----
    template <int N, bool DO_YI>
    static cudaLaunchConfig_t xy_config(cudaLaunchAttribute* attr, int grid, cudaStream_t st) {
        typedef XyShape<N, kXyCluster> X;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(X::NT);
        cfg.dynamicSmemBytes = (size_t)(X::SLAB + X::XBUF) * sizeof(float2);
        cfg.stream = st;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kXyCluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cfg;
    }
    // persistent grid: as many clusters as fit on the device at once, at most one per
    // plane; cached per grid size (both variants share it)
    template <int N>
    static int xy_grid_n() {
        static int grid = 0;
        if (grid == 0) {
            cudaLaunchAttribute attr[1];
            cudaLaunchConfig_t cfg = xy_config<N, true>(attr, kXyCluster, nullptr);
            int nc0 = 0, nc1 = 0;
            if (set_smem(k_xy_cluster<N, kXyCluster, true>, cfg.dynamicSmemBytes) != cudaSuccess ||
                set_smem(k_xy_cluster<N, kXyCluster, false>, cfg.dynamicSmemBytes) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&nc0, k_xy_cluster<N, kXyCluster, true>, &cfg) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&nc1, k_xy_cluster<N, kXyCluster, false>, &cfg) != cudaSuccess)
                return 0;
            int nc = nc0 < nc1 ? nc0 : nc1;
            nc = nc < N ? nc : N;
            grid = nc * kXyCluster;
        }
        return grid;
    }
    template <int N, bool DO_YI>
    static cudaError_t xy_n(const void* W1, void* W2, KgDev* dev, double* ps, double* pm, const void* tw, double scale, double lam,
                            cudaStream_t st) {
        const int grid = xy_grid_n<N>();
        if (grid < kXyCluster) return cudaErrorInvalidConfiguration;
        auto kern = k_xy_cluster<N, kXyCluster, DO_YI>;
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = xy_config<N, DO_YI>(attr, grid, st);
        cudaError_t e = set_smem(kern, cfg.dynamicSmemBytes);
        if (e != cudaSuccess) return e;
        return cudaLaunchKernelEx(&cfg, kern, (const float2*)W1, (float2*)W2, dev, ps, pm, (const float2*)tw, scale, lam);
    }
    static cudaError_t xy_fused(int N, int do_yi, const void* W1, void* W2, KgDev* dev, double* ps, double* pm,
                                const void* tw, double scale, double lam, cudaStream_t st) {
        if constexpr (!std::is_same<P, PrecF32>::value) {
            return cudaErrorNotSupported;
        } else {
#define KG_XY_CASE(NN)                                                                       \
    case NN:                                                                                 \
        return do_yi ? xy_n<NN, true>(W1, W2, dev, ps, pm, tw, scale, lam, st)               \
                     : xy_n<NN, false>(W1, W2, dev, ps, pm, tw, scale, lam, st);
            switch (N) {
                KG_XY_CASE(64)
                KG_XY_CASE(128)
                KG_XY_CASE(256)
                KG_XY_CASE(512)
                default: return cudaErrorNotSupported;
            }
#undef KG_XY_CASE
        }
    }
    static int xy_parts(int N) {
        if constexpr (!std::is_same<P, PrecF32>::value) {
            return 0;
        } else {
            switch (N) {
                case 64: return xy_grid_n<64>();
                case 128: return xy_grid_n<128>();
                case 256: return xy_grid_n<256>();
                case 512: return xy_grid_n<512>();
                default: return 0;
            }
        }
    }

    // the ensemble's steps (kg_ensemble.cuh); schedules differ in tile shape and stage order,
    // not in shared memory (a unit's tiles always hold 2048 values)
    template <int SCHED>
    static size_t ens_smem_s() {
        typedef EnsUnits<P, 64, SCHED> U64;
        typedef EnsUnits<P, 128, SCHED> U128;
        size_t a = (size_t)U64::LPU * XShape<64>::PADM, b = (size_t)U128::LPU * XShape<128>::PADM;
        size_t c = (size_t)U64::TPU * 64 * U64::C, d = (size_t)U128::TPU * 128 * U128::C;
        size_t m = a > b ? a : b;
        m = m > c ? m : c;
        m = m > d ? m : d;
        return (m + kEnsTables) * sizeof(S);   // and both twiddle tables
    }
    template <int SCHED>
    static int ens_blocks_per_sm_s() {
        if (set_smem(k_ens_run<P, SCHED>, ens_smem_s<SCHED>()) != cudaSuccess) return 0;
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ens_run<P, SCHED>, kEnsThreads, ens_smem_s<SCHED>()) !=
            cudaSuccess)
            return 0;
        return n;
    }
    static int ens_blocks_per_sm(int sched) {
        switch (sched) {
            case 0: return ens_blocks_per_sm_s<0>();
            case 1: return ens_blocks_per_sm_s<1>();
            case 2: return ens_blocks_per_sm_s<2>();
            case 3: return ens_blocks_per_sm_s<3>();
            default: return 0;
        }
    }
    template <int SCHED>
    static cudaError_t ens_run_s(const EnsParams& p, int grid, int order, int steps, cudaStream_t st) {
        cudaError_t e = set_smem(k_ens_run<P, SCHED>, ens_smem_s<SCHED>());
        if (e != cudaSuccess) return e;
        k_ens_plan<P, SCHED><<<1, kEnsMaxInst, 0, st>>>(p, order, steps, grid);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(kEnsThreads);
        cfg.dynamicSmemBytes = ens_smem_s<SCHED>();
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k_ens_run<P, SCHED>, p);
    }
    static cudaError_t ens_run(const EnsParams& p, int grid, int sched, int order, int steps, cudaStream_t st) {
        switch (sched) {
            case 0: return ens_run_s<0>(p, grid, order, steps, st);
            case 1: return ens_run_s<1>(p, grid, order, steps, st);
            case 2: return ens_run_s<2>(p, grid, order, steps, st);
            case 3: return ens_run_s<3>(p, grid, order, steps, st);
            default: return cudaErrorInvalidValue;
        }
    }
    static cudaError_t ens_fill(const EnsInst* inst, int count, const EnsAxis* axis, const double* A, double lam,
                                const double2* coef64, const double2* coef128, cudaStream_t st) {
        // 64 CTAs an instance: one slot in ten a thread at 64^3
        k_ens_fill<P><<<dim3(64, count), 256, 0, st>>>(inst, axis, A, lam, EnsTab{nullptr, coef64},
                                                      EnsTab{nullptr, coef128});
        return cudaGetLastError();
    }
};

}  // namespace kg
