// kg_ensemble.cuh -- persistent launches that advance a batch of independent instances
// of the scheme (parametric studies of blow-up, Aseeri et al. section 1), on grids of
// 64^3 and 128^3, by several time steps each.
//
// A step of one instance is four passes (x, forward y, z with the update, inverse y), each cut
// into work units of 256 threads.  The units of a launch form one list: step by step and pass by
// pass, those of every live instance in turn.  CTAs draw runs of consecutive
// units from it in order.  A run waits until its instance's earlier passes are complete (a counter
// of finished units per instance); with the units of the other instances in between they nearly
// always are, so no pass ends with idle SMs.
// The earlier form (one launch per step, a grid barrier after each pass, static shares) had 2.7
// to 4 barrier and 4.6 to 8.8 memory stalls per issued instruction; ms per step, before and now
// in the untuned shape: 48 + 48 instances double-float 3.83 and 2.68, 256 x 64^3 FP32 1.42 and
// 0.79.  Measured and left out: the instances in groups whose arrays fit in L2, each group through
// all the steps (no faster at 10 units a CTA and pass, slower below: the groups wait for their own
// passes), and an L2 prefetch of the next run's data by the thread that draws it (10 % slower).
//
// A run only ever waits for units before it in the list, and every CTA of the (cooperative)
// launch is resident and works its units off in order, so the waits end; each is bounded all the
// same: past spin_limit polls it sets status = 1 and every CTA leaves the launch.
//
// max|u^n| of each instance is gathered during the x pass; an instance whose max exceeds the
// threshold is frozen at level n before its update (its later units do nothing), which is the
// per-instance blow-up flag.
#pragma once
#include "kg_kernels.cuh"

namespace kg {

constexpr int kEnsThreads = 256;
constexpr int kEnsMaxInst = 1024;

struct EnsInst {
    double2* S0;
    double2* S1;
    void* W1;            // x-lines
    void* W2;            // z-columns (struct Lay)
    long long level;
    long long blowup_level;
    int N;
    int phase;
    int frozen;
    unsigned maxkey;     // float bits of max|u| so far in the current step's x pass
    double maxabs;       // max |u^l| seen by the last step that ran
};

struct EnsTab {
    const void* tw;
    const double2* coef;
};

// the list of a launch, written by k_ens_plan: class 0 holds 64^3 instances, class 1 128^3
struct EnsList {
    int live[2];               // instances of the class in the list
    int first;                 // class whose units come first in a pass
    int steps;
    int run;                   // units of a run
    unsigned short inst[2][kEnsMaxInst];   // instance indexes, phase0 in the top bit:
};                                         // the array roles at the start of the launch
constexpr unsigned kEnsSwapped = 0x8000u;
struct EnsPlan {
    EnsList list;
    unsigned ticket;           // next run
    unsigned done[kEnsMaxInst];    // finished units of instance i in this launch; kEnsFrozen once it blew up
    unsigned zdone[kEnsMaxInst];   // finished z units
};
constexpr unsigned kEnsFrozen = 0x80000000u;

struct EnsParams {
    EnsInst* inst;
    EnsPlan* plan;
    int count;
    EnsTab tab[2];
    int* status;               // 0 ok, 1 a wait timed out
    const int* order_idx;      // instance visiting order (length count)
    double lam;
    unsigned thr_key;          // float bits of the blow-up threshold (0xffffffff: off)
    int run;                   // most units of a run
    int missing;               // test hook: waits ask for one unit more than there are
    long long spin_limit;
};

// Launch schedules of the ensemble step, chosen by the autotuner (kg_ens_tune):
//   bit 0: column tiles of half the default width (64-byte instead of 128-byte rows;
//          twice the tiles per unit);
//   bit 1: the short radix stage first in transforms whose length is not a power of 8
//          (128-point columns and x-line pairs, 32-point FP32 x-lines; FftShape).
// Every schedule computes the same step; a tile width changes nothing of the arithmetic,
// the stage order changes the rounding of the transforms (double-float/FP32 level).
constexpr int kEnsSchedules = 4;
template <int SCHED>
struct EnsSched {
    static constexpr int cdiv = (SCHED & 1) ? 2 : 1;
    static constexpr bool remfirst = (SCHED & 2) != 0;
};

// work units per pass for a grid of size N (256 threads each)
template <class P, int N, int SCHED = 0>
struct EnsUnits {
    static constexpr int C = ColShape<P>::C / EnsSched<SCHED>::cdiv;
    static constexpr int TPP = (N / 2 + 1 + C - 1) / C;              // column tiles per plane
    static constexpr int TPU = kEnsThreads / (C * N / 8);             // tiles per unit
    static constexpr int col_units = (N * TPP + TPU - 1) / TPU;
    static constexpr int LPU = kEnsThreads / (N / 16);                // x-lines per unit
    static constexpr int x_units = N * N / LPU;
    static constexpr int step_units = x_units + 3 * col_units;
    static_assert(TPU >= 1 && LPU >= 1, "unit shape");
};

// a column tile of a unit: NT threads, synchronised on their own (the tiles of a unit are
// independent)
template <class P, int C, int NT>
struct TileSmem {
    typename P::S* base;
    int c;
    unsigned bar;
    __device__ __forceinline__ void put(int row, cx<typename P::R> v) { base[col_slot<P, C>(row, c)] = P::pack(v); }
    __device__ __forceinline__ cx<typename P::R> get(int row) const { return P::load(base[col_slot<P, C>(row, c)]); }
    __device__ __forceinline__ void sync() const {
        if (NT <= 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;\n" ::"r"(bar), "r"(NT) : "memory");
    }
};

// dynamic shared memory of the launch: both twiddle tables (64, then 128 entries), then the
// exchange space of a unit
template <class S>
__device__ __forceinline__ S* ens_smem() {
    extern __shared__ __align__(16) unsigned char smraw[];
    return reinterpret_cast<S*>(smraw);
}
template <class S, int N>
__device__ __forceinline__ const S* ens_twiddles() {
    return ens_smem<S>() + (N == 64 ? 0 : 64);
}
constexpr int kEnsTables = 192;

// The bodies of the four passes, one unit each.  Functions of their own, so that each gets the
// whole register budget and the unit loop keeps nothing alive across them.
template <class P, int N, int SCHED>
__device__ __noinline__ void ens_x(typename P::S* W1, int unit, double lam, unsigned* maxkey) {
    typedef typename P::S S;
    const S* tw = ens_twiddles<S, N>();
    S* sm = ens_smem<S>() + kEnsTables;
    typedef EnsUnits<P, N, SCHED> U;
    constexpr bool RF = EnsSched<SCHED>::remfirst;
    Stats<P> st;
    st.init();
    if constexpr (XPaired<P>::value) {
        // lines in pairs through one N-point transform (a pair fits in one warp here)
        typedef XpShape<N> XP;
        static_assert(!XP::CTA_SYNC, "ensemble grids keep a line pair inside a warp");
        const int pi = threadIdx.x / XP::T, jp = threadIdx.x % XP::T;
        const size_t pair = (size_t)unit * (U::LPU / 2) + pi;
        LineSmemX<P, false> lsm{sm + pi * XP::PADN, 0u, 0u};
        x_pair_body<P, N, MODE_STEP, LineSmemX<P, false>, RF>(W1 + 2 * pair * Lay<N>::PITCH, jp, lsm, tw,
                                                              1.0 / ((double)N * N * N), P::from_f64(lam), false, st);
    } else {
        constexpr int T = N / 16;
        const int li = threadIdx.x / T, j = threadIdx.x % T;
        const size_t line = (size_t)unit * U::LPU + li;
        LineSmem<P> lsm{sm + li * XShape<N>::PADM};
        x_line_body<P, N, MODE_STEP, const S*, S* __restrict__, RF>(W1 + line * Lay<N>::PITCH,
                                                                    W1 + line * Lay<N>::PITCH, j, lsm, tw,
                                                                    1.0 / ((double)N * N * N), P::from_f64(lam), false,
                                                                    st);
    }
    const unsigned wmax = __reduce_max_sync(0xffffffffu, st.fkey());
    if ((threadIdx.x & 31) == 0) atomicMax(maxkey, wmax);
}

template <class P, int N, int SCHED>
struct EnsTile {
    typedef EnsUnits<P, N, SCHED> U;
    static constexpr int C = U::C, NT = C * N / 8;
    int plane, kx, j;
    bool valid;
    TileSmem<P, C, NT> csm;
    __device__ __forceinline__ explicit EnsTile(int unit) {
        typename P::S* sm = ens_smem<typename P::S>() + kEnsTables;
        const int sub = threadIdx.x / NT, t = threadIdx.x % NT;
        const int tile = unit * U::TPU + sub;
        const bool ok = tile < N * U::TPP;
        j = t / C;
        plane = ok ? tile / U::TPP : 0;
        kx = (ok ? tile % U::TPP : 0) * C + t % C;
        valid = ok && kx < N / 2 + 1;
        csm = TileSmem<P, C, NT>{sm + sub * (N * C), t % C, 1u + (unsigned)sub};
    }
};

template <class P, int N, int SCHED, int SIGN, int DIR>
__device__ __noinline__ void ens_y(const typename P::S* src, typename P::S* dst, int unit) {
    EnsTile<P, N, SCHED> t(unit);
    col_body<P, P, P, N, SIGN, DIR, false, decltype(t.csm), EnsSched<SCHED>::remfirst>(
        src, dst, t.plane, t.kx, t.valid, t.j, t.csm, ens_twiddles<typename P::S, N>(), LayLg<P, N>::value);
}

template <class P, int N, int SCHED>
__device__ __noinline__ void ens_z(typename P::S* W2, const double2* cur, double2* old, int unit,
                                   const double2* coef) {
    EnsTile<P, N, SCHED> t(unit);
    z_body<P, N, decltype(t.csm), EnsSched<SCHED>::remfirst>(W2, cur, old, t.kx, t.plane, t.valid, t.j, t.csm,
                                                             ens_twiddles<typename P::S, N>(), coef);
}

// the run of units a ticket stands for
struct EnsRun {
    int cls, inst, pass, first, count;
    int swapped;     // uh^n is in S1
    unsigned need;   // finished units of the instance it waits for
    unsigned zlast;  // z units of a step
    void *W1, *W2;
    double2 *S0, *S1;
};

template <class U64, class U128>
__device__ __forceinline__ bool ens_decode(const EnsList* pl, unsigned ticket, EnsRun& u) {
    const unsigned len = (unsigned)pl->run, l0 = (unsigned)pl->live[0], l1 = (unsigned)pl->live[1];
    // runs of a pass per instance of each class, and of a whole x or column pass
    const unsigned xr0 = (U64::x_units + len - 1) / len, xr1 = (U128::x_units + len - 1) / len;
    const unsigned cr0 = (U64::col_units + len - 1) / len, cr1 = (U128::col_units + len - 1) / len;
    const unsigned xs = l0 * xr0 + l1 * xr1, cs = l0 * cr0 + l1 * cr1, step = xs + 3 * cs;
    if (step == 0) return false;
    const unsigned k = ticket / step;
    if (k >= (unsigned)pl->steps) return false;
    ticket -= k * step;
    u.pass = 0;
    if (ticket >= xs) {
        ticket -= xs;
        const unsigned pp = ticket / cs;
        ticket -= pp * cs;
        u.pass = 1 + (int)pp;
    }
    // the class in the order asked for, the instance within it, the run within its pass
    const unsigned r0 = u.pass == 0 ? xr0 : cr0, r1 = u.pass == 0 ? xr1 : cr1;
    const unsigned lead = pl->first ? l1 * r1 : l0 * r0;
    int c = pl->first;
    if (ticket >= lead) {
        ticket -= lead;
        c = 1 - c;
    }
    const unsigned runs = c ? r1 : r0, i = ticket / runs, r = ticket - i * runs;
    const unsigned xu = c ? U128::x_units : U64::x_units, cu = c ? U128::col_units : U64::col_units;
    const unsigned units = u.pass == 0 ? xu : cu;
    u.cls = c;
    const unsigned e = pl->inst[c][i];
    u.inst = (int)(e & ~kEnsSwapped);
    u.swapped = (int)(((e & kEnsSwapped) != 0) ^ (k & 1u));   // a live instance swaps every step
    u.first = (int)(r * len);
    u.count = (int)(r + 1 < runs ? len : units - r * len);
    u.need = k * (xu + 3 * cu) + (u.pass == 0 ? 0u : xu + (unsigned)(u.pass - 1) * cu);
    u.zlast = cu;
    return true;
}

// The list of a launch of `steps` steps (EnsPlan): the live instances of each class in visiting
// order, the counters at zero.  One CTA; a kernel of its own, so that every CTA of the launch sees the same list whatever
// freezes meanwhile.
template <class P, int SCHED>
__global__ void __launch_bounds__(kEnsMaxInst) k_ens_plan(EnsParams p, int order, int steps, int grid) {
    typedef EnsUnits<P, 64, SCHED> U64;
    typedef EnsUnits<P, 128, SCHED> U128;
    __shared__ int s_warp[2][kEnsMaxInst / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int i = t < p.count ? p.order_idx[t] : -1;
    const bool live = i >= 0 && !p.inst[i].frozen;
    const int cls = i >= 0 && p.inst[i].N == 128;
    EnsPlan* pl = p.plan;
    EnsList* ls = &pl->list;
    pl->done[t] = 0u;
    pl->zdone[t] = 0u;
    unsigned mine[2];
    for (int c = 0; c < 2; c++) {
        mine[c] = __ballot_sync(0xffffffffu, live && cls == c);
        if (lane == 0) s_warp[c][w] = __popc(mine[c]);
    }
    __syncthreads();
    if (t < 2) {
        int run = 0;
        for (int q = 0; q < kEnsMaxInst / 32; q++) {
            const int n = s_warp[t][q];
            s_warp[t][q] = run;
            run += n;
        }
        ls->live[t] = run;
    }
    __syncthreads();
    if (live)
        ls->inst[cls][s_warp[cls][w] + __popc(mine[cls] & ((1u << lane) - 1u))] =
            (unsigned short)(i | (p.inst[i].phase ? kEnsSwapped : 0u));
    if (t == 0) {
        const int units = ls->live[0] * U64::col_units + ls->live[1] * U128::col_units;   // of a column pass
        ls->first = order == 1 ? 1 : cls;   // order 0: the grid of the first instance comes first
        ls->steps = steps;
        ls->run = max(1, min(p.run, units / (3 * grid)));   // about three runs a CTA and pass, or single units
        pl->ticket = 0u;
    }
}

// resident CTAs per SM the step kernel is compiled for (the autotuner picks up to this many).  At 64
// registers the double-float z bodies spill 180 to 272 bytes and the FP32 ones up to 96 (128^3,
// half-width tiles or the short stage first), and four CTAs are still the fastest of those measured: FP32
// compiled for five and six spilled more and was 8 and 14 % slower
template <class P>
struct EnsMinBlocks {
    static constexpr int value = 2;
};
template <>
struct EnsMinBlocks<PrecDF> {
    static constexpr int value = 4;
};
template <>
struct EnsMinBlocks<PrecF32> {
    static constexpr int value = 4;
};

template <class P, int SCHED>
__global__ void __launch_bounds__(kEnsThreads, EnsMinBlocks<P>::value) k_ens_run(EnsParams p) {
    typedef typename P::S S;
    typedef EnsUnits<P, 64, SCHED> U64;
    typedef EnsUnits<P, 128, SCHED> U128;
    S* tws = ens_smem<S>();
    __shared__ EnsRun s_run;
    __shared__ EnsList s_list;
    __shared__ int s_go;        // 1: do the run, 2: nothing to do for it, 0: leave the launch
    unsigned ticket = 0;        // thread 0: the next ticket, drawn one ahead (a CTA's runs keep their order)

    for (int i = threadIdx.x; i < 64; i += kEnsThreads)
        if (p.tab[0].tw) tws[i] = ((const S*)p.tab[0].tw)[i];
    for (int i = threadIdx.x; i < 128; i += kEnsThreads)
        if (p.tab[1].tw) tws[64 + i] = ((const S*)p.tab[1].tw)[i];
    for (int i = threadIdx.x; i < (int)(sizeof(EnsList) / 4); i += kEnsThreads)
        reinterpret_cast<unsigned*>(&s_list)[i] = reinterpret_cast<const unsigned*>(&p.plan->list)[i];
    if (threadIdx.x == 0) ticket = atomicAdd(&p.plan->ticket, 1u);
    __syncthreads();

    for (;;) {
        if (threadIdx.x == 0) {
            EnsRun u;
            int go = 0;
            if (ens_decode<U64, U128>(&s_list, ticket, u)) {
                ticket = atomicAdd(&p.plan->ticket, 1u);
                const EnsInst* in = p.inst + u.inst;
                u.W1 = in->W1;
                u.W2 = in->W2;
                u.S0 = in->S0;
                u.S1 = in->S1;
                const unsigned need = u.need + (p.missing ? 1u : 0u);
                volatile unsigned* done = p.plan->done + u.inst;
                go = 1;
                long long spins = 0;
                unsigned d;
                while (((d = *done) & ~kEnsFrozen) < need) {
                    if (++spins > p.spin_limit || *((volatile int*)p.status) != 0) {
                        atomicExch(p.status, 1);
                        go = 0;
                        break;
                    }
                    __nanosleep(20);
                }
                __threadfence();   // what those units wrote is visible from here on
                if (go) {
                    if (d & kEnsFrozen) go = 2;
                    else if (u.pass == 2 && *((volatile unsigned*)&p.inst[u.inst].maxkey) > p.thr_key) go = 2;
                }
                s_run = u;
            }
            s_go = go;
        }
        __syncthreads();
        const int go = s_go;
        if (go == 0) return;
        if (go == 1) {
            unsigned* maxkey = &p.inst[s_run.inst].maxkey;
            S* W1 = (S*)s_run.W1;
            S* W2 = (S*)s_run.W2;
            const int pass = s_run.pass, cls = s_run.cls, last = s_run.first + s_run.count;
            const double2* cur = s_run.swapped ? s_run.S1 : s_run.S0;
            double2* old = s_run.swapped ? s_run.S0 : s_run.S1;
            // a thread's part of the exchange space is that of its own tile or line in every unit,
            // so the units of a run need no barrier between them
#pragma unroll 1
            for (int unit = s_run.first; unit < last; unit++) {
                if (pass == 0) {
                    if (cls == 0) ens_x<P, 64, SCHED>(W1, unit, p.lam, maxkey);
                    else ens_x<P, 128, SCHED>(W1, unit, p.lam, maxkey);
                } else if (pass == 1) {
                    if (cls == 0) ens_y<P, 64, SCHED, -1, COL_YF>(W1, W2, unit);
                    else ens_y<P, 128, SCHED, -1, COL_YF>(W1, W2, unit);
                } else if (pass == 2) {
                    if (cls == 0) ens_z<P, 64, SCHED>(W2, cur, old, unit, p.tab[0].coef);
                    else ens_z<P, 128, SCHED>(W2, cur, old, unit, p.tab[1].coef);
                } else {
                    if (cls == 0) ens_y<P, 64, SCHED, +1, COL_YI>(W2, W1, unit);
                    else ens_y<P, 128, SCHED, +1, COL_YI>(W2, W1, unit);
                }
            }
        }
        __syncthreads();   // the run's writes precede its count; its exchange space is free
        if (threadIdx.x == 0) {
            __threadfence();
            const int inst = s_run.inst;
            const unsigned n = (unsigned)s_run.count;
            unsigned count = n;
            if (s_run.pass == 2 && (atomicAdd(p.plan->zdone + inst, n) + n) % s_run.zlast == 0u) {
                // the instance's last z units of the step: blow-up flag, level, array roles; the
                // next pass waits for this run's count too
                __threadfence();
                volatile EnsInst* v = p.inst + inst;
                if (!v->frozen) {
                    const unsigned key = v->maxkey;
                    v->maxabs = (double)__uint_as_float(key);
                    if (key > p.thr_key) {
                        v->frozen = 1;
                        v->blowup_level = v->level;
                        count += kEnsFrozen;
                    } else {
                        v->level = v->level + 1;
                        v->phase = v->phase ^ 1;
                        v->maxkey = 0u;
                    }
                }
                __threadfence();
            }
            atomicAdd(p.plan->done + inst, count);
        }
    }
}

// ---------------------------------------------------------------------------
// Set-up of the Gaussian instances.  u0 = A exp(-|x|^2/s^2) is a product g(x) g(y) g(z) on the grid,
// and so is u0^3; their transforms are products of 1D ones, and the yz-inverse of uh^0 that W1
// holds is N^2 A g(z) g(y) G(kx).  So a set-up is 130 sums of N terms and one pass that writes the
// arrays, in place of three 3D transforms in FP64: kg_ens_init of 48 + 48 double-float instances 36.1
// -> 5.7 ms, of 256 x 64^3 FP32 ones 35.9 -> 5.4 ms (most of what is left is allocation)
// ---------------------------------------------------------------------------
// per instance: g_j (N values), G(m) and the transform of g^3 (m = 0..N/2 each; both real, since
// the grid has x_{N-j} = -x_j), compensated FP64 sums
struct EnsAxis {
    double g[128], G[65], G3[65];
};

__global__ void __launch_bounds__(128) k_ens_axis(const EnsInst* inst, const double* s, double L, const double2* tw64,
                                                  const double2* tw128, EnsAxis* out);

// S0 = uh^0, S1 = uh^{-1} = c uh^0 + beta F^0 (v0 = 0) and, with W1 in FP64 or double-float, its
// x-lines; the slots of padding get zeros
template <class P, int N>
__device__ __forceinline__ void ens_fill(const EnsInst& in, const EnsAxis& ax, double A, double lam,
                                         const double2* __restrict__ coef) {
    typedef ModeIndex<N, false> MI;
    typedef typename P::S S;
    constexpr unsigned PITCH = Lay<N>::PITCH;
    constexpr int LG = LayLg<P, N>::value;
    const double A3 = lam * (A * A * A), An2 = A * ((double)N * N);
    S* W1 = (S*)in.W1;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < MI::slots(LG); i += gridDim.x * blockDim.x) {
        const MI mi(i, LG);
        double a = 0.0, b = 0.0;
        if (mi.valid) {
            const int my = mi.ky <= N / 2 ? mi.ky : N - mi.ky, mz = mi.kz <= N / 2 ? mi.kz : N - mi.kz;
            const double2 cf = coef[mi.m2];
            a = A * (ax.G[mi.kx] * ax.G[my] * ax.G[mz]);
            b = 0.5 * cf.x * a + 0.5 * cf.y * (A3 * (ax.G3[mi.kx] * ax.G3[my] * ax.G3[mz]));
        }
        in.S0[i] = make_double2(a, 0.0);
        in.S1[i] = make_double2(b, 0.0);
    }
    if constexpr (sizeof(S) == 16) {
        for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (unsigned)Lay<N>::kSlots; i += gridDim.x * blockDim.x) {
            const unsigned row = i / PITCH, kx = i - row * PITCH;
            const double w = kx <= N / 2 ? An2 * (ax.g[row / N] * ax.g[row % N] * ax.G[kx]) : 0.0;
            W1[i] = P::pack(cmake<typename P::R>(P::from_f64(w), P::from_f64(0.0)));
        }
    }
}

template <class P>
__global__ void __launch_bounds__(256) k_ens_fill(const EnsInst* inst, const EnsAxis* axis, const double* A, double lam,
                                                  EnsTab t64, EnsTab t128) {
    __shared__ EnsAxis ax;
    const int i = blockIdx.y;
    const EnsInst in = inst[i];
    const double* src = reinterpret_cast<const double*>(axis + i);
    for (int k = threadIdx.x; k < (int)(sizeof(EnsAxis) / 8); k += blockDim.x) reinterpret_cast<double*>(&ax)[k] = src[k];
    __syncthreads();
    if (in.N == 64) ens_fill<P, 64>(in, ax, A[i], lam, t64.coef);
    else ens_fill<P, 128>(in, ax, A[i], lam, t128.coef);
}

}  // namespace kg
