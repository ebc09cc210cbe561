// kg_plane.cuh -- inverse y, x and forward y passes of one z-plane in one kernel, for grids that
// are bound by launches (real field, double-float work array, N <= 64).
//
// What bounds a step of a small grid is not its arithmetic (64^3: 2 us of FP32 lanes) but the
// chain of dependent kernels, some 4 us each.  The three passes between two z passes mix values
// within one z-plane only, and a plane fits in the shared memory of one CTA (N <= 32) or of two
// (N = 64: 34 KB; two so that 128 SMs share the work and not 64).  So a step is two kernels,
// this one and the z pass, instead of four; the finalisers ride in the last CTA of the z pass.
// Measured (us a step, before and after): 18.0 -> 11.5 at 16^3, 18.9 -> 13.0 at 32^3, 21.2 -> 18.0 at
// 64^3; a step with its energy read 65 -> 50 at 64^3.  What is left is each kernel's start, its first
// loads and the instruction stream of eight points a thread, one warp a scheduler.
//
// CTA r of the CL of a plane owns the kx columns [r CW, (r+1) CW) (the last one also the Nyquist
// column) for the y transforms and the rows [r RPC, (r+1) RPC) for the x transforms.  Each phase
// stores its results where the next one reads them: the inverse y transforms into the row blocks
// of the CTA that transforms them along x, these into the column slabs (stores into the other CTA
// of the cluster, which nothing waits for before the cluster barrier).  A pair of x-lines
// exchanges inside its own row block.  The work array stays in z-columns, read and written in
// place: a plane's part of it belongs to its cluster alone.
//
// The transforms, the statistics of u^n and the cube are those of the separate passes
// (kg_kernels.cuh), so the spectra agree bit for bit.
#pragma once
#include <cooperative_groups.h>

#include "kg_kernels.cuh"

namespace kg {

template <int N>
struct PlaneShape {
    static constexpr int CL = N >= 64 ? 2 : 1;             // CTAs per plane
    static constexpr int NX = N / 2 + 1;
    static constexpr int T = N / 8;                         // threads per column and per pair of x-lines
    static constexpr int CW = (N / 2) / CL, RPC = N / CL;
    static constexpr int PAIRS = RPC / 2;
    static constexpr int NT = ((CW + 1) * T + 31) / 32 * 32;
    static constexpr int CC = NT / T;                       // column slots and row blocks: idle threads transform
                                                            // zeros in those beyond the plane
    static constexpr int PADN = N + N / 8;                  // padded exchange slots of a pair = its row block
    static constexpr int LDX = PADN / 2;                    // row pitch inside a block
    static constexpr int SLAB = N * CC, LINES = CC * PADN;   // values
    static_assert(LDX >= NX && CC >= CW + 1 && CC >= PAIRS && 32 % T == 0 && NT <= 1024, "plane kernel shape");
};

// every thread of every CTA of the cluster: stores before it, into any CTA's shared memory, are
// visible after it
template <int CL>
__device__ __forceinline__ void plane_barrier() {
    if (CL > 1) {
        asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
    } else {
        __syncthreads();
    }
}

// the exchange space of a transform: a column of the slab (rows ld values apart) or a row block (one
// pad slot every eight values)
template <class P>
struct PlaneSmem {
    typename P::S* base;
    int ld, pad;
    __device__ __forceinline__ typename P::S* at(int i) const { return base + i * ld + (i >> 3) * pad; }
    __device__ __forceinline__ void put(int i, cx<typename P::R> v) { *at(i) = P::pack(v); }
    __device__ __forceinline__ cx<typename P::R> get(int i) const { return P::load(*at(i)); }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
};

// W: z-inverse z-columns in, F's y-transform out.  ahead (kind FIN_X_AHEAD, or none): the pass runs
// ahead of its step for kg_energy: sum u^4 in any case, and the CTA that draws the last ticket
// advances the run state, which before and after (host memory) receive as it was and as it is then.
// phase_clk (may be NULL): clocks of the first CTA at the start and after each phase.
template <class P, int N>
__global__ void __launch_bounds__(PlaneShape<N>::NT)
    k_plane(typename P::S* __restrict__ W, KgDev* dev, double* __restrict__ part_sum,
            const typename P::S* __restrict__ tw, double scale, double lam, FinArgs ahead,
            KgDev* before, KgDev* after, long long* phase_clk) {
    typedef typename P::S S;
    typedef typename P::R R;
    typedef cx<R> C;
    typedef PlaneShape<N> X;
    typedef Lay<N> Ly;
    namespace cgx = cooperative_groups;
    constexpr int CL = X::CL, T = X::T, CC = X::CC, NT = X::NT, LG = LayLg<P, N>::value;
    extern __shared__ __align__(16) unsigned char smraw[];
    S* slab = reinterpret_cast<S*>(smraw);   // [row][column slot]
    S* lines = slab + X::SLAB;               // [pair][PADN]
    __shared__ df dred[NT / 32];
    __shared__ unsigned kred[NT / 32];
    const int tid = threadIdx.x;
    const int rank = CL > 1 ? (int)(blockIdx.x % CL) : 0, z = (int)blockIdx.x / CL;
    // the row block or slab slot p of CTA r of the cluster
    auto at = [&](S* p, int r) -> S* {
        if constexpr (CL > 1) return cgx::this_cluster().map_shared_rank(p, (unsigned)r);
        else return p;
    };
    auto stamp = [&](int i) {
        if (phase_clk && blockIdx.x == 0 && tid == 0) phase_clk[i] = clock64();
    };

    // y transforms: thread j of the column in slot c; x transforms: thread jp of the pair of x-lines
    // in row block p
    const int c = tid % CC, j = tid / CC;
    const int p = tid / T, jp = tid % T;
    const int kx = rank * X::CW + c;
    const bool valid = c < (rank == CL - 1 ? X::CW + 1 : X::CW);
    S* __restrict__ col = W + (valid ? Ly::zcol(0, kx, LG) + ((size_t)z << LG) : 0);
    const size_t cs = Ly::ky_stride(LG);
    const C zero = cmake<R>(P::from_f64(0.0), P::from_f64(0.0));
    S* L1 = lines + p * X::PADN;   // the pair's rows; also its exchange space

    if (CL > 1) asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
    for (int i = X::PAIRS * X::PADN + tid; i < X::LINES; i += NT) lines[i] = P::pack(zero);   // idle row blocks
    tw = stage_table_any(tw, lines + X::LINES, N);   // first touches of the table would wait in every stage
    pdl_wait();
    stamp(0);
    const bool want_sum = ahead.kind != FIN_NONE || kg_recording(dev);
    const R rlam = P::from_f64(lam);
    Stats<P> st;
    st.init();

    C v[8];
#pragma unroll
    for (int s = 0; s < 8; s++) v[s] = valid ? P::load(col[(j + T * s) * cs]) : zero;
    // inverse y, inverse x, forward x, forward y through one copy of the transform's code: a kernel
    // of a few microseconds waits for its instructions too (three copies made a step 12.4, 14.8 and
    // 20.0 us at 16, 32 and 64^3, one 13.1, 14.3 and 19.1; recording 22, 26.3 and 32 against 22, 24.7
    // and 29.3)
#pragma unroll 1
    for (int ph = 0; ph < 4; ph++) {
        const bool xph = ph == 1 || ph == 2;
        PlaneSmem<P> sm{xph ? L1 : slab + c, xph ? 1 : CC, xph ? 1 : 0};
        fft<P, N, PlaneSmem<P>, false, false, false>(v, xph ? jp : j, tw, 1, sm, ph < 2 ? +1 : -1);
        if (ph == 0) {
            if (CL > 1) asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");   // every CTA has started
            if (valid) {
#pragma unroll
                for (int s = 0; s < 8; s++) {
                    const int row = j + T * s, lr = row % X::RPC;
                    *at(lines + (lr >> 1) * X::PADN + (lr & 1) * X::LDX + kx, row / X::RPC) = P::pack(v[s]);
                }
            }
            plane_barrier<CL>();
            stamp(1);
            x_pair_load<P, N>(L1, L1 + X::LDX, jp, v);
            __syncthreads();   // the rows are read; the transform exchanges there
        } else if (ph == 1) {
#pragma unroll
            for (int s = 0; s < 8; s++) {
                v[s].re = P::scale2(v[s].re, scale);   // u1, u2 at x = jp + T s; scale = 1/N^3
                v[s].im = P::scale2(v[s].im, scale);
                st.take2(v[s], want_sum);
            }
#pragma unroll
            for (int s = 0; s < 8; s++) {
                v[s].re = P::cube(v[s].re, rlam);
                v[s].im = P::cube(v[s].im, rlam);
            }
        } else if (ph == 2) {
#pragma unroll
            for (int s = 0; s < 8; s++) sm.put(jp + T * s, v[s]);
            sm.sync();
            const int row = rank * X::RPC + 2 * p;
#pragma unroll
            for (int s = 0; s < 8; s++) {
                const int k = jp + T * s;
                if (k <= N / 2 && p < X::PAIRS) {
                    const C Z = v[s];
                    const C Zm = conj(sm.get((N - k) & (N - 1)));
                    const C A = P::cadd(Z, Zm), B = P::csub(Z, Zm);      // 2 X1, 2 i X2
                    const int r = k / X::CW < CL - 1 ? k / X::CW : CL - 1;
                    S* dst = slab + row * CC + (k - r * X::CW);
                    *at(dst, r) = P::pack(P::cscale2(A, 0.5));
                    *at(dst + CC, r) = P::pack(P::cscale2(P::cmul_negi(B), 0.5));
                }
            }
            const unsigned key = __reduce_max_sync(0xffffffffu, st.fkey());
            if ((tid & 31) == 0) kred[tid >> 5] = key;
            if (want_sum) {
                df t = st.total_df();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    t = df_add_lazy(t, df_make(__shfl_down_sync(0xffffffffu, t.hi, o), __shfl_down_sync(0xffffffffu, t.lo, o)));
                if ((tid & 31) == 0) dred[tid >> 5] = t;
            }
            plane_barrier<CL>();   // no store into another CTA after this one
            stamp(2);
            // max |u| into the run state, where the z pass reads it before it updates
            if (tid == 0) {
                if (want_sum) {
                    df t = dred[0];
                    for (int w = 1; w < NT / 32; w++) t = df_add_lazy(t, dred[w]);
                    part_sum[blockIdx.x] = f2d_int(t.hi) + f2d_int(t.lo);
                }
                unsigned k = kred[0];
                for (int w = 1; w < NT / 32; w++) k = kred[w] > k ? kred[w] : k;
                atomicMax(&dev->xkey, (unsigned long long)__double_as_longlong(f2d_int(__uint_as_float(k))));
            }
#pragma unroll
            for (int s = 0; s < 8; s++) v[s] = valid ? P::load(slab[(j + T * s) * CC + c]) : zero;
            __syncthreads();   // the slab is the columns' exchange space
        }
    }
    if (valid) {
#pragma unroll
        for (int s = 0; s < 8; s++) col[(j + T * s) * cs] = P::pack(v[s]);
    }
    stamp(3);

    if (ahead.kind != FIN_NONE) {
        __shared__ int last;
        if (tid == 0) {
            __threadfence();   // the partial and the maximum are visible before the ticket
            last = atomicAdd(&dev->ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (last && tid < 32) {
            __threadfence();
            const double P = warp_total(part_sum, ahead.count);
            if (tid == 0) {
                KgDev run = *dev;
                run.xkey = __ldcg(&dev->xkey);
                run.ticket = 0u;
                *before = run;
                state_after_x(&run, true, true, __longlong_as_double((long long)run.xkey), ahead.norm * P);
                run.xkey = 0ull;
                *after = run;
                *dev = run;
            }
        }
    }
}

}  // namespace kg
