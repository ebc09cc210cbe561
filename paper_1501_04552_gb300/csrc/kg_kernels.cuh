// kg_kernels.cuh -- kernel templates of the step passes, the set-up and the read-out.
#pragma once
#include <type_traits>
#include "kg_fft.cuh"
#include "kg_launch.h"

namespace kg {

// ---------------------------------------------------------------------------
// Pass X.  MODE_STEP: C2R along x, stats, F = lam u^3, R2C along x, in place.
//          MODE_PEEK: C2R along x and stats only (W untouched).
// One line = N/2+1 complex values; T = N/16 threads per line.
// ---------------------------------------------------------------------------
constexpr int kXThreads = 256;

// threads per CTA of the stepping x pass: 256, and below 128^3 few enough that the grid still
// spreads over the SMs (a 32^3 pass is 2048 threads: with 64 CTAs of 32 in place of 8 of 256
// the whole double-float step went from 20.4 to 18.9 us; 16^3 20.9 to 18.0, 64^3 22.6 to 21.2)
template <int N>
struct XStep {
    static constexpr int NT = N >= 128 ? kXThreads : N >= 64 ? 64 : 32;
};

template <int N, int NT = kXThreads>
struct XShape {
    static constexpr int M = N / 2;
    static constexpr int T = M / 8;
    static constexpr int LPC = NT / T;                  // lines per CTA
    static constexpr int PADM = M + M / 8 + (N == 16);  // padded smem slots per line (even: a line lands in 16-byte copies)
    static_assert(T <= 32, "one line must fit in a warp");
};

// LIN: a pointer to the line's N/2+1 values, or any type whose operator[] yields them
// (the cluster-fused pass reads lines spread over the shared memory of several CTAs)
template <class P, int N, class LIN = const typename P::S*>
__device__ __forceinline__ void x_load_c2r(LIN line, int j, const typename P::S* __restrict__ tw,
                                           cx<typename P::R> (&v)[8]) {
    typedef typename P::R R;
    typedef cx<R> C;
    constexpr int M = N / 2, T = XShape<N>::T;
    constexpr bool kPow = sizeof(R) == 4;   // FP32: twiddles by products (L1TEX-bound pass)
    C wr[8];
    if constexpr (kPow) twiddle_run<P>(tw, j, T, +1, wr);
#pragma unroll
    for (int s = 0; s < 8; s++) {
        const int k = j + T * s;
        C X = P::load(line[k]);
        C Xp = P::load(line[M - k]);       // k = 0 pairs with the Nyquist entry k = M
        if (k == 0) {                      // real parts only at kx = 0 and kx = N/2
            X.im = P::from_f64(0.0);
            Xp.im = P::from_f64(0.0);
        }
        C A = P::cadd(X, conj(Xp));
        C B = P::csub(X, conj(Xp));
        C Bw;                                                // B exp(+2 pi i k / N)
        if constexpr (kPow) Bw = P::ctw(B, wr[s]);
        else Bw = P::ctw(B, twiddle<P>(tw, k, +1));
        v[s] = P::cnorm(P::cadd(A, mul_i(Bw)));
    }
}

// One x-line (T = N/16 threads, thread j): C2R, scale, stats, and in MODE_STEP the
// cube, R2C and write-back.  The line is read from Lin (global memory, or the line's
// landing slot in shared memory, which may be lsm's own storage) and written to L
// (pointers, or element accessors as for x_load_c2r; every read precedes every write).
template <class P, int N, int MODE, class LIN = const typename P::S*, class LOUT = typename P::S* __restrict__,
          bool RF = false>
__device__ __forceinline__ void x_line_body(LIN Lin, LOUT L, int j,
                                            LineSmem<P>& lsm, const typename P::S* __restrict__ tw, double scale,
                                            typename P::R rlam, bool want_sum, Stats<P>& st) {
    typedef typename P::R R;
    typedef cx<R> C;
    constexpr int M = N / 2, T = XShape<N>::T;
    C v[8];
    x_load_c2r<P, N, LIN>(Lin, j, tw, v);
    lsm.sync();   // every lane has read Lin before the first exchange writes lsm
    // inverse transform, then (stepping pass) the forward one, through one copy of the code
#pragma unroll 1
    for (int dir = 0; dir < (MODE == MODE_STEP ? 2 : 1); dir++) {
        // the FP32 x pass is bound by the L1TEX pipe: twiddle powers by products there
        fft<P, M, LineSmem<P>, sizeof(typename P::R) == 4, RF>(v, j, tw, 2, lsm, dir == 0 ? +1 : -1);
        if (dir == 0) {
#pragma unroll
            for (int s = 0; s < 8; s++) {
                v[s].re = P::scale2(v[s].re, scale);   // scale = 1/N^3, a power of two
                v[s].im = P::scale2(v[s].im, scale);
                st.take(v[s].re, want_sum);
                st.take(v[s].im, want_sum);
            }
            if (MODE == MODE_STEP) {
#pragma unroll
                for (int s = 0; s < 8; s++) {
                    v[s].re = rlam * (v[s].re * v[s].re * v[s].re);
                    v[s].im = rlam * (v[s].im * v[s].im * v[s].im);
                }
            }
        }
    }
    if (MODE == MODE_STEP) {
        // real-to-complex post-processing: X[k] = (Z_k + conj Z_{M-k})/2 - i W^k (Z_k - conj Z_{M-k})/2
#pragma unroll
        for (int s = 0; s < 8; s++) lsm.put(j + T * s, v[s]);
        lsm.sync();
        const double half = 0.5;
        constexpr bool kPow = sizeof(R) == 4;
        C wf[8];
        if constexpr (kPow) twiddle_run<P>(tw, j, T, -1, wf);
#pragma unroll
        for (int s = 0; s < 8; s++) {
            const int k = j + T * s;
            C Z = v[s];
            C Zp = lsm.get((M - k) & (M - 1));
            C A = P::cadd(Z, conj(Zp));
            C B = P::csub(Z, conj(Zp));
            C D;                                                // i B exp(-2 pi i k / N)
            if constexpr (kPow) D = mul_i(P::ctw(B, wf[s]));
            else D = mul_i(P::ctw(B, twiddle<P>(tw, k, -1)));
            C out = P::cnorm(P::csub(A, D));
            out.re = P::scale2(out.re, half);
            out.im = P::scale2(out.im, half);
            L[k] = P::pack(out);
            if (k == 0) L[M] = P::pack(cmake<R>(Z.re - Z.im, P::from_f64(0.0)));
        }
        lsm.sync();
    }
}

// Two x-lines of a real field through one N-point complex transform.  Over the Hermitian
// extensions of both half spectra (real parts only at kx = 0 and N/2, the C2R rule),
// Z[k] = X1[k] + i X2[k] has the inverse transform u1 + i u2; after the cube, the forward
// transform of F1 + i F2 splits again as
//     X1[k] = (Z[k] + conj Z[N-k]) / 2,    X2[k] = -i (Z[k] - conj Z[N-k]) / 2,
// which needs no twiddle product (the one-line form packs each line into an N/2-point
// transform with a twiddle product per point on the way in and on the way out).
template <int N, int NT = kXThreads>
struct XpShape {
    static constexpr int T = N / 8;              // threads per line pair
    static constexpr int PPC = NT / T;           // pairs per CTA
    static constexpr int PADN = N + N / 8;       // padded exchange slots per pair
    static constexpr bool CTA_SYNC = T > 32;     // a pair spans more than one warp
    static_assert(2 * PPC == XShape<N, NT>::LPC && PPC * PADN <= XShape<N, NT>::LPC * XShape<N, NT>::PADM,
                  "same lines per CTA as the one-line form, within its shared memory");
    static_assert(!CTA_SYNC || PPC <= 15, "one named barrier per pair");
};

// v[s] = X1[k] + i X2[k], k = j + T s, from the half spectra L1, L2 of two x-lines
// (Hermitian extension; the kx = 0 and N/2 entries contribute their real parts).  No const
// __restrict__ pointers: the ensemble's lines are written again within the launch.
template <class P, int N>
__device__ __forceinline__ void x_pair_load(const typename P::S* L1, const typename P::S* L2, int j,
                                            cx<typename P::R> (&v)[8]) {
    typedef typename P::R R;
    typedef cx<R> C;
    constexpr int T = N / 8;
    const R zero = P::from_f64(0.0);
#pragma unroll
    for (int s = 0; s < 8; s++) {
        const int k = j + T * s;
        const int kk = k <= N / 2 ? k : N - k;
        C X1 = P::load(L1[kk]), X2 = P::load(L2[kk]);
        if (kk == 0 || kk == N / 2) {      // real parts only
            X1.im = zero;
            X2.im = zero;
        }
        if (k > N / 2) {                    // Hermitian extension
            X1 = conj(X1);
            X2 = conj(X2);
        }
        // X1 + i X2, left unnormalised: the transform's first stage takes lazy sums of it
        v[s] = P::cadd_i(X1, X2);
    }
}

// the half spectra of two real lines from Z = FFT(x1 + i x2) held as v[s] = Z[j + T s]:
// X1 = (Z + conj Zm) / 2, X2 = -i (Z - conj Zm) / 2, Zm the mirrored entry
template <class P, int N, class SM>
__device__ __forceinline__ void x_pair_unpack(typename P::S* __restrict__ L1, typename P::S* __restrict__ L2, int j,
                                              SM& lsm, const cx<typename P::R> (&v)[8]) {
    typedef typename P::R R;
    typedef cx<R> C;
    constexpr int T = N / 8;
#pragma unroll
    for (int s = 0; s < 8; s++) lsm.put(j + T * s, v[s]);
    lsm.sync();
#pragma unroll
    for (int s = 0; s < 8; s++) {
        const int k = j + T * s;
        if (k <= N / 2) {
            const C Z = v[s];
            const C Zm = conj(lsm.get((N - k) & (N - 1)));
            const C A = P::cadd(Z, Zm), B = P::csub(Z, Zm);      // 2 X1, 2 i X2
            // stored unnormalised: every reader of W starts with lazy sums or an exact
            // conversion of both words
            L1[k] = P::pack(P::cscale2(A, 0.5));
            L2[k] = P::pack(P::cscale2(P::cmul_negi(B), 0.5));
        }
    }
    lsm.sync();
}

template <class P, int N, int MODE, class SM, bool RF = false>
__device__ __forceinline__ void x_pair_body(typename P::S* __restrict__ L1, int j, SM& lsm,
                                            const typename P::S* __restrict__ tw, double scale, typename P::R rlam,
                                            bool want_sum, Stats<P>& st) {
    typedef typename P::R R;
    typedef cx<R> C;
    typename P::S* __restrict__ L2 = L1 + Lay<N>::PITCH;
    C v[8];
    x_pair_load<P, N>(L1, L2, j, v);
#pragma unroll 1
    for (int dir = 0; dir < (MODE == MODE_STEP ? 2 : 1); dir++) {
        // outputs left unnormalised: the statistics read the rounded sum of both words, the
        // cube and the unpacking take lazy products and sums
        fft<P, N, SM, false, RF, false>(v, j, tw, 1, lsm, dir == 0 ? +1 : -1);
        if (dir == 0) {
#pragma unroll
            for (int s = 0; s < 8; s++) {
                v[s].re = P::scale2(v[s].re, scale);   // u1, u2 at x = j + T s; scale = 1/N^3
                v[s].im = P::scale2(v[s].im, scale);
                st.take2(v[s], want_sum);
            }
            if (MODE == MODE_STEP) {
#pragma unroll
                for (int s = 0; s < 8; s++) {
                    v[s].re = P::cube(v[s].re, rlam);
                    v[s].im = P::cube(v[s].im, rlam);
                }
            }
        }
    }
    if (MODE == MODE_STEP) x_pair_unpack<P, N>(L1, L2, j, lsm, v);
}

// The double-float and FP64 passes take x-lines in pairs (x_pair_body): fewer
// arithmetic operations per point, which is what bounds them.
template <class P>
struct XPaired {
    static constexpr bool value = false;
};
template <>
struct XPaired<PrecDF> {
    static constexpr bool value = true;
};
template <>
struct XPaired<PrecF64> {
    static constexpr bool value = true;
};

// resident threads per SM the x pass is compiled for: the paired double-float body fits
// 1024 (64 registers and 8 to 20 bytes of spills; 1.61 -> 1.44 ms at 512^3 against 512 when it
// was measured); the pipelined
// FP32 body measured slower at 768 (0.48 -> 0.51 ms), and the FP64 body needs its registers.
// Below 128^3 the grid does not fill the SMs and every body keeps its registers.
template <class P, int N>
struct XMinBlocks {
    static constexpr int kThreads = std::is_same<P, PrecDF>::value ? 1024 : 512;
    static constexpr int value = N >= 128 ? kThreads / XStep<N>::NT : 1;
};

// How pass X walks W.  Pipelined (the FP32 pass, bound by latency and the L1TEX pipe): a
// persistent grid walks the batches, and while a CTA transforms one batch from shared
// memory the next one lands in the other half of a double buffer (cp.async).  Direct
// (the double-float and FP64 passes, bound by their arithmetic pipes, where the copy loop
// and the extra barriers cost more than they hide): one batch per CTA, loaded from global
// memory straight into registers.
template <class P>
struct XPipelined {
    static constexpr bool value = true;
};
template <>
struct XPipelined<PrecDF> {
    static constexpr bool value = false;
};
template <>
struct XPipelined<PrecF64> {
    static constexpr bool value = false;
};

// Pass X.  A batch is LPC consecutive x-lines of W1 (rows of PITCH values, 16-byte aligned, so
// a line lands in 16-byte copies: two FP32 values each); a landed batch serves as the lines'
// FFT exchange space.  Each CTA writes one max key and one Sigma u^4 partial when the step
// records or `record` is set (kg_energy's pass).
template <class P, int N, int MODE>
__global__ void __launch_bounds__(XStep<N>::NT, XMinBlocks<P, N>::value)
    k_pass_x(typename P::S* __restrict__ W, KgDev* __restrict__ dev, double* __restrict__ part_sum,
             double* __restrict__ part_max, const typename P::S* __restrict__ tw, double scale, double lam, int record) {
    typedef typename P::S S;
    constexpr int NT = XStep<N>::NT;
    typedef XShape<N, NT> X;
    constexpr int T = X::T, NH = N / 2 + 1, LPC = X::LPC, PADM = X::PADM, PITCH = Lay<N>::PITCH;
    constexpr int NB = N * N / LPC;     // batches
    constexpr int VPC = 16 / (int)sizeof(S);              // values per 16-byte copy
    constexpr int CPL = (NH + VPC - 1) / VPC;             // copies per line (the last may bring one slot of padding)
    static_assert(PADM >= CPL * VPC && PADM % VPC == 0 && PITCH >= CPL * VPC, "a line lands in its exchange slot");
    extern __shared__ __align__(16) unsigned char smraw[];
    S* buf = reinterpret_cast<S*>(smraw);   // (2 when pipelined) x LPC x PADM values
    __shared__ double red[96];

    const int li = threadIdx.x / T, j = threadIdx.x % T;
    pdl_wait();
    const bool want_sum = (MODE == MODE_PEEK) || record || kg_recording(dev);
    const typename P::R rlam = P::from_f64(lam);
    Stats<P> st;
    st.init();

    if constexpr (!XPipelined<P>::value && XPaired<P>::value) {
        typedef XpShape<N, NT> XP;
        const int pi = threadIdx.x / XP::T, jp = threadIdx.x % XP::T;
        const size_t pair = (size_t)blockIdx.x * XP::PPC + pi;
        LineSmemX<P, XP::CTA_SYNC> lsm{buf + pi * XP::PADN, 1u + (unsigned)pi, (unsigned)XP::T};
        x_pair_body<P, N, MODE>(W + 2 * pair * PITCH, jp, lsm, tw, scale, rlam, want_sum, st);
    } else if constexpr (!XPipelined<P>::value) {
        const size_t line = (size_t)blockIdx.x * LPC + li;
        LineSmem<P> lsm{buf + li * PADM};
        x_line_body<P, N, MODE>(W + line * PITCH, W + line * PITCH, j, lsm, tw, scale, rlam, want_sum, st);
    } else {
        auto issue = [&](int batch, S* dst) {
            const S* src = W + (size_t)batch * LPC * PITCH;
            for (int e = threadIdx.x; e < LPC * CPL; e += NT) {
                const int l = e / CPL, k = (e - l * CPL) * VPC;
                cp_async16(dst + l * PADM + k, src + l * PITCH + k);
            }
        };
        int b = blockIdx.x;
        if (b < NB) issue(b, buf);
        cp_async_commit();
        for (int it = 0; b < NB; b += gridDim.x, ++it) {
            S* cur = buf + (it & 1) * (LPC * PADM);
            if (b + (int)gridDim.x < NB) issue(b + gridDim.x, buf + ((it + 1) & 1) * (LPC * PADM));
            cp_async_commit();
            cp_async_wait_1();
            __syncthreads();
            LineSmem<P> lsm{cur + li * PADM};
            x_line_body<P, N, MODE>(cur + li * PADM, W + ((size_t)b * LPC + li) * PITCH, j, lsm, tw, scale, rlam, want_sum,
                                    st);
            __syncthreads();   // the buffer is the target of the copy issued next iteration
        }
        cp_async_wait_all();
    }

    // the max every step (integer keys), the compensated FP64 sum only when it is wanted
    block_max_to<NT>(st, part_max + blockIdx.x);
    if (want_sum) {
        if constexpr (XPaired<P>::value && !std::is_same<P, PrecF64>::value) {
            __shared__ df dred[NT / 32];
            const df t = block_sum_df<NT>(st.total_df(), dred);
            if (threadIdx.x == 0) part_sum[blockIdx.x] = f2d_int(t.hi) + f2d_int(t.lo);
        } else {
            NSum acc;
            acc.s = st.total();
            acc.c = 0.0;
            double unused = 0.0;
            block_reduce<NT>(acc, unused, red);
            if (threadIdx.x == 0) part_sum[blockIdx.x] = acc.value();
        }
    }
}

// ---------------------------------------------------------------------------
// Finalisers: reduce the partials of a pass and advance the run state.  Those of a step run in
// one more CTA of the y pass that follows (FIN_X in the forward, FIN_Z in the inverse one, both
// before the next reader of the state starts).  As kernels of one CTA, and without programmatic
// dependent launch, they made a double-float step 33 us at 32^3 and 72 us at 64^3 recording
// every level; so 18.9 and 34 us (13.0 and 28.5 with k_plane, whose finalisers ride in the z pass).
// ---------------------------------------------------------------------------
constexpr int kFinThreads = 1024;
constexpr int kFinSmem = 128;   // doubles of shared memory a finaliser needs

// compensated sums of the first 2 from lanes of a warp -> lane 0
__device__ __forceinline__ void warp_merge(NSum& v, int from = 16, unsigned mask = 0xffffffffu) {
    for (int o = from; o > 0; o >>= 1) {
        NSum b;
        b.s = __shfl_down_sync(mask, v.s, o);
        b.c = __shfl_down_sync(mask, v.c, o);
        nsum_merge(v, b);
    }
}

// the sum of count partials by one warp -> lane 0
__device__ __forceinline__ double warp_total(const double* part, int count) {
    NSum acc;
    acc.s = acc.c = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x & 31; i < count; i += 32) acc.add(__ldcg(part + i));
    warp_merge(acc);
    return acc.value();
}

// v of the first `count` threads of an NT-thread CTA (of all of them when it has fewer) -> thread 0.
// The SM makes two FP64 operations a clock, so the warps that hold nothing stay out (a step with its
// energy read at 64^3: 72 -> 57 us).
template <int NT>
__device__ __forceinline__ void block_sum_of(NSum& v, int count, double* sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int NW = (NT + 31) / 32;   // grids of 16^3 have CTAs of half a warp
    const int nw = count >= NT ? NW : (count + 31) / 32;
    if (w < nw) warp_merge(v, NT >= 32 ? 16 : NT / 2, NT >= 32 ? 0xffffffffu : (1u << (NT & 31)) - 1u);
    if (nw > 1) {
        __syncthreads();
        if (lane == 0 && w < nw) {
            sh[w] = v.s;
            sh[32 + w] = v.c;
        }
        __syncthreads();
        if (w == 0) {
            v.s = lane < nw ? sh[lane] : 0.0;
            v.c = lane < nw ? sh[32 + lane] : 0.0;
            warp_merge(v, nw > 16 ? 16 : nw > 8 ? 8 : nw > 4 ? 4 : nw > 2 ? 2 : 1);
        }
    }
}

// all NT threads of the CTA; red: kFinSmem doubles
template <int NT>
__device__ __forceinline__ void fin_reduce(const double* part_sum, const double* part_max, int count, NSum& acc,
                                           double& mx, double* red) {
    acc.s = 0.0;
    acc.c = 0.0;
    unsigned long long key = 0ull;
    for (int i = threadIdx.x; i < count; i += NT) {
        if (part_sum) acc.add(part_sum[i]);
        if (part_max) {
            const unsigned long long k = (unsigned long long)__double_as_longlong(part_max[i]);
            key = k > key ? k : key;
        }
    }
    if (part_max) key = block_max_key<NT>(key, reinterpret_cast<unsigned long long*>(red + 96));
    mx = __longlong_as_double((long long)key);
    if (part_sum) block_sum_of<NT>(acc, count, red);
}

// the run state after the x pass of a step, whose largest |u| is mx and whose P^l (when rec) is P;
// ahead: the next step's x pass, run by kg_energy; its max |u| waits in maxabs_peek until that step
// runs (kg_status reports the last step's)
__device__ __forceinline__ void state_after_x(KgDev* dev, bool ahead, bool rec, double mx, double P) {
    if (ahead && dev->frozen) dev->maxabs_peek = dev->maxabs_last;
    // the composed scheme checks the field at integer times only (its first substep)
    if (dev->sub == 0 && !dev->frozen) {
        if (ahead) dev->maxabs_peek = mx;
        else dev->maxabs_last = mx;
        if (rec) {
            dev->P_last = P;
            dev->P_last_level = dev->level;
        }
        if (dev->threshold > 0.0 && !(mx <= dev->threshold)) {
            dev->frozen = 1;
            dev->blowup_level = dev->level;
        }
    }
}

// the run state after the update: Q^{l+1/2} (when rec) and the level advance
__device__ __forceinline__ void state_after_z(KgDev* dev, bool rec, double Q) {
    if (dev->frozen) return;
    if (rec) {
        dev->Q_last = Q;
        dev->Q_last_level = dev->level;
    }
    if (dev->scheme == 0) {
        dev->level += 1;
        dev->phase ^= 1;
    } else {   // composed scheme: the state arrays stay put; a step is three substeps
        dev->sub = dev->sub == 2 ? 0 : dev->sub + 1;
        if (dev->sub == 0) dev->level += 1;
    }
}

template <int NT>
__device__ __noinline__ void finalise(const FinArgs f, double* red) {
    KgDev* dev = f.dev;
    NSum acc;
    double mx;
    // Whether the level records decides which threads reach the barriers of the reductions, and thread 0
    // advances the level in the last branch: every thread reads the decision here, once, and a barrier
    // stands between this and the advance, so that a warp which comes late takes the branch of the
    // others.  (A barrier right here would do as well, but hold back the loads of the partials: 180
    // FP32 steps at 16^3, with set-up and read-out, took 2572 us against 2453 without it.)
    const bool recording = kg_recording(dev);
    if (f.kind == FIN_X || f.kind == FIN_X_AHEAD) {
        // after a stepping x pass: blow-up check and P^l; norm = lam h^3 / 4
        const bool ahead = f.kind == FIN_X_AHEAD;
        const bool rec = recording || ahead;
        fin_reduce<NT>(rec ? f.part_sum : nullptr, f.part_max, f.count, acc, mx, red);
        if (dev->complex_field) mx = sqrt(mx);   // the keys were |u|^2
        if (threadIdx.x == 0) state_after_x(dev, ahead, rec, mx, rec ? f.norm * acc.value() : 0.0);
    } else if (f.kind == FIN_AHEAD_DONE) {
        // the step whose x pass ran ahead: its max |u| becomes the last step's
        if (threadIdx.x == 0) dev->maxabs_last = dev->maxabs_peek;
    } else if (f.kind == FIN_PEEK) {
        fin_reduce<NT>(f.part_sum, f.part_max, f.count, acc, mx, red);
        if (dev->complex_field) mx = sqrt(mx);
        if (threadIdx.x == 0) {
            dev->P_peek = f.norm * acc.value();
            dev->maxabs_peek = mx;
        }
    } else {
        // after the update; norm = h^3/N^3
        if (recording) fin_reduce<NT>(f.part_sum, nullptr, f.count, acc, mx, red);
        __syncthreads();
        if (threadIdx.x == 0) state_after_z(dev, recording, recording ? f.norm * acc.value() : 0.0);
    }
}

// ---------------------------------------------------------------------------
// Column FFT: C consecutive kx columns of one plane, all N rows (layouts: struct Lay).
// COL_YF: plane z, x-lines -> z-columns; COL_YI: plane z, z-columns -> x-lines;
// COL_Z: plane ky, z-columns, in place or between storage formats (set-up / read-out).
// ---------------------------------------------------------------------------
enum { COL_YF = 0, COL_YI = 1, COL_Z = 2 };

template <class P>
struct ColShape {
    static constexpr int C = 128 / (int)sizeof(typename P::S);
};
// Column tiles of the y passes (and the FP64 z columns): 128-byte rows, except the FP32 ones
// (64-byte rows: twice the CTAs for the same occupancy, and the width of a row of z-columns) and
// the double-float ones at 512^3 (four CTAs of 256 threads per SM instead of two of 512 wait less
// at barriers: 0.509 and 0.543 ms against 0.543 and 0.584; at 256^3 0.065 and 0.068 against 0.064
// and 0.064)
template <class P, int N, bool YPASS>
struct ColStep {
    static constexpr bool kNarrow = YPASS && (sizeof(typename P::S) == 8 || (std::is_same<P, PrecDF>::value && N >= 512));
    static constexpr int C = (kNarrow ? 64 : 128) / (int)sizeof(typename P::S);
};

// where column kx of a plane starts in a source (DST == false) or destination array, and
// the distance of its rows
template <int N, int DIR, bool CPLX, bool DST>
struct ColAddr {
    typedef Lay<N, CPLX> Ly;
    static constexpr bool kLines = DST ? DIR == COL_YI : DIR == COL_YF;   // x-lines
    static __device__ __forceinline__ size_t stride(int lg) {
        return DIR == COL_Z ? (size_t)1 << lg : kLines ? (size_t)Ly::PITCH : Ly::ky_stride(lg);
    }
    static __device__ __forceinline__ size_t base(int plane, int kx, int lg) {
        if (DIR == COL_Z) return Ly::zcol(plane, kx, lg);
        return kLines ? (size_t)plane * N * Ly::PITCH + kx : Ly::zcol(0, kx, lg) + ((size_t)plane << lg);
    }
};

// the layout a kernel of precision P works in: its own, or for FP64 the context's
template <class P, int N>
__device__ __forceinline__ int lay_lg(int lg) {
    return std::is_same<P, PrecF64>::value ? lg : LayLg<P, N>::value;
}

// one column (T = N/8 threads, thread j) of a tile; valid == false for the columns
// of the last tile beyond the plane (they compute on zeros and store nothing)
template <class Pin, class P, class Pout, int N, int SIGN, int DIR, bool CPLX, class SM, bool RF = false>
__device__ __forceinline__ void col_body(const typename Pin::S* src, typename Pout::S* dst, int plane, int kx,
                                         bool valid, int j, SM& csm, const typename P::S* __restrict__ tw, int lg) {
    typedef typename P::R R;
    typedef ColAddr<N, DIR, CPLX, false> In;
    typedef ColAddr<N, DIR, CPLX, true> Out;
    constexpr int T = N / 8;
    cx<R> v[8];
    {
        const typename Pin::S* s0 = src + In::base(plane, kx, lg);
        const size_t st = In::stride(lg);
#pragma unroll
        for (int s = 0; s < 8; s++) {
            if (valid) v[s] = Convert<Pin, P>::go(Pin::load(s0[(size_t)(j + T * s) * st]));
            else v[s] = cmake<R>(P::from_f64(0.0), P::from_f64(0.0));
        }
    }
    fft<P, N, SM, false, RF, false, false>(v, j, tw, 1, csm, SIGN);   // outputs go to W or FP64
    if (valid) {
        typename Pout::S* d0 = dst + Out::base(plane, kx, lg);
        const size_t st = Out::stride(lg);
#pragma unroll
        for (int s = 0; s < 8; s++) d0[(size_t)(j + T * s) * st] = Pout::pack(Convert<P, Pout>::go(v[s]));
    }
}

// resident threads per SM a column kernel is compiled for: 1024 (64 registers) for 16-byte
// values, 2048 (32) for FP32.  Left to itself ptxas took 74 for the double-float y passes, one
// CTA of 512 threads per SM: 0.74 against 0.55 ms at 512^3; the FP32 ones took 0.250 ms
// compiled for 1024 threads against 0.227.  Grids below 128^3 have too few CTAs to fill the
// SMs anyway and keep their registers.
template <class P, int NT, int N>
struct ColMinBlocks {
    static constexpr int kThreads = sizeof(typename P::S) == 8 ? 2048 : 1024;
    static constexpr int value = N >= 128 && kThreads / NT > 1 ? kThreads / NT : 1;
};

template <class Pin, class P, class Pout, int N, int SIGN, int DIR, bool CPLX, int CW>
__global__ void __launch_bounds__(CW * N / 8, ColMinBlocks<P, CW * N / 8, N>::value) k_col(const typename Pin::S* src, typename Pout::S* dst,
                                                    const typename P::S* __restrict__ tw, int lg, FinArgs fin) {
    constexpr int C = CW;
    extern __shared__ __align__(16) unsigned char smraw[];
    typename P::S* sm = reinterpret_cast<typename P::S*>(smraw);
    const int plane = (int)blockIdx.y - (fin.kind != FIN_NONE);   // a finaliser takes the first row of CTAs
    if (plane < 0) {
        pdl_wait();
        if (blockIdx.x == 0) finalise<CW * N / 8>(fin, reinterpret_cast<double*>(smraw));
        return;
    }
    const int c = threadIdx.x % C, j = threadIdx.x / C;
    const int kx = blockIdx.x * C + c;
    ColSmem<P, C> csm{sm, c};
    tw = stage_table(tw, sm + N * C, N);
    pdl_wait();
    col_body<Pin, P, Pout, N, SIGN, DIR, CPLX, ColSmem<P, C>>(src, dst, plane, kx, kx < Lay<N, CPLX>::NX, j, csm, tw,
                                                               lay_lg<P, N>(lg));
}

// inverse z column FFT from an FP64 spectral array into W2 (precision P); the source is
// src1 when dev != NULL and dev->phase == 1, src0 otherwise (the current level's array)
template <class P, int N, bool CPLX, int CW>
__global__ void __launch_bounds__(CW * N / 8, ColMinBlocks<P, CW * N / 8, N>::value) k_col_sel(const double2* src0, const double2* src1, const KgDev* dev,
                                                        typename P::S* dst, const typename P::S* __restrict__ tw,
                                                        int lg) {
    constexpr int C = CW;
    extern __shared__ __align__(16) unsigned char smraw[];
    typename P::S* sm = reinterpret_cast<typename P::S*>(smraw);
    pdl_wait();
    const double2* src = (dev != nullptr && dev->phase) ? src1 : src0;
    const int c = threadIdx.x % C, j = threadIdx.x / C;
    const int kx = blockIdx.x * C + c;
    ColSmem<P, C> csm{sm, c};
    tw = stage_table(tw, sm + N * C, N);
    col_body<PrecF64, P, P, N, +1, COL_Z, CPLX, ColSmem<P, C>>(src, dst, (int)blockIdx.y, kx, kx < Lay<N, CPLX>::NX, j,
                                                                  csm, tw, lay_lg<P, N>(lg));
}

// ---------------------------------------------------------------------------
// Fused z column of the batched ensemble: forward z FFT -> F^n, FP64 update, inverse z FFT,
// in one pass over W2.  coef[m2] = (2 c_k, 2 beta_k) for integer m2 = mx^2 + my^2 + mz^2.
// One (ky, kx) column (T = N/8 threads, thread j).
// cur and old change their roles every step of a launch, so cur is not read-only for the kernel's
// life, and it was last written by another SM: it is no const __restrict__ pointer, whose loads may
// take the path that nothing keeps coherent.
// ---------------------------------------------------------------------------
template <class P, int N, class SM, bool RF = false>
__device__ __forceinline__ void z_body(typename P::S* __restrict__ W, const double2* cur,
                                       double2* __restrict__ old, int kx, int ky, bool valid, int j,
                                       SM& csm, const typename P::S* __restrict__ tw,
                                       const double2* __restrict__ coef) {
    typedef typename P::R R;
    typedef cx<R> Cx;
    constexpr int T = N / 8, LG = LayLg<P, N>::value, RS = 1 << LG;
    const size_t base = Lay<N>::zcol(ky, kx, LG);

    Cx v[8];
#pragma unroll
    for (int s = 0; s < 8; s++) {
        if (valid) v[s] = P::load(W[base + (size_t)(j + T * s) * RS]);
        else v[s] = cmake<R>(P::from_f64(0.0), P::from_f64(0.0));
    }
    // forward z transform, the update, then the inverse z transform; the double-float and
    // FP64 bodies are large, so they run both transforms through one copy of the FFT code
    constexpr bool kShare = sizeof(typename P::S) == 16;
#pragma unroll(kShare ? 1 : 2)
    for (int dir = 0; dir < 2; dir++) {
        fft<P, N, SM, false, RF, false>(v, j, tw, 1, csm, dir == 0 ? -1 : +1);
        if (dir == 1) break;
        const int my = ky <= N / 2 ? ky : ky - N;
        const int mxy2 = kx * kx + my * my;
#pragma unroll
        for (int s = 0; s < 8; s++) {
            const int kz = j + T * s;
            const int mz = kz <= N / 2 ? kz : kz - N;
            const int m2 = mxy2 + mz * mz;
            if (valid) {
                const size_t idx = base + (size_t)kz * RS;
                const double2 cf = __ldg(coef + m2);
                const double2 a = cur[idx];
                const double2 b = old[idx];
                double nre = P::fma_into(cf.y, v[s].re, fma(cf.x, a.x, -b.x));
                double nim = P::fma_into(cf.y, v[s].im, fma(cf.x, a.y, -b.y));
                old[idx] = make_double2(nre, nim);
                v[s] = cmake<R>(P::from_f64(nre), P::from_f64(nim));
            }
        }
    }
    if (valid) {
#pragma unroll
        for (int s = 0; s < 8; s++) W[base + (size_t)(j + T * s) * RS] = P::pack(v[s]);
    }
}

// ---------------------------------------------------------------------------
// Time-stepping schemes of the per-mode update.
// SCHEME 0, Eq. (2): cur = uh^n, old = uh^{n-1};
//     uh^{n+1} = 2 c_k uh^n - uh^{n-1} + 2 beta_k F^n_k   written over old.
// SCHEME 1, the fourth-order composition (triple jump) of Eq. (2) in kick-drift-kick
// form: cur = a (= uh), old = P (velocity variable); substep s = dev->sub of a step
//     P <- P + K_s (F - omega^2 a),   a <- a + h_s P       (both written back)
// with the merged kick K_s = (h_{s-1}/2)/(1 + omega^2 h_{s-1}^2/4) + (h_s/2)/(1 + omega^2
// h_s^2/4) (h_{-1} = h_2 = h_0) and h = (g1, g2, g1) dt.  One F per substep; with one
// substep of length dt this is Eq. (2) itself.
// ---------------------------------------------------------------------------
// (the tables and substep lengths travel in C4Args, kg_launch.h)

// The per-mode update of one step (or substep) at mode index idx with integer norm m2, F the
// transform of the cube there in the pass precision; writes the state (unless frozen) and
// returns the new uh in FP64, the value the inverse transforms start from.  a = cur[idx], b = old[idx].
template <class P, int SCHEME>
__device__ __forceinline__ double2 mode_update(cx<typename P::R> f, double2* cur, double2* old, size_t idx, int m2,
                                               const double2* __restrict__ coef, const C4Args& c4, int sub,
                                               bool update, double2 a, double2 b) {
    if constexpr (SCHEME == 0) {
        const double2 cf = __ldg(coef + m2);
        const double nre = P::fma_into(cf.y, f.re, fma(cf.x, a.x, -b.x));
        const double nim = P::fma_into(cf.y, f.im, fma(cf.x, a.y, -b.y));
        if (update) old[idx] = make_double2(nre, nim);
        return make_double2(nre, nim);
    } else {
        const double2 kc = __ldg(c4.kick + (size_t)sub * c4.stride + m2);
        const double pre = P::fma_into(kc.x, f.re, fma(-kc.y, a.x, b.x));
        const double pim = P::fma_into(kc.x, f.im, fma(-kc.y, a.y, b.y));
        const double h = sub == 1 ? c4.h[1] : c4.h[0];   // h = (g1, g2, g1) dt
        const double2 n = make_double2(fma(h, pre, a.x), fma(h, pim, a.y));
        if (update) {
            old[idx] = make_double2(pre, pim);
            cur[idx] = n;
        }
        return n;
    }
}

// ---------------------------------------------------------------------------
// Streaming update between the forward and the inverse z FFT.  W holds F^n_k on entry
// and uh^{n+1}_k in the pass precision on exit; the state update and the Q terms are
// those of z_body.
// ---------------------------------------------------------------------------
// The mode in slot i of an array of z-columns (struct Lay, tiles of 2^lg columns): the half
// spectrum of a real field (kx = 0..N/2) or the full spectrum of a complex field (kx = 0..N-1 in FFT
// order).  m2 = mx^2 + my^2 + mz^2 indexes the coefficient tables; w is the Parseval weight of the
// mode in the energy sums; slots of padding hold no mode (valid == false).
template <int N, bool CPLX>
struct ModeIndex {
    typedef Lay<N, CPLX> Ly;
    static_assert(Ly::kSlots < (1ll << 31), "slot indexes fit 32 bits");
    int m2, kx, ky, kz;
    bool twice, valid;
    static __host__ __device__ __forceinline__ unsigned slots(int lg) { return (unsigned)N * (unsigned)Ly::ky_stride(lg); }
    __device__ __forceinline__ ModeIndex(unsigned i, int lg) {
        const unsigned row = i >> lg, tile = row / N, tl = (unsigned)Ly::tiles(lg);
        kz = (int)(row % N);
        ky = (int)(tile / tl);
        kx = (int)((tile - ky * tl) << lg) + (int)(i & ((1u << lg) - 1u));
        const int mx = (CPLX && kx > N / 2) ? kx - N : kx;
        const int my = ky <= N / 2 ? ky : ky - N, mz = kz <= N / 2 ? kz : kz - N;
        m2 = mx * mx + my * my + mz * mz;
        twice = !CPLX && kx != 0 && kx != N / 2;
        valid = kx < Ly::NX;
    }
};

constexpr int kUpdThreads = 256;

// One term of Q^{n+1/2} without its constant factor 1/(2 dt^2):
//     w_k ( |a1 - a0|^2 + r_k |a1 + a0|^2 ),   r_k = qr omega_k^2,  qr = dt^2 / 4,
// (the Q definition of kg.h multiplied by 2 dt^2).  Only the cancelling differences
// a1 - a0 are formed in FP64; the sums a1 + a0, r_k, the squares and their sums are
// formed in double-float on the FP32 pipe (the FP64 pipe already carries the update),
// except for the IEEE FP64 passes, which stay in FP64.
template <class P>
struct QTerm {
    typedef df T;
    static __device__ __forceinline__ T zero() { return df_make(0.f, 0.f); }
    // the cancelling differences in FP64, then squares and sums in double-float left
    // unnormalised: D, S and r S are sums of non-negative terms (n + a adds two values of
    // the same mode), so an unnormalised pair still holds each to within u^2 of its size,
    // and value() converts both words exactly
    static __device__ __forceinline__ T term(double n_re, double n_im, double2 a, double w2, double qr, bool twice) {
        const df dre = d2df_int(n_re - a.x), dim = d2df_int(n_im - a.y);
        const df sre = df_add_lazy(d2df_int(n_re), d2df_int(a.x)), sim = df_add_lazy(d2df_int(n_im), d2df_int(a.y));
        const df D = df_add_lazy(df_mul_lazy(dre, dre), df_mul_lazy(dim, dim));
        const df S = df_add_lazy(df_mul_lazy(sre, sre), df_mul_lazy(sim, sim));
        const df t = df_add_lazy(D, df_mul_lazy(df_mul_lazy(d2df_int(w2), d2df_int(qr)), S));
        return twice ? df_scale2(t, 2.0f) : t;
    }
    static __device__ __forceinline__ T add(T x, T y) { return df_add_lazy(x, y); }
    static __device__ __forceinline__ T shfl_down(T x, int o) {
        return df_make(__shfl_down_sync(0xffffffffu, x.hi, o), __shfl_down_sync(0xffffffffu, x.lo, o));
    }
    static __device__ __forceinline__ double value(T x) { return f2d_int(x.hi) + f2d_int(x.lo); }
};
template <>
struct QTerm<PrecF64> {
    typedef double T;
    static __device__ __forceinline__ T zero() { return 0.0; }
    static __device__ __forceinline__ T term(double n_re, double n_im, double2 a, double w2, double qr, bool twice) {
        const double r = qr * w2;
        const double dre = n_re - a.x, dim = n_im - a.y, sre = n_re + a.x, sim = n_im + a.y;
        const double t = fma(r, fma(sre, sre, sim * sim), fma(dre, dre, dim * dim));
        return twice ? t + t : t;
    }
    static __device__ __forceinline__ T add(T x, T y) { return x + y; }
    static __device__ __forceinline__ T shfl_down(T x, int o) { return __shfl_down_sync(0xffffffffu, x, o); }
    static __device__ __forceinline__ double value(T x) { return x; }
};

// pairwise (tree) sum of one value per thread of an NT-thread CTA; the total lands in
// thread 0
template <class Q, int NT>
__device__ __forceinline__ typename Q::T block_tree_sum(typename Q::T v, typename Q::T* sm) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = Q::add(v, Q::shfl_down(v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sm[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < NT / 32 ? sm[l] : Q::zero();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = Q::add(v, Q::shfl_down(v, o));
    }
    return v;
}

// Streaming per-mode update of Eq. (2) between the forward and the inverse z column
// passes, one mode per thread (a full grid keeps enough loads in flight to stream at
// HBM rate and lets the FP64 update overlap them):
//     uh^{n+1} = 2 c_k uh^n - uh^{n-1} + 2 beta_k F^n_k        (FP64, over uh^{n-1})
// and W <- uh^{n+1} in the pass precision for the inverse transforms.  On recording
// steps each CTA also writes its partial sum of the Q terms (QTerm) times qc = 1/(2 dt^2).
template <class P, int N, bool CPLX = false, int SCHEME = 0>
__global__ void __launch_bounds__(kUpdThreads, 6) k_update(typename P::S* __restrict__ W, double2* S0, double2* S1,
                                                          KgDev* __restrict__ dev, double* __restrict__ part_sum,
                                                          const double2* __restrict__ coef,
                                                          const double* __restrict__ w2tab, double qr, double qc,
                                                          C4Args c4) {
    typedef typename P::R R;
    typedef QTerm<P> Q;
    typedef ModeIndex<N, CPLX> MI;
    __shared__ typename Q::T red[kUpdThreads / 32];
    pdl_wait();
    const bool want_q = SCHEME == 0 && kg_recording(dev);
    const bool update = dev->frozen == 0;
    double2* __restrict__ cur = dev->phase ? S1 : S0;
    double2* __restrict__ old = dev->phase ? S0 : S1;
    const unsigned i = blockIdx.x * kUpdThreads + threadIdx.x;
    typename Q::T q = Q::zero();
    const MI mi(i, LayLg<P, N>::value);
    if (i < MI::slots(LayLg<P, N>::value) && mi.valid) {
        const cx<R> f = P::load(W[i]);
        const double2 a = cur[i];
        const double2 n = mode_update<P, SCHEME>(f, cur, old, i, mi.m2, coef, c4, dev->sub, update, a, old[i]);
        W[i] = P::pack(cmake<R>(P::from_f64(n.x), P::from_f64(n.y)));
        if (want_q) q = Q::term(n.x, n.y, a, __ldg(w2tab + mi.m2), qr, mi.twice);
    }
    if (want_q) {
        q = block_tree_sum<Q, kUpdThreads>(q, red);
        if (threadIdx.x == 0) part_sum[blockIdx.x] = qc * Q::value(q);
    }
}

// ---------------------------------------------------------------------------
// z pass of the single-state step in one kernel: per (ky, kx) column, the forward z
// FFT -> F^n_k, the update of k_update (uh^{n+1} over uh^{n-1}, W <- uh^{n+1} in the pass
// precision, Q terms on recording steps), then the inverse z FFT of uh^{n+1}.  One pass
// over W2: 2 W + 3 S per launch instead of 6 W + 3 S for the three kernels.
// C columns of N rows per CTA (ZStepShape).  The state is read with plain loads after the forward
// transform; on large grids, whose arrays do not stay in L2, one thread has asked L2 for the
// tile's two contiguous state runs before it (one bulk prefetch each).  The pass by itself, with
// tiles of eight columns, 512^3: 1.561 -> 1.548 ms double-float, 0.777 -> 0.746 ms FP32; 256^3: 0.185 ->
// 0.179 and 0.118 -> 0.106 ms.
// ---------------------------------------------------------------------------
// [p, p + bytes) of global memory into L2 (16-byte aligned, a multiple of 16 bytes)
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

// columns per CTA: one tile of z-columns from N = 32 on.  Four double-float columns make CTAs of 256
// threads at 512^3, four per SM where eight made two of 512: their phases interleave more and wait
// less (1.543 -> 1.386 ms).
template <class P, int N>
struct ZStepShape {
    static constexpr int C = N >= 32 ? 1 << LayLg<P, N>::value : 16;
    static constexpr int NT = C * N / 8;
    static constexpr bool kPrefetch = N >= 256;
};
// resident threads per SM the kernel is compiled for: 1024 (64 registers; double-float 44 to 56
// bytes of spills, complex 72 to 92, composed 108 to 248); 1536 for the FP32 passes at N = 512: 40
// registers and 96 bytes of spills, which the extra loads in flight outweigh (0.798 -> 0.780 ms, 0.854
// -> 0.834 with the energy every 10 steps; not measured at other sizes, which keep 1024)
template <class P, int N>
struct ZStepMinBlocks {
    static constexpr int kThreads = (sizeof(typename P::S) == 8 && N >= 512) ? 1536 : 1024;
    static constexpr int value = N >= 128 && kThreads / ZStepShape<P, N>::NT > 1 ? kThreads / ZStepShape<P, N>::NT : 1;
};

// What a z pass does when its last CTA is done.  After k_plane the finalisers have no y pass to
// ride in: the CTA that draws the last ticket runs them, that of the x statistics (fx) and that of
// the update (fz); the others have read the run state by then.  Blow-up at this level must already
// stop the update, so every CTA compares the maximum that k_plane left in the run state.  A step
// that records no energies has nothing to reduce: its CTAs draw once the update is done, ahead of
// their stores, and the last one advances a copy of the run state that it has read by then.
// (Tickets after the stores and the general finalisers on every step cost 5 us of a 12 us pass.)
struct NoTail {};
struct ZTail {
    FinArgs fx, fz;
};

// bring a table entry into L1
__device__ __forceinline__ void touch(const double2* p) {
    double x, y;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];\n" : "=d"(x), "=d"(y) : "l"(p));
}

template <class P, int N, bool CPLX = false, int SCHEME = 0, class TAIL = NoTail>
__global__ void __launch_bounds__(ZStepShape<P, N>::NT, ZStepMinBlocks<P, N>::value)
    k_zstep(typename P::S* __restrict__ W, double2* S0, double2* S1, KgDev* __restrict__ dev,
            double* __restrict__ part_sum, const typename P::S* __restrict__ tw, const double2* __restrict__ coef,
            const double* __restrict__ w2tab, double qr, double qc, C4Args c4, TAIL tail) {
    typedef typename P::R R;
    typedef typename P::S S;
    typedef QTerm<P> Q;
    typedef Lay<N, CPLX> Ly;
    constexpr bool kTail = std::is_same<TAIL, ZTail>::value;
    constexpr int T = N / 8, C = ZStepShape<P, N>::C, NT = ZStepShape<P, N>::NT, LG = LayLg<P, N>::value, RS = 1 << LG;
    extern __shared__ __align__(16) unsigned char smraw[];
    S* sm = reinterpret_cast<S*>(smraw);
    __shared__ typename Q::T red[NT / 32];
    const int c = threadIdx.x % C, j = threadIdx.x / C;
    const int kx = blockIdx.x * C + c, ky = blockIdx.y;
    const bool valid = kx < Ly::NX;   // columns of the last tile beyond the plane compute on zeros
    ColSmem<P, C> csm{sm, c};
    const size_t base = Ly::zcol(ky, kx, LG);
    if (ZStepShape<P, N>::kPrefetch && threadIdx.x == 0) {
        prefetch_l2(S0 + base, (unsigned)(N * C * sizeof(double2)));
        prefetch_l2(S1 + base, (unsigned)(N * C * sizeof(double2)));
    }
    if constexpr (kTail) {
        if (SCHEME == 0 && valid) {
            const int my = ky <= N / 2 ? ky : ky - N;
#pragma unroll
            for (int s = 0; s < 8; s++) {
                const int kz = j + T * s, mz = kz <= N / 2 ? kz : kz - N;
                touch(coef + (kx * kx + my * my + mz * mz));
            }
        }
        tw = stage_table_any(tw, sm + N * C, N);
    } else tw = stage_table(tw, sm + N * C, N);
    pdl_wait();

    cx<R> v[8];
#pragma unroll
    for (int s = 0; s < 8; s++) {
        if (valid) v[s] = P::load(W[base + (size_t)(j + T * s) * RS]);
        else v[s] = cmake<R>(P::from_f64(0.0), P::from_f64(0.0));
    }
    // a small grid waits for each load in turn and has registers to spare: everything that the
    // update reads is on its way before the forward transform
    double2 pre0[kTail ? 8 : 1], pre1[kTail ? 8 : 1];
    KgDev run;
    const unsigned ctas = gridDim.x * gridDim.y;
    unsigned ticket = 0u;
    bool rec = false;
    if constexpr (kTail) {
        run = *dev;
#pragma unroll
        for (int s = 0; s < 8; s++) {
            pre0[s] = pre1[s] = make_double2(0.0, 0.0);
            if (valid) {
                pre0[s] = S0[base + (size_t)(j + T * s) * RS];
                pre1[s] = S1[base + (size_t)(j + T * s) * RS];
            }
        }
    }
    typename Q::T q = Q::zero();
    // the 16-byte bodies are large: both transforms run through one copy of the FFT code
    constexpr bool kShare = sizeof(S) == 16;
#pragma unroll(kShare ? 1 : 2)
    for (int dir = 0; dir < 2; dir++) {
        // F^n goes to the update through exact conversions of both words, uh^{n+1} to W
        fft<P, N, ColSmem<P, C>, false, false, false>(v, j, tw, 1, csm, dir == 0 ? -1 : +1);
        if (dir == 1) break;
        // the run state is read only now, so that nothing of it is live across the
        // forward transform (at 64 registers: 132 -> 8 bytes of spills, 1.98 -> 1.91 ms
        // for the double-float pass at 512^3 in the layout before; 56 bytes now)
        const KgDev* rs = dev;
        if constexpr (kTail) rs = &run;
        rec = kg_recording(rs);
        const bool want_q = SCHEME == 0 && rec;
        bool update = rs->frozen == 0;
        if constexpr (kTail) {
            if (run.threshold > 0.0 && run.sub == 0 && !(__longlong_as_double((long long)run.xkey) <= run.threshold))
                update = false;
        }
        double2* __restrict__ cur = rs->phase ? S1 : S0;
        double2* __restrict__ old = rs->phase ? S0 : S1;
        const int mx = (CPLX && kx > N / 2) ? kx - N : kx;
        const int my = ky <= N / 2 ? ky : ky - N;
        const int mxy2 = mx * mx + my * my;
        const bool twice = !CPLX && kx != 0 && kx != N / 2;
        const int sub = SCHEME == 0 ? 0 : rs->sub;
#pragma unroll
        for (int s = 0; s < 8; s++) {
            const int kz = j + T * s;
            const int mz = kz <= N / 2 ? kz : kz - N;
            const int m2 = mxy2 + mz * mz;
            if (valid) {
                const size_t idx = base + (size_t)kz * RS;
                double2 a, n;
                if constexpr (kTail) {
                    a = run.phase ? pre1[s] : pre0[s];
                    n = mode_update<P, SCHEME>(v[s], cur, old, idx, m2, coef, c4, sub, update, a,
                                               run.phase ? pre0[s] : pre1[s]);
                    pre0[s] = a;   // kept for the Q terms
                    pre1[s] = n;
                } else {
                    a = cur[idx];
                    n = mode_update<P, SCHEME>(v[s], cur, old, idx, m2, coef, c4, sub, update, a, old[idx]);
                    if (want_q) q = Q::add(q, Q::term(n.x, n.y, a, __ldg(w2tab + m2), qr, twice));
                }
                v[s] = cmake<R>(P::from_f64(n.x), P::from_f64(n.y));
            }
        }
        // the Q terms' code (eight copies, 40 KB) stays out of the other steps' way, which had to fetch
        // around it: 13.1 -> 11.5, 14.3 -> 13.0, 19.1 -> 18.0 us a step at 16, 32, 64^3
        if constexpr (kTail) {
            if (want_q && valid) {
#pragma unroll
                for (int s = 0; s < 8; s++) {
                    const int kz = j + T * s, mz = kz <= N / 2 ? kz : kz - N;
                    q = Q::add(q, Q::term(pre1[s].x, pre1[s].y, pre0[s], __ldg(w2tab + mxy2 + mz * mz), qr, twice));
                }
            }
        }
    }
    // the inverse transform's exchanges have passed: every thread of the CTA has read the run state
    if (kTail && threadIdx.x == 0 && !rec) ticket = atomicAdd(&dev->ticket, 1u);
    if (valid) {
#pragma unroll
        for (int s = 0; s < 8; s++) W[base + (size_t)(j + T * s) * RS] = P::pack(v[s]);
    }
    if (SCHEME == 0 && (kTail ? rec : kg_recording(dev))) {
        q = block_tree_sum<Q, NT>(q, red);
        if (threadIdx.x == 0) part_sum[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = qc * Q::value(q);
    }
    if constexpr (kTail) {
        if (rec) {
            __shared__ int last;
            __syncthreads();   // the CTA is done with smraw
            if (threadIdx.x == 0) {
                __threadfence();   // the partial is visible before the ticket
                last = atomicAdd(&dev->ticket, 1u) == ctas - 1;
            }
            __syncthreads();
            if (last) {
                // the first warp sums P's partials, the last one Q's; one thread advances the state
                __threadfence();
                double* tot = reinterpret_cast<double*>(smraw);
                const int w = threadIdx.x >> 5;
                const bool p_now = tail.fx.kind == FIN_X;
                if (p_now && w == 0) {
                    const double P = warp_total(tail.fx.part_sum, tail.fx.count);
                    if (threadIdx.x == 0) tot[0] = tail.fx.norm * P;
                }
                if (w == NT / 32 - 1) {
                    const double Q = warp_total(tail.fz.part_sum, tail.fz.count);
                    if ((threadIdx.x & 31) == 0) tot[1] = tail.fz.norm * Q;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    if (p_now) {
                        state_after_x(&run, false, true, __longlong_as_double((long long)run.xkey), tot[0]);
                        run.xkey = 0ull;
                    } else {
                        run.maxabs_last = run.maxabs_peek;
                    }
                    state_after_z(&run, true, tot[1]);
                    run.ticket = 0u;
                    *dev = run;
                }
            }
        } else if (threadIdx.x == 0 && ticket == ctas - 1) {
            if (tail.fx.kind == FIN_AHEAD_DONE) {
                run.maxabs_last = run.maxabs_peek;
            } else {
                state_after_x(&run, false, false, __longlong_as_double((long long)run.xkey), 0.0);
                run.xkey = 0ull;
            }
            state_after_z(&run, false, 0.0);
            run.ticket = 0u;
            *dev = run;
        }
    }
}

#ifdef KG_DEFINE_COMMON_KERNELS   // defined by exactly one translation unit
// a finaliser in a kernel of its own (one CTA): the fused xy form, kg_energy's passes.
// before / after (host memory, may be NULL) receive the run state around it.
__global__ void __launch_bounds__(kFinThreads) k_fin(FinArgs f, KgDev* before, KgDev* after) {
    __shared__ double red[kFinSmem];
    if (before && threadIdx.x == 0) *before = *f.dev;
    __syncthreads();
    finalise<kFinThreads>(f, red);
    __syncthreads();
    if (after && threadIdx.x == 0) *after = *f.dev;
}
#endif  // KG_DEFINE_COMMON_KERNELS

// ---------------------------------------------------------------------------
// FP64 set-up and read-out kernels
// ---------------------------------------------------------------------------
// forward R2C along x of physical lines: out[line][k] = sum_x f(u[line][x]) e^{-2 pi i k x/N},
// f(u) = u (cube == 0) or lam u^3 (cube == 1).  Same line mapping as pass X.
template <int N>
__global__ void __launch_bounds__(kXThreads) k_x_forward(const double* __restrict__ u, double2* __restrict__ out,
                                                         const double2* __restrict__ tw, int cube, double lam) {
    typedef PrecF64 P;
    typedef cx<double> C;
    typedef XShape<N> X;
    constexpr int M = X::M, T = X::T;
    extern __shared__ __align__(16) unsigned char smraw[];
    double2* sm = reinterpret_cast<double2*>(smraw);
    const int li = threadIdx.x / T, j = threadIdx.x % T;
    const size_t line = (size_t)blockIdx.x * X::LPC + li;
    const double* __restrict__ ul = u + line * N;
    double2* __restrict__ L = out + line * Lay<N>::PITCH;
    LineSmem<P> lsm{sm + li * X::PADM};
    C v[8];
#pragma unroll
    for (int s = 0; s < 8; s++) {
        const int m = j + T * s;
        double a = ul[2 * m], b = ul[2 * m + 1];
        if (cube) {
            a = lam * (a * a * a);
            b = lam * (b * b * b);
        }
        v[s] = cmake<double>(a, b);
    }
    fft<P, M>(v, j, tw, 2, lsm, -1);
#pragma unroll
    for (int s = 0; s < 8; s++) lsm.put(j + T * s, v[s]);
    lsm.sync();
#pragma unroll
    for (int s = 0; s < 8; s++) {
        const int k = j + T * s;
        C Z = v[s];
        C Zp = lsm.get((M - k) & (M - 1));
        C A = Z + conj(Zp);
        C B = Z - conj(Zp);
        C w = twiddle<P>(tw, k, -1);
        C D = mul_i(cmul(w, B));
        L[k] = make_double2(0.5 * (A.re - D.re), 0.5 * (A.im - D.im));
        if (k == 0) L[M] = make_double2(Z.re - Z.im, 0.0);
    }
}

// inverse C2R along x to physical lines, times scale; optionally sum u^4 (per CTA)
template <int N>
__global__ void __launch_bounds__(kXThreads) k_x_inverse(const double2* __restrict__ in, double* __restrict__ u,
                                                         const double2* __restrict__ tw, double scale,
                                                         double* __restrict__ part_sum) {
    typedef PrecF64 P;
    typedef cx<double> C;
    typedef XShape<N> X;
    constexpr int M = X::M, T = X::T;
    extern __shared__ __align__(16) unsigned char smraw[];
    double2* sm = reinterpret_cast<double2*>(smraw);
    __shared__ double red[96];
    const int li = threadIdx.x / T, j = threadIdx.x % T;
    const size_t line = (size_t)blockIdx.x * X::LPC + li;
    LineSmem<P> lsm{sm + li * X::PADM};
    C v[8];
    x_load_c2r<P, N>(in + line * Lay<N>::PITCH, j, tw, v);
    fft<P, M>(v, j, tw, 2, lsm, +1);
    NSum acc;
    acc.s = 0.0;
    acc.c = 0.0;
#pragma unroll
    for (int s = 0; s < 8; s++) {
        const int m = j + T * s;
        const double a = v[s].re * scale, b = v[s].im * scale;
        if (u) {
            u[line * N + 2 * m] = a;
            u[line * N + 2 * m + 1] = b;
        }
        if (part_sum) {
            const double a2 = a * a, b2 = b * b;
            acc.add(a2 * a2);
            acc.add(b2 * b2);
        }
    }
    if (part_sum) {
        double mx = 0.0;
        block_reduce<kXThreads>(acc, mx, red);
        if (threadIdx.x == 0) part_sum[blockIdx.x] = acc.value();
    }
}

// Set-up and read-out along x in the pass precision, two physical x-lines per N-point
// complex transform (the pair form of the x pass), one pair per N/8 threads:
// FWD: physical FP64 lines u_in (lam u^3 when cube) -> their half spectra, unnormalised,
//      in the pass precision in spec (x-lines, struct Lay);
// else: half spectra in spec -> physical lines times scale, FP64, into u_out.
template <class P, int N, bool FWD>
__global__ void __launch_bounds__(kXThreads) k_x_pair_io(const double* __restrict__ u_in, typename P::S* __restrict__ spec,
                                                         double* __restrict__ u_out,
                                                         const typename P::S* __restrict__ tw, int cube, double lam,
                                                         double scale) {
    typedef typename P::R R;
    typedef cx<R> C;
    typedef XpShape<N> X;
    constexpr int T = X::T;
    extern __shared__ __align__(16) unsigned char smraw[];
    typename P::S* sm = reinterpret_cast<typename P::S*>(smraw);
    const int pi = threadIdx.x / T, j = threadIdx.x % T;
    const size_t pair = (size_t)blockIdx.x * X::PPC + pi;
    LineSmemX<P, X::CTA_SYNC> lsm{sm + pi * X::PADN, 1u + (unsigned)pi, (unsigned)T};
    typename P::S* __restrict__ L1 = spec + 2 * pair * Lay<N>::PITCH;
    typename P::S* __restrict__ L2 = L1 + Lay<N>::PITCH;
    C v[8];
    if constexpr (FWD) {
        const double* __restrict__ u1 = u_in + 2 * pair * N;
        const double* __restrict__ u2 = u1 + N;
        const R rlam = P::from_f64(lam);
#pragma unroll
        for (int s = 0; s < 8; s++) {
            const int x = j + T * s;
            R a = P::from_f64(u1[x]), b = P::from_f64(u2[x]);
            if (cube) {
                a = rlam * (a * a * a);
                b = rlam * (b * b * b);
            }
            v[s] = cmake<R>(a, b);
        }
        fft<P, N>(v, j, tw, 1, lsm, -1);
        x_pair_unpack<P, N>(L1, L2, j, lsm, v);
    } else {
        x_pair_load<P, N>(L1, L2, j, v);
        fft<P, N>(v, j, tw, 1, lsm, +1);
        double* __restrict__ o1 = u_out + 2 * pair * N;
        double* __restrict__ o2 = o1 + N;
#pragma unroll
        for (int s = 0; s < 8; s++) {
            const int x = j + T * s;
            const cx<double> w = Convert<P, PrecF64>::go(
                cmake<R>(P::scale2(v[s].re, scale), P::scale2(v[s].im, scale)));
            o1[x] = w.re;
            o2[x] = w.im;
        }
    }
}

// uh^{-1} = c_k uh^0 - dt vh^0 + beta_k F^0 (coef holds 2c, 2 beta); b holds vh^0 on entry
template <int N, bool CPLX = false>
__global__ void k_startup(const double2* __restrict__ a, double2* __restrict__ b, const double2* __restrict__ f,
                          const double2* __restrict__ coef, double dt, int lg) {
    typedef ModeIndex<N, CPLX> MI;
    const size_t total = MI::slots(lg);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const MI mi((unsigned)i, lg);
        if (!mi.valid) continue;
        const double2 cf = coef[mi.m2];
        const double c = 0.5 * cf.x, beta = 0.5 * cf.y;
        const double2 a0 = a[i], v0 = b[i], f0 = f[i];
        b[i] = make_double2(c * a0.x - dt * v0.x + beta * f0.x, c * a0.y - dt * v0.y + beta * f0.y);
    }
}

// startup of the composed scheme: b holds vh^0 on entry and the stored velocity variable
// P^0 = vh^0 - (h_0/2)(F^0 - omega^2 uh^0)/(1 + omega^2 h_0^2/4) on exit (the first
// merged kick then applies only the opening half kick); kick0 = (K_0, K_0 omega^2) with
// K_0 = h_0/(1 + omega^2 h_0^2/4)
template <int N>
__global__ void k_startup_c4(const double2* __restrict__ a, double2* __restrict__ b, const double2* __restrict__ f,
                             const double2* __restrict__ kick0, int lg) {
    typedef ModeIndex<N, false> MI;
    const size_t total = MI::slots(lg);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const MI mi((unsigned)i, lg);
        if (!mi.valid) continue;
        const double2 kc = kick0[mi.m2];
        const double2 a0 = a[i], v0 = b[i], f0 = f[i];
        b[i] = make_double2(v0.x - 0.5 * (kc.x * f0.x - kc.y * a0.x), v0.y - 0.5 * (kc.x * f0.y - kc.y * a0.y));
    }
}

// Q(x, y) partials for arbitrary FP64 spectral pairs (energy outside the recorded steps)
template <int N, bool CPLX = false>
__global__ void __launch_bounds__(256) k_energy_q(const double2* __restrict__ x, const double2* __restrict__ y,
                                                  const double* __restrict__ w2tab, double inv_dt,
                                                  double* __restrict__ part_sum, int lg) {
    typedef ModeIndex<N, CPLX> MI;
    __shared__ double red[96];
    const size_t total = MI::slots(lg);
    NSum acc;
    acc.s = 0.0;
    acc.c = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const MI mi((unsigned)i, lg);
        if (!mi.valid) continue;
        const double w = mi.twice ? 2.0 : 1.0;
        const double2 a = x[i], b = y[i];
        const double dre = (a.x - b.x) * inv_dt, dim = (a.y - b.y) * inv_dt;
        const double sre = a.x + b.x, sim = a.y + b.y;
        acc.add(w * (0.5 * (dre * dre + dim * dim) + 0.125 * w2tab[mi.m2] * (sre * sre + sim * sim)));
    }
    double mx = 0.0;
    block_reduce<256>(acc, mx, red);
    if (threadIdx.x == 0) part_sum[blockIdx.x] = acc.value();
}

// z-columns <-> the packed order [kz][ky][kx] of checkpoints and kg_fetch_spectral
template <int N, bool CPLX, bool TO_PACKED>
__global__ void k_repack(const double2* __restrict__ in, double2* __restrict__ out, int lg) {
    typedef ModeIndex<N, CPLX> MI;
    const size_t total = MI::slots(lg);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const MI mi((unsigned)i, lg);
        if (!mi.valid) continue;
        const size_t p = ((size_t)mi.kz * N + mi.ky) * MI::Ly::NX + mi.kx;
        if (TO_PACKED) out[p] = in[i];
        else out[i] = in[p];
    }
}

#ifdef KG_DEFINE_COMMON_KERNELS
// plain Neumaier total of partials into *out (times norm)
__global__ void __launch_bounds__(kFinThreads) k_fin_sum(const double* part_sum, int count, double norm, double* out) {
    __shared__ double red[kFinSmem];
    NSum acc;
    double mx;
    fin_reduce<kFinThreads>(part_sum, nullptr, count, acc, mx, red);
    if (threadIdx.x == 0) *out = norm * acc.value();
}

#endif  // KG_DEFINE_COMMON_KERNELS

}  // namespace kg
