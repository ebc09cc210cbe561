// kg_mlp.cu -- the blow-up ranker network: training and inference on the GPU.
//
// The paper motivates parametric studies of blow-up (section 1) but has no learned
// component; this network is the project's.  Network 6 -> 128 -> 128 -> 2 (ReLU),
// heads z0 = blow-up logit and z1 = predicted log blow-up time.  Loss, mean over the
// batch: BCE(z0, y) + y (z1 - l)^2 + (1 - y) relu(log T - z1)^2 (runs that did not
// blow up by T only bound t_b from below).  Adam on FP32 master weights.
//
// Arithmetic: BF16 operands (inputs, weights, activations h1, h2 and the activation
// gradients dz, dh2, dh1, rounded to nearest even where they are stored) on the
// tensor cores with FP32 accumulation (mma.sync m16n8k16, operands by ldmatrix from rows
// padded to 16 bytes past a multiple of 128); biases, the loss and the weight gradients are
// FP32.  One CTA of 32 warps takes tiles of 128 batch rows with all weights in shared memory:
// warp w has 16 rows (w mod 8) and 32 columns (w / 8) of the activations, and 16 x 32 of dW2
// (summed over the tile's rows in one chain of products).
// A training step is latency: 26 MFLOP in a chain of six products.  With 8 warps per CTA,
// operands gathered by 2-byte shared loads, gradients added by atomics and the host waiting for
// the loss after every epoch it took 120 us (batch 256); now 18 us, and a prediction of 65 536 rows
// 75 us in place of 518 (buffers kept between calls, the sigmoid on the device).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/kg.h"
#include "kg_fft.cuh"
#include "kg_launch.h"

namespace {

constexpr int DIN = 6, DH = 128, DOUT = 2;
constexpr int KIN = 16;                          // padded input width (one MMA k-step)
constexpr int K3 = 16;                           // padded output width of W3 / dz
constexpr int BT = 128;                          // batch rows of a tile
constexpr int NTH = 1024;
constexpr int RT = BT / 16;                      // row tiles: warp w has row tile w % RT, columns 32 (w / RT) ..
static_assert(RT * (DH / 32) == NTH / 32, "the warps tile the activations");
// CTAs (and partial gradients) of a backward launch.  Batches up to 16384 rows have a CTA a tile, larger
// ones several tiles a CTA.  Training on large batches waits for the host, which draws the row order
// (16384 rows a batch: 98 us with 64 and 128 alike); a gradient by itself does not (kg_mlp_grad of 65 536
// rows: 205 us with 64, 145 with 128).
constexpr int kMostParts = 128;
constexpr int NPARAM = DIN * DH + DH + DH * DH + DH + DH * DOUT + DOUT;
// offsets of the tensors in the flat parameter vector (order W1, b1, W2, b2, W3, b3)
constexpr int OW1 = 0, OB1 = OW1 + DIN * DH, OW2 = OB1 + DH, OB2 = OW2 + DH * DH, OW3 = OB2 + DH,
              OB3 = OW3 + DH * DOUT;

typedef unsigned short bf;   // raw bfloat16 bits

__device__ __forceinline__ bf to_bf(float f) { return __bfloat16_as_ushort(__float2bfloat16_rn(f)); }
__device__ __forceinline__ float from_bf(bf b) { return __bfloat162float(__ushort_as_bfloat16(b)); }

__device__ __forceinline__ void mma_16x8x16(float c[4], const unsigned a[4], const unsigned b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
template <bool TRANS>
__device__ __forceinline__ void ldsm4(unsigned r[4], const bf* p) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(p);
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(sa));
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(sa));
}
// Operands by ldmatrix: lane l gives the row address of 8x8 matrix l / 8.  A (16 x 16 at m0, k0)
// from an array [m][k] or, transposed, [k][m]; B (16 x 16 at k0, n0: two tiles of eight columns,
// b[0..1] and b[2..3]) from [n][k] or, transposed, [k][n]; ld is the row pitch
__device__ __forceinline__ void load_a(unsigned a[4], const bf* p, int ld, int m0, int k0) {
    const int l = threadIdx.x & 31, q = l >> 3;
    ldsm4<false>(a, p + (m0 + (l & 7) + (q & 1) * 8) * ld + k0 + (q >> 1) * 8);
}
__device__ __forceinline__ void load_at(unsigned a[4], const bf* p, int ld, int m0, int k0) {
    const int l = threadIdx.x & 31, q = l >> 3;
    ldsm4<true>(a, p + (k0 + (l & 7) + (q >> 1) * 8) * ld + m0 + (q & 1) * 8);
}
__device__ __forceinline__ void load_b(unsigned b[4], const bf* p, int ld, int k0, int n0) {
    const int l = threadIdx.x & 31, q = l >> 3;
    ldsm4<false>(b, p + (n0 + (l & 7) + (q >> 1) * 8) * ld + k0 + (q & 1) * 8);
}
__device__ __forceinline__ void load_bt(unsigned b[4], const bf* p, int ld, int k0, int n0) {
    const int l = threadIdx.x & 31, q = l >> 3;
    ldsm4<true>(b, p + (k0 + (l & 7) + (q & 1) * 8) * ld + n0 + (q >> 1) * 8);
}

constexpr int LH = DH + 8;     // row pitch of 128-wide arrays (272 bytes: eight rows hit eight bank groups)
constexpr int LK = 16 + 8;     // row pitch of 16-wide arrays (48 bytes: the same)

struct Smem {
    bf w1[KIN * LH];
    bf w2[DH * LH];
    bf w3[DH * LK];
    bf x[BT * LK];
    bf h1[BT * LH];
    bf h2[BT * LH];     // reused for dh1 in the backward pass
    bf dh2[BT * LH];
    bf dz[BT * LK];
    float b1[DH], b2[DH], b3[DOUT];
    float red[3 * RT];   // per row tile: loss, db3
};

struct Params {   // device pointers
    const float* master;     // NPARAM fp32
    const bf* w1b;           // KIN x DH
    const bf* w2b;           // DH x DH
    const bf* w3b;           // DH x K3
};

// the weights into padded rows, 16 bytes a copy
__device__ __forceinline__ void load_weights(Smem& s, const Params& P) {
    for (int i = threadIdx.x; i < KIN * DH / 8; i += NTH)
        kg::cp_async16(s.w1 + (i / (DH / 8)) * LH + (i % (DH / 8)) * 8, P.w1b + 8 * i);
    for (int i = threadIdx.x; i < DH * DH / 8; i += NTH)
        kg::cp_async16(s.w2 + (i / (DH / 8)) * LH + (i % (DH / 8)) * 8, P.w2b + 8 * i);
    for (int i = threadIdx.x; i < DH * K3 / 8; i += NTH)
        kg::cp_async16(s.w3 + (i / (K3 / 8)) * LK + (i % (K3 / 8)) * 8, P.w3b + 8 * i);
    kg::cp_async_commit();
    if (threadIdx.x < DH) s.b1[threadIdx.x] = P.master[OB1 + threadIdx.x];
    else if (threadIdx.x < 2 * DH) s.b2[threadIdx.x - DH] = P.master[OB2 + threadIdx.x - DH];
    else if (threadIdx.x < 2 * DH + DOUT) s.b3[threadIdx.x - 2 * DH] = P.master[OB3 + threadIdx.x - 2 * DH];
}
// rows row0.. of X (gathered through idx when given), zero beyond n and in the padded inputs
__device__ __forceinline__ void load_rows(Smem& s, const float* X, const int* idx, int n, int row0) {
    for (int i = threadIdx.x; i < BT * KIN; i += NTH) {
        const int r = i / KIN, c = i % KIN, row = row0 + r;
        float v = 0.f;
        if (c < DIN && row < n) v = X[(size_t)(idx ? idx[row] : row) * DIN + c];
        s.x[r * LK + c] = to_bf(v);
    }
}

// the two values of a fragment pair (c, c + 1) as one bf16x2 word
__device__ __forceinline__ void put2(bf* p, float a, float b) {
    *reinterpret_cast<unsigned*>(p) = (unsigned)to_bf(a) | ((unsigned)to_bf(b) << 16);
}

// h1 and h2 of the tile, then z = h2 W3 + b3 in c3 of warps 0 .. RT - 1 (rows 16 w ..; columns 0 and 1 live in
// c3[0], c3[1] (row g) and c3[2], c3[3] (row g + 8) of the lanes with t == 0).  Ends with every warp
// past the barrier after h2.
__device__ __forceinline__ void forward_tile(Smem& s, float c3[4]) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int r0 = 16 * (w % RT), n0 = 32 * (w / RT);
    unsigned a[4], b[4];
    {   // h1 = relu(x W1 + b1)
        load_a(a, s.x, LK, r0, 0);
#pragma unroll
        for (int q = 0; q < 2; q++) {
            load_bt(b, s.w1, LH, 0, n0 + 16 * q);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                float c[4] = {0.f, 0.f, 0.f, 0.f};
                mma_16x8x16(c, a, b + 2 * h);
                const int col = n0 + 16 * q + 8 * h + 2 * t;
                const float ba = s.b1[col], bb = s.b1[col + 1];
                put2(s.h1 + (r0 + g) * LH + col, fmaxf(c[0] + ba, 0.f), fmaxf(c[1] + bb, 0.f));
                put2(s.h1 + (r0 + g + 8) * LH + col, fmaxf(c[2] + ba, 0.f), fmaxf(c[3] + bb, 0.f));
            }
        }
    }
    __syncthreads();
    {   // h2 = relu(h1 W2 + b2)
        float c[4][4] = {};
#pragma unroll
        for (int kt = 0; kt < DH / 16; kt++) {
            load_a(a, s.h1, LH, r0, 16 * kt);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                load_bt(b, s.w2, LH, 16 * kt, n0 + 16 * q);
                mma_16x8x16(c[2 * q], a, b);
                mma_16x8x16(c[2 * q + 1], a, b + 2);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int col = n0 + 8 * q + 2 * t;
            const float ba = s.b2[col], bb = s.b2[col + 1];
            put2(s.h2 + (r0 + g) * LH + col, fmaxf(c[q][0] + ba, 0.f), fmaxf(c[q][1] + bb, 0.f));
            put2(s.h2 + (r0 + g + 8) * LH + col, fmaxf(c[q][2] + ba, 0.f), fmaxf(c[q][3] + bb, 0.f));
        }
    }
    __syncthreads();
    if (w < RT) {   // z
#pragma unroll
        for (int q = 0; q < 4; q++) c3[q] = 0.f;
#pragma unroll
        for (int kt = 0; kt < DH / 16; kt++) {
            load_a(a, s.h2, LH, r0, 16 * kt);
            load_bt(b, s.w3, LK, 16 * kt, 0);   // columns 8..15 are padding
            mma_16x8x16(c3, a, b);
        }
        if (t == 0) {
            c3[0] += s.b3[0];
            c3[1] += s.b3[1];
            c3[2] += s.b3[0];
            c3[3] += s.b3[1];
        }
    }
}

// p = sigmoid(z0) and z1 of n rows (either may be NULL); the grid walks the tiles
__global__ void __launch_bounds__(NTH) k_mlp_forward(Params P, const float* X, int n, float* prob, float* logt) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem& s = *reinterpret_cast<Smem*>(raw);
    load_weights(s, P);
    for (int row0 = blockIdx.x * BT; row0 < n; row0 += gridDim.x * BT) {
        load_rows(s, X, nullptr, n, row0);
        kg::cp_async_wait_all();
        __syncthreads();
        float c3[4];
        forward_tile(s, c3);
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        if (w < RT && t == 0) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int row = row0 + 16 * w + g + 8 * h;
                if (row < n) {
                    if (prob) prob[row] = 1.f / (1.f + expf(-c3[2 * h]));
                    if (logt) logt[row] = c3[2 * h + 1];
                }
            }
        }
    }
}

// partial gradients of the mean loss over rows idx[0..n) (idx may be NULL: rows 0..n), scaled by
// inv_n, of this CTA's tiles into part[blockIdx.x], its loss sum into loss_part[blockIdx.x].  A CTA
// with several tiles adds each one's gradients to its part in global memory, with rounding: left in the
// accumulators, whose additions truncate, they drifted with the number of tiles: 65 536 and 262 144
// rows were 8.9e-7 and 4.1e-6 of the gradient from 64 bits, and are 2.3e-7 and 7.0e-7.
__global__ void __launch_bounds__(NTH) k_mlp_backward(Params P, const float* X, const float* Y, const float* ELL,
                                                      const int* idx, int n, float inv_n, float logT, float* part,
                                                      float* loss_part) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem& s = *reinterpret_cast<Smem*>(raw);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int r0 = 16 * (w % RT), n0 = 32 * (w / RT);
    // the labels of this lane's rows (t == 0 of the row warps) are asked for with the inputs
    float yv[2] = {0.f, 0.f}, lv[2] = {0.f, 0.f};
    auto load_labels = [&](int row0) {
        if (w < RT && t == 0) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int row = row0 + r0 + g + 8 * h;
                if (row < n) {
                    const int src = idx ? idx[row] : row;
                    yv[h] = Y[src];
                    lv[h] = ELL[src];
                }
            }
        }
    };
    load_rows(s, X, idx, n, blockIdx.x * BT);
    load_labels(blockIdx.x * BT);
    for (int i = threadIdx.x; i < BT * LK; i += NTH) s.dz[i] = 0;   // columns 2..15 stay zero
    kg::pdl_wait();   // the weights of the step before
    load_weights(s, P);
    float lsum = 0.f, db3a = 0.f, db3b = 0.f;
    float* out = part + (size_t)blockIdx.x * NPARAM;
    unsigned a[4], b[4];
    for (int row0 = blockIdx.x * BT; row0 < n; row0 += gridDim.x * BT) {
        if (row0 != (int)blockIdx.x * BT) {
            __syncthreads();   // the tile before is done with its rows
            load_rows(s, X, idx, n, row0);
            load_labels(row0);
        }
        kg::cp_async_wait_all();
        __syncthreads();
        float d1[4] = {}, d2[4][4] = {}, d3[4] = {}, db = 0.f;   // dW1, dW2, dW3, db1 or db2 of the tile
        float c3[4];
        forward_tile(s, c3);
        if (w < RT && t == 0) {   // dz = dL/dz per row
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int r = r0 + g + 8 * h, row = row0 + r;
                float e0 = 0.f, e1 = 0.f;
                if (row < n) {
                    const float y = yv[h], ell = lv[h];
                    const float z0 = c3[2 * h], z1 = c3[2 * h + 1];
                    const float sig = 1.f / (1.f + expf(-z0));
                    const float cens = fmaxf(logT - z1, 0.f);
                    lsum += fmaxf(z0, 0.f) - y * z0 + log1pf(expf(-fabsf(z0))) + y * (z1 - ell) * (z1 - ell) +
                            (1.f - y) * cens * cens;
                    e0 = (sig - y) * inv_n;
                    e1 = (2.f * y * (z1 - ell) - 2.f * (1.f - y) * cens) * inv_n;
                }
                const bf q0 = to_bf(e0), q1 = to_bf(e1);
                s.dz[r * LK] = q0;
                s.dz[r * LK + 1] = q1;
                db3a += from_bf(q0);
                db3b += from_bf(q1);
            }
        }
        __syncthreads();
        {   // dh2 = (dz W3^T) masked by h2 > 0
            load_a(a, s.dz, LK, r0, 0);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                load_b(b, s.w3, LK, 0, n0 + 16 * q);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
                    mma_16x8x16(c, a, b + 2 * h);
                    const int col = n0 + 16 * q + 8 * h + 2 * t;
#pragma unroll
                    for (int e = 0; e < 2; e++) {
                        const int at = (r0 + g + 8 * e) * LH + col;
                        put2(s.dh2 + at, from_bf(s.h2[at]) > 0.f ? c[2 * e] : 0.f,
                             from_bf(s.h2[at + 1]) > 0.f ? c[2 * e + 1] : 0.f);
                    }
                }
            }
        }
        if (w < 8) {   // dW3 += h2^T dz: warp w owns features 16 w ..
#pragma unroll
            for (int kt = 0; kt < BT / 16; kt++) {
                load_at(a, s.h2, LH, 16 * w, 16 * kt);
                load_bt(b, s.dz, LK, 16 * kt, 0);
                mma_16x8x16(d3, a, b);
            }
        }
        __syncthreads();   // dh2 complete; h2 is free from here on
        bf* dh1 = s.h2;
        {   // dh1 = (dh2 W2^T) masked by h1 > 0, written over h2
            float c[4][4] = {};
#pragma unroll
            for (int kt = 0; kt < DH / 16; kt++) {
                load_a(a, s.dh2, LH, r0, 16 * kt);
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    load_b(b, s.w2, LH, 16 * kt, n0 + 16 * q);
                    mma_16x8x16(c[2 * q], a, b);
                    mma_16x8x16(c[2 * q + 1], a, b + 2);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int col = n0 + 8 * q + 2 * t;
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    const int at = (r0 + g + 8 * e) * LH + col;
                    put2(dh1 + at, from_bf(s.h1[at]) > 0.f ? c[q][2 * e] : 0.f,
                         from_bf(s.h1[at + 1]) > 0.f ? c[q][2 * e + 1] : 0.f);
                }
            }
        }
        // dW2 += h1^T dh2: warp w owns rows 16 (w mod 8) .. and columns 32 (w / 8) ..
#pragma unroll
        for (int kt = 0; kt < BT / 16; kt++) {
            load_at(a, s.h1, LH, 16 * (w & 7), 16 * kt);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                load_bt(b, s.dh2, LH, 16 * kt, 32 * (w >> 3) + 16 * q);
                mma_16x8x16(d2[2 * q], a, b);
                mma_16x8x16(d2[2 * q + 1], a, b + 2);
            }
        }
        __syncthreads();   // dh1 complete
        if (w < 16) {   // dW1 += x^T dh1: warp w owns columns 8 w .. (the other half of a 16-wide load is unused)
#pragma unroll
            for (int kt = 0; kt < BT / 16; kt++) {
                load_at(a, s.x, LK, 0, 16 * kt);
                load_bt(b, dh1, LH, 16 * kt, 16 * (w >> 1));
                mma_16x8x16(d1, a, b + 2 * (w & 1));
            }
        } else if (w < 24) {   // db2, db1: column sums over the tile
            const int i = threadIdx.x - 512;
            const bf* col = (i < DH ? s.dh2 : dh1) + (i & (DH - 1));
#pragma unroll 16
            for (int r = 0; r < BT; r++) db += from_bf(col[r * LH]);
        }
        const bool add = row0 != (int)blockIdx.x * BT;
        auto put = [&](int at, float x, float y) {   // a thread's own pairs, the same in every tile
            float2* p = reinterpret_cast<float2*>(out + at);
            if (add) {
                const float2 v = *p;
                x += v.x;
                y += v.y;
            }
            *p = make_float2(x, y);
        };
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int at = OW2 + (16 * (w & 7) + g) * DH + 32 * (w >> 3) + 8 * q + 2 * t;
            put(at, d2[q][0], d2[q][1]);
            put(at + 8 * DH, d2[q][2], d2[q][3]);
        }
        if (w < 16 && g < DIN) put(OW1 + g * DH + 8 * w + 2 * t, d1[0], d1[1]);
        if (w < 8 && t == 0) {
            put(OW3 + (16 * w + g) * DOUT, d3[0], d3[1]);
            put(OW3 + (16 * w + g + 8) * DOUT, d3[2], d3[3]);
        }
        if (w >= 16 && w < 24) {
            const int i = threadIdx.x - 512, at = i < DH ? OB2 + i : OB1 + i - DH;
            out[at] = add ? out[at] + db : db;
        }
    }
    // loss and db3: warp sums, then the row warps in order
    if (w < RT) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            db3a += __shfl_xor_sync(0xffffffffu, db3a, o);
            db3b += __shfl_xor_sync(0xffffffffu, db3b, o);
        }
        if (lane == 0) {
            s.red[w] = lsum;
            s.red[RT + w] = db3a;
            s.red[2 * RT + w] = db3b;
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        float v = 0.f;
        for (int r = 0; r < RT; r++) v += s.red[RT * threadIdx.x + r];
        if (threadIdx.x == 0) loss_part[blockIdx.x] = v;
        else out[OB3 + threadIdx.x - 1] = v;
    }
}

// grad = sum of nparts partial gradients in order (kg_mlp_grad), loss likewise
__global__ void k_mlp_sum(const float* part, const float* loss_part, int nparts, float* grad, float* loss) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPARAM) {
        float v = 0.f;
        for (int c = 0; c < nparts; c++) v += part[(size_t)c * NPARAM + i];
        grad[i] = v;
    }
    if (i == 0) {
        float v = 0.f;
        for (int c = 0; c < nparts; c++) v += loss_part[c];
        *loss = v;
    }
}

// Adam on the master weights with the sum of nparts partial gradients (taken in order, so that a
// run repeats itself), then the bf16 copies (padded shapes); the batch's loss joins *loss.
// nparts == 0 only refreshes the copies.
__global__ void __launch_bounds__(256) k_mlp_adam(float* master, const float* part, const float* loss_part, int nparts,
                                                  float* m, float* v, float* loss, float lr, float b1, float b2,
                                                  float eps, float c1, float c2, bf* w1b, bf* w2b, bf* w3b) {
    kg::pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPARAM) {
        float wv = master[i];
        if (nparts > 0) {
            float gv = 0.f;
            for (int c = 0; c < nparts; c++) gv += part[(size_t)c * NPARAM + i];
            const float mv = b1 * m[i] + (1.f - b1) * gv;
            const float vv = b2 * v[i] + (1.f - b2) * gv * gv;
            m[i] = mv;
            v[i] = vv;
            wv -= lr * (mv * c1) / (sqrtf(vv * c2) + eps);
            master[i] = wv;
        }
        if (i < OB1) {
            const int r = i / DH, c = i % DH;
            w1b[r * DH + c] = to_bf(wv);
        } else if (i >= OW2 && i < OB2) {
            w2b[i - OW2] = to_bf(wv);
        } else if (i >= OW3 && i < OB3) {
            const int r = (i - OW3) / DOUT, c = (i - OW3) % DOUT;
            w3b[r * K3 + c] = to_bf(wv);
        }
    }
    if (i == 0 && loss_part) {
        float l = *loss;
        for (int c = 0; c < nparts; c++) l += loss_part[c];
        *loss = l;
    }
}
constexpr int kAdamCtas = (NPARAM + 255) / 256;

// rows of device memory a call's data are staged in, kept between calls (grown as needed, released
// by kg_mlp_finalize): a call that allocates and frees its own spends longer on that than on work
struct Staging {
    float *X = nullptr, *Y = nullptr, *E = nullptr;   // inputs; predictions use Y and E as outputs
    int* idx[2] = {nullptr, nullptr};                 // two epochs' row orders
    int* h_idx[2] = {nullptr, nullptr};               // pinned, to fill one while the other uploads
    cudaEvent_t sent[2] = {nullptr, nullptr};
    int rows = 0, idx_rows = 0;
};

struct Mlp {
    float* master = nullptr;
    float* part = nullptr;       // partial gradients of a backward launch, kMostParts of them
    float* loss_part = nullptr;
    float* grad = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    bf* w1b = nullptr;
    bf* w2b = nullptr;
    bf* w3b = nullptr;
    float* loss = nullptr;
    long long t = 0;
    Staging st;
    std::vector<void*> allocs;
};
Mlp* g_mlp = nullptr;

int mfail(int code, const std::string& msg) { return kg::set_last_error(code, msg); }

#define KG_MCK(call)                                                                               \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) return mfail(KG_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

int mlp_alloc(Mlp* M, void** p, size_t b) {
    if (cudaMalloc(p, b) != cudaSuccess) {
        cudaGetLastError();
        return mfail(KG_ENOMEM, "mlp allocation");
    }
    cudaMemset(*p, 0, b);
    M->allocs.push_back(*p);
    return KG_OK;
}

void release_rows(Staging& s) {
    cudaFree(s.X);
    cudaFree(s.Y);
    cudaFree(s.E);
    s.X = s.Y = s.E = nullptr;
    s.rows = 0;
}
void release_orders(Staging& s) {
    for (int k = 0; k < 2; k++) {
        cudaFree(s.idx[k]);
        cudaFreeHost(s.h_idx[k]);
        s.idx[k] = s.h_idx[k] = nullptr;
    }
    s.idx_rows = 0;
}

void mlp_destroy(Mlp* M) {
    if (!M) return;
    cudaDeviceSynchronize();
    for (void* p : M->allocs) cudaFree(p);
    release_rows(M->st);
    release_orders(M->st);
    for (cudaEvent_t e : M->st.sent)
        if (e) cudaEventDestroy(e);
    delete M;
}

int mlp_ensure() {
    if (g_mlp) return KG_OK;
    Mlp* M = new Mlp();
    int rc = mlp_alloc(M, (void**)&M->master, sizeof(float) * NPARAM);
    if (!rc) rc = mlp_alloc(M, (void**)&M->grad, sizeof(float) * NPARAM);
    if (!rc) rc = mlp_alloc(M, (void**)&M->part, sizeof(float) * NPARAM * kMostParts);
    if (!rc) rc = mlp_alloc(M, (void**)&M->loss_part, sizeof(float) * kMostParts);
    if (!rc) rc = mlp_alloc(M, (void**)&M->m, sizeof(float) * NPARAM);
    if (!rc) rc = mlp_alloc(M, (void**)&M->v, sizeof(float) * NPARAM);
    if (!rc) rc = mlp_alloc(M, (void**)&M->w1b, sizeof(bf) * KIN * DH);
    if (!rc) rc = mlp_alloc(M, (void**)&M->w2b, sizeof(bf) * DH * DH);
    if (!rc) rc = mlp_alloc(M, (void**)&M->w3b, sizeof(bf) * DH * K3);
    if (!rc) rc = mlp_alloc(M, (void**)&M->loss, sizeof(float));
    if (rc) {
        mlp_destroy(M);
        return rc;
    }
    g_mlp = M;
    return KG_OK;
}

Params params_of(const Mlp* M) { return Params{M->master, M->w1b, M->w2b, M->w3b}; }

int refresh_bf16(Mlp* M) {
    k_mlp_adam<<<kAdamCtas, 256>>>(M->master, nullptr, nullptr, 0, M->m, M->v, M->loss, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f,
                                   M->w1b, M->w2b, M->w3b);
    KG_MCK(cudaGetLastError());
    return KG_OK;
}

int set_smem_once() {
    static bool done = false;
    if (done) return KG_OK;
    KG_MCK(cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)));
    KG_MCK(cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)));
    done = true;
    return KG_OK;
}

// Test hook: KG_TEST_FAIL_STAGING=k makes the k-th allocation of a growing staging fail
int g_staging_allocs = 0;
template <class T>
bool staging_fails(cudaError_t (*alloc)(void**, size_t), T** p, size_t bytes) {
    const char* inj = std::getenv("KG_TEST_FAIL_STAGING");
    if (inj && ++g_staging_allocs == std::atoi(inj)) return true;
    if (alloc((void**)p, bytes) == cudaSuccess) return false;
    cudaGetLastError();
    *p = nullptr;
    return true;
}

// room for n rows of inputs, labels (or outputs), and with idx for two row orders; what cannot be
// had in full is given back
int reserve(Staging& s, int n, bool idx) {
    const auto device = [](void** p, size_t b) { return cudaMalloc(p, b); };
    const auto pinned = [](void** p, size_t b) { return cudaMallocHost(p, b); };
    g_staging_allocs = 0;
    if (n > s.rows) {
        release_rows(s);
        if (staging_fails<float>(device, &s.X, sizeof(float) * DIN * (size_t)n) ||
            staging_fails<float>(device, &s.Y, sizeof(float) * (size_t)n) ||
            staging_fails<float>(device, &s.E, sizeof(float) * (size_t)n)) {
            release_rows(s);
            return mfail(KG_ENOMEM, "mlp data allocation");
        }
        s.rows = n;
    }
    if (idx && n > s.idx_rows) {
        release_orders(s);
        for (auto& e : s.sent)
            if (!e) KG_MCK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        for (int k = 0; k < 2; k++) {
            if (staging_fails<int>(device, &s.idx[k], sizeof(int) * (size_t)n) ||
                staging_fails<int>(pinned, &s.h_idx[k], sizeof(int) * (size_t)n)) {
                release_orders(s);
                return mfail(KG_ENOMEM, "mlp row order allocation");
            }
        }
        s.idx_rows = n;
    }
    return KG_OK;
}

// What a call keeps for the next one is bounded: staging beyond kKeepRows goes back at its end,
// however it ends.
constexpr int kKeepRows = 1 << 20;
struct Bounded {
    Staging& s;
    explicit Bounded(Staging& st) : s(st) {}
    Bounded(const Bounded&) = delete;
    ~Bounded() {
        if (s.rows > kKeepRows) release_rows(s);
        if (s.idx_rows > kKeepRows) release_orders(s);
    }
};

int upload(Staging& s, const float* X, const float* y, const float* ell, int n) {
    KG_MCK(cudaMemcpyAsync(s.X, X, sizeof(float) * DIN * (size_t)n, cudaMemcpyHostToDevice, 0));
    if (y) KG_MCK(cudaMemcpyAsync(s.Y, y, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, 0));
    if (ell) KG_MCK(cudaMemcpyAsync(s.E, ell, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, 0));
    return KG_OK;
}

int parts_of(int n) {
    const int tiles = (n + BT - 1) / BT;
    return tiles < kMostParts ? tiles : kMostParts;
}

// launches on the default stream that may start while the kernel before drains
template <class... KA, class... A>
cudaError_t launch_after(void (*kernel)(KA...), int grid, int block, size_t smem, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

}  // namespace

extern "C" {

int kg_mlp_set_params(const float* params) {
    if (!params) return mfail(KG_EINVAL, "NULL params");
    for (int i = 0; i < NPARAM; i++)
        if (!std::isfinite(params[i])) return mfail(KG_EINVAL, "non-finite parameter");
    int rc = mlp_ensure();
    if (rc) return rc;
    KG_MCK(cudaMemcpy(g_mlp->master, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice));
    KG_MCK(cudaMemset(g_mlp->m, 0, sizeof(float) * NPARAM));
    KG_MCK(cudaMemset(g_mlp->v, 0, sizeof(float) * NPARAM));
    g_mlp->t = 0;
    return refresh_bf16(g_mlp);
}

int kg_mlp_get_params(float* params) {
    if (!g_mlp) return mfail(KG_ESTATE, "kg_mlp_get_params before kg_mlp_set_params");
    if (!params) return mfail(KG_EINVAL, "NULL params");
    KG_MCK(cudaMemcpy(params, g_mlp->master, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
    return KG_OK;
}

int kg_mlp_predict(const float* X, int n, float* p_blowup, float* logt) {
    if (!g_mlp) return mfail(KG_ESTATE, "kg_mlp_predict before kg_mlp_set_params");
    if (!X || n < 1) return mfail(KG_EINVAL, "bad arguments");
    int rc = set_smem_once();
    Staging& s = g_mlp->st;
    const Bounded bounded(s);
    if (!rc) rc = reserve(s, n, false);
    if (!rc) rc = upload(s, X, nullptr, nullptr, n);
    if (rc) return rc;
    int dev = 0, sms = 0;
    KG_MCK(cudaGetDevice(&dev));
    KG_MCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int tiles = (n + BT - 1) / BT;   // a CTA per SM, over several tiles
    k_mlp_forward<<<tiles < sms ? tiles : sms, NTH, sizeof(Smem)>>>(params_of(g_mlp), s.X, n, p_blowup ? s.Y : nullptr,
                                                                      logt ? s.E : nullptr);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && p_blowup) e = cudaMemcpyAsync(p_blowup, s.Y, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost, 0);
    if (e == cudaSuccess && logt) e = cudaMemcpyAsync(logt, s.E, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost, 0);
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    if (e != cudaSuccess) return mfail(KG_ECUDA, std::string("mlp forward: ") + cudaGetErrorString(e));
    return KG_OK;
}

int kg_mlp_grad(const float* X, const float* y, const float* logt, int n, double T, float* grad, double* loss) {
    if (!g_mlp) return mfail(KG_ESTATE, "kg_mlp_grad before kg_mlp_set_params");
    if (!X || !y || !logt || n < 1 || !(T > 0.0)) return mfail(KG_EINVAL, "bad arguments");
    int rc = set_smem_once();
    Staging& s = g_mlp->st;
    const Bounded bounded(s);
    if (!rc) rc = reserve(s, n, false);
    if (!rc) rc = upload(s, X, y, logt, n);
    if (rc) return rc;
    const int parts = parts_of(n);
    k_mlp_backward<<<parts, NTH, sizeof(Smem)>>>(params_of(g_mlp), s.X, s.Y, s.E, nullptr, n, 1.f / (float)n,
                                                 (float)std::log(T), g_mlp->part, g_mlp->loss_part);
    k_mlp_sum<<<kAdamCtas, 256>>>(g_mlp->part, g_mlp->loss_part, parts, g_mlp->grad, g_mlp->loss);
    KG_MCK(cudaGetLastError());
    if (grad) KG_MCK(cudaMemcpy(grad, g_mlp->grad, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
    float l = 0.f;
    KG_MCK(cudaMemcpy(&l, g_mlp->loss, sizeof(float), cudaMemcpyDeviceToHost));
    if (loss) *loss = (double)l / n;
    return KG_OK;
}

int kg_mlp_train(const float* X, const float* y, const float* logt, int n, const kg_mlp_cfg* cfg, double* final_loss) {
    if (!g_mlp) return mfail(KG_ESTATE, "kg_mlp_train before kg_mlp_set_params");
    if (!X || !y || !logt || n < 1 || !cfg || cfg->epochs < 0 || cfg->batch < 1 || !(cfg->lr > 0.0) ||
        !(cfg->T > 0.0))
        return mfail(KG_EINVAL, "bad arguments");
    int rc = set_smem_once();
    Mlp* M = g_mlp;
    Staging& s = M->st;
    const Bounded bounded(s);
    if (!rc) rc = reserve(s, n, true);
    if (!rc) rc = upload(s, X, y, logt, n);
    if (rc) return rc;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f, logT = (float)std::log(cfg->T), lr = (float)cfg->lr;
    const int batch = cfg->batch < n ? cfg->batch : n;
    const int parts = parts_of(batch);
    unsigned long long st = cfg->seed ? cfg->seed : 0x9E3779B97F4A7C15ull;
    for (int ep = 0; ep < cfg->epochs; ep++) {
        // the row order of one epoch is drawn while the GPU works on the one before
        const int k = ep & 1;
        if (ep >= 2) KG_MCK(cudaEventSynchronize(s.sent[k]));
        int* perm = s.h_idx[k];
        for (int i = 0; i < n; i++) perm[i] = i;
        for (int i = n - 1; i > 0; i--) {   // Fisher-Yates with a xorshift64 stream
            st ^= st << 13;
            st ^= st >> 7;
            st ^= st << 17;
            const int j = (int)(st % (unsigned long long)(i + 1));
            const int tmp = perm[i];
            perm[i] = perm[j];
            perm[j] = tmp;
        }
        KG_MCK(cudaMemcpyAsync(s.idx[k], perm, sizeof(int) * n, cudaMemcpyHostToDevice, 0));
        KG_MCK(cudaEventRecord(s.sent[k], 0));
        KG_MCK(cudaMemsetAsync(M->loss, 0, sizeof(float), 0));
        for (int b0 = 0; b0 + batch <= n; b0 += batch) {
            KG_MCK(launch_after(k_mlp_backward, parts, NTH, sizeof(Smem), params_of(M), s.X, s.Y, s.E, s.idx[k] + b0,
                                batch, 1.f / (float)batch, logT, M->part, M->loss_part));
            M->t += 1;
            const float c1 = 1.f / (1.f - std::pow(b1, (float)M->t));
            const float c2 = 1.f / (1.f - std::pow(b2, (float)M->t));
            KG_MCK(launch_after(k_mlp_adam, kAdamCtas, 256, 0, M->master, M->part, M->loss_part, parts, M->m, M->v,
                                M->loss, lr, b1, b2, eps, c1, c2, M->w1b, M->w2b, M->w3b));
        }
    }
    float lastloss = 0.f;
    if (cfg->epochs > 0) {
        KG_MCK(cudaMemcpy(&lastloss, M->loss, sizeof(float), cudaMemcpyDeviceToHost));
        lastloss /= (float)((n / batch) * batch);
    }
    KG_MCK(cudaDeviceSynchronize());
    if (final_loss) *final_loss = lastloss;
    return KG_OK;
}

int kg_mlp_adam_step(const float* grad, double lr) {
    if (!g_mlp) return mfail(KG_ESTATE, "kg_mlp_adam_step before kg_mlp_set_params");
    if (!grad || !(lr > 0.0)) return mfail(KG_EINVAL, "bad arguments");
    KG_MCK(cudaMemcpy(g_mlp->part, grad, sizeof(float) * NPARAM, cudaMemcpyHostToDevice));
    g_mlp->t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f / (1.f - std::pow(b1, (float)g_mlp->t)), c2 = 1.f / (1.f - std::pow(b2, (float)g_mlp->t));
    k_mlp_adam<<<kAdamCtas, 256>>>(g_mlp->master, g_mlp->part, nullptr, 1, g_mlp->m, g_mlp->v, g_mlp->loss, (float)lr, b1,
                                   b2, 1e-8f, c1, c2, g_mlp->w1b, g_mlp->w2b, g_mlp->w3b);
    KG_MCK(cudaGetLastError());
    KG_MCK(cudaDeviceSynchronize());
    return KG_OK;
}

int kg_mlp_param_count(void) { return NPARAM; }

int kg_mlp_finalize(void) {
    mlp_destroy(g_mlp);
    g_mlp = nullptr;
    return KG_OK;
}

}  // extern "C"
