// Learned cost model kernels (the scheduler's analogue of the paper's
// performance-aware task scheduling, Sec. IV: estimated per-task costs choose
// where and how each task runs). Never touches pixel values.
//
//   features_kernel  one pass over I and J of every tile: 16-bin histogram of
//                    I - J (bins of width 16), count of I >= 100 (blob pixels),
//                    count of J == 0 (fill-holes markers), J > I violations.
//                    Erosion tiles are counted on complemented values (the
//                    dilation problem the kernel actually solves); FillHoles
//                    tiles as complemented I with J = 0 (their interior marker)
//   finalize_kernel  counts -> 20 fp32 features per tile
//   mlp_forward      20 -> 64 -> 64 -> 2, ReLU hidden units, fp32
//   mlp_grad         forward + backward of L = 1/(2N) sum (Y - T)^2 over a
//                    mini-batch, gradients accumulated per CTA in shared memory
//   adam_kernel      Adam update (Kingma & Ba 2015, Algorithm 1); zeroes the gradient
//   train_kernel     every step of one epoch (forward, backward, Adam) in one launch
#include <algorithm>
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include "recon_learn.h"

namespace rl {

struct FeatTile {
    const uint8_t *I, *J;
    int H, W, pitch, op;
    int crow;   // rows per chunk (about CHUNK_PX pixels)
};

__device__ __forceinline__ int find_chunk_tile(const unsigned *chunk_base, int n, unsigned c)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (chunk_base[mid] <= c) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// counts: per tile NCOUNT u32: [0..15] histogram, [16] bright, [17] zero J, [18] violations
constexpr int NCOUNT = 19;
constexpr int CHUNK_PX = 1 << 16;   // pixels per chunk of a tile (a whole number of rows, at least one)

constexpr int FT = 256;   // threads of features_kernel

// Four pixels at once (bytes of a 32-bit word). d gets the per-byte
// difference a - b modulo 256 and the high bit of each byte of `borrow` is set
// where b > a (the bytes subtract independently: the high bit of each byte of
// a is set first so that no borrow crosses a byte boundary, then restored).
__device__ __forceinline__ void sub_bytes(uint32_t a, uint32_t b, uint32_t &d, uint32_t &borrow)
{
    constexpr uint32_t H = 0x80808080u;
    d = ((a | H) - (b & ~H)) ^ ((a ^ ~b) & H);
    borrow = ((~a & b) | (~(a ^ b) & d)) & H;
}

// Counts of one thread: the 16 histogram bins live in the thread's own column
// of a shared array (row = bin, column = thread: the 32 lanes of a warp always
// touch 32 different banks), with row 16 taking the pixels whose I - J bin is
// undefined (J > I); the blob-pixel, zero-marker and violation counts are
// registers, counted four pixels at a time.
struct Counts {
    unsigned *col;                       // &hist[threadIdx.x], rows FT apart
    unsigned bright = 0, zero = 0, bad = 0;

    // one 32-bit word of I and of J; op: 0 dilation, 1 erosion, 2 FillHoles
    __device__ __forceinline__ void add4(uint32_t i, uint32_t j, int op, int npx = 4)
    {
        if (op != 0) {
            i = ~i;
            j = (op == 2) ? 0u : ~j;
        }
        uint32_t d, jgt, e, lt100;
        sub_bytes(i, j, d, jgt);
        sub_bytes(i, 0x64646464u, e, lt100);   // bytes of I below 100
        const uint32_t z = ~(((j & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | j | 0x7F7F7F7Fu);   // bytes of J equal to 0
        const uint32_t valid = npx == 4 ? 0x80808080u : (0x80808080u >> (8 * (4 - npx)));
        bright += __popc(~lt100 & valid);
        zero += __popc(z & valid);
        bad += __popc(jgt & valid);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (b >= npx) break;
            const unsigned bin = ((jgt >> (8 * b + 7)) & 1u) ? 16u : ((d >> (8 * b + 4)) & 15u);
            col[bin * FT] += 1u;
        }
    }
};

__global__ void __launch_bounds__(FT) features_kernel(const FeatTile *T, int n, const unsigned *chunk_base,
                                                      unsigned nchunks, unsigned *counts)
{
    __shared__ unsigned hist[17 * FT];
    __shared__ unsigned sh[NCOUNT];
    for (unsigned c = blockIdx.x; c < nchunks; c += gridDim.x) {
        if (threadIdx.x < NCOUNT) sh[threadIdx.x] = 0;
        for (int b = 0; b < 17; ++b) hist[b * FT + threadIdx.x] = 0u;   // this thread's column
        __syncthreads();
        const int t = find_chunk_tile(chunk_base, n, c);
        const FeatTile d = T[t];
        const int y0 = (int)(c - chunk_base[t]) * d.crow;
        const int rows = min(d.H, y0 + d.crow) - y0;
        Counts loc;
        loc.col = &hist[threadIdx.x];
        const bool vec = ((d.pitch & 15) == 0) && (((uintptr_t)d.I & 15) == 0) && (((uintptr_t)d.J & 15) == 0);
        // every thread strides over the chunk's 16-byte vectors (rows x W/16),
        // so narrow tiles keep the whole CTA busy and each thread has several
        // loads in flight; the ragged column tail and unaligned tiles go byte by byte
        const int nv = vec ? d.W >> 4 : 0;
        const int nvec = rows * nv;
        // (row, vector) of index e, stepped by FT = q rows + rem vectors
        const int q = nv ? FT / nv : 0, rem = FT - q * nv;
        int r = nv ? (int)threadIdx.x / nv : 0, v = (int)threadIdx.x - r * nv;
#pragma unroll 2
        for (int e = threadIdx.x; e < nvec; e += FT) {
            const size_t o = (size_t)(y0 + r) * d.pitch;
            const uint4 a = __ldg((const uint4 *)(d.I + o) + v), b = __ldg((const uint4 *)(d.J + o) + v);
            loc.add4(a.x, b.x, d.op);
            loc.add4(a.y, b.y, d.op);
            loc.add4(a.z, b.z, d.op);
            loc.add4(a.w, b.w, d.op);
            r += q;
            v += rem;
            if (v >= nv) {
                v -= nv;
                ++r;
            }
        }
        const int tw = d.W - 16 * nv;   // pixels per row not covered by vectors
        for (int e = threadIdx.x; e < rows * tw; e += FT) {
            const int r = e / tw, x = 16 * nv + (e - r * tw);
            const size_t o = (size_t)(y0 + r) * d.pitch + x;
            loc.add4(d.I[o], d.J[o], d.op, 1);
        }
        if (loc.bright) atomicAdd(&sh[16], loc.bright);
        if (loc.zero) atomicAdd(&sh[17], loc.zero);
        if (loc.bad) atomicAdd(&sh[18], loc.bad);
        __syncthreads();
        {   // bin (thread & 15) over the 16 columns of thread group (thread >> 4)
            const int bin = threadIdx.x & 15, g = threadIdx.x >> 4;
            unsigned s = 0;
#pragma unroll
            for (int q = 0; q < FT / 16; ++q) s += hist[bin * FT + g * (FT / 16) + q];
            if (s) atomicAdd(&sh[bin], s);
        }
        __syncthreads();
        if (threadIdx.x < NCOUNT && sh[threadIdx.x]) atomicAdd(&counts[t * NCOUNT + threadIdx.x], sh[threadIdx.x]);
        __syncthreads();
    }
}

__global__ void finalize_kernel(const FeatTile *T, int n, const unsigned *counts, float *feat, int *violations)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const float px = (float)T[t].H * (float)T[t].W;
    const unsigned *c = counts + t * NCOUNT;
    float *f = feat + t * NFEAT;
    for (int k = 0; k < 16; ++k) f[k] = (float)c[k] / px;
    f[16] = (float)c[16] / px;
    f[17] = (float)c[17] / px;
    f[18] = log2f((float)T[t].H) / 12.0f;
    f[19] = log2f((float)T[t].W) / 12.0f;
    if (violations) violations[t] = c[18] ? 1 : 0;
}

// ---------------------------------------------------------------------------
// MLP: parameter blob layout W1 (64x20) b1 (64) W2 (64x64) b2 (64) W3 (2x64) b3 (2)

constexpr int D0 = NFEAT, D1 = 64, D2 = 64, D3 = 2;
constexpr int OW1 = 0, OB1 = OW1 + D1 * D0, OW2 = OB1 + D1, OB2 = OW2 + D2 * D1, OW3 = OB2 + D2,
              OB3 = OW3 + D3 * D2, NP = OB3 + D3;
static_assert(NP == MLP_NPARAMS, "parameter count");

__global__ void __launch_bounds__(64) mlp_forward(const float *theta, const float *X, int n, float *Y)
{
    __shared__ float P[NP];
    __shared__ float x[D0], a1[D1], a2[D2];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) P[i] = theta[i];
    __syncthreads();
    const int j = threadIdx.x;
    for (int s = blockIdx.x; s < n; s += gridDim.x) {
        if (j < D0) x[j] = X[(size_t)s * D0 + j];
        __syncthreads();
        float z = P[OB1 + j];
        for (int i = 0; i < D0; ++i) z = fmaf(P[OW1 + j * D0 + i], x[i], z);
        a1[j] = fmaxf(z, 0.0f);
        __syncthreads();
        z = P[OB2 + j];
        for (int k = 0; k < D1; ++k) z = fmaf(P[OW2 + j * D1 + k], a1[k], z);
        a2[j] = fmaxf(z, 0.0f);
        __syncthreads();
        if (j < D3) {
            float y = P[OB3 + j];
            for (int k = 0; k < D2; ++k) y = fmaf(P[OW3 + j * D2 + k], a2[k], y);
            Y[(size_t)s * D3 + j] = y;
        }
        __syncthreads();
    }
}

// Gradient of L over the samples idx[0..nb) (idx NULL: 0..nb-1), added into grad.
__global__ void __launch_bounds__(64) mlp_grad(const float *theta, const float *X, const float *T,
                                               const int *idx, int nb, float *grad, float *loss)
{
    __shared__ float P[NP];
    __shared__ float G[NP];
    __shared__ float x[D0], z1[D1], a1[D1], z2[D2], a2[D2], dz2[D2], dy[D3];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) { P[i] = theta[i]; G[i] = 0.0f; }
    __syncthreads();
    const int j = threadIdx.x;
    const float invN = 1.0f / (float)nb;
    float lsum = 0.0f;
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        const int s = idx ? idx[b] : b;
        if (j < D0) x[j] = X[(size_t)s * D0 + j];
        __syncthreads();
        float z = P[OB1 + j];
        for (int i = 0; i < D0; ++i) z = fmaf(P[OW1 + j * D0 + i], x[i], z);
        z1[j] = z;
        a1[j] = fmaxf(z, 0.0f);
        __syncthreads();
        z = P[OB2 + j];
        for (int k = 0; k < D1; ++k) z = fmaf(P[OW2 + j * D1 + k], a1[k], z);
        z2[j] = z;
        a2[j] = fmaxf(z, 0.0f);
        __syncthreads();
        if (j < D3) {
            float y = P[OB3 + j];
            for (int k = 0; k < D2; ++k) y = fmaf(P[OW3 + j * D2 + k], a2[k], y);
            const float e = y - T[(size_t)s * D3 + j];
            dy[j] = e * invN;
            lsum += 0.5f * e * e * invN;
        }
        __syncthreads();
        // output layer
        for (int o = 0; o < D3; ++o) G[OW3 + o * D2 + j] += dy[o] * a2[j];
        if (j < D3) G[OB3 + j] += dy[j];
        float g2 = 0.0f;
        for (int o = 0; o < D3; ++o) g2 = fmaf(dy[o], P[OW3 + o * D2 + j], g2);
        dz2[j] = z2[j] > 0.0f ? g2 : 0.0f;
        __syncthreads();
        // hidden layer 2: thread j owns row j of W2
        for (int k = 0; k < D1; ++k) G[OW2 + j * D1 + k] += dz2[j] * a1[k];
        G[OB2 + j] += dz2[j];
        // hidden layer 1: thread j = unit j of layer 1
        float g1 = 0.0f;
        for (int k = 0; k < D2; ++k) g1 = fmaf(dz2[k], P[OW2 + k * D1 + j], g1);
        const float dz1 = z1[j] > 0.0f ? g1 : 0.0f;
        for (int i = 0; i < D0; ++i) G[OW1 + j * D0 + i] += dz1 * x[i];
        G[OB1 + j] += dz1;
        __syncthreads();
    }
    for (int i = threadIdx.x; i < NP; i += blockDim.x)
        if (G[i] != 0.0f) atomicAdd(&grad[i], G[i]);
    if (loss && j < D3 && lsum != 0.0f) atomicAdd(loss, lsum);
}

__global__ void adam_kernel(float *theta, float *grad, float *m, float *v, int t, float lr, float b1,
                            float b2, float eps)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NP) return;
    const float g = grad[i];
    const float mi = b1 * m[i] + (1.0f - b1) * g;
    const float vi = b2 * v[i] + (1.0f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / (1.0f - powf(b1, (float)t));
    const float vh = vi / (1.0f - powf(b2, (float)t));
    theta[i] -= lr * mh / (sqrtf(vh) + eps);
    grad[i] = 0.0f;
}

// One epoch of mini-batch Adam in one launch: a cluster of CL CTAs shares every
// step. Each CTA holds all weights in shared memory and takes a CL-th of the
// batch's samples, TS at a time; the CTAs' gradients are added over distributed
// shared memory, each CTA updates its CL-th of the parameters (Adam's moments
// stay with it for the whole epoch) and writes them into every CTA's copy. Two
// cluster barriers a step replace two launches and the global atomics.
// A step is bound by latency and shared-memory loads, not arithmetic (6 x 5504
// weights x 256 samples = 8.5 MFLOP): mlp_grad's 16 CTAs of 64 threads took one
// sample at a time, with 32-way bank conflicts in the 64 x 64 layer (a thread per
// row of stride 64); here the rows are 65 apart, a thread works on one unit of
// four samples, and the next samples are on their way while these are worked on.
// An epoch of 16 steps takes 216 us a call, 2473 with those launches (which remain
// for a device that cannot place sixteen CTAs together: rl_train_fits).
namespace cg = cooperative_groups;
constexpr int S1 = D0 + 1, S2 = D1 + 1;           // weight row strides: odd, so that a column has no bank conflicts
constexpr int PW1 = 0, PB1 = PW1 + D1 * S1, PW2 = PB1 + D1, PB2 = PW2 + D2 * S2, PW3 = PB2 + D2,
              PB3 = PW3 + D3 * D2, PPAD = (PB3 + D3 + 3) / 4 * 4;

constexpr int CL = 16;                             // CTAs (a cluster of more than eight is not portable)
constexpr int TT = 256, TS = 16;                   // threads; samples at a time: four a unit and thread group
struct TrainSmem {
    float P[PPAD];                                 // weights, padded rows
    float G[(NP + 3) / 4 * 4];                     // this CTA's gradient, flat layout
    alignas(16) float a1[TS][D1], a2[TS][D2], dz1[TS][D1], dz2[TS][D2];
    alignas(16) float x[TS][D0];
    float t[TS][D3], dy[TS][D3];
    float loss;
};

__device__ __forceinline__ int padded(int i)       // flat parameter index -> place in TrainSmem::P
{
    if (i < OB1) return PW1 + i / D0 * S1 + i % D0;
    if (i < OW2) return PB1 + (i - OB1);
    if (i < OB2) return PW2 + (i - OW2) / D1 * S2 + (i - OW2) % D1;
    return PB2 + (i - OB2);                        // b2, W3 and b3 follow each other in both
}
static_assert(PW3 - PB2 == OW3 - OB2 && PB3 - PB2 == OB3 - OB2, "layout");

__global__ void __launch_bounds__(TT) train_kernel(float *theta, float *m, float *v, const float *X, const float *T,
                                                   const int *idx, int n, int batch, int step0, float lr, float b1,
                                                   float b2, float eps, float *loss)
{
    constexpr int NG = TT / 64;                             // thread groups, 4 samples each
    constexpr int OWN = (NP + CL - 1) / CL, OPT = (OWN + TT - 1) / TT;   // parameters a CTA (a thread) updates
    constexpr int RW = D2 / NG, IW = D0 / NG;               // W2 rows, inputs of W1 whose gradients a thread adds up
    constexpr int NF = (TS * (D0 + D3) + TT - 1) / TT;      // inputs and targets a thread fetches
    static_assert(TS == 4 * NG && D0 % NG == 0 && D2 % NG == 0, "four samples a group, whole rows and columns");
    extern __shared__ __align__(16) unsigned char train_smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(train_smem);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int j = tid & 63, g = tid >> 6;
    for (int i = tid; i < NP; i += TT) S.P[padded(i)] = theta[i];
    float mo[OPT], vo[OPT];                        // Adam's moments of this thread's parameters
#pragma unroll
    for (int q = 0; q < OPT; ++q) {
        const int o = tid + q * TT, i = rank * OWN + o;
        const bool mine = o < OWN && i < NP;
        mo[q] = mine ? m[i] : 0.0f;
        vo[q] = mine ? v[i] : 0.0f;
    }
    // this CTA's samples of the batch at s0: [lo, hi) of it, in chunks of TS (at least one, maybe empty)
    auto share = [&](int s0, int &lo, int &hi) {
        const int nb = min(batch, n - s0), per = (nb + CL - 1) / CL;
        lo = min(nb, rank * per);
        hi = min(nb, lo + per);
    };
    float next[NF];                                // the next chunk's inputs and targets
    auto fetch = [&](int s0, int c0, int hi) {
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            const int e = tid + q * TT, s = e / (D0 + D3), f = e - s * (D0 + D3);
            next[q] = 0.0f;
            if (s < TS && c0 + s < hi) {
                const size_t row = (size_t)idx[s0 + c0 + s];
                next[q] = f < D0 ? X[row * D0 + f] : T[row * D3 + f - D0];
            }
        }
    };
    float lsum = 0.0f;
    int step = step0, lo, hi;
    share(0, lo, hi);
    fetch(0, lo, hi);
    for (int s0 = 0; s0 < n; s0 += batch) {
        const float invN = 1.0f / (float)min(batch, n - s0);
        const bool last = n - s0 <= batch;
        float gw2[RW], gw1[IW], gb2 = 0.0f, gb1 = 0.0f, gw3 = 0.0f, gb3 = 0.0f;
#pragma unroll
        for (int q = 0; q < RW; ++q) gw2[q] = 0.0f;
#pragma unroll
        for (int q = 0; q < IW; ++q) gw1[q] = 0.0f;
        int c0 = lo;
        do {
            const int nc = min(TS, hi - c0);       // (negative or 0 when there is nothing to do)
            __syncthreads();                       // the chunk before (or the weights' update) is done with S
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                const int e = tid + q * TT, s = e / (D0 + D3), f = e - s * (D0 + D3);
                if (s < TS) (f < D0 ? S.x[s][f] : S.t[s][f - D0]) = next[q];
            }
            __syncthreads();
            if (c0 + TS < hi) {
                fetch(s0, c0 + TS, hi);
            } else if (!last) {
                int l2, h2;
                share(s0 + batch, l2, h2);
                fetch(s0 + batch, l2, h2);
            }
            float z[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = S.P[PB1 + j];
#pragma unroll
            for (int i = 0; i < D0; i += 4) {
                const float *w = &S.P[PW1 + j * S1 + i];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 a = *(const float4 *)&S.x[4 * g + q][i];
                    z[q] = fmaf(w[3], a.w, fmaf(w[2], a.z, fmaf(w[1], a.y, fmaf(w[0], a.x, z[q]))));
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) S.a1[4 * g + q][j] = 4 * g + q < nc ? fmaxf(z[q], 0.0f) : 0.0f;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = S.P[PB2 + j];
#pragma unroll 4
            for (int k = 0; k < D1; k += 4) {
                float4 a[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = *(const float4 *)&S.a1[4 * g + q][k];
                const float *w = &S.P[PW2 + j * S2 + k];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    z[q] = fmaf(w[3], a[q].w, fmaf(w[2], a[q].z, fmaf(w[1], a[q].y, fmaf(w[0], a[q].x, z[q]))));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) S.a2[4 * g + q][j] = 4 * g + q < nc ? fmaxf(z[q], 0.0f) : 0.0f;
            __syncthreads();
            {   // output layer: eight threads per sample and output, eight products each
                const int s = tid >> 4, o = (tid >> 3) & 1, p = tid & 7;
                float y = 0.0f;
#pragma unroll
                for (int k = 0; k < D2 / 8; ++k) y = fmaf(S.P[PW3 + o * D2 + 8 * k + p], S.a2[s][8 * k + p], y);
#pragma unroll
                for (int d = 4; d; d >>= 1) y += __shfl_xor_sync(0xFFFFFFFFu, y, d);
                if (p == 0) {
                    const float e = s < nc ? y + S.P[PB3 + o] - S.t[s][o] : 0.0f;
                    S.dy[s][o] = e * invN;
                    lsum += 0.5f * e * e * invN;
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int s = 4 * g + q;
                const float d = fmaf(S.dy[s][1], S.P[PW3 + D2 + j], fmaf(S.dy[s][0], S.P[PW3 + j], 0.0f));
                S.dz2[s][j] = S.a2[s][j] > 0.0f ? d : 0.0f;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = 0.0f;
#pragma unroll 4
            for (int k = 0; k < D2; k += 4) {
                float4 d[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) d[q] = *(const float4 *)&S.dz2[4 * g + q][k];
                const float *w = &S.P[PW2 + k * S2 + j];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    z[q] = fmaf(d[q].w, w[3 * S2], fmaf(d[q].z, w[2 * S2], fmaf(d[q].y, w[S2], fmaf(d[q].x, w[0], z[q]))));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) S.dz1[4 * g + q][j] = S.a1[4 * g + q][j] > 0.0f ? z[q] : 0.0f;
            __syncthreads();
            // gradients of the chunk, all in one pass over its samples: W2 rows RW g ..., column j; W1 row j,
            // columns g, g + NG, ...; the biases and W3 where a thread has their terms at hand
#pragma unroll 4
            for (int s = 0; s < TS; ++s) {
                const float a = S.a1[s][j], d1 = S.dz1[s][j];
#pragma unroll
                for (int q = 0; q < RW; q += 4) {
                    const float4 d = *(const float4 *)&S.dz2[s][RW * g + q];
                    gw2[q] = fmaf(d.x, a, gw2[q]);
                    gw2[q + 1] = fmaf(d.y, a, gw2[q + 1]);
                    gw2[q + 2] = fmaf(d.z, a, gw2[q + 2]);
                    gw2[q + 3] = fmaf(d.w, a, gw2[q + 3]);
                }
#pragma unroll
                for (int q = 0; q < IW; ++q) gw1[q] = fmaf(d1, S.x[s][g + q * NG], gw1[q]);
                if (g == 0) gb1 += d1;
                else if (g == 1) gb2 += S.dz2[s][j];
                if (g >= NG - 2) gw3 = fmaf(S.dy[s][g - (NG - 2)], S.a2[s][j], gw3);
                if (tid < D3) gb3 += S.dy[s][tid];
            }
            c0 += TS;
        } while (c0 < hi);
#pragma unroll
        for (int q = 0; q < RW; ++q) S.G[OW2 + (RW * g + q) * D1 + j] = gw2[q];
#pragma unroll
        for (int q = 0; q < IW; ++q) S.G[OW1 + j * D0 + g + q * NG] = gw1[q];
        if (g == 0) S.G[OB1 + j] = gb1;
        else if (g == 1) S.G[OB2 + j] = gb2;
        if (g >= NG - 2) S.G[OW3 + (g - (NG - 2)) * D2 + j] = gw3;
        if (tid < D3) S.G[OB3 + tid] = gb3;
        ++step;
        const float k1 = 1.0f - powf(b1, (float)step), k2 = 1.0f - powf(b2, (float)step);
        cl.sync();                                 // every CTA's gradient is in place
#pragma unroll
        for (int q = 0; q < OPT; ++q) {
            const int o = tid + q * TT, i = rank * OWN + o;
            if (o < OWN && i < NP) {
                float gr[CL], grad = 0.0f;
#pragma unroll
                for (int r = 0; r < CL; ++r) gr[r] = *cl.map_shared_rank(&S.G[i], r);
#pragma unroll
                for (int r = 0; r < CL; ++r) grad += gr[r];
                mo[q] = b1 * mo[q] + (1.0f - b1) * grad;
                vo[q] = b2 * vo[q] + (1.0f - b2) * grad * grad;
                const float mh = mo[q] / k1, vh = vo[q] / k2;
                float *p = &S.P[padded(i)];
                const float w = *p - lr * mh / (sqrtf(vh) + eps);
#pragma unroll
                for (int r = 0; r < CL; ++r) *cl.map_shared_rank(p, r) = w;
            }
        }
        cl.sync();                                 // every CTA has the new weights; the gradients may be overwritten
        if (!last) share(s0 + batch, lo, hi);
        else break;                                // (s0 + batch may not fit an int)
    }
#pragma unroll
    for (int q = 0; q < OPT; ++q) {
        const int o = tid + q * TT, i = rank * OWN + o;
        if (o < OWN && i < NP) {
            theta[i] = S.P[padded(i)];
            m[i] = mo[q];
            v[i] = vo[q];
        }
    }
    if (tid == 0) S.loss = 0.0f;
    __syncthreads();
    if (lsum != 0.0f) atomicAdd(&S.loss, lsum);
    __syncthreads();
    if (tid == 0 && loss) atomicAdd(loss, S.loss);
}

}  // namespace rl

// ---------------------------------------------------------------------------
// host-side launchers (internal)

cudaError_t rl_features(const rl_tile *tiles, int n, void *scratch, size_t scratch_bytes, float *feat_dev,
                        int *viol_dev, int sms, cudaStream_t st, void *host_stage, size_t stage_bytes)
{
    static int occ = 0;   // resident CTAs of features_kernel per SM (it is latency-bound: fill the SMs)
    if (!occ && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, rl::features_kernel, rl::FT, 0) != cudaSuccess)
        occ = 4;
    const int grid = std::max(1, occ) * std::max(1, sms);
    // scratch: [FeatTile n][chunk_base n+1][counts n*NCOUNT]
    const size_t o_base = ((sizeof(rl::FeatTile) * n + 15) / 16) * 16;
    const size_t o_cnt = ((o_base + sizeof(unsigned) * (n + 1) + 15) / 16) * 16;
    const size_t need = o_cnt + sizeof(unsigned) * n * rl::NCOUNT;
    if (scratch_bytes < need || stage_bytes < o_cnt) return cudaErrorInvalidValue;
    unsigned char *h = (unsigned char *)host_stage;
    rl::FeatTile *F = (rl::FeatTile *)h;
    unsigned *base = (unsigned *)(h + o_base);
    unsigned acc = 0;
    for (int t = 0; t < n; ++t) {
        F[t].I = tiles[t].I; F[t].J = tiles[t].J; F[t].H = tiles[t].H; F[t].W = tiles[t].W;
        F[t].pitch = tiles[t].pitch; F[t].op = tiles[t].op;
        F[t].crow = std::max(1, std::min(tiles[t].H, rl::CHUNK_PX / std::max(tiles[t].W, 1)));
        base[t] = acc;
        acc += (unsigned)((tiles[t].H + F[t].crow - 1) / F[t].crow);
    }
    base[n] = acc;
    unsigned char *d = (unsigned char *)scratch;
    cudaError_t e = cudaMemcpyAsync(d, h, o_cnt, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d + o_cnt, 0, sizeof(unsigned) * n * rl::NCOUNT, st);
    if (e != cudaSuccess) return e;
    rl::features_kernel<<<grid, rl::FT, 0, st>>>((const rl::FeatTile *)d, n, (const unsigned *)(d + o_base), acc,
                                             (unsigned *)(d + o_cnt));
    rl::finalize_kernel<<<(n + 127) / 128, 128, 0, st>>>((const rl::FeatTile *)d, n, (const unsigned *)(d + o_cnt),
                                                         feat_dev, viol_dev);
    return cudaGetLastError();
}

size_t rl_features_scratch(int n)
{
    const size_t o_base = ((sizeof(rl::FeatTile) * n + 15) / 16) * 16;
    const size_t o_cnt = ((o_base + sizeof(unsigned) * (n + 1) + 15) / 16) * 16;
    return o_cnt + sizeof(unsigned) * n * rl::NCOUNT;
}

size_t rl_features_stage(int n)
{
    const size_t o_base = ((sizeof(rl::FeatTile) * n + 15) / 16) * 16;
    return ((o_base + sizeof(unsigned) * (n + 1) + 15) / 16) * 16;
}

cudaError_t rl_forward(const float *theta, const float *X, int n, float *Y, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    rl::mlp_forward<<<n < 1216 ? n : 1216, 64, 0, st>>>(theta, X, n, Y);
    return cudaGetLastError();
}

cudaError_t rl_grad(const float *theta, const float *X, const float *T, const int *idx, int nb, float *grad,
                    float *loss, cudaStream_t st)
{
    if (nb <= 0) return cudaSuccess;
    int g = (nb + 15) / 16;
    if (g > 304) g = 304;
    rl::mlp_grad<<<g, 64, 0, st>>>(theta, X, T, idx, nb, grad, loss);
    return cudaGetLastError();
}

cudaError_t rl_adam(float *theta, float *grad, float *m, float *v, int t, float lr, cudaStream_t st)
{
    rl::adam_kernel<<<(MLP_NPARAMS + 255) / 256, 256, 0, st>>>(theta, grad, m, v, t, lr, 0.9f, 0.999f, 1e-8f);
    return cudaGetLastError();
}

static cudaLaunchConfig_t train_config(cudaLaunchAttribute *attr, cudaStream_t st)
{
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = rl::CL;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(rl::CL);
    cfg.blockDim = dim3(rl::TT);
    cfg.dynamicSmemBytes = sizeof(rl::TrainSmem);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

bool rl_train_fits()
{
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = train_config(&attr, nullptr);
    int clusters = 0;
    cudaError_t e = cudaFuncSetAttribute(rl::train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(rl::TrainSmem));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(rl::train_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, rl::train_kernel, &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && clusters > 0;
}

cudaError_t rl_train_epoch(float *theta, float *m, float *v, const float *X, const float *T, const int *idx, int n,
                           int batch, int step0, float lr, float *loss, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = train_config(&attr, st);
    return cudaLaunchKernelEx(&cfg, rl::train_kernel, theta, m, v, X, T, idx, n, batch, step0, lr, 0.9f, 0.999f, 1e-8f,
                              loss);
}
