// Distance transform (Table II, "Distance Transform": for each foreground pixel
// the distance to the closest background pixel). What Algorithm 1's wavefront
// propagates towards -- every pixel holding the nearest background pixel
// ("site") -- is computed directly, in two separable steps (Saito and Toriwaki
// 1994): the nearest background pixel of each pixel's column, then, along the
// row, the smallest dx^2 + (column distance)^2. The result is exact and does
// not depend on any order; of equally near sites the one with the lower index
// is taken. (A wavefront passes on only the site a pixel holds, so it can miss
// the nearest one; where it does not, the two agree.)
//
//   mask_kernel    32 rows of a column per 32-bit word (bit set: background)
//   column_kernel  signed distance to the nearest background row of the column,
//                  by bit scans of the column's words (16 bits a pixel)
//   row_kernel     a row of squared column distances in shared memory; each
//                  pixel searches outwards until dx^2 reaches its best, past 128
//                  columns in runs of 32 that a run's minimum can rule out
//
// The work per pixel is a few bit operations plus about two instructions per
// column within its distance; no step waits for another pixel's result. A
// 4096^2 mask of the space between objects (distances up to 97, 112 wavefront
// levels, each a launch of dependent global loads) takes 0.141 ms, 2.63 ms as a
// wavefront; the objects of a 2048 x 3000 mask 35 us, 297 us before. The row
// search is two thirds of it (60% of the issue slots, 4.4 instructions per pixel
// and column of distance); masks and columns are bound by memory latency.
#include <algorithm>
#include <cuda_runtime.h>
#include <stdint.h>

#include "recon_check.h"
#include "recon_dt.h"

namespace dt {

constexpr unsigned INF = 0x7FFFFFFFu;   // above every squared distance (2 * 32767^2); INF + dx^2 fits 32 bits
constexpr uint32_t FAR = 32767u + 1u;   // more than any distance within a column
constexpr int LONG_WALK = 256;          // strips of a column worth a look before the walk (more than 8192 rows)
constexpr uint32_t EMPTY = 0xFFFFu;     // no background in the whole mask (its square is negative as an int)
constexpr int WMAX = 32768;             // widest row
constexpr int PAD = 128;                // columns of INF at both ends of a row in shared memory

// A kernel may be launched when the last CTAs of the one before it run, and
// waits for all of that one's results before it reads any: 4 and 5 us of a call on
// the two masks above.
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Whether the mask has any background at all: mask_kernel's warps write the call's
// number to one of 32 words, each in a line of its own (one word for all cost 2 us on a
// 4096^2 mask).
__device__ __noinline__ bool any_background(const unsigned *some, unsigned call)
{
    for (int k = 0; k < 32; k += 8) {
        bool any = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) any |= some[32 * (k + i)] == call;
        if (any) return true;
    }
    return false;
}

// A thread packs four columns of a strip of 32 rows.
__global__ void __launch_bounds__(128) mask_kernel(const uint8_t *B, int H, int W, uint32_t *M, unsigned *some,
                                                   unsigned call)
{
    const int x = 4 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    allow_next();
    if (x >= W) return;
    const bool vec = (W & 3) == 0 && ((uintptr_t)B & 3) == 0;
    const int y1 = min(H - (int)blockIdx.y * 32, 32);
    const uint8_t *p = B + (size_t)blockIdx.y * 32 * W + x;
    uint32_t m[4] = {0u, 0u, 0u, 0u};
    for (int r0 = 0; r0 < y1; r0 += 16) {   // 16 rows' loads in flight
        uint32_t v[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            v[r] = 0xFFFFFFFFu;
            if (r0 + r < y1) {
                const uint8_t *q = p + (size_t)(r0 + r) * W;
                if (vec) {
                    v[r] = __ldg((const uint32_t *)q);
                } else {
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if (x + b < W && q[b] == 0) v[r] &= ~(0xFFu << (8 * b));
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 16; ++r)
#pragma unroll
            for (int b = 0; b < 4; ++b) m[b] |= (((v[r] >> (8 * b)) & 255u) == 0u ? 1u : 0u) << (r0 + r);
    }
    if (m[0] | m[1] | m[2] | m[3]) some[32 * ((4 * (blockIdx.x + blockIdx.y) + (threadIdx.x >> 5)) & 31)] = call;
    uint32_t *o = M + (size_t)blockIdx.y * W + x;
    if ((W & 3) == 0) {
        *(uint4 *)o = make_uint4(m[0], m[1], m[2], m[3]);
    } else {
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (x + b < W && RK_CHECK(blockIdx.y < gridDim.y && 32 * (int)blockIdx.y < H, CK_WORD)) o[b] = m[b];
    }
}

// For a strip of two columns without background: EMPTY when the mask has none at all.
// Looked at after the walks to both ends of the column, and before them where they are
// LONG: a mask without background took 2.2 ms at 4096^2 and 88 ms at 16384^2, and takes
// 97 us and 0.80 ms. (Asked within every walk it takes 64 us, but other masks of 4096^2
// 1 us more; asked before every walk, those of 8192^2 8 us more.)
__device__ __noinline__ bool empty_strip(const unsigned *some, unsigned call, uint16_t *G, int y0, int y1, int pitch)
{
    if (any_background(some, call)) return false;
    // (in row WMAX - 1, EMPTY is the distance to row 0: that row is searched)
    for (int y = y0; y < y1; ++y) *(uint32_t *)(G + (size_t)y * pitch) = (y == WMAX - 1 ? FAR : EMPTY) * 0x10001u;
    return true;
}

// A thread takes two columns of a strip of 32 rows. The nearest background above
// and below the strip comes from the words of the strips around it, eight at a
// time (a walk word by word waits for one load after another). Then, as two u16
// lanes, the distance downwards for all rows (kept in registers) and upwards. G:
// rows of `pitch` (even) distances, FAR or more without background; with SITE
// bit 15 says "upwards" (a tie goes up, to the lower index) and FAR alone means
// none. EMPTY everywhere says that the mask has no background at all, so that the
// rows are not searched from end to end for nothing.
template <bool SITE, bool LONG>
__global__ void __launch_bounds__(128) column_kernel(const uint32_t *M, int H, int W, uint16_t *G, int pitch,
                                                     const unsigned *some, unsigned call)
{
    const int x = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    allow_next();
    wait_previous();
    if (x >= W) return;
    const int s = blockIdx.y, ns = gridDim.y, y0 = 32 * s, xb = min(x + 1, W - 1);
    const uint32_t m[2] = {M[(size_t)s * W + x], M[(size_t)s * W + xb]};
    if (LONG && !m[0] && empty_strip(some, call, G + x, y0, min(H, y0 + 32), pitch)) return;
    uint32_t up, dn;   // distances from the row before / after the strip
    auto word = [&](int t, int c) {
        return RK_CHECK(t >= 0 && t < ns && c < W, CK_WORD) ? M[(size_t)t * W + c] : 0u;
    };
    {
        uint32_t u[2] = {FAR, FAR}, d[2] = {FAR, FAR};
        // a strip whose first (last) row is background needs no look above (below)
        bool more0 = !(m[0] & 1u), more1 = !(m[1] & 1u);
        for (int t = s - 1; t >= 0 && (more0 || more1); t -= 8) {
            uint32_t a[8], b[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                a[k] = more0 && t - k >= 0 ? word(t - k, x) : 0u;
                b[k] = more1 && t - k >= 0 ? word(t - k, xb) : 0u;
            }
#pragma unroll
            for (int k = 7; k >= 0; --k) {
                if (a[k]) { u[0] = (uint32_t)(y0 - 1 - (32 * (t - k) + 31 - __clz(a[k]))); more0 = false; }
                if (b[k]) { u[1] = (uint32_t)(y0 - 1 - (32 * (t - k) + 31 - __clz(b[k]))); more1 = false; }
            }
        }
        more0 = !(m[0] >> 31);
        more1 = !(m[1] >> 31);
        for (int t = s + 1; t < ns && (more0 || more1); t += 8) {
            uint32_t a[8], b[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                a[k] = more0 && t + k < ns ? word(t + k, x) : 0u;
                b[k] = more1 && t + k < ns ? word(t + k, xb) : 0u;
            }
#pragma unroll
            for (int k = 7; k >= 0; --k) {
                if (a[k]) { d[0] = (uint32_t)(32 * (t + k) + __ffs(a[k]) - 1 - (y0 + 32)); more0 = false; }
                if (b[k]) { d[1] = (uint32_t)(32 * (t + k) + __ffs(b[k]) - 1 - (y0 + 32)); more1 = false; }
            }
        }
        if (!m[0] && u[0] == FAR && d[0] == FAR && empty_strip(some, call, G + x, y0, min(H, y0 + 32), pitch)) return;
        up = u[0] | u[1] << 16;
        dn = d[0] | d[1] << 16;
    }
    // lanes of ones where row r is background: bit r of both words moved to the sign and spread
    auto bg = [&](int r) {
        uint32_t o;
        asm("prmt.b32 %0, %1, %2, 0xFFBB;" : "=r"(o) : "r"(m[0] << (31 - r)), "r"(m[1] << (31 - r)));
        return o;
    };
    uint32_t down[32];
#pragma unroll
    for (int r = 31; r >= 0; --r) {
        dn = (dn + 0x00010001u) & ~bg(r);
        down[r] = dn;
    }
    const int rows = min(H - y0, 32);
    uint16_t *o = G + (size_t)y0 * pitch + x;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        up = (up + 0x00010001u) & ~bg(r);
        if (r < rows) {
            uint32_t v;
            asm("min.u16x2 %0, %1, %2;" : "=r"(v) : "r"(up), "r"(down[r]));
            if (SITE) {
                uint32_t w = 0;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const uint32_t g = (v >> (16 * c)) & 0xFFFFu, u = (up >> (16 * c)) & 0xFFFFu;
                    w |= (g >= FAR ? FAR : (u == g && g ? g | 0x8000u : g)) << (16 * c);
                }
                v = w;
            }
            if (RK_CHECK(y0 + r < H && x + 1 < pitch, CK_COLUMN)) *(uint32_t *)(o + (size_t)r * pitch) = v;
        }
    }
}

// A row of squared column distances in shared memory (q, PAD x INF before and
// PAD + 2 behind it) and the minimum of each run of 32 (low). All threads.
template <bool SITE>
__device__ __forceinline__ void load_row(const uint16_t *row, int W, int pitch, int y, uint32_t *q, uint32_t *low, uint16_t *gs)
{
    for (int x = threadIdx.x; x < (W + 31) / 32 * 32; x += blockDim.x) {
        const uint32_t raw = x < pitch ? row[x] : FAR;   // (an odd row is followed by a copy of its last distance)
        uint32_t g = raw, v;
        if (SITE) {
            if (raw != EMPTY || y == WMAX - 1) g &= 0x7FFFu;   // (there: row 0)
            v = raw == FAR ? INF : g * g;
        } else {
            v = raw - FAR <= 32u ? INF : g * g;
        }
        if (x < pitch && RK_CHECK(x < W + PAD + 2, CK_ROW)) {
            q[x] = v;
            if (SITE && x < W) gs[x] = (uint16_t)raw;
        }
        const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, v);
        if ((threadIdx.x & 31) == 0) low[x >> 5] = mn;
    }
}

__device__ __forceinline__ void pad_row(int W, uint32_t *q)
{
    for (int i = threadIdx.x; i < PAD + 2; i += blockDim.x) {
        if (i < PAD) q[i - PAD] = INF;
        q[W + i] = INF;
    }
}

// Columns further than PAD from x: whole runs of 32 are skipped when even their
// minimum is too far. take(column, squared offset), beyond(lower bound): no use.
template <class Take, class Beyond>
__device__ __forceinline__ void search_far(int x, int W, const uint32_t *low, Take take, Beyond beyond)
{
    for (int c = x - PAD - 1; c >= 0; --c) {
        const uint32_t d = (uint32_t)((x - c) * (x - c));
        if (beyond(d)) break;
        if ((c & 31) == 31 && beyond(d + low[c >> 5])) { c -= 31; continue; }
        take(c, d);
    }
    for (int c = x + PAD + 1; c < W; ++c) {
        const uint32_t d = (uint32_t)((c - x) * (c - x));
        if (beyond(d)) break;
        if ((c & 31) == 0 && beyond(d + low[c >> 5])) { c += 31; continue; }
        take(c, d);
    }
}

// Distances only. Two neighbouring pixels a thread: a pair of columns (one
// 64-bit load) gives each of them two candidates, one add-and-min instruction
// each, so a column costs 1.5 instructions a pixel and side (one pixel a thread
// with 32-bit loads nearly doubles the 4096^2 mask's call).
__global__ void row_kernel(const uint16_t *G, int H, int W, int pitch, unsigned *d2)
{
    extern __shared__ __align__(16) uint32_t dt_smem[];
    uint32_t *const q = dt_smem + PAD, *const low = q + (W + 1) / 2 * 2 + PAD + 2;
    pad_row(W, q);
    wait_previous();
    for (int y = blockIdx.x; y < H; y += gridDim.x) {
        __syncthreads();                                            // the row before is done with
        load_row<false>(G + (size_t)y * pitch, W, pitch, y, q, low, nullptr);
        __syncthreads();
        for (int x = 2 * threadIdx.x; x < W; x += 2 * blockDim.x) {
            const uint2 own = *(const uint2 *)&q[x];
            uint32_t b0 = __viaddmin_u32(own.y, 1u, own.x), b1 = __viaddmin_u32(own.x, 1u, own.y);
            int j = 2;                                              // columns x - j, x - j + 1 and x + j, x + j + 1
            for (; j <= PAD; j += 4) {
                if ((j - 1) * (j - 1) >= max((int)b0, (int)b1)) break;   // (at once for EMPTY: both are negative)
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    if (!RK_CHECK(x - j - k >= -PAD && x + j + k + 1 < W + PAD + 2, CK_ROW)) continue;
                    const uint2 l = *(const uint2 *)&q[x - j - k], r = *(const uint2 *)&q[x + j + k];
                    const uint32_t s0 = (uint32_t)((j + k - 1) * (j + k - 1)), s1 = (uint32_t)((j + k) * (j + k)),
                                   s2 = (uint32_t)((j + k + 1) * (j + k + 1));
                    b0 = __viaddmin_u32(l.x, s1, __viaddmin_u32(l.y, s0, b0));
                    b1 = __viaddmin_u32(l.x, s2, __viaddmin_u32(l.y, s1, b1));
                    b0 = __viaddmin_u32(r.x, s1, __viaddmin_u32(r.y, s2, b0));
                    b1 = __viaddmin_u32(r.x, s0, __viaddmin_u32(r.y, s1, b1));
                }
            }
            if (j > PAD) {
                search_far(x, W, low, [&](int c, uint32_t d) { if (RK_CHECK(c >= 0 && c < W, CK_ROW)) b0 = min(b0, q[c] + d); }, [&](uint32_t d) { return d >= b0; });
                if (x + 1 < W)
                    search_far(x + 1, W, low, [&](int c, uint32_t d) { if (RK_CHECK(c >= 0 && c < W, CK_ROW)) b1 = min(b1, q[c] + d); },
                               [&](uint32_t d) { return d >= b1; });
            }
            unsigned *o = d2 + (size_t)y * W + x;
            b0 = b0 >= INF ? 0xFFFFFFFFu : b0;
            b1 = b1 >= INF ? 0xFFFFFFFFu : b1;
            if ((W & 1) == 0 && ((uintptr_t)d2 & 7) == 0) {
                *(uint2 *)o = make_uint2(b0, b1);
            } else {
                o[0] = b0;
                if (x + 1 < W) o[1] = b1;
            }
        }
    }
}

// Distances and sites: of equally near sites the one with the lowest index, so
// columns at exactly the best distance count too.
__global__ void row_site_kernel(const uint16_t *G, int H, int W, int pitch, unsigned *d2, int *site)
{
    extern __shared__ __align__(16) uint32_t dt_smem[];
    uint32_t *const q = dt_smem + PAD, *const low = q + (W + 1) / 2 * 2 + PAD + 2;
    uint16_t *const gs = (uint16_t *)(low + (W + 31) / 32);         // the column distances with their direction
    pad_row(W, q);
    wait_previous();
    for (int y = blockIdx.x; y < H; y += gridDim.x) {
        __syncthreads();
        load_row<true>(G + (size_t)y * pitch, W, pitch, y, q, low, gs);
        __syncthreads();
        auto site_of = [&](int c) {
            if (!RK_CHECK(c >= 0 && c < W, CK_ROW)) return 0;
            const int g = gs[c];
            return (y + (g & 0x8000 ? -(g & 0x7FFF) : g)) * W + c;
        };
        for (int x = threadIdx.x; x < W; x += blockDim.x) {
            uint32_t best = q[x];
            int bs = best >= INF ? 0x7FFFFFFF : site_of(x);
            auto take = [&](int c, uint32_t d) {
                if (!RK_CHECK(c >= -PAD && c < W + PAD + 2, CK_ROW)) return;
                const uint32_t v = q[c] + d;
                if (v > best || v >= INF) return;
                const int s = site_of(c);
                if (v < best || s < bs) bs = s;
                best = v;
            };
            auto beyond = [&](uint32_t d) { return d > best; };
            int dx = 1;
            for (; dx <= PAD; ++dx) {
                const uint32_t d = (uint32_t)(dx * dx);
                if ((int)d > (int)best) break;   // (at once for EMPTY, which is negative)
                take(x - dx, d);
                take(x + dx, d);
            }
            if (dx > PAD) search_far(x, W, low, take, beyond);
            const size_t p = (size_t)y * W + x;
            d2[p] = best >= INF ? 0xFFFFFFFFu : best;
            site[p] = best >= INF ? -1 : bs;
        }
    }
}

}  // namespace dt

RK_CHECK_READER(dt_read_checks)

static size_t mask_bytes(int H, int W) { return (((size_t)((H + 31) / 32) * W * sizeof(uint32_t)) + 255) / 256 * 256; }
static int g_pitch(int W) { return (W + 1) / 2 * 2; }

// Shared memory of the row kernels: the padded row, its runs' minima, with sites the distances with their direction.
static size_t row_smem(int W, bool site)
{
    return sizeof(uint32_t) * ((size_t)(W + 1) / 2 * 2 + 2 * dt::PAD + 2 + (W + 31) / 32) +
           (site ? sizeof(uint16_t) * (size_t)W : 0);
}

size_t dt_scratch_bytes(int H, int W)
{
    return DT_HEADER + mask_bytes(H, W) + (size_t)H * g_pitch(W) * sizeof(uint16_t);
}

// Launches a kernel behind the one before it on the stream, as its dependent.
template <class... P, class... A>
static cudaError_t launch_after(void (*f)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f, P(args)...);
}

int dt_run(const uint8_t *B, int H, int W, int *site, unsigned *d2, void *scratch, unsigned call, int sms, cudaStream_t st)
{
    unsigned *some = (unsigned *)scratch;
    uint32_t *M = (uint32_t *)((unsigned char *)scratch + DT_HEADER);
    uint16_t *G = (uint16_t *)((unsigned char *)M + mask_bytes(H, W));
    const int ns = (H + 31) / 32, pitch = g_pitch(W);
    dt::mask_kernel<<<dim3((W + 511) / 512, ns), 128, 0, st>>>(B, H, W, M, some, call);
    const dim3 cg((W + 255) / 256, ns);
    cudaError_t e = cudaGetLastError();
    const bool far = ns > dt::LONG_WALK;
    if (e == cudaSuccess)
        e = launch_after(site ? (far ? dt::column_kernel<true, true> : dt::column_kernel<true, false>)
                              : (far ? dt::column_kernel<false, true> : dt::column_kernel<false, false>),
                         cg, 128, 0, st, M, H, W, G, pitch, some, call);
    // a CTA per row; more threads where a wide row's shared memory leaves room for few CTAs
    const int px = site ? W : (W + 1) / 2;
    const int T = W > 8192 ? 1024 : std::min(256, (px + 31) / 32 * 32);
    const size_t smem = row_smem(W, site != nullptr);
    // the limit belongs to the kernel, not to the call: the same for every call (that of the widest row),
    // so that calls of other threads cannot lower it between this line and the launch
    const void *fn = site ? (const void *)dt::row_site_kernel : (const void *)dt::row_kernel;
    if (smem > 48 * 1024 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)row_smem(dt::WMAX, site != nullptr)) != cudaSuccess)
        return DT_ECUDA;
    const int grid = std::min(H, 64 * std::max(1, sms));
    if (e == cudaSuccess)
        e = site ? launch_after(dt::row_site_kernel, dim3(grid), T, smem, st, G, H, W, pitch, d2, site)
                 : launch_after(dt::row_kernel, dim3(grid), T, smem, st, G, H, W, pitch, d2);
    return e == cudaSuccess ? DT_OK : DT_ECUDA;
}
